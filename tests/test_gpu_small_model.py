"""A caller's model of three states (tests/models/pdg_model_vertical.cuh): the
fixed-point PIPG against the FP64 loop (a thread count above the fixed-point
loop's) over chained SCP iterations with forced counts, ragged grids."""
import os

import numpy as np
import pytest

from gpu_helpers import assert_scaled_close

pytestmark = pytest.mark.gpu
HEADER = os.path.join(os.path.dirname(os.path.abspath(__file__)), "models", "pdg_model_vertical.cuh")


def test_three_states(inputs, tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_18034_gb300 import build
    from paper_2404_18034_gb300.pdg_mc import Solver
    lib = build.build_model(HEADER, str(tmp_path / "libpdg_mc_vertical.so"))
    p = inputs.load_params(model="3dof")
    keep = [0, 4, 7]  # m, v_x, y of the 3-DoF model
    P_x = np.asarray(p["P_x"])[keep]
    p.update(model="custom", P_x=P_x, z_f=np.asarray(p["z_f"])[keep], fix_f=[0, 1, 0])
    Ns = np.array([13, 2, 5, 12], np.int32)
    B, n, nx, nu = len(Ns), 13, 3, 4
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    x0 = inputs.dispersion(inputs.load_params(model="3dof"), B, 3, "bj")[:, [0, 4]]
    X, U = np.zeros((B, n, nx)), np.zeros((B, n, nu))
    for b, N in enumerate(Ns):
        t = np.linspace(0, 1, N)[:, None]
        X[b, :N, :2] = (1 - t) * x0[b] + t * np.array([0.5 * (x0[b, 0] + p["m_dry"]), p["z_f"][1]])
        U[b, :N, 0] = X[b, :N, 0] * np.linalg.norm(p["g_I"])
        U[b, :N, 3] = p["tf_guess"]
    res = []
    for threads in (0, 288):
        S = Solver(p, n, library=lib)
        assert S.nx == nx
        S.set_threads(threads)
        ws = {k: torch.zeros(B, *s, dtype=torch.float64, device="cuda") for k, s in
              dict(xh=(n, nx), uh=(n, nu), mup=(n - 1, nx), mum=(n - 1, nx), phi=(n - 1, nx), th=(n - 1,)).items()}
        gX, gU = d(X), d(U)
        for fp, fj in ((20, 45), (20, 120)):
            S.scp_step(d(x0), gX, gU, ws, d(Ns), d(np.array([[fp, fj]] * B, np.int32)))
        torch.cuda.synchronize()
        res.append(dict(X=gX.cpu().numpy(), U=gU.cpu().numpy(), **{k: v.cpu().numpy() for k, v in ws.items()}))
        S.close()
    assert np.isfinite(res[1]["X"]).all() and np.abs(res[1]["X"] - X).max() > 1e-3
    scale = dict(X=P_x, U=np.asarray(p["P_u"])[:nu])
    for k in res[0]:
        assert_scaled_close(res[0][k], res[1][k], scale.get(k, 1.0), what=k)
