"""The plain form's discretization by column classes against the oracle, through
single SCP iterations whose updated trajectories depend on every block: grids
where a wave ends inside a warp (one interval, 16 and 17, the largest), both
models and control sizes, path constraints active (their row is the one the
single columns integrate), FP64 and FP32."""
import numpy as np
import pytest

from gpu_helpers import RTOL, assert_scaled_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("model,nu", [("6dof", 4), ("6dof", 7), ("3dof", 4)])
def test_defect_and_step_on_ragged_waves(oracle, inputs, model, nu, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_18034_gb300.pdg_mc import Solver
    p = inputs.load_params(model=model, nu=nu, glide_slope=1)
    Ns = np.array([2, 3, 9, 16, 17, 18, 31, 32], np.int32)
    n, B, nx = 32, len(Ns), len(p["P_x"])
    x0 = inputs.dispersion(p, B, 17, "bj")
    rng = np.random.default_rng(8)
    X, U = np.zeros((B, n, nx)), np.zeros((B, n, nu))
    for b, N in enumerate(Ns):
        X[b, :N], U[b, :N] = oracle.init_guess(p, int(N), x0[b])
        X[b, 1:N] += 0.03 * p["P_x"] * rng.normal(size=(N - 1, nx))
        U[b, :N] += 0.03 * p["P_u"][:nu] * rng.normal(size=(N, nu))
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    z = lambda *s: torch.zeros(B, *s, dtype=torch.float64, device="cuda")  # noqa: E731
    S = Solver(p, n, precision)
    ws = dict(xh=z(n, nx), uh=z(n, nu), mup=z(n - 1, nx), mum=z(n - 1, nx), phi=z(n - 1, nx), th=z(n - 1))
    gX, gU = d(X), d(U)
    o = S.scp_step(d(x0), gX, gU, ws, d(Ns), d(np.array([[40, 20]] * B, np.int32)))
    torch.cuda.synchronize()
    # FP32: 40 RK4 stages, 40 power and 20 PIPG iterations at 6e-8 a rounding,
    # their squares in the norm, on blocks of up to 1e2: 1e-3 of the scales
    rtol = RTOL if precision == 0 else 1e-3
    for b, N in enumerate(Ns):
        oX, oU, ow = X[b, :N].copy(), U[b, :N].copy(), oracle.PDState(int(N), nu, model)
        r = oracle.scp_iterate(p, x0[b], oX, oU, ow, force_pow=40, force_pipg=20)
        assert abs(o["defect"][b].item() - r["defect"]) <= rtol * max(r["defect"], 1.0)
        assert abs(o["sigma"][b].item() - r["sigma"]) <= rtol * r["sigma"]
        assert_scaled_close(gX[b, :N].cpu().numpy(), oX, p["P_x"], rtol, what=f"X N={N}")
        assert_scaled_close(gU[b, :N].cpu().numpy(), oU, p["P_u"][:nu], rtol, what=f"U N={N}")
