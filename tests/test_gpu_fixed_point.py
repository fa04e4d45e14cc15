"""The fixed-point PIPG loop of FP64 instances (phase_pipg_fx): chained SCP
iterations with forced counts against the oracle at the sizes where its work
split is ragged (groups that end inside a warp, one interval, the largest
grid), both control sizes and both models; counts that end between its looks
at the magnitudes; a warm start far above the cold start's range (a coarser
unit) and one that no unit suits (the FP64 loop behind it)."""
import numpy as np
import pytest

from gpu_helpers import RTOL, assert_scaled_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _chain(torch, oracle, inputs, model, nu, Ns, counts, scale=0.0, **ov):
    from paper_2404_18034_gb300.pdg_mc import Solver
    p = inputs.load_params(model=model, nu=nu, **ov)
    n = int(max(Ns))
    B, nx = len(Ns), len(p["P_x"])
    S = Solver(p, n)
    x0 = inputs.dispersion(p, B, 31, "bj")
    X, U = np.zeros((B, n, nx)), np.zeros((B, n, nu))
    ws = {k: np.zeros((B, n if k in ("xh", "uh") else n - 1) + {"uh": (nu,), "th": ()}.get(k, (nx,)))
          for k in ("xh", "uh", "mup", "mum", "phi", "th")}
    rng = np.random.default_rng(4)
    ows = []
    for b, N in enumerate(Ns):
        X[b, :N], U[b, :N] = oracle.init_guess(p, int(N), x0[b])
        o = oracle.PDState(int(N), nu, model)
        if scale:
            o.phi[...] = scale * rng.normal(size=o.phi.shape)
            ws["phi"][b, :N - 1] = o.phi
        ows.append(o)
    oX = [X[b, :N].copy() for b, N in enumerate(Ns)]
    oU = [U[b, :N].copy() for b, N in enumerate(Ns)]
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    gX, gU, gw = d(X), d(U), {k: d(v) for k, v in ws.items()}
    gone = set()  # instances that diverged in the oracle: a few power iterations can miss sigma
    for fp, fj in counts:
        S.scp_step(d(x0), gX, gU, gw, d(np.asarray(Ns, np.int32)), d(np.array([[fp, fj]] * B, np.int32)))
        torch.cuda.synchronize()
        assert S.launch_info()["pipg_form"] == 1
        for b, N in enumerate(Ns):
            if b in gone:
                continue
            oracle.scp_iterate(p, x0[b], oX[b], oU[b], ows[b], force_pow=fp, force_pipg=fj)
            if not np.isfinite(oX[b]).all():  # then it diverges here too, and holds no values to compare
                assert not torch.isfinite(gX[b, :N]).all()
                gone.add(b)
                continue
            assert_scaled_close(gX[b, :N].cpu().numpy(), oX[b], p["P_x"], what=f"X N={N}")
            assert_scaled_close(gU[b, :N].cpu().numpy(), oU[b], p["P_u"][:nu], what=f"U N={N}")
            for k in ws:
                ref = getattr(ows[b], k)
                assert_scaled_close(gw[k][b].cpu().numpy()[:ref.shape[0]], ref, max(1.0, scale), what=f"{k} N={N}")
    return gone


@pytest.mark.parametrize("model,nu", [("6dof", 4), ("6dof", 7), ("3dof", 4)])
@pytest.mark.parametrize("Ns", [[2, 3, 4, 5], [8, 9, 12, 13], [16, 17, 31, 32]], ids=["small", "middle", "large"])
def test_ragged_grids(torch_cuda, oracle, inputs, model, nu, Ns):
    _chain(torch_cuda, oracle, inputs, model, nu, Ns, [(7, 1), (5, 43), (9, 120)])


@pytest.mark.parametrize("scale", [3e4, 1e70])
def test_large_warm_starts(torch_cuda, oracle, inputs, scale):
    """RTOL is relative to the largest of each array and the warm start's
    scale: the iteration is linear in the warm start wherever it projects
    nothing, so both sides carry it alike."""
    assert RTOL == 1e-6
    _chain(torch_cuda, oracle, inputs, "6dof", 4, [10, 15], [(7, 3)], scale=scale)


def test_stop_tests_off_the_window(torch_cuda, oracle, inputs):
    """Stop tests every 1, 7 and 25 iterations (the magnitudes are looked at
    every 10): counts and results equal the oracle's free runs."""
    torch = torch_cuda
    from paper_2404_18034_gb300.pdg_mc import Solver
    for jc in (1, 7, 25):
        p = inputs.load_params(pipg_jcheck=jc, pipg_eps_rel=1e-4)
        x0 = inputs.dispersion(p, 3, 12, "bj")
        S = Solver(p, 10)
        o = S.solve(torch.from_numpy(x0).cuda(), mode=0)
        torch.cuda.synchronize()
        for b in range(3):
            r = oracle.solve(p, 10, x0[b])
            assert int(o["status"][b]) == r["status"] and int(o["scp_iters"][b]) == r["scp_iters"]
            assert int(o["pipg_iters"][b]) == int(r["pipg_iters"])
            if r["status"] == 0:
                assert_scaled_close(o["X"][b].cpu().numpy(), r["X"], p["P_x"], what=f"X jcheck={jc}")
