"""Which PIPG loop ran: the fixed-point one on ordinary data, in every form
that uses it, the FP64 one behind it where the data does not suit, and none of
either where the launch chooses another loop."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _step(torch, S, p, oracle, x0, Ns, counts, phi=0.0):
    n, nx, nu, B = int(max(Ns)), len(p["P_x"]), int(p["nu"]), len(Ns)
    X, U = np.zeros((B, n, nx)), np.zeros((B, n, nu))
    for b, N in enumerate(Ns):
        X[b, :N], U[b, :N] = oracle.init_guess(p, int(N), x0[b])
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    z = lambda *s: torch.zeros(B, *s, dtype=torch.float64, device="cuda")  # noqa: E731
    ws = dict(xh=z(n, nx), uh=z(n, nu), mup=z(n - 1, nx), mum=z(n - 1, nx), phi=z(n - 1, nx) + phi, th=z(n - 1))
    S.scp_step(d(x0), d(X), d(U), ws, d(np.asarray(Ns, np.int32)), d(np.array([counts] * B, np.int32)))


@pytest.mark.parametrize("model,nu", [("6dof", 4), ("6dof", 7), ("3dof", 4)])
def test_steps_run_in_fixed_point(torch_cuda, oracle, inputs, model, nu):
    from paper_2404_18034_gb300.pdg_mc import Solver
    p = inputs.load_params(model=model, nu=nu)
    Ns = [2, 3, 8, 13, 17, 24, 31, 32]
    x0 = inputs.dispersion(p, len(Ns), 5, "bj")
    S = Solver(p, 32)
    assert S.pipg_loops() == dict(fixed_point=0, again=0, fp64=0)
    _step(torch_cuda, S, p, oracle, x0, Ns, (20, 60))
    r = S.pipg_loops()
    assert r["fixed_point"] == len(Ns) and r["fp64"] == 0
    _step(torch_cuda, S, p, oracle, x0, Ns, (20, 3), phi=1e70)  # no unit suits
    r = S.pipg_loops()
    assert r["fixed_point"] == len(Ns) and r["fp64"] == len(Ns)
    S.set_threads(512)  # outside the fixed-point loop's thread counts
    _step(torch_cuda, S, p, oracle, x0, Ns, (20, 60))
    assert S.pipg_loops() == r
    S.close()


def test_solves_run_in_fixed_point(torch_cuda, inputs):
    """Every solve's SCP iterations count one loop each, in all modes, the
    no-allocation entry point and the gradient."""
    from paper_2404_18034_gb300.pdg_mc import Solver
    torch = torch_cuda
    p = inputs.load_params(scp_jmax=2, pipg_jmax=100)
    B = 5
    x0 = torch.from_numpy(inputs.dispersion(p, B, 6, "bj")).cuda()
    N = torch.tensor([10, 9, 10, 12, 12], dtype=torch.int32, device="cuda")
    S = Solver(p, 12)
    want = 0
    calls = [lambda m=m: S.solve(x0, N, mode=m) for m in (0, 1, 2)] + [lambda: S.solve_noalloc(x0, N), lambda: S.grad(x0, N)]
    for call in calls:
        call()
        want += 2 * B
        r = S.pipg_loops()
        assert r["fixed_point"] == want and r["fp64"] == 0
    S.close()
    S = Solver(p, 5)  # whole solves on fewer than six nodes: the FP64 loop's kernels
    for mode in (0, 1):
        S.solve(x0, mode=mode)
    assert S.pipg_loops() == dict(fixed_point=0, again=0, fp64=0)
    S.close()
    for args in ((inputs.load_params(scp_jmax=2, pipg_jmax=100, soc_thrust=1), 0), (p, 1)):
        S = Solver(args[0], 12, args[1])  # the thrust projection; FP32
        S.solve(x0, N)
        assert S.pipg_loops() == dict(fixed_point=0, again=0, fp64=0)
        S.close()
