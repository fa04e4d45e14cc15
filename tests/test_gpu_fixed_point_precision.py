"""The fixed-point PIPG loop against the FP64 loop (a thread count outside the
fixed-point loop's range) on the same reference and warm start, short and long
forced counts: exact-penalty weights far above every iterate."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# Both loops' errors are of the size of FP64 rounding carried through the
# iterations, at most some 1e-14 of an array's largest entry after 500.
TOL = 1e-12


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _both(torch, oracle, p, x0, Ns, counts, phi=0.0):
    """Chained SCP iterations in fixed point from phi; each is repeated from
    the same state by the FP64 loop.  Returns the two sides after every
    iteration and the handle's counts."""
    from paper_2404_18034_gb300.pdg_mc import Solver
    n, nx, nu, B = int(max(Ns)), len(p["P_x"]), int(p["nu"]), len(Ns)
    X, U = np.zeros((B, n, nx)), np.zeros((B, n, nu))
    for b, N in enumerate(Ns):
        X[b, :N], U[b, :N] = oracle.init_guess(p, int(N), x0[b])
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    s = dict(X=d(X), U=d(U))
    for k, sh in dict(xh=(n, nx), uh=(n, nu), mup=(n - 1, nx), mum=(n - 1, nx), phi=(n - 1, nx), th=(n - 1,)).items():
        s[k] = torch.zeros(B, *sh, dtype=torch.float64, device="cuda")
    s["phi"] += phi
    fx, fp = Solver(p, n), Solver(p, n)
    fp.set_threads(512)
    out = []
    for c in counts:
        t = {k: v.clone() for k, v in s.items()}
        for S, a in ((fx, s), (fp, t)):
            S.scp_step(d(x0), a["X"], a["U"], a, d(np.asarray(Ns, np.int32)), d(np.array([c] * B, np.int32)))
        torch.cuda.synchronize()
        out.append(({k: v.cpu().numpy() for k, v in s.items()}, {k: v.cpu().numpy() for k, v in t.items()}))
    r = fx.pipg_loops()
    assert fp.pipg_loops() == dict(fixed_point=0, again=0, fp64=0)
    fx.close(), fp.close()
    return out, r


def _close(out, what):
    for i, (a, b) in enumerate(out):
        for k in ("xh", "uh", "mup", "mum", "phi", "th"):
            for n in range(len(b[k])):
                # (the CTCS duals against the duals' scale: they start from zero)
                top = max(np.abs(b[k][n]).max(), np.abs(b["phi"][n]).max() if k == "th" else 0.0)
                err = np.abs(a[k][n] - b[k][n]).max()
                assert err <= TOL * top, f"{what}, iteration {i}, {k} of instance {n}: {err:.2e} of {top:.2e}"


@pytest.mark.parametrize("w_ep", [1e2, 1e6, 1e8, 1e13, 1e20])
def test_penalty_weight(torch_cuda, oracle, inputs, w_ep):
    """The weight is no iterate: it must not set the unit they are held in."""
    p = inputs.load_params(w_ep=w_ep)
    Ns = [10, 15, 12]
    out, r = _both(torch_cuda, oracle, p, inputs.dispersion(p, len(Ns), 8, "bj"), Ns,
                   [(30, 20), (30, 60), (30, 20), (30, 500)])
    assert r["fixed_point"] == 4 * len(Ns) and r["fp64"] == 0
    _close(out, f"w_ep {w_ep:g}")
