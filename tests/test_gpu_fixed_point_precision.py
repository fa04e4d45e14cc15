"""The fixed-point PIPG loop against the FP64 loop (a thread count outside the
fixed-point loop's range) on the same reference and warm start, short and long
forced counts: exact-penalty weights far above every iterate; parameters of
other scales, where the FP64 loop has to take over; iterates that outgrow the
unit; stop tests at every distance from the looks at the magnitudes."""
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


def _scaled(inputs, key=None, part=None, f=1.0, **ov):
    p = inputs.load_params(**ov)
    if key:
        p[key] = np.array(p[key], float)
        p[key][part] *= f
    return p


@pytest.mark.parametrize("ov", [dict(pipg_omega=1e-6), dict(w_prox=1e6),
                                dict(key="P_x", part=slice(11, 14), f=1e-4)], ids=["omega", "w_prox", "rates"])
def test_other_scales(torch_cuda, oracle, inputs, ov):
    """Where the controls' or the duals' entries sink far below the largest
    iterate, one unit for all of them would cost their precision."""
    p = _scaled(inputs, **ov)
    Ns = [10, 15]
    out, r = _both(torch_cuda, oracle, p, inputs.dispersion(p, 2, 8, "bj"), Ns, [(30, 20), (30, 200), (30, 500)])
    assert r["fixed_point"] + r["fp64"] == 3 * len(Ns) and r["fp64"] >= len(Ns)
    _close(out, str(ov))


@pytest.mark.parametrize("model,nu,Ns", [("6dof", 4, [3, 10, 24]), ("6dof", 7, [8, 15]), ("3dof", 4, [4, 15, 32])])
def test_outgrown_unit(torch_cuda, oracle, inputs, model, nu, Ns):
    """A warm start that is hardly there sets a fine unit; the iterates leave
    its range and the part is run again, with and without virtual controls."""
    for w_ep in (100.0, 1.0):
        p = inputs.load_params(model=model, nu=nu, w_ep=w_ep)
        out, r = _both(torch_cuda, oracle, p, inputs.dispersion(p, len(Ns), 8, "bj"), Ns, [(30, 5), (30, 11), (30, 300)],
                       phi=1e-9)
        assert r["again"] > 0 and r["fixed_point"] > 0
        _close(out, f"w_ep {w_ep:g}")


@pytest.mark.parametrize("jcheck", [1, 2, 9, 10, 11, 21, 30])
def test_stop_tests(torch_cuda, inputs, jcheck):
    """Free runs with a stop test every jcheck iterations: the same counts as
    the FP64 loop's (looks at the magnitudes lie ten iterations apart)."""
    from paper_2404_18034_gb300.pdg_mc import Solver
    torch = torch_cuda
    p = inputs.load_params(pipg_jcheck=jcheck, pipg_eps_rel=1e-3, scp_jmax=3)
    x0 = torch.from_numpy(inputs.dispersion(p, 4, 12, "bj")).cuda()
    res = []
    for threads in (0, 512):
        S = Solver(p, 10)
        S.set_threads(threads)
        res.append(S.solve(x0, mode=0, trace=True))
        torch.cuda.synchronize()
        S.close()
    a, b = res
    n, cap = a["trace"][..., 1], p["pipg_jmax"]
    assert torch.equal(a["trace"], b["trace"])
    assert ((n % jcheck == 0) | (n == cap)).all() and (n < cap).any()
    assert (a["X"] - b["X"]).abs().max() <= 1e-9 * b["X"].abs().max()
