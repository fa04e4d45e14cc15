"""The thrust projection of the plain form's PIPG kernel reads the reference
controls of its own instance: with several waves of CTAs an instance's step
equals the step of that instance alone."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_soc_step_does_not_depend_on_the_batch(inputs, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_18034_gb300.pdg_mc import Solver
    p = inputs.load_params(soc_thrust=1)
    n, B, at = 17, 1500, [0, 700, 1499]
    x0 = inputs.dispersion(p, B, 9, "bj")
    t = np.linspace(0.0, 1.0, n)[None, :, None]
    X = np.concatenate([(1 - t) * x0[:, None, :] + t * p["z_f"][None, None, :-1], np.zeros((B, n, 1))], 2)
    # reference thrusts that differ from instance to instance, many outside the sector
    U = np.random.default_rng(3).normal(size=(B, n, 4)) * 0.5 + np.array([2.0, 0.0, 0.0, 5.0])

    def step(idx):
        d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
        z = lambda *s: torch.zeros(len(idx), *s, dtype=torch.float64, device="cuda")  # noqa: E731
        S = Solver(p, n, precision)
        ws = dict(xh=z(n, 15), uh=z(n, 4), mup=z(n - 1, 15), mum=z(n - 1, 15), phi=z(n - 1, 15), th=z(n - 1))
        Xg, Ug = d(X[idx]), d(U[idx])
        S.scp_step(d(x0[idx]), Xg, Ug, ws, force=torch.tensor([[9, 40]] * len(idx), dtype=torch.int32, device="cuda"))
        torch.cuda.synchronize()
        return Xg.cpu().numpy(), Ug.cpu().numpy()

    Xa, Ua = step(np.arange(B))
    for b in at:
        Xb, Ub = step(np.array([b]))
        assert np.array_equal(Xa[b], Xb[0]) and np.array_equal(Ua[b], Ub[0])
