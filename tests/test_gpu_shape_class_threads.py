"""Shape classes (mode 2) with a thread setting that takes n_max out of the
fixed-point loop: the smaller classes, which choose their own CTA size, then
ask for more shared memory than n_max."""
import numpy as np
import pytest

from gpu_helpers import assert_scaled_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_max,threads", [(15, 288), (15, 96), (20, 128), (30, 512)])
def test_classes_fit_whatever_the_setting(inputs, n_max, threads):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_18034_gb300.pdg_mc import Solver
    # two SCP iterations of 60 PIPG iterations: the two loops differ by rounding
    p = inputs.load_params(scp_jmax=2, pipg_jmax=60)
    Ns = np.array([n_max, n_max - 1, n_max - 1, 10, 2, n_max], np.int32)
    x0 = torch.from_numpy(inputs.dispersion(p, len(Ns), 6, "bj")).cuda()
    N = torch.from_numpy(Ns).cuda()
    S = Solver(p, n_max)
    ref = S.solve(x0, N, mode=1)
    S.set_threads(threads)
    out = S.solve(x0, N, mode=2)
    torch.cuda.synchronize()
    assert torch.equal(out["status"], ref["status"]) and torch.equal(out["pipg_iters"], ref["pipg_iters"])
    assert_scaled_close(out["X"].cpu().numpy(), ref["X"].cpu().numpy(), p["P_x"], what="X")
    assert_scaled_close(out["U"].cpu().numpy(), ref["U"].cpu().numpy(), p["P_u"][:4], what="U")
    S.close()
