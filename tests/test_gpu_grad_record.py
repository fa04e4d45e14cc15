"""Gradients behind a solve whose PIPG loop runs in FP64 (a thread count
outside the fixed-point loop's range): that solve records the last loop's
checkpoints for the adjoint, which otherwise reruns the loop.  Both against
central differences of the oracle's last SCP iteration."""
import numpy as np
import pytest

from test_gpu_grad import _fd, _grads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads", [0, 288], ids=["reruns", "records"])
@pytest.mark.parametrize("model,nu,N", [("6dof", 4, 10), ("6dof", 7, 12), ("3dof", 4, 15)])
def test_gradient(oracle, inputs, model, nu, N, threads):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_18034_gb300.pdg_mc import Solver
    p = inputs.load_params(model=model, nu=nu)
    S = Solver(p, N)
    S.set_threads(threads)
    x0 = inputs.dispersion(p, 2, inputs.config_seed(3), "bj")
    o = _grads(torch, S, x0)
    assert (S.pipg_loops()["fixed_point"] == 0) == (threads == 288)
    assert np.isin(o["status"], (0, 1)).any()
    for b in np.flatnonzero(np.isin(o["status"], (0, 1))):
        X, U, ws, sig, n = oracle.final_iteration_state(p, N, x0[b], o["trace"][b], int(o["scp_iters"][b]))
        fd = _fd(oracle, p, x0[b], X, U, ws, sig, n)
        assert np.all(np.abs(o["g_fuel"][b] - fd[:, 0]) <= 1e-6 + 1e-5 * np.abs(fd[:, 0]))
        assert np.all(np.abs(o["g_touch"][b] - fd[:, 1]) <= 1e-9 + 1e-4 * np.abs(fd[:, 1]))
    S.close()
