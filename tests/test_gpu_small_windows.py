"""Window 32, whose pass takes one line of a transform per lane group or packed
line pairs by the number of positions of a launch: either side of each line
against the oracle, with the first and the last tile of the object, and object
and intensity arrays that start off 16-byte alignment."""
import numpy as np
import pytest

from oracle import ptycho_oracle as orc
from tests.parity_util import TOL_EPOCH, TOL_FWD, TOL_GRAD, c64, err, f32pos, problem, to_dev
from tests.test_gpu_pair_pass import _shifted

pytestmark = pytest.mark.gpu


def _sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


def _positions(N, H, W, J, seed):
    """J positions all over the object, the first and the last whole and fractional tiles among them."""
    lo, hi = N / 2.0, np.array([H - N / 2.0, W - N / 2.0]) - 1.0 / 64
    pos = lo + np.random.default_rng(seed).random((J, 2)) * (hi - lo)
    pos[:3] = [[lo, lo], hi, np.floor(hi - lo) + lo]
    return f32pos(pos)


@pytest.mark.parametrize("shift", [0, 1, 2])
@pytest.mark.parametrize("M,per_sm,more", [(1, 2, 0), (1, 2, 1), (2, 1, 0), (2, 1, 1)])
def test_window_32_matches_oracle(M, per_sm, more, shift):
    import torch
    from paper_2510_20929_gb300 import api
    N, H, W, J = 32, 56, 59, per_sm * _sms() + more
    p = problem(N=N, M=M, H=H, W=W, J=J, seed=J, step=0.5, counts=300.0)
    O, P, I_m, pos = c64(p["O"]), c64(p["P"]), np.float32(p["I_m"]).astype(np.float64), _positions(N, H, W, J, M)
    dO, dP = _shifted(O, torch.complex64, shift), to_dev(P, torch.complex64)
    dpos, dI = to_dev(pos, torch.float32), _shifted(I_m, torch.float32, shift)
    assert err(api.forward(dO, dP, dpos).cpu().numpy(), orc.forward(O, P, pos)) < TOL_FWD
    for noise, nz in (("gaussian", orc.GAUSSIAN), ("poisson", orc.POISSON)):
        ref = orc.loss_and_gradients(O, P, pos, I_m, nz, 1.0)
        loss, gO, gP, gr = api.adjoint(dO, dP, dpos, dI, noise, eps=1.0, batch=J)
        assert abs(loss.item() - ref[0]) / abs(ref[0]) < TOL_FWD
        assert err(gO.cpu().numpy(), ref[1]) < TOL_GRAD and err(gP.cpu().numpy(), ref[2], axis=0) < TOL_GRAD
        assert err(gr.cpu().numpy(), ref[3], axis=1) < TOL_GRAD


@pytest.mark.parametrize("M,more", [(1, 0), (2, 0), (2, 1)])
def test_window_32_epoch_matches_oracle(M, more):
    from tests.test_gpu_step_pass import _epoch
    J = _sms() + more
    _epoch(32, M, J, J, 67, 0, 0)


@pytest.mark.parametrize("K,M,J", [(3, 1, 310), (2, 2, 160)])
def test_window_32_relaxed_probe_packed_matches_oracle(K, M, J):
    from paper_2510_20929_gb300 import api
    from tests.parity_util import opr_problem
    from tests.test_gpu_opr import _dev, _epoch_case, _host
    h = _host(opr_problem(N=32, K=K, M=M, H=58, W=63, J=J, step=1.0))
    d = _dev(h)
    assert err(api.forward_opr(*d[:5]).cpu().numpy(), orc.forward_opr(*h[:5])) < TOL_FWD
    e, _ = _epoch_case(32, K, M, 58, 63, J, 1.0, J, True)
    assert max(e.values()) < TOL_EPOCH
