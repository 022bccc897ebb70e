"""Multislice windows 16 and 32, whose passes take one line of a transform per lane
group or packed line pairs by the number of positions of a launch: either side
of each line against the oracle, with the first and the last tile of the object."""
import numpy as np
import pytest

from oracle import ptycho_oracle as orc
from tests.parity_util import err, to_dev
from tests.test_gpu_multislice import LAM, PX, TOL_FWD, TOL_GRAD, _dev, ms_problem
from tests.test_gpu_small_windows import _positions, _sms

pytestmark = pytest.mark.gpu


def _ms(N, M, S, J):
    Os, P, _, Hf, I_m = ms_problem(N, M, S, N + 23, N + 26, J, 0.3, 5e-6)
    pos = _positions(N, N + 23, N + 26, J, S)
    return (Os, P, pos, Hf, I_m), _dev(Os, P, pos, I_m)


@pytest.mark.parametrize("more", [0, 1])
@pytest.mark.parametrize("N,M,S,per_sm", [(16, 1, 3, 6), (32, 2, 2, 2)])
def test_multislice_forward_matches_oracle(N, M, S, per_sm, more):
    from paper_2510_20929_gb300 import api
    J = per_sm * _sms() + more
    (Os, P, pos, Hf, _), (dO, dP, dpos, _) = _ms(N, M, S, J)
    I = api.forward_ms(dO, dP, dpos, api.make_multislice(S, 5e-6, LAM, PX), batch=J).cpu().numpy()
    assert err(I, orc.forward_ms(Os, P, pos, Hf)) < TOL_FWD


@pytest.mark.parametrize("recompute", [False, True])
@pytest.mark.parametrize("more", [0, 1])
@pytest.mark.parametrize("N,M,S,per_sm", [(16, 2, 3, 4), (32, 1, 2, 1)])
def test_multislice_gradients_match_oracle(N, M, S, per_sm, more, recompute):
    from paper_2510_20929_gb300 import api
    J = per_sm * _sms() + more
    (Os, P, pos, Hf, I_m), dev = _ms(N, M, S, J)
    ms = api.make_multislice(S, 5e-6, LAM, PX, recompute=recompute)
    loss, gO, gP, gr = api.adjoint_ms(*dev, ms, "gaussian", eps=1.0, batch=J)
    ref = orc.loss_and_gradients_ms(Os, P, pos, Hf, I_m, orc.GAUSSIAN, 1.0)
    assert abs(loss.item() - ref[0]) / abs(ref[0]) < TOL_FWD
    assert err(gO.cpu().numpy(), ref[1], axis=0) < TOL_GRAD and err(gP.cpu().numpy(), ref[2], axis=0) < TOL_GRAD
    assert err(gr.cpu().numpy(), ref[3], axis=1) < TOL_GRAD


@pytest.mark.parametrize("N,M,S,per_sm,more", [(16, 2, 2, 2, 0), (16, 2, 2, 2, 1), (32, 1, 3, 1, 0), (32, 1, 3, 1, 1),
                                               (32, 2, 2, 1, 0)])
def test_multislice_epoch_matches_oracle(N, M, S, per_sm, more):
    import torch
    from paper_2510_20929_gb300 import api
    J = per_sm * _sms() + more
    (Os, P, pos, Hf, I_m), (dO, dP, dpos, dI) = _ms(N, M, S, J)
    kw = dict(batch=J, delta_o=0.1, delta_p=0.1, lam=1e-6, eps=1.0)
    order = np.arange(J, dtype=np.int32)[::-1].copy()
    O1, P1, L1, a1 = orc.lsqml_epoch_ms(Os, P, pos, I_m, order, Hf, orc.LsqmlOptions(**kw))
    loss, alpha = api.lsqml_epoch_ms(dO, dP, dpos, dI, to_dev(order, torch.int32), api.make_multislice(S, 5e-6, LAM, PX),
                                     want_alpha=True, **kw)
    e = (err(dO.cpu().numpy(), O1, axis=0), err(dP.cpu().numpy(), P1, axis=0), err(alpha.cpu().numpy(), a1, axis=1))
    print(f"ms N={N} M={M} S={S} J={J}:", e)
    assert max(e) < TOL_GRAD and abs(loss.item() - L1) / abs(L1) < TOL_FWD
