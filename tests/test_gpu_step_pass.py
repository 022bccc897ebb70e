"""The two launches of the step-size pass (sums that walk over the positions,
then the update in bands) against the oracle: minibatches that are no multiple
of the four positions of a reduction tree, a single position, several trees per
CTA, odd and shifted objects, and each update switched off; and the rule that
chooses them by the minibatch's size."""
import numpy as np
import pytest

from oracle import ptycho_oracle as orc
from tests.parity_util import TOL_EPOCH, TOL_FWD, c64, err, f32pos, problem, to_dev

pytestmark = pytest.mark.gpu


def _epoch(N, M, J, batch, W, shift, variant, update_object=True, update_probe=True):
    import torch
    from paper_2510_20929_gb300 import api
    p = problem(N=N, M=M, H=N + 21, W=W, J=J, seed=N + J, step=2.0 if J <= 70 else 1.0)
    O, P, pos, I_m = c64(p["O"]), c64(p["P"]), f32pos(p["pos"]), np.float32(p["I_m"]).astype(np.float64)
    buf = torch.zeros(O.size + shift, dtype=torch.complex64, device="cuda")
    dO = buf[shift:].view(O.shape)
    dO.copy_(to_dev(O, torch.complex64))
    dP, dpos, dI = to_dev(P, torch.complex64), to_dev(pos, torch.float32), to_dev(I_m, torch.float32)
    order = np.random.default_rng(J).permutation(J).astype(np.int32)
    kw = dict(batch=batch, delta_o=0.1, delta_p=0.1, lam=1e-6, eps=1e-6, update_object=update_object,
              update_probe=update_probe)
    if variant:
        api.set_tuning(api.dims_of(dO, dP, dpos), batch, 0, variant, 0)
    O1, P1, L1, a1 = orc.lsqml_epoch(O, P, pos, I_m, order, orc.LsqmlOptions(**kw))
    loss, alpha = api.lsqml_epoch(dO, dP, dpos, dI, to_dev(order, torch.int32), want_alpha=True,
                                  autotune=bool(variant), **kw)
    e = (err(dO.cpu().numpy(), O1), err(dP.cpu().numpy(), P1, axis=0), err(alpha.cpu().numpy(), a1, axis=1))
    print(f"N={N} M={M} {J}/{batch} W={W}+{shift}:", e)
    assert max(e) < TOL_EPOCH and abs(loss.item() - L1) / abs(L1) < TOL_FWD


@pytest.mark.parametrize("N,M,J,batch,W,shift", [
    (16, 1, 9, 9, 40, 0), (16, 3, 1, 1, 41, 0), (32, 2, 11, 6, 56, 1), (64, 1, 7, 5, 87, 0), (64, 5, 4, 4, 88, 0),
    (128, 1, 70, 70, 150, 0), (192, 2, 5, 5, 214, 0), (256, 1, 6, 3, 279, 0), (256, 4, 3, 3, 280, 1)])
def test_two_launches_match_oracle(N, M, J, batch, W, shift):
    _epoch(N, M, J, batch, W, shift, 1)


@pytest.mark.parametrize("N", [32, 128, 192])
@pytest.mark.parametrize("update_object,update_probe", [(False, True), (True, False)])
def test_two_launches_with_one_update_off(N, update_object, update_probe):
    _epoch(N, 2, 5, 5, N + 24, 0, 1, update_object, update_probe)


@pytest.mark.parametrize("N,J", [(64, 153), (64, 214), (128, 213)])
def test_rule_by_minibatch_matches_oracle(N, J):
    # past one position per SM at 64, and either side of a last wave 0.7 full
    _epoch(N, 1, J, J, N + 30, 0, 0)


@pytest.mark.parametrize("N,M,S,W,update_object,update_probe", [
    (16, 5, 2, 37, True, True), (32, 1, 3, 58, True, True), (64, 4, 3, 87, True, True), (128, 2, 1, 151, True, True),
    (192, 1, 2, 215, True, True), (256, 2, 2, 280, True, True), (64, 2, 2, 88, False, True)])
def test_multislice_directions_and_updates_in_bands(N, M, S, W, update_object, update_probe):
    # more modes than slices and fewer, odd and even object widths
    import torch
    from paper_2510_20929_gb300 import api
    from tests.test_gpu_multislice import LAM, PX, TOL_GRAD, _dev, ms_problem
    dz, J = 5e-6, 5
    Os, P, pos, Hf, I_m = ms_problem(N, M, S, N + 23, W, J, 2.0, dz)
    dO, dP, dpos, dI = _dev(Os, P, pos, I_m)
    kw = dict(batch=3, delta_o=0.1, delta_p=0.1, lam=1e-6, eps=1e-6, update_object=update_object,
              update_probe=update_probe)
    order = np.arange(J, dtype=np.int32)[::-1].copy()
    O1, P1, L1, a1 = orc.lsqml_epoch_ms(Os, P, pos, I_m, order, Hf, orc.LsqmlOptions(**kw))
    loss, alpha = api.lsqml_epoch_ms(dO, dP, dpos, dI, to_dev(order, torch.int32), api.make_multislice(S, dz, LAM, PX),
                                     want_alpha=True, **kw)
    e = (err(dO.cpu().numpy(), O1, axis=0), err(dP.cpu().numpy(), P1, axis=0), err(alpha.cpu().numpy(), a1, axis=1))
    print(f"ms N={N} M={M} S={S} W={W}:", e)
    assert max(e) < TOL_GRAD and abs(loss.item() - L1) / abs(L1) < TOL_FWD
