"""A position whose object tile or measured pattern does not arrive is given up
as a whole: none of its CTAs adds to the gradients, the status says so, and the
next call on the same workspace is right again."""
import ctypes

import numpy as np
import pytest

from tests.parity_util import TOL_FWD, TOL_GRAD, c64, err, f32pos, problem, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("copy", [1, 2])
@pytest.mark.parametrize("N,S,M,J", [(32, 1, 2, 400), (64, 1, 1, 3), (128, 1, 2, 3), (192, 1, 1, 3), (256, 1, 2, 3),
                                     (64, 2, 2, 3), (128, 2, 1, 3), (192, 2, 2, 3), (256, 3, 1, 3)])
def test_given_up_positions_add_nothing(N, S, M, J, copy):
    import torch
    from paper_2510_20929_gb300 import api
    p = problem(N=N, M=M, H=N + 33, W=N + 36, J=J, seed=N, step=1.0)
    O, P = to_dev(c64(p["O"]), torch.complex64), to_dev(c64(p["P"]), torch.complex64)
    pos, I = to_dev(f32pos(p["pos"]), torch.float32), to_dev(np.float32(p["I_m"]), torch.float32)
    ms = None
    if S > 1:
        O, ms = O.expand(S, -1, -1).contiguous(), api.make_multislice(S, 2e-6, 0.1e-9, 10e-9)
        d = api._ms_dims(O, P, pos, ms)
        ws = api._ms_workspace(d, ms, J, O.device)
        call = lambda: api.adjoint_ms(O, P, pos, I, ms, eps=1.0, batch=J)
    else:
        d = api.dims_of(O, P, pos)
        ws = api.workspace(d, J, O.device)
        call = lambda: api.adjoint(O, P, pos, I, eps=1.0, batch=J)
    want = call()
    gO, gP = torch.zeros_like(O), torch.zeros_like(P)
    loss = torch.zeros((), dtype=torch.float64, device=O.device)
    api._check(api.lib().ptycho_selftest_copy_timeout(
        ctypes.byref(d), ctypes.byref(ms) if ms else None, copy, *map(api._ptr, (O, P, pos, I, gO, gP, loss)),
        api._P(ws.ptr), ws.nbytes, api._stream()), "selftest")
    assert ws.status() == 5   # PTYCHO_ERR_TIMEOUT
    assert not torch.view_as_real(gO).any() and not torch.view_as_real(gP).any()
    assert copy == 2 or N > 128 or loss.item() == 0.0
    got = call()
    assert abs(got[0].item() - want[0].item()) <= TOL_FWD * abs(want[0].item())
    for a, b in zip(got[1:3], want[1:3]):
        assert err(a.cpu().numpy(), b.cpu().numpy()) < TOL_GRAD


def test_other_copies_are_refused():
    from paper_2510_20929_gb300 import api
    d = api.Dims(80, 80, 64, 1, 1)
    for copy in (0, 3):
        assert api.lib().ptycho_selftest_copy_timeout(ctypes.byref(d), None, copy, *[None] * 7, None, 0, None) == 1
