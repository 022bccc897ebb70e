"""The split-BF16 far field's pipeline at its edges: one mode (no far field is
staged again), two, three; several positions per persistent CTA; predicted
intensities written to an array that is not 16-byte aligned."""
import ctypes

import numpy as np
import pytest

from oracle import ptycho_oracle as orc
from tests.parity_util import c64, err, f32pos, problem, to_dev

pytestmark = pytest.mark.gpu

TOL_BF16 = 1e-3   # the bar of the split-BF16 form


@pytest.mark.parametrize("N,M,J,noise", [(32, 1, 320, "poisson"), (32, 3, 7, "gaussian"), (64, 1, 3, "gaussian"),
                                         (64, 2, 160, "poisson"), (128, 1, 3, "poisson"), (128, 2, 3, "gaussian"),
                                         (128, 3, 156, "gaussian")])
def test_modes_and_positions_per_cta(N, M, J, noise):
    import torch
    from paper_2510_20929_gb300 import api
    p = problem(N=N, M=M, H=N + 24, W=N + 26, J=J, seed=N + M, step=1.0, counts=2e4)
    O, P, pos, I_m = c64(p["O"]), c64(p["P"]), f32pos(p["pos"]), np.float32(p["I_m"]).astype(np.float64)
    nz = orc.GAUSSIAN if noise == "gaussian" else orc.POISSON
    ref = orc.loss_and_gradients(O, P, pos, I_m, nz, 1.0)
    dev = (to_dev(O, torch.complex64), to_dev(P, torch.complex64), to_dev(pos, torch.float32))
    loss, gO, gP, gr = api.adjoint(*dev, to_dev(I_m, torch.float32), noise, eps=1.0, batch=J, precision="bf16x3")
    d = api.dims_of(*dev)
    I = torch.empty(J * N * N + 1, device="cuda")[1:].view(J, N, N)   # (not 16-byte aligned)
    ws = api.workspace(d, J, "cuda")
    api._check(api.lib().ptycho_forward_ex(ctypes.byref(d), api._precision("bf16x3"), J, *map(api._ptr, dev), api._ptr(I),
                                           api._P(ws.ptr), ws.nbytes, api._stream()), "ptycho_forward_ex")
    I = I.cpu().numpy()
    e = (abs(loss.item() - ref[0]) / abs(ref[0]), err(gO.cpu().numpy(), ref[1]), err(gP.cpu().numpy(), ref[2], axis=0),
         err(gr.cpu().numpy(), ref[3], axis=1), err(I, orc.forward(O, P, pos)))
    print(f"N={N} M={M} J={J} {noise}:", " ".join(f"{x:.2e}" for x in e))
    assert max(e) < TOL_BF16
