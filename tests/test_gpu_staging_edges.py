"""The staged object tile and measured pattern at their edges, where
test_gpu_pair_pass.py does not reach: the cluster windows 192 and 256 (bands of 32
rows, the last ending the plane; the pattern as strips of 32 columns), and the
multislice pass on every window, with slices of an odd number of pixels (every
other one starts off 16-byte alignment) and with object and intensity arrays
that are not aligned themselves."""
import numpy as np
import pytest

from oracle import ptycho_oracle as orc
from tests.parity_util import err, to_dev
from tests.test_gpu_multislice import LAM, PX, TOL_FWD, TOL_GRAD, ms_problem
from tests.test_gpu_pair_pass import _shifted, test_edges_match_oracle as edges
from tests.test_gpu_small_windows import _positions

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("noise", ["gaussian", "poisson"])
@pytest.mark.parametrize("N,W,shift", [(N, W, s) for N in (192, 256) for W, s in ((N + 6, 0), (N + 7, 0), (N + 7, 1))])
def test_cluster_windows_match_oracle(N, W, shift, noise):
    edges(N, W, shift, noise)


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("N,M,S,J", [(16, 1, 3, 4), (16, 1, 3, 640), (32, 1, 3, 4), (32, 2, 2, 170), (64, 2, 3, 4),
                                     (128, 1, 3, 4), (192, 2, 2, 4), (256, 1, 3, 4)])
def test_multislice_matches_oracle(N, M, S, J, shift):
    import torch
    from paper_2510_20929_gb300 import api
    H, W = N + 23, N + 25   # odd
    Os, P, _, Hf, I_m = ms_problem(N, M, S, H, W, J, 0.3, 5e-6)
    pos = _positions(N, H, W, J, N)
    dO, dP = _shifted(Os, torch.complex64, shift), to_dev(P, torch.complex64)
    dpos, dI = to_dev(pos, torch.float32), _shifted(I_m, torch.float32, shift)
    ms = api.make_multislice(S, 5e-6, LAM, PX)
    assert err(api.forward_ms(dO, dP, dpos, ms, batch=J).cpu().numpy(), orc.forward_ms(Os, P, pos, Hf)) < TOL_FWD
    loss, gO, gP, gr = api.adjoint_ms(dO, dP, dpos, dI, ms, "gaussian", eps=1.0, batch=J)
    ref = orc.loss_and_gradients_ms(Os, P, pos, Hf, I_m, orc.GAUSSIAN, 1.0)
    assert abs(loss.item() - ref[0]) / abs(ref[0]) < TOL_FWD
    assert err(gO.cpu().numpy(), ref[1], axis=0) < TOL_GRAD and err(gP.cpu().numpy(), ref[2], axis=0) < TOL_GRAD
    assert err(gr.cpu().numpy(), ref[3], axis=1) < TOL_GRAD
