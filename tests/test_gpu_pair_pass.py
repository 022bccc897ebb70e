"""The line-pair pass (windows 32, 64, 128) at its edges: object tiles that end
the object, rows of odd pitch, object and intensity arrays that are not 16-byte
aligned (plain loads instead of bulk copies), zero counts, and an eps outside
the range of the data term's fast square roots."""
import numpy as np
import pytest

from oracle import ptycho_oracle as orc
from tests.parity_util import TOL_FWD, TOL_GRAD, c64, err, f32pos, problem, to_dev

pytestmark = pytest.mark.gpu


def _shifted(x, dtype, shift):
    """A contiguous device copy of x that starts `shift` elements into its storage."""
    import torch
    t = to_dev(x, dtype)
    buf = torch.zeros(t.numel() + shift, dtype=dtype, device="cuda")
    buf[shift:] = t.reshape(-1)
    return buf[shift:].view(t.shape)


@pytest.mark.parametrize("noise", ["gaussian", "poisson"])
@pytest.mark.parametrize("N,W,shift", [(N, W, s) for N in (32, 64, 128) for W, s in ((N + 6, 0), (N + 7, 0), (N + 7, 1))])
def test_edges_match_oracle(N, W, shift, noise):
    import torch
    from paper_2510_20929_gb300 import api
    H, M = N + 5, 2
    p = problem(N=N, M=M, H=H, W=W, J=4, seed=N + W, step=1.0, counts=300.0)
    O, P, I_m = c64(p["O"]), c64(p["P"]), np.float32(p["I_m"]).astype(np.float64)
    # the first and the last tile of the object, whole and fractional
    lo, hy, hx = N / 2.0, H - N / 2.0 - 1.0, W - N / 2.0 - 1.0
    pos = f32pos([[lo, lo], [hy, hx], [hy + 0.984375, hx + 0.984375], [hy + 0.5, lo + 0.25]])
    assert (I_m == 0).any()
    dO, dP = _shifted(O, torch.complex64, shift), to_dev(P, torch.complex64)
    dpos, dI = to_dev(pos, torch.float32), _shifted(I_m, torch.float32, shift)
    assert err(api.forward(dO, dP, dpos).cpu().numpy(), orc.forward(O, P, pos)) < TOL_FWD
    nz = orc.GAUSSIAN if noise == "gaussian" else orc.POISSON
    ref = orc.loss_and_gradients(O, P, pos, I_m, nz, 1.0)
    loss, gO, gP, gr = api.adjoint(dO, dP, dpos, dI, noise, eps=1.0, batch=3)
    assert abs(loss.item() - ref[0]) / abs(ref[0]) < TOL_FWD
    assert err(gO.cpu().numpy(), ref[1]) < TOL_GRAD and err(gP.cpu().numpy(), ref[2], axis=0) < TOL_GRAD
    assert err(gr.cpu().numpy(), ref[3], axis=1) < TOL_GRAD


@pytest.mark.parametrize("scale", [1.0, 1e-18])
def test_data_term_outside_the_fast_range(scale):
    # intensities scaled to about 1e-36 .. 1e-32, where the loss takes sqrtf
    import torch
    from paper_2510_20929_gb300 import api
    p = problem(N=32, M=1, H=48, W=50, J=3, seed=4, step=4.0)
    O, P, pos = c64(p["O"]), c64(p["P"] * scale), f32pos(p["pos"])
    I_m = np.float32(p["I_m"] * scale ** 2).astype(np.float64)
    loss, _, _, _ = api.adjoint(to_dev(O, torch.complex64), to_dev(P, torch.complex64), to_dev(pos, torch.float32),
                                to_dev(I_m, torch.float32), "gaussian", eps=0.0)
    ref = sum(orc.pattern_loss(i, m, orc.GAUSSIAN, 0.0) for i, m in zip(orc.forward(O, P, pos), I_m))
    assert abs(loss.item() - ref) / ref < TOL_FWD


@pytest.mark.parametrize("N", [32, 64, 128])
def test_non_finite_and_zero_predictions_keep_their_values(N):
    # a dark pattern with eps = 0: 0 counts give rho = 0 / 0, counts give 1 / 0;
    # an infinite or negative count is reported
    import torch
    from paper_2510_20929_gb300 import api
    O = torch.zeros(N + 4, N + 4, dtype=torch.complex64, device="cuda")
    P = torch.ones(1, N, N, dtype=torch.complex64, device="cuda")
    pos = torch.full((1, 2), N / 2 + 1.0, device="cuda")
    I = torch.full((1, N, N), 4.0, device="cuda")
    loss, gO, _, _ = api.adjoint(O, P, pos, I, "gaussian", eps=0.0)
    assert loss.item() == 4.0 * N * N and torch.isnan(torch.view_as_real(gO)).any()
    for bad in (float("inf"), -1.0):
        I[0, N - 1, N - 1] = bad
        with pytest.raises(api.PtychoError):
            api.adjoint(O + 1, P, pos, I, "gaussian", eps=1.0)
