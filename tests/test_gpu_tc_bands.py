"""Position gradients of the split-BF16 form, whose overlap-add splits a position
into bands of 32 rows: the bands' shares are summed in FP64 and rounded once, so
the gradient does not depend on the order in which the bands finish."""
import numpy as np
import pytest

from tests.parity_util import c64, f32pos, problem, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,J,batch", [(32, 40, 40), (64, 300, 128), (128, 300, 300)])
def test_position_gradient_repeats_bit_for_bit(N, J, batch):
    import torch
    from paper_2510_20929_gb300 import api
    p = problem(N=N, M=1, H=N + 34, W=N + 37, J=J, seed=N, step=1.0, counts=2e4)
    dev = (to_dev(c64(p["O"]), torch.complex64), to_dev(c64(p["P"]), torch.complex64),
           to_dev(f32pos(p["pos"]), torch.float32), to_dev(np.float32(p["I_m"]), torch.float32))
    first = api.adjoint(*dev, "gaussian", eps=1.0, batch=batch, precision="bf16x3")[3]
    assert first.abs().min(1).values.max() > 0
    for _ in range(12):
        again = api.adjoint(*dev, "gaussian", eps=1.0, batch=batch, precision="bf16x3")[3]
        assert torch.equal(first, again)
