"""The relaxed probe's batch sums and weight step over every number of
eigenmodes, with minibatches that are no multiple of the slots a CTA, a warp or
a load group takes."""
import pytest

from tests.parity_util import TOL_EPOCH
from tests.test_gpu_opr import _epoch_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,J,batch", [(16, 1, 3, 3), (16, 2, 13, 13), (32, 3, 9, 5), (32, 4, 8, 8), (32, 5, 37, 37),
                                         (64, 6, 7, 6), (64, 7, 6, 1), (32, 8, 75, 70)])
def test_weight_step_matches_oracle(N, K, J, batch):
    e, moved = _epoch_case(N, K, 1, N + 26, N + 31, J, 2.0, batch, True)
    print(f"N={N} K={K} {J}/{batch}:", " ".join(f"{k} {v:.2e}" for k, v in e.items()), f"moved {moved:.1e}")
    assert max(e.values()) < TOL_EPOCH and moved > 1e-4
