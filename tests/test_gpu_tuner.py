"""The autotuner times each kernel once: where several accepted numbers name one
form of the per-position pass, they report one time and the first is chosen."""
import pytest

from tests.parity_util import c64, f32pos, problem, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,forms,accepted", [(16, 2, 2), (64, 1, 2), (128, 1, 3), (256, 1, 1)])
def test_one_time_per_form(N, forms, accepted):
    import torch
    from paper_2510_20929_gb300 import api
    p = problem(N=N, M=2, H=N + 31, W=N + 33, J=6, seed=N, step=3.0)
    O, P = to_dev(c64(p["O"]), torch.complex64), to_dev(c64(p["P"]), torch.complex64)
    pos, I = to_dev(f32pos(p["pos"]), torch.float32), to_dev(p["I_m"], torch.float32)
    api.lsqml_epoch(O, P, pos, I, batch=6, eps=1.0, autotune=True)
    t = api.tuning(api.dims_of(O, P, pos), 6)
    ms = t["pass1_ms"]
    assert min(ms[:accepted]) > 0 and not any(ms[accepted:]) and t["pass1"] < forms
    assert forms > 1 or len(set(ms[:accepted])) == 1
