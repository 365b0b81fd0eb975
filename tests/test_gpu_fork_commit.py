"""kvr_fork_commit where every row of prefix + tail has a thread (up to 128 and
up to 256 rows) and one row past that, against the oracle."""
import pytest
import torch

from paper_2608_15797_gb300 import inputs
from tests import harness

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    torch.cuda.set_device(0)


# (prefix rows, tail rows, B, W): 127 to 129 and 255 to 257 rows; budgets that
# cut the prefix itself, that reach into the tail and that cut nothing; no
# budget (only the window stays); no window; the second sequence of every case
# has a prefix a row shorter than the budget needs, or none.
@pytest.mark.parametrize("np_,nt,B,W", [
    (124, 3, 60, 8), (120, 8, 100, 24), (126, 3, 126, 2), (126, 3, 200, 2),
    (250, 5, 20, 0), (240, 16, 0, 9), (253, 4, 250, 4), (9, 30, 3, 5),
    (1, 1, 1, 0)])
@pytest.mark.parametrize("d,dtype", [(128, "bf16"), (64, "f32")])
def test_commit_shapes(np_, nt, B, W, d, dtype):
    w = inputs.Workload("fc", 1, 2, 2, d, dtype, B, W, 0, 0, sigma=1.0)
    c, o = harness.make_pair(w, 500 + np_, 2, cap=np_ + nt + 2,
                             prompt_lens=[np_, max(0, B + W - nt - 1)
                                          if B + W - nt - 1 < np_ else 0])
    o2, _, _ = harness.fork_lockstep(c, o, w, 500 + np_, 2, nt, B, W)
    assert (c.lengths() == o2.len.max(axis=2)).all()
    harness.check_guards(c)
    if B and np_ + nt < 200:
        harness.lockstep(c, o2, w, 500 + np_, 2, B, W, step0=100)
