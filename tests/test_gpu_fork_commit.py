"""kvr_fork_commit where every row of prefix + tail has a thread (up to 128 and
up to 256 rows) and one row past that, against the oracle."""
import numpy as np
import pytest
import torch

from paper_2608_15797_gb300 import inputs, kvr
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


@pytest.mark.parametrize("np_", [72, 300])  # by rank, and by select
def test_commit_past_the_capacity_is_refused(np_):
    """A 16-token tail on a parent with one free row: a budget that keeps all of
    it is refused on the host with the fork as it was; one that fits commits."""
    w = inputs.Workload("fc", 1, 2, 2, 128, "bf16", np_ + 56, 8, 0, 0, sigma=1.0)
    c, o = harness.make_pair(w, 510, 2, cap=np_ + 1, prompt_lens=[np_, 5])
    f = harness.guarded_fork(c, 2, 16)
    for t in range(16):
        f.attend_score(*(harness.dev(a, w.dtype)[None].expand(
            2, *a.shape).contiguous() for a in inputs.step_inputs(w, 510, t, 2)))
    before = c.export(0)
    launches = c.launch_count()
    with pytest.raises(kvr.KvrError) as e:
        f.commit(np.array([1, 0], np.int32), np_ + 56, 8)
    assert e.value.status == kvr.KVR_ECAPACITY
    assert c.launch_count() == launches
    assert c.lengths().tolist() == [[np_], [5]]
    after = c.export(0)
    for name in ("K", "V", "score", "pos", "len"):
        assert np.array_equal(before[name], after[name], equal_nan=True)
    f.commit(np.array([1, 0], np.int32), np_ - 7, 8)      # np_ + 1 rows: the capacity
    assert c.lengths().tolist() == [[np_ + 1], [21]]
    c.sync_status()
    harness.check_guards(c, f)
