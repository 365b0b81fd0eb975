"""The generic step's one launch (shapes outside the bf16, head_dim 128
kernels; at most 256 rows with the appended one), against the oracle: at its
row limit and one past it, cuts of one and of many rows, ragged units."""
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


@pytest.mark.parametrize("d,dtype", [(64, "f32"), (128, "f32"), (64, "bf16")])
@pytest.mark.parametrize("B,W,lens,launches", [
    (16, 8, [24, 9, 0], 4),        # steady state beside growing units
    (5, 0, [255, 40, 6], 4),       # 256 rows cut to 5; no window
    (0, 3, [30, 3, 2], 4),         # no budget
    (247, 8, [255, 255, 255], 4),  # the limit, one row a step
    (248, 8, [256, 200, 256], 8),  # 257 rows: attend, then the eviction
])
def test_generic_step(d, dtype, B, W, lens, launches):
    w = inputs.Workload("gs", 1, 2, 3, d, dtype, B, W, 0, 0, sigma=1.0)
    c, o = harness.make_pair(w, 150 + B, 3, cap=max(lens) + 5, prompt_lens=lens)
    n0 = c.launch_count()
    harness.lockstep(c, o, w, 150 + B, 4, B, W)
    assert c.launch_count() - n0 == launches
    harness.check_guards(c)
