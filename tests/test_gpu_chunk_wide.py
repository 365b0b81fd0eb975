"""The chunked step's groups of four warps (64-row chunks) and of two, against
the oracle: unit lengths at the edges of tiles and chunks, one and several
units an SM, with and without eviction, accumulated attention and R-KV."""
import pytest
import torch

from paper_2608_15797_gb300 import inputs
from tests import harness
from tests.test_gpu_rkv import rkv_lockstep

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    torch.cuda.set_device(0)


# Rows with the appended one: the kernel's shortest, one short of, on and past
# a 64-row chunk's end, on and past a 16-row tile's, the longest.
@pytest.mark.parametrize("rows,G,out", [
    (161, 7, "f32"), (191, 8, "bf16"), (192, 1, "f32"), (193, 7, "bf16"),
    (208, 2, "bf16"), (209, 4, "f32"), (521, 7, "bf16"), (1024, 8, "f32")])
@pytest.mark.parametrize("chunk", [(0, 0), (2, 2)])
def test_plain_step_lengths(rows, G, out, chunk):
    """(0, 0): a few units, so one group of four warps an SM; (2, 2) names
    groups of two.  Units of very different lengths, one of them empty; the
    longest evicts from its first step on, the next from its third."""
    B, W = rows - 9, 8
    w = inputs.Workload("cw", 1, 2, G, 128, "bf16", B, W, 0, 0, sigma=1.0)
    c, o = harness.make_pair(w, 200 + rows, 4, cap=rows + 1, out_dtype=out,
                             prompt_lens=[rows - 1, rows - 3, 0, 47],
                             chunk=chunk)
    n0 = c.launch_count()
    harness.lockstep(c, o, w, 200 + rows, 4, B, W)
    assert c.launch_count() - n0 == 4
    assert c.last_chunk_groups() == ((1, 4) if chunk == (0, 0) else (2, 2))
    harness.check_guards(c)


# (units an SM, rows, R-KV, warps a group): the lines of the rule that picks the
# groups.  Two; three (pairs); four and six at lengths below and above the
# line; lengths at which two groups of four do not fit.
@pytest.mark.parametrize("per,rows,rkv,warps", [
    (2, 200, False, 4), (3, 400, False, 2), (4, 400, False, 4),
    (4, 425, False, 4), (6, 400, False, 2), (6, 425, False, 4),
    (2, 800, False, 2), (2, 200, True, 4), (4, 489, True, 4),
    (6, 470, True, 2), (2, 800, True, 2)])
def test_units_an_sm(per, rows, rkv, warps):
    """Several units an SM; the oracle holds two of the sequences, one of
    them in the last round of units."""
    L = 10
    S = per * torch.cuda.get_device_properties(0).multi_processor_count // L
    B, W = rows - 9, 8
    w = inputs.Workload("cu", L, 1, 7, 128, "bf16", B, W, rows - 1, 0,
                        sigma=1.0)
    sample = [0, S - 1]
    c, o = harness.make_pair(w, 300 + rows, S, cap=rows + 1, sample=sample)
    if rkv:
        rkv_lockstep(c, o, w, 300 + rows, 2, B, W, 0.1, fused=True,
                     sample=sample)
    else:
        harness.lockstep(c, o, w, 300 + rows, 2, B, W, sample=sample)
    assert c.last_chunk_groups()[1] == warps
    harness.check_guards(c)


@pytest.mark.parametrize("rows,G", [(193, 7), (256, 8), (700, 3)])
def test_rkv_groups_of_two(rows, G):
    """R-KV in pairs of warps, which a few units no longer take by default."""
    B, W = rows - 9, 8
    w = inputs.Workload("cr", 1, 2, G, 128, "bf16", B, W, 0, 0, sigma=1.0)
    c, o = harness.make_pair(w, 400 + rows, 2, cap=rows + 1,
                             prompt_lens=[rows - 1, rows - 40], chunk=(2, 2))
    rkv_lockstep(c, o, w, 400 + rows, 4, B, W, 0.1, fused=True)
    assert c.last_chunk_groups() == (2, 2)
    harness.check_guards(c)
