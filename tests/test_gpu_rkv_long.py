"""kvr_decode_step_rkv on units of 161 to 1,024 rows (the chunked kernel with
the kept key sum), against the oracle's reading of R-KV."""
import numpy as np
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


# 161 and 1,024 rows with the appended one are the kernel's limits; 192 and
# 193 end on and one past a 32-row chunk; G = 8 leaves no spare query column;
# W = 0 lets the new row itself be the one that goes.
@pytest.mark.parametrize("B,W,G", [(152, 8, 7), (183, 8, 8), (184, 8, 1),
                                   (512, 128, 7), (1015, 8, 3), (200, 0, 7)])
@pytest.mark.parametrize("lam", [0.0, 0.1, 1.0])
def test_rkv_chunked_step_shapes(B, W, G, lam):
    w = inputs.Workload("rc", 2, 3, G, 128, "bf16", B, W, B + W, 0, sigma=1.0)
    c, o = harness.make_pair(w, 130 + B, 2, cap=B + W + 1,
                             prompt_lens=[B + W, B + W - 1])
    n0 = c.launch_count()
    rkv_lockstep(c, o, w, 130 + B, 5, B, W, lam, fused=True)
    assert c.launch_count() - n0 == 10   # the (mostly empty) sums, the step
    harness.check_guards(c)


def test_rkv_chunked_kept_sum_across_other_calls():
    """The kept sum over many steps, dropped by a plain step, an import and a
    copy, and carried over from the one-launch kernel's smaller units."""
    B, W = 180, 8
    w = inputs.Workload("rk", 1, 2, 7, 128, "bf16", B, W, 0, 0, sigma=1.0)
    c, o = harness.make_pair(w, 140, 2, cap=B + W + 1, prompt_lens=[150, B + W])
    rkv_lockstep(c, o, w, 140, 60, B, W, 0.1, fused=True)
    harness.lockstep(c, o, w, 140, 2, B, W, step0=60)
    rkv_lockstep(c, o, w, 140, 4, B, W, 0.1, step0=62, fused=True)
    for s in range(2):
        c.import_state(s, c.export(s))
    rkv_lockstep(c, o, w, 140, 4, B, W, 0.1, step0=66, fused=True)
    d = harness.guarded_cache(2, 1, 2, 7, 128, B + W + 1, kv_dtype="bf16",
                              out_dtype="f32")
    d.copy_from(c, np.arange(2, dtype=np.int32), np.arange(2, dtype=np.int32))
    rkv_lockstep(d, o, w, 140, 4, B, W, 0.1, step0=70, fused=True)
    harness.check_guards(d)


def test_rkv_chunked_duplicate_and_zero_keys():
    """lambda = 0: 21 identical keys are the most redundant rows (their mean
    cosine is at least 20/200 more than chance, and chance is a sum of 200
    cosines of deviation 128^-1/2 over 200: 0.0063, 16 deviations less), and
    the one at the highest position goes; a zero key (cosine 0) stays."""
    n = 200
    w = inputs.Workload("rd", 1, 1, 2, 128, "bf16", n - 2, 2, n, 0, sigma=1.0)
    c, o = harness.make_pair(w, 141, 1, cap=n + 1, prompt_lens=[n])
    e = c.export(0)
    for a in (e["K"][0, 0], o.K[0, 0, 0]):
        a[50:150:5] = a[20]
        a[152] = 0.0
    c.import_state(0, e)
    rkv_lockstep(c, o, w, 141, 1, n - 2, 2, 0.0, fused=True)
    kept = c.export(0, kv=False)["pos"][0, 0, :n].tolist()
    assert 145 not in kept and {20, 50, 140, 152} <= set(kept)
