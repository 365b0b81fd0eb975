"""The candidate step as tiles on 5th-generation tensor cores (kernel 5),
against the oracle: candidate counts (whole and half-filled pairs), group
sizes, prefixes and tails at the ends of their blocks; and the library's choice
of it, with more units than CTAs and prefixes and tails of several blocks."""
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


# (N, G, prefix rows of the two sequences, tokens): a block holds 128 prefix
# rows, or 16 * (8 // N) tail rows of each candidate.
@pytest.mark.parametrize("N,G,lens,tokens", [
    (8, 8, [72, 72], 18), (8, 7, [128, 1], 3), (8, 1, [127, 16], 34),
    (7, 5, [0, 31], 17), (5, 8, [127, 113], 2), (4, 7, [120, 15], 33),
    (3, 2, [128, 64], 4), (2, 8, [48, 0], 65), (1, 7, [100, 17], 20)])
@pytest.mark.parametrize("out_dtype", ["bf16", "f32"])
def test_fork_tile_shapes(N, G, lens, tokens, out_dtype):
    w = inputs.Workload("ft", 1, 2, G, 128, "bf16", 40, 8, 0, 0, sigma=1.0)
    c, o = harness.make_pair(w, 160 + N, 2, cap=max(max(lens), 48) + tokens + 1,
                             prompt_lens=lens, out_dtype=out_dtype)
    o2, _, st = harness.fork_lockstep(c, o, w, 160 + N, N, tokens, w.budget,
                                      w.window, kernel=5)
    assert st.kernels == [5] * tokens
    harness.lockstep(c, o2, w, 160 + N, 2, w.budget, w.window, step0=500)


def test_fork_tile_is_the_choice_for_many_units():
    """Four units for each SM, of ragged prefixes up to three blocks, N = 8,
    tails crossing a block: every CTA works through several units, reusing
    its buffers.  Three candidates, or half the layers, go elsewhere."""
    layers = -(-torch.cuda.get_device_properties(0).multi_processor_count // 4)
    w = inputs.Workload("fm", layers, 4, 1, 128, "bf16", 24, 8, 0, 0, sigma=1.0)
    c, o = harness.make_pair(w, 170, 4, cap=280, prompt_lens=[257, 7, 129, 0],
                             out_dtype="bf16")
    _, _, st = harness.fork_lockstep(c, o, w, 170, 8, 18, w.budget, w.window)
    assert st.kernels == [5] * 18
    q, k, v = (np.stack([x, x, x]) for x in inputs.step_inputs(w, 170, 900, 4))
    dq, dk, dv = (harness.dev(a, w.dtype) for a in (q, k, v))
    f = harness.guarded_fork(c, 3, 2)
    f.attend_score(dq, dk, dv)
    assert f.last_kernel() == 1


def test_fork_tile_layer_ranges():
    """Calls over parts of the layers, whose tails differ in length meanwhile,
    give what one call over all of them gives."""
    w = inputs.Workload("fm", 11, 8, 2, 128, "bf16", 24, 8, 0, 0, sigma=1.0)
    c, o = harness.make_pair(w, 170, 8, cap=80, prompt_lens=[32, 7, 40, 0, 33,
                                                             16, 31, 48])
    f = harness.guarded_fork(c, 2, 3, kernel=5)
    q, k, v = (np.stack([x, x]) for x in inputs.step_inputs(w, 170, 900, 8))
    dq, dk, dv = (harness.dev(a, w.dtype) for a in (q, k, v))
    whole = f.attend_score(dq, dk, dv)
    harness.check_guards(f)
    del f
    g = harness.guarded_fork(c, 2, 3, kernel=5)
    part = [g.attend_score(*(a[:, :, lo:hi].contiguous() for a in (dq, dk, dv)),
                           layers=(lo, hi)) for lo, hi in ((0, 4), (4, 11))]
    assert g.last_kernel() == 5
    assert torch.equal(whole, torch.cat(part, 2))
    harness.check_guards(c, g)


# (N, prefix, the first tail that goes elsewhere, the kernel it goes to): against
# one warp a candidate, against the chunked kernel, and a prefix too short.
@pytest.mark.parametrize("N,prefix,last,other", [
    (8, 72, 42, 1), (4, 136, 50, 1), (8, 20, 0, 1), (8, 300, 151, 2),
    (5, 330, 99, 1)])
def test_long_tails_go_elsewhere(N, prefix, last, other):
    layers = torch.cuda.get_device_properties(0).multi_processor_count
    c = kvr.Cache(1, layers, 4, 1, 128, prefix + 1, kv_dtype="bf16",
                  out_dtype="bf16")
    g = torch.Generator(device="cuda")
    g.manual_seed(N)

    def rnd(*shape):
        return torch.randn(shape, generator=g, device="cuda").bfloat16()
    c.load(0, rnd(layers, 4, prefix, 128), rnd(layers, 4, prefix, 128))
    f = kvr.Fork(c, N, last + 1)
    q, k, v = (rnd(N, 1, layers, 4, 128) for _ in range(3))
    for t in range(last + 1):
        f.attend_score(q, k, v)
        assert f.last_kernel() == (5 if t < last else other), f"tail {t}"
