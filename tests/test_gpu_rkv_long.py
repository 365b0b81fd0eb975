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


def _kept_sum(c):
    """The units' kept key sums: the cache buffer's last array."""
    n = c.S * c.L * c.H * c.d * 4
    need = c.buf.numel() // 256 * 256
    return c.buf[need - n:need].view(torch.float32).view(c.S, c.L, c.H, c.d)


def _rkv_steps(caches, steps, seed, B, W, mark=None):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    for _ in range(steps):
        c = caches[0]
        q, k, v = (torch.randn(c.S, c.L, h, c.d, generator=gen, device="cuda")
                   .bfloat16() for h in (c.H * c.G, c.H, c.H))
        if mark is not None:
            q[..., 0] = mark
        for x in caches:
            x.step_rkv(q, k, v, B, W, 0.1)


def test_rkv_chunked_kept_sum_does_not_drift():
    """After 2,000 steps, in which every row has left but the last few, the kept
    sum is off the sum of the live rows' keys by what a sum of 208 keys is off by:
    rms some 2^-24 of partial sums of 1 to 2 and of each key's norm, below 2e-7.
    Roundings that added up, two a step, would make 60 times 2^-25 of the sum."""
    B, W, S, H = 200, 8, 2, 2
    c = harness.guarded_cache(S, 1, H, 7, 128, B + W + 1, kv_dtype="bf16",
                              out_dtype="bf16")
    for s in range(S):
        c.load(s, *(torch.randn(1, H, B + W, 128, device="cuda").bfloat16()
                    for _ in range(2)))

    def rms():
        k = torch.stack([torch.from_numpy(c.export(s)["K"][:, :, :B + W])
                         for s in range(S)]).double()
        want = torch.nn.functional.normalize(k, dim=-1).sum(-2)
        return (_kept_sum(c).cpu().double() - want).square().mean().sqrt().item()
    _rkv_steps([c], 2, 1, B, W)
    assert rms() < 3e-7
    _rkv_steps([c], 2000, 3, B, W)
    assert rms() < 3e-7
    harness.check_guards(c)


def test_rkv_chunked_infinite_key_leaves_with_its_row():
    """A key with an infinite element (its logits are -inf, its probability 0)
    makes its unit's sum, and every z, NaN while its row lives.  The row is the
    first to go (of equal z the highest position), and the steps after it rank
    as a cache that forms the sum anew does."""
    B, W = 200, 8
    c, d = (harness.guarded_cache(1, 1, 2, 8, 128, B + W + 1, kv_dtype="bf16",
                                  out_dtype="bf16") for _ in range(2))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(8)
    k, v = (torch.randn(1, 2, B + W, 128, generator=gen, device="cuda").bfloat16()
            for _ in range(2))
    k[0, 0, B, 0] = float("inf")  # (the newest candidate once a row is appended)
    c.load(0, k, v)
    _rkv_steps([c], 1, 9, B, W, mark=-1.0)
    e = c.export(0)
    assert np.isfinite(e["K"][..., :B + W, :]).all()
    assert B not in e["pos"][0, 0, :B + W]
    for t in range(3):
        d.import_state(0, c.export(0))
        _rkv_steps([c, d], 1, 10 + t, B, W, mark=-1.0)
        a, b = c.export(0, kv=False), d.export(0, kv=False)
        assert np.array_equal(a["pos"][..., :B + W], b["pos"][..., :B + W])
    c.sync_status()
