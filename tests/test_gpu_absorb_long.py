"""kvr_absorb_chunk beyond the one-launch kernels' limits, bf16 outputs (the
blocked tensor-core path), against the oracle: units and chunks at the edges
of its 128-row key blocks, 256-row score items and query tiles of 128 // G
whole tokens."""
import numpy as np
import pytest
import torch

from oracle import parity
from paper_2608_15797_gb300 import inputs
from tests import harness
from tests.test_gpu_absorb import absorb_lockstep

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    torch.cuda.set_device(0)


# (G, rows before the chunk, chunk): one and several query tiles, an odd
# number of tiles, a last tile of one token; units ending on, one before and
# one past a block or an item; an empty unit beside a full one; a one-token
# chunk; G = 1 (128 tokens a tile) and 8 (16).
SHAPES = [(7, [192, 0], 1), (7, [250, 131], 18), (7, [0, 0], 127),
          (7, [128, 1], 128), (7, [120, 0], 136), (7, [0, 255], 257),
          (7, [640, 640], 57), (1, [3, 300], 129), (1, [0, 128], 256),
          (8, [129, 257], 65), (8, [0, 240], 16), (3, [500, 11], 43),
          (5, [0, 100], 300)]


@pytest.mark.parametrize("G,old,chunk", SHAPES)
def test_absorb_long_shapes(G, old, chunk):
    w = inputs.Workload("al", 2, 2, G, 128, "bf16", 48, 8, 0, 0, sigma=1.0)
    c, o = harness.make_pair(w, 90 + G, 2, cap=max(old) + chunk + 1,
                             prompt_lens=old, out_dtype="bf16")
    absorb_lockstep(c, o, w, 90 + G, chunk, w.budget, w.window)
    assert c.last_absorb_kernel() == 3
    harness.check_guards(c)
    harness.lockstep(c, o, w, 90 + G, 2, w.budget, w.window, step0=100)


@pytest.mark.parametrize("G,old,chunk", [(7, [640, 633], 57), (7, [0, 0], 200),
                                         (3, [500, 11], 43), (1, [3, 250], 130)])
def test_absorb_long_beside_slots_that_nothing_has_written(G, old, chunk):
    """Query tiles that end within 16 rows of the unit's end, in a cache with
    room behind it: PV's last step reads slots that hold NaN, with P = 0."""
    w = inputs.Workload("al", 1, 2, G, 128, "bf16", 48, 8, 0, 0, sigma=1.0)
    c, o = harness.make_pair(w, 95 + G, 2, cap=max(old) + chunk + 16,
                             prompt_lens=old, out_dtype="bf16")
    absorb_lockstep(c, o, w, 95 + G, chunk, w.budget, w.window)
    assert c.last_absorb_kernel() == 3
    harness.check_guards(c)


def test_absorb_long_without_eviction_and_budget_edges():
    """No eviction (every unit grows), then a chunk cut to a budget of one
    row and no window; peaked logits (scores of 3-sigma keys) move the online
    softmax's reference between blocks."""
    w = inputs.Workload("al", 1, 2, 7, 128, "bf16", 1, 0, 0, 0, sigma=2.0,
                        heavy_frac=0.05)
    c, o = harness.make_pair(w, 97, 2, cap=600, prompt_lens=[260, 30],
                             out_dtype="bf16")
    absorb_lockstep(c, o, w, 97, 70, 0, 0, evict=False)
    assert c.last_absorb_kernel() == 3
    assert c.lengths().tolist() == [[330], [100]]
    absorb_lockstep(c, o, w, 97, 200, 1, 0, step0=30_000)
    assert c.lengths().tolist() == [[1], [1]]


def test_absorb_long_layer_range():
    """Layers [1, 3) of four: the other layers' units stay as they were."""
    w = inputs.Workload("al", 4, 2, 7, 128, "bf16", 100, 8, 0, 0, sigma=1.0)
    c, o = harness.make_pair(w, 98, 2, cap=400, prompt_lens=[200, 180],
                             out_dtype="bf16")
    toks = [inputs.step_inputs(w, 98, 40_000 + j, 2) for j in range(90)]
    q, kn, vn = (np.stack([t[i] for t in toks], axis=2) for i in range(3))
    out = c.absorb(*(harness.dev(a[:, 1:3], "bf16") for a in (q, kn, vn)),
                   100, 8, layers=(1, 3))
    assert c.last_absorb_kernel() == 3
    ref = o.absorb(q, kn, vn, B=100, W=8, evict=True)
    torch.cuda.synchronize()
    parity.check_out(out.float().cpu().numpy(), ref[:, 1:3])
    assert c.lengths().tolist() == [[200, 108, 108, 200], [180, 108, 108, 180]]
    e = c.export(0, kv=False)
    assert (e["score"][0, :, :200] == 0).all()
    c.sync_status()


def test_absorb_long_prompt_beyond_one_append_grid():
    """33,000 tokens in one call: more rows than the append's CTAs take in one
    round.  Sampled tokens' outputs against fp64; every row in its slot."""
    n = 33_000
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    q, k, v = (torch.randn(1, 1, n, 1, 128, generator=g, device="cuda").bfloat16()
               for _ in range(3))
    c = harness.guarded_cache(1, 1, 1, 1, 128, n, kv_dtype="bf16",
                              out_dtype="bf16")
    out = c.absorb(q, k, v, evict=False)[0, 0, :, 0]
    assert c.last_absorb_kernel() == 3
    c.sync_status()
    score, pos, _ = c.scores_view()
    assert (pos[0, 0, 0, :n].cpu() == torch.arange(n)).all()
    # every token's probabilities sum to one
    assert abs(score[0, 0, 0, :n].double().sum().item() - n) < 1e-5 * n
    e = c.export(0)
    assert (torch.from_numpy(e["K"][0, 0]) == k[0, 0, :, 0].float().cpu()).all()
    kk, vv = k[0, 0, :, 0].double(), v[0, 0, :, 0].double()
    for t in (0, 1, 127, 128, 20_000, 32_767, 32_768, n - 1):
        p = torch.softmax(kk[:t + 1] @ q[0, 0, t, 0].double() / 128 ** 0.5, 0)
        ref = p @ vv[:t + 1]
        # one rounding to bf16 of outputs, fp32 sums before it
        assert ((out[t].double() - ref).abs() <= 2.0 ** -8 * ref.abs() + 2e-5).all()
    harness.check_guards(c)


def test_absorb_long_scores_are_not_biased():
    """Scores against fp64, 5% of the keys three times as long.  Roundings go
    either way; what they leave in the mean is 1 / G's (7: 4.5e-8 high) and half
    a step of the scale (3e-8).  Logits that the contraction cuts towards zero
    and nothing makes up for give 1.9e-7: the normalisers lack more of the
    longest keys' terms than the other rows' scores do of theirs."""
    S, L, H, G, m, c = 2, 2, 4, 7, 640, 57
    g = torch.Generator(device="cuda")
    g.manual_seed(12)

    def rnd(*shape, heavy=False):
        x = torch.randn(shape, generator=g, device="cuda")
        if heavy:
            x[torch.rand(shape[:-1], generator=g, device="cuda") < 0.05] *= 3
        return x.bfloat16()
    cache = harness.guarded_cache(S, L, H, G, 128, m + c, kv_dtype="bf16",
                                  out_dtype="bf16")
    old = [rnd(L, H, m, 128, heavy=True) for _ in range(S)]
    for s in range(S):
        cache.load(s, old[s], rnd(L, H, m, 128))
    q, k, v = (rnd(S, L, c, H * G, 128), rnd(S, L, c, H, 128, heavy=True),
               rnd(S, L, c, H, 128))
    cache.absorb(q, k, v, evict=False)
    assert cache.last_absorb_kernel() == 3
    got = cache.scores_view()[0][..., :m].double()
    errs = []
    hidden = (torch.arange(m + c, device="cuda")[None] >
              m + torch.arange(c, device="cuda")[:, None])
    for s in range(S):
        kk = torch.cat([old[s], k[s].transpose(1, 2)], 2).double()   # [L][H][m+c]
        qq = q[s].double().unflatten(2, (H, G)).permute(0, 2, 1, 3, 4)
        x = torch.einsum("lhcgd,lhnd->lhcgn", qq, kk) / 128 ** 0.5
        p = torch.softmax(x.masked_fill(hidden[:, None], -float("inf")), -1)
        want = p.mean(3).sum(2)[..., :m]
        errs.append((got[s] - want) / want)
    err = torch.stack(errs)
    assert abs(err.mean().item()) < 1.1e-7
    assert err.square().mean().sqrt().item() < 2e-7
