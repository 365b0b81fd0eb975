"""A non-finite value in one token's V reaches the queries that see the token
and no others: the tensor-core tiles hold tokens, or candidates, that do not
see one another's rows."""
import pytest
import torch

from paper_2608_15797_gb300 import kvr

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    torch.cuda.set_device(0)


def _rnd(seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return lambda *s: torch.randn(s, generator=gen, device="cuda").bfloat16()


def _same(a, b):
    """Equal but for the bf16 rounding of fp32 sums in another order: a step
    of 2^-8 of the value, or of the sums' own 1e-5 near zero."""
    a, b = a.float(), b.float()
    return bool(((a - b).abs() <= 2.0 ** -7 * b.abs() + 1e-4).all())


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("G,m,chunk", [(7, 300, 57), (1, 140, 130), (8, 0, 200)])
def test_absorbed_tokens_see_no_later_row(G, m, chunk, bad):
    S, L, H, at = 1, 2, 2, chunk // 2
    runs = []
    for dirty in (False, True):
        r = _rnd(7 + G)
        c = kvr.Cache(S, L, H, G, 128, m + chunk + 3, kv_dtype="bf16",
                      out_dtype="bf16")
        c.load(0, r(L, H, m, 128), r(L, H, m, 128))
        q, k, v = r(S, L, chunk, H * G, 128), r(S, L, chunk, H, 128), r(S, L, chunk, H, 128)
        if dirty:
            v[0, 1, at, 0, 5] = bad       # one element, layer 1, head 0
        out = c.absorb(q, k, v, evict=False)
        assert c.last_absorb_kernel() == 3
        c.sync_status()
        runs.append((out.unflatten(-2, (H, G)), c.scores_view()[0][..., :m + chunk]))
    (a, sa), (b, sb) = runs
    assert torch.equal(sa, sb)
    hit = torch.zeros_like(a, dtype=torch.bool)
    hit[0, 1, at:, 0, :, 5] = True
    assert not b[hit].isfinite().any()
    assert _same(b[~hit], a[~hit])


@pytest.mark.parametrize("out_dtype", ["bf16", "f32"])
@pytest.mark.parametrize("N,G,m,at", [(8, 7, 72, 2), (3, 8, 130, 0), (2, 1, 0, 17)])
def test_candidates_see_no_other_tail(N, G, m, at, out_dtype):
    S, L, H, tokens = 1, 1, 4, at + 3
    runs = []
    for dirty in (False, True):
        r = _rnd(70 + N)
        c = kvr.Cache(S, L, H, G, 128, m + 1, kv_dtype="bf16", out_dtype=out_dtype)
        c.load(0, r(L, H, m, 128), r(L, H, m, 128))
        f = kvr.Fork(c, N, tokens, kernel=5 if m <= 128 else 1)
        outs = []
        for t in range(tokens):
            q, k, v = r(N, S, L, H * G, 128), r(N, S, L, H, 128), r(N, S, L, H, 128)
            if dirty and t == at:
                v[1, 0, 0, 2, 9] = float("nan")
            outs.append(f.attend_score(q, k, v).unflatten(-2, (H, G)))
            assert f.last_kernel() == (5 if m <= 128 else 1)
        c.sync_status()
        runs.append(torch.stack(outs))
    a, b = runs
    hit = torch.zeros_like(a, dtype=torch.bool)
    hit[at:, 1, 0, 0, 2, :, 9] = True
    assert b[hit].isnan().all()
    assert _same(b[~hit], a[~hit])
