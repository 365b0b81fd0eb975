"""Near ties of the blocked absorb: rows whose scores lie within a few roundings
of each other at the cut.  The rows that stay, and their slots, must be those
that the same call keeps token by token from the same state: its sums run in
another order, so scores alone settle nothing there."""
import pytest
import torch

from paper_2608_15797_gb300 import kvr

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    torch.cuda.set_device(0)


def _absorbed(G, m, chunk, cap, budget, window, fused, spread):
    """One absorb into 2 x 2 x 4 units of m rows with the same key each (every
    token adds the same to all of them) and scores spread over a few roundings
    just below 2, where a sum's rounding step doubles on the way."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1000 * G + m + chunk)

    def rnd(*shape):
        return torch.randn(shape, generator=gen, device="cuda").bfloat16()
    S, L, H = 2, 2, 4
    c = kvr.Cache(S, L, H, G, 128, cap, kv_dtype="bf16", out_dtype="bf16")
    c.set_fused(fused)
    for s in range(S):
        c.load(s, rnd(L, H, 1, 128).expand(L, H, m, 128).contiguous(),
               rnd(L, H, m, 128))
    score = c.scores_view()[0]
    score[..., :m] = 1.98 + spread * torch.rand(
        (S, L, H, m), generator=gen, device="cuda")
    c.absorb(rnd(S, L, chunk, H * G, 128), 0.2 * rnd(S, L, chunk, H, 128),
             rnd(S, L, chunk, H, 128), budget, window)
    c.sync_status()
    assert c.last_absorb_kernel() == (3 if fused else 2)
    assert (c.lengths() == budget + window).all()
    got, pos, _ = c.scores_view()
    keep = budget + window
    return got[..., :keep].clone(), pos[..., :keep].clone()


# (G, rows, chunk, capacity, budget, window): eviction by rank (up to 256 rows)
# and by histogram, 256 and 1,024 threads; room for the sums and none (G = 1
# and 2 in a cache that the chunk fills).
SHAPES = [(7, 300, 20, 330, 150, 8), (7, 200, 30, 230, 100, 0),
          (8, 640, 57, 697, 300, 128), (1, 300, 20, 320, 150, 8),
          (2, 210, 40, 250, 120, 8), (4, 2100, 18, 2200, 1000, 8)]


@pytest.mark.parametrize("G,m,chunk,cap,budget,window", SHAPES)
def test_near_ties_keep_the_rows_of_token_by_token(G, m, chunk, cap, budget,
                                                   window):
    # some 25 tied rows around the cut: the band is 1.2e-6 either way
    spread = m * 2e-7 * 1.98
    a = _absorbed(G, m, chunk, cap, budget, window, True, spread)
    b = _absorbed(G, m, chunk, cap, budget, window, False, spread)
    moved = (a[1] != b[1]).any(-1).sum().item()
    assert moved == 0, f"{moved} of 16 units keep other rows"
    # one rounding a token on one side: 64 steps of 2^-24 are the most
    assert ((a[0] - b[0]).abs() <= 64 * 2.0 ** -24 * b[0] + 1e-7).all()
