"""The step on units longer than 2,048 rows (a cluster of eight CTAs a unit)
and the eviction's selection over more than 256 rows, at the edges of their
row shares, stages and thread counts."""
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


# Ragged units in one launch: the longest sets the kernel; units of one stage,
# of fewer rows than CTAs of the cluster, one row past a share, and empty.
@pytest.mark.parametrize("G,lens", [(7, [2048, 0, 5]), (1, [4096, 511, 512]),
                                    (8, [2112, 64, 2111]), (3, [7001, 448, 449])])
@pytest.mark.parametrize("out_dtype", ["bf16", "f32"])
def test_long_step_ragged(G, lens, out_dtype):
    w = inputs.Workload("ls", 1, 2, G, 128, "bf16", 40, 8, 0, 0, sigma=1.0)
    c, o = harness.make_pair(w, 110 + G, 3, cap=max(lens) + 2, prompt_lens=lens,
                             out_dtype=out_dtype)
    harness.lockstep(c, o, w, 110 + G, 3, w.budget, w.window)
    harness.check_guards(c)


def test_long_step_matches_the_generic_kernel_in_fp32():
    """fp32 outputs keep fp32's precision: P is taken as three bf16 terms.
    Both kernels' errors against fp64 are a few 2^-24 of the probability-
    weighted |v| (about 1): 4e-6 allows an order of magnitude."""
    w = inputs.Workload("lf", 1, 2, 7, 128, "bf16", 40, 8, 0, 0, sigma=1.0)
    outs = []
    for fused in (True, False):
        c, _ = harness.make_pair(w, 121, 1, cap=3001, prompt_lens=[3000],
                                 fused=fused)
        q, k, v = (harness.dev(a, w.dtype)
                   for a in inputs.step_inputs(w, 121, 0, 1))
        outs.append((c.attend_score(q, k, v), c.export(0, kv=False)["score"]))
    assert (outs[0][0] - outs[1][0]).abs().max().item() < 4e-6
    np.testing.assert_allclose(outs[0][1][..., :3001], outs[1][1][..., :3001],
                               rtol=4e-6)


@pytest.mark.parametrize("n", [257, 700, 2047, 2048, 2049, 9000])
@pytest.mark.parametrize("B,W", [(0, 3), (1, 0), (64, 8), (200, 31)])
def test_eviction_of_equal_scores_keeps_the_lower_positions(n, B, W):
    """q = 0: every row gains exactly the same score, so the retained set is
    positions 0..B-1 and the W newest, through the radix select's tie rule.
    Slots hold random positions, so lower positions are not lower slots."""
    c = kvr.Cache(1, 1, 2, 2, 64, n + 1, kv_dtype="f32", out_dtype="f32")
    rng = np.random.default_rng(n + B)
    st = {x: rng.standard_normal((1, 2, n + 1, 64)).astype(np.float32)
          for x in ("K", "V")}
    st["score"] = np.zeros((1, 2, n + 1), np.float32)
    st["pos"] = np.stack([np.append(rng.permutation(n), 0) for _ in range(2)]
                         )[None].astype(np.int32)
    st["len"] = np.full((1, 2), n, np.int32)
    st["next_pos"] = np.full((1, 2), n, np.int32)
    c.import_state(0, st)
    z = torch.zeros(1, 1, 4, 64, device="cuda")
    c.attend_score(z, z[:, :, :2].contiguous(), z[:, :, :2].contiguous())
    c.evict(B, W)
    c.sync_status()
    e = c.export(0)
    for h in range(2):
        assert e["len"][0, h] == B + W
        got = e["pos"][0, h, :B + W]
        assert sorted(got) == list(range(B)) + list(range(n + 1 - W, n + 1))
        # the rows moved with their positions
        slot_of = {int(p): s for s, p in enumerate(st["pos"][0, h, :n])}
        for s, p in enumerate(got):
            if p < n:
                assert (e["K"][0, h, s] == st["K"][0, h, slot_of[int(p)]]).all()
