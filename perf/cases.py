"""The workloads that the library is timed on, and what each must return.

A case is one call sequence of a program that decodes with an evicted KV
cache: an evicting decode step, the same with the R-KV policy, the first step
on a loaded prompt, a prompt or an accepted step absorbed in one call, a step
of best-of-N candidates, the full-context helper's step, the entropy test of
the degeneration detector.  Geometries (layers, KV heads, query heads per KV
head, head dim) are those of paper_2608_15797_gb300/inputs.py.

Inputs follow that file's recipe for peaked attention: q, k, v ~ N(0, 1) with
5% of the keys scaled by 3.  Before a steady-state call a cache holds budget +
window rows whose scores come from one decode step, so that an eviction has
scores of real spread to rank.  Outputs are the attention output and, where
the call updates them, the scores and positions of the retained slots.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2608_15797_gb300 import inputs, kvr

# layers, KV heads, query heads per KV head, head dim, element type
GEOMETRY = {
    name: (w.n_layers, w.n_kv_heads, w.group, w.head_dim, w.dtype)
    for name, w in (("tiny", inputs.WORKLOADS["tiny"]),
                    ("7b", inputs.WORKLOADS["7b_b64"]),
                    ("72b", inputs.WORKLOADS["72b_bon8"]),
                    ("1p5b", inputs.WORKLOADS["1p5b_full16k"]))
}
HEAVY_FRAC, HEAVY_SCALE = 0.05, 3.0
LAM = 0.1            # the paper's R-KV mix weight
HELPER_SLACK = 256   # tokens a helper sequence decodes before it starts again


def listed():
    return [
        # The smallest call: one layer, one sequence, fp32, head dim 64 (a
        # reference run of the method); latency and launches.
        dict(name="decode_tiny_f32", kind="decode", geometry="tiny", n_seq=1,
             budget=16, window=8, by_layer=False),
        # A single user's sequence decoded as a model does it, one call a
        # layer (each layer's query needs the layer before): 28 small calls.
        dict(name="decode_7b_1seq_by_layer", kind="decode", geometry="7b",
             n_seq=1, budget=64, window=8, by_layer=True),
        # The benchmark's batch: 64 sequences at budget 64.
        dict(name="decode_7b_64seq_b64", kind="decode", geometry="7b",
             n_seq=64, budget=64, window=8, by_layer=False),
        # The same batch at the sweep's largest budget.
        dict(name="decode_7b_64seq_b512", kind="decode", geometry="7b",
             n_seq=64, budget=512, window=8, by_layer=False),
        # The paper's own policy at its own setting: R-KV, budget 512, window
        # 128 (the crossover measurement's batch of 16 sequences).
        dict(name="rkv_7b_16seq_b512_w128", kind="rkv", geometry="7b",
             n_seq=16, budget=512, window=128, by_layer=False),
        # Prompts of very different lengths enter the cache and the first
        # step cuts each to budget + window.
        dict(name="first_step_7b_4seq", kind="first", geometry="7b", n_seq=4,
             budget=64, window=8, shortest=700, longest=16384),
        # Two prompts absorbed into empty sequences, so that the retained
        # rows are those their own prefill attention ranks first.
        dict(name="prefill_7b_2seq_1000", kind="prefill", geometry="7b",
             n_seq=2, budget=128, window=8, chunk=1000),
        # An accepted 64-token helper step absorbed by the whole batch.
        dict(name="absorb_7b_64seq_c64", kind="absorb", geometry="7b",
             n_seq=64, budget=64, window=8, chunk=64),
        # The same at the paper's budget and window, a step of odd length.
        dict(name="absorb_7b_16seq_b512_c57", kind="absorb", geometry="7b",
             n_seq=16, budget=512, window=128, chunk=57),
        # One reasoning step of best-of-8 at 72B: fork, 16 tokens of every
        # candidate, commit of the chosen one.
        dict(name="candidates_72b_4seq_n8", kind="candidates", geometry="72b",
             n_seq=4, budget=64, window=8, n_cand=8, tokens=16),
        # The helper's decode over its whole context.
        dict(name="helper_1p5b_16seq_16k", kind="helper", geometry="1p5b",
             n_seq=16, context=16384),
        # The detector over the candidates of 64 problems, full vocabulary.
        dict(name="entropy_512x152064_bf16", kind="entropy", rows=512,
             vocab=inputs.VOCAB, dtype="bf16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: batch, budget, lengths, chunk and
    row counts spread over their logarithm, odd sizes included."""
    kind = rng.choice(["decode", "decode", "rkv", "first", "prefill",
                       "absorb", "absorb", "candidates", "helper", "entropy"])
    if kind in ("decode", "rkv"):
        geometry = rng.choice(["7b", "7b", "72b", "1p5b", "tiny"])
        layers, heads = GEOMETRY[geometry][:2]
        budget, window = _log_int(rng, 16, 512), rng.choice([4, 8, 32, 128])
        n_seq = _log_int(rng, 1, 64)
        most = 7168 * 520 // (layers * heads * (budget + window))
        return dict(kind=kind, geometry=geometry, n_seq=min(n_seq, most),
                    budget=budget, window=window,
                    by_layer=rng.random() < 0.3)
    if kind == "first":
        lo, hi = sorted(_log_int(rng, 512, 16384) for _ in range(2))
        return dict(kind=kind, geometry="7b", n_seq=rng.randint(1, 4),
                    budget=rng.choice([64, 128, 256, 512]), window=8,
                    shortest=lo, longest=hi)
    if kind == "prefill":
        chunk = _log_int(rng, 100, 1024)
        return dict(kind=kind, geometry=rng.choice(["7b", "7b", "1p5b"]),
                    n_seq=rng.randint(1, max(1, min(4, 2000 // chunk))),
                    budget=rng.choice([64, 128, 512]),
                    window=rng.choice([8, 128]), chunk=chunk)
    if kind == "absorb":
        budget, window = _log_int(rng, 16, 512), rng.choice([8, 128])
        n_seq = _log_int(rng, 1, 64)
        most = 16 * 640 // (budget + window)
        return dict(kind=kind, geometry="7b", n_seq=max(1, min(n_seq, most)),
                    budget=budget, window=window, chunk=_log_int(rng, 4, 64))
    if kind == "candidates":
        geometry = rng.choice(["7b", "72b"])
        return dict(kind=kind, geometry=geometry, n_seq=rng.randint(1, 4),
                    budget=rng.choice([64, 128]), window=8,
                    n_cand=rng.randint(2, 8), tokens=rng.randint(3, 16))
    if kind == "helper":
        return dict(kind=kind, geometry="1p5b", n_seq=rng.randint(1, 16),
                    context=_log_int(rng, 512, 16384))
    return dict(kind="entropy", rows=_log_int(rng, 1, 512),
                vocab=rng.choice([inputs.VOCAB, 151936, 50001, 32000]),
                dtype=rng.choice(["bf16", "bf16", "f32"]))


# ---- inputs -----------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _normal(g, shape, dtype):
    return torch.randn(shape, generator=g, device="cuda", dtype=dtype)


def _keys(g, shape, dtype):
    """N(0, 1) keys [..., d], 5% of the rows scaled by 3."""
    k = _normal(g, shape, dtype)
    heavy = torch.rand(shape[:-1], generator=g, device="cuda") < HEAVY_FRAC
    k[heavy] *= HEAVY_SCALE
    return k


def _lengths(case):
    """Prompt lengths of a "first" case: from the shortest to the longest in
    equal ratios."""
    n, lo, hi = case["n_seq"], case["shortest"], case["longest"]
    if n == 1:
        return [hi]
    return [int(round(lo * (hi / lo) ** (s / (n - 1)))) for s in range(n)]


def _token(g, lead, H, G, d, dt):
    """One token's (q, k, v): [*lead][H*G][d] and [*lead][H][d]."""
    return (_normal(g, (*lead, H * G, d), dt), _keys(g, (*lead, H, d), dt),
            _normal(g, (*lead, H, d), dt))


def _inputs(case, seed):
    """Every random tensor of a case, in the layout the calls take."""
    g = _gen(seed)
    x = {}
    if case["kind"] == "entropy":
        dt = kvr.TORCH_DTYPES[case["dtype"]]
        # a spread per row for which a coherent candidate's entropy stays
        # below the detector's threshold: no row stops
        sigma = 3.6 + 1.4 * torch.rand(case["rows"], 1, generator=g,
                                       device="cuda")
        x["logits"] = (torch.randn((case["rows"], case["vocab"]), generator=g,
                                   device="cuda") * sigma).to(dt)
        return x
    L, H, G, d, dtype = GEOMETRY[case["geometry"]]
    dt = kvr.TORCH_DTYPES[dtype]
    S, kind = case["n_seq"], case["kind"]
    if kind == "helper":
        x["k"] = [_keys(g, (L, H, case["context"], d), dt) for _ in range(S)]
        x["v"] = [_normal(g, (L, H, case["context"], d), dt) for _ in range(S)]
        x["token"] = _token(g, (S, L), H, G, d, dt)
        return x
    if kind == "first":
        x["k"] = [_keys(g, (L, H, n, d), dt) for n in _lengths(case)]
        x["v"] = [_normal(g, (L, H, n, d), dt) for n in _lengths(case)]
        x["token"] = _token(g, (S, L), H, G, d, dt)
        return x
    if kind == "prefill":
        x["token"] = _token(g, (S, L, case["chunk"]), H, G, d, dt)
        return x
    # Steady state: budget + window - 1 loaded rows and one decoded token.
    n = case["budget"] + case["window"] - 1
    x["k"] = [_keys(g, (L, H, n, d), dt) for _ in range(S)]
    x["v"] = [_normal(g, (L, H, n, d), dt) for _ in range(S)]
    x["warm"] = _token(g, (S, L), H, G, d, dt)
    if kind == "absorb":
        x["token"] = _token(g, (S, L, case["chunk"]), H, G, d, dt)
    elif kind == "candidates":
        x["token"] = _token(g, (case["tokens"], case["n_cand"], S, L), H, G, d,
                            dt)
        x["chosen"] = np.random.default_rng(seed).integers(
            0, case["n_cand"], size=S).astype(np.int32)
    else:
        x["token"] = _token(g, (S, L), H, G, d, dt)
    return x


# ---- the calls ---------------------------------------------------------------

def _cache(case, capacity):
    L, H, G, d, dtype = GEOMETRY[case["geometry"]]
    return kvr.Cache(case["n_seq"], L, H, G, d, capacity, kv_dtype=dtype,
                     out_dtype=dtype)


def _retained(cache, rows):
    """Scores and positions of slots [0, rows), viewed in place."""
    score, pos, _ = cache.scores_view()
    return {"score": score[..., :rows], "pos": pos[..., :rows]}


def prepare(case, seed):
    x = _inputs(case, seed)
    st = {"case": case, "token": x.get("token")}
    kind = case["kind"]
    if kind == "entropy":
        st["det"] = kvr.EntropyDetector(case["rows"], case["vocab"],
                                        logits_dtype=case["dtype"])
        st["logits"] = x["logits"]
        return st
    L, H, G, d, dtype = GEOMETRY[case["geometry"]]
    S = case["n_seq"]
    if kind == "helper":
        ctx = case["context"]
        st["prompt"] = _cache(case, ctx)
        for s in range(S):
            st["prompt"].load(s, x["k"][s], x["v"][s])
        st["cache"] = _cache(case, ctx + HELPER_SLACK)
        st["seqs"] = np.arange(S, dtype=np.int32)
        st["cache"].copy_from(st["prompt"], st["seqs"], st["seqs"])
        st["left"] = HELPER_SLACK
        st["out"] = st["cache"].new_out(L)
        need = kvr.kvr_decode_attend_workspace_bytes(st["cache"].handle, 0, L)
        st["workspace"] = torch.empty(2 * need, dtype=torch.uint8,
                                      device="cuda")
        return st
    keep = case["budget"] + case["window"]
    if kind == "first":
        st["k"], st["v"] = x["k"], x["v"]
        st["cache"] = _cache(case, max(_lengths(case)) + 1)
        st["out"] = st["cache"].new_out(L)
        st["kept"] = _retained(st["cache"], min(keep, min(_lengths(case)) + 1))
        return st
    if kind == "prefill":
        st["cache"] = _cache(case, case["chunk"])
        st["none"] = torch.empty(L, H, 0, d, dtype=kvr.TORCH_DTYPES[dtype],
                                 device="cuda")
        st["out"] = torch.empty_like(st["token"][0])
        st["kept"] = _retained(st["cache"], min(keep, case["chunk"]))
        return st
    cache = _cache(case, keep + (case["chunk"] if kind == "absorb" else 1))
    for s in range(S):
        cache.load(s, x["k"][s], x["v"][s])
    cache.attend_score(*x["warm"])
    st["cache"], st["kept"] = cache, _retained(cache, keep)
    if kind == "absorb":
        st["out"] = torch.empty_like(st["token"][0])
    elif kind == "candidates":
        st["chosen"] = x["chosen"]
        nbytes = kvr.kvr_fork_required_bytes(cache.handle, case["n_cand"],
                                             case["tokens"])
        st["fork_buf"] = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        st["out"] = torch.empty_like(st["token"][0])
    elif case["by_layer"]:
        st["token"] = [[t[:, l:l + 1].contiguous() for t in st["token"]]
                       for l in range(L)]
        st["out"] = torch.empty(L, *st["token"][0][0].shape,
                                dtype=cache.out_torch_dtype, device="cuda")
    else:
        st["out"] = cache.new_out(L)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "entropy":
        entropy, mean, stopped = st["det"].step(st["logits"])
        return {"entropy": entropy, "mean": mean, "stopped": stopped}
    cache, out = st["cache"], st["out"]
    if kind == "helper":
        if st["left"] == 0:  # the trajectory starts again from its prompt
            cache.copy_from(st["prompt"], st["seqs"], st["seqs"])
            st["left"] = HELPER_SLACK
        st["left"] -= 1
        kvr.attend_full(cache, *st["token"], out=out,
                        workspace=st["workspace"])
        return {"out": out}
    B, W = case["budget"], case["window"]
    if kind == "first":
        for s in range(case["n_seq"]):
            cache.load(s, st["k"][s], st["v"][s])
        cache.step(*st["token"], B, W, out=out)
    elif kind == "prefill":
        for s in range(case["n_seq"]):
            cache.load(s, st["none"], st["none"])
        cache.absorb(*st["token"], B, W, out=out)
    elif kind == "absorb":
        cache.absorb(*st["token"], B, W, out=out)
    elif kind == "candidates":
        fork = kvr.Fork(cache, case["n_cand"], case["tokens"],
                        buf=st["fork_buf"])
        q, k, v = st["token"]
        for t in range(case["tokens"]):
            fork.attend_score(q[t], k[t], v[t], out=out[t])
        fork.commit(st["chosen"], B, W)
    else:
        if case["by_layer"]:
            calls = [(out[l], (l, l + 1), t) for l, t in enumerate(st["token"])]
        else:
            calls = [(out, None, st["token"])]
        for o, layers, (q, k, v) in calls:
            if kind == "rkv":
                cache.step_rkv(q, k, v, B, W, LAM, out=o, layers=layers)
            else:
                cache.step(q, k, v, B, W, out=o, layers=layers)
    return {"out": out, **st["kept"]}


# ---- what a pass cannot do without --------------------------------------------

def work(case):
    """Each input read once and each output written once: the live K and V
    rows, q, the new rows, the outputs, scores and positions; two operations
    a multiply-add of the attention products."""
    kind = case["kind"]
    if kind == "entropy":
        n = case["rows"] * case["vocab"]
        es = 2 if case["dtype"] == "bf16" else 4
        return {"bytes": n * es + case["rows"] * 76, "flops": 4 * n}
    L, H, G, d, dtype = GEOMETRY[case["geometry"]]
    es = 2 if dtype == "bf16" else 4
    units = case["n_seq"] * L * H
    kv, qo = 2 * d * es, 2 * G * d * es   # one row's K and V; one token's q, out
    mac = 4 * G * d                       # QK and PV of one row and token
    if kind == "helper":
        n = case["context"] + 1
        return {"bytes": units * (n * kv + kv + qo), "flops": units * n * mac}
    keep = case["budget"] + case["window"]
    if kind == "first":
        # loading: rows read and written; the step: rows read again, the
        # retained rows' scores and positions written, at most the retained
        # rows moved
        rows = L * H * sum(_lengths(case))
        return {"bytes": 3 * rows * kv + 8 * rows + units * (qo + 3 * keep * kv),
                "flops": rows * mac}
    if kind == "prefill":
        c = case["chunk"]
        return {"bytes": units * (c * (kv + qo) + min(c, keep) * (kv + 8)),
                "flops": units * mac * c * (c + 1) // 2}
    if kind == "absorb":
        c = case["chunk"]
        return {"bytes": units * (keep * (kv + 16) + c * (kv + qo)
                                  + min(c, keep) * kv),
                "flops": units * mac * (c * keep + c * (c + 1) // 2)}
    if kind == "candidates":
        N, T = case["n_cand"], case["tokens"]
        per_token = keep * kv + N * (2 * kv + qo) + N * 8 * keep
        tails = N * (T - 1) * T // 2 * (kv + 8)
        return {"bytes": units * (T * per_token + tails + N * 4 * keep
                                  + (keep + T) * 8 + min(T, keep) * kv),
                "flops": units * N * mac * (T * keep + T * (T + 1) // 2)}
    flops = units * (keep + 1) * mac
    if kind == "rkv":
        flops += units * keep * 4 * d     # norms and dots with the key sum
    return {"bytes": units * (keep * (kv + 12) + 2 * kv + qo), "flops": flops}


def tolerance(case):
    """bf16 outputs: probabilities and sums in fp32, one rounding to 8 bits at
    the end, so two correct kernels differ by roundings that fall the other
    way (measured: outputs 1.7e-3 off their 64-bit values, which is that
    rounding).  Scores are fp32 sums, but rows whose scores agree to about
    1e-7 may trade places at an eviction, and then a slot holds another row
    with another score and position: hence the wide largest difference and
    the small share of positions."""
    if case["kind"] == "entropy":
        return {"rel": 1e-5}
    if case["kind"] == "helper":
        return {"rel": 4e-3, "max": 0.03}
    if GEOMETRY[case["geometry"]][4] == "f32":
        return {"rel": 1e-5, "differ": 0.001}
    return {"rel": 4e-3, "max": 0.99, "differ": 0.001}


# ---- the same in 64 bits --------------------------------------------------------

def _attend64(q, k, v):
    """q [..., G, d] over k, v [..., n, d]: outputs and probabilities."""
    p = torch.softmax(q @ k.transpose(-1, -2) / math.sqrt(q.shape[-1]), -1)
    return p @ v, p


def _heads(t, H):
    """[..., H*G, d] -> [..., H, G, d] in double."""
    return t.double().unflatten(-2, (H, t.shape[-2] // H))


def _cut64(rank, B, W):
    """The slots retained of rows in position order: the last W and the B
    best-ranked others (ties to the lower position).  A retained row below
    B + W keeps its slot; the freed slots there take the retained rows from
    above, both in ascending order.  rank [..., n] -> slots [..., B+W]."""
    n, keep = rank.shape[-1], B + W
    if n <= keep:
        return torch.arange(n, device=rank.device).expand(*rank.shape)
    order = torch.sort(rank[..., :n - W], dim=-1, descending=True, stable=True)[1]
    kept = torch.zeros(rank.shape, dtype=torch.bool, device=rank.device)
    kept.scatter_(-1, order[..., :B], True)
    kept[..., n - W:] = True
    slot = torch.arange(n, device=rank.device).expand(*rank.shape)
    movers = torch.sort(torch.where(kept[..., keep:], slot[..., keep:], n),
                        -1)[0]
    holes = ~kept[..., :keep]
    nth = (holes.cumsum(-1) - 1).clamp(0, movers.shape[-1] - 1)
    return torch.where(holes, movers.gather(-1, nth), slot[..., :keep])


def _rkv64(score, k, W, lam):
    """R-KV's z of rows in position order (the last W are never ranked)."""
    n = k.shape[-2]
    kn = torch.nn.functional.normalize(k, dim=-1)
    r = ((kn @ kn.sum(-2).unsqueeze(-1)).squeeze(-1) - 1) / (n - 1)
    cand = n - W
    z = torch.zeros_like(score)
    total = score[..., :cand].sum(-1, keepdim=True)
    z[..., :cand] = lam * score[..., :cand] / total - (1 - lam) * torch.softmax(
        r[..., :cand], -1)
    return z


def exact(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    if kind == "entropy":
        H = torch.cat([torch.special.entr(torch.softmax(r.double(), -1)).sum(-1)
                       for r in x["logits"].split(16)])
        return {"entropy": H, "mean": H, "stopped": None}
    L, H, G, d, dtype = GEOMETRY[case["geometry"]]
    S = case["n_seq"]
    if kind == "helper":
        q, kt, vt = x["token"]
        outs = []
        for s in range(S):
            o = []
            for l in range(L):
                k, v = (torch.cat([a[s][l].double(), t[s, l].double()[:, None]], 1)
                        for a, t in ((x["k"], kt), (x["v"], vt)))
                o.append(_attend64(_heads(q[s, l], H), k, v)[0].flatten(0, 1))
            outs.append(torch.stack(o))
        return {"out": torch.stack(outs)}
    B, W = case["budget"], case["window"]
    outs, scores, poss = [], [], []
    for s in range(S):
        o_l, s_l, p_l = [], [], []
        for l in range(L):
            o, sc, slots = _exact_layer(case, x, s, l, H, B, W)
            o_l.append(o)
            s_l.append(sc.gather(-1, slots))
            p_l.append(slots)
        outs.append(torch.stack(o_l, -3))
        scores.append(torch.stack(s_l))
        poss.append(torch.stack(p_l))
    if kind == "first":
        rows = min(min(a.shape[-1] for a in scores), B + W)
        scores = [a[..., :rows] for a in scores]
        poss = [a[..., :rows] for a in poss]
    if kind in ("prefill", "absorb"):        # [S][chunk][L] -> [S][L][chunk]
        out = torch.stack(outs).transpose(1, 2)
    elif kind == "candidates":               # [S][T][N][L] -> [T][N][S][L]
        out = torch.stack(outs, 2)
    elif case.get("by_layer"):               # [S][L] -> [L][S][1]
        out = torch.stack(outs).transpose(0, 1).unsqueeze(2)
    else:
        out = torch.stack(outs)
    return {"out": out, "pos": torch.stack(poss), "score": torch.stack(scores)}


def _exact_layer(case, x, s, l, H, B, W):
    """One sequence's layer: outputs [..., H*G, d], the scores of all rows in
    position order [H][n], and the slots' rows [H][B+W] after the cut."""
    kind = case["kind"]
    if kind == "prefill":
        k = v = score = None
    else:
        k, v = x["k"][s][l].double(), x["v"][s][l].double()
        score = torch.zeros(k.shape[:2], dtype=torch.float64, device=k.device)
    steps = []
    if "warm" in x:
        steps.append(tuple(t[s, l] for t in x["warm"]))
    if kind in ("decode", "rkv", "first"):
        steps.append(tuple(t[s, l] for t in x["token"]))
    out = None
    for q, kt, vt in steps:
        k, v = (torch.cat([a, t.double()[:, None]], 1)
                for a, t in ((k, kt), (v, vt)))
        out, p = _attend64(_heads(q, H), k, v)
        score = torch.cat([score, score.new_zeros(H, 1)], 1) + p.mean(-2)
        out = out.flatten(0, 1)
    if kind in ("prefill", "absorb"):
        q, kt, vt = (t[s, l] for t in x["token"])
        out, k, score = _causal64(_heads(q, H).transpose(0, 1), k, v, score,
                                  kt.double().transpose(0, 1),
                                  vt.double().transpose(0, 1))
        out = out.transpose(0, 1).flatten(1, 2)
    elif kind == "candidates":
        q, kt, vt = (t[:, :, s, l] for t in x["token"])   # [T][N][H..][d]
        o, sc = [], None
        for c in range(case["n_cand"]):
            oc, _, scc = _causal64(_heads(q[:, c], H).transpose(0, 1), k, v,
                                   score, kt[:, c].double().transpose(0, 1),
                                   vt[:, c].double().transpose(0, 1))
            o.append(oc.transpose(0, 1).flatten(1, 2))
            if c == int(x["chosen"][s]):
                sc = scc
        out, score = torch.stack(o, 1), sc
    rank = _rkv64(score, k, W, LAM) if kind == "rkv" else score
    return out, score, _cut64(rank, B, W)


def _causal64(q, k, v, score, kt, vt):
    """A chunk of c tokens, each attending the old rows and the chunk's rows
    up to its own.  q [H][c][G][d], old k, v [H][m][d] (or None), kt, vt
    [H][c][d] -> out [H][c][G][d], all keys [H][m+c][d], scores [H][m+c]."""
    H, c, G, d = q.shape
    k = kt if k is None else torch.cat([k, kt], 1)
    v = vt if v is None else torch.cat([v, vt], 1)
    m = k.shape[1] - c
    score = torch.cat([score if score is not None else k.new_zeros(H, 0),
                       k.new_zeros(H, c)], 1)
    row = torch.arange(m + c, device=k.device)
    hidden = row[None, :] > m + torch.arange(c, device=k.device)[:, None]
    logits = q @ k.transpose(1, 2).unsqueeze(1) / math.sqrt(d)
    p = torch.softmax(logits.masked_fill(hidden[None, :, None], -math.inf), -1)
    return p @ v.unsqueeze(1), k, score + p.mean(2).sum(1)
