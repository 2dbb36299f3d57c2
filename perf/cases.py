"""The work a user of this library has it do, as cases that can be timed and compared.

Every case is one call (or one short sequence of calls) of the public entry points in
``paper_2506_03762_b200.binding``, at the shapes of the repository's own configurations and of
their neighbourhood.  Operations:

``evict``    one layer's eviction step (score, select, compact) after prefill, or a later round with a
             carried score; optionally a budget per head, optionally a token-major cache layout
``ragged``   the eviction step for a batch whose sequences differ in length and budget
``step``     one generation step on an ordered cache: score update, selection, compaction in place
``slots``    one generation step on a cache kept as slots
``causal``   accumulation over all query rows (the H2O-style score of the ablation)
``entropy``  the row entropies a caller tunes the softmax scale with

Inputs: N(0, 1) queries, keys and values.  Where tokens are kept by their score, as many tokens as the
budget has room for are heavy hitters (keys aligned with a random observation query, positions uniform
outside the recent window): the tokens worth keeping stand clear of the rest, so the kept set does not
hang on the last bits of a score and two correct implementations keep the same rows.
"""
from __future__ import annotations

import torch

from paper_2506_03762_b200 import binding as ab

DEV = "cuda"
DTYPE = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
CODE = {"f32": ab.F32, "f16": ab.F16, "bf16": ab.BF16}
HITTER_COS = 0.9


def _evict(name, B, Hq, Hkv, d, n, dtype, r, Br, Bud, **kw):
    c = {"name": name, "op": "evict", "B": B, "Hq": Hq, "Hkv": Hkv, "d": d, "n": n, "dtype": dtype, "r": r, "Br": Br,
         "Bud": Bud, "prior": True, "carried": False, "head_budgets": False, "token_major": False}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest configuration: four float32 heads of 512 tokens, where launches and host work are all there is
        _evict("evict_tiny_f32", 1, 4, 4, 64, 512, "f32", 32, 32, 128),
        # float32 inputs at an ordinary size with an odd number of tokens (offline evaluation in full precision)
        _evict("evict_3k_f32", 1, 8, 8, 128, 3001, "f32", 32, 64, 500),
        # LLaMA-2-7B-shaped layer after the prefill of one request
        _evict("evict_4k_f16", 1, 32, 32, 128, 4096, "f16", 64, 64, 512),
        # LLaMA-3-8B-shaped layer with grouped queries, a small prefill batch
        _evict("evict_gqa_16k_bf16", 4, 32, 8, 128, 16384, "bf16", 64, 128, 1024),
        # long-context prefill batch, the largest configuration: 262144 tokens x 32 heads a layer
        _evict("evict_long_32k_f16", 8, 32, 32, 128, 32768, "f16", 128, 128, 2048),
        # seven query heads a KV head, one very long request of odd length in a token-major cache, budgets per head
        _evict("evict_gqa7_70k_bf16", 1, 28, 4, 128, 70001, "bf16", 32, 128, 4096, head_budgets=True, token_major=True),
        # a decode-time eviction round: budget 2048 + 32 new tokens for 16 sequences, carried score, no value prior
        _evict("evict_round_bf16", 16, 32, 8, 128, 2080, "bf16", 32, 64, 2048, prior=False, carried=True),
        # a serving batch of eight requests of 2K to 32K tokens, each keeping a quarter
        {"name": "evict_ragged_f16", "op": "ragged", "B": 8, "Hq": 32, "Hkv": 32, "d": 128, "n_min": 2048, "n": 32768,
         "dtype": "f16", "r": 128, "Br": 128, "keep": 0.25},
        # one generation step, evicting at every step, rows kept in order
        {"name": "step_bf16", "op": "step", "B": 16, "Hq": 32, "Hkv": 8, "d": 128, "Bud": 2048, "Br": 64, "dtype": "bf16"},
        # the same step on a slot cache: one call a layer and token
        {"name": "slots_bf16", "op": "slots", "B": 16, "Hq": 32, "Hkv": 8, "d": 128, "Bud": 2048, "Br": 64, "dtype": "bf16"},
        # the score accumulated over every query row of an 8K prompt (the comparison methods' score)
        {"name": "causal_8k_f16", "op": "causal", "B": 1, "Hq": 32, "Hkv": 32, "d": 128, "n": 8192, "r": 128, "dtype": "f16"},
        # row entropies of the observation rows over a long context (choosing the softmax scale)
        {"name": "entropy_32k_f16", "op": "entropy", "B": 2, "Hq": 32, "Hkv": 32, "d": 128, "n": 32768, "r": 128, "dtype": "f16"},
    ]


# ---- more cases of the same ranges ------------------------------------------------------------------

def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def _heads(rng):
    """(query heads, KV heads) of the model families the repository names: one to eight query heads a KV head."""
    g = rng.choice((1, 1, 2, 4, 4, 7, 8))
    hkv = rng.choice((1, 2, 4, 8, 8, 16, 32)) if g < 7 else rng.choice((1, 2, 4))
    return g * hkv, hkv


def draw(rng):
    op = rng.choice(("evict",) * 5 + ("evict_f32", "evict_round", "ragged", "step", "slots", "causal", "entropy"))
    d = rng.choice((64, 128, 128, 128))
    dtype = rng.choice(("f16", "bf16"))
    if op == "evict":
        Hq, Hkv = _heads(rng)
        n = _log_int(rng, 256, 70000)
        r = rng.choice((16, 32, 64, 100, 128))
        r = min(r, 256 // (Hq // Hkv), n // 4)
        Br = rng.choice((0, r, 64, 128))
        Bud = max(Br + 16, 48, int(n / rng.choice((2, 4, 8, 16))))
        Br = min(Br, Bud // 2)
        r = max(1, min(r, (Bud - Br) // (2 * (Hq // Hkv))))        # the budget has room for what every row attends to
        cap = max(1, min(8, (1 << 31) // (n * Hkv * d * 2)))       # at most the bytes of the largest listed case
        rows = -(-r * (Hq // Hkv) // 128) * 128
        cap = max(1, min(cap, 1_000_000_000 // (n * Hkv * rows)))
        return {k: v for k, v in _evict("", _log_int(rng, 1, cap), Hq, Hkv, d, n, dtype, r, Br, Bud,
                                        head_budgets=rng.random() < 0.2, token_major=rng.random() < 0.3,
                                        prior=rng.random() < 0.85).items() if k != "name"}
    if op == "evict_f32":
        Hq, Hkv = rng.choice(((4, 4), (8, 8), (8, 2), (16, 4)))
        n = _log_int(rng, 256, 6000)
        r = min(rng.choice((16, 32, 32)), 64 // (Hq // Hkv), n // 16)
        return {k: v for k, v in _evict("", 1, Hq, Hkv, d, n, "f32", r, r, max(80, n // rng.choice((3, 4, 8)))).items()
                if k != "name"}
    if op == "evict_round":
        Hq, Hkv = _heads(rng)
        r = rng.choice((16, 32, 64))
        r = min(r, 256 // (Hq // Hkv))
        Bud = _log_int(rng, 512, 4096)
        B = _log_int(rng, 1, max(1, min(16, 400 // Hkv)))
        return {k: v for k, v in _evict("", B, Hq, Hkv, d, Bud + r, dtype, r, max(64, r), Bud, prior=False,
                                        carried=True).items() if k != "name"}
    if op == "ragged":
        Hq, Hkv = _heads(rng)
        r = rng.choice((32, 64, 128))
        r = min(r, 256 // (Hq // Hkv))
        n = _log_int(rng, 4096, 32768)
        return {"op": "ragged", "B": rng.randint(2, max(2, min(8, 256 // Hkv))), "Hq": Hq, "Hkv": Hkv, "d": d,
                "n_min": n // rng.choice((4, 8, 16)), "n": n, "dtype": dtype, "r": r, "Br": r, "keep": rng.choice((0.125, 0.25, 0.5))}
    if op in ("step", "slots"):
        Hq, Hkv = _heads(rng)
        Bud = _log_int(rng, 512, min(8192, 40960 // (Hq // Hkv) - 1))
        B = _log_int(rng, 1, max(1, min(32, 300000 // (Hkv * Bud))))
        return {"op": op, "B": B, "Hq": Hq, "Hkv": Hkv, "d": d, "Bud": Bud, "Br": rng.choice((32, 64, 128)), "dtype": dtype}
    if op == "causal":
        Hq, Hkv = rng.choice(((8, 8), (16, 16), (32, 32), (32, 8), (16, 2)))
        r = min(rng.choice((64, 128)), 256 // (Hq // Hkv))
        return {"op": "causal", "B": 1, "Hq": Hq, "Hkv": Hkv, "d": d, "n": _log_int(rng, 1024, 8192), "r": r, "dtype": dtype}
    Hq, Hkv = _heads(rng)
    n = _log_int(rng, 1024, 32768)
    r = min(rng.choice((32, 64, 100, 128)), 256 // (Hq // Hkv))
    return {"op": "entropy", "B": _log_int(rng, 1, max(1, min(4, 64 // Hq))), "Hq": Hq, "Hkv": Hkv, "d": d, "n": n, "r": r, "dtype": dtype}


# ---- inputs ----------------------------------------------------------------------------------------------

def _randn(g, shape, dtype):
    return torch.randn(shape, generator=g, device=DEV, dtype=DTYPE[dtype])


def _plant_hitters(g, q, k, Br, counts):
    """Gives `counts[b, h]` tokens of each (sequence, KV head), outside the recent window and seen by every
    observation row, keys of length sqrt(d) at HITTER_COS to one of the queries of the group, taken in turn."""
    B, Hq, r, d = q.shape
    Hkv, n = k.shape[1], k.shape[2]
    G, most = Hq // Hkv, int(counts.max())
    pos = torch.rand((B, Hkv, n - max(Br, r)), generator=g, device=DEV).argsort(dim=-1)[..., :most]
    b = torch.arange(B, device=DEV).view(B, 1, 1).expand_as(pos)
    h = torch.arange(Hkv, device=DEV).view(1, Hkv, 1).expand_as(pos)
    which = torch.arange(most, device=DEV).view(1, 1, most).expand_as(pos)
    live = which < counts.to(DEV).unsqueeze(-1)
    b, h, pos, which = b[live], h[live], pos[live], which[live]
    for s in range(0, pos.numel(), 1 << 20):
        bb, hh, pp, ww = b[s:s + (1 << 20)], h[s:s + (1 << 20)], pos[s:s + (1 << 20)], which[s:s + (1 << 20)]
        u = q[bb, hh * G + ww % G, (ww // G) % r].float()
        u = u / u.norm(dim=-1, keepdim=True)
        z = k[bb, hh, pp].float()
        z = z - (z * u).sum(-1, keepdim=True) * u
        z = z / z.norm(dim=-1, keepdim=True)
        k[bb, hh, pp] = (d ** 0.5 * (HITTER_COS * u + (1 - HITTER_COS ** 2) ** 0.5 * z)).to(k.dtype)


def _carried_score(g, B, Hkv, n, Br, evicted, new_rows):
    """F of the earlier rounds: survivors carry a clear score, as many tokens as this round evicts have gone stale,
    and the new rows start at zero."""
    f = 2.0 + 2.0 * torch.rand((B, Hkv, n), generator=g, device=DEV)
    if evicted > 0:
        stale = torch.rand((B, Hkv, n - max(Br, new_rows)), generator=g, device=DEV).argsort(dim=-1)[..., :evicted]
        f.scatter_(-1, stale, 1e-3 * torch.rand(stale.shape, generator=g, device=DEV))
    if new_rows > 0:
        f[..., n - new_rows:] = 0.0
    return f


def _lengths(c):
    """Lengths of a ragged batch: spread evenly over the logarithm from n_min to n, not round numbers except the longest."""
    m = max(1, c["B"] - 1)
    return [c["n"] if b == m else int(round(c["n_min"] * (c["n"] / c["n_min"]) ** (b / m))) for b in range(c["B"])]


def _budget(c, n):
    return max(c["Br"] + 16, int(n * c["keep"]))


def _token_major(t):
    """The same values as [B, n, H, d] in memory, and the element strides (batch, head, token) that say so."""
    B, H, n, d = t.shape
    return t.transpose(1, 2).contiguous(), (n * H * d, d, H * d)


def prepare(case, seed):
    c = case
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000003 + 17)
    B, Hq, Hkv, d, dtype = c["B"], c["Hq"], c["Hkv"], c["d"], c["dtype"]
    code = CODE[dtype]
    if c["op"] == "evict":
        n, r, Br, Bud = c["n"], c["r"], c["Br"], c["Bud"]
        q, k, v = (_randn(g, s, dtype) for s in ((B, Hq, r, d), (B, Hkv, n, d), (B, Hkv, n, d)))
        p = ab.Params(B, Hq, Hkv, d, n, r, Br, Bud, dtype=code, flags=ab.FLAG_VALUE_PRIOR if c["prior"] else 0,
                      n_total=32768 + n if c["carried"] else None)
        budgets, prev = None, None
        if c["carried"]:
            prev = _carried_score(g, B, Hkv, n, Br, n - Bud, r)
        else:
            counts = torch.full((B, Hkv), Bud, dtype=torch.int32)
            if c["head_budgets"]:
                span = torch.rand((B, Hkv), generator=g, device=DEV).cpu()
                counts = (Bud - (Bud - Br) // 2 * span).to(torch.int32)
                budgets = counts.to(DEV)
            _plant_hitters(g, q, k, Br, counts - Br)
        if c["token_major"]:
            k, p.k_stride = _token_major(k)
            v, p.v_stride = _token_major(v)
        return {"op": "evict", "p": p, "in": (q, k, v, prev), "budgets": budgets, "out": tuple(t.zero_() for t in ab.alloc_outputs(p, DEV)),
                "ws": ab.alloc_workspace(p, DEV)}
    if c["op"] == "ragged":
        n, r, Br = c["n"], c["r"], c["Br"]
        q = _randn(g, (B, Hq, r, d), dtype)
        k, v = torch.zeros((B, Hkv, n, d), dtype=DTYPE[dtype], device=DEV), torch.zeros((B, Hkv, n, d), dtype=DTYPE[dtype], device=DEV)
        seqs = []
        for b, nb in enumerate(_lengths(c)):
            kb = _randn(g, (1, Hkv, nb, d), dtype)
            _plant_hitters(g, q[b:b + 1], kb, Br, torch.full((1, Hkv), _budget(c, nb) - Br, dtype=torch.int32))
            k[b, :, :nb] = kb[0]
            v[b, :, :nb] = _randn(g, (Hkv, nb, d), dtype)
            seqs.append((nb, _budget(c, nb), nb))
        p = ab.Params(B, Hq, Hkv, d, n, r, Br, _budget(c, n), dtype=code, flags=ab.FLAG_VALUE_PRIOR)
        return {"op": "ragged", "p": p, "seqs": seqs, "in": (q, k, v, None), "out": tuple(t.zero_() for t in ab.alloc_outputs(p, DEV)),
                "ws": ab.alloc_workspace(p, DEV)}
    if c["op"] in ("step", "slots"):
        Bud, Br = c["Bud"], c["Br"]
        n = Bud + 1
        p = ab.Params(B, Hq, Hkv, d, n, 1, Br, Bud, dtype=code, n_total=32768 + n, flags=0)
        k, v = _randn(g, (B, Hkv, n, d), dtype), _randn(g, (B, Hkv, n, d), dtype)
        f = _carried_score(g, B, Hkv, n, Br, 0, 1)
        q = _randn(g, (B, Hq, 1, d), dtype)
        if c["op"] == "step":
            # the attention layer has written the new token's rows behind the kept ones
            return {"op": "step", "p": p, "in": (q, f), "cache": (k, v, torch.zeros_like(f)),
                    "idx": torch.zeros((B, Hkv, Bud), dtype=torch.int32, device=DEV)}
        # slots hold distinct positions in no order; the free one is anywhere, the recent window is in the cache
        f = _carried_score(g, B, Hkv, n, Br, 0, 0)
        order = torch.rand((B, Hkv, n), generator=g, device=DEV).argsort(dim=-1)
        pos = (32768 + order).to(torch.int32)                      # positions 32768 .. 32768 + Bud
        free = (order == Bud).int().argmax(dim=-1).to(torch.int32)
        pos.scatter_(-1, free.long().unsqueeze(-1), -1)
        k_t, v_t = _randn(g, (B, Hkv, 1, d), dtype), _randn(g, (B, Hkv, 1, d), dtype)
        p.n_total = 32768 + Bud
        return {"op": "slots", "p": p, "in": (q, k_t, v_t), "cache": (k, v, f, pos, free)}
    n, r = c["n"], c["r"]
    k = _randn(g, (B, Hkv, n, d), dtype)
    Bud = max(64, n // 8)
    if c["op"] == "causal":
        p = ab.Params(B, Hq, Hkv, d, n, r, 64, Bud, dtype=code, flags=ab.FLAG_VALUE_PRIOR)
        return {"op": "causal", "p": p, "in": (_randn(g, (B, Hq, n, d), dtype), k, _randn(g, (B, Hkv, n, d), dtype)),
                "score": torch.zeros((B, Hkv, n), dtype=torch.float32, device=DEV), "ws": ab.alloc_workspace(p, DEV)}
    p = ab.Params(B, Hq, Hkv, d, n, r, 64, Bud, dtype=code, flags=0)
    return {"op": "entropy", "p": p, "in": (_randn(g, (B, Hq, r, d), dtype), k),
            "h": torch.zeros((B, Hq, r), dtype=torch.float32, device=DEV)}


# ---- one pass ----------------------------------------------------------------------------------------------

def run(state):
    s, p = state, state["p"]
    if s["op"] == "evict":
        q, k, v, prev = s["in"]
        k_out, v_out, s_out, idx = s["out"]
        if s["budgets"] is None:
            ab.ahakv_evict(p, q, k, v, prev, k_out, v_out, s_out, idx, s["ws"])
        else:
            ab.ahakv_evict_head_budgets(p, s["budgets"], q, k, v, prev, k_out, v_out, s_out, idx, s["ws"])
        return s["out"]
    if s["op"] == "ragged":
        q, k, v, prev = s["in"]
        k_out, v_out, s_out, idx = s["out"]
        ab.ahakv_evict_ragged(p, s["seqs"], q, k, v, prev, k_out, v_out, s_out, idx, s["ws"])
        return s["out"]
    if s["op"] == "step":
        (q, f_prev), (k, v, f) = s["in"], s["cache"]
        ab.ahakv_score_step(p, q, k, f_prev, f)
        ab.ahakv_select(p, f, s["idx"])
        ab.ahakv_compact_inplace(p, k, v, f, s["idx"])
        return k, v, f, s["idx"]
    if s["op"] == "slots":
        p.n_total += 1                                             # one more token has been generated
        ab.ahakv_step_slots(p, *s["in"], *s["cache"])
        return s["cache"]
    if s["op"] == "causal":
        ab.ahakv_score_full_causal(p, *s["in"], None, s["score"], s["ws"])
        return s["score"]
    return ab.ahakv_row_entropy(p, *s["in"], s["h"])


# ---- what a pass cannot do without ------------------------------------------------------------------------

def work(case):
    c = case
    B, Hq, Hkv, d = c["B"], c["Hq"], c["Hkv"], c["d"]
    es = 4 if c["dtype"] == "f32" else 2
    row = d * es
    if c["op"] in ("evict", "ragged"):
        if c["op"] == "evict":
            seqs = [(c["n"], min(c["n"], c["Bud"]))] * B
        else:
            seqs = [(n, min(n, _budget(c, n))) for n in _lengths(c)]
        r, prior, carried = c["r"], c.get("prior", True), c.get("carried", False)
        tokens, kept = sum(n for n, _ in seqs) * Hkv, sum(m for _, m in seqs) * Hkv
        values = tokens if prior else kept                          # without the value prior only the kept V rows are read
        return {"bytes": (tokens + values) * row + 2 * kept * row + B * Hq * r * row + kept * 8 + (tokens * 4 if carried else 0),
                "flops": 2.0 * Hq // Hkv * r * d * tokens}
    if c["op"] in ("step", "slots"):
        rows = B * Hkv * (c["Bud"] + 1)
        flops = 2.0 * B * Hq * (c["Bud"] + 1) * d
        if c["op"] == "slots":                                      # keys, positions, the score in and out
            return {"bytes": rows * (row + 12) + 4 * B * Hkv * row + B * Hq * row, "flops": flops}
        moved = rows // 2                                           # rows behind the evicted one, half of them on average
        return {"bytes": rows * (row + 12) + 3 * moved * row + B * Hq * row, "flops": flops}
    n = c["n"]
    if c["op"] == "causal":
        return {"bytes": B * (Hq + 2 * Hkv) * n * row + B * Hkv * n * 4, "flops": float(B * Hq) * n * (n + 1) * d}
    return {"bytes": B * Hkv * n * row + B * Hq * c["r"] * (row + 4), "flops": 2.0 * B * Hq * c["r"] * n * d}


def tolerance(case):
    """Kept indices and copied rows are the same; scores and entropies agree to the rounding of FP32 sums of
    exponentials whose arguments (tens, in log2 units) carry FP32 rounding themselves."""
    return {"rel": 1e-5 if case["dtype"] == "f32" else 1e-4}
