"""Calls that a decoding program makes to this library, at the sizes it makes them.

A diffusion language model decodes a sequence block by block. Per block and layer it runs one dense step (every row of
the sequence over all keys), one refresh (block attention over all keys, saliency, pooling, top-k and gather of the kept
entries into the compacted cache) and some thirty reuse steps (block attention over the compacted cache and the block's
own fresh rows). A case is one of these calls, or one step through a stack of layers, through `LayerCache`:

  op           "refresh", "reuse" or "dense"
  layers       layers called one after the other in a pass, each with tensors and a cache of its own
  batch        sequences; seq_len is the longest one's length, and `ragged` spreads the others' below it
  after        positions from the start of the decoding block to the end of the sequence
  score, pool, select, window, retention   the policy of the refresh

Inputs follow the recipe of `paper_2508_02558_b200/workloads.py`, drawn on the GPU: Gaussian rows of variance 1/D, a few
keys per head planted along the mean block query (alone or in spans), and optional sink tokens at the front.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2508_02558_b200 import binding as B
from paper_2508_02558_b200.session import LayerCache

DEV = "cuda:0"
DTYPE = {"bf16": (torch.bfloat16, B.BF16), "f32": (torch.float32, B.F32)}
SCORE = {"logit": B.SCORE_LOGIT_MEAN, "prob": B.SCORE_PROB_MEAN}
POOL = {"max": B.POOL_MAX, "avg": B.POOL_AVG}
SELECT = {"joint": B.SELECT_JOINT_FLOOR, "region": B.SELECT_PER_REGION_CEIL, "prefix": B.SELECT_PREFIX_ONLY}

# Attention geometries of the configurations: query heads, KV heads, head dimension, share of planted keys, sink tokens,
# whether the planted keys come in spans.
TINY = dict(dtype="f32", q_heads=2, kv_heads=2, dim=64, planted=0.02, sink=1, spans=False)
LLADA = dict(dtype="bf16", q_heads=32, kv_heads=32, dim=128, planted=0.02, sink=0, spans=False)
DREAM = dict(dtype="bf16", q_heads=28, kv_heads=4, dim=128, planted=0.01, sink=4, spans=False)
LONG = dict(dtype="bf16", q_heads=32, kv_heads=8, dim=128, planted=0.005, sink=0, spans=True)
NARROW = dict(dtype="bf16", q_heads=16, kv_heads=8, dim=64, planted=0.02, sink=0, spans=False)

# Most key rows (batch x KV heads x length) and most dense multiply-adds of a case: those of the largest listed ones.
MAX_ROWS = 16 * 32 * 4352
MAX_DENSE = 32768 * 32768 * 32 * 128


def _case(op, geometry, seq_len, **kw):
    c = dict(op=op, layers=1, batch=1, seq_len=seq_len, ragged=False, block=32, after=256, retention=0.5, window=3, score="logit",
             pool="max", select="joint")
    c.update(geometry)
    c.update(kw)
    return c


def listed():
    cases = [
        # the smallest call: the fp32 configuration, latency and launches only
        _case("refresh", TINY, 256, after=128, name="tiny_f32_refresh"),
        # what a decoding program does most: one denoising step that reuses the caches of a whole stack of 32 layers
        _case("reuse", LLADA, 1280, layers=32, name="llada_reuse_32_layers"),
        # once per block and layer of the same stack
        _case("refresh", LLADA, 1280, name="llada_refresh"),
        # the same with the probability saliency, average pooling and per-region quotas
        _case("refresh", LLADA, 1280, score="prob", pool="avg", select="region", window=7, name="llada_refresh_prob"),
        # grouped heads, a 4k sequence: one layer's step in a single-user session
        _case("reuse", DREAM, 4096, retention=0.25, name="dream_reuse"),
        _case("refresh", DREAM, 4096, retention=0.25, name="dream_refresh"),
        # long context
        _case("reuse", LONG, 32768, name="long_reuse"),
        _case("refresh", LONG, 32768, name="long_refresh"),
        # ragged serving batches
        _case("reuse", LLADA, 3909, batch=4, ragged=True, name="serving4_reuse"),
        _case("refresh", LLADA, 4352, batch=16, ragged=True, name="serving16_refresh"),
        # the dense step that opens a block, ordinary and long
        _case("dense", LLADA, 1280, name="llada_dense"),
        _case("dense", LONG, 32768, name="long_dense"),
    ]
    return cases


def _log_between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any operation, geometry, block length and policy, lengths and batch sizes over their whole range."""
    geometry = rng.choice([TINY, LLADA, LLADA, LLADA, DREAM, LONG, NARROW])
    if geometry is TINY:
        op = rng.choice(["refresh", "reuse"])             # the dense step is bf16 only
        batch, seq_len = rng.choice([1, 1, 2]), _log_between(rng, 128, 2048)
    else:
        op = rng.choice(["refresh", "reuse", "dense"])
        batch = _log_between(rng, 1, 16)
        most = MAX_ROWS // (batch * geometry["kv_heads"])
        if op == "dense":
            most = min(most, int(math.sqrt(MAX_DENSE / (batch * geometry["q_heads"] * geometry["dim"]))))
        seq_len = _log_between(rng, 256, max(256, min(32768, most)))
    group = geometry["q_heads"] // geometry["kv_heads"]
    block = rng.choice([b for b in (8, 16, 32, 32, 32, 64) if b * group <= 256])
    score = "prob" if op == "refresh" and geometry is not TINY and block % 16 == 0 and rng.random() < 0.15 else "logit"
    return _case(op, geometry, seq_len, batch=batch, ragged=batch > 1 and rng.random() < 0.7, block=block,
                 layers=rng.choice([1, 1, 4]) if op == "reuse" and batch == 1 else 1,
                 after=min(seq_len, block * rng.randint(1, max(1, 256 // block))), retention=rng.choice([0.1, 0.25, 0.5, 0.5, 0.5, 0.7, 0.9]),
                 window=rng.choice([1, 3, 3, 3, 5, 7, 9]), score=score, pool=rng.choice(["max", "max", "max", "avg"]),
                 select=rng.choice(["joint", "joint", "joint", "region", "prefix"]))


def _lengths(case):
    """Lengths of the batch's sequences: all alike, or spread uniformly between an eighth of the longest one's and it."""
    n, longest = case["batch"], case["seq_len"]
    if not case["ragged"]:
        return [longest] * n
    rng = random.Random(longest * 131 + n)
    low = min(longest, max(longest // 8, case["after"]))
    lengths = [rng.randint(low, longest) for _ in range(n)]
    lengths[rng.randrange(n)] = longest
    return lengths


def _desc(case):
    """What the number of kept entries depends on."""
    return B.make_desc(batch=case["batch"], n_q_heads=case["q_heads"], n_kv_heads=case["kv_heads"], head_dim=case["dim"],
                       seq_len_max=case["seq_len"], block_len=case["block"], dtype=DTYPE[case["dtype"]][1], retention=case["retention"],
                       select=SELECT[case["select"]])


def _normal(gen, dtype, *shape):
    return torch.randn(shape, generator=gen, dtype=dtype, device=DEV).mul_(shape[-1] ** -0.5)


def _sequence_inputs(case, gen, lengths):
    """(q_blk, k, v): the block's queries and the keys and values of all positions, planted keys and sink tokens included."""
    n, hq, hkv, dim, L, b = (case[x] for x in ("batch", "q_heads", "kv_heads", "dim", "seq_len", "block"))
    dtype = DTYPE[case["dtype"]][0]
    q, k, v = _normal(gen, dtype, n, hq, b, dim), _normal(gen, dtype, n, hkv, L, dim), _normal(gen, dtype, n, hkv, L, dim)
    u = torch.nn.functional.normalize(q.float().reshape(n, hkv, -1, dim).mean(2), dim=-1)
    mask = torch.rand((n, hkv, L), generator=gen, device=DEV)
    if case["spans"]:
        span = torch.rand((n, hkv, (L + 63) // 64), generator=gen, device=DEV) < 2 * case["planted"]
        mask = (mask < 0.5) & span.repeat_interleave(64, dim=-1)[..., :L]
    else:
        mask = mask < case["planted"]
    mask[..., :case["sink"]] = False
    for i, length in enumerate(lengths):
        o = length - case["after"]
        mask[i, :, o:o + b] = False
    i, h, p = mask.nonzero(as_tuple=True)
    k[i, h, p] = (k[i, h, p].float() + 3.0 * u[i, h]).to(dtype)
    if case["sink"]:
        k[:, :, :case["sink"]] = (k[:, :, :case["sink"]].float() + 6.0 * u[:, :, None]).to(dtype)
    return q, k, v


def _layer(case, gen, lengths, seq_len, block_off, scratch):
    n, hq, hkv, dim, L, b = (case[x] for x in ("batch", "q_heads", "kv_heads", "dim", "seq_len", "block"))
    dtype, code = DTYPE[case["dtype"]]
    cache = LayerCache(batch=n, n_q_heads=hq, n_kv_heads=hkv, head_dim=dim, seq_len_max=L, block_len=b, dtype=code,
                       retention=case["retention"], pool_window=case["window"], pool=POOL[case["pool"]], score=SCORE[case["score"]],
                       select=SELECT[case["select"]], device=DEV, share_scratch_with=scratch)
    q, k, v = _sequence_inputs(case, gen, lengths)
    out = torch.zeros_like(q)
    if case["op"] == "refresh":
        return cache, (q, k, v), out
    if case["op"] == "dense":
        rows = _normal(gen, dtype, n, hq, L, dim)
        return cache, (rows, k, v), torch.zeros_like(rows)
    cache.refresh(q, k, v, seq_len, block_off, out)         # a reuse step finds the cache of its block filled
    drift = 0.05

    def step(x):
        return (x.float() + drift * _normal(gen, torch.float32, *x.shape)).to(dtype)

    rows = [x.new_empty((n, hkv, b, dim)) for x in (k, v)]
    for i, length in enumerate(lengths):
        o = length - case["after"]
        for r, x in zip(rows, (k, v)):
            r[i] = step(x[i, :, o:o + b])
    return cache, (step(q), rows[0], rows[1]), out


def prepare(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    lengths = _lengths(case)
    seq_len = torch.tensor(lengths, dtype=torch.int32, device=DEV)
    block_off = torch.tensor([n - case["after"] for n in lengths], dtype=torch.int32, device=DEV)
    layers = []
    for _ in range(case["layers"]):
        layers.append(_layer(case, gen, lengths, seq_len, block_off, layers[0][0] if layers else None))
    return case["op"], layers, seq_len, block_off


def run(state):
    op, layers, seq_len, block_off = state
    if op == "reuse":
        return [cache.sparse_step(q, k, v, out) for cache, (q, k, v), out in layers]
    cache, (q, k, v), out = layers[0]
    if op == "dense":
        return cache.dense_step(q, k, v, seq_len, out)
    cache.refresh(q, k, v, seq_len, block_off, out)
    return {"out": out, "pooled": cache.pooled, "kept_idx": cache.kept_idx, "kept_cnt": cache.kept_cnt, "k_c": cache.k_c, "v_c": cache.v_c}


def work(case):
    """Every input read once and every output written once; rows past a sequence's end and unused cache rows are not counted."""
    hq, hkv, dim, b = (case[x] for x in ("q_heads", "kv_heads", "dim", "block"))
    size = 2 if case["dtype"] == "bf16" else 4
    desc, nbytes, flops = _desc(case), 0, 0
    for n in _lengths(case):
        kept = B.keep_count(desc, n, n - case["after"])[0]
        if case["op"] == "dense":
            nbytes += 2 * n * (hq + hkv) * dim * size
            flops += 4 * n * n * hq * dim
        elif case["op"] == "reuse":
            nbytes += (2 * (kept + b) * hkv + 2 * b * hq) * dim * size
            flops += 4 * b * (kept + b) * hq * dim
        else:       # K, V, Q in; O, pooled scores, indices and the compacted rows out
            nbytes += (2 * n * hkv + 2 * b * hq + 2 * kept * hkv) * dim * size + 4 * hkv * (n - b) + 4 * hkv * kept
            flops += 4 * b * n * hq * dim + 2 * n * hkv * dim
    return {"bytes": nbytes * case["layers"], "flops": flops * case["layers"]}


def tolerance(case):
    """bf16: probabilities and outputs are rounded to 8 bits. fp32: sums of up to a few thousand products. Whole numbers (kept
    positions) may differ where two keys' scores are equal but for the rounding of an fp32 sum."""
    return {"rel": 1e-5, "max": 1e-4, "differ": 0.01} if case["dtype"] == "f32" else {"rel": 1e-2, "max": 0.1, "differ": 0.01}
