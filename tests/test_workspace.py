"""One workspace serves every attention call of a layer: the counters that a call expects at zero lie where no call keeps data."""
import subprocess

import numpy as np
import pytest
import torch

import oracle
from paper_2508_02558_b200 import binding as B
from paper_2508_02558_b200 import workloads as W


def test_no_plan_keeps_data_among_the_counters(host_program):
    """Every planner of the library, the overrides of the key splits included, over batches, heads, blocks and lengths."""
    exe = host_program("workspace_ranges.cpp")
    res = subprocess.run([exe], capture_output=True, text=True)
    assert res.returncode == 0, res.stdout + res.stderr
    assert all(int(x) > 0 for x in res.stdout.split()), res.stdout        # the walk met every kind of user


@pytest.mark.gpu
@pytest.mark.parametrize("batch,heads,block,L,r,score", [
    (1, 32, 16, 1280, 0.5, B.SCORE_PROB_MEAN),          # cut dense units, then four key splits that meet through counters
    (1, 96, 32, 2048, 0.5, B.SCORE_LOGIT_MEAN),         # ... then the resident walk, which hands out its units with a counter
    (10, 32, 32, 768, 0.9, B.SCORE_LOGIT_MEAN),         # refresh without counters, then a reuse step by the resident walk
])
def test_dense_refresh_and_reuse_on_one_layer_cache(batch, heads, block, L, r, score):
    import parity_util as U
    from paper_2508_02558_b200.session import LayerCache
    D, o = 128, L - 256
    rng = np.random.default_rng(heads + L)

    def draw(*shape):
        return W.round_to_dtype((rng.standard_normal(shape) / np.sqrt(D)).astype(np.float32), "bf16")

    check = [(0, 0), (batch - 1, heads - 1), (batch // 2, 7)]           # (sequence, head) pairs that the oracle recomputes
    k, v, rows = draw(batch, heads, L, D), draw(batch, heads, L, D), draw(batch, heads, L, D)
    q, q2, kn, vn = (draw(batch, heads, block, D) for _ in range(4))
    kd, vd, rd, qd, q2d, knd, vnd = (U.to_dev(x, "bf16") for x in (k, v, rows, q, q2, kn, vn))
    bo = torch.full((batch,), o, dtype=torch.int32, device="cuda")
    cache = LayerCache(batch=batch, n_q_heads=heads, n_kv_heads=heads, head_dim=D, seq_len_max=L, block_len=block, retention=r, score=score)

    def nan_like(x):
        return torch.full_like(x, float("nan"))

    def dense():
        out = nan_like(rd)
        cache.dense_step(rd, kd, vd, None, out)
        for i, h in check:
            at = [0, 255, 256, L - 1]
            ref, _ = oracle.dense_attention(rows[i, h:h + 1], k[i, h:h + 1], v[i, h:h + 1], rows=at)
            U.assert_close(U.to_host_f32(out[i, h:h + 1, at]), ref, "bf16", f"dense seq {i} head {h}")

    def refresh():
        out, lse = nan_like(qd), torch.full((batch, heads, block), float("nan"), device="cuda")
        cache.refresh(qd, kd, vd, None, bo, out, lse)
        torch.cuda.synchronize()
        g = U.GpuRefresh(cache, U.to_host_f32(out), lse.cpu().numpy(), cache.pooled.cpu().numpy(), cache.kept_idx.cpu().numpy(),
                         cache.kept_cnt.cpu().numpy(), kd, vd)
        for i, h in check:
            U.check_refresh_against_oracle(g, q, k, v, [L] * batch, [o] * batch, "bf16", r, 3, seqs=[i], heads=[h], score=score)
        return g

    def reuse(g):
        out = nan_like(qd)
        cache.sparse_step(q2d, knd, vnd, out)
        for i, h in check:
            U.check_sparse_against_oracle(g, U.to_host_f32(out), q2, kn, vn, "bf16", seqs=[i], heads=[h])

    dense()
    reuse(refresh())
    dense()
    reuse(refresh())
    assert B.read_status(cache.workspace) == 0
