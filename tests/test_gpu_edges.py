"""Kernel variants at the sizes where they can go wrong: the edges of tiles, remainders, the ends of their ranges."""
import numpy as np
import pytest
import torch

import oracle
from paper_2508_02558_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cand", [1, 31, 512, 513, 1536, 1537, 3073, 5120, 5121, 8192, 8193, 32768, 32769, 65537])
@pytest.mark.parametrize("heads,mode,r", [(2, B.SELECT_JOINT_FLOOR, 0.5), (150, B.SELECT_JOINT_FLOOR, 0.9), (3, B.SELECT_PER_REGION_CEIL, 0.3)])
def test_select_compact_at_the_ends_of_each_variant(cand, heads, mode, r):
    """One launch or two, one CTA or a cluster per head, full and partial last items: kept positions and rows against a
    stable sort, with ties, infinities and NaN among the scores."""
    if cand > 8193 and heads > 8:
        heads, r = 8, 0.03
    b, D, o = 16, 64, cand // 3
    L = cand + b
    rng = np.random.default_rng(cand + heads)
    sc = rng.standard_normal((1, heads, L)).astype(np.float32)
    sc[:, :, ::7] = np.round(sc[:, :, ::7])
    sc[:, :, 3::41] = -np.inf
    sc[:, 1::2, 5::23] = np.nan
    d = B.make_desc(batch=1, n_q_heads=heads, n_kv_heads=heads, head_dim=D, seq_len_max=L, block_len=b, dtype=B.BF16, retention=r,
                    select=mode, n_keep_max=cand)
    k = torch.arange(heads * L, dtype=torch.int32, device="cuda").reshape(1, heads, L, 1).repeat(1, 1, 1, D // 2).contiguous()
    v = -k
    idx = torch.full((1, heads, cand), -5, dtype=torch.int32, device="cuda")
    cnt = torch.zeros((1,), dtype=torch.int32, device="cuda")
    kc, vc = (torch.full((1, heads, cand, D // 2), -7, dtype=torch.int32, device="cuda") for _ in range(2))
    B.select_compact(d, torch.from_numpy(sc).cuda(), None, torch.tensor([o], dtype=torch.int32, device="cuda"), k, v, idx, cnt, kc, vc)
    torch.cuda.synchronize()
    n, n_pre, n_suf = B.keep_count(d, L, o)
    assert cnt.item() == n
    pos = oracle.candidate_positions(L, b, o)
    x = np.where(np.isnan(sc), -np.inf, sc)[0][:, pos]
    x = np.where(np.isnan(sc[0][:, pos]), np.finfo(np.float64).min * np.ones_like(x, np.float64), np.maximum(x, -1e300).astype(np.float64))
    for h in range(heads):
        segments = [(0, cand, n)] if mode == B.SELECT_JOINT_FLOOR else [(0, o, n_pre), (o, cand, n_suf)]
        want = np.concatenate([pos[lo + np.sort(np.argsort(-x[h, lo:hi], kind="stable")[:m])] for lo, hi, m in segments])
        got = idx[0, h].cpu().numpy()
        np.testing.assert_array_equal(got[:n], want)
        assert (got[n:] == -1).all()
        rows = np.where(np.arange(cand) < n, h * L + got, 0)
        assert (kc[0, h, :, 0].cpu().numpy() == rows).all() and (vc[0, h, :, -1].cpu().numpy() == -rows).all()
