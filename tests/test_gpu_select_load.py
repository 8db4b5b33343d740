"""Pooling and fusing inside the selection kernel against the stage entry points, bit for bit: the fused call's own scores go
through cc_fuse_prior_pool and cc_topk_select, which have their own code for both.  Lengths around a thread's four items, a
part of the slice (four per thread) and a CTA's share; every width of the pooling window's two-tap steps."""
import math

import pytest
import torch

from paper_2604_10235_b200 import binding as cc

from gpu_util import ctx

pytestmark = pytest.mark.gpu
POOLS = [(cc.CC_POOL_NONE, 1), (cc.CC_POOL_MAX, 1), (cc.CC_POOL_MAX, 3), (cc.CC_POOL_AVG, 5), (cc.CC_POOL_MAX, 7),
         (cc.CC_POOL_AVG, 63), (cc.CC_POOL_MAX, 63)]


@pytest.mark.parametrize("pool", POOLS)
@pytest.mark.parametrize("cap", [0.0, 0.3])
@pytest.mark.parametrize("lens", [(1,), (3,), (509, 512, 515), (2047,), (2049,), (4097, 8193, 5), (40001,), (16385,) * 20])
def test_fused_load_matches_the_stages(pool, cap, lens):
    g = torch.Generator("cuda").manual_seed(len(lens) + lens[0])
    kind, size = pool
    budgets = tuple(max(1, n // 5) for n in lens)
    d = cc.Desc(4, 2, 16, seq_lens=lens, budgets=budgets, pool_kind=kind, pool_size=size, alpha=1.0, beta=0.01,
                force_threshold=0.9 if cap == 0.0 else 0.6, span_ratio=cap, span_min=1)
    n, b = sum(lens), sum(budgets)
    q = torch.randn(len(lens), 16, 4, 128, generator=g, device="cuda", dtype=torch.bfloat16)
    k, v = (torch.randn(n, 2, 128, generator=g, device="cuda", dtype=torch.bfloat16) for _ in range(2))
    prior = torch.rand(n, generator=g, device="cuda")
    k_out, v_out = (torch.empty(b, 2, 128, device="cuda", dtype=torch.bfloat16) for _ in range(2))
    idx = torch.full((2, b), -9, dtype=torch.int32, device="cuda")
    count = torch.full((len(lens), 2), -9, dtype=torch.int32, device="cuda")
    ws = ctx().workspace(d)
    cc.cc_compress_layer(ctx(), d, q, k, v, prior, k_out, v_out, idx, count, ws=ws)
    assert ctx().poll() == 0
    scores, fused = (t.clone() for t in cc.cc_workspace_views(ctx(), d, ws))
    assert math.isfinite(float(scores.sum()))
    staged = torch.empty_like(fused)
    cc.cc_fuse_prior_pool(ctx(), d, scores, prior, staged)
    assert torch.equal(staged, fused)
    idx2, count2 = torch.full_like(idx, -9), torch.full_like(count, -9)
    cc.cc_topk_select(ctx(), d, fused, prior, idx2, count2)
    assert torch.equal(idx, idx2) and torch.equal(count, count2)
