"""Pooling and fusing inside the selection kernel against the stage entry points, bit for bit: the fused call's own scores go
through cc_fuse_prior_pool, which has its own code for both; the indices are those of cc_topk_select, whose load is another one but
whose search and emission are the same code, and of cc_topk_select_static, a kernel of its own.  Lengths around a thread's four items, a
part of the slice (four per thread) and a CTA's share; every width of the pooling window's two-tap steps."""
import math

import pytest
import torch

from paper_2604_10235_b200 import binding as cc

from gpu_util import ctx
from test_launch_rules import _shape

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
    for select in (cc.cc_topk_select, cc.cc_topk_select_static):
        idx2, count2 = torch.full_like(idx, -9), torch.full_like(count, -9)
        select(ctx(), d, fused, prior, idx2, count2)
        assert torch.equal(idx, idx2) and torch.equal(count, count2)


@pytest.mark.parametrize("cap", [0.0, 0.3])
@pytest.mark.parametrize("shape,chunk,heads,lens", [
    ((1, 1024), 1, 1, (3001,)), ((1, 512), 10, 2, (701, 33, 9, 2005)), ((1, 512), 33, 8, (11999, 640)), ((1, 1024), 2, 1, (4383,)),
    ((1, 1024), 10, 8, (30007,) * 15), ((2, 1024), 2, 8, (15423,) * 5), ((4, 512), 2, 1, (8817, 3)), ((4, 512), 10, 8, (20011,)),
    ((4, 1024), 2, 8, (17735, 17001)), ((8, 512), 2, 1, (10141,)), ((8, 512), 10, 8, (32768,)), ((8, 1024), 2, 1, (35673,)),
    ((8, 1024), 4, 8, (131071,))])
def test_every_shape_matches_the_single_cta(shape, chunk, heads, lens, cap):
    """Each compiled shape that the lengths above leave out, by sequences it is chosen for: raw scores (the fused call) and fused
    values (cc_topk_select) against the general kernel, bit for bit, with a last chunk that is cut."""
    items = -(-max(lens) // chunk)
    for fused_input in (0, 1):
        assert _shape(items, len(lens), heads, chunk, fused_input) == shape
    g = torch.Generator("cuda").manual_seed(chunk + lens[0])
    budgets = tuple(max(1, n // 5) for n in lens)
    d = cc.Desc(heads, heads, 16, seq_lens=lens, budgets=budgets, pool_kind=cc.CC_POOL_NONE, chunk_size=chunk, alpha=1.0, beta=0.01,
                force_threshold=0.98 if cap == 0.0 else 0.9, span_ratio=cap, span_min=1)
    n, b = sum(lens), sum(budgets)
    q = torch.randn(len(lens), 16, heads, 128, generator=g, device="cuda", dtype=torch.bfloat16)
    k = torch.randn(n, heads, 128, generator=g, device="cuda", dtype=torch.bfloat16)
    prior = torch.rand(n, generator=g, device="cuda")
    k_out, v_out = (torch.empty(b, heads, 128, device="cuda", dtype=torch.bfloat16) for _ in range(2))
    idx = torch.full((heads, b), -9, dtype=torch.int32, device="cuda")
    count = torch.full((len(lens), heads), -9, dtype=torch.int32, device="cuda")
    ws = ctx().workspace(d)
    cc.cc_compress_layer(ctx(), d, q, k, k, prior, k_out, v_out, idx, count, ws=ws)
    assert ctx().poll() == 0
    scores, fused = (t.clone() for t in cc.cc_workspace_views(ctx(), d, ws))
    staged = torch.empty_like(fused)
    cc.cc_fuse_prior_pool(ctx(), d, scores, prior, staged)
    assert torch.equal(staged, fused)
    for select in (cc.cc_topk_select, cc.cc_topk_select_static):
        idx2, count2 = torch.full_like(idx, -9), torch.full_like(count, -9)
        select(ctx(), d, fused, prior, idx2, count2)
        assert ctx().poll() == 0
        assert torch.equal(idx, idx2) and torch.equal(count, count2)
