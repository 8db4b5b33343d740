"""Chunk scoring on masked logits: -inf, or the lowest value of the type, wherever a thread's first
vectors, a whole warp, the odd ends of a row or all but a few places of it are masked.  Tolerance as in
test_gpu_ppl.py, plus the 8e-5 that one exponential may be off where a few of them make up the sum."""
import numpy as np
import pytest
import torch

from oracle import codecomp_oracle as orc
from paper_2604_10235_b200 import binding as cc

from gpu_util import ctx

pytestmark = pytest.mark.gpu
TOL = 5e-5 + 8e-5


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("lowest", [False, True])
@pytest.mark.parametrize("chunks,t,v", [(1, 3, 7), (2, 3, 4099), (3, 2, 50257), (2, 4, 128256)])
def test_masked_logits(dtype, lowest, chunks, t, v):
    rng = np.random.Generator(np.random.PCG64(v + 7 * lowest))
    x = torch.from_numpy((rng.standard_normal((6, chunks, t, v)) * 3.0).astype(np.float32)).to(dtype)
    mask = torch.finfo(dtype).min if lowest else -float("inf")
    tgt = rng.integers(v // 2, v, size=t).astype(np.int32)
    places = torch.zeros(v, dtype=torch.bool)
    places[torch.from_numpy(rng.integers(0, v, size=3))] = True
    places[torch.from_numpy(tgt).long()] = True
    x[0, ..., :v // 2] = mask                     # the first vectors of every thread
    x[1, ..., -(v // 3 + 1):] = mask              # the last ones, the targets among them at times
    x[2, ..., ~places] = mask                     # all but a few places: most threads meet nothing else
    x[3, ..., torch.from_numpy(rng.random(v) < 0.7)] = mask
    x[4, ..., 1:] = mask                          # one value left, in front of the first whole vector
    x[5] = mask                                   # nothing left: NaN, which ranks last
    x = x.reshape(6 * chunks, t, v)
    nll = torch.full((6 * chunks, t), -1.0, device="cuda")
    score = torch.full((6 * chunks,), -1.0, device="cuda")
    cc.cc_ppl_chunk_scores(ctx(), x.cuda(), torch.from_numpy(tgt).cuda(), nll, score)
    assert ctx().poll() == 0, ctx().lib.cc_last_error(ctx().handle)
    with np.errstate(invalid="ignore"):
        _, ref = orc.ppl_chunk_scores(x.double().numpy(), tgt)
    ref[5 * chunks:] = np.nan
    np.testing.assert_allclose(nll.cpu().numpy(), ref, atol=TOL, rtol=2e-7)      # (lowest: 3e38 to f32's place)


@pytest.mark.parametrize("dtype,v", [(torch.float32, 50257), (torch.float32, 32000), (torch.bfloat16, 50257)])
def test_one_value_carries_the_sum(dtype, v):
    """Every exponential of f32 logits, and of rows off the 16-byte grid, is evaluated by ex2 (relative
    error 2^-22): where one value of magnitude 4 carries the sum, three more roundings to f32 of values
    below 8 are left, 2^-22 + 3 * 2^-22 in all, wherever in a vector the value lies."""
    t = 256                                       # enough rows that a row is one CTA, whose threads take vectors in pairs
    x = torch.full((2, t, v), -40.0, dtype=dtype)
    x[:, torch.arange(t), torch.arange(t) * 37 % 1000] = 4.0
    tgt = np.full(t, v - 1, np.int32)
    nll = torch.full((2, t), -1.0, device="cuda")
    score = torch.full((2,), -1.0, device="cuda")
    cc.cc_ppl_chunk_scores(ctx(), x.cuda(), torch.from_numpy(tgt).cuda(), nll, score)
    assert ctx().poll() == 0
    _, ref = orc.ppl_chunk_scores(x.double().numpy(), tgt)
    np.testing.assert_allclose(nll.cpu().numpy(), ref, atol=2.0 ** -20, rtol=2.0 ** -24)   # (the subtraction of -40)
