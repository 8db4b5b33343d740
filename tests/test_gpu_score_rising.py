"""Score parity where a row's logits rise far above its first keys': the running reference of pass 1 is looked
at before the first and the last 32 keys of a tile only, and a tile whose other keys overflow it is gone through again."""
import numpy as np
import pytest
import torch

from oracle import codecomp_oracle as orc
from paper_2604_10235_b200 import binding as cc
from paper_2604_10235_b200 import inputs as gen

from gpu_util import ctx
from test_gpu_score import check_against_oracle

pytestmark = pytest.mark.gpu

# The polynomial's 7.8e-5 enters a score twice (its value, its row's sum), and f32 products of logits up to 700
# are good to 700 * 2^-23 / ln 2 = 1.2e-4.
TOL = 4e-4


@pytest.mark.parametrize("w,hq,hkv", [(16, 8, 2), (64, 8, 2), (100, 8, 2), (128, 8, 2)])
@pytest.mark.parametrize("at", [0, 31, 32, 63, 64, 95, 96, 127, 128 + 40, 5 * 128 + 70])
@pytest.mark.parametrize("jump", [40.0, 60.0, 100.0, 700.0])
def test_scores_of_rows_that_rise(w, hq, hkv, at, jump):
    """One key, every query's best by `jump` nats (58, 87, 144, 1010 powers of two), at each place of a tile."""
    wl = gen.Workload("rise", 29, 1, hq, hkv, 128, w, gen.POOL_MAX, 7, 1, n=1500)
    x = gen.make_layer(wl, layer=at, with_v=False)
    q = orc.bf16_bits_to_f64(x.q_win).astype(np.float32)
    q[..., 0] = 4.0
    x.q_win = gen.f32_to_bf16_bits(q)
    k = orc.bf16_bits_to_f64(x.k).astype(np.float32)
    k[:, :, 0] = 0.0
    k[at, :, 0] = jump * np.sqrt(128.0) / 4.0
    x.k = gen.f32_to_bf16_bits(k)
    check_against_oracle(wl, x, cc.CC_MODE_BF16, TOL)


@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("w", [16, 64, 96, 128])
def test_rises_in_later_tiles_of_a_span(w, causal):
    """Seventeen tiles per CTA, one to four row blocks.  Every 23 tiles, so mostly well inside a span: heads 0 to 3 have four
    tiles of keys 57 powers of two up, which the reference stays below, and in the next one, which the set that had the first of
    them goes through again, a key 72 up, in the chunk of the head's number; 3 % of a row is left to the keys of before, whose
    sum has to come through that.  Heads 4 to 7 rise by 72 and, in the set's next tile of that row block, by 80 more."""
    n, hkv, every = 40000, 8, 23
    tiles = -(-n // 128)
    assert tiles * hkv > 4 * torch.cuda.get_device_properties(0).multi_processor_count
    wl = gen.Workload("later", 37, 1, 32, hkv, 128, w, gen.POOL_MAX, 7, 1, n=n, causal=causal)
    x = gen.make_layer(wl, layer=w, with_v=False)
    q = orc.bf16_bits_to_f64(x.q_win).astype(np.float32)
    q[..., 0] = 4.0
    x.q_win = gen.f32_to_bf16_bits(q)
    k = orc.bf16_bits_to_f64(x.k).astype(np.float32) * 0.25
    k[:, :, 0] = 0.0
    up = np.log(2.0) * np.sqrt(128.0) / 4.0      # one power of two, in channel 0 of a key
    for tile in range(2, tiles - 8, every):
        for h in range(4):
            k[tile * 128:(tile + 4) * 128, h, 0] = 57.0 * up
            k[(tile + 4) * 128 + 32 * h + 11, h, 0] = 72.0 * up
        for h in range(4, 8):
            k[tile * 128 + 32 * (h - 4) + 11, h, 0] = 72.0 * up
            k[(tile + 4) * 128 + 32 * ((h - 3) % 4) + 11, h, 0] = 152.0 * up
    x.k = gen.f32_to_bf16_bits(k)
    check_against_oracle(wl, x, cc.CC_MODE_BF16, TOL)


def test_lanes_without_rows_do_not_slow_the_others():
    """48 rows: half a warp, and two whole ones, multiply what lies behind the rows of Q, among it keys by keys.  Where all keys are
    large in a channel that the queries are small in, those products are out of every reference's range; going through such
    items again had cost 16 to 20 % here, and 0 to 2 % is left."""
    w, hq, hkv, causal = 12, 32, 8, True
    n = 65536
    d = cc.Desc(hq, hkv, w, n=n, budget=1, causal=causal)
    g = torch.Generator("cuda").manual_seed(w)
    q = torch.randn(1, w, hq, 128, generator=g, device="cuda", dtype=torch.bfloat16)
    q[..., 0] = 0.0
    q[..., 70] *= 0.1
    plain = torch.randn(n, hkv, 128, generator=g, device="cuda", dtype=torch.bfloat16)
    large = plain.clone()
    large[..., 0] = large[..., 70] = 300.0
    u = torch.empty(hkv, n, device="cuda")
    times = {}
    for turn in range(12):
        for name, k in (("plain", plain), ("large", large)):
            begin, end = torch.cuda.Event(True), torch.cuda.Event(True)
            begin.record()
            for _ in range(20):
                cc.cc_score_window(ctx(), d, q, k, u, None)
            end.record()
            torch.cuda.synchronize()
            times.setdefault(name, []).append(begin.elapsed_time(end))
    assert ctx().poll() == 0
    assert np.median(times["large"][2:]) < 1.08 * np.median(times["plain"][2:]), times
