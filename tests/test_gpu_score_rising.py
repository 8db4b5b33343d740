"""Score parity where a row's logits rise far above its first keys': the running reference of pass 1 is looked
at before the first and the last 32 keys of a tile only, and a tile whose other keys overflow it is gone through again."""
import numpy as np
import pytest
import torch

from oracle import codecomp_oracle as orc
from paper_2604_10235_b200 import binding as cc
from paper_2604_10235_b200 import inputs as gen

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
