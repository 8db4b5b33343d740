"""Score parity where the tensor-core kernel cuts tiles at their middle between two CTAs (few tiles
per SM: fewer than half a tile each, a last or first half, several problems in a span), contiguous,
paged and causal, and where a span holds many short problems."""
import numpy as np
import pytest

from oracle import codecomp_oracle as orc
from paper_2604_10235_b200 import binding as cc
from paper_2604_10235_b200 import inputs as gen

from test_gpu_score import check_against_oracle, run_scores

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,hq,hkv,lens,page,causal", [
    (64, 28, 4, (2000,), 0, False), (64, 32, 8, (1000,), 0, False), (128, 32, 8, (777,), 16, False),
    (64, 28, 4, (10007,), 0, True), (64, 8, 2, (11000,), 0, False), (128, 8, 2, (700, 40, 1300), 32, False),
    (128, 8, 2, (150,) * 40, 0, False), (64, 28, 4, (500,) * 30, 16, True)])
def test_scores_of_cut_tiles_and_short_problems(w, hq, hkv, lens, page, causal):
    wl = gen.Workload("spans", 27, 1, hq, hkv, 128, w, gen.POOL_MAX, 7, 0, seq_lens=lens, budget_frac=0.1,
                      page_size=page, causal=causal)
    check_against_oracle(wl, gen.make_layer(wl, layer=sum(lens), with_v=False), cc.CC_MODE_BF16, 2e-3)


@pytest.mark.parametrize("w,hq,hkv", [(16, 2, 2), (32, 2, 2), (96, 2, 2), (112, 2, 2), (36, 8, 2), (56, 8, 2), (68, 8, 2),
                                      (48, 28, 4), (100, 8, 2), (50, 28, 4), (64, 28, 4)])
@pytest.mark.parametrize("lens,page", [((20000,), 0), ((500, 130, 77) * 3, 16)])
def test_scores_where_the_last_block_of_rows_is_not_full(w, hq, hkv, lens, page):
    """16 to 448 rows, one to four blocks of 128, the last of which has 0 to 3 warps without rows."""
    wl = gen.Workload("padded", 28, 1, hq, hkv, 128, w, gen.POOL_MAX, 7, 0, seq_lens=lens, budget_frac=0.1, page_size=page)
    check_against_oracle(wl, gen.make_layer(wl, layer=w, with_v=False), cc.CC_MODE_BF16, 2e-3)


# Error budget: the polynomial's 7.8e-5 twice (value and row sum) and f32 products and references below 64, 2^-18.
@pytest.mark.parametrize("w,hq,hkv", [(16, 8, 8), (12, 32, 8), (16, 56, 8), (50, 32, 8), (96, 32, 8), (64, 56, 8), (128, 32, 8)])
@pytest.mark.parametrize("lens,page,causal", [((41000,), 0, False), ((5000, 130, 77, 300, 9000, 1, 700, 26000), 16, False),
                                              ((40000, 300), 0, True)])
def test_scores_whose_row_sums_the_product_subtracts(w, hq, hkv, lens, page, causal):
    """Sixteen items per CTA and more, 16 to 512 rows in one to four blocks, problems of one tile up to hundreds."""
    wl = gen.Workload("added", 30, 1, hq, hkv, 128, w, gen.POOL_MAX, 7, 0, seq_lens=lens, budget_frac=0.1, page_size=page,
                      causal=causal)
    check_against_oracle(wl, gen.make_layer(wl, layer=w, with_v=False), cc.CC_MODE_BF16, 2e-4)


@pytest.mark.parametrize("w,hq,hkv", [(16, 8, 8), (12, 32, 8), (50, 32, 8), (96, 32, 8), (128, 32, 8)])
@pytest.mark.parametrize("lens,page,causal", [((41000,), 0, False), ((5000, 130, 77, 300, 9000, 1, 700, 26000), 16, False),
                                              ((40000, 300), 0, True)])
def test_equal_keys_have_equal_scores(w, hq, hkv, lens, page, causal):
    """The tie rule (equal values: the lower index first) decides among equal keys, so nothing else may: wherever a key lies in its
    tile, in the span of its CTA and in the sequence, its score is the same bit for bit, as long as the same rows attend to it."""
    wl = gen.Workload("equal", 36, 1, hq, hkv, 128, w, gen.POOL_MAX, 7, 0, seq_lens=lens, budget_frac=0.1, page_size=page,
                      causal=causal)
    x = gen.make_layer(wl, layer=w, with_v=False)
    period = 61                                  # a prime: every key falls on every place of a tile
    for s, n in enumerate(lens):
        rows = orc.paged_rows(x.page_table[s], n, page) if page else np.arange(x.tok_offsets[s], x.tok_offsets[s] + n)
        x.k[rows] = x.k[rows[:period]][np.arange(n) % period]
    u, _ = run_scores(wl, x, cc.CC_MODE_BF16, want_lse=False)
    for s, n in enumerate(lens):
        lo = int(x.tok_offsets[s])
        seen = n - w + 1 if causal else n        # keys that all rows attend to
        own = u[:, lo:lo + seen]
        np.testing.assert_array_equal(own, own[:, np.arange(seen) % period])


@pytest.mark.parametrize("w,hq,hkv", [(16, 1, 1), (24, 1, 1), (128, 1, 1), (64, 7, 1), (128, 4, 1)])
@pytest.mark.parametrize("lens", [(19000,), (40000,), (7, 18500, 200, 21000)])
def test_scores_of_one_head_spread_over_all_ctas(w, hq, hkv, lens):
    """Up to 148 spans of a (sequence, head) to merge, 16 to 512 rows: sixteen threads for a pair of rows, or two."""
    wl = gen.Workload("merge", 31, 1, hq, hkv, 128, w, gen.POOL_MAX, 7, 0, seq_lens=lens, budget_frac=0.1)
    check_against_oracle(wl, gen.make_layer(wl, layer=w, with_v=False), cc.CC_MODE_BF16, 2e-4)
