"""The cut-off search of the cluster selection kernel where its branches turn: bins of the first
histogram with one value, with more keys than are ranked directly (a second histogram), with
enough to be narrowed before ranking, with every key equal; slices at the edges of a warp's step, of
a CTA and of the cluster widths.  Bit for bit against the oracle."""
import numpy as np
import pytest

from oracle import codecomp_oracle as orc

from test_gpu_stages import run_select

pytestmark = pytest.mark.gpu


def _values(kind, rng, hkv, n):
    if kind == "equal":
        return np.full((hkv, n), 0.25, np.float32)
    if kind == "few":                           # crowded bins of one value each
        return rng.integers(0, 5, (hkv, n)).astype(np.float32)
    if kind == "outlier":                       # everything but one item in the lowest bin
        x = (1.0 + rng.random((hkv, n)) * 1e-4).astype(np.float32)
        x[:, n // 2] = 1e30
        return x
    if kind == "negative":
        return (-rng.random((hkv, n))).astype(np.float32)
    return np.exp(rng.standard_normal((hkv, n))).astype(np.float32)


@pytest.mark.parametrize("kind", ["equal", "few", "outlier", "negative", "spread"])
@pytest.mark.parametrize("n", [1, 31, 33, 511, 513, 1025, 4097, 16383, 40961])
def test_cut_off_search(kind, n):
    rng = np.random.Generator(np.random.PCG64(n + len(kind)))
    hkv = 3
    fused = _values(kind, rng, hkv, n)
    prior = (rng.random(n) < 0.05).astype(np.float32)
    for budget in sorted({1, n // 3, n // 2, n - 1} - {0}):
        for cap in (0.0, 0.3):
            idx, count = run_select(fused, prior, n, budget, 0.5, span_ratio=cap, span_min=2)
            keep = min(budget, n)
            for h in range(hkv):
                ref = orc.select_tokens(fused[h], prior, n, budget, 0.5, cap, 2)
                assert count[h] == keep
                np.testing.assert_array_equal(idx[h, :keep], ref, err_msg=f"{kind} n={n} B={budget} cap={cap} h={h}")


@pytest.mark.parametrize("kind", ["spread", "outlier", "few"])
@pytest.mark.parametrize("n,hkv,chunk", [(40000, 3, 1), (40961, 40, 1), (131072, 2, 1), (90007, 8, 3)])
def test_cap_cut_off_by_a_graded_prior_over_several_ctas(kind, n, hkv, chunk):
    """Both searches of the kernel list and rank candidates (or refine a crowded bin first) in clusters of
    two and more: the cap's among priors that differ everywhere, then the budget's."""
    rng = np.random.Generator(np.random.PCG64(n + hkv))
    fused = _values(kind, rng, hkv, -(-n // chunk))
    prior = rng.random(n).astype(np.float32)
    if kind == "outlier":                       # the protected tokens' priors in one bin of the first histogram
        prior[prior >= 0.5] = (0.5 + rng.random(int((prior >= 0.5).sum())) * 1e-4).astype(np.float32)
        prior[n // 3] = 1e30
    _, item_prior = orc.chunk_reduce(np.zeros((1, n), np.float32), prior, chunk, dtype=np.float32)
    for budget in (n // 4, n // 3):
        for cap in (0.3, 0.9):
            idx, count = run_select(fused, prior, n, budget, 0.5, span_ratio=cap, span_min=2, chunk=chunk)
            for h in range(hkv):
                ref = orc.select_tokens(fused[h], item_prior, n, budget, 0.5, cap, 2, chunk=chunk)
                assert count[h] == len(ref) == budget
                np.testing.assert_array_equal(idx[h], ref, err_msg=f"{kind} n={n} B={budget} cap={cap} h={h}")
