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
