"""Arguments of the exponentials of the tensor-core score kernel: their error (whole powers of two, where the polynomial of one
pair in three has one and the same error and only the argument's is left to see), and their range (logits that rise or lie where
the polynomial's exponent would wrap or its reference is no exact integer)."""
import numpy as np
import pytest
import torch

from paper_2604_10235_b200 import binding as cc
from paper_2604_10235_b200 import inputs as gen

from gpu_util import ctx
from oracle import codecomp_oracle as orc
from test_gpu_score import check_against_oracle
from test_gpu_score_rising import TOL

pytestmark = pytest.mark.gpu
LN2 = np.log(2.0)
SCALE = float(np.float32(0.12751743))        # powers of two per unit of a product: log2(e) / sqrt(128), rounded to f32


def bf16_pieces(x):
    """Three bf16 that add up to x, an f32."""
    rest, out = torch.tensor(float(np.float32(x)), dtype=torch.float64), []
    for _ in range(3):
        out.append(rest.to(torch.bfloat16))
        rest = rest - out[-1].double()
    assert float(rest) == 0.0
    return torch.stack(out)


def scores(d, q, k, rows_shape):
    u = torch.full((k.shape[1], k.shape[0]), -1.0, device="cuda")
    lse = torch.full(rows_shape, -1.0, device="cuda")
    cc.cc_score_window(ctx(), d, q, k, u, lse)
    assert ctx().poll() == 0
    return u.double().cpu().numpy(), lse.double().cpu().numpy()


@pytest.mark.parametrize("n", [16384, 16384 + 77])
def test_sums_of_keys_a_whole_power_below_the_reference(n):
    """Head c has the keys j = c modulo 32, one column of each chunk, at d powers of two below key 0; row t has the t-th d.
    log-sums of a head differ by what d makes of them, and by roundings: of the result below 6 (2^-22 each of logarithm,
    conversion to nats and sum with the reference, 0) and of at most 16 partial sums (2^-24 each), 1.2e-6 together."""
    depths = [0, 4, 5, 6, 7, 8, 9, 10, 11, 12, 4, 5, 6, 8, 10, 11]
    q = torch.zeros(16, 32, 128)
    k = torch.zeros(n, 32, 128)
    x = np.zeros(16)
    for t, d in enumerate(depths):
        q[t, :, 3 * t:3 * t + 3] = 1.0
        pieces = bf16_pieces(-d / SCALE)
        x[t] = float(pieces.double().sum()) * SCALE
        for c in range(32):
            k[:, c, 3 * t] = -30000.0
            k[c::32, c, 3 * t:3 * t + 3] = pieces.float()
    k[0] = 0.0
    _, lse = scores(cc.Desc(32, 32, 16, n=n, budget=1), q.bfloat16().cuda(), k.bfloat16().cuda(), (1, 32, 16))
    worst = 0.0
    for c in range(32):
        keys = len(range(c, n, 32)) - (c == 0)
        one = (np.exp(lse[0, c, 0]) - 1.0) / keys          # what 2^0 is in this column: 1, or the polynomial's value
        assert abs(one - 1.0) < 8e-5
        worst = max(worst, np.abs(lse[0, c] - np.log1p(keys * one * np.exp2(x))).max())
    assert worst < 1.2e-6, worst


def test_scores_of_whole_powers():
    """Row t of 16 has the keys j = t modulo 16, all at 0: sequences of 16 2^e keys have rows that sum to 2^e, and every score
    is 2^-e, up to the polynomial's value at 0 in its rows.  exp(-lse) is what the kernel has (2^-24 of at most 9.1 nats from its
    conversion, 5.4e-7); the argument itself is below 2^4 and good to 2^-21 powers of two (3.3e-7): 1.2e-6 with the sum's."""
    lens = tuple(16 << e for e in range(4, 14))
    n = sum(lens)
    q = torch.zeros(len(lens), 16, 4, 128)
    k = torch.full((n, 4, 128), -30000.0)
    for t in range(16):
        q[:, t, :, t] = 1.0
        k[t::16, :, t] = 0.0                               # (lengths are multiples of 16)
    d = cc.Desc(4, 4, 16, seq_lens=lens, budgets=(1,) * len(lens))
    u, lse = scores(d, q.bfloat16().cuda(), k.bfloat16().cuda(), (len(lens), 4, 16))
    ratio = [[] for _ in range(16)]
    lo = 0
    for s, m in enumerate(lens):
        for t in range(16):
            ratio[t].append((u[:, lo + t:lo + m:16] * np.exp(lse[s, :, t])[:, None]).ravel())
        lo += m
    for t in range(16):
        r = np.concatenate(ratio[t])
        assert abs(r.mean() - 1.0) < 8e-5
        centre = np.median(r)
        assert np.abs(r / centre - 1.0).max() < 1.2e-6, (t, np.abs(r / centre - 1.0).max())


def one_key(wl, at, logit, rest):
    """Every query's product with key `at` is logit sqrt(128) and with the others rest sqrt(128), besides N(0, 1) parts."""
    x = gen.make_layer(wl, layer=at, with_v=False)
    q = orc.bf16_bits_to_f64(x.q_win).astype(np.float32)
    q[..., 0] = 4.0
    x.q_win = gen.f32_to_bf16_bits(q)
    k = orc.bf16_bits_to_f64(x.k).astype(np.float32)
    k[:, :, 0] = rest * np.sqrt(128.0) / 4.0
    k[at, :, 0] = logit * np.sqrt(128.0) / 4.0
    x.k = gen.f32_to_bf16_bits(k)
    return x


@pytest.mark.parametrize("at", [32 + 4, 64 + 29, 128 + 32 + 17, 5 * 128 + 64 + 10])
@pytest.mark.parametrize("jump", [66.0, 72.0, 86.0, 100.0, 130.0, 260.0, 700.0])
def test_rises_in_columns_of_the_polynomial(at, jump):
    """95 to 1010 powers of two above the first keys: an exponent wraps from 128 on and comes round at 384."""
    wl = gen.Workload("rise", 33, 1, 8, 2, 128, 64, gen.POOL_MAX, 7, 1, n=1500)
    check_against_oracle(wl, one_key(wl, at, jump, 0.0), cc.CC_MODE_BF16, TOL)


@pytest.mark.parametrize("at", [4, 32 + 10, 64 + 29, 96 + 17, 128 + 96 + 5, 10 * 128 + 100])
@pytest.mark.parametrize("depth", [-80.0, -100.0, -1.0e3, -1.0e9, -1.0e13, -3.0e30])
def test_keys_far_below_in_columns_of_the_polynomial(at, depth):
    """Where 2^x underflows, where the cubic of the remainder is huge and where it overflows."""
    wl = gen.Workload("fall", 35, 1, 8, 2, 128, 64, gen.POOL_MAX, 7, 1, n=1500)
    check_against_oracle(wl, one_key(wl, at, depth, 0.0), cc.CC_MODE_BF16, TOL)


def check_one_key_with_all_of_every_row(n, at, logit, rest, causal, ulps):
    wl = gen.Workload("huge", 34, 1, 8, 2, 128, 64, gen.POOL_MAX, 7, 1, n=n, causal=causal)
    x = one_key(wl, at, logit, rest)
    d = cc.Desc(8, 2, 64, n=n, budget=1, causal=causal)
    q, k = (torch.from_numpy(a.view(np.int16)).view(torch.bfloat16).cuda() for a in (x.q_win, x.k))
    u, lse = scores(d, q, k, (1, 8, 64))
    assert np.isfinite(u).all() and np.isfinite(lse).all()
    off = 0.5 * np.spacing(np.float32(abs(logit) / LN2)) + ulps * SCALE * np.spacing(np.float32(abs(logit) * np.sqrt(128.0))) + 4e-4
    assert np.abs(np.log2(u[:, at] / 256.0)).max() < off
    assert u.sum() - u[:, at].sum() < 256.0 * 2e-4
    bits = orc.bf16_bits_to_f64(x.q_win).reshape(64, 8, 128), orc.bf16_bits_to_f64(x.k)[at]
    ref = np.einsum("whd,hd->hw", bits[0], np.repeat(bits[1], 4, axis=0)) / np.sqrt(128.0)
    np.testing.assert_allclose(lse[0], ref, rtol=1e-6, atol=0.2)


@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("at", [0, 31, 36, 100, 127, 128 + 80, 640 + 120])
@pytest.mark.parametrize("logit,rest", [(2.8e3, 0.0), (2.9e3, 0.0), (7.0e5, 0.0), (3.0e7, 0.0), (-1.0e3, -1.2e3),
                                        (-2.8e3, -4.0e3), (-7.3e5, -1.0e6), (-1.0e6, -4.0e6), (0.0, -1.0e9)])
def test_logits_of_any_size(at, logit, rest, causal):
    """References around 2^12 and far beyond, others far below: the one key has all of every row that attends to it.  Its scores are good to half a unit
    in the last place of the f32 row statistic and to one of the product, in powers of two."""
    check_one_key_with_all_of_every_row(1000, at, logit, rest, causal, 1)


@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("at", [5, 10 * 128 + 100, 41000, 79900])
@pytest.mark.parametrize("logit,rest", [(2.8e3, 0.0), (7.0e5, 0.0), (-2.8e3, -4.0e3), (-7.3e5, -1.0e6), (0.0, -1.0e9)])
def test_logits_of_any_size_in_a_long_call(at, logit, rest, causal):
    """The same where the product subtracts the row statistic (sixteen items per CTA and more): a rounding of it and one of its
    three parts' sum besides, each of at most a unit of the product."""
    check_one_key_with_all_of_every_row(80000, at, logit, rest, causal, 3)
