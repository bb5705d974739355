"""Sequences of at most 32 tokens: the kernel of its own that contracts two examples per hand-off."""
import math

import pytest
import torch

import paper_2510_00236_b200 as pe

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# one and two MMA steps, odd batches (a last unit of one example), one example, partial 128- and 32-column pieces, tiles on both sides of the
# number of pairs, batches split so finely that a slice holds one example, widths that go by way of padded copies (rows of 4 k and of odd length),
# whole tiles of many examples beside sliced ones, with and without copies
@pytest.mark.parametrize("B,T,d_in,d_out", [(1, 1, 8, 8), (5, 16, 136, 264), (4, 17, 128, 256), (33, 32, 200, 520), (2, 31, 264, 40), (9, 2, 96, 76 * 256),
                                            (3, 32, 1032, 21 * 256 + 8), (200, 3, 64, 72), (70, 9, 612, 1037), (64, 32, 333, 520), (49, 2, 1123, 5035),
                                            (90, 20, 1544, 2824)])
@pytest.mark.parametrize("zeros", [False, True])
def test_short_sequences_against_fp64(B, T, d_in, d_out, zeros):
    g = torch.Generator(device=DEV).manual_seed(B * T)
    X = torch.randn((B, T, d_in), generator=g, device=DEV).bfloat16()
    dY = (torch.randn((B, T, d_out), generator=g, device=DEV) * T ** -0.5).bfloat16()
    if zeros:       # columns, rows and whole examples whose G_b is exactly zero
        X[::2, :, ::3] = 0
        dY[1::3, :, 1::5] = 0
        X[B // 2] = 0
    new = lambda: torch.full((d_out, d_in), float("nan"), device=DEV)       # noqa: E731
    mean, square, sign, mean1, square1, mean2, sign2, square3, sign3 = (new() for _ in range(9))
    pe.pe_linear_stats_all(X, dY, mean, square, sign)
    pe.pe_linear_stats(X, dY, "square", mean1, square1)
    pe.pe_linear_stats(X, dY, "sign", mean2, sign2)
    pe.pe_linear_stats(X, dY, "square", None, square3)
    pe.pe_linear_stats(X, dY, "sign", None, sign3)
    more = [t.clone() for t in (mean1, square1)]
    pe.pe_linear_stats_accumulate(X, dY, "square", *more)
    assert pe.pe_get_async_status(DEV) == (0, 0)
    G = torch.einsum("bto,bti->boi", dY.double(), X.double())
    # a term of G_b is exact in fp32 and its sum is taken in fp32, truncated: (T + B) * 2^-23 of the sum of magnitudes at most
    mag = torch.einsum("bto,bti->boi", dY.double().abs(), X.double().abs())
    eps = (T + B) * 2.0 ** -23
    for got, times in ((mean, 1), (mean1, 1), (mean2, 1), (more[0], 2)):
        assert torch.all((got.double() - times * G.sum(0)).abs() <= times * eps * mag.sum(0))
    for got, times in ((square, 1), (square1, 1), (square3, 1), (more[1], 2)):
        assert torch.all((got.double() - times * (G * G).sum(0)).abs() <= times * 3 * eps * (mag * mag).sum(0))
    unsure = ((G.abs() <= eps * mag) & (mag > 0)).sum(0)
    for got in (sign, sign2, sign3):
        assert torch.all((got.double() - G.sign().sum(0)).abs() <= 2 * unsure)


# the 128 tiles of this layer are more than there are pairs: whole tiles over the batch where the 16-bit counts of the signs hold it (32767 examples:
# 65535 exactly), slices beyond
@pytest.mark.parametrize("B", [32767, 33000, 70000])
def test_counts_of_signs_do_not_overflow(B):
    T, d = 2, 2048
    g = torch.Generator(device=DEV).manual_seed(B)
    X = torch.randn((B, T, d), generator=g, device=DEV, dtype=torch.bfloat16)
    dY = torch.randn((B, T, d), generator=g, device=DEV, dtype=torch.bfloat16)
    sign = pe.pe_linear_stats_all(X, dY)[2]
    rows = torch.tensor([0, 1, 255, 256, 1000, 1337, 2046, 2047], device=DEV)
    want, unsure = 0, 0
    for b in range(0, B, 1000):
        x, y = X[b:b + 1000].double(), dY[b:b + 1000, :, rows].double()
        G, mag = torch.einsum("bto,bti->boi", y, x), torch.einsum("bto,bti->boi", y.abs(), x.abs())
        want, unsure = want + G.sign().sum(0), unsure + (G.abs() <= T * 2.0 ** -23 * mag).sum(0)
    assert torch.all((sign[rows].double() - want).abs() <= 2 * unsure)
    X.abs_().add_(0.5)
    dY.abs_().add_(0.5)
    assert torch.all(pe.pe_linear_stats_all(X, dY)[2] == B)
    assert pe.pe_get_async_status(DEV) == (0, 0)


# layers of more tiles than pairs by a fraction of a wave.  Rounding to nearest leaves u^2 / 6 on average (u = 2^-24); a sum of p examples at a time has an
# error of u sqrt(p / 6) against terms of either sign, u p / sqrt(18 B) against squares, beside the contraction's (T truncations in fp32, averaged over the batch)
@pytest.mark.parametrize("outputs,B,T,d_in,d_out,p", [(2, 2021, 24, 2336, 1728, 405), (3, 1545, 4, 1624, 2296, 309), (1, 1395, 5, 1696, 1336, 200)])
def test_precision_of_sums_over_many_examples(outputs, B, T, d_in, d_out, p):
    g = torch.Generator(device=DEV).manual_seed(B)
    X = torch.randn((B, T, d_in), generator=g, device=DEV, dtype=torch.bfloat16)
    dY = torch.randn((B, T, d_out), generator=g, device=DEV, dtype=torch.bfloat16)
    if outputs == 1:
        mean, square = None, torch.empty((d_out, d_in), device=DEV)
        pe.pe_linear_stats(X, dY, "square", None, square)
    else:
        mean, square = (pe.pe_linear_stats_all(X, dY) if outputs == 3 else pe.pe_linear_stats(X, dY, "square"))[:2]
    rows = torch.randperm(d_out, generator=torch.Generator().manual_seed(1))[:96].to(DEV)
    m, q = 0, 0
    for b in range(0, B, 64):
        G = torch.einsum("bto,bti->boi", dY[b:b + 64, :, rows].double(), X[b:b + 64].double())
        m, q = m + G.sum(0), q + (G * G).sum(0)
    u = 2.0 ** -24
    if mean is not None:
        assert (mean[rows].double() - m).norm() <= 1.25 * u * math.sqrt((p + B / p) / 6) * m.norm()
    assert (square[rows].double() - q).norm() <= 1.25 * u * math.sqrt(p * p / (18 * B) + B / p / 18 + T / 6) * q.norm()


# an infinity or a NaN of one example reaches its own column of the sums and nothing else: not the other example of its unit of two, the missing one of a
# last unit, the tokens past the sequence's end
@pytest.mark.parametrize("T", [2, 17, 32])
@pytest.mark.parametrize("bad", [0, 1, 4])
def test_infinities_and_nan_stay_in_their_columns(T, bad):
    B, d_in, d_out = 5, 136, 264
    g = torch.Generator(device=DEV).manual_seed(T)
    X = torch.randn((B, T, d_in), generator=g, device=DEV).bfloat16()
    dY = (torch.rand((B, T, d_out), generator=g, device=DEV) + 0.5).bfloat16()
    dY[:, :, ::3] *= -1
    X[bad, T - 1, 7], X[bad, 0, 70], X[bad, 0, 130] = float("inf"), float("-inf"), float("nan")
    new = lambda: torch.empty((d_out, d_in), device=DEV)       # noqa: E731
    mean, square, sign, mean1, square1, square2, mean3, sign3, sign4 = (new() for _ in range(9))
    pe.pe_linear_stats_all(X, dY, mean, square, sign)
    pe.pe_linear_stats(X, dY, "square", mean1, square1)
    pe.pe_linear_stats(X, dY, "square", None, square2)
    pe.pe_linear_stats(X, dY, "sign", mean3, sign3)
    pe.pe_linear_stats(X, dY, "sign", None, sign4)
    assert pe.pe_get_async_status(DEV) == (0, 0)
    G = torch.einsum("bto,bti->boi", dY.double(), X.double())
    mag = torch.einsum("bto,bti->boi", dY.double().abs(), X.double().abs().nan_to_num(0, 0, 0))
    finite = torch.ones(d_in, dtype=torch.bool, device=DEV)
    finite[[7, 70, 130]] = False
    eps = (T + B) * 2.0 ** -23
    for got in (mean, mean1, mean3):
        assert torch.all((got.double() - G.sum(0))[:, finite].abs() <= (eps * mag.sum(0))[:, finite])
        assert torch.equal(got[:, [7, 70]].double(), G.sum(0)[:, [7, 70]]) and torch.isnan(got[:, 130]).all()
    for got in (square, square1, square2):
        assert torch.all((got.double() - (G * G).sum(0))[:, finite].abs() <= (3 * eps * (mag * mag).sum(0))[:, finite])
        assert torch.isinf(got[:, [7, 70]]).all() and torch.isnan(got[:, 130]).all()
    number = torch.arange(d_in, device=DEV) != 130               # (the sign of a NaN is not specified)
    unsure = (G.abs() <= eps * mag).sum(0)
    for got in (sign, sign3, sign4):
        assert torch.all((got.double() - G.sign().sum(0))[:, number].abs() <= 2 * unsure[:, number])
