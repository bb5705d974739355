"""Examples of a single token (T = 1): the statistics as contractions of row-wise functions of the operands."""
import pytest
import torch

import paper_2510_00236_b200 as pe

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _layer(B, d_in, d_out, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    X, dY = torch.randn((B, 1, d_in), generator=g, device=DEV), torch.randn((B, 1, d_out), generator=g, device=DEV)
    # examples whose two factors differ by up to 2^100 (their squares leave fp32, the squares of their products do not), zeros
    k = torch.randint(-50, 51, (B, 1, 1), generator=g, device=DEV).float()
    X, dY = X * torch.exp2(k), dY * torch.exp2(-k)
    X[torch.rand(X.shape, generator=g, device=DEV) < 0.1] = 0
    dY[:, :, d_out // 2] = 0
    return X.bfloat16(), dY.bfloat16()


# B below, at and past multiples of the 64 rows of an accumulator, and no multiple of 16; widths past tiles of 256, no multiples of 8 and of 4
@pytest.mark.parametrize("B,d_in,d_out", [(512, 512, 520), (513, 256, 1032), (70, 1544, 1256), (1300, 333, 401), (33, 2050, 2044), (5000, 264, 264), (2, 8200, 8192)])
def test_one_token_against_fp64(B, d_in, d_out):
    assert pe.pe_linear_stats_padded_workspace_bytes(B, 1, d_in, d_out) >= 4 * 2 * B * (d_in + d_out), "four copies: the route under test"
    X, dY = _layer(B, d_in, d_out, B)
    x, y = X[:, 0].double(), dY[:, 0].double()
    want_mean, want_square, want_sign = y.T @ x, (y * y).T @ (x * x), y.sign().T @ x.sign()
    new = lambda: torch.full((d_out, d_in), float("nan"), device=DEV)       # noqa: E731
    mean, square, sign, mean1, square1, sign1 = (new() for _ in range(6))
    pe.pe_linear_stats_all(X, dY, mean, square, sign)
    pe.pe_linear_stats(X, dY, "square", mean1, square1)
    pe.pe_linear_stats(X, dY, "sign", None, sign1)
    square2 = new()
    pe.pe_linear_stats(X, dY, "square", None, square2)
    more_mean, more_square = mean.clone(), square.clone()
    pe.pe_linear_stats_accumulate(X, dY, "square", more_mean, more_square)
    assert pe.pe_get_async_status(DEV) == (0, 0)
    # products are exact; an accumulator takes 4 additions of 16 products, the 4 B / 64 accumulators are added, all in fp32, truncated at 2^-23
    eps = (16 + B // 16) * 2.0 ** -23
    mag = y.abs().T @ x.abs()
    for got in (mean, mean1, more_mean / 2):
        assert torch.all((got.double() - want_mean).abs() <= eps * mag)
    for got in (square, square1, square2, more_square / 2):
        assert torch.all((got.double() - want_square).abs() <= eps * want_square)
    assert torch.equal(sign.double(), want_sign) and torch.equal(sign1.double(), want_sign)


def test_infinite_and_undefined_inputs():
    X, dY = _layer(600, 520, 512, 7)
    X[5, 0, 3], dY[9, 0, 4], X[40, 0, 100] = float("inf"), float("-inf"), float("nan")
    x, y = X[:, 0].float(), dY[:, 0].float()
    want = torch.zeros((512, 520), device=DEV)
    sign = torch.zeros_like(want)
    for b in range(600):
        G = y[b][:, None] * x[b][None, :]
        want += G * G
        sign += (G > 0).float() - (G < 0).float()
    _, square, got_sign = pe.pe_linear_stats_all(X, dY)
    assert torch.equal(square.isnan(), want.isnan()) and torch.equal(square.isinf(), want.isinf())
    assert torch.equal(got_sign, sign)
