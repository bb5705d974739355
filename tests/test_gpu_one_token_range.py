"""Examples of a single token whose rows span a range that their squares, or the products of their entries, do not have in fp32: the
statistics are those of G_b in fp32."""
import pytest
import torch

import paper_2510_00236_b200 as pe

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
INF, NAN = float("inf"), float("nan")


def _rows(kind, n, d_in, d_out, g):
    x, y = torch.randn((n, d_in), generator=g, device=DEV), torch.randn((n, d_out), generator=g, device=DEV)
    small = torch.arange(d_in, device=DEV) % 2 == 1
    if kind == "zero row":                      # G = 0, whatever the other row holds
        return x * 0, y * 2.0 ** 100
    if kind == "subnormal row":
        return x * 2.0 ** -130, y * 2.0 ** 100
    if kind == "infinity beside 2^70":
        x, y = x * 2.0 ** 70, y * 2.0 ** -80
        x[:, 3] = INF
    elif kind == "undefined entry":
        x[:, 5], y[0, 7] = NAN, -INF
    elif kind == "entries 2^-90 below":         # squares of 2^-140, products of 2^-50 with the largest of the other row
        x, y = torch.where(small, x * 2.0 ** -70, x * 2.0 ** 20), y * 2.0 ** 20
    elif kind == "products of zero":            # below 2^-149: zero in fp32, for a part of the columns
        x, y = torch.where(small, x * 2.0 ** -100, x), y * 2.0 ** -60
    elif kind == "products of zero, all":
        x, y = x * 2.0 ** -90, y * 2.0 ** -90
    elif kind == "entries 2^-110 below":        # in both rows: no scale keeps the squares of both
        x, y = torch.where(small, x * 2.0 ** -90, x * 2.0 ** 20), torch.where(torch.arange(d_out, device=DEV) % 3 == 1, y * 2.0 ** -60, y * 2.0 ** 30)
    elif kind == "one row wide":                # the usual tails of a softmax; a scale that keeps the other row's squares, too
        y = torch.where(torch.arange(d_out, device=DEV) % 3 == 1, y * 2.0 ** -70, y)
    elif kind == "products of 2^57":            # sums of squares below 510 * (1.5^2 * 2^57)^2 < 2^126, close to the end of fp32
        x, y = x.clamp(-1.5, 1.5) * 2.0 ** 98, y.clamp(-1.5, 1.5) * 2.0 ** -41
    elif kind == "squares beyond fp32":         # infinite in half of the columns, 2^4 in the others
        x, y = torch.where(small, x, x * 2.0 ** 64), y * 4
    else:
        assert kind == "ordinary"
    return x, y


KINDS = ["ordinary", "zero row", "subnormal row", "infinity beside 2^70", "undefined entry", "entries 2^-90 below", "products of zero",
         "products of zero, all", "entries 2^-110 below", "one row wide", "products of 2^57", "squares beyond fp32"]


# all examples of the kind or a third of them between zeros; several chunks of 64 with a partial one; aligned and odd widths
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("B,d_in,d_out,every", [(510, 520, 512, 1), (1030, 333, 401, 3)])
def test_statistics_are_those_of_the_products_in_fp32(kind, B, d_in, d_out, every):
    assert pe.pe_linear_stats_padded_workspace_bytes(B, 1, d_in, d_out) > 0, "the route under test"
    g = torch.Generator(device=DEV).manual_seed(B + len(kind))
    X, dY = torch.zeros((B, 1, d_in), device=DEV), torch.zeros((B, 1, d_out), device=DEV)
    X[::every, 0], dY[::every, 0] = _rows(kind, len(range(0, B, every)), d_in, d_out, g)
    X, dY = X.bfloat16(), dY.bfloat16()
    want_square, want_sign = torch.zeros((d_out, d_in), dtype=torch.float64, device=DEV), torch.zeros((d_out, d_in), device=DEV)
    for b in range(0, B, every):
        G = dY[b, 0].float()[:, None] * X[b, 0].float()[None, :]
        want_square += (G * G).double()
        want_sign += (G > 0).float() - (G < 0).float()
    _, square, sign = pe.pe_linear_stats_all(X, dY)
    square1, sign1 = torch.full_like(square, NAN), torch.full_like(sign, NAN)
    pe.pe_linear_stats(X, dY, "square", None, square1)
    pe.pe_linear_stats(X, dY, "sign", None, sign1)
    more = [torch.ones_like(square), torch.ones_like(square)]
    pe.pe_linear_stats_accumulate(X, dY, "sign", more[0], more[1])
    assert pe.pe_get_async_status(DEV) == (0, 0)
    assert torch.equal(sign, want_sign) and torch.equal(sign1, want_sign) and torch.equal(more[1] - 1, want_sign)
    finite = want_square.isfinite()
    # the operands are exact, sums of 4 B products in fp32, truncated; a product below fp32's normal range may be lost
    eps, lost = (16 + B // 16) * 2.0 ** -23, 4 * B * 2.0 ** -126
    for got in (square, square1):
        assert torch.equal(got.isnan(), want_square.isnan()) and torch.equal(got.isinf(), want_square.isinf())
        assert torch.all(((got.double() - want_square).abs() <= eps * want_square + lost)[finite])
