"""fp32 layers of a few hundred rows and columns, which the kernel takes in tiles of 64 x 64 by blocks of 128 threads."""
import pytest
import torch

import paper_2510_00236_b200 as pe

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# whole and partial tiles, rows of whole groups of four and of odd length, sequences of whole chunks, of remainders of 1 and 8 tokens and shorter than a
# chunk, one and several batch slices (9 x 7: the rule's other side)
@pytest.mark.parametrize("B,T,d_in,d_out", [(10, 200, 800, 400), (64, 32, 500, 300), (20, 185, 406, 881), (5, 20, 1100, 1100), (9, 7, 700, 640), (23, 168, 247, 489)])
def test_against_fp64(B, T, d_in, d_out):
    g = torch.Generator(device=DEV).manual_seed(B * T)
    X = torch.randn((B, T, d_in), generator=g, device=DEV)
    dY = torch.randn((B, T, d_out), generator=g, device=DEV) * T ** -0.5
    new = lambda: torch.full((d_out, d_in), float("nan"), device=DEV)       # noqa: E731
    mean, square, sign, token = new(), new(), new(), new()
    pe.pe_linear_stats_f32(X, dY, "square", mean, square)
    pe.pe_linear_stats_f32(X, dY, "sign", None, sign)
    pe.pe_token_sqstats_f32(X, dY, token)
    assert pe.pe_last_path() == pe.PATH_SIMT
    if (B, T) != (9, 7):
        assert 4 in (pe.pe_plan_query(what, outputs, B, T, d_in, d_out, 148)[0] for what, outputs in ((pe.PLAN_SIMT_STATS, 1), (pe.PLAN_SIMT_STATS, 0), (pe.PLAN_SIMT_TOKEN, 0)))
    G, mag = torch.einsum("bto,bti->boi", dY.double(), X.double()), torch.einsum("bto,bti->boi", dY.double().abs(), X.double().abs())
    # sums of T products and of B terms, a rounding each
    eps = (T + B) * 2.0 ** -24
    assert torch.all((mean.double() - G.sum(0)).abs() <= eps * mag.sum(0))
    assert torch.all((square.double() - (G * G).sum(0)).abs() <= 3 * eps * (mag * mag).sum(0))
    assert torch.all((sign.double() - G.sign().sum(0)).abs() <= 2 * (G.abs() <= eps * mag).sum(0))
    want = dY.double().reshape(-1, d_out).square().T @ X.double().reshape(-1, d_in).square()
    assert torch.all((token.double() - want).abs() <= (B * T + 2) * 2.0 ** -24 * want)
