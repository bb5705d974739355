"""Per-token statistic of layers whose tiles leave pairs idle in whole slices: the rows of all tiles dealt out evenly."""
import pytest
import torch

import paper_2510_00236_b200 as pe

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# 16, 48 and 60 tiles, partial ones among them; rows that are no multiple of a stage; pairs that hold parts of one and of two tiles; 5 tiles
@pytest.mark.parametrize("rows,d_in,d_out", [(16384, 512, 2048), (9999, 776, 3000), (4127, 1016, 3848), (20001, 264, 520), (3000, 256, 1280)])
def test_rows_dealt_out_evenly(rows, d_in, d_out):
    g = torch.Generator(device=DEV).manual_seed(rows)
    X = torch.randn((1, rows, d_in), generator=g, device=DEV).bfloat16()
    dY = (torch.randn((1, rows, d_out), generator=g, device=DEV) * torch.rand((1, rows, 1), generator=g, device=DEV)).bfloat16()
    out = torch.full((d_out, d_in), float("nan"), device=DEV)
    for _ in range(2):
        pe.pe_token_sqstats(X, dY, out)
    assert pe.pe_get_async_status(DEV) == (0, 0)
    want = dY[0].double().square().T @ X[0].double().square()
    # both factors rounded to 11 bits: 2^-11 each; fp32 sums, truncated once per 8 rows at 2^-24 or so
    assert torch.all((out.double() - want).abs() <= (2.0 ** -10 + rows / 8 * 2.0 ** -24) * want)


# 38, 32, 56 and 64 tiles, which are whole or in two parts: two sums on zero are the same in either order
@pytest.mark.parametrize("rows,d_in,d_out", [(2000, 512, 4864), (16384, 1024, 2048), (4001, 1784, 2048), (3001, 1024, 4096)])
def test_tiles_of_two_parts_repeat_bit_for_bit(rows, d_in, d_out):
    g = torch.Generator(device=DEV).manual_seed(rows)
    X = torch.randn((1, rows, d_in), generator=g, device=DEV).bfloat16()
    dY = torch.randn((1, rows, d_out), generator=g, device=DEV).bfloat16()
    first = pe.pe_token_sqstats(X, dY, torch.full((d_out, d_in), float("nan"), device=DEV))
    want = dY[0].double().square().T @ X[0].double().square()
    assert torch.all((first.double() - want).abs() <= (2.0 ** -10 + rows / 8 * 2.0 ** -24) * want)
    for _ in range(6):
        assert torch.equal(first, pe.pe_token_sqstats(X, dY, torch.full((d_out, d_in), float("nan"), device=DEV)))
