"""Per-example norms of layers of many tiles: a pair takes tiles and slices of the batch in turn."""
import pytest
import torch

import paper_2510_00236_b200 as pe

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# slices of one example and of several, a shorter last one, one example, partial tiles, one stage and several per example
@pytest.mark.parametrize("B,T,d_in,d_out", [(16, 512, 1032, 4096), (50, 120, 1400, 2000), (37, 300, 2048, 1544), (1, 64, 4104, 4096), (211, 40, 520, 2600), (3, 17, 2600, 8 * 1001)])
def test_norms_against_fp64(B, T, d_in, d_out):
    g = torch.Generator(device=DEV).manual_seed(B * T)
    X = torch.randn((B, T, d_in), generator=g, device=DEV).bfloat16()
    dY = (torch.randn((B, T, d_out), generator=g, device=DEV) * T ** -0.5).bfloat16()
    got = pe.pe_example_sqnorms(X, dY, torch.full((B,), float("nan"), device=DEV))
    assert pe.pe_get_async_status(DEV) == (0, 0)
    want = torch.stack([(dY[b].double().T @ X[b].double()).square().sum() for b in range(B)])
    assert torch.allclose(got.double(), want, rtol=2e-5)         # squares of sums truncated once per 16 tokens, and fp32 sums of all of them


@pytest.mark.parametrize("B,T,d_in,d_out", [(40, 64, 1032, 4096), (7, 200, 264, 520)])
def test_infinities_and_nan_stay_with_their_examples(B, T, d_in, d_out):
    g = torch.Generator(device=DEV).manual_seed(B)
    X = torch.randn((B, T, d_in), generator=g, device=DEV).bfloat16()
    dY = (torch.randn((B, T, d_out), generator=g, device=DEV) * T ** -0.5).bfloat16()
    X[1, T - 1, 5], dY[B - 1, 0, d_out - 1], X[4, 3, d_in - 1] = float("inf"), float("-inf"), float("nan")
    got = pe.pe_example_sqnorms(X, dY, torch.empty(B, device=DEV))
    want = torch.stack([(dY[b].double().T @ X[b].double()).square().sum() for b in range(B)])
    assert torch.isnan(got[4]) and not torch.isfinite(got[[1, B - 1]]).any()          # (an infinity times a zero is a NaN)
    rest = [b for b in range(B) if b not in (1, 4, B - 1)]
    assert torch.allclose(got[rest].double(), want[rest], rtol=2e-5)
