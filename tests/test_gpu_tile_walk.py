"""Layers of more tiles than CTA pairs: one pair takes several tiles, and the last wave's tiles are split over the batch."""
import numpy as np
import pytest
import torch

import paper_2510_00236_b200 as pe

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# rows of tiles (of 256): a few more than the 74 pairs (the rest in slices), two whole waves, a batch of one example that no slice can
# share, more slices than examples; widths with a partial 192-, 128- and 32-column piece; T on both sides of the 32-token kernels
@pytest.mark.parametrize("B,T,d_in,d_out", [(9, 40, 200, 39 * 256 - 40), (24, 300, 192, 75 * 256), (5, 129, 136, 148 * 256 - 8), (1, 64, 512, 30 * 256 - 200),
                                            (3, 17, 1032, 21 * 256 + 8), (40, 8, 256, 76 * 256), (2, 32, 128, 149 * 256), (6, 600, 264, 80 * 256)])
def test_many_tiles_against_fp64(B, T, d_in, d_out):
    g = torch.Generator(device=DEV).manual_seed(B * T)
    X = torch.randn((B, T, d_in), generator=g, device=DEV).bfloat16()
    dY = (torch.randn((B, T, d_out), generator=g, device=DEV) * T ** -0.5).bfloat16()
    new = lambda: torch.full((d_out, d_in), float("nan"), device=DEV)       # noqa: E731
    mean, square, sign, mean1, square1, sign1, square2 = (new() for _ in range(7))
    pe.pe_linear_stats_all(X, dY, mean, square, sign)
    pe.pe_linear_stats(X, dY, "square", mean1, square1)
    pe.pe_linear_stats(X, dY, "sign", None, sign1)
    pe.pe_linear_stats(X, dY, "square", None, square2)
    clipped, norms = pe.pe_linear_clipped_sum(X, dY, 0.9 * (d_in * d_out) ** 0.5)
    assert pe.pe_get_async_status(DEV) == (0, 0)
    rng = np.random.default_rng(T)
    o = torch.as_tensor(np.unique(np.concatenate([np.arange(0, d_out, 256), np.arange(255, d_out, 256), [d_out - 1], rng.integers(0, d_out, 60)])), device=DEV)
    G = torch.einsum("bto,bti->boi", dY[:, :, o].double(), X.double())
    # a term of G_b is exact in fp32 and its sum is taken in fp32, truncated: (T + B) * 2^-23 of the sum of magnitudes at most
    mag = torch.einsum("bto,bti->boi", dY[:, :, o].double().abs(), X.double().abs())
    eps = (T + B) * 2.0 ** -23
    for got in (mean, mean1):
        assert torch.all((got[o].double() - G.sum(0)).abs() <= eps * mag.sum(0))
    for got in (square, square1, square2):
        assert torch.all((got[o].double() - (G * G).sum(0)).abs() <= 3 * eps * (mag * mag).sum(0))
    unsure = (G.abs() <= eps * mag).sum(0)
    for got in (sign, sign1):
        assert torch.all((got[o].double() - G.sign().sum(0)).abs() <= 2 * unsure)
    norm = torch.stack([(dY[b].double().T @ X[b].double()).norm() for b in range(B)])
    assert torch.allclose(norms.double().sqrt(), norm, rtol=1e-5)
    want = (G * (0.9 * (d_in * d_out) ** 0.5 / norm).clamp(max=1.0)[:, None, None]).sum(0)
    assert torch.all((clipped[o].double() - want).abs() <= (eps + 1e-5) * mag.sum(0))


def test_rest_of_the_tiles_takes_a_second_launch():
    X, dY = torch.randn((24, 300, 192), device=DEV).bfloat16(), torch.randn((24, 300, 75 * 256), device=DEV).bfloat16()
    mean, square = torch.empty((75 * 256, 192), device=DEV), torch.empty((75 * 256, 192), device=DEV)
    pe.pe_reset_launch_count()
    pe.pe_linear_stats(X, dY, "square", mean, square)
    assert pe.pe_launch_count() == 2       # one tile more than pairs: zeroed first, then contracted by all of them
