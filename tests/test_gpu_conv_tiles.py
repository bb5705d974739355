"""Convolutions of enough images for a block of the unfolding kernel to take several output rows."""
import pytest
import torch
import torch.nn.functional as F

import paper_2510_00236_b200 as pe
from paper_2510_00236_b200 import conv_unfold

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# eight, four and two output rows to a block, their number no multiple of that; image rows of odd length (single elements) and of even length whose
# first column is odd; stride, dilation, no padding; two tiles across; channels in several rounds; one column, one kernel row
@pytest.mark.parametrize("B,C,Fo,H,W,K,stride,padding,dilation", [
    (120, 3, 32, 43, 46, (7, 7), (2, 2), (3, 3), (1, 1)), (70, 2, 24, 37, 41, (5, 3), (1, 1), (2, 1), (1, 1)), (40, 4, 16, 45, 32, (3, 3), (1, 2), (0, 1), (2, 3)),
    (20, 1, 8, 33, 300, (3, 5), (1, 1), (1, 2), (1, 1)), (80, 40, 48, 21, 20, (3, 3), (1, 1), (1, 1), (1, 1)), (150, 2, 40, 50, 1, (4, 1), (1, 1), (0, 0), (1, 1)),
    (90, 3, 16, 9, 30, (1, 1), (1, 1), (0, 0), (1, 1))])
def test_several_output_rows_to_a_block(B, C, Fo, H, W, K, stride, padding, dilation):
    g = torch.Generator(device=DEV).manual_seed(B + C)
    x = torch.randn((B, C, H, W), generator=g, device=DEV).bfloat16()
    X = F.unfold(x.double(), K, padding=padding, stride=stride, dilation=dilation)
    T = X.shape[2]
    out = [(n + 2 * p - d * (k - 1) - 1) // s + 1 for n, p, d, k, s in zip((H, W), padding, dilation, K, stride)]
    gy = (torch.randn((B, Fo, *out), generator=g, device=DEV) * T ** -0.5).bfloat16()
    mean, square = conv_unfold.pe_conv2d_stats(x, gy, (Fo, C, *K), "square", stride, padding, dilation)
    assert pe.pe_get_async_status(DEV) == (0, 0)
    y = gy.double().reshape(B, Fo, T)
    G, mag = torch.einsum("bft,bit->bfi", y, X), torch.einsum("bft,bit->bfi", y.abs(), X.abs())
    # a term of G_b is exact in fp32 and its sum is taken in fp32, truncated: (T + B) * 2^-23 of the sum of magnitudes at most
    eps = (T + B) * 2.0 ** -23
    assert torch.all((mean.reshape(Fo, -1).double() - G.sum(0)).abs() <= eps * mag.sum(0))
    assert torch.all((square.reshape(Fo, -1).double() - (G * G).sum(0)).abs() <= 3 * eps * (mag * mag).sum(0))
