"""Widths TMA cannot address (rows that are no 16-byte multiples) on the tensor cores through padded copies, and the
convolution's unfolding kernel, against the oracle and the torch restatement of the operands."""
import numpy as np
import pytest
import torch

import oracle
import paper_2510_00236_b200 as pe
from paper_2510_00236_b200 import conv_unfold, inputs
from parity_util import SIGN_REL, check_sign, rel_frob

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
# Accumulated in the tensor core by truncation, at most 512 tokens = 32 instructions per accumulator: a deficit of up to 32 * 2^-24
# = 2e-6 of a sum and twice that of its square, beside fp32 rounding of the outer sums (sqrt(100) * 6e-8)
TOL = 5e-6


# d_in odd, d_in = 2 mod 4 and d_in = 4 mod 8 (the last one still has 16-byte output rows), X or dY or both to be padded, every
# shift of a row against a 16-byte word, tails that reach the end of the tensor, short and long sequences, split and whole batches
@pytest.mark.parametrize("B,T,d_in,d_out", [(4, 300, 513, 520), (8, 128, 512, 1029), (6, 400, 362, 379), (3, 700, 388, 392),
                                            (70, 16, 505, 511), (2, 1030, 385, 384), (16, 64, 1001, 515), (33, 32, 515, 513)])
def test_odd_widths_on_the_tensor_cores(B, T, d_in, d_out):
    assert pe.pe_linear_stats_padded_workspace_bytes(B, T, d_in, d_out) > 0
    li = inputs.heterogeneous_layer(B, T, d_in, d_out, seed=40 + B + d_in, device=DEV, with_weights=False)
    st = oracle.linear_stats(inputs.to_numpy_bits(li.X), inputs.to_numpy_bits(li.dY), small_rel=SIGN_REL)
    nan = lambda: torch.full((d_out, d_in), float("nan"), device=DEV)
    for both in (True, False):
        mean, sq, sg, ident = (nan() if both else None), nan(), nan(), nan()
        pe.pe_linear_stats(li.X, li.dY, "square", mean, sq)
        assert pe.pe_last_path() == pe.PATH_TENSOR
        pe.pe_linear_stats(li.X, li.dY, "sign", mean, sg)
        pe.pe_linear_stats(li.X, li.dY, "identity", mean, ident)
        if both:
            assert rel_frob(mean.cpu().numpy(), st.sum_g) <= TOL
        assert rel_frob(sq.cpu().numpy(), st.sum_g2) <= TOL and rel_frob(ident.cpu().numpy(), st.sum_g) <= TOL
        check_sign(sg.cpu().numpy(), st)
    outs = [nan() for _ in range(3)]
    pe.pe_linear_stats_all(li.X, li.dY, *outs)
    assert rel_frob(outs[0].cpu().numpy(), st.sum_g) <= TOL and rel_frob(outs[1].cpu().numpy(), st.sum_g2) <= TOL
    check_sign(outs[2].cpu().numpy(), st)
    acc = [torch.ones((d_out, d_in), device=DEV) for _ in range(2)]
    pe.pe_linear_stats_accumulate(li.X, li.dY, "square", *acc)
    assert rel_frob(acc[0].cpu().numpy() - 1.0, st.sum_g) <= 10 * TOL      # the added 1 costs up to 2^-24 of itself
    assert rel_frob(acc[1].cpu().numpy(), st.sum_g2 + 1.0) <= TOL
    assert pe.pe_get_async_status(DEV) == (0, 0)


# channel counts and kernels whose features are no multiples of 8, several channel rounds (C * K * K rows over the block's shared
# memory), rows cut into runs, borders on every side, unequal strides / paddings / dilations, small (SIMT) and large layers
@pytest.mark.parametrize("B,C,F,H,W,K,stride,padding,dilation", [
    (3, 3, 16, 21, 33, (3, 3), (1, 1), (1, 1), (1, 1)), (2, 5, 9, 30, 17, (5, 3), (2, 1), (0, 2), (1, 2)), (4, 64, 96, 28, 28, (3, 3), (1, 1), (1, 1), (1, 1)),
    (2, 24, 40, 40, 300, (7, 7), (1, 2), (3, 3), (1, 1)), (6, 3, 64, 64, 64, (7, 7), (2, 2), (3, 3), (1, 1)), (2, 1, 8, 9, 9, (1, 1), (1, 1), (0, 0), (1, 1)),
    (1, 130, 33, 14, 150, (3, 5), (1, 1), (2, 0), (2, 3))])
def test_unfolded_convolution(B, C, F, H, W, K, stride, padding, dilation):
    g = torch.Generator(device="cpu").manual_seed(B * 100 + C)
    x = torch.randn((B, C, H, W), generator=g).to(torch.bfloat16).to(DEV)
    Ho, Wo = ((n + 2 * p - d * (k - 1) - 1) // s + 1 for n, p, d, k, s in zip((H, W), padding, dilation, K, stride))
    gy = (torch.randn((B, F, Ho, Wo), generator=g) / 8).to(torch.bfloat16).to(DEV)
    assert pe.pe_conv2d_stats_workspace_bytes(B, C, H, W, F, *K, stride, padding, dilation) > 0
    X, dY = conv_unfold.conv2d_operands(x, gy, K, stride, padding, dilation)
    # (the reference in fp64 on the GPU: one batched product per image)
    G = torch.stack([dY[b].double().T @ X[b].double() for b in range(B)])
    for phi, want in (("square", (G * G).sum(0)), ("identity", G.sum(0))):
        mean, stat = conv_unfold.pe_conv2d_stats(x, gy, (F, C, *K), phi, stride, padding, dilation)
        aligned = C * K[0] * K[1] % 8 == 0 and F % 8 == 0      # those take one accumulator per image: ceil(T / 16) instructions
        TOL = max(5e-6, (Ho * Wo / 16 + 1) * 2.0 ** -23) if aligned else 5e-6
        assert mean.shape == (F, C, *K)
        assert rel_frob(mean.reshape(F, -1).cpu().numpy(), G.sum(0).cpu().numpy()) <= TOL
        assert rel_frob(stat.reshape(F, -1).cpu().numpy(), want.cpu().numpy()) <= TOL
    # other dtypes and layouts (identity, or the two sums: the same mean) of the same values
    mean2, _ = conv_unfold.pe_conv2d_stats(x.double(), gy.float().to(memory_format=torch.channels_last), (F, C, *K), "square", stride, padding, dilation)
    assert rel_frob(mean2.reshape(F, -1).cpu().numpy(), G.sum(0).cpu().numpy()) <= TOL
    assert pe.pe_get_async_status(DEV) == (0, 0)


def test_a_receptive_field_beyond_the_unfolding_kernel_goes_through_torch():
    g = torch.Generator(device="cpu").manual_seed(5)
    x = torch.randn((2, 8, 130, 130), generator=g).to(torch.bfloat16).to(DEV)
    gy = torch.randn((2, 8, 3, 3), generator=g).to(torch.bfloat16).to(DEV)
    assert pe.pe_conv2d_stats_workspace_bytes(2, 8, 130, 130, 8, 128, 128, (1, 1), (0, 0), (1, 1)) == 0
    X, dY = conv_unfold.conv2d_operands(x, gy, (128, 128))
    mean, _ = conv_unfold.pe_conv2d_stats(x, gy, (8, 8, 128, 128), "square")
    want = torch.einsum("bto,bti->oi", dY.double(), X.double())
    assert rel_frob(mean.reshape(8, -1).cpu().numpy(), want.cpu().numpy()) <= TOL
