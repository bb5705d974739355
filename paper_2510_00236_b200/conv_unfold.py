"""Convolution layers through the same contraction (Appendix B.4, "For convolutions ..."): an image is
unfolded into one row per output position holding that position's receptive field, after which the layer is
the dense sequence-level layer of Section 2.3 with T = H_out * W_out "tokens" and d_in = C * K_h * K_w, and its
per-example weight gradient is G_b = dY_b^T X_b reshaped to [F, C, K_h, K_w].

``pe_conv2d_stats`` is one library call: the operands are unfolded by a kernel straight into the layout the
contraction reads.  ``conv2d_operands`` gives them as tensors, by torch's unfold and a transpose.
"""
from __future__ import annotations

import torch
import torch.nn.functional as F

from . import binding

__all__ = ["conv2d_operands", "pe_conv2d_stats"]


def conv2d_operands(x: torch.Tensor, grad_out: torch.Tensor, kernel_size, stride=1, padding=0, dilation=1):
    """x: [B, C, H, W] layer input, grad_out: [B, F, H_out, W_out] cotangent of the layer output.
    Returns (X [B, T, C*K_h*K_w], dY [B, T, F]) in bf16, T = H_out * W_out, ready for pe_linear_stats.
    The feature order of X is torch's unfold order (channel-major, then kernel row, then kernel column), i.e.
    the order of weight.view(F, -1)."""
    if x.dim() != 4 or grad_out.dim() != 4 or x.shape[0] != grad_out.shape[0]:
        raise ValueError("x must be [B, C, H, W] and grad_out [B, F, H_out, W_out]")
    cols = F.unfold(x.float(), kernel_size, dilation=dilation, padding=padding, stride=stride)      # [B, C*K*K, T]
    B, Fo = grad_out.shape[:2]
    T = cols.shape[2]
    if grad_out.shape[2] * grad_out.shape[3] != T:
        raise ValueError("grad_out's spatial size does not match the convolution's output size")
    X = cols.transpose(1, 2).contiguous().to(torch.bfloat16)
    dY = grad_out.reshape(B, Fo, T).transpose(1, 2).contiguous().to(torch.bfloat16)
    return X, dY


def _pair(v):
    return (int(v), int(v)) if not isinstance(v, (tuple, list)) else ((int(v[0]), int(v[0])) if len(v) == 1 else (int(v[0]), int(v[1])))


def pe_conv2d_stats(x, grad_out, weight_shape, phi, stride=1, padding=0, dilation=1):
    """sum_b G_b and sum_b phi(G_b) of a conv2d weight [F, C, K_h, K_w]; both returned in the weight's shape."""
    Fo, C, Kh, Kw = weight_shape
    if x.dim() != 4 or grad_out.dim() != 4 or x.shape[0] != grad_out.shape[0]:
        raise ValueError("x must be [B, C, H, W] and grad_out [B, F, H_out, W_out]")
    sizes = [(n + 2 * p - d * (k - 1) - 1) // s + 1
             for n, p, d, k, s in zip(x.shape[2:], _pair(padding), _pair(dilation), (Kh, Kw), _pair(stride))]
    if tuple(x.shape[1:2]) == (C,) and tuple(grad_out.shape[1:]) == (Fo, *sizes) and x.is_cuda and x.device == grad_out.device:
        mean = x.new_empty((Fo, C * Kh * Kw), dtype=torch.float32)
        stat = torch.empty_like(mean)
        # the same rounding as conv2d_operands: unfolding moves values, so it commutes with the conversion
        xb = x if x.dtype == torch.bfloat16 else x.float().to(torch.bfloat16)
        if binding.pe_conv2d_stats(xb.contiguous(), grad_out.to(torch.bfloat16).contiguous(), (Kh, Kw), phi, _pair(stride), _pair(padding),
                                            _pair(dilation), mean, stat):
            return mean.view(Fo, C, Kh, Kw), stat.view(Fo, C, Kh, Kw)
    X, dY = conv2d_operands(x, grad_out, (Kh, Kw), stride, padding, dilation)
    mean, stat = binding.pe_linear_stats(X, dY, phi)
    return mean.view(Fo, C, Kh, Kw), stat.view(Fo, C, Kh, Kw)
