"""The staged per-token statistic of large layers: squares scaled by the maxima of 512-row chunks, unscaled chunk by chunk."""
import numpy as np
import pytest
import torch

import paper_2510_00236_b200 as pe

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# rows a multiple of the chunk, one short and one past it, widths beyond a 64-column group and a 256-column tile; columns whose
# magnitudes differ by 2^40, rows whose magnitudes differ by 2^12 (chunks get different scales), zero columns and zero chunks
@pytest.mark.parametrize("B,T,d_in,d_out", [(25, 512, 4096, 3800), (1, 16383, 1032, 5128), (7, 1829, 4104, 4096), (31, 413, 72, 8000)])
def test_chunked_staging_against_fp64(B, T, d_in, d_out):
    if B * T * (d_in + d_out) < 1e8:       # the last shape: one more factor of rows
        B *= 1 + int(1e8 / (B * T * (d_in + d_out)))
    need, rows = pe.pe_token_sqstats_staged_workspace_bytes(B, T, d_in, d_out), B * T
    assert need > (d_in + d_out) * (4 + 2 * rows) + 1024, "the layer must be large enough for the one-pass staging"
    g = torch.Generator(device=DEV).manual_seed(B + T)
    X = torch.randn((rows, d_in), generator=g, device=DEV) * torch.exp2(torch.randint(-20, 21, (d_in,), generator=g, device=DEV).float())
    dY = torch.randn((rows, d_out), generator=g, device=DEV) * torch.exp2(torch.randint(-6, 7, (rows, 1), generator=g, device=DEV).float())
    X[:, 3] = 0
    dY[512:1024] = 0
    X, dY = X.to(torch.bfloat16).view(B, T, d_in), dY.to(torch.bfloat16).view(B, T, d_out)
    out = torch.full((d_out, d_in), float("nan"), device=DEV)
    pe.pe_token_sqstats_staged(X, dY, out, torch.empty(need, dtype=torch.uint8, device=DEV))
    two_pass = torch.full((d_out, d_in), float("nan"), device=DEV)      # a workspace without room for the chunks' scales
    pe.pe_token_sqstats_staged(X, dY, two_pass, torch.empty((d_in + d_out) * (4 + 2 * rows) + 1024, dtype=torch.uint8, device=DEV))
    assert pe.pe_get_async_status(DEV) == (0, 0)
    rng = np.random.default_rng(B)
    o = torch.as_tensor(np.unique(np.concatenate([[0, 63, 64, 255, 256, d_out - 1], rng.integers(0, d_out, 60)])), device=DEV)
    i = torch.as_tensor(np.unique(np.concatenate([[0, 3, 63, 64, d_in - 1], rng.integers(0, d_in, 60)])), device=DEV)
    want = (dY.reshape(rows, -1)[:, o].double() ** 2).T @ (X.reshape(rows, -1)[:, i].double() ** 2)
    # two squares rounded to 11 bits, nearest even: at most 2 * 2^-11 per term, all terms non-negative, so per entry too
    for got in (out, two_pass):
        got = got[o][:, i].double()
        assert torch.isfinite(got).all()
        assert torch.all((got - want).abs() <= 2.0 ** -10 * 1.01 * want), float(((got - want).abs() / want.clamp_min(1e-300)).max())
    assert torch.all(out[:, 3] == 0)
