"""Packed batches one after the other on one workspace: a batch of whole 16-token groups, whose contraction reads nothing of the side
buffer, between batches that do."""
import pytest
import torch

import paper_2510_00236_b200 as pe

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _batch(lens, d_in, d_out, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    offs = torch.tensor([0] + lens, dtype=torch.int32).cumsum(0).to(torch.int32)
    X = torch.randn((int(offs[-1]), d_in), generator=g, device=DEV).bfloat16()
    dY = torch.randn((int(offs[-1]), d_out), generator=g, device=DEV).bfloat16()
    x, y = X.double(), dY.double()
    G = [y[a:b].T @ x[a:b] for a, b in zip(offs[:-1].tolist(), offs[1:].tolist())]
    mag = y.abs().T @ x.abs()
    return X, dY, offs.to(DEV), sum(G), sum(g * g for g in G), mag, torch.stack([(g * g).sum() for g in G])


# 75 and 2 tiles of 256 x 192: an unsplit batch and one in slices
@pytest.mark.parametrize("d_in,d_out", [(576, 6400), (200, 512)])
def test_batches_sharing_a_workspace(d_in, d_out):
    whole, tails = [16, 48, 32, 160], [17, 5, 33, 170]
    batches = [_batch(lens, d_in, d_out, k) for k, lens in enumerate((whole, tails))]
    workspace = torch.empty(pe.pe_linear_stats_ragged_workspace_bytes(4, d_in, d_out), dtype=torch.uint8, device=DEV)
    got = []
    for k in range(20):
        X, dY, offs = batches[k % 2][:3]
        got.append((pe.pe_linear_stats_ragged(X, dY, offs, "square", workspace=workspace),
                    pe.pe_example_sqnorms_ragged(X, dY, offs, workspace=workspace)))
    assert pe.pe_get_async_status(DEV) == (0, 0)
    eps = (170 + 4) * 2.0 ** -23             # products exact in fp32, sums of at most 170 tokens and 4 examples in fp32, truncated
    for k, ((mean, square), norms) in enumerate(got):
        _, _, _, want_mean, want_square, mag, want_norms = batches[k % 2]
        assert torch.all((mean.double() - want_mean).abs() <= eps * mag)
        assert torch.all((square.double() - want_square).abs() <= 3 * eps * mag * mag)
        assert torch.allclose(norms.double(), want_norms, rtol=1e-5, atol=0)
