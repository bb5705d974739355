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


# norms, clipped sums, packed batches and the update in one launch on the same tile: bf16 rows of whole groups of four and of odd length
@pytest.mark.parametrize("B,T,d_in,d_out", [(10, 200, 800, 400), (64, 32, 500, 300), (20, 185, 406, 881)])
def test_other_entry_points_against_fp64(B, T, d_in, d_out):
    assert {pe.pe_plan_query(what, 0, B, T, d_in, d_out, 148)[0] for what in (pe.PLAN_SIMT_STATS, pe.PLAN_SIMT_NORMS)} == {4}
    g = torch.Generator(device=DEV).manual_seed(B + T)
    X = torch.randn((B, T, d_in), generator=g, device=DEV).bfloat16()
    dY = (torch.randn((B, T, d_out), generator=g, device=DEV) * T ** -0.5).bfloat16()
    theta = torch.randn((d_out, d_in), generator=g, device=DEV)
    adam, m, v = theta.clone(), torch.zeros_like(theta), torch.zeros_like(theta)
    lens = torch.randint(0, T + 1, (B,), generator=torch.Generator().manual_seed(B))
    offs = torch.cat([torch.zeros(1, dtype=torch.long), lens.cumsum(0)]).int()
    Xp, Yp = (torch.cat([t[b, :n] for b, n in enumerate(lens.tolist())]).contiguous() for t in (X, dY))
    mean_p, square_p, mean, square = (torch.full((d_out, d_in), float("nan"), device=DEV) for _ in range(4))
    prev, prev_fused = pe.pe_set_path(pe.PATH_SIMT), pe.pe_set_fused_update(pe.FUSED_ALWAYS)
    try:
        norms = pe.pe_example_sqnorms(X, dY)
        clip = float(norms.median().sqrt())
        total, _ = pe.pe_linear_clipped_sum(X, dY, clip, norms)
        pe.pe_linear_stats_ragged(Xp, Yp, offs.to(DEV), "square", mean_p, square_p)
        pe.pe_linear_microadam_step(X, dY, adam, m, v, step=1, lr=1e-3, beta1=0.9, beta2=0.999, eps=1e-8, out_mean=mean, out_stat=square)
        torch.cuda.synchronize()
    finally:
        pe.pe_set_path(prev), pe.pe_set_fused_update(prev_fused)
    y, x = dY.double(), X.double()
    G, mag = torch.einsum("bto,bti->boi", y, x), torch.einsum("bto,bti->boi", y.abs(), x.abs())
    # sums of T products and of B terms, a rounding each
    eps = (T + B + 2) * 2.0 ** -24
    N = G.square().sum((1, 2))
    assert torch.allclose(norms.double(), N, rtol=2e-5)          # squares of sums of T products, and fp32 sums of all of them
    c = (clip / N.sqrt()).clamp(max=1)[:, None, None]
    assert torch.all((total.double() - (c * G).sum(0)).abs() <= (eps + 2e-5) * mag.sum(0))
    keep = (torch.arange(T)[None, :] < lens[:, None]).to(DEV).double()[:, :, None]
    Gp, magp = torch.einsum("bto,bti->boi", y * keep, x), torch.einsum("bto,bti->boi", y.abs() * keep, x.abs())
    for a, b, GG, mm in ((mean_p, square_p, Gp, magp), (mean, square, G, mag)):
        assert torch.all((a.double() - GG.sum(0)).abs() <= eps * mm.sum(0))
        assert torch.all((b.double() - GG.square().sum(0)).abs() <= 3 * eps * mm.square().sum(0))
    # the first step from zero moments: their bias corrections undo 1 - beta, which fp32 rounds by 2^-24 / 1e-3 = 6e-5 for v
    mu, nu = mean.double() / B, square.double() / B
    assert torch.allclose(m.double(), 0.1 * mu, rtol=1e-5) and torch.allclose(v.double(), 1e-3 * nu, rtol=2e-4)
    assert torch.all((adam.double() - theta.double() + 1e-3 * mu / (nu.sqrt() + 1e-8)).abs() <= 2e-4 * 1e-3 + 2.0 ** -23 * theta.double().abs())
