"""How launches divide their work, through the library's host-side query (no GPU)."""
import pytest

import paper_2510_00236_b200 as pe
from paper_2510_00236_b200 import build as pe_build

SMS = 148
MEAN, SQUARE, SIGN = 1, 2, 4


@pytest.fixture(scope="module", autouse=True)
def lib():
    pe_build.build_library()
    return pe.load_library()


# 128, 100, 64, 128, 512 and 2 tiles
@pytest.mark.parametrize("d_in,d_out", [(2048, 2048), (1600, 2048), (1024, 2048), (1024, 4096), (4096, 4096), (128, 512)])
def test_sign_counts_of_short_sequences_fit_16_bits(d_in, d_out):
    for B in [32766, 32767, 32768, 33000, 40000, 65534, 65535, 66000, 70000, 100000, 131072, 140000, 1 << 20]:
        whole, slices, longest = pe.pe_plan_query(pe.PLAN_SHORT, MEAN | SQUARE | SIGN, B, 2, d_in, d_out, SMS)
        assert longest == (B if whole else -(-B // slices))
        assert longest <= 32767


# the tiles of 128 x 64 (32 slices), 64 x 64 by 256 threads (16) and 128 x 64 (32) are what these layers take among the other four tiles: roundings of a
# sum over the batch are a slice's examples, the slices of a cluster of eight, the clusters
@pytest.mark.parametrize("B,T,d_in,d_out,others", [(60, 24, 900, 300, 32), (37, 187, 356, 126, 16), (49, 37, 948, 328, 32)])
def test_smaller_blocks_do_not_lengthen_fp32_sums(B, T, d_in, d_out, others):
    tile, slices, cluster = pe.pe_plan_query(pe.PLAN_SIMT_STATS, MEAN, B, T, d_in, d_out, SMS)
    chain = lambda s: -(-B // s) + min(s, 8) + -(-s // 8)        # noqa: E731
    assert tile == 4 and cluster == min(slices, 8)
    assert chain(slices) <= chain(others)
