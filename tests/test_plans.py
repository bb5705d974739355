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
