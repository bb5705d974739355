"""How launches divide their work, through the library's host-side query (no GPU)."""
import time

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
        whole, slices, longest, _ = pe.pe_plan_query(pe.PLAN_SHORT, MEAN | SQUARE | SIGN, B, 2, d_in, d_out, SMS)
        assert longest == (B if whole else -(-B // slices))
        assert longest <= 32767


# what a pair per tile and slice would have taken: five slices of 91 or 133 tiles, two of 99, and so on
@pytest.mark.parametrize("outputs,B,T,d_in,d_out,most", [
    (MEAN | SQUARE, 2021, 24, 2336, 1728, 405), (MEAN | SIGN, 2021, 24, 2336, 1728, 405), (MEAN | SQUARE | SIGN, 1545, 4, 1624, 2296, 309),
    (MEAN | SQUARE, 1854, 6, 2616, 1368, 464), (MEAN | SQUARE | SIGN, 285, 2, 832, 3888, 95), (MEAN | SQUARE | SIGN, 1858, 20, 1864, 2208, 310)])
def test_sums_of_short_sequences_are_not_lengthened(outputs, B, T, d_in, d_out, most):
    assert pe.pe_plan_query(pe.PLAN_SHORT, outputs, B, T, d_in, d_out, SMS)[2] <= most


# error variances up to a factor (examples in order, or runs and their sums, and the slices) against the slices of a pair per 256 x 256 tile and slice
@pytest.mark.parametrize("B,T,d_in,d_out,slices", [(1395, 5, 1696, 1336, 7), (665, 16, 832, 2528, 5), (1010, 6, 528, 3304, 5), (800, 32, 1024, 4096, 0), (28, 32, 1024, 1024, 4)])
def test_runs_of_the_square_alone(B, T, d_in, d_out, slices):
    whole, split, longest, run = pe.pe_plan_query(pe.PLAN_SHORT, SQUARE, B, T, d_in, d_out, SMS)
    variance = lambda p, r, parts: (r * r + p * p / r if r < p else p * p) + B * parts        # noqa: E731
    assert run in (16, 32, 64, 128, 256)
    p = -(-B // max(1, slices))
    assert variance(longest, run, 0 if whole or split == 1 else split) <= variance(p, p, slices)


# the tiles of 128 x 64 (32 slices), 64 x 64 by 256 threads (16) and 128 x 64 (32) are what these layers take among the other four tiles: roundings of a
# sum over the batch are a slice's examples, the slices of a cluster of eight, the clusters
@pytest.mark.parametrize("B,T,d_in,d_out,others", [(60, 24, 900, 300, 32), (37, 187, 356, 126, 16), (49, 37, 948, 328, 32)])
def test_smaller_blocks_do_not_lengthen_fp32_sums(B, T, d_in, d_out, others):
    tile, slices, cluster, _ = pe.pe_plan_query(pe.PLAN_SIMT_STATS, MEAN, B, T, d_in, d_out, SMS)
    chain = lambda s: -(-B // s) + min(s, 8) + -(-s // 8)        # noqa: E731
    assert tile == 4 and cluster == min(slices, 8)
    assert chain(slices) <= chain(others)


def test_sums_of_signs_alone_are_exact_in_any_number_of_slices():
    assert pe.pe_plan_query(pe.PLAN_SIMT_STATS, SIGN, 60, 24, 900, 300, SMS)[:2] == (4, 4)


def _parts(rows, d_in, d_out):
    """Per tile of the per-token statistic the chunks that each pair takes, by the plan."""
    chunks, tiles, slots = -(-rows // 32), -(-d_in // 256) * -(-d_out // 256), SMS // 2
    slices, deal_tiles, deal_pairs, pairs = pe.pe_plan_query(pe.PLAN_TOKEN, 0, 1, rows, d_in, d_out, SMS)
    if not deal_tiles:
        return slices, [[chunks * (z + 1) // slices - chunks * z // slices for z in range(slices)] for _ in range(tiles)]
    parts = [[] for _ in range(tiles)]
    assert deal_tiles <= deal_pairs and pairs <= slots
    for pair in range(pairs):
        group, i = divmod(pair, deal_pairs)
        in_group, n = min(deal_tiles, tiles - group * deal_tiles), min(deal_pairs, pairs - group * deal_pairs)
        first, last = chunks * in_group * i // n, chunks * in_group * (i + 1) // n
        assert first < last <= first // chunks * chunks + 2 * chunks            # one or two tiles to a pair
        for tile in range(first // chunks, -(-last // chunks)):
            parts[group * deal_tiles + tile].append(min(last, (tile + 1) * chunks) - max(first, tile * chunks))
    return slices, parts


def test_rows_of_the_per_token_statistic_dealt_out():
    dealt = 0
    for rows in (33, 64, 100, 1000, 2000, 4127, 16384, 100000):
        for d_in in (8, 256, 512, 776, 1024, 2304):
            for d_out in (8, 520, 1280, 2048, 3000, 4864, 8192):
                slices, parts = _parts(rows, d_in, d_out)
                dealt += any(len(p) != slices for p in parts)
                for p in parts:
                    assert sum(p) == -(-rows // 32) and min(p) > 0
                    # whole tiles and tiles in two parts repeat bit for bit, and they do so wherever whole slices would
                    assert len(p) <= 2 or slices > 2
    assert dealt > 20


# operands that L2 holds, or one small operand beside a large one that no two tiles share; 522, 338 and 134 MB that several tiles share
@pytest.mark.parametrize("rows,d_in,d_out,dealt", [(16384, 1280, 2560, True), (16384, 512, 2048, True), (60000, 256, 6656, True), (60000, 2048, 2304, False), (60000, 1024, 2560, False),
                                                   (16384, 2048, 2048, False)])
def test_rows_are_dealt_out_where_they_stay_in_l2(rows, d_in, d_out, dealt):
    assert (pe.pe_plan_query(pe.PLAN_TOKEN, 0, 1, rows, d_in, d_out, SMS)[1] > 0) == dealt


def test_the_plan_of_example_norms_takes_no_time():
    # 128 and 16 tiles; slices of the whole batch
    start = time.perf_counter()
    for _ in range(50):
        for d_in, d_out in ((2048, 4096), (512, 2048)):
            for B in (1 << 20, 1 << 24):
                slices, examples, order, _ = pe.pe_plan_query(pe.PLAN_NORMS, 0, B, 4, d_in, d_out, SMS)
                assert not examples or slices == -(-B // examples)
    assert time.perf_counter() - start < 1.0                  # one search through all lengths of slices took 5 ms at B = 2^20
    # the tile order, whose search is kept per layer and slices, is not searched anew for another batch
    for B in range(100, 300):
        slices, examples, order, _ = pe.pe_plan_query(pe.PLAN_NORMS, 0, B, 512, 2048, 4096, SMS)
        assert order == (1 if examples else slices)
