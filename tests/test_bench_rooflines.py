"""The work behind the roofline fractions of bench.py is what the kernels execute."""
import os
import re
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402

CSRC = os.path.join(ROOT, "paper_2509_07974_gb300", "csrc")


def _source(name):
    return open(os.path.join(CSRC, name)).read()


def test_sector_sums_are_counted_as_the_kernel_has_them():
    """Seven weights times K polynomials, K by the same line of powers as the launcher."""
    src = _source("gather_sector.cu")
    line, k0, k1 = map(int, re.search(r"const int K = L\.max_pow <= (\d+) \? (\d+) : (\d+);", src).groups())
    assert re.search(r"kMomRows = 7 \* K \+ 12;", src)
    for nmax in (7, 20, 21, 40):
        K = k0 if 2 * nmax + 6 <= line else k1
        assert bench.sector_flop_per_pair(nmax) == 7 + 18 * (K - 1) + 50
    # a fraction of one or more of the pipe would mean counting work that is not done
    assert bench.sector_flop_per_pair(20) < 0.15 * bench.gather_flop_per_pair(20)


@pytest.mark.parametrize("share,flop", [(0.0, 2160), (1.0, 255), (0.5, (2160 + 255) / 2)])
def test_gather_fraction_follows_the_kernel_that_took_the_centres(share, flop):
    r = bench.gather_roofline(1e9, 20, share, 4, 100.0, 80.0)
    assert r["achieved"] == pytest.approx(flop * 1e9 / 0.1 / 1e12) and r["frac"] == pytest.approx(r["achieved"] / 80.0)
    assert r["algorithmic_flop_per_pair"] == 2160 and r["ms_per_launch"] == 25.0


def test_split_fp16_contraction_counts_its_mmas():
    """2839 + 861 rows and 1655 tiles of 128 at n_max = 20, 10 bins; 80 columns of the four families' real and
    imaginary parts, 32 (20 and padding) for FW, three products of 128 real terms per 64 centres."""
    x, w = bench.basis_rows(20)
    assert sum(x) == 2839 and sum(w) == 861
    tiles = [sum(-(-n * 55 // 128) for n in k) for k in (x, w)]
    assert sum(tiles) == 1655
    assert bench.h16_mma_flop(64, 20, 10) == 3 * 2 * 128 * 128 * (tiles[0] * 80 + tiles[1] * 32)
    useful = 8 * (2839 * 4 + 861) * 55 * 10  # complex multiply-adds of the independent sums per centre
    assert 3 * useful < bench.h16_mma_flop(1, 20, 10) < 1.25 * 3 * useful
    assert bench.issued_flop("f16x3", 64, 20, 10) == bench.h16_mma_flop(64, 20, 10)
    assert bench.issued_flop("3xtf32", 1, 20, 10) == 3 * bench.reduced_contraction_flop(1, 20, 10)
    assert bench.h16_mma_flop(64, 2, 16) > 0 and bench.h16_mma_flop(64, 2, 1) > 0


def test_kernels_of_the_bench_line_have_a_traffic_figure_of_their_source():
    names = re.findall(r'measured_traffic\("(\w+)"', open(os.path.join(ROOT, "bench.py")).read())
    assert "gather_sector_kernel" in names and "contract_h16_kernel" in names
    for name in names + ["contract_tc_kernel"]:
        assert any(re.search(r"__global__[^;{]*\b%s\b" % name, _source(f)) for f in os.listdir(CSRC)), name
        assert bench.measured_traffic(name) is not None, name
