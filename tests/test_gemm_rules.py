"""How the contractions are cut along k (csrc/gemm_rules.h), compiled for the host."""
import ctypes
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2304_07006_gb300", "csrc")
SRC = """
#include "gemm_rules.h"
extern "C" int splits64(int m, int n, int r, int sm) { return xtc::gemm64_splits(m, n, r, sm); }
extern "C" int chains(int n, int tiles, int slots, int* q) { return xtc::chain_slices(n, 128, 32, 32, tiles, slots, q); }
"""
# (orbitals, grid points) of tests/test_gpu_chain_slices_cut.py and the slices of step (d) on 76 pairs of SMs
CUT = [(12, 4096, 2), (12, 4736, 3), (5, 13_000, 7), (23, 6000, 3)]


def step_d(n_orb, n_grid):
    """(ranges, tiles) of step (d): 4 values a point in ranges of 64, pairs of 128-row tiles x 128-column tiles."""
    rows = -(-(n_orb * (n_orb + 1) // 2) // 128)
    return 4 * (-(-n_grid // 128) * 128) // 64, (rows + 1) // 2 * rows



@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("rules")
    (d / "rules.cpp").write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "rules.so"), str(d / "rules.cpp")],
                   check=True)
    return ctypes.CDLL(str(d / "rules.so"))


@pytest.mark.parametrize("m_tiles,n_tiles", [(1, 1), (8, 20), (200, 1), (24000, 1), (313, 629)])
@pytest.mark.parametrize("n_ranges", [1, 7, 8, 625, 3200, 3201, 6400, 8192, 8193, 100_000])
def test_digit_sums_stay_inside_64_bits(rules, m_tiles, n_tiles, n_ranges):
    s = rules.splits64(m_tiles, n_tiles, n_ranges, 152)
    per = -(-n_ranges // s)
    assert s >= 1 and (s - 1) * per < n_ranges        # no empty slice
    # every digit at its largest, 2^8, and of one sign: diagonal d of a range is (d + 1) 64 2^16
    for diagonals in (range(0, 4), range(4, 8)):
        assert per * sum((d + 1) * 64 * 2**16 * 2**(27 - 9 * (d % 4)) for d in diagonals) < 2**63


@pytest.mark.parametrize("n_orb,n_grid,want", CUT + [(12, 2560, 1), (12, 2688, 1), (5, 4100, 1), (12, 4608, 1)])
def test_slices_of_the_sizes_under_test(rules, n_orb, n_grid, want):
    q = ctypes.c_int(0)
    assert rules.chains(*step_d(n_orb, n_grid), 76, ctypes.byref(q)) == want


@pytest.mark.parametrize("tiles", [1, 2, 10, 76, 77, 153, 400])
def test_slices_hold_whole_chains(rules, tiles):
    """Every slice but the first starts at a flush, and the last holds a flush of every column's chain (32 ranges) and more."""
    for n in range(1, 1400):
        q = ctypes.c_int(0)
        z = rules.chains(n, tiles, 76, ctypes.byref(q))
        if z > 1:
            step = 128 * q.value
            assert step >= 128 and z <= 16 and (z - 1) * step + 32 < n <= z * step
