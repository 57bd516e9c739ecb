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
"""


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
