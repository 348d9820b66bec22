"""CPU tests of the row-cost arithmetic (csrc/row_cost.cuh, plain C++ compiled
here): over every mesh the library accepts (up to 2^24 elements), the 32-bit
prefix sums of the rows' costs stay below 2^31, and the bound on the rows of a
CTA's range, which sizes its shared tables, is positive and holds."""
import ctypes
import shutil
import subprocess
from pathlib import Path

import numpy as np
import pytest

CSRC = Path(__file__).resolve().parents[1] / "paper_0704_2344_gb300" / "csrc"
SRC = """
#include "row_cost.cuh"
extern "C" {
int row_cost(int re, int im, int diag) { return fe::row_cost(re, im, diag != 0); }
int max_cost() { return fe::kMaxRowCost; }
int shift(long long rows) { return fe::cost_shift(rows); }
int scaled(int c, int s) { return fe::scaled_cost(c, s); }
long long rows_bound(long long n, long long total, int n_cta, int lo, int hi) {
    return fe::cta_rows_bound(n, total, n_cta, lo, hi);
}
}
"""


@pytest.fixture(scope="module")
def rc(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("row_cost")
    (d / "rc.cpp").write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-I", str(CSRC), str(d / "rc.cpp"), "-o",
                    str(d / "rc.so")], check=True)
    lib = ctypes.CDLL(str(d / "rc.so"))
    lib.shift.argtypes = [ctypes.c_longlong]
    lib.rows_bound.argtypes = [ctypes.c_longlong, ctypes.c_longlong] + [ctypes.c_int] * 3
    lib.rows_bound.restype = ctypes.c_longlong
    return lib


def test_largest_row_cost(rc):
    assert max(rc.row_cost(81, 81, 0), rc.row_cost(27, 0, 1)) == rc.max_cost()


# rows of the largest grids: a bar, a plate and a cube of 2^24 elements, a lossy checkerboard's size, small ones
@pytest.mark.parametrize("rows", [1, 8, 29666, 12_000_000, 257 ** 3, 4097 * 4097 * 2, 4 * (2 ** 24 + 1)])
def test_prefix_sums_fit_32_bits(rc, rows):
    s = rc.shift(rows)
    for cost in (9, 30, 110, 134, 150, 170):
        assert 1 <= rc.scaled(cost, s) and rows * rc.scaled(cost, s) < 2 ** 31
    if rows <= 12_000_000:
        assert s == 0


@pytest.mark.parametrize("rows,n_cta", [(257 ** 3, 152), (257 ** 3, 1), (4 * (2 ** 24 + 1), 114), (2197, 152), (5, 3)])
@pytest.mark.parametrize("cost", [30, 150, 170])
def test_rows_bound_of_equal_rows(rc, rows, n_cta, cost):
    c = rc.scaled(cost, rc.shift(rows))
    bound = rc.rows_bound(rows, rows * c, n_cta, c, c)
    assert -(-rows // n_cta) <= bound <= rows


@pytest.mark.parametrize("seed", range(20))
def test_rows_bound_holds_for_the_split(rc, seed):
    """Rows of random costs split as the solve splits them: no range is longer than the bound."""
    rng = np.random.default_rng(seed)
    n, n_cta = int(rng.integers(1, 5000)), int(rng.integers(1, 152))
    shift = int(rng.integers(0, 4))
    cost = np.array([rc.scaled(int(c), shift) for c in rng.integers(9, 171, n)])
    prefix = np.concatenate([[0], np.cumsum(cost)])
    total = int(prefix[-1])
    cut = [int(np.searchsorted(prefix, k * total // n_cta)) for k in range(n_cta)] + [n]
    bound = rc.rows_bound(n, total, n_cta, int(cost.min()), int(cost.max()))
    assert np.diff(cut).max() <= bound <= n
