"""The index arithmetic of the row blocks (csrc/rowshape.h) on the CPU, compiled
as plain C++: pieces of rows and their ends where 32 bits are nearly used up,
against Python's unbounded integers."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1504_06474_gb300", "csrc")
MAX_DIM = 2**31 - 1 - 256  # SSSPMV_MAX_DIM

SOURCE = """
#include "rowshape.h"
using namespace ssspmv;
extern "C" {
int32_t pieces(int32_t len, int32_t pl) { return row_pieces(len, pl); }
int32_t end_of(int32_t s, int32_t e, int32_t pl) { return piece_end(s, e, pl); }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("rowshape")
    src, out = d / "w.cpp", d / "w.so"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-fwrapv", "-shared", "-fPIC",
                    "-I", CSRC, str(src), "-o", str(out)], check=True)
    return ctypes.CDLL(str(out))


@pytest.mark.parametrize("pl", [10, 11])
@pytest.mark.parametrize("nnz", [100_000, 2_147_481_599, 2_147_481_600, 2_147_483_000, MAX_DIM])
def test_pieces_cover_a_row_that_ends_the_arrays(lib, pl, nnz):
    P = 1 << pl
    for n in (1, 5, P - 1, P, P + 1, 3 * P, 3 * P + 5, 6149, nnz):
        s = nnz - n
        count = lib.pieces(n, pl)
        assert count == -(-n // P)
        ks = range(count) if count < 100 else (0, 1, count // 2, count - 2, count - 1)
        for k in ks:
            at = s + k * P
            assert lib.end_of(at, nnz, pl) == min(at + P, nnz), (n, k)


@pytest.mark.parametrize("pl", [10, 11])
def test_no_entries_no_pieces(lib, pl):
    # (an invalid row_ptr's row may have a negative length)
    for n in (0, -1, -2048, -(2**31) + 1):
        assert lib.pieces(n, pl) == 0
    assert lib.end_of(MAX_DIM, MAX_DIM, pl) == MAX_DIM
