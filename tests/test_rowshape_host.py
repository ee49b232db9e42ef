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
void shape(int32_t m, int32_t nnz, int32_t val_bytes, int32_t *out)
{
    const RowShape s = row_shape(m, nnz, val_bytes);
    const RowUnits u = row_units(m, nnz, s);
    out[0] = s.gs;
    out[1] = s.us;
    out[2] = s.cap;
    out[3] = s.piece;
    out[4] = u.nbig;
    out[5] = u.nunits;
}
int64_t lists(int32_t m, int32_t nnz, int32_t val_bytes)
{
    const RowShape s = row_shape(m, nnz, val_bytes);
    return (int64_t)row_lists(nnz, s.cap, s.piece).bytes;
}
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


def _shape(lib, m, nnz, val_bytes):
    out = (ctypes.c_int32 * 6)()
    lib.shape(m, nnz, val_bytes, out)
    return dict(zip(("gs", "us", "cap", "piece", "nbig", "nunits"), out))


def test_the_gpu_cases_take_the_shapes_they_are_for(lib):
    from test_gpu_rowblock import LANES
    for kind, m, lanes in LANES:
        nnz = m * int(kind[5:]) if kind.startswith("const") else m * int(kind[4:]) // 2
        for val_bytes in (8, 4, 2):
            s = _shape(lib, m, nnz, val_bytes)
            assert (1 << s["gs"], s["us"]) == (lanes, 2), (kind, val_bytes, s)
            assert 0 < s["nbig"] < s["nunits"]


def test_units_cover_the_rows(lib):
    for m in (1, 31, 32, 33, 127, 9001, 400_003, 2_000_000_011, MAX_DIM):
        for mean in (0, 1, 10, 28, 60, 440):
            nnz = min(m * mean, MAX_DIM)
            for val_bytes in (8, 4, 2):
                s = _shape(lib, m, nnz, val_bytes)
                rows = 32 >> s["gs"]
                single = s["nunits"] - s["nbig"]
                covered = s["nbig"] * (rows << s["us"]) + single * rows
                assert 0 <= covered - m < rows, (m, mean, s)
                assert s["cap"] % 8 == 0


def test_short_rows_are_few_units(lib):
    # (a unit costs some 2 us of a warp's time however little it holds)
    for m, mean, most in ((20_000_000, 1, 161_000), (20_000_000, 3, 161_000),
                          (20_000_000, 20, 185_000), (2_000_000, 1, 20_500)):
        s = _shape(lib, m, m * mean, 8)
        assert s["us"] == 2 and s["nunits"] <= most, (m, mean, s)


def test_the_lists_fit_every_workspace(lib):
    # (the header takes the first 256 bytes; with less room a product would go by
    # tiles, see takes_rows)
    import random
    from paper_1504_06474_gb300 import _build
    from paper_1504_06474_gb300 import ssspmv as C
    _build.build()
    lib.lists.restype = ctypes.c_int64
    rng = random.Random(2)
    for i in range(30_000):
        m = int(2 ** rng.uniform(0, 31)) - 1
        nnz = int(2 ** rng.uniform(0, 31)) - 1
        if i < 3000:  # around the step in the pieces' length
            nnz = 15_000_000 + rng.randint(-2000, 800_000)
        m, nnz = min(max(m, 1), MAX_DIM), min(max(nnz, 1), MAX_DIM)
        vb = rng.choice((8, 4, 2))
        assert lib.lists(m, nnz, vb) <= C.ssspmv_workspace_bytes(m, nnz, vb, None) - 256, (m, nnz, vb)
