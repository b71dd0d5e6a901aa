"""csrc/extents.h: the sizes and index walks that the kernels and their launches
share, compiled for the host.  No GPU."""
import ctypes
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2608_02474_gb300", "csrc")
WRAP = """
#include "extents.h"
extern "C" {
size_t stage_bytes(int n) { return key_stage_bytes(n); }
int row_blocks(int n, int per) { return blocks_for_rows(n, per); }
// rows that the walk visits from `first` in steps of `step`, up to max of them
int row_walk(unsigned first, unsigned step, int n, int max, unsigned *rows) {
    int k = 0;
    for (RowWalk w{first, step}; w.below(n) && k < max; w.next()) rows[k++] = w.row;
    return k;
}
// pieces (row, piece) that thread t visits, up to max of them
int piece_walk(unsigned t, unsigned threads, unsigned C, int n, int max, unsigned *rows,
               unsigned *pieces) {
    int k = 0;
    for (PieceWalk w(t, threads, C); w.below(n) && k < max; w.next()) {
        rows[k] = w.row;
        pieces[k++] = w.piece;
    }
    return k;
}
}
"""


@pytest.fixture(scope="module")
def ext(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("extents")
    (d / "w.cpp").write_text(WRAP)
    subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-I" + CSRC, str(d / "w.cpp"),
                    "-o", str(d / "w.so")], check=True)
    return ctypes.CDLL(str(d / "w.so"))


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 7799, 7800, 10239, 51197, 51200])
def test_staged_keys_fit(ext, n):
    """The top-K kernels store keys as whole 16-byte groups at every multiple of four
    below n: the last one has to lie inside what the launch asks for."""
    ext.stage_bytes.restype = ctypes.c_size_t
    last_group = (n - 1) // 4
    assert 16 * (last_group + 1) <= ext.stage_bytes(n) < 16 * (last_group + 2)
    # and the launches ask for just that
    src = open(os.path.join(CSRC, "select.cu")).read()
    assert "const size_t key_bytes = key_stage_bytes(NT);" in src
    assert "key_stage_bytes(slice), st, keys" in src


INT32_MAX = 2 ** 31 - 1
GRID = 152 * 32 * 256                               # threads of the widest grid that walks


def _u32s(n):
    return (ctypes.c_uint32 * n)()


@pytest.mark.parametrize("n", [1, 7, 8, 9, 2 ** 30 + 1, INT32_MAX - 8, INT32_MAX])
@pytest.mark.parametrize("per", [1, 8])
def test_blocks_cover_the_rows(ext, n, per):
    b = ext.row_blocks(n, per)
    assert b * per >= n > (b - 1) * per


@pytest.mark.parametrize("n", [1, 8, 2 ** 30 + 1, INT32_MAX - 1, INT32_MAX])
@pytest.mark.parametrize("capped", [True, False])
def test_row_walk_ends_at_the_last_row(ext, n, capped):
    """With one row per warp the step is as large as the row count, and the row after
    the last one lies beyond INT32_MAX: it must not come back as a negative row."""
    blocks = ext.row_blocks(n, 8)
    if capped:
        blocks = min(blocks, 152 * 8)
    step = blocks * 8
    rows = _u32s(1 << 19)
    for first in {0, 1, 7, step - 8, step - 1}:
        k = ext.row_walk(first, step, n, len(rows), rows)
        want = range(first, n, step)
        assert k == len(want)
        assert k == 0 or (rows[0], rows[k - 1]) == (first, want[-1])


@pytest.mark.parametrize("n,C,threads", [
    (5, 3, 256), (1000, 64, 512), (300, 320, GRID), (INT32_MAX, 1, GRID), (INT32_MAX - 1, 1, GRID),
    (INT32_MAX, 3, GRID), (2 ** 30, 2, GRID),
])
def test_piece_walk_is_the_division(ext, n, C, threads):
    """Every thread's pieces are those that dividing its running index by the pieces of
    a row gives, to the last row a call accepts."""
    rows, pieces = _u32s(1 << 13), _u32s(1 << 13)
    for t in {0, 1, C - 1, C, threads // 2, threads - 1}:
        want = range(t, n * C, threads)
        k = ext.piece_walk(t, threads, C, n, len(rows), rows, pieces)
        assert k == len(want)
        for j in {0, 1, k // 2, k - 2, k - 1} & set(range(k)):
            assert (rows[j], pieces[j]) == divmod(want[j], C)
