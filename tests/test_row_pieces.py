"""Which columns the pieces of a decode to rows that start anywhere hold (csrc/row_pieces.h), compiled for the host: no GPU is
needed, and the column counts go up to the largest that a blob can have."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_00922_b200", "csrc")
# A warp's stores to row g of a row group (half = 0) or row g + 8, in the kernel's order: chunks kc0 .. kc1 - 1 as one run, four
# lanes a block, what is left over.  off: row g's.
HARNESS = r"""
#include "row_pieces.h"
using namespace huffllm;
extern "C" int64_t row_stores(uint64_t cols, uint32_t chunk_cols, uint32_t kc0, uint32_t kc1, uint32_t off, uint32_t half, int64_t *col, int32_t *n, int32_t *lane) {
    int64_t count = 0;
    const int32_t by = half ? row_half(off, cols) : 0;
    auto store = [&](uint32_t t, int64_t block, int32_t c, int32_t first, int32_t end) {
        const PieceCut cut = piece_cut(c, first, end);
        if (cut.lo < cut.hi) { col[count] = block + c + cut.lo; lane[count] = t; n[count++] = cut.hi - cut.lo; }
    };
    bool opens = true;
    for (uint32_t kc = kc0; kc < kc1; ++kc) {
        const uint32_t at = kc * chunk_cols;
        int32_t left = columns_left(cols, at);
        for (int32_t kb = 0; kb < (int32_t)chunk_cols / 32 && left > 0; ++kb, left -= 32, opens = false)
            for (uint32_t t = 0; t < 4; ++t) {
                const int32_t c = piece_column(t, off) + by;
                if (!opens && left >= 32) store(t, (int64_t)at + kb * 32, c, c, c + 8);
                else store(t, (int64_t)at + kb * 32, c, run_start(opens), left);
            }
    }
    const uint32_t at = (kc1 - 1) * chunk_cols;
    const int32_t left = columns_left(cols, at), end = left < (int32_t)chunk_cols ? left : (int32_t)chunk_cols, block = (end + 31) & ~31;
    for (uint32_t t = 0; t < 4; ++t)
        if (piece_column(t, off - by) < 0) store(t, (int64_t)at + block, piece_column(t, off - by), run_start(false), end - block);
    return count;
}
"""


@pytest.fixture(scope="module")
def row_stores(tmp_path_factory):
    d = tmp_path_factory.mktemp("row_pieces")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-ftrapv", "-shared", "-fPIC", "-I" + CSRC, "-o", str(d / "h.so"), str(d / "h.cpp")])
    f = ctypes.CDLL(str(d / "h.so")).row_stores
    f.restype = ctypes.c_int64
    f.argtypes = [ctypes.c_uint64] + [ctypes.c_uint32] * 5 + [ctypes.c_void_p] * 3

    def call(cols, chunk_cols, kc0, kc1, off, half):
        col, n, lane = np.zeros(4096, np.int64), np.zeros(4096, np.int32), np.zeros(4096, np.int32)
        k = f(cols, chunk_cols, kc0, kc1, off, half, col.ctypes.data, n.ctypes.data, lane.ctypes.data)
        return col[:k], n[:k], lane[:k]
    return call


@pytest.mark.parametrize("cols", [65, 66, 1027, 4099, 4101, (1 << 31) - 31, (1 << 31) - 3, (1 << 31) - 1])
@pytest.mark.parametrize("chunk_cols", [32, 256, 1024])
def test_every_column_is_stored_once_and_on_its_sector(row_stores, cols, chunk_cols):
    """... and nothing else: the pieces of a quad's even lanes start 32-byte sectors of the output, in rows g and g + 8 alike, which
    lie half a sector apart where the column count is odd, and only pieces at the ends of a run are cut."""
    chunks = -(-cols // chunk_cols)
    for kc0, kc1 in {(max(chunks - 3, 0), chunks), (chunks - 1, chunks), (max(chunks - 3, 0), max(chunks - 1, 1)), (0, 1)}:
        begin, end = kc0 * chunk_cols, min(kc1 * chunk_cols, cols)
        for off in range(16):
            for half in (0, 1):
                col, n, lane = row_stores(cols, chunk_cols, kc0, kc1, off, half)
                got = np.sort(np.concatenate([np.arange(c, c + k) for c, k in zip(col, n)]))
                assert np.array_equal(got, np.arange(begin, end)), (kc0, kc1, off, half)
                place = (off + 8 * cols * half + col) % 16                   # in the sector, counted in weights
                assert np.all((place == 8 * (lane % 2)) | (col == begin)), (kc0, kc1, off, half)
                assert np.all((n == 8) | (col == begin) | (col + n == end)), (kc0, kc1, off, half)
