"""Which columns the pieces of a decode to rows that start anywhere hold (csrc/row_pieces.h), compiled for the host: no GPU is
needed, and the column counts go up to the largest that a blob can have."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_00922_b200", "csrc")
# A warp's stores to one row, in the kernel's order: chunks kc0 .. kc1 - 1 as one run, four lanes a block, what is left over.
HARNESS = r"""
#include "row_pieces.h"
using namespace huffllm;
extern "C" int64_t row_stores(uint64_t cols, uint32_t chunk_cols, uint32_t kc0, uint32_t kc1, uint32_t off, int64_t *col, int32_t *n) {
    int64_t count = 0;
    auto store = [&](uint32_t at, int32_t c, int32_t first, int32_t end) {
        const PieceCut cut = piece_cut(c, first, end);
        if (cut.lo < cut.hi) { col[count] = (int64_t)at + c + cut.lo; n[count++] = cut.hi - cut.lo; }
    };
    for (uint32_t kc = kc0; kc < kc1; ++kc) {
        const uint32_t at = kc * chunk_cols;
        const int32_t left = columns_left(cols, at), blocks = ((left < (int32_t)chunk_cols ? left : (int32_t)chunk_cols) + 31) / 32;
        for (int32_t kb = 0; kb < blocks; ++kb)
            for (uint32_t t = 0; t < 4; ++t) {
                const int32_t c = piece_column(kb, t, off);
                if (kb >= (kc == kc0) && kb * 32 + 32 <= left) { col[count] = (int64_t)at + c; n[count++] = 8; }
                else store(at, c, run_start(kc > kc0), left);
            }
    }
    const uint32_t at = (kc1 - 1) * chunk_cols;
    const int32_t left = columns_left(cols, at), end = left < (int32_t)chunk_cols ? left : (int32_t)chunk_cols;
    for (uint32_t t = 0; t < 4; ++t)
        if (t * 8 < off) store(at, last_piece_column(end, t, off), 0, end);
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
    f.argtypes = [ctypes.c_uint64] + [ctypes.c_uint32] * 4 + [ctypes.c_void_p] * 2

    def call(cols, chunk_cols, kc0, kc1, off):
        col, n = np.zeros(4096, np.int64), np.zeros(4096, np.int32)
        k = f(cols, chunk_cols, kc0, kc1, off, col.ctypes.data, n.ctypes.data)
        return col[:k], n[:k]
    return call


@pytest.mark.parametrize("cols", [65, 66, 1027, 4099, 4101, (1 << 31) - 31, (1 << 31) - 3, (1 << 31) - 1])
@pytest.mark.parametrize("chunk_cols", [32, 256, 1024])
def test_every_column_is_stored_once_and_nothing_else(row_stores, cols, chunk_cols):
    chunks = -(-cols // chunk_cols)
    for kc0, kc1 in {(max(chunks - 3, 0), chunks), (chunks - 1, chunks), (max(chunks - 3, 0), max(chunks - 1, 1)), (0, 1)}:
        for off in range(16):
            col, n = row_stores(cols, chunk_cols, kc0, kc1, off)
            got = np.sort(np.concatenate([np.arange(c, c + k) for c, k in zip(col, n)]))
            assert np.array_equal(got, np.arange(kc0 * chunk_cols, min(kc1 * chunk_cols, cols))), (kc0, kc1, off)
