"""Where the device encoder's passes leave their numbers (csrc/encode_scratch.h), compiled for the host: the groups' sums must lie among
bits that nobody reads any more, for every number of chunks that is left over behind whole groups.  CPU only."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_00922_b200", "csrc")
# The stores of the launch that leaves the groups' sums, then what a scan CTA reads of the scratch: words in front of its chunks, and in
# the last one all chunks' bits and the most words.
HARNESS = r"""
#include <algorithm>
#include "encode_scratch.h"
using namespace huffllm;
extern "C" uint64_t bytes_of(uint64_t n) { return scratch_bytes(n); }
extern "C" void fill(void *scratch, uint64_t n, const uint32_t *bits, const uint32_t *words) {
    std::copy(bits, bits + n, scratch_bits(scratch));
    std::copy(words, words + n, scratch_words(scratch, n));
}
extern "C" void leave_sums(void *scratch, uint64_t n) {
    uint32_t *const bits = scratch_bits(scratch), *const words = scratch_words(scratch, n);
    for (uint32_t g = 0; g < group_count(n); ++g) {
        EncGroup sums = {};
        for (uint64_t c = (uint64_t)g * kScanThreads; c < std::min<uint64_t>(n, (uint64_t)(g + 1) * kScanThreads); ++c) {
            sums.words += words[c];
            sums.bits += bits[c];
            sums.most = std::max(sums.most, words[c]);
        }
        *group_at(bits, g) = sums;
    }
}
extern "C" void copy_words(void *scratch, uint64_t n, uint32_t *words) { std::copy(scratch_words(scratch, n), scratch_words(scratch, n) + n, words); }
extern "C" uint64_t words_in_front(void *scratch, uint64_t n, uint32_t cta) {
    uint64_t front = 0;
    for (uint32_t g = 0; g < cta; ++g) front += group_at(scratch_bits(scratch), g)->words;
    return front;
}
extern "C" void totals(void *scratch, uint64_t n, uint64_t *bits, uint32_t *most) {
    const uint32_t last = group_count(n);
    *bits = *most = 0;
    for (uint64_t c = (uint64_t)last * kScanThreads; c < n; ++c) {
        *bits += scratch_bits(scratch)[c];
        *most = std::max(*most, scratch_words(scratch, n)[c]);
    }
    for (uint32_t g = 0; g < last; ++g) {
        *bits += group_at(scratch_bits(scratch), g)->bits;
        *most = std::max(*most, group_at(scratch_bits(scratch), g)->most);
    }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("encode_scratch")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I" + CSRC, "-o", str(d / "h.so"), str(d / "h.cpp")])
    h = ctypes.CDLL(str(d / "h.so"))
    h.bytes_of.restype = h.words_in_front.restype = ctypes.c_uint64
    h.bytes_of.argtypes = [ctypes.c_uint64]
    h.fill.argtypes = [ctypes.c_void_p, ctypes.c_uint64, ctypes.c_void_p, ctypes.c_void_p]
    h.leave_sums.argtypes = [ctypes.c_void_p, ctypes.c_uint64]
    h.copy_words.argtypes = [ctypes.c_void_p, ctypes.c_uint64, ctypes.c_void_p]
    h.words_in_front.argtypes = [ctypes.c_void_p, ctypes.c_uint64, ctypes.c_uint32]
    h.totals.argtypes = [ctypes.c_void_p, ctypes.c_uint64, ctypes.c_void_p, ctypes.c_void_p]
    return h


@pytest.mark.parametrize("groups", [1, 2, 48, 60])
@pytest.mark.parametrize("rest", [0, 1, 2, 3, 4, 5, 6, 7, 8, 100, 1022, 1023])
def test_sums_of_groups_leave_every_chunks_words_alone(lib, groups, rest):
    n = 1024 * groups + rest
    rng = np.random.default_rng(n)
    bits, words = rng.integers(1, 1 << 18, n, dtype=np.uint32), rng.integers(1, 400, n, dtype=np.uint32)
    size = lib.bytes_of(n)
    assert size == 256 + 8 * n                               # (what callers of the library have sized theirs by)
    room = np.full(size + 64, 0x5A, dtype=np.uint8)
    at = room.ctypes.data
    lib.fill(at, n, bits.ctypes.data, words.ctypes.data)
    lib.leave_sums(at, n)
    assert np.all(room[:256] == 0x5A) and np.all(room[size:] == 0x5A)
    got = np.zeros(n, np.uint32)
    lib.copy_words(at, n, got.ctypes.data)
    assert np.array_equal(got, words)
    front = np.concatenate([[0], np.cumsum(words, dtype=np.uint64)])
    for cta in range(n // 1024 + 1):
        assert lib.words_in_front(at, n, cta) == front[1024 * cta]
    all_bits, most = np.zeros(1, np.uint64), np.zeros(1, np.uint32)
    lib.totals(at, n, all_bits.ctypes.data, most.ctypes.data)
    assert all_bits[0] == bits.sum(dtype=np.uint64) and most[0] == words.max()
