"""How far can damaged bits drive the device decoders?  (CPU only.)

The kernels read a chunk's coded rows from a shared-memory slot and never check a bit sequence against its length inside
the hot loop; what keeps a damaged blob from reading outside the CTA's shared memory is that a sequence is a pointer, that
every window is read from the rows under the pointer, and that the tables in shared memory hold no length above their
limit, whatever the blob's table says.  The library keeps 256 * (3 + rows * blocks) readable bytes behind the last slot
(huffllm_decode_smem_plan).

This file walks the pointers of all decoders: the table entries, the pointer's start, the address mask and the layout of the
tables are the kernels' own (csrc/decoder_tables.h, compiled for the host), the order of windows, lookups and shifts is
restated below.  Random and adversarial rows and tables; the furthest row ever addressed must lie inside slot + guard as the
library computes them, every table index inside the table, and the pointer's low 15 bits must be the sum of the lengths.  It
models addresses only: the decoded values are not its subject.
"""
import ctypes
import os
import subprocess

import pytest

import workloads as wl

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_00922_b200", "csrc")
HARNESS = r"""
#include "decoder_tables.h"
#include <algorithm>
#include <vector>
using namespace huffllm;
namespace {
uint64_t seed;
uint32_t rnd() { seed = seed * 6364136223846793005ull + 1442695040888963407ull; return (uint32_t)(seed >> 32); }
struct Walk {
    uint32_t base, furthest = 0, bad = 0;
    int mode;                                              // the rows: 0 random, 1 all ones, 2 all zeros
    uint32_t row(uint32_t pos, uint32_t ahead) {           // the word of row_addr(pos, col) + 256 * ahead
        const uint32_t addr = ((pos * 8u) & kRowMask) + 256u * ahead;
        if (addr < base) bad |= 1u;
        furthest = std::max(furthest, (addr - base) / 256u);
        return mode == 0 ? rnd() : mode == 1 ? ~0u : 0u;
    }
};
uint32_t funnel(uint32_t lo, uint32_t hi, uint32_t n) { return (uint32_t)((((uint64_t)hi << 32) | lo) >> (n & 31u)); }
struct Tables {
    int mode;                                              // the blob's table: 0 random, 1 all ones, 2 zeros, 3 the longest lengths, 4 all beyond 8 bits
    std::vector<uint32_t> words;
    Tables(int m, uint32_t n) : mode(m), words(n) {
        for (auto &w : words) w = m == 0 ? rnd() : m == 1 ? ~0u : m == 2 ? 0u : m == 3 ? (8u << 16) : (0xFFu << 16) | (rnd() & 0xFFFFu);
    }
};
// Entry of first-level piece v (source and field as the kernels load them), or of the whole table.
template <Decoder D> uint32_t first_level(Walk &k, const Tables &t, uint32_t v, uint32_t lut_bits) {
    if (v >= LutPlan<D>::kVecs) { k.bad |= 2u; return 0; }
    const uint32_t i = LutPlan<D>::source(v, lut_bits);
    if (i >= t.words.size()) { k.bad |= 4u; return 0; }
    return lut_entry<D>(t.words[i], LutPlan<D>::field(v));
}
template <Decoder D> uint32_t look(Walk &k, const Tables &t, uint32_t win, uint32_t field, uint32_t lut_bits) {
    const bool sixteen = D == kHalf || D == kHalf12 || D == kFlat || (D == kUpper && field);
    const uint32_t index = D == kBf9 ? (win >> 7) & 0x1FFu : D == kHalf7 ? (win >> 7) & 0x7Fu : win & 0xFFu;
    const uint32_t before = D == kUpper && field ? 2048u : field * 1024u;                  // 16-byte pieces in front of the field's table
    uint32_t e = first_level<D>(k, t, before + index * (sixteen ? 4u : 8u), lut_bits);
    if ((D == kBf12 || D == kHalf12) && (int32_t)e < 0) {
        const uint32_t i = (field << lut_bits) + (win & ((1u << lut_bits) - 1u));
        if (i >= t.words.size()) { k.bad |= 8u; return 0; }
        e = lut_entry<D>(t.words[i], 0u, false);
    }
    return e;
}
template <Decoder D> uint32_t weight(Walk &k, const Tables &t, uint32_t lo, uint32_t hi, uint32_t lut_bits) {      // FP16
    uint32_t win = D == kHalf7 ? lo << 7 : lo;
    const uint32_t e0 = look<D>(k, t, win, 0, lut_bits);
    if (both_flat(D)) return e0;
    if (D == kUpper) return e0 + look<D>(k, t, funnel(win, win, e0), 2, lut_bits);
    win = funnel(win, 0u, e0);
    const uint32_t e1 = look<D>(k, t, win, 1, lut_bits);
    win = D == kHalf12 ? funnel(lo, hi, e0 + e1) : funnel(win, 0u, e1);
    return e0 + e1 + look<D>(k, t, win, 2, lut_bits);
}
template <Decoder D> void walk(Walk &k, const Tables &t, uint32_t blocks, uint32_t lut_bits) {
    uint32_t pos = k.base / 8u + start_of(D);
    uint64_t bits = pos;
    auto add = [&](uint32_t e) { pos += e; bits += e & 0x7FFFu; };
    for (uint32_t w = 0; w < blocks * 8;) {
        if (D == kBf8) {
            uint32_t win = funnel(k.row(pos, 0), k.row(pos, 1), pos), sum[4];
            for (int i = 0; i < 4; ++i, ++w) { sum[i] = look<D>(k, t, win, 0, lut_bits); win = funnel(win, 0u, sum[i]); }
            for (uint32_t e : sum) add(e);
        } else if (D <= kBf12) {
            const uint32_t w0 = k.row(pos, 0), w1 = k.row(pos, 1), w2 = k.row(pos, 2), lo = funnel(w0, w1, pos), hi = funnel(w1, w2, pos);
            uint32_t win = lo;
            for (int h = 0; h < 2; ++h, w += 2) {
                const uint32_t a = look<D>(k, t, win, 0, lut_bits), b = look<D>(k, t, funnel(win, 0u, a), 0, lut_bits);
                add(a); add(b);
                win = funnel(lo, hi, a + b);
            }
        } else {
            uint32_t lo = 0, hi = 0, sum[2];
            for (int i = 0; i < 2; ++i, ++w) {
                if (i == 0 || D == kHalf12) {
                    const uint32_t w0 = k.row(pos, 0), w1 = k.row(pos, 1), w2 = k.row(pos, 2);
                    lo = funnel(w0, w1, pos);
                    hi = funnel(w1, w2, pos);
                }
                sum[i] = weight<D>(k, t, lo, hi, lut_bits);
                if (D == kHalf12) add(sum[i]);
                else if (i == 0) lo = funnel(lo, hi, sum[0]);
            }
            if (D != kHalf12) { add(sum[0]); add(sum[1]); }
        }
        if ((pos & 0x7FFFu) != (bits & 0x7FFFu)) k.bad |= 16u;
    }
}
}
extern "C" int64_t furthest_row(int lb, int fmt, uint32_t lut_bits, uint32_t blocks, uint32_t base, int rows, int table, uint64_t s) {
    seed = s;
    Walk k;
    k.base = base;
    k.mode = rows;
    const Tables t(table, (fmt ? 3u : 1u) << lut_bits);
    switch (decoder_of(lb, fmt)) {
    case kBf8: walk<kBf8>(k, t, blocks, lut_bits); break;
    case kBf9: walk<kBf9>(k, t, blocks, lut_bits); break;
    case kBf12: walk<kBf12>(k, t, blocks, lut_bits); break;
    case kHalf: walk<kHalf>(k, t, blocks, lut_bits); break;
    case kHalf7: walk<kHalf7>(k, t, blocks, lut_bits); break;
    case kHalf12: walk<kHalf12>(k, t, blocks, lut_bits); break;
    case kFlat: walk<kFlat>(k, t, blocks, lut_bits); break;
    case kFlatLanes: walk<kFlatLanes>(k, t, blocks, lut_bits); break;
    case kUpper: walk<kUpper>(k, t, blocks, lut_bits); break;
    }
    return k.bad ? -(int64_t)k.bad : (int64_t)k.furthest;
}
"""


@pytest.fixture(scope="module")
def furthest_row(tmp_path_factory):
    d = tmp_path_factory.mktemp("stream_bound")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I" + CSRC, "-o", str(d / "h.so"), str(d / "h.cpp")])
    f = ctypes.CDLL(str(d / "h.so")).furthest_row
    f.restype = ctypes.c_int64
    f.argtypes = [ctypes.c_int] * 2 + [ctypes.c_uint32] * 3 + [ctypes.c_int] * 2 + [ctypes.c_uint64]
    return f


# (dtype, index bits of the blob's table, kernel's table bits, kernel's format), as the launchers pair them
DECODERS = ([("bf16", b, 8 if b == 8 else 9 if b == 9 else 12, 0) for b in (8, 9, 10, 12)] + [("fp16", 7, 7, 1), ("fp16", 8, 8, 1)] +
            [("fp16", b, 12, 1) for b in (9, 10, 12)] + [("fp16", b, 8, f) for b in (7, 8) for f in (2, 3, 4)])


@pytest.mark.parametrize("dtype,bits,lb,fmt", DECODERS)
@pytest.mark.parametrize("chunk_elems", [512, 1024, 4096, 16384])
def test_no_stream_and_no_table_can_drive_a_decoder_past_the_guard(furthest_row, dtype, bits, lb, fmt, chunk_elems):
    import paper_2502_00922_b200 as hl
    w = (wl.gaussian_weights(16, chunk_elems // 16, 0.02, 3, "fp16") if dtype == "fp16"
         else wl.skewed_exponent_weights(16, chunk_elems // 16, 3))
    cb = hl.build_codebook(w, hl.FP16 if dtype == "fp16" else hl.BF16, bits)
    _, desc = hl.encode(cb, w, chunk_elems)
    cb.free()
    assert desc.lut_bits == bits
    plan = hl.decode_smem_plan(desc)
    blocks = desc.chunk_cols // 32
    assert plan["slot_bytes"] == desc.max_words * 256
    assert plan["guard_bytes"] == 256 * (3 + plan["refill_checks_per_block"] * blocks)
    worst = 0
    for base in (0x500, 0x2C600):                          # a first slot and one near the end of a CTA's shared memory
        for rows in range(3):
            for table in range(5):
                for seed in range(4 if rows == table == 0 else 1):
                    got = furthest_row(lb, fmt, bits, blocks, base, rows, table, 1000 * bits + seed)
                    assert got >= 0, f"fault bits {-got}"
                    worst = max(worst, got)
    # the furthest row lies inside slot + guard even for the smallest slot a record can have (one row), and for the last
    # slot of the CTA, behind which only the guard bytes are promised
    assert (worst + 1) * 256 <= 256 + plan["guard_bytes"]
    # the adversarial cases do reach the bound's order of magnitude: the budget is not idle
    assert worst >= blocks
