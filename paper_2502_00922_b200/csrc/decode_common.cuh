// Device code shared by the decode kernels: PTX helpers, the per-sequence decoder, the shared-memory plan.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

#include "decoder_tables.h"
#include "kernels.h"

namespace huffllm {

// ------------------------------------------------------------------------------ PTX helpers

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

template <int OFF = 0>
__device__ __forceinline__ uint32_t lds_stream(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(addr), "n"(OFF));
    return v;
}
// LUT reads: the table is constant once built, so the compiler may schedule these freely.
__device__ __forceinline__ uint32_t lds_lut(uint32_t addr) {
    uint32_t v;
    asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Arrival without a transaction count (a consumer hands a slot back).
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// One look at a barrier's phase, without waiting.
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bulk asynchronous copy global -> this CTA's shared memory, completion counted on `bar`.
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ uint4 ldg_stream16(const void *p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t ldg_stream2(const void *p) {
    uint16_t v;
    asm volatile("ld.global.nc.L1::no_allocate.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ void mma_f16_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                              uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                               uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Two mixed-precision multiply-adds: acc += w.lo * x.lo, then acc += w.hi * x.hi (bf16 halves of the two words).
// The products are exact in f32; each addition rounds once.
__device__ __forceinline__ void fma2_bf16(float &acc, uint32_t w, uint32_t x) {
    asm("{\n\t.reg .b16 wl, wh, xl, xh;\n\t"
        "mov.b32 {wl, wh}, %1;\n\t"
        "mov.b32 {xl, xh}, %2;\n\t"
        "fma.rn.f32.bf16 %0, wl, xl, %0;\n\t"
        "fma.rn.f32.bf16 %0, wh, xh, %0;\n\t}"
        : "+f"(acc)
        : "r"(w), "r"(x));
}

__device__ __forceinline__ void fma2_f16(float &acc, uint32_t w, uint32_t x) {
    asm("{\n\t.reg .b16 wl, wh, xl, xh;\n\t"
        "mov.b32 {wl, wh}, %1;\n\t"
        "mov.b32 {xl, xh}, %2;\n\t"
        "fma.rn.f32.f16 %0, wl, xl, %0;\n\t"
        "fma.rn.f32.f16 %0, wh, xh, %0;\n\t}"
        : "+f"(acc)
        : "r"(w), "r"(x));
}

// Arrival counter bump that publishes this warp's earlier stores and acquires the other arrivals' stores.
__device__ __forceinline__ uint32_t arrive_acq_rel(unsigned int *counter) {
    uint32_t old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(old) : "l"(counter) : "memory");
    return old;
}
// Programmatic dependent launch: let the next kernel in the stream be scheduled early / wait for the previous one.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait_prior_grid() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ------------------------------------------------------------------------------ lane decoder

// All that a decoder keeps of a bit sequence is its pointer: bits, counted from shared address 0 as if the sequence's rows
// were all there is (a row of a record holds one 32-bit word of each of the 64 sequences, 256 bytes), so that bits 5 and up
// times 8 are the address of the row that holds the next codeword and the low 5 bits say where in that word it starts.
// Whenever window bits are wanted, the two or three words at the pointer are read again: one multiplication and one logic
// operation for the address, and no registers from one step to the next.
// The pointer is advanced by adding whole table entries, which hold the length in their low bits and the symbol above bit
// 15 or higher: shared addresses have 18 bits, so bits 0..14 of the pointer are all that is read.
// What bounds these loops is the number of instructions (the SMs issue in four of five cycles) with the shared-memory pipe
// close behind (1.5 loads per BF16 weight).  Cycles per 32 weights and scheduler, 31 warps decoding from shared memory with
// nothing around them: window words kept in registers and refilled under a predicate 8.4 (28 instructions per four
// codewords), this 8.2 (27; and six registers fewer).
// Memory safety: the shared-memory copies of the tables hold no length above what the table's index bits allow
// (lut_entry), so a block moves a sequence by at most that many bits per codeword, whatever the stream and the table hold;
// the guard area behind the last slot covers it.

// Address of the row under the pointer, at byte `col` of it (4 * sequence).
__device__ __forceinline__ uint32_t row_addr(uint32_t pos, uint32_t col) {
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(d) : "r"(pos * 8u), "n"(kRowMask), "r"(col));
    return d;
}
// 32 bits of (hi:lo) from bit n % 32 on.
__device__ __forceinline__ uint32_t funnel(uint32_t lo, uint32_t hi, uint32_t n) {
    uint32_t t;
    asm("shf.r.wrap.b32 %0, %1, %2, %3;" : "=r"(t) : "r"(lo), "r"(hi), "r"(n));
    return t;
}
// The 32 bits at the pointer.  OFF = 0: the lane's first sequence (row g), 128: its second one (row g + 8).
template <int OFF>
__device__ __forceinline__ uint32_t window32(uint32_t pos, uint32_t col) {
    const uint32_t a = row_addr(pos, col);
    const uint32_t lo = lds_stream<OFF>(a), hi = lds_stream<OFF + 256>(a);
    return funnel(lo, hi, pos);
}
// The 64 bits at the pointer.
struct Window {
    uint32_t lo, hi;
};
template <int OFF>
__device__ __forceinline__ Window window64(uint32_t pos, uint32_t col) {
    const uint32_t a = row_addr(pos, col);
    const uint32_t w0 = lds_stream<OFF>(a), w1 = lds_stream<OFF + 256>(a), w2 = lds_stream<OFF + 512>(a);
    return {funnel(w0, w1, pos), funnel(w1, w2, pos)};
}
// A window shifted in place by an entry's length (its low 5 bits; the entry may be a sum of entries).
__device__ __forceinline__ uint32_t shift_by(uint32_t t, uint32_t e) { return funnel(t, 0u, e); }
// Table entry of the window's low byte: `stride` bytes per entry (byte dot product: index * stride + the lane's column).
__device__ __forceinline__ uint32_t lookup_byte0(uint32_t t, uint32_t stride, uint32_t lut_lane) { return lds_lut(__dp4a(t, stride, lut_lane)); }

// ---- BF16

// Two entries -> one word with the even weight's exponent at bits 7..14 and the odd one's at 23..30: the even entry's upper
// half plus the odd entry (a 16-bit dot product: one instruction of the multiplying pipe, where a byte permute would join
// the shifts on the integer pipe: 8.2 against 8.4 cycles).  Lengths end up among the mantissa bits.
__device__ __forceinline__ uint32_t merge_exponents(uint32_t e_even, uint32_t e_odd) { return __dp2a_lo(e_even, 0x00000100u, e_odd); }
// Exponents + the raw word of their group -> two bf16 weights packed in one register.
// A raw word holds the sign and mantissa bits of four consecutive weights of a row, laid out so that the first pair's
// bits already sit where a packed pair of bf16 words has them (mantissas at bits 0..6 and 16..22, signs at 15 and 31)
// and the second pair's do after a rotation by one byte; the other pair's bits lie in the exponent positions, which
// the select takes from the table entries.
__device__ __forceinline__ uint32_t pack_pair(uint32_t ex, uint32_t sm) {
    uint32_t w;   // sign and mantissa bits from sm, exponent bits from ex
    asm("lop3.b32 %0, %1, %2, 0x807F807F, 0xE4;" : "=r"(w) : "r"(sm), "r"(ex));
    return w;
}
__device__ __forceinline__ uint32_t rotr8(uint32_t v) { return prmt(v, v, 0x0321u); }

// One codeword of a longer code.  9 bits: the window is 7 bits behind the codeword, so the masked window is the address
// (the table lies on a boundary above the index bits).  Up to 12: the first level resolves codewords of up to 8 bits; a
// marked entry sends the lane to the whole table (one copy, 1 << lut_bits entries; full_mask = ((1 << lut_bits) - 1) * 4).
// Long codewords are rare, so the second level's bank conflicts do not matter.
template <Decoder D>
__device__ __forceinline__ uint32_t lookup_long(uint32_t t, uint32_t lut_lane, uint32_t full_base, uint32_t full_mask) {
    if (D == kBf9) {
        uint32_t addr;
        asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(addr) : "r"(t), "n"(0x1FFu << 7), "r"(lut_lane));
        return lds_lut(addr);
    }
    uint32_t e = lookup_byte0(t, D == kBf12 ? 128u : 64u, lut_lane);
    asm("{\n\t.reg .pred p;\n\t.reg .b32 i;\n\t"
        "setp.lt.s32 p, %0, 0;\n\t"
        "mad.lo.u32 i, %1, 4, 0;\n\t"
        "@p and.b32 i, i, %3;\n\t"
        "@p add.u32 i, i, %2;\n\t"
        "@p ld.shared.u32 %0, [i];\n\t}"
        : "+r"(e)
        : "r"(t), "r"(full_base), "r"(full_mask));
    return e;
}

// Four codewords of each of a lane's two sequences, the two chains interleaved; x: two words of merged exponents each.
// Codewords of up to 8 bits: the window's 32 bits hold four, taken out once and shifted in place; the pointer is not on
// the chain from one lookup to the next.  Longer ones: 64 bits are taken out, two codewords (at most 24 bits, 25 with the
// 9-bit table's lag) come from the low word, two from the 32 bits behind them.
template <Decoder D>
__device__ __forceinline__ void step4(uint32_t &pa, uint32_t &pb, uint32_t col, uint32_t lut_lane, uint32_t *xa, uint32_t *xb,
                                      uint32_t full_base, uint32_t full_mask) {
    uint32_t ea[4], eb[4];
    if (D == kBf8) {
        uint32_t ta = window32<0>(pa, col), tb = window32<128>(pb, col);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            ea[i] = lookup_byte0(ta, 128u, lut_lane);
            eb[i] = lookup_byte0(tb, 128u, lut_lane);
            if (i < 3) {
                ta = shift_by(ta, ea[i]);
                tb = shift_by(tb, eb[i]);
            }
        }
        pa = (pa + ea[0] + ea[1]) + (ea[2] + ea[3]);
        pb = (pb + eb[0] + eb[1]) + (eb[2] + eb[3]);
    } else {
        const Window wa = window64<0>(pa, col), wb = window64<128>(pb, col);
        uint32_t ta = wa.lo, tb = wb.lo;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            ea[2 * h] = lookup_long<D>(ta, lut_lane, full_base, full_mask);
            eb[2 * h] = lookup_long<D>(tb, lut_lane, full_base, full_mask);
            ta = shift_by(ta, ea[2 * h]);
            tb = shift_by(tb, eb[2 * h]);
            ea[2 * h + 1] = lookup_long<D>(ta, lut_lane, full_base, full_mask);
            eb[2 * h + 1] = lookup_long<D>(tb, lut_lane, full_base, full_mask);
            const uint32_t da = ea[2 * h] + ea[2 * h + 1], db = eb[2 * h] + eb[2 * h + 1];
            pa += da;
            pb += db;
            ta = funnel(wa.lo, wa.hi, da);
            tb = funnel(wb.lo, wb.hi, db);
        }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        xa[i] = merge_exponents(ea[2 * i], ea[2 * i + 1]);
        xb[i] = merge_exponents(eb[2 * i], eb[2 * i + 1]);
    }
}

// ---- FP16 {1,5,5,5}

// FP16 blobs code three fields per weight (exponent, upper and lower mantissa half: Section 3.1), each with its own table.
// A weight's entries are added up: its low 15 bits stand in the sum's upper half, its length in the low bits, which is what
// the next window and the pointer want.  Two weights come from one 64-bit window (at most 48 bits; the second one's 32 bits
// are taken out behind the first).
// The three tables of kHalf are 16 KB each, sixteen copies per entry (entry i of copy c at word 16 i + c; a lane uses copy
// lane % 16: a lookup takes two passes).  kHalf7's have 128 entries and a copy per lane: no conflicts; seven bits are no
// byte, so the window is moved up by 7 bits and masked.
// A FLAT code (all 32 symbols, 5 bits each: the canonical codeword of symbol s is s, written first bit first) needs no
// table: fp16-trained weights have it in both mantissa halves, bf16-trained ones in the upper half.  Its bits follow the
// exponent's codeword in reverse order.  The exponent's entry has them in its length, and the window is ROTATED by that
// length instead of shifted: what comes next (the second weight, or the lower half's codeword) stands at bit 0, and the flat
// bits at the top, in the order in which a bit reversal of both weights' halves at once puts them where they belong.
// The tables that are left have a copy per lane (kUpper's lower half and kFlat's one: sixteen).
template <Decoder D>
__device__ __forceinline__ uint32_t lookup_field(uint32_t t, int field, uint32_t lut_lane, uint32_t full_base, uint32_t full_mask) {
    if (D == kHalf7) {
        uint32_t addr;
        asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(addr) : "r"(t), "n"(0x7Fu << 7), "r"(lut_lane));
        return lds_lut(addr + 16384u * field);
    }
    if (D == kHalf12) return lookup_long<D>(t, lut_lane + 16384u * field, full_base + (full_mask + 4u) * field, full_mask);
    return lds_lut(__dp4a(t, 64u, lut_lane) + 16384u * field);
}
// One weight out of the 32 (kHalf12: 64) bits at its start: the sum of its entries, and the rotated window of the flat codes.
template <Decoder D>
__device__ __forceinline__ uint32_t weight_sum(const Window &w, uint32_t lut_lane, uint32_t lut_low, uint32_t full_base, uint32_t full_mask, uint32_t &rot) {
    uint32_t t = D == kHalf7 ? w.lo << 7 : w.lo;
    if (both_flat(D) || D == kUpper) {
        const uint32_t e0 = lookup_byte0(t, D == kFlat ? 64u : 128u, lut_lane);
        rot = funnel(t, t, e0);
        if (both_flat(D)) return e0;
        return e0 + lookup_byte0(rot, 64u, lut_low);
    }
    const uint32_t e0 = lookup_field<D>(t, 0, lut_lane, full_base, full_mask);
    t = shift_by(t, e0);
    const uint32_t e1 = lookup_field<D>(t, 1, lut_lane, full_base, full_mask);
    if (D == kHalf12) t = funnel(w.lo, w.hi, e0 + e1);
    else t = shift_by(t, e1);
    return e0 + e1 + lookup_field<D>(t, 2, lut_lane, full_base, full_mask);
}
// Two weights of each of a lane's two sequences -> their 15 bits each, as packed pairs (the sign positions hold anything).
template <Decoder D>
__device__ __forceinline__ void step2_fp16(uint32_t &pa, uint32_t &pb, uint32_t col, uint32_t lut_lane, uint32_t lut_low, uint32_t &xa, uint32_t &xb,
                                           uint32_t full_base, uint32_t full_mask) {
    Window wa = window64<0>(pa, col), wb = window64<128>(pb, col);
    uint32_t ea[2], eb[2], ra[2], rb[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        if (D == kHalf12 && i) {                      // (36 bits at most: the second weight has a window of its own)
            wa = window64<0>(pa, col);
            wb = window64<128>(pb, col);
        }
        ea[i] = weight_sum<D>(wa, lut_lane, lut_low, full_base, full_mask, ra[i]);
        eb[i] = weight_sum<D>(wb, lut_lane, lut_low, full_base, full_mask, rb[i]);
        if (D == kHalf12) {
            pa += ea[i];
            pb += eb[i];
        } else if (i == 0) {
            wa.lo = funnel(wa.lo, wa.hi, ea[0]);
            wb.lo = funnel(wb.lo, wb.hi, eb[0]);
        }
    }
    if (D != kHalf12) {
        pa += ea[0] + ea[1];
        pb += eb[0] + eb[1];
    }
    auto pair = [&](const uint32_t *e, const uint32_t *r) -> uint32_t {
        const uint32_t coded = both_flat(D) ? merge_exponents(e[0], e[1]) : prmt(e[0], e[1], 0x7632u);
        if (!both_flat(D) && D != kUpper) return coded;
        const uint32_t flat = __brev(prmt(r[0], r[1], 0x3276u));      // bits 0..9 / 16..25 (kUpper: 0..4 / 16..20): mantissa bits
        uint32_t x;
        if (both_flat(D)) asm("lop3.b32 %0, %1, %2, 0x03FF03FF, 0xE4;" : "=r"(x) : "r"(flat), "r"(coded));
        else asm("lop3.b32 %0, %1, %2, 0x03E003E0, 0xE4;" : "=r"(x) : "r"(flat * 32u), "r"(coded));
        return x;
    };
    xa = pair(ea, ra);
    xb = pair(eb, rb);
}

// ---- a block of 32 columns: 16 weights of this lane as 8 packed registers
// a[0..3] = row g, columns (0,1) (2,3) (4,5) (6,7);  a[4..7] = row g+8, same columns.
// raw: the lane's raw bytes of the block.  BF16: four words of sign and mantissa bits.  FP16: raw.x is a uint16, bit p = sign of
// the first weight of pair p, bit 8 + p = sign of its second weight.
template <Decoder D>
__device__ __forceinline__ void decode_block(uint32_t &pa, uint32_t &pb, uint32_t col, uint32_t lut_lane, uint32_t lut_low, const uint4 &raw,
                                             uint32_t (&a)[8], uint32_t full_base, uint32_t full_mask) {
    uint32_t x[8];
    if (D <= kBf12) {
#pragma unroll
        for (int i = 0; i < 4; i += 2) step4<D>(pa, pb, col, lut_lane, x + i, x + 4 + i, full_base, full_mask);
        const uint32_t sm[8] = {raw.x, rotr8(raw.x), raw.y, rotr8(raw.y), raw.z, rotr8(raw.z), raw.w, rotr8(raw.w)};
#pragma unroll
        for (int i = 0; i < 8; ++i) a[i] = pack_pair(x[i], sm[i]);
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) step2_fp16<D>(pa, pb, col, lut_lane, lut_low, x[i], x[4 + i], full_base, full_mask);
        const uint32_t s32 = prmt(raw.x, 0u, 0x4140u);     // first-weight signs in bits 0..7, second-weight signs in bits 16..23
#pragma unroll
        for (int p = 0; p < 8; ++p)                        // their sign bits at bits 15 and 31; mask bit set: the pair's, else the sign
            asm("lop3.b32 %0, %1, %2, 0x7FFF7FFF, 0xE4;" : "=r"(a[p]) : "r"(x[p]), "r"(s32 << (15 - p)));
    }
}

// ------------------------------------------------------------------------------ shared memory plan

// Dynamic shared memory, laid out at run time from the window's real start address:
//   [base, lut)            slot pairs (single slots where the launch says so), as many as fit
//   [lut, lut + LUTSZ)     per-lane LUT; lut = base rounded up to a multiple of LUTSZ, so that the
//                          index bits of a lookup address never overlap the table's base bits
//   [lut + LUTSZ, ...)     more slot pairs, then a guard area no valid stream ever reads (it may overlap the next area)
//   [end - part_bytes, end) the CTA's table of partial sums (fused product only)
struct SmemPlan {
    uint32_t lut;    // shared address of the table
    uint32_t warps;  // warps that own a slot pair
    uint32_t slotA;  // first slot pair before the table
    uint32_t nA;     // slot pairs before the table
    uint32_t slotB;  // first slot pair after it
};

__device__ __forceinline__ SmemPlan plan_smem(uint32_t base, const KernelArgs &k, uint32_t max_warps, uint32_t slots = 2) {   // k: launch-wide fields only
    SmemPlan p;
    const uint32_t lut_bytes = k.lut_align;
    uint32_t a0 = (base + 255u) & ~255u;     // (slots are whole rows of 256 bytes, on 256-byte boundaries)
    p.lut = (base + lut_bytes - 1) & ~(lut_bytes - 1);        // lut_align is a power of two
    p.slotA = a0;
    // (divisions by the slot pair's size as a multiplication by its rounded-down reciprocal and one correction: this
    // runs in every warp of a launch's set-up, which is bound by instruction issue)
    const uint32_t pair = slots == 2 ? 2 * k.slot_bytes : k.slot_bytes;
    auto div_pair = [&](uint32_t x) -> uint32_t {
        uint32_t q = __umulhi(x, k.pair_recip);
        return x - q * pair >= pair ? q + 1 : q;
    };
    p.nA = p.lut > a0 ? div_pair(p.lut - a0) : 0;  // a stream that overruns here reads the table: harmless
    p.slotB = p.lut + k.lut_size;
    uint32_t end = base + k.dyn_smem_bytes - k.part_bytes;
    // the guard area (read only, and only by a corrupt stream) may lie over what follows the slots; what it needs beyond that stays free
    const uint32_t guard_extra = k.guard_bytes > k.part_bytes ? k.guard_bytes - k.part_bytes : 0;
    uint32_t roomB = end > p.slotB + guard_extra ? end - p.slotB - guard_extra : 0;
    p.warps = min(max_warps, p.nA + div_pair(roomB));
    return p;
}

// Slot `which` of a decoder warp (two slots per warp).
__device__ __forceinline__ uint32_t slot_addr(const SmemPlan &p, uint32_t warp, uint32_t which, uint32_t slot_bytes) {
    uint32_t pair = warp < p.nA ? p.slotA + warp * 2 * slot_bytes : p.slotB + (warp - p.nA) * 2 * slot_bytes;
    return pair + which * slot_bytes;
}
// The one slot of a decoder warp where warps have single slots.
__device__ __forceinline__ uint32_t slot_addr_single(const SmemPlan &p, uint32_t warp, uint32_t slot_bytes) {
    return warp < p.nA ? p.slotA + warp * slot_bytes : p.slotB + (warp - p.nA) * slot_bytes;
}

constexpr int kMaxWarps = 32;
constexpr int kThreads = 1024;   // threads per CTA of the decode kernels (one CTA per SM)
constexpr uint32_t kWaitLimit = 1u << 22;
constexpr uint32_t kErrOverrun = 0x40000000u;     // error flag: this bit + (chunk + 1): the chunk's bits ran past its record
constexpr uint32_t kFeederIdleLimit = 1u << 22;   // polls of 100 ns without any slot coming back before the feeder gives up

}  // namespace huffllm
