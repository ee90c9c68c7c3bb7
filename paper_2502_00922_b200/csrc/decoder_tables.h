// The decoders, what their tables in shared memory hold and where those stand, and where a bit sequence's pointer starts: what the
// bound on a decoder's reads rests on (decode_common.cuh).
#pragma once
#include <cstdint>

#include "host_device.h"

namespace huffllm {

// Bits of 8 times a pointer that are the address of its row.
constexpr uint32_t kRowMask = 0x3FF00u;

// The decoders, by the blobs' format and code lengths (LB = index bits of the tables, 12 for all above 9; FMT: see huff_kernel).
enum Decoder {
    kBf8,      // BF16, codewords of at most 8 bits: table once per lane
    kBf9,      // BF16, 9 bits: table once per lane
    kBf12,     // BF16, up to 12 bits: two levels
    kHalf,     // FP16, three tables of 8 bits, sixteen copies each
    kHalf7,    // FP16, three tables of 7 bits, once per lane
    kHalf12,   // FP16, up to 12 bits per field: two levels
    kFlat,     // FP16, both mantissa halves carry the flat code (codewords of at most 8 bits): sixteen copies
    kFlatLanes,  // the same, table once per lane
    kUpper,    // FP16, the upper mantissa half carries the flat code (codewords of at most 8 bits)
};
HUFFLLM_HD constexpr Decoder decoder_of(int lb, int fmt) {
    return fmt == 0 ? (lb == 8 ? kBf8 : lb == 9 ? kBf9 : kBf12) : fmt == 1 ? (lb == 8 ? kHalf : lb == 7 ? kHalf7 : kHalf12) : fmt == 2 ? kFlat : fmt == 4 ? kFlatLanes : kUpper;
}
// Where a sequence's pointer starts: on its first codeword, behind the leading zero bits (7, FP16: 6); kBf9 stays 7 bits
// behind, so that the index stands where the address wants it.
HUFFLLM_HD constexpr uint32_t lag_of(Decoder d) { return d <= kBf12 ? 7u : 6u; }
HUFFLLM_HD constexpr uint32_t start_of(Decoder d) { return d == kBf9 ? 0u : lag_of(d); }
// Longest codeword (per field).
HUFFLLM_HD constexpr uint32_t longest_of(Decoder d) { return d == kBf9 ? 9u : d == kHalf7 ? 7u : d == kBf12 || d == kHalf12 ? 12u : 8u; }
// FP16 with both mantissa halves flat.
HUFFLLM_HD constexpr bool both_flat(Decoder d) { return d == kFlat || d == kFlatLanes; }
constexpr uint32_t kLongMark = 0x80000000u;

// Shared-memory form of a blob's table entry (length << 16 | symbol bits): the length in the low bits, the symbol above.
// BF16: exponent at bits 23..30.  FP16: the field where it belongs in the weight, 16 bits up; the exponent's entry of the
// decoders that read flat codes without a table has their bits added to its length.  A codeword of more than the first
// level's 8 bits is only marked there.
template <Decoder D>
HUFFLLM_HD uint32_t lut_entry(uint32_t e, uint32_t field, bool first_level = true) {
    const uint32_t len = e >> 16;
    if ((D == kBf12 || D == kHalf12) && first_level && len > 8u) return kLongMark;
    const uint32_t flat_bits = both_flat(D) ? 10u : D == kUpper && field == 0 ? 5u : 0u;
    return ((D <= kBf12 ? e & 0x7F80u : e & 0x7FFFu) << 16) | ((len < longest_of(D) ? len : longest_of(D)) + flat_bits);
}

// The tables in shared memory, by decoder, in 16-byte pieces (copies of one entry).
template <Decoder D>
struct LutPlan {
    // 16-byte pieces of the first level
    static constexpr uint32_t kVecs = D == kBf9 ? 4096u : D <= kBf12 || D == kFlatLanes ? 2048u : D == kFlat ? 1024u : 3072u;
    // entry index in the blob's tables (of 1 << lut_bits entries each) and field of piece v
    static HUFFLLM_HD uint32_t source(uint32_t v, uint32_t lut_bits) {
        if (D <= kBf12) return v >> 3;
        if (D == kHalf7) return (field(v) << lut_bits) + ((v >> 3) & 127u);
        if (D == kHalf || D == kHalf12) return (field(v) << lut_bits) + ((v >> 2) & 255u);
        // (tables of 7 bits serve as tables of 8 whose upper half repeats the lower one)
        const uint32_t in = D == kFlat ? v >> 2 : field(v) ? (v >> 2) & 255u : v >> 3;
        return (field(v) << lut_bits) + (in & ((1u << lut_bits) - 1u));
    }
    static HUFFLLM_HD uint32_t field(uint32_t v) { return D <= kBf12 || both_flat(D) ? 0u : D == kUpper ? (v >> 11) * 2u : v >> 10; }
};
// A lane's column of the table(s), and of kUpper's second one.
template <Decoder D>
HUFFLLM_HD uint32_t lut_column(uint32_t lut, uint32_t lane) { return lut | (D == kHalf || D == kHalf12 || D == kFlat ? lane & 15u : lane) << 2; }
template <Decoder D>
HUFFLLM_HD uint32_t lut_low_column(uint32_t lut, uint32_t lane) { return D == kUpper ? lut + 32768u + ((lane & 15u) << 2) : 0u; }
// Bytes of the first level, behind which the whole tables of the two-level decoders lie.
template <Decoder D>
constexpr uint32_t kLutBytes = LutPlan<D>::kVecs * 16u;

}  // namespace huffllm
