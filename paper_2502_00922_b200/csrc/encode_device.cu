// Device-side encoder: builds the same blob as huffllm_encode, byte for byte, from weights that already sit in
// device memory.  Compression is an offline, one-time step (Section 3.1); on the host it takes seconds per decoder
// layer, here it is three short passes over the tensor, so a model can be compressed while it is being loaded.
//
// A warp takes a chunk, its lanes the format's lanes: two bit sequences each (rows g and g + 8), one after the other in the loops
// below, so that a lane has two chains under way and what a chunk costs besides its weights is paid once per 128 of a lane's.
//   pass 1  code lengths only -> words per sequence and coded bits of every chunk; a CTA of its own writes code lengths and table
//   scan    record offsets (the index section), payload size, largest record
//   pass 2  raw part and coded part of every record (nothing if the scan found the tensor or the buffer unfit)
//   pass 3  the checksum term of every record, a warp each (many short records: a thread); the last one completes the header
// The host waits once, behind the last pass.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstring>
#include <type_traits>

#include "decode_common.cuh"
#include "encode_scratch.h"
#include "internal.h"

namespace huffllm {

struct EncTotals {
    unsigned long long payload_units, coded_bits, checksum;
    uint32_t max_words, bad;     // bad: 1 = a symbol without codeword, 2 = payload beyond the 32-bit record index, 4 = a wait ran out
    uint32_t summed;             // CTAs whose records' checksums are in
};

static_assert(sizeof(EncTotals) <= kScratchTotals, "the chunks' bits and words follow in the scratch");

constexpr uint32_t kWriteWarps = 4;          // of a CTA of pass 2
__host__ __device__ constexpr uint32_t write_ctas(bool vec) { return vec ? 6 : 5; }     // of an SM (80 and 96 registers)
constexpr uint32_t kNoCode = 1u << 14;       // length of a symbol without codeword: no sum of a sequence's codewords reaches it (768 of 12 bits)

constexpr uint32_t kUnfit = 0xFFFFFFFFu;

struct EncArgs {
    const uint16_t *w;
    uint64_t rows, cols, n_chunks;
    uint32_t Kc, KC, fp16, lag_bits, pad, vec_ok;
    uint32_t stage_rows;         // rows of a record that a warp of pass 2 has room for in shared memory
    uint64_t max_units;          // what the blob has room for
    uint32_t *bits, *words;      // per chunk: coded bits, words per sequence (kUnfit: a symbol without codeword)
    uint32_t *index;
    uint8_t *blob, *payload;
    EncTotals *totals;
    uint32_t code[256];          // a symbol's codeword, first bit in bit 31 | its length (FP16: three fields of 32 symbols)
    uint8_t lengths[256];        // the section of code lengths
    huffllm_desc desc;           // the header, but for what the totals say
};

__device__ __forceinline__ bool enc_fits(const EncArgs &A) {
    return __ldcg(&A.totals->bad) == 0u && __ldcg(&A.totals->payload_units) <= A.max_units;
}

// byte of a group's 32-bit word that takes weight j's mantissa bits, and the one that takes its sign (the raw-byte layout)
__host__ __device__ constexpr uint32_t raw_mant_byte(uint32_t j) { return ((j & 1u) << 1) | (j >> 1); }
__host__ __device__ constexpr uint32_t raw_sign_byte(uint32_t j) { return (raw_mant_byte(j) + 1u) & 3u; }
static_assert(raw_mant_byte(0) == kRawMantByte[0] && raw_mant_byte(1) == kRawMantByte[1] && raw_mant_byte(2) == kRawMantByte[2] &&
              raw_mant_byte(3) == kRawMantByte[3], "raw-byte layout");
// the same as byte selectors over two words of two weights each: weight j's low byte is byte 2 j, its high byte byte 2 j + 1
__host__ __device__ constexpr uint32_t raw_sel(bool sign) {
    uint32_t sel = 0;
    for (uint32_t j = 0; j < 4; ++j) sel |= (2 * j + (sign ? 1 : 0)) << (4 * (sign ? raw_sign_byte(j) : raw_mant_byte(j)));
    return sel;
}
constexpr uint32_t kRawMantSel = raw_sel(false), kRawSignSel = raw_sel(true);
static_assert(raw_sign_byte(0) == kRawSignByte[0] && raw_sign_byte(1) == kRawSignByte[1] && raw_sign_byte(2) == kRawSignByte[2] &&
              raw_sign_byte(3) == kRawSignByte[3], "raw-byte layout");

__device__ __forceinline__ uint32_t enc_blocks_of(const EncArgs &A, uint32_t kc) {
    uint64_t left = A.cols - (uint64_t)kc * A.Kc;
    return (uint32_t)(((left < A.Kc ? left : A.Kc) + 31) / 32);
}
__device__ __forceinline__ uint32_t enc_raw_bytes(const EncArgs &A, uint32_t nkb) {
    return A.fp16 ? (nkb * 64u + 127u) & ~127u : nkb * 512u;
}

// A lane of the warp that takes chunk c: its weights are, in every block of 32 columns, eight in row g and eight in row g + 8.
struct EncLane {
    uint32_t nkb, whole;        // blocks of the chunk; those that lie inside the tensor, with the 16-byte pieces around their rows' ends
    const uint16_t *row[2];     // the weights in the first block
    int32_t left[2];            // columns (at most) before the row ends, 0 for rows outside the tensor
    uint32_t off;               // bytes from a 16-byte boundary to the weights, in both rows
};
__device__ __forceinline__ EncLane enc_lane(const EncArgs &A, uint32_t c, uint32_t lane) {           // (fewer than 2^31 chunks)
    EncLane L;
    const uint32_t rg = c / A.KC, kc = c - rg * A.KC;
    const uint64_t r = (uint64_t)rg * 16 + (lane >> 2), first = (uint64_t)kc * A.Kc, col0 = first + (lane & 3) * 8;
    const uint32_t cols = (uint32_t)min(A.cols - first, (uint64_t)A.Kc);
    L.nkb = (cols + 31) / 32;
    L.whole = (uint64_t)rg * 16 + 16 <= A.rows ? cols / 32 : 0u;
    // (nothing outside the tensor is read: off 16-byte boundaries the pieces of its first row begin in front of it, and those of its last
    // row may reach up to eight weights behind the chunk)
    if (!A.vec_ok && (c == 0 || ((uint64_t)rg * 16 + 16 >= A.rows && first + cols + 8 > A.cols))) L.whole = 0;
    L.row[0] = A.w + r * A.cols + col0;
    L.row[1] = L.row[0] + 8 * A.cols;
    const int32_t left = (int32_t)cols - (int32_t)(lane & 3) * 8;
    L.left[0] = r < A.rows ? left : 0;
    L.left[1] = r + 8 < A.rows ? left : 0;
    L.off = (uint32_t)(uintptr_t)L.row[0] & 15u;
    return L;
}
// A block's eight weights of one row as four words, weight by weight, pad words outside the tensor.  (VEC: the columns are a multiple of
// eight, so all eight are there or none.)
template <bool VEC>
__device__ __forceinline__ uint4 enc_edge(const EncArgs &A, const uint16_t *p, int32_t left) {
    if (VEC) {
        const uint32_t pads = A.pad | A.pad << 16;
        return left > 0 ? __ldg((const uint4 *)p) : make_uint4(pads, pads, pads, pads);
    }
    uint32_t x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t lo = 2 * i < left ? p[2 * i] : A.pad, hi = 2 * i + 1 < left ? p[2 * i + 1] : A.pad;
        x[i] = lo | hi << 16;
    }
    return make_uint4(x[0], x[1], x[2], x[3]);
}
// The 16 bytes that start `off` bytes (an even number) into two neighbouring pieces.
__device__ __forceinline__ uint4 enc_shifted(const uint4 &p, const uint4 &n, uint32_t off) {
    const bool two = off & 8u, one = off & 4u;
    const uint32_t sel = (off & 2u) ? 0x5432u : 0x3210u;
    const uint32_t a0 = two ? p.z : p.x, a1 = two ? p.w : p.y, a2 = two ? n.x : p.z, a3 = two ? n.y : p.w, a4 = two ? n.z : n.x, a5 = two ? n.w : n.y;
    const uint32_t b0 = one ? a1 : a0, b1 = one ? a2 : a1, b2 = one ? a3 : a2, b3 = one ? a4 : a3, b4 = one ? a5 : a4;
    return make_uint4(__byte_perm(b0, b1, sel), __byte_perm(b1, b2, sel), __byte_perm(b2, b3, sel), __byte_perm(b3, b4, sel));
}
// f(weights in row g, weights in row g + 8) for every block of the chunk in turn, the loads of the next AHEAD blocks under way.  VEC: rows
// start on 16-byte boundaries; otherwise a row's weights are cut out of two pieces.
template <bool VEC, int AHEAD, typename F>
__device__ __forceinline__ void enc_blocks(const EncArgs &A, const EncLane &L, F &&f) {
    const uint4 *pa = (const uint4 *)((const char *)L.row[0] - (VEC ? 0u : L.off)), *pb = (const uint4 *)((const char *)L.row[1] - (VEC ? 0u : L.off));
    uint4 a[AHEAD], b[AHEAD], a1[AHEAD], b1[AHEAD];
    auto load = [&](int i) {
        a[i] = __ldg(pa + 4 * i);
        b[i] = __ldg(pb + 4 * i);
        if (!VEC) {
            a1[i] = __ldg(pa + 4 * i + 1);
            b1[i] = __ldg(pb + 4 * i + 1);
        }
    };
#pragma unroll
    for (int i = 0; i < AHEAD; ++i)
        if ((uint32_t)i < L.whole) load(i);
    uint32_t left = L.whole;
#pragma unroll 1
    while (left) {
        pa += 4 * AHEAD;
        pb += 4 * AHEAD;
#pragma unroll
        for (int i = 0; i < AHEAD; ++i) {
            if (VEC) {
                f(a[i], b[i]);
                if (left > AHEAD) load(i);
            } else {
                const uint4 va = enc_shifted(a[i], a1[i], L.off), vb = enc_shifted(b[i], b1[i], L.off);
                if (left > AHEAD) load(i);
                f(va, vb);
            }
            if (--left == 0) break;
        }
    }
#pragma unroll 1
    for (uint32_t kb = L.whole; kb < L.nkb; ++kb)
        f(enc_edge<VEC>(A, L.row[0] + kb * 32u, L.left[0] - (int32_t)(kb * 32u)), enc_edge<VEC>(A, L.row[1] + kb * 32u, L.left[1] - (int32_t)(kb * 32u)));
}
__device__ __forceinline__ uint32_t lds16(uint32_t addr) {
    uint16_t v;
    asm("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr));
    return v;
}
// FP16: the exponent and the upper mantissa half of a weight, its bits 5 .. 14, are looked up together: a table of 1024 entries in front of
// the lower half's 32.
constexpr uint32_t kPairEntries = 1024;

// Pass 1.  Bound by the read of the tensor (BF16) and by the lookups, whose addresses are byte or halfword dot products of the weights
// as they are, so that a BF16 weight costs 5.5 instructions (8.7 with a shift and a mask per weight, 64 threads a chunk and the
// table read anew for every few of them).  FP16 lengths are 16 bits wide: half as many words for the lanes to meet in.
// Four blocks' loads are in flight (two: 18.7 us instead of 17.3).  Rows off 16-byte boundaries are cut out of two 16-byte loads.
// (11008 x 4096, in a whole call, before / now, us: BF16 23.6 / 17.3, 11007 x 4099 in chunks of 2048 42.9 / 27, FP16 41.6 / 29.0, chunks
// of 512 79 / 50.)
constexpr uint32_t kSizeWarps = 8;           // of a CTA of pass 1
__host__ __device__ constexpr uint32_t size_ctas(bool vec) { return vec ? 3 : 4; }      // of an SM (80 and 64 registers)
// Code lengths and decode table of the blob, as the host writes them; the header's bytes are zero until the last kernel completes it.
__device__ __forceinline__ void enc_fixed_sections(const EncArgs &A) {
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    for (uint32_t i = threadIdx.x; i < (uint32_t)A.desc.off_index / 16; i += blockDim.x) ((uint4 *)A.blob)[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < 256; i += blockDim.x)
        if (A.lengths[i]) A.blob[A.desc.off_codebook + i] = A.lengths[i];
    for (uint32_t i = warp; i < (A.fp16 ? 96u : 256u); i += warps) {
        const uint32_t e = A.code[i], len = e & 31u, field = A.fp16 ? i >> 5 : 0u;
        if (!len) continue;
        uint32_t *const table = (uint32_t *)(A.blob + A.desc.off_lut) + ((size_t)field << A.desc.lut_bits);
        const uint32_t value = len << 16 | (A.fp16 ? (i & 31u) << (10 - 5 * field) : i << 7), seq = __brev(e & ~31u);
        for (uint32_t hi = lane; hi < 1u << (A.desc.lut_bits - len); hi += 32) table[seq | hi << len] = value;
    }
}
template <bool FP16, bool VEC>
__global__ void __launch_bounds__(32 * kSizeWarps, size_ctas(VEC)) encode_size_kernel(const __grid_constant__ EncArgs A) {
    pdl_launch_dependents();
    if (blockIdx.x == gridDim.x - 1) {                       // (the CTA behind those of the chunks)
        enc_fixed_sections(A);
        return;
    }
    __shared__ __align__(4) typename std::conditional<FP16, uint16_t, uint32_t>::type s_len[FP16 ? kPairEntries + 32 : 256];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto length = [&](uint32_t i) -> uint32_t { return A.code[i] ? A.code[i] & 31u : kNoCode; };
    if (FP16) {
        const uint32_t upper = length(32 + lane);
        for (uint32_t e = warp; e < 32; e += kSizeWarps) s_len[32 * e + lane] = min(length(e) + upper, kNoCode);
        if (warp == 0) s_len[kPairEntries + lane] = length(64 + lane);
    } else {
        s_len[threadIdx.x] = length(threadIdx.x);
    }
    __syncthreads();
    const uint32_t table = (uint32_t)__cvta_generic_to_shared(s_len), low = table + 2 * kPairEntries;
    auto bits_of = [&](const uint4 &v) -> uint32_t {
        const uint32_t x[4] = {v.x, v.y, v.z, v.w};
        uint32_t bits = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (FP16) {
                const uint32_t u = x[i] >> 5 & 0x03FF03FFu, l = x[i] & 0x001F001Fu;
                bits += lds16(__dp2a_lo(u, 0x0002u, table)) + lds16(__dp2a_lo(u, 0x0200u, table));
                bits += lds16(__dp2a_lo(l, 0x0002u, low)) + lds16(__dp2a_lo(l, 0x0200u, low));
            } else {
                const uint32_t y = x[i] * 2u;                                // exponents in bytes 1 and 3
                bits += lds_lut(__dp4a(y, 0x00000400u, table)) + lds_lut(__dp4a(y, 0x04000000u, table));
            }
        }
        return bits;
    };
#pragma unroll 1
    for (uint32_t c = blockIdx.x * kSizeWarps + warp; c < A.n_chunks; c += (gridDim.x - 1) * kSizeWarps) {
        const EncLane L = enc_lane(A, c, lane);
        uint32_t ba = 0, bb = 0;
        enc_blocks<VEC, VEC ? 4 : 1>(A, L, [&](const uint4 &va, const uint4 &vb) {
            ba += bits_of(va);
            bb += bits_of(vb);
        });
        const uint32_t most = __reduce_max_sync(0xFFFFFFFFu, max(ba, bb)), sum = __reduce_add_sync(0xFFFFFFFFu, ba + bb);
        if (lane == 0) {
            A.words[c] = most >= kNoCode ? kUnfit : max(1u, (most + A.lag_bits + 31) / 32);
            A.bits[c] = sum;
        }
    }
}

// Record offsets: an exclusive prefix sum of the record sizes (in 128-byte units).  A CTA takes 1024 chunks and sums up the words of all
// chunks in front of them itself (the raw parts in front are known without a sum), so that no CTA waits for another; the one at the end of the
// index, which sees them all, leaves the totals: nothing has to be cleared or added up by atomics in front of this.  Sums over every
// chunk in front grow with the square of the chunks: from kGroupsFrom on a launch of its own leaves those of 1024 chunks each (GROUPS),
// where the chunks' bits were; what is left over behind whole groups are the last scan CTA's own chunks.
// (Time behind pass 1 at 11008 / 88064 / 234 000 / 1.05 M chunks, us: 3.9 / 5.4 / 9.9 / 19.5; pass 1 adding up every 1024 by atomics, behind a launch that
// clears them, 6.3 / 7 / 16 / 30, and 50 us of pass 1 instead of 28 at 88064; without groups 4.2 / 11 / 77 / 224.  The last warp of pass 1 to
// come from every 1024 chunks doing this, for which it has to order its words before the others' counts: 17.3 -> 38 us for that pass.)
constexpr uint64_t kGroupsFrom = 49152;
__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}
__global__ void __launch_bounds__(kScanThreads) encode_groups_kernel(const __grid_constant__ EncArgs A) {
    __shared__ EncGroup s_warp[32];
    pdl_launch_dependents();
    pdl_wait_prior_grid();
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t c = (uint64_t)blockIdx.x * kScanThreads + threadIdx.x;    // (a CTA for every whole group)
    const uint32_t W = __ldcg(A.words + c), bits = __ldcg(A.bits + c);
    const EncGroup sums = {warp_sum(W), warp_sum(bits), __reduce_max_sync(0xFFFFFFFFu, W)};
    if (lane == 0) s_warp[warp] = sums;
    __syncthreads();                                         // (all of the group's bits have been read)
    if (warp) return;
    const EncGroup all = {warp_sum(s_warp[lane].words), warp_sum(s_warp[lane].bits), __reduce_max_sync(0xFFFFFFFFu, s_warp[lane].most)};
    if (lane == 0) *group_at(A.bits, blockIdx.x) = all;
}
template <bool GROUPS>
__global__ void __launch_bounds__(kScanThreads) encode_scan_kernel(const __grid_constant__ EncArgs A) {
    __shared__ unsigned long long s_front[32], s_bits[32];
    __shared__ uint32_t s_words[32], s_most[32];
    pdl_wait_prior_grid();
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, begin = blockIdx.x * kScanThreads;
    const uint64_t c = (uint64_t)begin + tid;
    const uint32_t last = group_count(A.n_chunks);           // the CTA at the end of the index, behind all whole groups
    unsigned long long front = 0, bits = 0;                  // words of the chunks in front of the CTA's; in the last one all chunks' bits and
    uint32_t most = 0;                                       // the most words
    const uint32_t W = c < A.n_chunks ? __ldcg(A.words + c) : 0u;
    if (GROUPS && blockIdx.x <= last) {
        if (blockIdx.x == last) {
            if (c < A.n_chunks) bits = __ldcg(A.bits + c);
            most = W;
        }
        for (uint32_t g = tid; g < blockIdx.x; g += kScanThreads) {
            const EncGroup *const sums = group_at(A.bits, g);
            front += __ldcg(&sums->words);
            if (blockIdx.x == last) {
                bits += __ldcg(&sums->bits);
                most = max(most, __ldcg(&sums->most));
            }
        }
    } else if (blockIdx.x == last) {
        if (c < A.n_chunks) bits = __ldcg(A.bits + c);
        most = W;
#pragma unroll 4
        for (uint32_t i = tid; i < begin; i += kScanThreads) {
            const uint32_t w = __ldcg(A.words + i);
            front += w;
            bits += __ldcg(A.bits + i);
            most = max(most, w);
        }
    } else if (blockIdx.x < last) {
#pragma unroll 8
        for (uint32_t i = tid; i < begin; i += kScanThreads) front += __ldcg(A.words + i);
    }
    uint32_t incl = W;                                      // (1024 chunks: fewer than 2^19 words)
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t n = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= (uint32_t)o) incl += n;
    }
    front = warp_sum(front);
    if (blockIdx.x == last) {
        bits = warp_sum(bits);
        most = __reduce_max_sync(0xFFFFFFFFu, most);
    }
    if (lane == 31) {
        s_words[warp] = incl;
        s_front[warp] = front;
        s_bits[warp] = bits;
        s_most[warp] = most;
    }
    __syncthreads();
    const unsigned long long before = warp_sum(s_front[lane] + (lane < warp ? s_words[lane] : 0u)) + (incl - W);
    if (blockIdx.x == last) {
        bits = warp_sum(s_bits[lane]);
        most = __reduce_max_sync(0xFFFFFFFFu, s_most[lane]);
    }
    if (c <= A.n_chunks) {                                  // (one entry more than chunks: the payload's end)
        const uint32_t raw_full = enc_raw_bytes(A, enc_blocks_of(A, 0)) / kRecordUnit, raw_last = enc_raw_bytes(A, enc_blocks_of(A, A.KC - 1)) / kRecordUnit;
        const uint32_t row = (uint32_t)c / A.KC, kc = (uint32_t)c - row * A.KC;        // raw parts in front: whole rows of chunks, then full chunks of this one
        const unsigned long long at = row * ((uint64_t)(A.KC - 1) * raw_full + raw_last) + (uint64_t)kc * raw_full + 2ull * before;
        A.index[c] = (uint32_t)at;
        if (c == A.n_chunks) *A.totals = {at, bits, 0ull, most, (most == kUnfit ? 1u : 0u) | (at > 0xFFFFFFFFull ? 2u : 0u), 0u};
    } else if (c < ((A.n_chunks + 64) & ~63ull)) {
        A.index[c] = 0;                                     // the section's padding to 256 bytes
    }
}

__device__ __forceinline__ uint32_t shl_pair(uint32_t hi, uint32_t lo, uint32_t n) {       // upper word of (hi:lo) << n % 32
    uint32_t d;
    asm("shf.l.wrap.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(lo), "r"(hi), "r"(n));
    return d;
}
__device__ __forceinline__ uint32_t shr_pair(uint32_t hi, uint32_t lo, uint32_t n) {       // lower word of (hi:lo) >> n % 32
    uint32_t d;
    asm("shf.r.wrap.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(lo), "r"(hi), "r"(n));
    return d;
}
// A sequence being written: its last 64 bits, the newest in bit 0, how many there are so far (bits 0 .. 5 are looked at), and where its
// next word goes, 256 bytes behind the one before: in shared memory (STAGED, the word's first bit on top) or in the record.
template <bool STAGED>
struct EncSequence {
    uint32_t hi, lo, n;
    typename std::conditional<STAGED, uint32_t, uint64_t>::type out;
    __device__ __forceinline__ void push(uint32_t e) {                 // the codeword of a table entry
        hi = shl_pair(hi, lo, e);
        lo = shl_pair(lo, e, e);
    }
    __device__ __forceinline__ void advance(uint32_t by) {             // up to 32 bits were pushed: if that made a word full, out with it
        const uint32_t was = n;
        n += by;
        const uint32_t word = shr_pair(hi, lo, n);
        if constexpr (STAGED)
            asm volatile("{\n\t.reg .pred p, q;\n\t.reg .b32 t;\n\tsetp.ne.u32 q, 0, 0;\n\tlop3.or.b32 t|p, %1, %2, 32, 0x28, q;\n\t"
                         "@p st.shared.u32 [%0], %3;\n\t@p add.u32 %0, %0, 256;\n\t}" : "+r"(out) : "r"(was), "r"(n), "r"(word) : "memory");
        else
            asm volatile("{\n\t.reg .pred p, q;\n\t.reg .b32 t;\n\tsetp.ne.u32 q, 0, 0;\n\tlop3.or.b32 t|p, %1, %2, 32, 0x28, q;\n\t"
                         "@p st.global.u32 [%0], %3;\n\t@p add.u64 %0, %0, 256;\n\t}" : "+l"(out) : "r"(was), "r"(n), "r"(__brev(word)) : "memory");
    }
    __device__ __forceinline__ void put(uint32_t word) {
        if constexpr (STAGED) asm volatile("st.shared.u32 [%0], %1;" ::"r"(out), "r"(word) : "memory");
        else asm volatile("st.global.u32 [%0], %1;" ::"l"(out), "r"(__brev(word)) : "memory");
        out += 256;
    }
    template <typename P>
    __device__ __forceinline__ void finish(P end) {                    // what is left of the last word, and zeros up to the record's end
        if (n & 31u) put(shr_pair(lo, 0u, n));
        while (out < end) put(0u);
    }
    template <bool SHORT>
    __device__ __forceinline__ void append_bf16(const uint4 &v, uint32_t table) {
        const uint32_t x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; i += 2) {
            const uint32_t y0 = x[i] * 2u, y1 = x[i + 1] * 2u;                            // exponents in bytes 1 and 3
            const uint32_t e0 = lds_lut(__dp4a(y0, 0x00000400u, table)), e1 = lds_lut(__dp4a(y0, 0x04000000u, table));
            const uint32_t e2 = lds_lut(__dp4a(y1, 0x00000400u, table)), e3 = lds_lut(__dp4a(y1, 0x04000000u, table));
            push(e0);
            push(e1);
            if (!SHORT) advance(e0 + e1);
            push(e2);
            push(e3);
            advance(SHORT ? e0 + e1 + e2 + e3 : e2 + e3);
        }
    }
    template <bool SHORT>
    __device__ __forceinline__ void append_fp16(const uint4 &v, uint32_t table) {
        const uint32_t x[4] = {v.x, v.y, v.z, v.w}, low = table + 4 * kPairEntries;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t u = x[i] >> 5 & 0x03FF03FFu, l = x[i] & 0x001F001Fu;
            const uint32_t e0 = lds_lut(__dp2a_lo(u, 0x0004u, table)), e1 = lds_lut(__dp2a_lo(l, 0x0004u, low));
            const uint32_t e2 = lds_lut(__dp2a_lo(u, 0x0400u, table)), e3 = lds_lut(__dp2a_lo(l, 0x0400u, low));
            push(e0);
            if (!SHORT) advance(e0);
            push(e1);
            advance(SHORT ? e0 + e1 : e1);
            push(e2);
            if (!SHORT) advance(e2);
            push(e3);
            advance(SHORT ? e2 + e3 : e3);
        }
    }
};

// Pass 2.  The coded part is collected in shared memory, row by row as the record has it: stored straight from the lanes, whose sequences
// run apart, the words go to L2 one by one as partial sectors.  Only records of more rows than a warp has room for (stage_rows, 32 or what
// the code can reach: chunks of 4096 stay below it, 12.7 bits a weight among FP16-trained ones included) are.
// An entry has its codeword on top and its length in the low bits, which is where a funnel shift wants both: two of them move the last
// 64 bits on by a codeword.  Whether a word is full shows in bit 5 of the count; four codewords of up to 8 bits (two of up to 12, an FP16
// weight) are pushed between two such looks.  The words' bits are turned around on their way from shared memory to the record.
// BF16 moves 161 MB in 29.2 us, 0.84 of a copy's rate; FP16 is bound by instruction issue (24 per weight).
// (11008 x 4096, in a whole call, codewords shifted and or-ed into a word / this, us: BF16 42.0 / 29.2, codes of 12 bits 44 / 30.3, 11007 x 4099
// 52 / 37, FP16 in chunks of 2048 83.9 / 52.9, chunks of 512 91 / 57; 28672 x 8192 188 / 141.  Two warps a chunk that meet at a barrier 42.9; stores
// through generic addresses, which one loop could share with the straight ones, 31.8 and 61.6 (FP16).)
template <bool FP16, bool SHORT, bool VEC>
__global__ void __launch_bounds__(32 * kWriteWarps, write_ctas(VEC)) encode_write_kernel(const __grid_constant__ EncArgs A) {
    extern __shared__ __align__(16) uint32_t s_coded[];
    __shared__ uint32_t s_code[FP16 ? kPairEntries + 32 : 256];
    if (!enc_fits(A)) return;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (FP16) {
        const uint32_t h = A.code[32 + lane];
        for (uint32_t i = warp; i < 32; i += kWriteWarps) {
            const uint32_t e = A.code[i];
            s_code[32 * i + lane] = (e & ~31u) | ((h & ~31u) >> (e & 31u)) | ((e & 31u) + (h & 31u));
        }
        if (warp == 0) s_code[kPairEntries + lane] = A.code[64 + lane];
    } else {
        for (uint32_t i = threadIdx.x; i < 256; i += 32 * kWriteWarps) s_code[i] = A.code[i];
    }
    __syncthreads();
    const uint32_t table = (uint32_t)__cvta_generic_to_shared(s_code);
    uint32_t *const stage = s_coded + warp * A.stage_rows * 64;
#pragma unroll 1
    for (uint32_t c = blockIdx.x * kWriteWarps + warp; c < A.n_chunks; c += gridDim.x * kWriteWarps) {
        const EncLane L = enc_lane(A, c, lane);
        const uint32_t W = __ldg(A.words + c), raw_bytes = enc_raw_bytes(A, L.nkb);
        uint8_t *const raw = A.payload + (uint64_t)__ldg(A.index + c) * kRecordUnit;
        uint8_t *raw_to = raw + lane * (FP16 ? 2 : 16);
        auto write = [&](auto &sa, auto &sb) {
            sb.out = sa.out + 128;
            const auto end = sa.out + W * 256u;
            sa.hi = sa.lo = sb.hi = sb.lo = 0;
            sa.n = sb.n = A.lag_bits;
            enc_blocks<VEC, VEC ? 2 : 1>(A, L, [&](const uint4 &va, const uint4 &vb) {
                const uint32_t x[8] = {va.x, va.y, va.z, va.w, vb.x, vb.y, vb.z, vb.w};
                if (FP16) {
                    // signs: bit p for the first weight of pair p, bit 8 + p for its second, row g's pairs first
                    uint32_t u = x[0] & 0x80008000u;
#pragma unroll
                    for (int i = 1; i < 8; ++i) u = u >> 1 | (x[i] & 0x80008000u);
                    *(uint16_t *)raw_to = (uint16_t)__byte_perm(u, 0u, 0x4431);
                    raw_to += 64;
                    sa.template append_fp16<SHORT>(va, table);
                    sb.template append_fp16<SHORT>(vb, table);
                } else {
                    uint32_t word[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {                     // bytes in the raw layout's order: low bytes' mantissas, high bytes' signs
                        const uint32_t m = __byte_perm(x[2 * i], x[2 * i + 1], kRawMantSel), sg = __byte_perm(x[2 * i], x[2 * i + 1], kRawSignSel);
                        asm("lop3.b32 %0, %1, %2, 0x7F7F7F7F, 0xE4;" : "=r"(word[i]) : "r"(m), "r"(sg));
                    }
                    *(uint4 *)raw_to = make_uint4(word[0], word[1], word[2], word[3]);
                    raw_to += 512;
                    sa.template append_bf16<SHORT>(va, table);
                    sb.template append_bf16<SHORT>(vb, table);
                }
            });
            sa.finish(end);
            sb.finish(end + 128);
        };
        if (W <= A.stage_rows) {
            EncSequence<true> sa, sb;
            sa.out = (uint32_t)__cvta_generic_to_shared(stage + lane);
            write(sa, sb);
            __syncwarp();
            for (uint32_t i = lane; i < W * 16; i += 32) {
                const uint4 v = ((const uint4 *)stage)[i];
                ((uint4 *)(raw + raw_bytes))[i] = make_uint4(__brev(v.x), __brev(v.y), __brev(v.z), __brev(v.w));
            }
            __syncwarp();                                             // (the next chunk's words go to the same place)
        } else {
            EncSequence<false> sa, sb;
            sa.out = (uint64_t)(raw + raw_bytes) + 4 * lane;
            write(sa, sb);
        }
        if (FP16 && (L.nkb & 1u)) *(uint16_t *)(raw + L.nkb * 64 + lane * 2) = 0;      // padding of the sign plane
        if (c + 1 == A.n_chunks) {                                    // the zero bytes behind the payload
            uint4 *tail = (uint4 *)(A.payload + __ldcg(&A.totals->payload_units) * kRecordUnit);
            for (uint32_t i = lane; i < kTailSlack / 16; i += 32) tail[i] = make_uint4(0, 0, 0, 0);
        }
    }
}

inline void (*write_kernel_of(bool fp16, bool short_codes, bool vec))(EncArgs) {
    if (fp16) return short_codes ? (vec ? encode_write_kernel<true, true, true> : encode_write_kernel<true, true, false>)
                                 : (vec ? encode_write_kernel<true, false, true> : encode_write_kernel<true, false, false>);
    return short_codes ? (vec ? encode_write_kernel<false, true, true> : encode_write_kernel<false, true, false>)
                       : (vec ? encode_write_kernel<false, false, true> : encode_write_kernel<false, false, false>);
}

// ------------------------------------------------------------------------------ checksum of the records

// The format's checksum of a record is byte-serial (h = (h ^ byte) * P mod 2^64, the FNV-1a hash).  Taken as written it
// leaves the GPU idle: one thread per record spent 193 us on an 11008 x 4096 tensor's 72 MB, most of it waiting for one
// 16-byte load after the other.  Two facts take it apart:
//   * The exclusive-or touches only the low byte of h.  With x_i = the low byte before byte b_i, h ^ b_i = h + d_i with
//     d_i = (x_i ^ b_i) - x_i = b_i - 2 (x_i & b_i), so h_end = h_0 P^n + sum_i d_i P^(n - i): a sum that can be taken in any
//     order once the x_i are known.
//   * The x_i form a chain of their own, x' = (x ^ b) * P mod 256, in which bit k of x' is bit k of x ^ b plus something that
//     depends on the bits below k only.  So if the bits below k are known everywhere, bit k at the end of a stretch of
//     bytes is bit k at its start, exclusive-or a value that the stretch alone determines: an exclusive-or scan over the
//     stretches gives bit k at the start of each.  Eight rounds, one per bit, give every stretch its starting x.
// A warp takes a record; a lane walks four stretches of 4 M bytes at a time, one in each byte of a register (stretch 32 s + l
// in byte s of lane l), each in two halves, which gives it two chains.  A round of a bit takes two instructions per four bytes: the
// low four bits times 3 (P mod 16) stay in their bytes, and so do the upper four, whose two bits of overflow end among the bits that
// the next mask takes away, once what the lower four add to them has been worked out for every byte (C below).  The weighted sum
// goes to the tensor cores as an 8-bit product: the record's bytes (and x & b, lower and upper four bits apart) times the eight byte limbs
// of the powers of P, exact in 32-bit integers.
// Bound by the integer pipe and what keeps it waiting: 40 instructions per four bytes, 20 of them there, at 57 % of its rate (a round
// settles its bit in six dependent shuffles).  (11008 records of 1600 to 1664 words 48.4 -> 43.8 us, 22016 FP16 records 74.6 -> 60, 5504 of twice the
// size 58 -> 41.7, against rounds of four instructions for the upper bits, even and odd bytes apart, in one chain, steps of 7, 6 and 3
// copied piece by piece.  Steps of 5 and 4 only, 24 warps an SM instead of 16: 50.)
constexpr uint64_t kFnvPrime = 1099511628211ull, kFnvStart = 1469598103934665603ull;
__host__ __device__ constexpr uint64_t fnv_pow(uint64_t base, uint32_t e) {
    uint64_t r = 1;
    for (; e; e >>= 1, base *= base)
        if (e & 1u) r *= base;
    return r;
}
constexpr uint64_t fnv_inverse() {                 // P^-1 mod 2^64 (Newton's iteration doubles the correct bits: 3, 6, ..., 96)
    uint64_t x = kFnvPrime;
    for (int i = 0; i < 5; ++i) x *= 2 - kFnvPrime * x;
    return x;
}
constexpr uint64_t kFnvInverse = fnv_inverse();
static_assert(kFnvInverse * kFnvPrime == 1, "inverse of the hash's multiplier");
// The sum's weights for stretches of M words: byte j of stretch 32 s + 4 g + t has weight P^(512 M - (32 s + 4 g + t) 4 M - j).
// The factor of g is taken out (row_factor); limb n of the rest is the B operand: for the product of bytes j = 2 i, 2 i + 1 and
// the same of the stretch's other half, 2 M further on (A registers in this order), lane 4 n + t holds in byte s of word 0 the limb
// for the first, of word 1 for the third; the odd j, rows g + 8 of A, carry one factor P^-1 more.
template <int M>
struct FnvWeights {
    uint32_t b[M][32][2];
    uint64_t row_factor[8];
    constexpr FnvWeights() : b(), row_factor() {
        for (int i = 0; i < M; ++i)
            for (int h = 0; h < 2; ++h)
                for (int t = 0; t < 4; ++t)
                    for (int s = 0; s < 4; ++s) {
                        const uint64_t w = fnv_pow(kFnvPrime, 512 * M - (32 * s + t) * 4 * M - (2 * i + 2 * M * h));
                        for (int n = 0; n < 8; ++n) b[i][4 * n + t][h] |= (uint32_t)(w >> (8 * n) & 0xFFu) << (8 * s);
                    }
        for (int g = 0; g < 8; ++g) row_factor[g] = fnv_pow(kFnvInverse, 16 * M * g);
    }
};
__device__ const FnvWeights<7> g_fnv7{};
__device__ const FnvWeights<6> g_fnv6{};
__device__ const FnvWeights<4> g_fnv4{};
__device__ const FnvWeights<3> g_fnv3{};

__device__ __forceinline__ uint32_t xor_and(uint32_t a, uint32_t b, uint32_t m) {       // (a ^ b) & m
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, 0x28;" : "=r"(d) : "r"(a), "r"(b), "r"(m));
    return d;
}
__device__ __forceinline__ uint32_t byte_perm(uint32_t a, uint32_t b, uint32_t sel) { return __byte_perm(a, b, sel); }
__device__ __forceinline__ void mma_u8(int32_t (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.u8.u8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// A record's hash on its way: every lane's part of it as if the record ended here (their sum is the hash), and the low byte, the same in
// all lanes.
struct FnvState {
    uint64_t part;
    uint32_t low;
};
// 512 M bytes of a record (`words`, in shared memory).
template <int M>
__device__ __forceinline__ void fnv_step(FnvState &F, const uint32_t *words, const FnvWeights<M> &wt, uint32_t lane, uint32_t three) {
    constexpr int N = 4 * M, H = 2 * M;            // bytes of a stretch, of its halves
    constexpr uint32_t kLow = 0x0F0F0F0Fu, kHigh = 0xF0F0F0F0u;
    uint32_t G[N];                                 // G[j]: byte j of the lane's four stretches
    uint32_t all[2] = {0, 0};
#pragma unroll
    for (int m = 0; m < M; ++m) {
        const uint32_t a = words[lane * M + m], b = words[(32 + lane) * M + m], c = words[(64 + lane) * M + m], d = words[(96 + lane) * M + m];
        const uint32_t t0 = byte_perm(a, b, 0x5140), t1 = byte_perm(c, d, 0x5140), t2 = byte_perm(a, b, 0x7362), t3 = byte_perm(c, d, 0x7362);
        G[4 * m] = byte_perm(t0, t1, 0x5410);
        G[4 * m + 1] = byte_perm(t0, t1, 0x7632);
        G[4 * m + 2] = byte_perm(t2, t3, 0x5410);
        G[4 * m + 3] = byte_perm(t2, t3, 0x7632);
    }
#pragma unroll
    for (int j = 0; j < N; ++j) all[j / H] ^= G[j];
    const uint32_t first = F.low * 0x01010101u;
    uint32_t X[2] = {0, 0};                        // the halves' starting low bytes, as far as they are known
    // e: the bits `bits` of each byte at the end of a half if they were 0 at its start; settles them in X
    auto settle = [&](const uint32_t (&e)[2], uint32_t bits, bool two = false) {
        const uint32_t own = xor_and(e[0], e[1], bits);
        uint32_t v = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1)
            asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 up;\n\tshfl.sync.up.b32 up|p, %0, %1, 0, 0xFFFFFFFF;\n\t@p xor.b32 %0, %0, up;\n\t}" : "+r"(v) : "r"(o));
        // what the stretches in the bytes below add (one bit: the lowest of the sum of their up to three totals is the exclusive or)
        const uint32_t total = __shfl_sync(0xFFFFFFFFu, v, 31);
        const uint32_t before = two ? total << 8 ^ total << 16 ^ total << 24 : total * 0x01010100u;
        const uint32_t at = v ^ own ^ before ^ first;
        X[0] |= at & bits;
        X[1] |= xor_and(at, e[0], bits);
    };
    // (bits 0 and 1 together: what bit 0 adds to bit 1 over a half's even number of bytes does not depend on where it started)
#pragma unroll
    for (uint32_t k = 1; k <= 3; ++k) {
        uint32_t z[2] = {X[0], X[1]};
#pragma unroll
        for (int j = 0; j < H; ++j)
#pragma unroll
            for (int h = 0; h < 2; ++h) z[h] = xor_and(z[h], G[h * H + j], kLow) * three;
        settle(z, k == 1 ? 0x03030303u : 0x01010101u << k, k == 1);
    }
    // The low four bits are known.  What they add to the upper four of (x ^ b) * P mod 256 is worked out once: P mod 256 is 16 * 11 + 3.
    int32_t sb[4] = {0, 0, 0, 0}, sv[4] = {0, 0, 0, 0};
    uint32_t C[N], zl[2] = {X[0], X[1]}, odd[2] = {all[0], all[1]};
    auto weights = [&](int i) -> uint2 { return __ldg((const uint2 *)&wt.b[i][lane][0]); };
    // four bytes j of half h: f(v's, number of the first byte)
#pragma unroll
    for (int j = 0; j < H; j += 2) {
        uint32_t v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int h = i >> 1, n = h * H + j + (i & 1);
            const uint32_t g = G[n], y = xor_and(zl[h], g, kLow);
            v[i] = zl[h] & g & kLow;
            zl[h] = y * three;
            C[n] = y * 176u + (zl[h] & kHigh);
            odd[h] ^= C[n];
        }
        const uint2 w = weights(j / 2);
        mma_u8(sb, G[j], G[j + 1], G[H + j], G[H + j + 1], w.x, w.y);
        mma_u8(sv, v[0], v[1], v[2], v[3], w.x, w.y);
    }
    settle(odd, 0x10101010u);
#pragma unroll 1
    for (uint32_t k = 5; k <= 7; ++k) {
        uint32_t z[2] = {X[0], X[1]};
#pragma unroll
        for (int j = 0; j < H; ++j)
#pragma unroll
            for (int h = 0; h < 2; ++h) z[h] = xor_and(z[h], G[h * H + j], kHigh) * three + C[h * H + j];
        settle(z, 0x01010101u << k);
    }
    uint32_t z[2] = {X[0], X[1]};
#pragma unroll
    for (int j = 0; j < H; j += 2) {
        uint32_t v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int h = i >> 1, n = h * H + j + (i & 1);
            v[i] = z[h] & G[n] & kHigh;
            z[h] = xor_and(z[h], G[n], kHigh) * three + C[n];
        }
        const uint2 w = weights(j / 2);
        mma_u8(sv, v[0], v[1], v[2], v[3], w.x, w.y);
    }
    F.low = __shfl_sync(0xFFFFFFFFu, (z[1] & kHigh) | (zl[1] & kLow), 31) >> 24;
    const uint32_t t = lane & 3u;
    auto limbs = [&](int32_t lo, int32_t hi) -> uint64_t { return ((uint64_t)(int64_t)lo + ((uint64_t)(int64_t)hi << 8)) << (16u * t); };
    const uint64_t sum = (limbs(sb[0] - 2 * sv[0], sb[1] - 2 * sv[1]) + limbs(sb[2] - 2 * sv[2], sb[3] - 2 * sv[3]) * kFnvInverse) *
                         __ldg((const unsigned long long *)&wt.row_factor[lane >> 2]);
    constexpr uint64_t kOver = fnv_pow(kFnvPrime, 512 * M);
    F.part = F.part * kOver + sum;
}

// What the totals add to the header.
__host__ __device__ inline void enc_fill_totals(huffllm_desc &d, const volatile EncTotals &t) {
    d.max_words = t.max_words;
    d.payload_bytes = t.payload_units * kRecordUnit;
    d.blob_bytes = d.off_payload + d.payload_bytes + kTailSlack;
    d.coded_bits = t.coded_bits;
    d.payload_checksum = t.checksum;
}

// One thread of every checksum CTA, with the CTA's sum; the last one to come completes the header.
__device__ __forceinline__ void finish_checksum(const EncArgs &A, unsigned long long term) {
    atomicAdd(&A.totals->checksum, term);
    __threadfence();
    if (atomicAdd(&A.totals->summed, 1u) != gridDim.x - 1u) return;
    __threadfence();
    huffllm_desc d = A.desc;
    enc_fill_totals(d, *(const volatile EncTotals *)A.totals);
    *(huffllm_desc *)A.blob = d;
}

// A warp goes through its records a step (7, 6, 4 or 3 times 512 bytes) at a time, while a bulk copy brings the next step's bytes to its
// other buffer.  (Beside the packing in one kernel, which would leave the record in shared memory, 110 us instead of 46 + 51 by the kernels
// of the time: too few warps to pack with.)
constexpr uint32_t kSumWarps = 4, kSumCtas = 4, kSumBuf = 7 * 128;       // CTAs of an SM (128 registers); words of a step
constexpr uint32_t kSumSmem = kSumWarps * 2 * kSumBuf * 4;
__global__ void __launch_bounds__(32 * kSumWarps, kSumCtas) encode_checksum_kernel(const __grid_constant__ EncArgs A) {
    extern __shared__ __align__(16) uint32_t s_steps[];
    __shared__ unsigned long long s_term[kSumWarps];
    __shared__ __align__(8) uint64_t s_landed[kSumWarps][2];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_chunks = (uint32_t)A.n_chunks, stride = gridDim.x * kSumWarps;
    if (!enc_fits(A)) return;
    uint32_t *const buf = s_steps + warp * 2 * kSumBuf;
    const uint32_t bar = smem_u32(&s_landed[warp][0]);
    if (lane == 0) {
        mbar_init(bar, 1);
        mbar_init(bar + 8, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    // 3, as a value the compiler does not know: times 3 as a shifted addition would join the logic instructions on the
    // integer pipe that bounds this kernel, as a multiplication it runs beside them
    const uint32_t three = 3u + (uint32_t)(A.n_chunks >> 32);
    // a step's size: two of 4 rather than 7 and 3, FP16 records of 4 KB among others
    auto step_of = [](uint32_t left) -> uint32_t { return left > 32u ? 7u : left > 28u ? 4u : left > 24u ? 7u : left > 16u ? 6u : left > 12u ? 4u : 3u; };
    // (sizes and places in the format's units of 128 bytes: `at`, from the payload on; as many of the `left` as a step may have)
    auto fetch = [&](uint32_t at, uint32_t left, uint32_t to) {
        if (lane) return;
        const uint32_t bytes = min(left, 4 * step_of(left)) * kRecordUnit;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(bar + 8 * to, bytes);
        bulk_g2s(smem_u32(buf + to * kSumBuf), A.payload + (uint64_t)at * kRecordUnit, bytes, bar + 8 * to);
    };
    auto open = [&](uint32_t r, uint32_t &at, uint32_t &left) {
        left = 0;
        if (r >= n_chunks) return;
        at = __ldg(A.index + r);
        left = __ldg(A.index + r + 1) - at;
    };
    const FnvState start = {lane == 0 ? kFnvStart : 0ull, (uint32_t)kFnvStart & 0xFFu};
    FnvState F = start;
    // the record at hand, from the step at hand on, and the warp's next one
    uint32_t c = blockIdx.x * kSumWarps + warp, step = 0, at = 0, left, next_at = 0, next_left;
    open(c, at, left);
    open(c + stride, next_at, next_left);
    if (lane == 0) s_term[warp] = 0;
    if (left) fetch(at, left, 0);
#pragma unroll 1
    for (; left; ++step) {
        const uint32_t which = step & 1u, m = step_of(left), here = min(left, 4 * m);
        const bool last = left <= 4 * m;
        __syncwarp();                                        // (all lanes are done with the other buffer)
        if (!last) fetch(at + 4 * m, left - 4 * m, which ^ 1u);
        else if (next_left) fetch(next_at, next_left, which ^ 1u);
        uint32_t spins = 0;
        bool done = mbar_try_wait(bar + 8 * which, step >> 1 & 1u);
        while (!__all_sync(0xFFFFFFFFu, done) && ++spins < kWaitLimit) done = mbar_try_wait(bar + 8 * which, step >> 1 & 1u);
        if (spins == kWaitLimit) break;                      // (the copy never came)
        uint32_t *const words = buf + which * kSumBuf;
        for (uint32_t i = here * 32 + lane; i < m * 128; i += 32) words[i] = 0;        // (zeros behind the record add nothing)
        __syncwarp();
        if (m == 7u) fnv_step<7>(F, words, g_fnv7, lane, three);
        else if (m == 6u) fnv_step<6>(F, words, g_fnv6, lane, three);
        else if (m == 4u) fnv_step<4>(F, words, g_fnv4, lane, three);
        else fnv_step<3>(F, words, g_fnv3, lane, three);
        if (last) {
            uint64_t h = F.part;
#pragma unroll
            for (int o = 16; o; o >>= 1) h += __shfl_xor_sync(0xFFFFFFFFu, (unsigned long long)h, o);
            // the zero bytes behind the record multiplied h by P each
            constexpr uint64_t kUnitBack = fnv_pow(kFnvInverse, kRecordUnit);
            for (uint32_t p = here; p < 4 * m; ++p) h *= kUnitBack;
            if (lane == 0) s_term[warp] += h * (2ull * c + 1);
            F = start;
            c += stride;
            at = next_at;
            left = next_left;
            open(c + stride, next_at, next_left);            // (wanted a record later)
        } else {
            at += 4 * m;
            left -= 4 * m;
        }
    }
    if (left) {
        // The call fails.  What is under way to the shared memory, this step and the one behind it, is waited for once more, again with a limit,
        // before another CTA may get it.
        atomicOr(&A.totals->bad, 4u);
        const uint32_t under_way = left > 4 * step_of(left) || next_left ? 2u : 1u;
        for (uint32_t i = 0; i < under_way; ++i, ++step)
            for (uint32_t spins = 0; spins < kWaitLimit && !mbar_try_wait(bar + 8 * (step & 1u), step >> 1 & 1u); ++spins) {}
    }
    __syncthreads();
    if (threadIdx.x) return;
    unsigned long long term = 0;
    for (uint32_t i = 0; i < kSumWarps; ++i) term += s_term[i];
    finish_checksum(A, term);
}

static uint32_t reverse_word(uint32_t v) {
    v = (v >> 1 & 0x55555555u) | (v & 0x55555555u) << 1;
    v = (v >> 2 & 0x33333333u) | (v & 0x33333333u) << 2;
    v = (v >> 4 & 0x0F0F0F0Fu) | (v & 0x0F0F0F0Fu) << 4;
    return v << 24 | (v & 0xFF00u) << 8 | (v >> 8 & 0xFF00u) | v >> 24;
}

// The device's SMs, whose number the checksum's CTAs go by, and the kernel's shared memory allowed, once per device.
static cudaError_t prepare_checksum(int *sms) {
    static std::atomic<int> known[64];               // set twice by racing threads at worst: to the same value
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64 && (*sms = known[dev].load(std::memory_order_acquire)) != 0) return cudaSuccess;
    if ((e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(encode_checksum_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSumSmem)) != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) known[dev].store(*sms, std::memory_order_release);
    return cudaSuccess;
}

// The same with a thread per record, as the hash is written: six instructions per byte where the warps above spend ten, but one byte
// after the other, 20 cycles each (16 of them the exclusive-or and the multiplication that wait for one another), which is
// the time of a launch as long as every scheduler has a warp at most.  Four pieces of 32 bytes are on their way to registers (with
// one of 16 bytes, 28672 x 8192 took 215 us instead of 145).  Both grow with the record, so the line is a number of records, which rises
// with their size because from 19000 on threads share schedulers.  (Warps / threads, us, 11008 x 4096: chunks of 512 119 / 33, 1024 66 / 35,
// 2048 45.5 / 47.0 and FP16 60.0 / 51.8, 4096 43.8 / 70; 28672 x 8192 in chunks of 4096 180 / 145, 28672 x 4096 in chunks of 8192 91 / 126.)
constexpr uint32_t kEachThreads = 128;
inline bool checksum_each(uint64_t n_chunks, uint32_t chunk_elems) { return n_chunks >= 13000ull + 4ull * chunk_elems; }
inline uint32_t each_threads(uint64_t n_chunks) { return n_chunks >= 65536 ? kEachThreads : 32; }       // (few records: a warp for every scheduler)
struct Piece32 {
    uint32_t w[8];
};
__device__ __forceinline__ Piece32 ldg_32(const uint8_t *p) {
    Piece32 v;
    asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v.w[0]), "=r"(v.w[1]), "=r"(v.w[2]), "=r"(v.w[3]), "=r"(v.w[4]), "=r"(v.w[5]), "=r"(v.w[6]), "=r"(v.w[7])
                 : "l"(p)
                 : "memory");
    return v;
}
__global__ void __launch_bounds__(kEachThreads) encode_checksum_each_kernel(const __grid_constant__ EncArgs A) {
    __shared__ unsigned long long s_term[kEachThreads / 32];
    const uint64_t c = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (!enc_fits(A)) return;
    unsigned long long term = 0;
    if (c < A.n_chunks) {
        constexpr uint32_t kPrimeLow = (uint32_t)kFnvPrime;          // P = 2^40 + this
        static_assert(kFnvPrime == (1ull << 40) + kPrimeLow, "the hash's multiplier");
        const uint32_t r0 = A.index[c];
        uint32_t units = A.index[c + 1] - r0;                        // (at least one)
        const uint8_t *p = A.payload + (uint64_t)r0 * kRecordUnit;
        uint32_t lo = (uint32_t)kFnvStart, hi = (uint32_t)(kFnvStart >> 32);
        Piece32 v[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) v[s] = ldg_32(p + 32 * s);
#pragma unroll 1
        for (; units; --units) {
            p += kRecordUnit;
#pragma unroll
            for (int s = 0; s < 4; ++s) {
#pragma unroll
                for (int k = 0; k < 32; ++k) {
                    const uint32_t x = lo ^ ((v[s].w[k >> 2] >> (8 * (k & 3))) & 0xFFu);
                    const uint64_t m = (uint64_t)x * kPrimeLow;
                    lo = (uint32_t)m;
                    hi = hi * kPrimeLow + (uint32_t)(m >> 32) + (x << 8);
                }
                if (units > 1) v[s] = ldg_32(p + 32 * s);
            }
        }
        term = ((unsigned long long)hi << 32 | lo) * (2 * c + 1);
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) term += __shfl_xor_sync(0xFFFFFFFFu, term, o);
    if ((threadIdx.x & 31) == 0) s_term[threadIdx.x >> 5] = term;
    __syncthreads();
    if (threadIdx.x) return;
    term = 0;
    for (uint32_t i = 0; i < blockDim.x / 32; ++i) term += s_term[i];
    finish_checksum(A, term);
}

}  // namespace huffllm

using namespace huffllm;

extern "C" huffllm_status huffllm_encode_device_scratch_bytes(uint64_t rows, uint64_t cols, uint32_t chunk_elems, size_t *bytes) {
    clear_error();
    if (!bytes) return fail(HUFFLLM_ERR_INVALID_ARG, "null output");
    if (rows == 0 || cols == 0 || rows > (1ull << 31) || cols > (1ull << 31) || chunk_elems % 512 || chunk_elems < 512 || chunk_elems > 16384)
        return fail(HUFFLLM_ERR_INVALID_ARG, "bad shape or chunk_elems");
    const uint64_t Kc = chunk_elems / kTileRows, n_chunks = ((rows + 15) / 16) * ((cols + Kc - 1) / Kc);
    *bytes = (size_t)scratch_bytes(n_chunks);
    return HUFFLLM_OK;
}

extern "C" huffllm_status huffllm_encode_device(const huffllm_codebook *cb, const uint16_t *w_dev, uint64_t rows, uint64_t cols,
                                                uint32_t chunk_elems, void *blob_dev, size_t blob_cap, void *scratch_dev,
                                                size_t scratch_bytes, huffllm_desc *desc, huffllm_stream stream) {
    clear_error();
    if (!cb || !w_dev || !blob_dev || !scratch_dev || !desc) return fail(HUFFLLM_ERR_INVALID_ARG, "null pointer");
    size_t need = 0;
    huffllm_status st = huffllm_encode_device_scratch_bytes(rows, cols, chunk_elems, &need);
    if (st != HUFFLLM_OK) return st;
    if (scratch_bytes < need) return fail(HUFFLLM_ERR_BUFFER_TOO_SMALL, "scratch needs %llu bytes", (unsigned long long)need);
    if (((uintptr_t)w_dev & 1u) || ((uintptr_t)blob_dev & 255u) || ((uintptr_t)scratch_dev & 255u))
        return fail(HUFFLLM_ERR_INVALID_ARG, "blob and scratch must be 256-byte aligned");
    const uint32_t Kc = chunk_elems / kTileRows, RG = (uint32_t)((rows + 15) / 16), KC = (uint32_t)((cols + Kc - 1) / Kc);
    huffllm_desc d;
    fill_desc_fixed(cb, rows, cols, chunk_elems, Kc, RG, KC, &d);
    if (blob_cap < d.off_payload) return fail(HUFFLLM_ERR_BUFFER_TOO_SMALL, "blob capacity below the fixed sections");
    if (d.n_chunks > 0x7FFFFFFFull) return fail(HUFFLLM_ERR_UNSUPPORTED, "too many chunks");

    cudaStream_t s = (cudaStream_t)stream;
    uint8_t *blob = (uint8_t *)blob_dev, *scr = (uint8_t *)scratch_dev;
    EncArgs A = {};
    A.w = w_dev;
    A.rows = rows;
    A.cols = cols;
    A.n_chunks = d.n_chunks;
    A.Kc = Kc;
    A.KC = KC;
    A.fp16 = d.dtype == HUFFLLM_FP16 ? 1u : 0u;
    A.lag_bits = d.lag_bits;
    A.pad = d.pad_word;
    A.vec_ok = (cols % 8 == 0 && ((uintptr_t)w_dev & 15u) == 0) ? 1u : 0u;
    A.max_units = blob_cap >= d.off_payload + kTailSlack ? (blob_cap - d.off_payload - kTailSlack) / kRecordUnit : 0;
    A.totals = (EncTotals *)scr;
    A.bits = scratch_bits(scr);
    A.words = scratch_words(scr, d.n_chunks);
    A.index = (uint32_t *)(blob + d.off_index);
    A.blob = blob;
    A.payload = blob + d.off_payload;
    A.desc = d;
    code_length_section(cb, A.lengths);
    uint8_t len[256];
    uint32_t bits[256], longest = 1;
    encoder_tables(cb, len, bits);
    for (int i = 0; i < 256; ++i) {
        A.code[i] = reverse_word(bits[i]) | len[i];
        longest = std::max<uint32_t>(longest, len[i]);
    }
    const uint32_t steps = Kc / kBlockCols * 8 * (A.fp16 ? 3 : 1), most_words = (d.lag_bits + steps * longest + 31) / 32;
    A.stage_rows = std::min(most_words, 32u);

    cudaError_t e;
    auto cuda_fail = [&](const char *what) { return fail(HUFFLLM_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e)); };
    const auto size_kernel = A.fp16 ? (A.vec_ok ? encode_size_kernel<true, true> : encode_size_kernel<true, false>)
                                    : (A.vec_ok ? encode_size_kernel<false, true> : encode_size_kernel<false, false>);
    const auto write_kernel = write_kernel_of(A.fp16 != 0, longest <= 8, A.vec_ok != 0);
    const uint32_t smem = kWriteWarps * A.stage_rows * 256;
    int sms = 0;
    if ((e = prepare_checksum(&sms)) != cudaSuccess) return cuda_fail("device attributes");
    // (What the GPU is given comes last and without a pause: it waits for the host otherwise.  The small kernels behind pass 1 start while it
    // ends.  Not the passes behind them, whose CTAs go where there is room first and then share what they find there unevenly: 11008 x 4096
    // both passes 3 us later, chunks of 2048 with a thread per record 36.)
    auto ctas = [&](uint32_t warps, uint32_t per_sm) { return (uint32_t)std::min<uint64_t>((d.n_chunks + warps - 1) / warps, (uint64_t)per_sm * sms); };
    auto launch = [&](void (*kernel)(EncArgs), uint32_t grid, uint32_t threads, uint32_t shared, bool early) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(grid);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = shared;
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = early ? 1 : 0;
        return cudaLaunchKernelEx(&cfg, kernel, A);
    };
    const bool groups = d.n_chunks >= kGroupsFrom;
    const bool a_thread_each = checksum_each(d.n_chunks, chunk_elems);
    const uint32_t each = each_threads(d.n_chunks);
    if ((e = launch(size_kernel, std::min(ctas(kSizeWarps, size_ctas(A.vec_ok)) + 1, size_ctas(A.vec_ok) * (uint32_t)sms), 32 * kSizeWarps, 0, false)) != cudaSuccess ||
        (groups && (e = launch(encode_groups_kernel, group_count(d.n_chunks), kScanThreads, 0, true)) != cudaSuccess) ||
        (e = launch(groups ? encode_scan_kernel<true> : encode_scan_kernel<false>, (uint32_t)((d.n_chunks + 64 + kScanThreads - 1) / kScanThreads), kScanThreads, 0, true)) != cudaSuccess ||
        (e = launch(write_kernel, ctas(kWriteWarps, write_ctas(A.vec_ok)), 32 * kWriteWarps, smem, false)) != cudaSuccess ||
        (e = a_thread_each ? launch(encode_checksum_each_kernel, (uint32_t)((d.n_chunks + each - 1) / each), each, 0, false)
                           : launch(encode_checksum_kernel, ctas(kSumWarps, kSumCtas), 32 * kSumWarps, kSumSmem, false)) != cudaSuccess)
        return cuda_fail("encoder launches");
    EncTotals tot;
    if ((e = cudaMemcpyAsync(&tot, scr, sizeof(tot), cudaMemcpyDeviceToHost, s)) != cudaSuccess || (e = cudaStreamSynchronize(s)) != cudaSuccess)
        return cuda_fail("encoder");
    if (tot.bad & 4u) return fail(HUFFLLM_ERR_CUDA, "a copy of a record did not arrive");
    if (tot.bad & 1u) return fail(HUFFLLM_ERR_INVALID_ARG, "a weight uses a symbol the codebook has no codeword for");
    if (tot.bad & 2u) return fail(HUFFLLM_ERR_UNSUPPORTED, "payload exceeds the 32-bit record index");
    enc_fill_totals(d, tot);
    if (tot.payload_units > A.max_units)
        return fail(HUFFLLM_ERR_BUFFER_TOO_SMALL, "blob needs %llu bytes, capacity is %llu", (unsigned long long)d.blob_bytes, (unsigned long long)blob_cap);
    *desc = d;
    return HUFFLLM_OK;
}
