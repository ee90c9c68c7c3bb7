// Small-batch product on the 5th-generation tensor cores (tcgen05), batch 9..64.
//
// Same decoder as the matrix-vector kernel (one table lookup per weight, two bit sequences per lane), but the
// decoded 16-bit weights are not multiplied from registers: every warp stores its 16 rows x 32 columns of a
// block into TENSOR MEMORY as the A operand of a 128-row tile, the activations of the same 32 columns go to
// shared memory as the B operand, and one thread issues tcgen05.mma (M = 128, N = padded batch, K = 16)
// whose fp32 accumulator also lives in tensor memory.  The decoded weights are consumed where they are
// produced (Section 1 of the paper: decompress only to multiply) and one pass over the compressed bytes
// serves the whole batch; the tensor pipe only takes the batch-fold of multiply-adds off the issue slots.
//
// Geometry of a CTA: 4 tiles of 8 warps; a tile is 128 rows (8 row groups of 16), warp (q = warp % 4, h = warp / 4 % 2)
// of a tile owns tensor-memory lanes 32 q + 16 h .. + 15, which is what the 16x256b store shape of a warp can reach.
// The tiles are dealt to `tc_slices` slices of the columns (1, 2 or 4): with one slice the four tiles are four times 128
// rows; with four they are the same 128 rows in four neighbouring column ranges, whose accumulators the epilogue adds.
// More slices mean fewer rows per CTA and therefore fewer CTAs per row to add up in global memory: that sum is what a
// launch over a small matrix would otherwise spend a third of its time on (a 4096 x 4096 matrix at 32 vectors: 16 column
// ranges of 496 rows, of which the last CTA to finish read 1 MB of pieces for 9 of the launch's 27 us).  The host picks the
// slices with the column ranges (tc_best).
// The CTA's LAST warp does not decode: it issues the MMAs.  A CTA's rows are therefore 8 row groups per tile of a slice,
// less one where all four tiles are in use (31, 15 or 7: the last 16 rows of a slice's last tile are never read).
// Tensor memory (512 columns): 4 accumulators of N columns, then stages x 4 tiles x 32 columns of A (a stage = two
// blocks of 32 weight columns = four K = 16 steps; a chunk's odd last block makes a stage of one block).
// A work item is (the CTA's row groups) x (a range of column chunks); partial results of the ranges of one row tile are
// added in a fixed order by whoever finishes last (arrival counters, nobody waits).
//
// Stage protocol: a decoder warp fills its rows of stage s of A (each block into its half of the stage as soon as it is
// decoded), arrives on the stage's "full" mbarrier and goes on decoding; no warp waits for another one except through the
// depth of the stage ring.  The activations of a slice are brought to shared memory by a warp that does not decode (8-byte
// cp.async, as the B operand's permuted columns want them); the issuer waits for a stage to be full, issues its MMAs and a
// tcgen05.commit onto the stage's "empty" mbarrier, which the others wait on (with a limit) before they reuse the stage.
// (With the issue taking turns among the decoder warps and a barrier after every block, each block cost the CTA its decode
// time plus the 2000 cycles one warp needs to issue the MMAs: that warp had to decode its next block before the next barrier
// could open.  With the activations carried through the first decoder warps' registers, every decoder paid for their
// predicates, pointers and sixteen registers; with cp.async from those warps, all waited for them: a 7B-shaped layer at 32
// vectors 153 us against 134.)
// BF16 and FP16 {1,5,5,5} blobs share the kernel (template parameter FMT): tables, raw part and operand format differ.
#include <atomic>
#include <type_traits>

#include "decode_common.cuh"

namespace huffllm {

constexpr int kTcStages = 3;      // most stages; A.tc_stages are in use (shared memory is short at wide paddings and many slices)
constexpr int kTcTiles = 4;
constexpr uint32_t kPollsAlone = 64;      // polls of a barrier before a warp sees to it that the kernel in front is over
static_assert(kPollsAlone < kWaitLimit, "a wait that ran out is reported behind the kernel in front");

// 8 bytes global -> shared without a register in between.
__device__ __forceinline__ void cp_async8(uint32_t dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t smem_dst, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// 16 lanes x 512 bits: thread (g = lane / 4, t = lane % 4) supplies, for rows g and g + 8, the 32-bit columns
// 2t, 2t+1 (r0, r1 | r2, r3) and 8 + 2t, 8 + 2t + 1 (r4, r5 | r6, r7).
__device__ __forceinline__ void tc_st_16x256b_x2(uint32_t taddr, const uint32_t (&r)[8]) {
    asm volatile("tcgen05.st.sync.aligned.16x256b.x2.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr), "r"(r[0]),
                 "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}
__device__ __forceinline__ void tc_mma_f16_tmem_a(uint32_t d, uint32_t a, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d),
        "r"(a), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
template <int N>
__device__ __forceinline__ void tc_ld_32x32b(uint32_t taddr, uint32_t (&v)[N]);
template <>
__device__ __forceinline__ void tc_ld_32x32b<2>(uint32_t taddr, uint32_t (&v)[2]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(v[0]), "=r"(v[1]) : "r"(taddr) : "memory");
}
template <>
__device__ __forceinline__ void tc_ld_32x32b<4>(uint32_t taddr, uint32_t (&v)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(taddr) : "memory");
}
template <>
__device__ __forceinline__ void tc_ld_32x32b<8>(uint32_t taddr, uint32_t (&v)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(taddr)
                 : "memory");
}
template <>
__device__ __forceinline__ void tc_ld_32x32b<16>(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]),
          "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr)
        : "memory");
}
template <>
__device__ __forceinline__ void tc_ld_32x32b<32>(uint32_t taddr, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, "
        "%18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]),
          "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]),
          "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]),
          "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr)
        : "memory");
}

// Shared-memory matrix descriptor of a K-major operand without swizzle: 8-row x 16-byte core matrices,
// `lbo` bytes between core matrices along K, `sbo` bytes between 8-row groups.  Low word: address and lbo, in units of 16 bytes.
__device__ __forceinline__ uint32_t smem_desc_lo(uint32_t addr, uint32_t lbo) { return ((addr & 0x3FFFFu) >> 4) | ((lbo >> 4) << 16); }
__device__ __forceinline__ uint64_t smem_desc(uint32_t lo, uint32_t sbo) { return (uint64_t)lo | ((uint64_t)(sbo >> 4) << 32) | (1ull << 46); }
// One thread of the (converged) warp.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}

// LB = table index bits; NPAD = batch rounded up to 16, 32 or 64 (the MMA's N); FMT = 0: BF16 blobs, 1: FP16 {1,5,5,5} blobs, 2 to 4: those with flat mantissa codes, see huff_kernel
// (three tables, sign words as the raw part, f16 operands).
// MULTI: the launch works through several matrices (a launch over one matrix reads its arguments without an index).
template <int LB, int NPAD, int FMT, bool MULTI>
__global__ void __launch_bounds__(1024, 1) huff_gemm_tc_kernel(const __grid_constant__ TcArgs T) {
    const KernelArgs &A = T.k;
    constexpr uint32_t kRawBlock = FMT ? 64u : 512u;          // raw bytes of one block of a record
    constexpr uint32_t kRawLane = FMT ? 2u : 16u;             // of which one lane's share
    auto raw_part = [](uint32_t nkb) -> uint32_t { return FMT ? (nkb * 64u + 127u) & ~127u : nkb * 512u; };
    auto load_raw = [](const uint8_t *p) -> uint4 {
        if (FMT) return make_uint4(ldg_stream2(p), 0, 0, 0);
        return ldg_stream16(p);
    };
    constexpr Decoder D = decoder_of(LB, FMT);
    constexpr uint32_t kBStage = NPAD * 128;                // bytes of B per slice and stage: NPAD rows x 64 columns (two blocks) of bf16
    constexpr uint32_t kLbo = 128, kSbo = 1024;             // core matrices: 8 along K side by side, then the next 8 rows
    constexpr uint32_t kACol0 = kTcTiles * NPAD;            // first tensor-memory column of the A stages
    // instruction descriptor: fp32 accumulate, bf16 x bf16, both K-major, N = NPAD, M = 128
    constexpr uint32_t kIdesc = (1u << 4) | (FMT ? 0u : (1u << 7) | (1u << 10)) | ((uint32_t)(NPAD >> 3) << 17) | ((128u >> 4) << 24);

    extern __shared__ __align__(128) uint8_t dyn_smem[];
    __shared__ __align__(8) uint64_t bars[kMaxWarps * 2];   // per warp: its two coded-copy barriers
    __shared__ __align__(8) uint64_t ring_bars[2 * kTcStages];   // stage may be refilled (arrived on by tcgen05.commit); every decoder warp's share is in place
    __shared__ uint32_t s_tmem_base, s_last;

    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    pdl_launch_dependents();   // the next kernel in the stream may be scheduled early; it waits for this one before it reads results
    // the matrix this CTA works in (the launch's CTAs are dealt to its matrices; a CTA builds one table), and the CTA's
    // number among that matrix's CTAs: it takes the matrix's work items J, J + n_cta, ...
    uint32_t mi = 0;
    if (MULTI)
        while (mi + 1 < A.n_mats && blockIdx.x >= A.m[mi + 1].cta_first) ++mi;
    const MatArgs &k = A.m[MULTI ? mi : 0];
    const uint32_t J = blockIdx.x - k.cta_first, n_cta = k.cta_count;
    const uint32_t smem_base = smem_u32(dyn_smem);
    // `na` row tiles of `n_rg` row groups, in each of `slices` column slices.  Warp w belongs to slice w / (8 na), has row group
    // `rgi` there and decodes if the CTA has that many.  Where all 32 warps belong to slices (four tiles) a slice's warp that does
    // not decode carries its activations, the very last one, the issuer, only where its slice has no other; with fewer tiles
    // (one slice) the first warp behind the tiles carries them and the others in front of the issuer leave at once.  A tile's further
    // warps without a row group arrive at every stage like the others, so that they are there for the epilogue.  (With the
    // issuer carrying them there too, chunks of 8192 elements took, back to back, 230 us against 172 for 8192 x 28672 at 64 vectors,
    // 111 against 94 for 12288 x 12288 at 32.)
    const uint32_t S = A.tc_stages, slices = A.tc_slices, na = A.tc_tiles, tiles = na * slices, issuer = 31u;
    const uint32_t n_rg = A.tc_row_groups, n_dec = n_rg * slices;
    const uint32_t slice = warp == issuer || warp >= tiles * 8u ? slices - 1u : warp / (8u * na), li = warp - warp / (8u * na) * 8u * na;
    const uint32_t tile = warp >> 3, q = warp & 3, h = (warp >> 2) & 1, rgi = (li & ~7u) + q * 2 + h;
    const bool decodes = warp < tiles * 8u && rgi < n_rg, serves = warp != issuer && (tiles == 4u ? rgi == n_rg : warp == tiles * 8u);
    const bool issuer_carries = tiles == 4u && n_rg == na * 8u - 1u;
    const uint32_t a_lane = (32u * q + 16u * h) << 16;
    const uint32_t KC = k.col_chunks, RG = (uint32_t)((k.rows + 15) / 16);
    const uint32_t *index = (const uint32_t *)(k.blob + k.off_index);
    const uint8_t *payload = k.blob + k.off_payload;
    const uint32_t ksplit = T.ksplit[MULTI ? mi : 0], n_items = T.m_tiles[MULTI ? mi : 0] * ksplit;
    auto blocks_of = [&](uint32_t kc) -> uint32_t {
        uint32_t left = (uint32_t)k.cols - kc * k.chunk_cols;
        return (min(left, k.chunk_cols) + 31u) >> 5;
    };
    // column chunks [k0, k1) of work item `it`, and of them those of slice sl: the first slices take what does not divide
    auto item_range = [&](uint32_t it, uint32_t &k0, uint32_t &k1) {
        const uint32_t ks_i = it % ksplit;
        k0 = KC * ks_i / ksplit;                            // (at most 2^26 column chunks and 16 ranges)
        k1 = KC * (ks_i + 1) / ksplit;
    };
    auto slice_beg = [&](uint32_t k0, uint32_t k1, uint32_t sl) -> uint32_t { return k0 + (((k1 - k0) * sl + slices - 1) >> (slices >> 1)); };   // (1, 2, 4 slices)
    // first and last chunk of this warp's row group in a work item (false: nothing to decode there)
    auto item_chunks = [&](uint32_t it, uint32_t &cb, uint32_t &ce) -> bool {
        uint32_t k0, k1;
        item_range(it, k0, k1);
        const uint32_t rg_i = it / ksplit * n_rg + rgi;
        cb = rg_i * KC + slice_beg(k0, k1, slice);
        ce = rg_i * KC + slice_beg(k0, k1, slice + 1);
        return rg_i < RG && cb < ce;
    };

    // ---- set-up: table, barriers, tensor memory.  The offsets of the warp's first two records are asked for before anything
    // else and their copies started between the table's loads and stores (a warp's barriers are its own, so the copies need
    // nothing that the CTA has to meet for): the records arrive while the table is built.  (With the copies started behind
    // the set-up a CTA's first block was decoded 7.3 us after its start; now 4.4.)
    uint32_t cb = 0, ce = 0, o0 = 0, o1 = 0, o2 = 0;
    bool primed = decodes && J < n_items && item_chunks(J, cb, ce);      // the item's first two record copies are under way
    if (primed && lane == 0) {
        o0 = __ldg(index + cb);
        o1 = __ldg(index + cb + 1);
        if (cb + 1 < ce) o2 = __ldg(index + cb + 2);
    }
    const SmemPlan plan = plan_smem(smem_base, A, n_dec);
    if (plan.warps < n_dec) {                                   // the entry point sizes shared memory so that this cannot happen
        pdl_wait_prior_grid();
        if (tid == 0 && A.err) atomicExch(A.err, -3);
        return;
    }
    const uint32_t b_base = smem_base + A.dyn_smem_bytes - A.part_bytes;   // the stages of B behind everything else
    uint32_t lut_lane = lut_column<D>(plan.lut, lane), lut_low = lut_low_column<D>(plan.lut, lane);
    asm volatile("mov.u32 %0, %0;" : "+r"(lut_lane));
    if (D == kUpper) asm volatile("mov.u32 %0, %0;" : "+r"(lut_low));
    const uint32_t bar0 = smem_u32(&bars[warp * 2]);
    // (The ring's address is worked out once: the compiler takes a shared variable's address anew at every use, three instructions
    // of which one waits for a special register, 28672 x 8192 at 32 vectors 109.2 us against 106.2.  Not at the widest padding,
    // where the register is missed elsewhere: 28672 x 8192 at 64 142.3 with it, 139.4 without.  The kernel has 64 registers a thread and
    // uses them all; what the compiler makes of the decoders' loop, and with it every time here, moves by a few per cent with such things,
    // so they are chosen by measurement for each padding.)
    uint32_t ring = smem_u32(ring_bars);
    if (NPAD < 64) asm volatile("mov.u32 %0, %0;" : "+r"(ring));
    auto empty_bar = [&](uint32_t st) -> uint32_t { return ring + st * 8u; };
    auto full_bar = [&](uint32_t st) -> uint32_t { return ring + kTcStages * 8u + st * 8u; };
    const uint32_t slot0 = slot_addr(plan, decodes ? slice * n_rg + rgi : 0u, 0, A.slot_bytes);    // (this kernel always runs with two slots per warp)
    auto record_ok = [&](uint32_t r0, uint32_t r1, uint32_t nkb) -> bool {
        return r1 > r0 && r1 <= k.payload_units && (r1 - r0) * 128u > raw_part(nkb) &&
               (r1 - r0) * 128u - raw_part(nkb) <= A.slot_bytes;
    };
    auto issue_record = [&](uint32_t kc, uint32_t which, uint32_t r0, uint32_t r1) {       // kc: the chunk's column chunk
        uint32_t nkb = blocks_of(kc), bar = bar0 + which * 8;
        if (record_ok(r0, r1, nkb)) {
            uint32_t bytes = (r1 - r0) * 128u - raw_part(nkb);
            mbar_expect_tx(bar, bytes);
            bulk_g2s(slot0 + which * A.slot_bytes, payload + (uint64_t)r0 * 128u + raw_part(nkb), bytes, bar);
        } else {
            mbar_expect_tx(bar, 0);
        }
    };
    auto issue = [&](uint32_t c, uint32_t which) { issue_record(c % KC, which, __ldg(index + c), __ldg(index + c + 1)); };
    {
        if (lane == 0) {
            mbar_init(bar0, 1);
            mbar_init(bar0 + 8, 1);
        }
        // the table goes to shared memory in 16-byte pieces: four neighbouring copies of one entry per piece
        constexpr uint32_t kLutVecs = LutPlan<D>::kVecs;
        constexpr int kLutLoads = (kLutVecs + 1023) / 1024;
        const uint32_t *lut_g = (const uint32_t *)(k.blob + k.off_lut);
        uint32_t lut_v[kLutLoads];
#pragma unroll
        for (int i = 0; i < kLutLoads; ++i) {
            const uint32_t v = tid + i * 1024u;
            lut_v[i] = v < kLutVecs ? __ldg(lut_g + LutPlan<D>::source(v, A.lut_bits)) : 0u;
        }
        if (tid < S) {
            mbar_init(empty_bar(tid), 1);
            mbar_init(full_bar(tid), tiles == 4u ? 31u : tiles * 8u + 1u);      // (every warp but the issuer, decoding or not)
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (warp == issuer) {
            tmem_alloc(smem_u32(&s_tmem_base), 512);
            tmem_relinquish();
        }
        if (primed && lane == 0) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            const uint32_t kc_b = cb % KC;
            issue_record(kc_b, 0, o0, o1);
            if (cb + 1 < ce) issue_record(kc_b + 1, 1, o1, o2);
        }
        uint4 *lut_s = (uint4 *)(dyn_smem + (plan.lut - smem_base));
#pragma unroll
        for (int i = 0; i < kLutLoads; ++i) {
            const uint32_t v = tid + i * 1024u, e = lut_entry<D>(lut_v[i], LutPlan<D>::field(v));
            if (v < kLutVecs) lut_s[v] = make_uint4(e, e, e, e);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem_base;
    if (warp > tiles * 8u && warp != issuer) {    // in no tile: only the teardown barrier is left
        tc_fence_before();
        __syncthreads();
        return;
    }

    // The kernel in front of this one in the stream may still be producing the activations, or using the workspace: the warps that issue
    // or carry activations wait for it here, all others before they write anything.  The decoders, who read the blob alone, run ahead by the
    // depth of the stage ring.  (All warps waiting here / this, us: 4096 x 14336 at 16 vectors 34.2 / 32.6, the 7B-shaped layer at 32
    // 133.1 / 127.6, 8192 x 28672 at 64 120.8 / 118.5, 1024 x 4096 at 32 13.5 / 11.1, FP16 4096 x 11008 at 24 51.5 / 45.9: a product behind the same
    // product, which lets it start early and leaves SMs free while it ends.  Behind a kernel that does not, nothing is gained.)
    if (warp == issuer || serves) pdl_wait_prior_grid();

    float *const tc_partial = T.partial[MULTI ? mi : 0];
    unsigned int *const tc_ticket = T.ticket[MULTI ? mi : 0];
    uint32_t phase = 0;                  // coded-copy barrier parities
    uint32_t st_s = 0, st_use = 0;       // the stage ring: the next stage and how often the ring has gone round
    auto next_stage = [&]() {
        if (++st_s == S) {
            st_s = 0;
            ++st_use;
        }
    };
    bool failed = false;                 // a wait ran out: stop waiting, keep moving, report

    // (Whether a wait has run out is asked first where that is faster.  Asked first / behind the poll alone, us: 4096 x 14336 at 16 vectors 32.4 /
    // 31.8, 8192 x 8192 at 16 in chunks of 8192 41.3 / 39.2; the 7B-shaped layer at 32 124.1 / 126.6; 8192 x 28672 at 64 116.4 / 119.6.)
    auto bounded_wait = [&](uint32_t bar, uint32_t parity) {
        if (NPAD > 16 && failed) return;
        uint32_t spins = 0;
        while (!__all_sync(0xFFFFFFFFu, mbar_try_wait(bar, parity))) {
            if (failed) return;
            if (++spins > kWaitLimit) {
                failed = true;
                if (A.err && lane == 0) atomicExch(A.err, -2);
                return;
            }
            // (what is missing may be behind the warps that wait for the kernel in front: that takes as long as it takes)
            if (spins == kPollsAlone) pdl_wait_prior_grid();
        }
    };
    auto stage_free = [&]() {            // the stage's last MMAs are done (the first time round: the phase in front of the first one has passed)
        bounded_wait(empty_bar(st_s), (st_use - 1) & 1u);
    };

    // The activations of a block: vector n's K positions 8 kap .. 8 kap + 7 (kap = 0 .. 3) of the tile hold its columns
    // base .. base + 3 and base + 8 .. base + 11 of the block, base = 16 (kap & 1) + 4 (kap >> 1), each four a copy of 8 bytes.
    // Eight lanes take a vector's 64 bytes, a warp instruction four vectors (whole sectors are read, and four lines at a
    // time: with four lanes to a vector it was eight).  `nblk` blocks (1 or 2) from column `col` on go to stage `st`; vectors
    // of the padding are left as they are: they reach no column of the product that is written.  The issuer's instructions are what
    // the carrying costs (eight cycles each, as above), so sixteen vectors that are all there are copied without a predicate, and
    // addresses are a base and a 32-bit stride.  (Sizes and pointers of
    // every copy selected by whether its vector exists / predicates on every copy / this, us: 25088 x 7168 at 64 vectors in chunks of 2048
    // 124.2 / 125.4 / 112.5, 11008 x 4096 at 48 34.6 / 34.0 / 30.3, 14336 x 4096 at 40 42.4 / 39.4 / 36.8.)
    auto carry_x = [&](uint32_t col, uint32_t nblk, uint32_t st) {
        const uint32_t kap = (lane >> 1) & 3u, half = lane & 1u;
        uint32_t n = lane >> 3;
        const uint32_t dst = b_base + (st * slices + slice) * kBStage + kap * kLbo + n * 16u + half * 8u;
        const uint16_t *src = k.x + (uint64_t)min(n, A.batch - 1) * k.cols + col + (kap & 1) * 16 + (kap >> 1) * 4 + half * 8;
        const uint32_t step = (uint32_t)k.cols;             // (at most 2^31)
        const char *sp = (const char *)src;
#pragma unroll
        for (int i0 = 0; i0 < NPAD / 4; i0 += 4, n += 16) {
            if (nblk > 1 && A.batch >= 4u * i0 + 16u) {
#pragma unroll
                for (int i = i0; i < i0 + 4; ++i) {
                    const uint32_t to = dst + (i >> 1) * kSbo + (i & 1) * 64u;
                    cp_async8(to, sp + (uint64_t)step * (8u * i));
                    cp_async8(to + 4 * kLbo, sp + (uint64_t)step * (8u * i) + 64);
                }
            } else {
#pragma unroll
                for (int i = i0; i < i0 + 4; ++i) {
                    const uint32_t to = dst + (i >> 1) * kSbo + (i & 1) * 64u;
                    if (n + 4 * (i - i0) < A.batch) {
                        cp_async8(to, sp + (uint64_t)step * (8u * i));
                        if (nblk > 1) cp_async8(to + 4 * kLbo, sp + (uint64_t)step * (8u * i) + 64);
                    }
                }
            }
        }
    };
    auto x_landed = [&]() {                                  // the B slice must be visible to the tensor core's reads
        asm volatile("cp.async.wait_all;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
    };
    // this warp's rows of the A operand
    const uint32_t a_dst0 = tmem + a_lane + kACol0 + tile * 32;

    // One block of the stage protocol, decoder side.  `a` = this warp's decoded 16 rows x 32 columns, block `half` of the
    // stage's `nblk`.  The warp stores its share, says so on the stage's "full" barrier and goes on decoding: nobody waits for
    // the other warps here.  A warp can run ahead of the slowest one by the depth of the stage ring and no further (it
    // needs the stage back, which the issuer's tcgen05.commit announces on the "empty" barrier).
    auto stage_block = [&](const uint32_t *a, uint32_t half, uint32_t nblk) {
        if (half == 0) {
            stage_free();
            tc_fence_after();
        }
        // lane (g, t): row g's weights 0..3 -> 32-bit columns 2t, 2t+1; weights 4..7 -> columns 8 + 2t, 8 + 2t + 1
        const uint32_t r[8] = {a[0], a[1], a[4], a[5], a[2], a[3], a[6], a[7]};
        tc_st_16x256b_x2(a_dst0 + st_s * 128 + half * 16, r);
        if (half + 1 < nblk) return;
        tc_wait_st();
        tc_fence_before();
        __syncwarp();
        if (NPAD > 16 ? lane == 0 : elect_one()) mbar_arrive(full_bar(st_s));   // (4096 x 14336 at 16 vectors 33.0 us / 31.9 elected, 8192 x 28672 at 64 117.1 / 118.5)
        next_stage();
    };
    // A stage to which this warp has nothing to add (rows outside the matrix, a slice that is done).
    auto stage_nothing = [&]() {
        stage_free();
        if (lane == 0) mbar_arrive(full_bar(st_s));
        next_stage();
    };
    // The same stage, issuer side: when every warp has arrived, one lane issues the stage's MMAs for every tile and commits
    // them onto the stage's "empty" barrier.  halves(sl): blocks of slice sl in the stage.  (After a wait that ran out the
    // commit still goes out: the stage ring keeps moving and the kernel ends with its error flag set.)
    // What bounds this warp is the number of instructions per MMA (its scheduler has seven decoding warps to serve, so each
    // costs some eight cycles): the thread is elected, not chosen by its number, and every operand is a base and a constant,
    // so that addresses and descriptors are worked out on the uniform datapath, where the MMA wants them.  (28672 x 8192 at
    // 32 vectors: 154 us with a loop over runtime strides in lane 0, 127 so; a stage's 16 MMAs take 500 to 600 cycles.
    // Unrolled for fewer tiles too, those launches took 1 to 2 % less, but those of four tiles up to 1 % more.)
    auto issue_tiles = [&](auto n_slices, bool first_of_item) {                    // a stage of four tiles whose slices all have two blocks
        constexpr uint32_t SL = decltype(n_slices)::value, NA = 4u / SL;
        const uint32_t ac = tmem + kACol0 + st_s * 128u;
        const uint32_t bd = smem_desc_lo(b_base + st_s * SL * kBStage, kLbo);
#pragma unroll
        for (uint32_t t = 0; t < 4; ++t)
#pragma unroll
            for (uint32_t j = 0; j < 4; ++j)
                tc_mma_f16_tmem_a(tmem + t * NPAD, ac + t * 32u + j * 8u, smem_desc(bd + ((t / NA * kBStage + j * 2u * kLbo) >> 4), kSbo), kIdesc,
                                  j == 0 ? (first_of_item ? 0u : 1u) : 1u);
    };
    auto issue_stage = [&](bool first_of_item, bool full, auto halves) {           // full: four tiles, two blocks of every slice
        bounded_wait(full_bar(st_s), st_use & 1u);
        if (elect_one()) {
            tc_fence_after();
            if (failed) {
            } else if (full && slices == 1u) {
                issue_tiles(std::integral_constant<uint32_t, 1>{}, first_of_item);
            } else if (full && slices == 2u) {
                issue_tiles(std::integral_constant<uint32_t, 2>{}, first_of_item);
            } else if (full) {
                issue_tiles(std::integral_constant<uint32_t, 4>{}, first_of_item);
            } else {
                uint32_t ac = tmem + kACol0 + st_s * 128u;
                for (uint32_t sl = 0; sl < slices; ++sl) {
                    const uint32_t steps = 2 * halves(sl);                // K = 16 steps: four per full stage, two for an odd last block
                    const uint32_t bd = smem_desc_lo(b_base + (st_s * slices + sl) * kBStage, kLbo);
                    for (uint32_t tl = 0; tl < na; ++tl, ac += 32u)
                        for (uint32_t j = 0; j < steps; ++j)
                            tc_mma_f16_tmem_a(tmem + (sl * na + tl) * NPAD, ac + j * 8u, smem_desc(bd + (j * 2u * kLbo >> 4), kSbo), kIdesc,
                                              (first_of_item && j == 0) ? 0u : 1u);
                }
            }
            tc_commit(empty_bar(st_s));
        }
        __syncwarp();
        next_stage();
    };

    // The end of a work item: the warps of a quarter of the lanes share the columns of the row tiles' accumulators; a warp adds
    // its columns of the slices' accumulators up, in slice order, and either writes them or leaves them as the piece of its
    // range, which the last range to arrive adds up in range order.
    auto epilogue = [&](auto n_slices, uint32_t item, uint32_t mt, uint32_t k0, uint32_t k1) {
        constexpr uint32_t SL = decltype(n_slices)::value;
        constexpr int CW = NPAD / (2 * SL);
        pdl_wait_prior_grid();                               // (over by now, as the issuer waited for it; but every warp that writes asks)
        const uint32_t col0 = (warp >> 2) * CW, acc_tile = col0 / NPAD, n0 = col0 % NPAD;
        float v[CW];
#pragma unroll
        for (uint32_t sl = 0; sl < SL; ++sl) {
            if (sl && slice_beg(k0, k1, sl) == slice_beg(k0, k1, sl + 1)) continue;      // (no chunk: nothing was accumulated)
            uint32_t t[CW];
            tc_ld_32x32b<CW>(tmem + ((32u * q) << 16) + sl * (4 / SL) * NPAD + col0, t);
            tc_wait_ld();
#pragma unroll
            for (int i = 0; i < CW; ++i) v[i] = sl ? v[i] + __uint_as_float(t[i]) : __uint_as_float(t[i]);
        }
        tc_fence_before();
        // thread `lane` holds row 32 q + lane of the tile, columns n = n0 + i
        const uint64_t row = (uint64_t)(mt * n_rg + acc_tile * 8) * 16 + 32u * q + lane;
        const bool row_ok = row < k.rows && acc_tile * 8 + 2 * q + (lane >> 4) < n_rg;   // (row groups behind the CTA's belong to the next item)
        auto write = [&](const float (&out)[CW]) {
#pragma unroll
            for (int i = 0; i < CW; ++i)
                if (n0 + i < A.batch && row_ok) k.y[(uint64_t)(n0 + i) * k.rows + row] = out[i];
        };
        if (ksplit == 1) {
            write(v);
            return;
        }
        // piece of (item, warp): [CW][32] floats, 32 piece slots per item
        float *piece = tc_partial + ((size_t)item * 32 + warp) * CW * 32;
#pragma unroll
        for (int i = 0; i < CW; ++i) piece[i * 32 + lane] = v[i];
        __syncwarp();
        uint32_t last = 0;
        if (SL == 1) {                                       // every warp finds its own pieces: a counter per row tile and warp
            if (lane == 0) {
                unsigned int *ctr = tc_ticket + mt * 32 + warp;
                last = arrive_acq_rel(ctr) == ksplit - 1 ? 1u : 0u;
                if (last) *ctr = 0;
            }
            last = __shfl_sync(0xFFFFFFFFu, last, 0);
        } else {                                             // small pieces: one counter per row tile (all 32 warps are here)
            __syncthreads();
            if (tid == 0) {
                unsigned int *ctr = tc_ticket + mt;
                s_last = arrive_acq_rel(ctr) == ksplit - 1 ? 1u : 0u;
                if (s_last) *ctr = 0;
            }
            __syncthreads();
            last = s_last;
        }
        if (!last) return;
        // 32 independent loads in flight: every column of as many ranges as make 32; every output adds its pieces in range order
        constexpr int U = CW >= 32 ? 1 : 32 / CW;
        constexpr size_t kRange = (size_t)32 * CW * 32;
        const float *pc = tc_partial + ((size_t)mt * ksplit * 32 + warp) * CW * 32 + lane;
#pragma unroll
        for (int i = 0; i < CW; ++i) v[i] = 0.f;
        uint32_t r = 0;
#pragma unroll 1
        for (; r + U <= ksplit; r += U, pc += U * kRange) {
            float p[U][CW];
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int i = 0; i < CW; ++i) p[u][i] = __ldcg(pc + u * kRange + i * 32);
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int i = 0; i < CW; ++i) v[i] += p[u][i];
        }
#pragma unroll 1
        for (; r < ksplit; ++r, pc += kRange)
#pragma unroll
            for (int i = 0; i < CW; ++i) v[i] += __ldcg(pc + i * 32);
        write(v);
    };

#pragma unroll 1
    for (uint32_t item = J; item < n_items; item += n_cta) {
        const uint32_t mt = item / ksplit;
        uint32_t k0, k1;
        item_range(item, k0, k1);
        const uint32_t kc0 = slice_beg(k0, k1, slice), kc1 = slice_beg(k0, k1, slice + 1);
        const uint32_t rg = mt * n_rg + rgi;
        const bool active = decodes && rg < RG && kc0 < kc1;
        // The slices go through their chunks side by side: a chunk's stages (pairs of blocks), `steps` times.  (One slice: the
        // stages of the chunk at hand; several: those of a full chunk, some of which the row's last chunk leaves empty.)
        const uint32_t steps = slice_beg(k0, k1, 1) - k0, full_stages = (k.chunk_cols / 32u + 1u) >> 1;
        const uint32_t col_lo = kc0 * k.chunk_cols;         // the slice's first column
        // blocks of the chunk that slice sl has in step j, and of those in the stage that holds its pair p
        auto step_blocks = [&](uint32_t sl, uint32_t j) -> uint32_t {
            const uint32_t kc = slice_beg(k0, k1, sl) + j;
            return kc < slice_beg(k0, k1, sl + 1) ? blocks_of(kc) : 0u;
        };
        auto halves = [](uint32_t nkb, uint32_t p) -> uint32_t { return nkb > 2 * p ? min(nkb - 2 * p, 2u) : 0u; };
        auto stages_of = [&](uint32_t j) -> uint32_t { return slices == 1u ? (blocks_of(k0 + j) + 1u) >> 1 : full_stages; };

        if (warp == issuer) {
            // The activations of the stages behind the one at hand, all but one of the ring's, are always under way.  (Of the next
            // stage alone / of the next two, us: 28672 x 8192 at 32 vectors 110.4 / 106.4, the 7B-shaped layer at 32 126.2 / 124.6.)
            uint32_t own = step_blocks(slice, 0), cj = 0, cp = 0, c_s = st_s, c_use = st_use;   // the stage to be carried next, and its place in the ring
            auto carry_next = [&]() {
                if (cj < steps) {
                    bounded_wait(empty_bar(c_s), (c_use - 1) & 1u);
                    const uint32_t n2 = halves(own, cp);
                    if (n2) carry_x(col_lo + cj * k.chunk_cols + cp * 64u, n2, c_s);
                    if (++c_s == S) {
                        c_s = 0;
                        ++c_use;
                    }
                    if (++cp == stages_of(cj)) {
                        cp = 0;
                        own = ++cj < steps ? step_blocks(slice, cj) : 0u;
                    }
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
            };
            if (issuer_carries)
                for (uint32_t i = 1; i < S; ++i) carry_next();
            for (uint32_t j = 0; j < steps; ++j) {          // stages are cut like the decoders': pairs of blocks inside a chunk
                const uint32_t n_st = stages_of(j);
                uint32_t nkb[4], least = ~0u;               // blocks of every slice in this step, and the fewest
#pragma unroll
                for (uint32_t sl = 0; sl < 4; ++sl) {
                    nkb[sl] = sl < slices ? step_blocks(sl, j) : 0u;
                    if (sl < slices) least = min(least, nkb[sl]);
                }
                for (uint32_t p = 0; p < n_st; ++p) {
                    if (issuer_carries) {
                        if (S == 3u) asm volatile("cp.async.wait_group 1;" ::: "memory");
                        else asm volatile("cp.async.wait_group 0;" ::: "memory");
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        __syncwarp();
                    }
                    issue_stage(j == 0 && p == 0, tiles == 4u && least >= 2 * p + 2, [&](uint32_t sl) -> uint32_t {
                        return halves(sl == 0 ? nkb[0] : sl == 1 ? nkb[1] : sl == 2 ? nkb[2] : nkb[3], p);
                    });
                    if (issuer_carries) carry_next();
                }
            }
        } else if (serves) {
            for (uint32_t j = 0; j < steps; ++j) {
                const uint32_t own = step_blocks(slice, j), n_st = stages_of(j);
                for (uint32_t p = 0; p < n_st; ++p) {
                    stage_free();
                    const uint32_t n2 = halves(own, p);
                    if (n2) carry_x(col_lo + j * k.chunk_cols + p * 64u, n2, st_s);
                    x_landed();
                    if (lane == 0) mbar_arrive(full_bar(st_s));
                    next_stage();
                }
            }
        } else if (active) {
            const uint32_t c_beg = rg * KC + kc0, c_end = rg * KC + kc1;
            if (lane == 0 && !primed) {
                issue(c_beg, 0);
                if (c_beg + 1 < c_end) issue(c_beg + 1, 1);
            }
            uint32_t kc = kc0;
            // record offsets are known two chunks ahead, the first raw block of a record is asked for in the last block of the
            // one before: a chunk's start waits for neither
            uint32_t r0 = __ldg(index + c_beg), r1 = __ldg(index + c_beg + 1), r2 = c_beg + 1 < c_end ? __ldg(index + c_beg + 2) : r1;
            bool raw_there = false;
            const uint8_t *const raw0 = payload + lane * kRawLane;
            const uint8_t *raw_p = raw0;
            uint4 raw_cur = make_uint4(0, 0, 0, 0), raw_b = make_uint4(0, 0, 0, 0);
#pragma unroll 1
            for (uint32_t c = c_beg; c < c_end; ++c, ++kc) {
                const uint32_t which = (c - c_beg) & 1u;
                const uint32_t nkb = blocks_of(kc);
                const bool ok = record_ok(r0, r1, nkb), has_next = c + 1 < c_end;
                const uint32_t r3 = c + 2 < c_end ? __ldg(index + c + 3) : r2;
                if (ok && !raw_there) {
                    raw_p = raw0 + (uint64_t)r0 * 128u;
                    raw_cur = load_raw(raw_p);
                }
                bounded_wait(bar0 + which * 8, (phase >> which) & 1u);
                phase ^= 1u << which;
                if (!ok && A.err && lane == 0) {
                    pdl_wait_prior_grid();                  // (it may be clearing or reading the flag)
                    atomicExch(A.err, (int32_t)min(c + 1, 0x7FFFFFFFu));
                }
                if (!ok) {
                    const uint32_t zero[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
                    for (uint32_t kb = 0; kb < nkb; ++kb) stage_block(zero, kb & 1u, (kb & 1u) || kb + 1 < nkb ? 2u : 1u);
                    raw_there = false;
                } else {
                    uint32_t pa = (slot0 + which * A.slot_bytes) / 8u + start_of(D), pb = pa;
                    // one block: fetch the next block's raw bytes into the other register set (behind the record's last one: the
                    // next record's first, an address inside the blob whatever its offsets turn out to be), decode this one, hand
                    // it to the tensor core
                    auto block = [&](const uint4 &raw_c, uint4 &raw_n, bool last, uint32_t half, uint32_t nblk) {
                        raw_p += kRawBlock;
                        if (last) raw_p = raw0 + (uint64_t)r1 * 128u;
                        if (!last || has_next) raw_n = load_raw(raw_p);
                        // the block behind that one is asked into L2: a register load one block ahead waits for DRAM otherwise.  (It may
                        // lie in the coded part or behind the record, up to 1 KB behind the payload: the blob has 4 KB there.)
                        // Not for FP16, whose raw part is a sixteenth.  (us, without / with it / two blocks further on: 4096 x 14336 at 16
                        // vectors 35.1 / 34.2 / 35.1, 7B-shaped layer at 32 135.5 / 133.1 / 135.1; 28672 x 8192 at 32 in chunks of 8192 160.5 /
                        // 148.6.  Padding 64: 12288 x 12288 90.1 / 86.6, in chunks of 8192 101.9 / 92.9, 28672 x 8192 147.6 / 143.7.  The record's
                        // whole raw part at once, with its copy: 36.8 and 139.6 for the first two.)
                        if (FMT == 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(raw_p + kRawBlock));
                        uint32_t a[8];
                        decode_block<D>(pa, pb, lane << 2, lut_lane, lut_low, raw_c, a, 0u, 0u);
                        stage_block(a, half, nblk);
                    };
                    uint32_t kb = 0;
#pragma unroll 1
                    for (; kb + 2 <= nkb; kb += 2) {                  // the usual case: pairs of blocks, two register sets in turn
                        block(raw_cur, raw_b, false, 0, 2);
                        block(raw_b, raw_cur, kb + 2 == nkb, 1, 2);
                    }
                    if (kb < nkb) {                                   // odd block count (a ragged last chunk): a stage of one block
                        block(raw_cur, raw_b, true, 0, 1);
                        raw_cur = raw_b;
                    }
                    raw_there = has_next;
                }
                if (slices > 1u)
                    for (uint32_t p = (nkb + 1u) >> 1; p < full_stages; ++p) stage_nothing();
                __syncwarp();
                if (lane == 0 && c + 2 < c_end) issue_record(kc + 2, which, r2, r3);
                r0 = r1;
                r1 = r2;
                r2 = r3;
            }
            for (uint32_t j = kc1 - kc0; j < steps; ++j)    // steps in which only other slices have a chunk
                for (uint32_t p = 0; p < full_stages; ++p) stage_nothing();
        } else {
            for (uint32_t j = 0; j < steps; ++j)            // nothing to decode for this warp: its arrivals are still waited for
                for (uint32_t p = stages_of(j); p; --p) stage_nothing();
        }

        // both slots are free again: the next item's first records are asked for now, so that they arrive behind the epilogue
        primed = false;
        if (decodes && item + n_cta < n_items) {
            uint32_t nb, ne;
            if (item_chunks(item + n_cta, nb, ne)) {
                if (lane == 0) {
                    issue(nb, 0);
                    if (nb + 1 < ne) issue(nb + 1, 1);
                }
                primed = true;
            }
        }

        // wait for the last stage's MMAs.  (The issuer has a share in the epilogue like every warp; with fewer than four tiles
        // only the tiles' warps have one.)
        if (warp < tiles * 8u) {
            const uint32_t ls = st_s == 0 ? S - 1u : st_s - 1u, lu = st_s == 0 ? st_use - 1u : st_use;
            bounded_wait(empty_bar(ls), lu & 1u);
            tc_fence_after();
            if (slices == 1u) epilogue(std::integral_constant<uint32_t, 1>{}, item, mt, k0, k1);
            else if (slices == 2u) epilogue(std::integral_constant<uint32_t, 2>{}, item, mt, k0, k1);
            else epilogue(std::integral_constant<uint32_t, 4>{}, item, mt, k0, k1);
        }
    }

    // ---- teardown
    tc_fence_before();
    __syncthreads();
    if (warp == issuer) tmem_dealloc(tmem, 512);
}

template <int LB, int NPAD, int FMT, bool MULTI>
static cudaError_t launch_tc_m(const TcArgs &t, uint32_t grid, cudaStream_t stream) {
    const KernelArgs &k = t.k;
    auto fn = huff_gemm_tc_kernel<LB, NPAD, FMT, MULTI>;
    static std::atomic<bool> attr_set[64];   // set twice by racing threads at worst: the call is idempotent
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64 || !attr_set[dev].load(std::memory_order_acquire)) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k.dyn_smem_bytes);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev].store(true, std::memory_order_release);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(1024);
    cfg.dynamicSmemBytes = k.dyn_smem_bytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // set-up overlaps the previous kernel's tail
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fn, t);
}

template <int LB, int NPAD, int FMT>
static cudaError_t launch_tc_one(const TcArgs &t, uint32_t grid, cudaStream_t stream) {
    if (t.k.n_mats > 1) return launch_tc_m<LB, NPAD, FMT, true>(t, grid, stream);
    return launch_tc_m<LB, NPAD, FMT, false>(t, grid, stream);
}

cudaError_t launch_gemm_tc(const TcArgs &t, uint32_t grid, cudaStream_t stream) {
    const KernelArgs &k = t.k;
    if (k.fmt && k.fp16_flat == kFlatUpper) {
        if (k.tc_npad == 16) return launch_tc_one<8, 16, 3>(t, grid, stream);
        if (k.tc_npad == 32) return launch_tc_one<8, 32, 3>(t, grid, stream);
        return launch_tc_one<8, 64, 3>(t, grid, stream);
    }
    if (k.fmt && k.fp16_flat == kFlatBoth) {
        if (k.tc_npad == 16) return launch_tc_one<8, 16, 2>(t, grid, stream);
        if (k.tc_npad == 32) return launch_tc_one<8, 32, 2>(t, grid, stream);
        return launch_tc_one<8, 64, 2>(t, grid, stream);
    }
    if (k.fmt && k.fp16_flat == kFlatBothLanes) {
        if (k.tc_npad == 16) return launch_tc_one<8, 16, 4>(t, grid, stream);
        if (k.tc_npad == 32) return launch_tc_one<8, 32, 4>(t, grid, stream);
        return launch_tc_one<8, 64, 4>(t, grid, stream);
    }
    if (k.fmt) {
        if (k.tc_npad == 16) return launch_tc_one<8, 16, 1>(t, grid, stream);
        if (k.tc_npad == 32) return launch_tc_one<8, 32, 1>(t, grid, stream);
        return launch_tc_one<8, 64, 1>(t, grid, stream);
    }
    if (k.lut_bits == 8) {
        if (k.tc_npad == 16) return launch_tc_one<8, 16, 0>(t, grid, stream);
        if (k.tc_npad == 32) return launch_tc_one<8, 32, 0>(t, grid, stream);
        return launch_tc_one<8, 64, 0>(t, grid, stream);
    }
    if (k.tc_npad == 16) return launch_tc_one<9, 16, 0>(t, grid, stream);
    if (k.tc_npad == 32) return launch_tc_one<9, 32, 0>(t, grid, stream);
    return launch_tc_one<9, 64, 0>(t, grid, stream);
}

}  // namespace huffllm
