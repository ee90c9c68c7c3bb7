// C-ABI entry points that run on the device: argument checks, launch geometry, launches.
// No allocation and no synchronisation here (huffllm_decode_gemm_host, which exists to be timed
// end to end with host buffers, is the one call that waits for its stream).
#include <cuda_runtime.h>
#include <atomic>
#include <cstdlib>
#include <cstring>

#include "internal.h"
#include "kernels.h"

using namespace huffllm;

namespace {

constexpr uint32_t kMaxGrid = 512;        // CTAs the scratch layout provides for
constexpr uint32_t kKernelBatch = 8;      // activation vectors one launch multiplies
constexpr uint32_t kStaticSmem = 2048;    // barriers and tables the kernel declares statically (rounded up)

// Per-device facts, looked up once.  Threads may race to fill an entry: they write the same values, and `known` is
// published last.
struct DeviceSlot {
    std::atomic<bool> known{false};
    std::atomic<int> sms{0}, smem_optin{0};
};
DeviceSlot g_dev[64];
struct DeviceInfo {
    int sms = 0, smem_optin = 0;
};

huffllm_status device_info(DeviceInfo *out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return fail(HUFFLLM_ERR_CUDA, "cudaGetDevice: %s", cudaGetErrorString(e));
    if (dev < 0 || dev >= 64) return fail(HUFFLLM_ERR_UNSUPPORTED, "device ordinal %d out of range", dev);
    DeviceSlot &d = g_dev[dev];
    if (!d.known.load(std::memory_order_acquire)) {
        int sms = 0, smem = 0;
        if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
            (e = cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess)
            return fail(HUFFLLM_ERR_CUDA, "cudaDeviceGetAttribute: %s", cudaGetErrorString(e));
        d.sms.store(sms, std::memory_order_relaxed);
        d.smem_optin.store(smem, std::memory_order_relaxed);
        d.known.store(true, std::memory_order_release);
    }
    out->sms = d.sms.load(std::memory_order_relaxed);
    out->smem_optin = d.smem_optin.load(std::memory_order_relaxed);
    return HUFFLLM_OK;
}

// Scratch layout of one matrix's workspace:
//   [0, 4096)            arrival counters of the register-path kernel (one per CTA)
//   [4096, partial_off)  arrival counters of the tensor-core kernel, sized for its smallest tile
//   [partial_off, ...)   partial sums: of the register path's CTAs, or of the tensor-core path's work items
// Everything in front of partial_off is zero between calls; what lies behind it is overwritten freely by either path.
size_t ws_ctrl_bytes(const huffllm_desc *) { return 4096; }
size_t ws_partial_offset(const huffllm_desc *d) {
    const size_t max_m_tiles = (d->row_groups + 7) / 8;      // tensor-core row tiles at their smallest (128 rows)
    return ws_ctrl_bytes(d) + (max_m_tiles * 32 * 4 + 255) / 256 * 256;
}
// Partial sums of the register path: [kMaxGrid * 2][16 * b] CTA pieces, and, with two tiles of activations (batch
// 9..16), [kMaxGrid][2 * 32][16 * b] pieces that the warps of one CTA exchange (shared memory has no room for them).
constexpr uint32_t kTwoTileBatch = 16;    // most activation vectors of the register path with two tiles
bool two_tile_blob(const huffllm_desc *d) { return d->dtype == HUFFLLM_BF16 && d->lut_bits == 8; }
// blobs the tensor-core kernel takes: tables of up to 9 bits (FP16: field codes of up to 8 bits)
bool tc_blob(const huffllm_desc *d) { return d->dtype == HUFFLLM_FP16 ? d->lut_bits == 8u : d->lut_bits <= 9u; }
size_t ws_cta_pieces_bytes(uint32_t b) { return (size_t)kMaxGrid * 2 * 16 * b * sizeof(float); }
// (a workspace sized for `batch` vectors serves every smaller batch too)
size_t ws_bytes_for(const huffllm_desc *d, uint32_t batch) {
    size_t need = ws_cta_pieces_bytes(batch < kKernelBatch ? batch : kKernelBatch);
    if (batch > kKernelBatch && two_tile_blob(d)) {
        const uint32_t b = batch < kTwoTileBatch ? batch : kTwoTileBatch;
        need = ws_cta_pieces_bytes(b) + (size_t)kMaxGrid * 2 * 32 * 16 * b * sizeof(float);
    }
    return ws_partial_offset(d) + need;
}

// What a blob asks of a decoder CTA's shared memory.
struct SmemNeeds {
    uint32_t table_align, table_bytes;   // window of the decode table(s)
    uint32_t slot_bytes;                 // one slot: the W rows of the largest record
    uint32_t checks_per_block;           // rows a sequence may move on in a block of 32 columns, as budgeted
    uint32_t guard_bytes;                // readable bytes kept behind the last slot
};
// Which mantissa halves of an FP16 blob carry the flat code and can be read without a table (codes of at most 8 bits).
uint32_t flat_of(const huffllm_desc *d) {
    if (d->dtype != HUFFLLM_FP16 || d->lut_bits > 8) return kFlatNone;
    return (d->flat_fields & 6u) == 6u ? kFlatBoth : d->flat_fields & 2u ? kFlatUpper : kFlatNone;
}
// ... and of several blobs.
uint32_t flat_of_both(uint32_t a, uint32_t b) { return a == b ? a : a == kFlatNone || b == kFlatNone ? kFlatNone : kFlatUpper; }
// Bytes of the FP16 tables (first level): three of 16 KB; the exponent's with a copy per lane and the lower half's with
// sixteen; the exponent's alone, with sixteen or with one per lane (a launch's choice, see finish_args and tc_choose).
uint32_t fp16_table_bytes(uint32_t flat) { return flat == kFlatBoth ? 16384u : flat == kFlatBothLanes ? 32768u : 49152u; }
SmemNeeds smem_needs(const huffllm_desc *desc) {
    SmemNeeds n;
    const bool fmt = desc->dtype == HUFFLLM_FP16;
    // BF16 tables of up to 9 bits are replicated per lane; longer ones are looked up in two levels: a per-lane table of the
    // first 8 bits, then one copy of the whole table behind it
    // (FP16: three sixteen-fold tables of 8 bits; fields of 9 bits and more take the second level too)
    const bool two_level = desc->lut_bits > (fmt ? 8u : 9u);
    // (FP16 blobs with flat mantissa codes need fewer tables; a launch over several matrices takes what all of them allow, see
    // fp16_table_bytes)
    n.table_align = fmt ? 16384u : 128u << (two_level ? 8u : desc->lut_bits);
    n.table_bytes = fmt ? fp16_table_bytes(two_level ? kFlatNone : flat_of(desc)) + (two_level ? 3u * (4u << desc->lut_bits) : 0u)
                        : (two_level ? (128u << 8) + (4u << desc->lut_bits) : 128u << desc->lut_bits);
    // a slot holds the W rows of a record; the windows run up to two rows ahead of the pointer, and what they read
    // past the last row lies in the next slot, the table or the guard area and is never used
    n.slot_bytes = desc->max_words * 256;
    // No table in shared memory holds a length above what its index bits allow (lut_entry), so a block moves a sequence by
    // 64 bits (8-bit BF16 tables) to 288 (FP16, fields of up to 12 bits), two to nine rows, whatever its bits and whatever
    // the blob's table says.  The budget is that of decoders that took a check per row (three to 24 a block): it covers
    // these too, for a slot of any size.
    n.checks_per_block = fmt ? (two_level ? 24 : 8) : (desc->lut_bits == 8 ? 3 : 4);
    n.guard_bytes = 256 * (3 + n.checks_per_block * (desc->chunk_cols / kBlockCols));
    return n;
}

// How many decoder warps get their slots: the kernels' own shared-memory plan (plan_smem in decode_common.cuh) worked out
// on the host.  Slots lie in front of and behind the decode table, which sits on a boundary of `lut_align` bytes, so up to a
// slot pair's bytes are lost on either side; where the dynamic window starts depends on the kernel's static shared memory,
// which the host does not know exactly: the smallest count over every 128-byte start within kStaticSmem + 1 KB is taken.
uint32_t planned_warps(uint32_t lut_align, uint32_t lut_size, uint64_t pair_bytes, uint32_t dyn_smem, uint32_t part_bytes,
                       uint32_t guard_bytes) {
    // (32-bit arithmetic, whose divisions are cheap: a launch asks this a dozen times; check_desc bounds the records)
    const uint32_t guard_extra = guard_bytes > part_bytes ? guard_bytes - part_bytes : 0, pair = (uint32_t)pair_bytes;
    uint32_t least = 64;
    for (uint32_t base = 0; base <= kStaticSmem + 1024; base += 128) {
        const uint32_t lut = (base + lut_align - 1) & ~(lut_align - 1);      // (a power of two)
        const uint32_t slot_a = (base + 255) / 256 * 256, n_a = lut > slot_a ? (lut - slot_a) / pair : 0;
        const uint32_t slot_b = lut + lut_size, end = base + dyn_smem - part_bytes;
        const uint32_t n_b = end > slot_b + guard_extra ? (end - slot_b - guard_extra) / pair : 0;
        if (n_a + n_b < least) least = n_a + n_b;
    }
    return least;
}

// ---- the tensor-core small-batch path (batch 9..64)
// What a CTA of a launch decodes side by side: `na` tiles of 128 rows in each of `slices` column slices, at most four tiles in
// all (eight warps each), and the stages through which they hand it to the tensor core.
struct TcShape {
    uint32_t na, slices, stages, row_groups;
    uint32_t decoders() const { return row_groups * slices; }
    bool part_filled() const { return slices == 1 && na == 2 && row_groups < 16; }     // (shape 4: the second tile has rows left over)
    uint32_t part_bytes(uint32_t npad) const { return stages * slices * npad * 128; }  // the stages of activations
    uint32_t piece_columns(uint32_t npad) const { return npad / (2 * slices); }        // columns of a warp's share of the accumulators
};
uint32_t tc_npad_of(uint32_t batch) { return batch <= 16 ? 16 : (batch <= 32 ? 32 : 64); }
// Do the slot pairs of the shape's decoder warps fit beside the tables and the stages of activations (the guard area may lie
// over those), for the largest records among the launch's matrices?
uint32_t tc_room(const huffllm_desc *const *d, uint32_t n, uint32_t npad, const TcShape &sh, uint32_t flat, uint32_t dyn_smem) {
    SmemNeeds need = smem_needs(d[0]);
    if (d[0]->dtype == HUFFLLM_FP16 && d[0]->lut_bits <= 8) need.table_bytes = fp16_table_bytes(flat);   // (a launch-wide choice)
    for (uint32_t i = 1; i < n; ++i) {
        const SmemNeeds o = smem_needs(d[i]);
        if (o.slot_bytes > need.slot_bytes) need.slot_bytes = o.slot_bytes;
        if (o.guard_bytes > need.guard_bytes) need.guard_bytes = o.guard_bytes;
    }
    return planned_warps(need.table_align, need.table_bytes, 2ull * need.slot_bytes, dyn_smem, sh.part_bytes(npad), need.guard_bytes);
}
bool tc_fits(const huffllm_desc *const *d, uint32_t n, uint32_t npad, const TcShape &sh, uint32_t flat, uint32_t dyn_smem) {
    return tc_room(d, n, npad, sh, flat, dyn_smem) >= sh.decoders();
}
// The shapes a launch chooses from: 0 = one slice, as many tiles of rows as find room; 1 = one slice and a warp of its own for
// the activations (at the widest batch padding: there the issuer, which carries them otherwise, bounds the CTA, 8192 x 28672
// at 64 vectors 149 us against 133 with one decoder fewer); 2, 3 = two and four slices; 4 = one slice and as many row groups as
// have room, where whole tiles would be eight (large records, as FP16 has: a CTA of eight warps waits for its lookups).
// False: it does not fit or apply.
constexpr uint32_t kTcShapes = 5;
bool tc_shape(const huffllm_desc *const *d, uint32_t n, uint32_t npad, uint32_t which, uint32_t flat, uint32_t dyn_smem, TcShape *sh) {
    const uint32_t slices = which < 2 || which == 4 ? 1 : which == 2 ? 2 : 4;
    // three stages, two at the widest batch padding, where tensor memory holds no more; the CTA's last warp issues the MMAs
    *sh = TcShape{4 / slices, slices, npad == 64 ? 2u : 3u, 32 / slices - (which == 1 ? 2 : 1)};
    if (which == 0) {
        for (; sh->na; --sh->na) {
            sh->row_groups = sh->na == 4 ? 31 : 8 * sh->na;
            if (tc_fits(d, n, npad, *sh, flat, dyn_smem)) return true;
        }
        return false;
    }
    if (which == 4) {                                        // (its room does not depend on the row groups)
        sh->row_groups = tc_room(d, n, npad, *sh, flat, dyn_smem);
        sh->na = 2;
        return sh->row_groups > 8 && sh->row_groups < 16;
    }
    if (which == 1 && npad != 64) return false;
    if (slices == 4 && npad == 64) return false;             // (seven row groups' worth of rows do not pay for 64 columns of sums)
    for (; sh->stages >= 2; --sh->stages)
        if (tc_fits(d, n, npad, *sh, flat, dyn_smem)) return true;
    return false;
}

// The plan of one matrix: its row tiles and the ranges its column chunks are cut into.
struct TcPlan {
    uint32_t m_tiles, ksplit, items;
    uint32_t chunks;          // most column chunks that one accumulator adds up
    uint64_t span;            // estimated time of the CTA that works longest, and of the last sum
    size_t ticket_off, partial_off, bytes;
};
// Estimated costs, in 1/32 of the time that a CTA of one slice takes for a block of 32 columns (0.93 us, 31 decoders).  Time
// stamps: with two slices (30 decoders) a block takes 0.99 us, with four (28) 1.14; an item's start and epilogue take 5 to 6 us,
// with several slices, whose pieces are smaller, 4.5; the last CTA's sum of a row tile's pieces 9 us for 16 ranges of 16 columns
// per warp, 5.5 for 5 of 16, 6 for 14 of 8.  (The term for that sum is a line through the origin: 4.7 and 6.5 us for the last two;
// 14.9 for the first, where it stands against plans of 16 ranges and one slice, which no measured shape was better off with.)
// At the widest padding two slices leave one slice's activations to the issuer, beside 16 MMAs per stage: 36 instead of 34.  (With
// 34, 28672 x 4096 at 64 vectors took two slices, 99 us, instead of one and a warp for the activations, 91; with 38, 25088 x 7168
// in chunks of 2048 would go the other way, 153 instead of 141.)
// With nine to fifteen row groups (shape 4) a block takes longer than with the eight of shape 0, because the warps share issue slots, and so does
// an item: least squares over 130 launches measured in both shapes, the estimate 4 % (FP16) and 7 % (BF16) off.
constexpr uint32_t kTcUnit = 32;
struct TcCost {
    uint32_t block, item;
};
TcCost tc_cost(const TcShape &sh, uint32_t npad, bool fp16) {
    if (sh.part_filled()) return {fp16 ? 39u : 36u, 8 * kTcUnit};
    return {sh.slices == 1 ? kTcUnit : sh.slices == 2 ? (npad == 64 ? 36u : 34u) : 39u, 5 * kTcUnit};
}
uint32_t tc_sum_cost(const TcShape &sh, uint32_t npad, uint32_t ks) { return ks > 1 ? 2 * ks * sh.piece_columns(npad) : 0; }
// The longest any CTA works when `ks` column ranges of `m_tiles` row tiles are dealt to `sms` CTAs: CTA b takes items b,
// b + grid, ... in turn.  Item i is of range i mod ks, so what a CTA gets depends on b mod ks and on whether it has an item
// in the last round: one sum per residue instead of one per CTA.  (Walking every item of every candidate took 15 to 30 us
// of host time per matrix and launch: the four launches of a 7B-shaped layer at 32 vectors were bound by it, 225 us a layer
// for 165 us of GPU time.)
uint64_t tc_span(const huffllm_desc *d, const TcShape &sh, TcCost price, uint32_t m_tiles, uint32_t ks, uint32_t sms) {
    const uint64_t items = (uint64_t)m_tiles * ks;
    const uint32_t grid = (uint32_t)(items < sms ? items : sms), rounds = (uint32_t)((items + grid - 1) / grid);
    const uint32_t in_last = (uint32_t)(items - (uint64_t)(rounds - 1) * grid);      // CTAs with an item in the last round: the first ones
    const uint32_t chunk_cost = d->chunk_cols / kBlockCols * price.block, step = grid % ks;
    uint64_t cost[16];                                                               // of an item of range r
    for (uint32_t r = 0, at = 0; r < ks; ++r) {
        const uint32_t end = d->col_chunks * (r + 1) / ks;       // (at most 2^26 chunks: the product fits)
        cost[r] = (uint64_t)((end - at + sh.slices - 1) / sh.slices) * chunk_cost + price.item;
        at = end;
    }
    uint64_t span = 0;
    for (uint32_t rho = 0; rho < ks && rho < grid; ++rho) {
        const uint32_t n = rho < in_last ? rounds : rounds - 1;                      // CTA rho has the most items of its residue
        uint64_t sum = 0;
        for (uint32_t i = 0, r = rho; i < n; ++i) {
            sum += cost[r];
            r = r + step >= ks ? r + step - ks : r + step;
        }
        if (sum > span) span = sum;
    }
    return span;
}
// `sms`: the CTAs this matrix can have (all SMs, or its share of a launch over several matrices); `max_bytes`: the workspace
// at hand (column ranges whose pieces would not fit are not considered: a share of the SMs can favour more ranges than the
// whole GPU, for which workspaces are sized); `max_chunks`: the most column chunks that one accumulator may add up; `min_ranges`: the
// fewest ranges.
TcPlan tc_plan(const huffllm_desc *d, uint32_t npad, uint32_t sms, const TcShape &sh, size_t max_bytes, uint32_t max_chunks,
               uint32_t min_ranges = 1) {
    TcPlan p;
    p.m_tiles = (d->row_groups + sh.row_groups - 1) / sh.row_groups;
    const size_t item_bytes = (size_t)32 * sh.piece_columns(npad) * 32 * sizeof(float);
    // Column ranges: in shape 0 (no limit on the chunks) the count whose items are done first, their sums not considered (fewer,
    // longer ranges would be a little faster, but an accumulator's error grows with the columns it adds up: 1e-6 for 1024,
    // 3.8e-6 for 3584); in the others all costs count, and no accumulator may add up more columns than in shape 0.  For row groups that
    // fill no tile ranges are counted as if blocks and items were cheaper than they are, which makes for more of them and shorter
    // sums (20000 x 1024 FP16 at 32 in two ranges 30.3 us and 6.4e-7 from 64 bits, in four 32.5 and 3.4e-7); whether it pays is up to what they cost.
    const bool base = max_chunks == ~0u;
    const TcCost price = tc_cost(sh, npad, d->dtype == HUFFLLM_FP16);
    const TcCost ranges_price = sh.part_filled() ? TcCost{kTcUnit * (14 + sh.row_groups) / (14 + 8), 5 * kTcUnit} : price;
    uint32_t best = 0;
    uint64_t best_span = ~0ull;
    for (uint32_t ks = min_ranges; ks <= 16 && ks <= d->col_chunks; ++ks) {
        if (ks > 1 && ws_partial_offset(d) + (size_t)p.m_tiles * ks * item_bytes > max_bytes) break;
        const uint32_t range = (d->col_chunks + ks - 1) / ks;
        if ((range + sh.slices - 1) / sh.slices > max_chunks) continue;
        const uint64_t span = tc_span(d, sh, ranges_price, p.m_tiles, ks, sms) + (base ? 0 : tc_sum_cost(sh, npad, ks));
        if (span < best_span) { best_span = span; best = ks; }
    }
    if (best && sh.part_filled()) best_span = tc_span(d, sh, price, p.m_tiles, best, sms) + tc_sum_cost(sh, npad, best);
    p.ksplit = best;                                     // (0: no number of ranges is within the limits)
    p.items = p.m_tiles * best;
    // (at the widest padding an issuer that carries the activations of four tiles as well makes a block take an eighth longer)
    p.span = !best ? ~0ull : !base ? best_span : (npad == 64 && sh.na == 4 ? best_span * 9 / 8 : best_span) + tc_sum_cost(sh, npad, best);
    p.chunks = best ? ((d->col_chunks + best - 1) / best + sh.slices - 1) / sh.slices : 0;
    // the counters' region is sized for the smallest tile (most row tiles), so that plans for different batch sizes
    // sharing one workspace never put partial sums where another plan keeps counters
    p.ticket_off = ws_ctrl_bytes(d);
    p.partial_off = ws_partial_offset(d);
    p.bytes = p.partial_off + (best > 1 ? p.items * item_bytes : 0);
    return p;
}
// The shape and plans of a launch over n matrices with cta[i] CTAs each: the shape whose slowest matrix is done first among those
// whose plans fit `max_bytes` of workspace.  No accumulator may add up more columns than in shape 0 without a limit on the
// workspace: what a caller hands over as workspace decides about time, not about rounding.  (With the limit taken from a shape-0
// plan that the workspace had already cut, 28672 x 4096 at 64 vectors in a workspace of exactly the size asked for added up 2048
// columns instead of 1024.)  Only where no plan of any shape is within both, the cut shape-0 plan is the measure.
// False: no shape fits.
bool tc_best(const huffllm_desc *const *d, uint32_t n, uint32_t npad, const uint32_t *cta, uint32_t flat, uint32_t dyn_smem, size_t max_bytes,
             TcShape *shape, TcPlan *plans) {
    TcShape base;
    if (!tc_shape(d, n, npad, 0, flat, dyn_smem, &base)) return false;
    for (size_t base_bytes = ~(size_t)0;; base_bytes = max_bytes) {
        uint64_t best_span = ~0ull;
        uint32_t most[kMaxMats], ranges[kMaxMats];
        for (uint32_t which = 0; which < kTcShapes; ++which) {
            TcShape sh = base;
            // Row groups that fill no tile can pay where a CTA of whole tiles has eight and every CTA has 32 chunks or more to decode; the
            // estimate decides.  (Whole tiles / this, us: FP16 28672 x 8192 at 32 vectors 276 / 263, 11008 x 4096 at 32 61.5 / 58.3, 20000 x 1024 at
            // 32 36.6 / 32.4, 4096 x 14336 at 64 79.5 / 73.4; 9-bit BF16 in chunks of 8192 12288 x 12288 at 32 139 / 127; BF16 in chunks of 16384 20000 x
            // 4096 at 24 97 / 91.  67 launches of drawn sizes, records and formats that took it: 0.95 to 1.63 times as fast, four of them slower than
            // whole tiles.  With a block cost of 14 + n for n row groups and an item cost of 5 units 28 of 89 were slower, FP16 25088 x 7168
            // at 64 218 / 286.  30 chunks a CTA, 9000 x 2048 at 64 26.6 / 27.6, 15, 9000 x 1024 at 17 14.2 / 16.1.  Sixteen warps and more use the
            // issue slots already: BF16 20000 x 4096 at 32 in chunks of 8192 70.5 / 74.1, FP16 12288 x 12288 at 32 in chunks of 2048 109.6 / 121.3.)
            // A row is cut into no fewer ranges than in shape 0: its error grows with the columns of an average range as well, 11008 x 4096
            // FP16 at 32 in four ranges of four chunks is 1.25e-6 from 64 bits, in five 1.03e-6, in seven, as it is now, 0.77e-6.
            if (which == 4) {
                bool pays = base.na == 1;
                for (uint32_t i = 0; i < n; ++i) pays = pays && d[i]->n_chunks >= 32ull * cta[i];
                if (!pays) continue;
            }
            if (which && !tc_shape(d, n, npad, which, flat, dyn_smem, &sh)) continue;
            TcPlan p[kMaxMats];
            uint64_t span = 0;
            for (uint32_t i = 0; i < n; ++i) {
                p[i] = tc_plan(d[i], npad, cta[i], sh, which ? max_bytes : base_bytes, which ? most[i] : ~0u, which == 4 ? ranges[i] : 1u);
                const uint64_t t = p[i].bytes > max_bytes ? ~0ull : p[i].span;
                if (t > span) span = t;
                if (which == 0) {
                    most[i] = p[i].chunks;
                    ranges[i] = p[i].ksplit ? p[i].ksplit : 1u;
                }
            }
            if (span < best_span) {
                best_span = span;
                *shape = sh;
                for (uint32_t i = 0; i < n; ++i) plans[i] = p[i];
            }
        }
        if (best_span != ~0ull) return true;
        if (base_bytes == max_bytes) return false;
    }
}

// The same with the choice of the exponent's table where FP16 mantissa codes are flat: a copy per lane where no accumulator adds up
// more chunks for the 16 KB (the workspace at hand does not decide).  With fewer tiles a CTA because of it, 12288 x 12288 at 32
// vectors in chunks of 2048 took 121.5 us and was 4.9e-6 from 64 bits, with sixteen copies 117.8 and 1.7e-6; in chunks of 1024, where
// all tiles fit either way, 8192 x 8192 at 24 took 56.0 us with a copy per lane and 58.0 with sixteen.
bool tc_choose(const huffllm_desc *const *d, uint32_t n, uint32_t npad, const uint32_t *cta, uint32_t *flat, uint32_t dyn_smem, size_t max_bytes,
               TcShape *shape, TcPlan *plans) {
    // (room for 32 decoders beside the larger table and the most stages that a shape has: every shape fits beside either table, and
    // so the plans are the same)
    const uint32_t slices = npad == 64 ? 2 : 4;
    if (*flat == kFlatBoth && tc_fits(d, n, npad, TcShape{4 / slices, slices, npad == 64 ? 2u : 3u, 32 / slices}, kFlatBothLanes, dyn_smem))
        *flat = kFlatBothLanes;
    if (*flat != kFlatBoth) return tc_best(d, n, npad, cta, *flat, dyn_smem, max_bytes, shape, plans);
    TcShape wide;
    TcPlan wide_plans[kMaxMats];
    const bool tight = tc_best(d, n, npad, cta, kFlatBoth, dyn_smem, ~(size_t)0, shape, plans);
    bool lanes = tc_best(d, n, npad, cta, kFlatBothLanes, dyn_smem, ~(size_t)0, &wide, wide_plans);
    for (uint32_t i = 0; lanes && tight && i < n; ++i) lanes = wide_plans[i].chunks <= plans[i].chunks;
    if (!lanes && !tight) return false;
    if (lanes) {
        *flat = kFlatBothLanes;
        *shape = wide;
        for (uint32_t i = 0; i < n; ++i) plans[i] = wide_plans[i];
    }
    for (uint32_t i = 0; i < n; ++i)
        if (plans[i].bytes > max_bytes) return tc_best(d, n, npad, cta, *flat, dyn_smem, max_bytes, shape, plans);
    return true;
}

// Start a launch description.
void begin_args(KernelArgs *k, uint32_t batch, const DeviceInfo &dev) {
    memset(k, 0, sizeof(*k));
    k->batch = batch;
    k->dyn_smem_bytes = (uint32_t)dev.smem_optin - kStaticSmem;
}

// Append one matrix to a launch description (checks the descriptor and the blob pointer).
huffllm_status add_matrix(KernelArgs *k, const huffllm_desc *desc, const void *blob) {
    huffllm_status st = check_desc(desc);
    if (st != HUFFLLM_OK) return st;
    if (!blob || ((uintptr_t)blob & 255)) return fail(HUFFLLM_ERR_INVALID_ARG, "blob must be a 256-byte aligned device pointer");
    const uint32_t fmt = desc->dtype == HUFFLLM_FP16 ? 1u : 0u;

    if (k->n_mats && k->fmt != fmt) return fail(HUFFLLM_ERR_UNSUPPORTED, "matrices of one call must share the dtype");
    k->fmt = fmt;
    if (k->n_mats == kMaxMats) return fail(HUFFLLM_ERR_UNSUPPORTED, "at most %u matrices per call", kMaxMats);
    if (k->n_mats && k->lut_bits != desc->lut_bits)
        return fail(HUFFLLM_ERR_UNSUPPORTED, "matrices of one call must share max_code_len");
    if (desc->n_chunks + k->total_chunks >= (1ull << 31)) return fail(HUFFLLM_ERR_UNSUPPORTED, "too many chunks for one launch");
    MatArgs &m = k->m[k->n_mats++];
    m.blob = (const uint8_t *)blob;
    m.off_lut = desc->off_lut;
    m.off_index = desc->off_index;
    m.off_payload = desc->off_payload;
    m.payload_units = (uint32_t)(desc->payload_bytes / kRecordUnit);
    m.rows = desc->rows;
    m.cols = desc->cols;
    m.n_chunks = (uint32_t)desc->n_chunks;
    m.chunk_cols = desc->chunk_cols;
    m.col_chunks = desc->col_chunks;
    k->total_chunks += m.n_chunks;
    k->lut_bits = desc->lut_bits;
    // (flat mantissa codes: those that every matrix of the launch has)
    k->fp16_flat = k->n_mats == 1 ? flat_of(desc) : flat_of_both(k->fp16_flat, flat_of(desc));
    const SmemNeeds need = smem_needs(desc);
    k->lut_align = need.table_align;
    k->lut_size = need.table_bytes;
    if (need.slot_bytes > k->slot_bytes) k->slot_bytes = need.slot_bytes;
    if (need.guard_bytes > k->guard_bytes) k->guard_bytes = need.guard_bytes;
    return HUFFLLM_OK;
}

// The tensor-core kernel's part of a launch description.
void set_tc_shape(KernelArgs *k, uint32_t npad, const TcShape &sh, uint32_t flat) {
    k->fp16_flat = flat;
    if (k->fmt) k->lut_size = fp16_table_bytes(flat);
    k->part_bytes = sh.part_bytes(npad);
    k->slots = 2;
    k->pair_recip = (uint32_t)(0x100000000ull / (2ull * k->slot_bytes));
    k->tc_npad = npad;
    k->tc_tiles = sh.na;
    k->tc_slices = sh.slices;
    k->tc_stages = sh.stages;
    k->tc_row_groups = sh.row_groups;
}

// Does a decode send its rows through shared memory?  Rows of a multiple of 8 columns start on 16-byte boundaries (the output
// does) and are stored directly, also where multiples of 8 that are not multiples of 16 make rows straddle sectors: the detour
// reads a word behind a piece whose row starts on a 32-byte boundary, for which a tile's last row has no room (it never does
// off 16 bytes), and has little to give there (28672 x 8184 stored directly takes 250 us, 28672 x 8188 through shared memory 245).
// Other rows pay for the detour from 64 columns and 3/4 2^20 weights on: below that a launch is bound by its set-up and a warp's
// few blocks, and direct stores, many as they are, take less (BF16, chunks of 4096, direct / through shared memory:
// 100000 x 7 12.2 / 15.7 us, 100000 x 33 19.2 / 19.6, 1000 x 515 13.6 / 13.3; 4096 x 257 14.2 / 14.2, 30000 x 65 15.5 / 14.3,
// 1000 x 1027 15.6 / 14.4, 11007 x 4099 186 / 59).
bool rows_through_smem(const MatArgs &m) { return m.cols % 8 && m.cols >= 64 && m.rows * m.cols >= 3ull << 18; }

// Close a launch description: shared-memory budget and grid size.
huffllm_status finish_args(KernelArgs *k, bool product, const DeviceInfo &dev, uint32_t *grid, uint32_t *warps_at_least = nullptr) {
    // (pieces that warps of a CTA exchange: in shared memory up to 8 vectors, in the workspace above)
    if (product) k->part_bytes = k->batch <= kKernelBatch ? 2 * 32 * 16 * k->batch * (uint32_t)sizeof(float) : 0;
    // Two slots per decoder warp, so that a warp's next record lands while it decodes this one.  Where records are so large
    // that this would leave fewer than 31 warps a slot pair, and single slots serve at least a quarter more warps, every
    // warp gets one slot: more decoders at work outweigh the wait for a copy at every chunk start.
    const uint64_t max_w = 31;                                       // decoder warps of a CTA of 1024 threads
    // (decode with rows that go through shared memory: every warp takes room for the rows it works on, as many warps as find
    // both a slot and that room; one always does: its room is no larger than the guard area)
    const bool row_bufs = !product && rows_through_smem(k->m[0]);
    auto warps_with = [&](uint64_t pair_bytes) -> uint64_t {
        uint64_t best = 0;
        for (uint64_t n = row_bufs ? max_w : 1; n > best; --n) {
            if (row_bufs) k->part_bytes = (uint32_t)n * 16 * kRowBuf;
            const uint64_t w = planned_warps(k->lut_align, k->lut_size, pair_bytes, k->dyn_smem_bytes, k->part_bytes, k->guard_bytes);
            const uint64_t got = row_bufs ? (w < n ? w : n) : (w < max_w ? w : max_w);
            if (got > best) best = got;
            if (!row_bufs) break;
        }
        return best;
    };
    // slots and warps with the table(s) that `flat` asks for; false: not even one warp finds its slots
    uint32_t warps = 0;
    auto fit = [&](uint32_t flat) -> bool {
        k->fp16_flat = flat;
        if (k->fmt && k->lut_bits <= 8) k->lut_size = fp16_table_bytes(flat);
        const bool single_ok = k->fmt || k->lut_bits == 8;            // (the kernels that exist with single slots)
        const uint64_t w2 = warps_with(2ull * k->slot_bytes), w1 = single_ok && w2 < max_w ? warps_with(k->slot_bytes) : 0;
        k->slots = w1 && 4 * w1 >= 5 * w2 ? 1u : 2u;
        warps = (uint32_t)(k->slots == 1 ? w1 : w2);
        if (row_bufs) k->part_bytes = warps * 16 * kRowBuf;
        return warps != 0;
    };
    // (flat FP16 mantissa codes, see below: a table per lane that leaves decode a warp, or a product all of them, needs no comparison)
    const uint32_t flat = k->fp16_flat;
    bool lanes = flat == kFlatBoth && fit(kFlatBothLanes);
    const uint32_t lanes_warps = lanes ? warps : 0, lanes_slots = k->slots;
    lanes = lanes && (!product || warps == max_w);
    if (!lanes && !fit(flat)) return fail(HUFFLLM_ERR_UNSUPPORTED, "chunk records too large for shared memory (slot %u bytes)", k->slot_bytes);
    uint64_t g = k->total_chunks < (uint64_t)dev.sms ? k->total_chunks : (uint64_t)dev.sms;
    *grid = (uint32_t)(g < kMaxGrid ? g : kMaxGrid);
    // deal the CTAs out to the matrices: one each, then always to the matrix with the most chunks per CTA, so that
    // the largest piece is as small as it can be and no CTA works in two matrices
    if (*grid < k->n_mats) return fail(HUFFLLM_ERR_UNSUPPORTED, "more matrices than SMs");
    uint32_t cnt[kMaxMats];
    for (uint32_t i = 0; i < k->n_mats; ++i) cnt[i] = 1;
    for (uint32_t left = *grid - k->n_mats; left; --left) {
        uint32_t best = k->n_mats;
        for (uint32_t i = 0; i < k->n_mats; ++i) {
            if (cnt[i] >= k->m[i].n_chunks) continue;
            if (best == k->n_mats || (uint64_t)k->m[i].n_chunks * cnt[best] > (uint64_t)k->m[best].n_chunks * cnt[i]) best = i;
        }
        if (best == k->n_mats) break;
        ++cnt[best];
    }
    uint32_t first = 0;
    for (uint32_t i = 0; i < k->n_mats; ++i) {
        k->m[i].cta_first = first;
        k->m[i].cta_count = cnt[i];
        k->m[i].cta_chunks = k->m[i].n_chunks / cnt[i];
        k->m[i].cta_extra = k->m[i].n_chunks % cnt[i];
        first += cnt[i];
    }
    *grid = first;
    // Flat FP16 mantissa codes: the exponent's table with a copy per lane has no bank conflicts, but takes 16 KB that decoder warps
    // want for their slots.  It is taken where no warp's accumulators add up more chunks for it, nor, in chunks so long that warps
    // have single slots, any warp is lost (decode adds up nothing).  FP16 11008 x 4096, sixteen copies / one per lane, us and the
    // relative error against 64 bits: one vector, chunks of 4096 (26 / 24 warps) 29.2, 2.30e-7 / 31.4, 2.39e-7, chunks of 2048 (27 /
    // 25, six chunks a warp either way) 27.0, 2.31e-7 / 29.5, 2.11e-7; 8 vectors, chunks of 1024 (31 / 31) 36.6 / 35.8 and no
    // difference, of 4096 (24 / 22) 35.6, 9.5e-7 / 32.0, 10.3e-7, of 8192 (12 / 10) 42.7, 1.76e-6 / 41.0, 2.05e-6.
    if (flat == kFlatBoth && !lanes && lanes_warps) {
        auto longest_sum = [&](const MatArgs &m, uint32_t with) -> uint32_t {
            const uint32_t chunks = (m.cta_chunks + (m.cta_extra ? 1u : 0u) + with - 1) / with;
            return chunks < m.col_chunks ? chunks : m.col_chunks;
        };
        lanes = k->slots == 2 || lanes_warps >= warps;
        for (uint32_t i = 0; lanes && i < k->n_mats; ++i) lanes = longest_sum(k->m[i], lanes_warps) <= longest_sum(k->m[i], warps);
        if (lanes) {
            k->fp16_flat = kFlatBothLanes;
            k->lut_size = fp16_table_bytes(kFlatBothLanes);
            k->slots = lanes_slots;
            warps = lanes_warps;
        }
    }
    if (warps_at_least) *warps_at_least = warps;
    k->pair_recip = (uint32_t)(0x100000000ull / ((uint64_t)k->slots * k->slot_bytes));
    return HUFFLLM_OK;
}

}  // namespace

extern "C" {

huffllm_status huffllm_workspace_bytes(const huffllm_desc *desc, uint32_t batch, size_t *bytes) {
    clear_error();
    if (!bytes) return fail(HUFFLLM_ERR_INVALID_ARG, "bytes is null");
    huffllm_status st = check_desc(desc);
    if (st != HUFFLLM_OK) return st;
    if (batch == 0 || batch > 64) return fail(HUFFLLM_ERR_INVALID_ARG, "batch must be in [1, 64]");
    *bytes = ws_bytes_for(desc, batch);     // (above 8 vectors: what passes of 8 need, should the tensor-core kernel not fit)
    if (batch > kKernelBatch) {      // the tensor-core path keeps partial tiles of its column ranges here
        DeviceInfo dev;       // without a device (a host-only caller sizing buffers): the B200's figures
        const bool have = device_info(&dev) == HUFFLLM_OK;
        clear_error();
        const int sms = have ? dev.sms : 148;
        const uint32_t dyn = (have ? (uint32_t)dev.smem_optin : 232448u) - kStaticSmem;
        const uint32_t cta = (uint32_t)sms;
        // The plan that will run for this and for every smaller batch, and the shape-0 plan, which a launch over several matrices
        // may fall back on; with all three FP16 tables, and with those that flat codes leave.
        for (uint32_t npad = 16; npad <= tc_npad_of(batch); npad *= 2)
            for (uint32_t flat : {kFlatNone, kFlatUpper, kFlatBoth, kFlatBothLanes}) {
                const uint32_t have_flat = flat == kFlatBothLanes ? kFlatBoth : flat;
                if (flat != kFlatNone && flat_of_both(have_flat, flat_of(desc)) != have_flat) continue;
                TcShape sh;
                TcPlan p;
                if (!tc_best(&desc, 1, npad, &cta, flat, dyn, ~(size_t)0, &sh, &p)) continue;
                if (p.bytes > *bytes) *bytes = p.bytes;
                if (!tc_shape(&desc, 1, npad, 0, flat, dyn, &sh)) continue;
                p = tc_plan(desc, npad, cta, sh, ~(size_t)0, ~0u);
                if (p.bytes > *bytes) *bytes = p.bytes;
            }
    }
    return HUFFLLM_OK;
}

huffllm_status huffllm_workspace_control_bytes(const huffllm_desc *desc, size_t *bytes) {
    clear_error();
    if (!bytes) return fail(HUFFLLM_ERR_INVALID_ARG, "bytes is null");
    huffllm_status st = check_desc(desc);
    if (st != HUFFLLM_OK) return st;
    *bytes = ws_partial_offset(desc);
    return HUFFLLM_OK;
}

huffllm_status huffllm_decode_smem_plan(const huffllm_desc *desc, uint32_t *table_bytes, uint32_t *slot_bytes,
                                        uint32_t *refill_checks_per_block, uint32_t *guard_bytes) {
    clear_error();
    huffllm_status st = check_desc(desc);
    if (st != HUFFLLM_OK) return st;
    const SmemNeeds n = smem_needs(desc);
    if (table_bytes) *table_bytes = n.table_bytes;
    if (slot_bytes) *slot_bytes = n.slot_bytes;
    if (refill_checks_per_block) *refill_checks_per_block = n.checks_per_block;
    if (guard_bytes) *guard_bytes = n.guard_bytes;
    return HUFFLLM_OK;
}

huffllm_status huffllm_decode_launch_plan(const huffllm_desc *desc, uint32_t batch, uint32_t smem_bytes_per_cta,
                                          uint32_t *slots_per_warp, uint32_t *decoder_warps) {
    clear_error();
    huffllm_status st = check_desc(desc);
    if (st != HUFFLLM_OK) return st;
    if (batch > kKernelBatch) return fail(HUFFLLM_ERR_INVALID_ARG, "the plan is that of the register path: batch 0 (decode) to %u", kKernelBatch);
    DeviceInfo dev = {};
    dev.sms = 148;
    dev.smem_optin = smem_bytes_per_cta ? smem_bytes_per_cta : 232448;
    KernelArgs k;
    uint32_t grid = 0, warps = 0;
    begin_args(&k, batch ? batch : 1, dev);
    if ((st = add_matrix(&k, desc, (const void *)256)) != HUFFLLM_OK) return st;     // (the pointer is only checked for alignment)
    if ((st = finish_args(&k, batch != 0, dev, &grid, &warps)) != HUFFLLM_OK) return st;
    if (slots_per_warp) *slots_per_warp = k.slots;
    if (decoder_warps) *decoder_warps = warps;
    return HUFFLLM_OK;
}

huffllm_status huffllm_gemm_launch_plan(uint32_t n, const huffllm_desc *const *descs, uint32_t batch, size_t workspace_bytes_each,
                                        uint32_t *column_slices, uint32_t *row_groups, uint32_t *ranges, uint32_t *work_items,
                                        uint32_t *chunks_per_sum) {
    clear_error();
    if (!descs) return fail(HUFFLLM_ERR_INVALID_ARG, "null pointer");
    if (n == 0 || n > kMaxMats) return fail(HUFFLLM_ERR_INVALID_ARG, "between 1 and %u matrices per call", kMaxMats);
    if (batch <= kKernelBatch || batch > 64) return fail(HUFFLLM_ERR_INVALID_ARG, "the plan is that of the tensor-core path: batch %u to 64", kKernelBatch + 1);
    DeviceInfo dev;
    if (device_info(&dev) != HUFFLLM_OK) {
        clear_error();
        dev.sms = 148;
        dev.smem_optin = 232448;
    }
    KernelArgs k;
    uint32_t grid = 0, cta[kMaxMats];
    begin_args(&k, batch, dev);
    huffllm_status st;
    for (uint32_t i = 0; i < n; ++i) {
        if ((st = add_matrix(&k, descs[i], (const void *)256)) != HUFFLLM_OK) return st;     // (the pointer is only checked for alignment)
        if (!tc_blob(descs[i])) return fail(HUFFLLM_ERR_UNSUPPORTED, "the tensor-core path takes tables of up to 9 bits (FP16: 8)");
    }
    uint32_t flat = k.fp16_flat;
    if (n > 1 && (st = finish_args(&k, true, dev, &grid)) != HUFFLLM_OK) return st;
    for (uint32_t i = 0; i < n; ++i) cta[i] = n > 1 ? k.m[i].cta_count : (uint32_t)dev.sms;
    TcShape sh;
    TcPlan plans[kMaxMats];
    if (!tc_choose(descs, n, tc_npad_of(batch), cta, &flat, k.dyn_smem_bytes, workspace_bytes_each ? workspace_bytes_each : ~(size_t)0, &sh, plans))
        return fail(HUFFLLM_ERR_UNSUPPORTED, "chunk records too large for the tensor-core kernel's slots");
    if (column_slices) *column_slices = sh.slices;
    if (row_groups) *row_groups = sh.row_groups;
    for (uint32_t i = 0; i < n; ++i) {
        if (ranges) ranges[i] = plans[i].ksplit;
        if (work_items) work_items[i] = plans[i].items;
        if (chunks_per_sum) chunks_per_sum[i] = plans[i].chunks;
    }
    return HUFFLLM_OK;
}

huffllm_status huffllm_decode(const huffllm_desc *desc, const void *blob, uint16_t *out, int32_t *err_flag, huffllm_stream stream) {
    clear_error();
    DeviceInfo dev;
    huffllm_status st = device_info(&dev);
    if (st != HUFFLLM_OK) return st;
    if (!out || ((uintptr_t)out & 15)) return fail(HUFFLLM_ERR_INVALID_ARG, "out must be a 16-byte aligned device pointer");
    KernelArgs k;
    uint32_t grid;
    begin_args(&k, 1, dev);
    if ((st = add_matrix(&k, desc, blob)) != HUFFLLM_OK) return st;
    if ((st = finish_args(&k, false, dev, &grid)) != HUFFLLM_OK) return st;
    k.m[0].out = out;
    k.err = err_flag;
    cudaError_t e = launch_decode(k, grid, (cudaStream_t)stream);
    if (e != cudaSuccess) return fail(HUFFLLM_ERR_CUDA, "decode launch: %s", cudaGetErrorString(e));
    return HUFFLLM_OK;
}

// Checks shared by the product entry points for one matrix of a call.
static huffllm_status check_product_args(const huffllm_desc *desc, const uint16_t *x, const float *y, const void *workspace,
                                         size_t workspace_bytes, uint32_t batch) {
    if (!x || !y || !workspace) return fail(HUFFLLM_ERR_INVALID_ARG, "null pointer");
    if (((uintptr_t)x & 15) || ((uintptr_t)y & 3) || ((uintptr_t)workspace & 255))
        return fail(HUFFLLM_ERR_INVALID_ARG, "x must be 16-byte, y 4-byte, workspace 256-byte aligned");
    huffllm_status st = check_desc(desc);
    if (st != HUFFLLM_OK) return st;
    if (workspace_bytes < ws_bytes_for(desc, batch)) return fail(HUFFLLM_ERR_BUFFER_TOO_SMALL, "workspace too small");
    if (desc->cols % kBlockCols) return fail(HUFFLLM_ERR_UNSUPPORTED, "fused products need cols to be a multiple of 32");
    return HUFFLLM_OK;
}

huffllm_status huffllm_decode_gemm_multi(uint32_t n, const huffllm_desc *const *descs, const void *const *blobs,
                                         const uint16_t *const *xs, uint32_t batch, float *const *ys, void *const *workspaces,
                                         size_t workspace_bytes_each, int32_t *err_flag, huffllm_stream stream) {
    clear_error();
    DeviceInfo dev;
    huffllm_status st = device_info(&dev);
    if (st != HUFFLLM_OK) return st;
    if (!descs || !blobs || !xs || !ys || !workspaces) return fail(HUFFLLM_ERR_INVALID_ARG, "null pointer");
    if (n == 0 || n > kMaxMats) return fail(HUFFLLM_ERR_INVALID_ARG, "between 1 and %u matrices per call", kMaxMats);
    if (batch == 0 || batch > 64) return fail(HUFFLLM_ERR_INVALID_ARG, "batch must be in [1, 64]");
    if (batch > kTwoTileBatch) {
        // 17..64 vectors: the tensor-core kernel, its CTAs dealt to the matrices like the other kernels'
        TcArgs t;
        memset(&t, 0, sizeof(t));
        KernelArgs &k = t.k;
        uint32_t grid;
        begin_args(&k, batch, dev);
        for (uint32_t i = 0; i < n; ++i) {
            if ((st = check_product_args(descs[i], xs[i], ys[i], workspaces[i], workspace_bytes_each, batch)) != HUFFLLM_OK) return st;
            if (!tc_blob(descs[i]))
                return fail(HUFFLLM_ERR_UNSUPPORTED, "more than %u vectors per call over several matrices take tables of up to 9 bits (FP16: 8)", kTwoTileBatch);
            for (uint32_t j = 0; j < i; ++j)
                if (workspaces[j] == workspaces[i]) return fail(HUFFLLM_ERR_INVALID_ARG, "matrices %u and %u share a workspace", j, i);
            if ((st = add_matrix(&k, descs[i], blobs[i])) != HUFFLLM_OK) return st;
            k.m[i].x = xs[i];
            k.m[i].y = ys[i];
        }
        uint32_t flat = k.fp16_flat;
        if ((st = finish_args(&k, true, dev, &grid)) != HUFFLLM_OK) return st;      // (deals the CTAs to the matrices by their chunks)
        const uint32_t npad = tc_npad_of(batch);
        uint32_t cta[kMaxMats];
        for (uint32_t i = 0; i < n; ++i) cta[i] = k.m[i].cta_count;
        TcShape sh;
        TcPlan plans[kMaxMats];
        if (!tc_choose(descs, n, npad, cta, &flat, k.dyn_smem_bytes, workspace_bytes_each, &sh, plans))
            return fail(HUFFLLM_ERR_UNSUPPORTED, "chunk records too large for the tensor-core kernel's slots");
        set_tc_shape(&k, npad, sh, flat);
        uint32_t first = 0;
        for (uint32_t i = 0; i < n; ++i) {
            const TcPlan &tp = plans[i];
            if (workspace_bytes_each < tp.bytes) return fail(HUFFLLM_ERR_BUFFER_TOO_SMALL, "workspace of matrix %u too small for batch %u", i, batch);
            t.m_tiles[i] = tp.m_tiles;
            t.ksplit[i] = tp.ksplit;
            t.ticket[i] = (unsigned int *)((uint8_t *)workspaces[i] + tp.ticket_off);
            t.partial[i] = (float *)((uint8_t *)workspaces[i] + tp.partial_off);
            k.m[i].cta_first = first;
            if (tp.items < k.m[i].cta_count) k.m[i].cta_count = tp.items;
            first += k.m[i].cta_count;
        }
        k.err = err_flag;
        cudaError_t e = launch_gemm_tc(t, first, (cudaStream_t)stream);
        if (e != cudaSuccess) return fail(HUFFLLM_ERR_CUDA, "tensor-core product launch: %s", cudaGetErrorString(e));
        return HUFFLLM_OK;
    }
    KernelArgs k;
    uint32_t grid;
    begin_args(&k, batch, dev);
    for (uint32_t i = 0; i < n; ++i) {
        if ((st = check_product_args(descs[i], xs[i], ys[i], workspaces[i], workspace_bytes_each, batch)) != HUFFLLM_OK) return st;
        if (batch > kKernelBatch && !two_tile_blob(descs[i]))
            return fail(HUFFLLM_ERR_UNSUPPORTED, "more than %u vectors per call take BF16 blobs of max_code_len 8", kKernelBatch);
        for (uint32_t j = 0; j < i; ++j)
            if (workspaces[j] == workspaces[i]) return fail(HUFFLLM_ERR_INVALID_ARG, "matrices %u and %u share a workspace", j, i);
        if ((st = add_matrix(&k, descs[i], blobs[i])) != HUFFLLM_OK) return st;
        MatArgs &m = k.m[i];
        m.x = xs[i];
        m.y = ys[i];
        m.ws_ticket = (unsigned int *)workspaces[i];
        m.ws_partial = (float *)((uint8_t *)workspaces[i] + ws_partial_offset(descs[i]));
        m.ws_warp_pieces = (float *)((uint8_t *)workspaces[i] + ws_partial_offset(descs[i]) + ws_cta_pieces_bytes(batch));   // (used above 8 vectors)
    }
    if ((st = finish_args(&k, true, dev, &grid)) != HUFFLLM_OK) return st;
    k.err = err_flag;
    cudaError_t e = launch_gemm(k, grid, (cudaStream_t)stream);
    if (e != cudaSuccess) return fail(HUFFLLM_ERR_CUDA, "product launch: %s", cudaGetErrorString(e));
    return HUFFLLM_OK;
}

huffllm_status huffllm_decode_gemm(const huffllm_desc *desc, const void *blob, const uint16_t *x, uint32_t batch, float *y,
                                   void *workspace, size_t workspace_bytes, int32_t *err_flag, huffllm_stream stream) {
    clear_error();
    DeviceInfo dev;
    huffllm_status st = device_info(&dev);
    if (st != HUFFLLM_OK) return st;
    if (batch == 0 || batch > 64) return fail(HUFFLLM_ERR_INVALID_ARG, "batch must be in [1, 64]");
    if ((st = check_product_args(desc, x, y, workspace, workspace_bytes, batch)) != HUFFLLM_OK) return st;
    // Paths for more than 8 vectors.  Each returns HUFFLLM_OK with `done` set if it launched, HUFFLLM_OK without if it does
    // not apply here (the next path decides), or an error.
    bool done = false;
    auto two_tiles = [&]() -> huffllm_status {
        // 9..16 vectors on the default BF16 blobs: the register path with two tiles of activations per decoded block
        if (batch > kTwoTileBatch || !two_tile_blob(desc)) return HUFFLLM_OK;
        KernelArgs k;
        uint32_t grid;
        begin_args(&k, batch, dev);
        huffllm_status s2 = add_matrix(&k, desc, blob);
        if (s2 != HUFFLLM_OK) return s2;
        if (finish_args(&k, true, dev, &grid) != HUFFLLM_OK) {
            clear_error();      // records too large for shared memory: another path decides
            return HUFFLLM_OK;
        }
        k.m[0].x = x;
        k.m[0].y = y;
        k.m[0].ws_ticket = (unsigned int *)workspace;
        k.m[0].ws_partial = (float *)((uint8_t *)workspace + ws_partial_offset(desc));
        k.m[0].ws_warp_pieces = (float *)((uint8_t *)workspace + ws_partial_offset(desc) + ws_cta_pieces_bytes(batch));
        k.err = err_flag;
        cudaError_t e = launch_gemm(k, grid, (cudaStream_t)stream);
        if (e != cudaSuccess) return fail(HUFFLLM_ERR_CUDA, "product launch: %s", cudaGetErrorString(e));
        done = true;
        return HUFFLLM_OK;
    };
    auto tensor_core = [&](bool other_path_left) -> huffllm_status {
        // one pass over the compressed weights for the whole batch (tables of up to 9 bits; longer codes take passes of 8
        // vectors through the register-path kernel and its two-level lookup)
        if (!tc_blob(desc)) return HUFFLLM_OK;
        // (column ranges are planned within the workspace at hand)
        const uint32_t npad = tc_npad_of(batch), cta = (uint32_t)dev.sms;
        TcShape sh;
        TcPlan tp;
        uint32_t flat = flat_of(desc);
        if (!tc_choose(&desc, 1, npad, &cta, &flat, (uint32_t)dev.smem_optin - kStaticSmem, workspace_bytes, &sh, &tp))
            return HUFFLLM_OK;      // records too large for this kernel's slots
        TcArgs t;
        memset(&t, 0, sizeof(t));
        KernelArgs &k = t.k;
        begin_args(&k, batch, dev);
        huffllm_status s2 = add_matrix(&k, desc, blob);
        if (s2 != HUFFLLM_OK) return s2;
        set_tc_shape(&k, npad, sh, flat);
        if (workspace_bytes < tp.bytes) {
            if (other_path_left) return HUFFLLM_OK;     // (the register path needs less)
            return fail(HUFFLLM_ERR_BUFFER_TOO_SMALL, "workspace too small for batch %u", batch);
        }
        k.m[0].x = x;
        k.m[0].y = y;
        t.m_tiles[0] = tp.m_tiles;
        t.ksplit[0] = tp.ksplit;
        t.ticket[0] = (unsigned int *)((uint8_t *)workspace + tp.ticket_off);
        t.partial[0] = (float *)((uint8_t *)workspace + tp.partial_off);
        k.err = err_flag;
        const uint32_t grid = tp.items < (uint32_t)dev.sms ? tp.items : (uint32_t)dev.sms;
        k.m[0].cta_first = 0;
        k.m[0].cta_count = grid;
        cudaError_t e = launch_gemm_tc(t, grid, (cudaStream_t)stream);
        if (e != cudaSuccess) return fail(HUFFLLM_ERR_CUDA, "tensor-core product launch: %s", cudaGetErrorString(e));
        done = true;
        return HUFFLLM_OK;
    };
    if (batch > kKernelBatch) {
        // 9..16 vectors: the tensor-core kernel, whose time does not grow with the batch below its padding of 16, is the
        // faster one for matrices that are at least as wide as tall (few row groups per SM make the register path's
        // cross-CTA sums of 16-vector pieces expensive), unless they have so few rows that it gets few row tiles; measured
        // at 12 and 16 vectors on seven shapes from 1024 x 8192 to 28672 x 8192, before that kernel had column slices (the line has
        // not been drawn again).  Above 16 vectors it is the only one.
        const bool wide = desc->cols >= desc->rows && desc->rows >= 2048;
        if (!wide && (st = two_tiles()) != HUFFLLM_OK) return st;
        if (!done && (st = tensor_core(wide && batch <= kTwoTileBatch && two_tile_blob(desc))) != HUFFLLM_OK) return st;
        if (!done && wide && (st = two_tiles()) != HUFFLLM_OK) return st;
        if (done) return HUFFLLM_OK;
        // neither applies (long codes, or chunk records too large for the slots): passes of 8 vectors
    }
    for (uint32_t b0 = 0; b0 < batch; b0 += kKernelBatch) {
        uint32_t nb = batch - b0 < kKernelBatch ? batch - b0 : kKernelBatch;
        KernelArgs k;
        uint32_t grid;
        begin_args(&k, nb, dev);
        if ((st = add_matrix(&k, desc, blob)) != HUFFLLM_OK) return st;
        if ((st = finish_args(&k, true, dev, &grid)) != HUFFLLM_OK) return st;
        k.m[0].x = x + (uint64_t)b0 * desc->cols;
        k.m[0].y = y + (uint64_t)b0 * desc->rows;
        k.m[0].ws_ticket = (unsigned int *)workspace;
        k.m[0].ws_partial = (float *)((uint8_t *)workspace + ws_partial_offset(desc));
        k.err = err_flag;
        cudaError_t e = launch_gemm(k, grid, (cudaStream_t)stream);
        if (e != cudaSuccess) return fail(HUFFLLM_ERR_CUDA, "product launch: %s", cudaGetErrorString(e));
    }
    return HUFFLLM_OK;
}

huffllm_status huffllm_decode_gemv(const huffllm_desc *desc, const void *blob, const uint16_t *x, float *y, void *workspace,
                                   size_t workspace_bytes, int32_t *err_flag, huffllm_stream stream) {
    return huffllm_decode_gemm(desc, blob, x, 1, y, workspace, workspace_bytes, err_flag, stream);
}

huffllm_status huffllm_decode_gemm_multi_host_async(uint32_t n, const huffllm_desc *const *descs, const void *const *blobs,
                                                    const uint16_t *const *xs_host, uint32_t batch, float *const *ys_host,
                                                    uint16_t *const *x_stages, float *const *y_stages, void *const *workspaces,
                                                    size_t workspace_bytes_each, int32_t *err_flag, huffllm_stream stream) {
    clear_error();
    if (!descs || !xs_host || !ys_host || !x_stages || !y_stages) return fail(HUFFLLM_ERR_INVALID_ARG, "null pointer");
    if (n == 0 || n > kMaxMats) return fail(HUFFLLM_ERR_INVALID_ARG, "between 1 and %u matrices per call", kMaxMats);
    if (batch == 0 || batch > 64) return fail(HUFFLLM_ERR_INVALID_ARG, "batch must be in [1, 64]");
    cudaStream_t s = (cudaStream_t)stream;
    for (uint32_t i = 0; i < n; ++i) {     // nothing is enqueued before every argument has been looked at
        if (!descs[i] || !xs_host[i] || !ys_host[i] || !x_stages[i] || !y_stages[i]) return fail(HUFFLLM_ERR_INVALID_ARG, "null pointer");
        huffllm_status st = check_product_args(descs[i], x_stages[i], y_stages[i], workspaces ? workspaces[i] : nullptr,
                                               workspace_bytes_each, batch);
        if (st != HUFFLLM_OK) return st;
        if (!blobs || !blobs[i] || ((uintptr_t)blobs[i] & 255))
            return fail(HUFFLLM_ERR_INVALID_ARG, "blob must be a 256-byte aligned device pointer");
        if (batch > kKernelBatch && batch <= kTwoTileBatch && !two_tile_blob(descs[i]))
            return fail(HUFFLLM_ERR_UNSUPPORTED, "9 to %u vectors per call over several matrices take BF16 blobs of max_code_len 8", kTwoTileBatch);
        if (batch > kTwoTileBatch && !tc_blob(descs[i]))
            return fail(HUFFLLM_ERR_UNSUPPORTED, "more than %u vectors per call over several matrices take tables of up to 9 bits (FP16: 8)", kTwoTileBatch);
    }
    for (uint32_t i = 0; i < n; ++i) {
        cudaError_t e = cudaMemcpyAsync(x_stages[i], xs_host[i], (size_t)batch * descs[i]->cols * 2, cudaMemcpyHostToDevice, s);
        if (e != cudaSuccess) return fail(HUFFLLM_ERR_CUDA, "copy of x: %s", cudaGetErrorString(e));
    }
    huffllm_status st = huffllm_decode_gemm_multi(n, descs, blobs, (const uint16_t *const *)x_stages, batch, y_stages, workspaces,
                                                  workspace_bytes_each, err_flag, stream);
    if (st != HUFFLLM_OK) return st;
    for (uint32_t i = 0; i < n; ++i) {
        cudaError_t e = cudaMemcpyAsync(ys_host[i], y_stages[i], (size_t)batch * descs[i]->rows * 4, cudaMemcpyDeviceToHost, s);
        if (e != cudaSuccess) return fail(HUFFLLM_ERR_CUDA, "copy of y: %s", cudaGetErrorString(e));
    }
    return HUFFLLM_OK;
}

huffllm_status huffllm_decode_gemm_multi_host(uint32_t n, const huffllm_desc *const *descs, const void *const *blobs,
                                              const uint16_t *const *xs_host, uint32_t batch, float *const *ys_host,
                                              uint16_t *const *x_stages, float *const *y_stages, void *const *workspaces,
                                              size_t workspace_bytes_each, int32_t *err_flag, huffllm_stream stream) {
    huffllm_status st = huffllm_decode_gemm_multi_host_async(n, descs, blobs, xs_host, batch, ys_host, x_stages, y_stages, workspaces,
                                                             workspace_bytes_each, err_flag, stream);
    if (st != HUFFLLM_OK) return st;
    cudaError_t e = cudaStreamSynchronize((cudaStream_t)stream);
    if (e != cudaSuccess) return fail(HUFFLLM_ERR_CUDA, "waiting for the stream: %s", cudaGetErrorString(e));
    return HUFFLLM_OK;
}

huffllm_status huffllm_decode_gemm_host(const huffllm_desc *desc, const void *blob, const uint16_t *x_host, uint32_t batch,
                                        float *y_host, uint16_t *x_stage, float *y_stage, void *workspace,
                                        size_t workspace_bytes, int32_t *err_flag, huffllm_stream stream) {
    clear_error();
    if (!desc || !x_host || !y_host || !x_stage || !y_stage) return fail(HUFFLLM_ERR_INVALID_ARG, "null pointer");
    if (batch == 0 || batch > 64) return fail(HUFFLLM_ERR_INVALID_ARG, "batch must be in [1, 64]");
    huffllm_status st0 = check_product_args(desc, x_stage, y_stage, workspace, workspace_bytes, batch);
    if (st0 != HUFFLLM_OK) return st0;       // nothing is enqueued for a call that will be refused
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = cudaMemcpyAsync(x_stage, x_host, (size_t)batch * desc->cols * 2, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return fail(HUFFLLM_ERR_CUDA, "copy of x: %s", cudaGetErrorString(e));
    huffllm_status st = huffllm_decode_gemm(desc, blob, x_stage, batch, y_stage, workspace, workspace_bytes, err_flag, stream);
    if (st != HUFFLLM_OK) return st;
    e = cudaMemcpyAsync(y_host, y_stage, (size_t)batch * desc->rows * 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return fail(HUFFLLM_ERR_CUDA, "copy of y: %s", cudaGetErrorString(e));
    return HUFFLLM_OK;
}

}  // extern "C"

// Scratch of huffllm_decode_gemm_static.  In host code this name is only a handle for the runtime, not a
// device address: the address the kernels get comes from cudaGetSymbolAddress, once per device.
static __device__ __align__(256) unsigned char g_static_scratch[HUFFLLM_STATIC_SCRATCH_BYTES];
static std::atomic<void *> g_static_scratch_addr[64];

extern "C" {

huffllm_status huffllm_decode_gemm_static(const huffllm_desc *desc, const void *blob, const uint16_t *x, uint32_t batch,
                                          float *y, int32_t *err_flag, huffllm_stream stream) {
    clear_error();
    if (batch == 0) return fail(HUFFLLM_ERR_INVALID_ARG, "batch must be at least 1");
    huffllm_status st = check_desc(desc);
    if (st != HUFFLLM_OK) return st;
    if (batch > HUFFLLM_STATIC_MAX_BATCH || ws_bytes_for(desc, batch) > sizeof(g_static_scratch))
        return fail(HUFFLLM_ERR_BUFFER_TOO_SMALL,
                    "this matrix with %u vectors needs %zu bytes of scratch; the built-in array has %u (and takes at most %u vectors)",
                    batch, ws_bytes_for(desc, batch), (unsigned)HUFFLLM_STATIC_SCRATCH_BYTES, (unsigned)HUFFLLM_STATIC_MAX_BATCH);
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return fail(HUFFLLM_ERR_CUDA, "cudaGetDevice: %s", cudaGetErrorString(e));
    if (dev < 0 || dev >= 64) return fail(HUFFLLM_ERR_UNSUPPORTED, "device ordinal %d out of range", dev);
    void *ws = g_static_scratch_addr[dev].load(std::memory_order_acquire);
    if (!ws) {   // set-up, once per device, with that device current (racing threads look up the same address)
        e = cudaGetSymbolAddress(&ws, g_static_scratch);
        if (e != cudaSuccess || !ws) return fail(HUFFLLM_ERR_CUDA, "cudaGetSymbolAddress: %s", cudaGetErrorString(e));
        g_static_scratch_addr[dev].store(ws, std::memory_order_release);
    }
    // Everything that can refuse the call is checked before anything is enqueued: a refused call leaves the array alone.
    DeviceInfo info;
    if ((st = device_info(&info)) != HUFFLLM_OK) return st;
    if ((st = check_product_args(desc, x, y, ws, sizeof(g_static_scratch), batch)) != HUFFLLM_OK) return st;
    {
        KernelArgs k;
        uint32_t grid;
        begin_args(&k, batch, info);
        if ((st = add_matrix(&k, desc, blob)) != HUFFLLM_OK) return st;
        if ((st = finish_args(&k, true, info, &grid)) != HUFFLLM_OK) return st;
    }
    // the array keeps whatever the last call (finished or not) left: the control words must start at zero
    e = cudaMemsetAsync(ws, 0, ws_partial_offset(desc), (cudaStream_t)stream);
    if (e != cudaSuccess) return fail(HUFFLLM_ERR_CUDA, "clearing the built-in scratch: %s", cudaGetErrorString(e));
    return huffllm_decode_gemm(desc, blob, x, batch, y, ws, sizeof(g_static_scratch), err_flag, stream);
}

huffllm_status huffllm_stage_copy(void *dst, const void *src, size_t bytes, huffllm_stream stream) {
    clear_error();
    DeviceInfo dev;
    huffllm_status st = device_info(&dev);
    if (st != HUFFLLM_OK) return st;
    if (!dst || !src) return fail(HUFFLLM_ERR_INVALID_ARG, "null pointer");
    if (bytes % 16 || ((uintptr_t)dst & 15) || ((uintptr_t)src & 15)) return fail(HUFFLLM_ERR_INVALID_ARG, "size and pointers must be multiples of 16 bytes");
    cudaError_t e = launch_stage_copy(dst, src, bytes, (uint32_t)dev.sms, (cudaStream_t)stream);
    if (e != cudaSuccess) return fail(HUFFLLM_ERR_CUDA, "copy launch: %s", cudaGetErrorString(e));
    return HUFFLLM_OK;
}

huffllm_status huffllm_plain_gemv_multi(uint32_t n, const uint16_t *const *ws, const uint64_t *rows, const uint64_t *cols,
                                        const uint16_t *const *xs, float *const *ys, huffllm_stream stream) {
    clear_error();
    DeviceInfo dev;
    huffllm_status st = device_info(&dev);
    if (st != HUFFLLM_OK) return st;
    if (!ws || !rows || !cols || !xs || !ys) return fail(HUFFLLM_ERR_INVALID_ARG, "null pointer");
    if (n == 0 || n > kMaxMats) return fail(HUFFLLM_ERR_INVALID_ARG, "between 1 and %u matrices per call", kMaxMats);
    PlainArgs a;
    memset(&a, 0, sizeof(a));
    a.n_mats = n;
    uint64_t total = 0;
    for (uint32_t i = 0; i < n; ++i) {
        if (!ws[i] || !xs[i] || !ys[i] || rows[i] == 0 || cols[i] == 0) return fail(HUFFLLM_ERR_INVALID_ARG, "null pointer or empty matrix");
        if (cols[i] % 8 || ((uintptr_t)ws[i] & 15) || ((uintptr_t)xs[i] & 15))
            return fail(HUFFLLM_ERR_UNSUPPORTED, "cols must be a multiple of 8 and pointers 16-byte aligned");
        a.m[i].w = ws[i];
        a.m[i].x = xs[i];
        a.m[i].y = ys[i];
        a.m[i].rows = rows[i];
        a.m[i].cols = cols[i];
        a.m[i].row_first = (uint32_t)total;
        total += rows[i];
        if (total >= (1ull << 31)) return fail(HUFFLLM_ERR_UNSUPPORTED, "too many rows for one launch");
    }
    a.total_rows = (uint32_t)total;
    cudaError_t e = launch_plain_gemv(a, (uint32_t)dev.sms, (cudaStream_t)stream);
    if (e != cudaSuccess) return fail(HUFFLLM_ERR_CUDA, "plain gemv launch: %s", cudaGetErrorString(e));
    return HUFFLLM_OK;
}

huffllm_status huffllm_plain_gemv(const uint16_t *w, uint64_t rows, uint64_t cols, const uint16_t *x, float *y, huffllm_stream stream) {
    return huffllm_plain_gemv_multi(1, &w, &rows, &cols, &x, &y, stream);
}

}  // extern "C"
