// Bit-field split explorer (Section 3.1, entropy table): how many bits per parameter would each way of cutting a
// 16-bit weight into separately coded fields cost?  The device part counts, for every field of a split, how often
// each of its values occurs in a weight tensor that already sits in device memory; the host part turns counts into
// entropies and Huffman code costs.
//
// Counting is one streaming pass over the weights (2 bytes per weight from HBM).  Every CTA keeps private counters in
// shared memory and adds them to the global 64-bit counters at the end.  What bounds it is the shared-memory atomic unit,
// one counter update per weight and counted piece, so neighbouring narrow fields of a large tensor are counted together, as one
// piece of up to ten bits, and told apart when the CTA adds its counters up.  LLM weights are very skewed (a handful of exponent values
// cover almost all weights), so a piece's counters are replicated 32 times, one copy per lane: the lanes of a warp never
// touch the same address or the same bank, whatever the data.  Wider fields get fewer copies; a field whose counters do
// not fit is counted in several launches, each owning a range of values.
// Where the word is cut into two pieces a CTA of 1024 threads has an SM to itself: its counters are cleared, added up and sent to L2 once
// per SM, its threads have registers for eight loads in flight.  An update takes the atomic unit two cycles, 20 of the 22 us that splits of two pieces take at 45 M weights.
// (Kernel alone, two CTAs an SM, four loads at a time, shifts as kernel arguments / this, us: 45 M weights 1-8-7 25.6 / 22.2, 1-5-5-5 26.8 / 26.0;
// 16.8 M 13.9 / 10.7; 235 M 95 / 83, 0.87 of a copy's rate.  At first, every field counted on its own, 40 and 49 us.)
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "internal.h"

namespace huffllm {

constexpr uint32_t kHistThreads = 1024;
constexpr uint32_t kHistBudgetWords = 48u * 1024u;   // shared-memory counters of one launch (192 KB)
constexpr uint32_t kFieldWords = 8u * 1024u;         // target size of a wide field's counters, copies included
constexpr uint32_t kPieceBits = 10;                  // most bits of a piece of several fields: 1024 counters, 32 copies, 128 KB
// From this many counter updates on (weights times fields) fields are counted together.  Below, clearing and adding up the larger
// tables costs a CTA more than its weights do.  (Apart / together, us: 1-5-5-5 at 10^6 weights 10.0 / 14.4, at 4 10^6 14.3 / 16.3, at
// 45 10^6 53 / 36; 1-8-7 10.2 / 12.2, 14.2 / 15.7, 45 / 33; sixteen fields of one bit 17.5 / 23.5, 33 / 25.6, 169 / 45.)
constexpr uint64_t kMergeFrom = 1ull << 25;

struct PiecePlan {
    uint32_t shift, mask;        // value of the piece = (word >> shift) & mask
    uint32_t bin_lo, bin_n;      // values counted by this launch: bin_lo .. bin_lo + bin_n - 1
    uint32_t smem_off;           // first counter, in 32-bit words
    uint32_t rep_log2;           // log2 of the copies per value
    uint32_t ranged;             // 1 if the launch covers only a part of the piece's values
    uint32_t field_first, n_fields;
};
struct FieldPlan {
    uint32_t shift, width;       // inside its piece
    uint32_t out_off;            // index of the field's value 0 in the output counters
};
struct HistArgs {
    const uint16_t *w;
    uint64_t n;
    unsigned long long *counts;
    uint32_t n_pieces, smem_words;
    PiecePlan p[HUFFLLM_MAX_FIELDS];
    FieldPlan f[HUFFLLM_MAX_FIELDS];
};

__device__ __forceinline__ void red_shared_inc(uint32_t addr) {
    asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(addr) : "memory");
}
template <int OFF>
__device__ __forceinline__ void red_shared_inc(uint32_t addr) {
    asm volatile("red.shared.add.u32 [%0+%1], 1;" ::"r"(addr), "n"(OFF) : "memory");
}

// LOW: the word is cut into two unranged pieces whose counters are 32-fold, LOW bits and the 16 - LOW above (the splits of the two
// formats); 0: any pieces
template <int LOW>
__global__ void __launch_bounds__(kHistThreads, LOW ? 1 : 2) split_histogram_kernel(const __grid_constant__ HistArgs A) {
    extern __shared__ __align__(16) uint32_t hist[];
    const uint32_t tid = threadIdx.x, lane = tid & 31;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(hist);

    // 16-byte vectors of eight weights; the last n % 8 weights go to one thread
    const uint64_t n_vec = A.n / 8;
    const uint4 *const src = (const uint4 *)A.w;
    auto clear = [&]() {
        for (uint32_t i = tid; i < A.smem_words / 4; i += kHistThreads) ((uint4 *)hist)[i] = make_uint4(0, 0, 0, 0);
        for (uint32_t i = (A.smem_words & ~3u) + tid; i < A.smem_words; i += kHistThreads) hist[i] = 0;
        __syncthreads();
    };
    // n_words words of two weights each (one with `single`): a piece at a time, its plan read once for all of them
    auto count_words = [&](const uint32_t *word, auto n_words, bool single) {
#pragma unroll 1
        for (uint32_t pi = 0; pi < A.n_pieces; ++pi) {
            const PiecePlan &p = A.p[pi];
            const uint32_t lane_off = base + ((p.smem_off + (lane & ((1u << p.rep_log2) - 1u))) << 2);
            const uint32_t step = 4u << p.rep_log2, sh = p.shift, mask = p.mask, lo = p.bin_lo, nb = p.bin_n;
            if (!p.ranged) {
#pragma unroll
                for (int i = 0; i < decltype(n_words)::value; ++i) {
                    red_shared_inc(lane_off + ((word[i] >> sh) & mask) * step);
                    if (!single) red_shared_inc(lane_off + ((word[i] >> (sh + 16)) & mask) * step);
                }
            } else {
#pragma unroll
                for (int i = 0; i < decltype(n_words)::value; ++i) {
                    const uint32_t b0 = ((word[i] >> sh) & mask) - lo, b1 = ((word[i] >> (sh + 16)) & mask) - lo;
                    if (b0 < nb) red_shared_inc(lane_off + b0 * step);
                    if (!single && b1 < nb) red_shared_inc(lane_off + b1 * step);
                }
            }
        }
    };
    const uint32_t lane_base = base + (lane << 2);
    auto count = [&](const uint4 &q) {
        const uint32_t word[4] = {q.x, q.y, q.z, q.w};
        if constexpr (LOW == 0) {
            count_words(word, std::integral_constant<int, 4>{}, false);
        } else {
            // A counter's 32 copies are 128 bytes: a halfword dot product takes the value of either weight times 128 to the lane's
            // column.  (All shifts and masks are constants, so a weight's two updates cost three and a half instructions besides.)
            constexpr uint32_t kLow = ((1u << LOW) - 1u) * 0x10001u, kHigh = ((1u << (16 - LOW)) - 1u) * 0x10001u;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t h = word[i] >> LOW & kHigh, l = word[i] & kLow;
                red_shared_inc<0>(__dp2a_lo(h, 0x0080u, lane_base));
                red_shared_inc<0>(__dp2a_lo(h, 0x8000u, lane_base));
                red_shared_inc<128 << (16 - LOW)>(__dp2a_lo(l, 0x0080u, lane_base));
                red_shared_inc<128 << (16 - LOW)>(__dp2a_lo(l, 0x8000u, lane_base));
            }
        }
    };
    if constexpr (LOW == 0) {                                // dealt to the grid's threads in turn
        clear();
        const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
        for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + tid; v < n_vec; v += stride) count(__ldg(src + v));
    } else {
        // A CTA takes a contiguous piece.  Eight loads are in flight per thread throughout, the first ones while the counters are cleared: a
        // vector's registers are loaded anew as soon as it has been counted.
        constexpr int kAhead = 8;
        const uint64_t first = n_vec * blockIdx.x / gridDim.x;
        int32_t left = (int32_t)(n_vec * (blockIdx.x + 1) / gridDim.x - first) - (int32_t)tid;    // (fewer than 2^35 / 148 vectors a CTA)
        const uint4 *at = src + first + tid;
        uint4 q[kAhead];
#pragma unroll
        for (int i = 0; i < kAhead; ++i)
            if (left > i * (int)kHistThreads) q[i] = __ldg(at + i * kHistThreads);
        clear();
#pragma unroll 1
        for (; left > 0; left -= kAhead * (int)kHistThreads) {
            at += kAhead * kHistThreads;
#pragma unroll
            for (int i = 0; i < kAhead; ++i) {
                if (left > i * (int)kHistThreads) count(q[i]);
                if (left > (kAhead + i) * (int)kHistThreads) q[i] = __ldg(at + i * kHistThreads);
            }
        }
    }
    if (blockIdx.x == 0 && tid == 0)
        for (uint64_t i = n_vec * 8; i < A.n; ++i) {
            const uint32_t word = A.w[i];
            count_words(&word, std::integral_constant<int, 1>{}, true);
        }
    __syncthreads();

    // add the CTA's counters to the global ones, copies of a value summed first, zero sums skipped: a piece of one field at
    // once; of several, the copies are summed into the first one (which no other thread reads), then a thread or a warp per
    // field value sums the piece's values that have it
    bool several = false;
    for (uint32_t pi = 0; pi < A.n_pieces; ++pi) {
        const PiecePlan &p = A.p[pi];
        const uint32_t reps = 1u << p.rep_log2;
        several = several || p.n_fields > 1;
        for (uint32_t b = tid; b < p.bin_n; b += blockDim.x) {
            uint32_t s = 0;
            for (uint32_t r = 0; r < reps; ++r) s += hist[p.smem_off + (b << p.rep_log2) + ((r + tid) & (reps - 1u))];
            if (p.n_fields > 1) hist[p.smem_off + (b << p.rep_log2)] = s;
            else if (s) atomicAdd(A.counts + A.f[p.field_first].out_off + p.bin_lo + b, (unsigned long long)s);
        }
    }
    if (!several) return;
    __syncthreads();
    for (uint32_t pi = 0; pi < A.n_pieces; ++pi) {
        const PiecePlan &p = A.p[pi];
        if (p.n_fields == 1) continue;
        for (uint32_t fi = p.field_first; fi < p.field_first + p.n_fields; ++fi) {
            const FieldPlan &f = A.f[fi];
            const uint32_t others = p.bin_n >> f.width;        // piece values with a given field value
            auto at = [&](uint32_t val, uint32_t i) -> uint32_t {
                const uint32_t b = ((i >> f.shift) << (f.shift + f.width)) | (val << f.shift) | (i & ((1u << f.shift) - 1u));
                return hist[p.smem_off + (b << p.rep_log2)];
            };
            if (others <= 8u) {                                // few: a thread per field value
                for (uint32_t val = tid; val < 1u << f.width; val += kHistThreads) {
                    uint32_t s = 0;
                    for (uint32_t i = 0; i < others; ++i) s += at(val, i);
                    if (s) atomicAdd(A.counts + f.out_off + val, (unsigned long long)s);
                }
                continue;
            }
            for (uint32_t val = tid >> 5; val < 1u << f.width; val += kHistThreads / 32) {
                uint32_t s = 0;
                for (uint32_t i = lane; i < others; i += 32) s += at(val, i);
#pragma unroll
                for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
                if (lane == 0 && s) atomicAdd(A.counts + f.out_off + val, (unsigned long long)s);
            }
        }
    }
}

// The kernel of a word cut into two pieces above its `low` lower bits (pieces have ten bits at most).
static void (*two_pieces(uint32_t low))(HistArgs) {
    switch (low) {
        case 6: return split_histogram_kernel<6>;
        case 7: return split_histogram_kernel<7>;
        case 8: return split_histogram_kernel<8>;
        case 9: return split_histogram_kernel<9>;
        case 10: return split_histogram_kernel<10>;
        default: return split_histogram_kernel<0>;
    }
}

static huffllm_status check_widths(const uint8_t *widths, uint32_t n_fields, size_t *total_bins) {
    if (!widths || n_fields == 0 || n_fields > HUFFLLM_MAX_FIELDS) return fail(HUFFLLM_ERR_INVALID_ARG, "a split has 1..%d fields", HUFFLLM_MAX_FIELDS);
    uint32_t sum = 0;
    size_t bins = 0;
    for (uint32_t i = 0; i < n_fields; ++i) {
        if (widths[i] < 1 || widths[i] > 16) return fail(HUFFLLM_ERR_INVALID_ARG, "field %u has width %u", i, (unsigned)widths[i]);
        sum += widths[i];
        bins += (size_t)1 << widths[i];
    }
    if (sum != 16) return fail(HUFFLLM_ERR_INVALID_ARG, "the field widths add up to %u, not 16", sum);
    if (total_bins) *total_bins = bins;
    return HUFFLLM_OK;
}

}  // namespace huffllm

using namespace huffllm;

extern "C" huffllm_status huffllm_split_counts_size(const uint8_t *widths, uint32_t n_fields, size_t *n_counts) {
    clear_error();
    if (!n_counts) return fail(HUFFLLM_ERR_INVALID_ARG, "null output");
    return check_widths(widths, n_fields, n_counts);
}

extern "C" huffllm_status huffllm_split_histogram(const uint16_t *w_dev, uint64_t n_weights, const uint8_t *widths,
                                                  uint32_t n_fields, uint64_t *counts_dev, huffllm_stream stream) {
    clear_error();
    size_t bins = 0;
    huffllm_status st = check_widths(widths, n_fields, &bins);
    if (st != HUFFLLM_OK) return st;
    if (!w_dev || !counts_dev) return fail(HUFFLLM_ERR_INVALID_ARG, "null device pointer");
    if (((uintptr_t)w_dev & 15u) || ((uintptr_t)counts_dev & 7u)) return fail(HUFFLLM_ERR_INVALID_ARG, "weights must be 16-byte aligned, counters 8-byte aligned");
    if (n_weights >> 38) return fail(HUFFLLM_ERR_UNSUPPORTED, "more than 2^38 weights in one call");   // a CTA's 32-bit counters cannot overflow below that
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e;
    int dev = 0, sms = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess || (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
        return fail(HUFFLLM_ERR_CUDA, "device query: %s", cudaGetErrorString(e));

    // the pieces to count: neighbouring fields of up to kPieceBits bits together (large tensors), a wider field, or a range of a wide
    // field's values, each with its counters' size.  (A split has 16 bits, so two pieces are the least there can be, and no
    // split of fields of up to ten bits needs more than three.)
    std::vector<PiecePlan> pieces;
    FieldPlan fields[HUFFLLM_MAX_FIELDS] = {};
    uint32_t hi = 16, out_off = 0;
    const bool merge = n_weights * n_fields >= kMergeFrom;
    for (uint32_t i = 0; i < n_fields;) {
        uint32_t bits = widths[i], last = i + 1;
        while (merge && last < n_fields && bits + widths[last] <= kPieceBits) bits += widths[last++];
        const uint32_t n_bins = 1u << bits;
        PiecePlan p = {};
        p.shift = hi - bits;
        p.mask = n_bins - 1u;
        p.field_first = i;
        p.n_fields = last - i;
        for (uint32_t rel = bits; i < last; ++i) {
            rel -= widths[i];
            fields[i].shift = rel;
            fields[i].width = widths[i];
            fields[i].out_off = out_off;
            out_off += 1u << widths[i];
        }
        const uint32_t target = merge && bits <= kPieceBits ? n_bins << 5 : kFieldWords;
        while (p.rep_log2 < 5u && (n_bins << (p.rep_log2 + 1u)) <= target) ++p.rep_log2;
        const uint32_t per_piece = std::min(n_bins, kHistBudgetWords / 2u >= n_bins ? n_bins : 32u * 1024u);
        for (uint32_t lo = 0; lo < n_bins; lo += per_piece) {
            p.bin_lo = lo;
            p.bin_n = per_piece;
            p.ranged = per_piece < n_bins ? 1u : 0u;
            pieces.push_back(p);
        }
        hi -= bits;
    }
    // launches: pieces in order, as many as fit the shared-memory budget.  All of them are planned before the first call that the GPU
    // sees: planned behind the clearing of the counters, the counting waited for the host.
    struct Launch {
        void (*kernel)(HistArgs);
        HistArgs args;
    };
    std::vector<Launch> launches;
    size_t p = 0;
    while (n_weights && p < pieces.size()) {
        launches.push_back({});
        HistArgs &A = launches.back().args;
        A.w = w_dev;
        A.n = n_weights;
        A.counts = (unsigned long long *)counts_dev;
        memcpy(A.f, fields, sizeof(fields));
        uint32_t words = 0;
        bool plain = true;
        while (p < pieces.size() && A.n_pieces < HUFFLLM_MAX_FIELDS) {
            PiecePlan f = pieces[p];
            const uint32_t need = f.bin_n << f.rep_log2;
            if (A.n_pieces && words + need > kHistBudgetWords) break;
            f.smem_off = words;
            words += need;
            plain = plain && !f.ranged && f.rep_log2 == 5u;
            A.p[A.n_pieces++] = f;
            ++p;
        }
        A.smem_words = words;
        launches.back().kernel = plain && A.n_pieces == 2 ? two_pieces(A.p[0].shift) : split_histogram_kernel<0>;
        if ((e = cudaFuncSetAttribute(launches.back().kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kHistBudgetWords * 4u))) != cudaSuccess)
            return fail(HUFFLLM_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
    }
    if ((e = cudaMemsetAsync(counts_dev, 0, bins * sizeof(uint64_t), s)) != cudaSuccess) return fail(HUFFLLM_ERR_CUDA, "cudaMemsetAsync: %s", cudaGetErrorString(e));
    for (const Launch &l : launches) {
        const size_t smem = (size_t)l.args.smem_words * 4u;
        const uint32_t per_sm = l.kernel == split_histogram_kernel<0> && smem <= 100u * 1024u ? 2u : 1u;
        const uint32_t grid = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>((uint64_t)sms * per_sm, (n_weights / 8 + kHistThreads - 1) / kHistThreads));
        l.kernel<<<grid, kHistThreads, smem, s>>>(l.args);
        if ((e = cudaGetLastError()) != cudaSuccess) return fail(HUFFLLM_ERR_CUDA, "split_histogram_kernel: %s", cudaGetErrorString(e));
    }
    return HUFFLLM_OK;
}

extern "C" huffllm_status huffllm_split_entropy(const uint64_t *counts_host, const uint8_t *widths, uint32_t n_fields,
                                                double *entropy_bits, double *huffman_bits) {
    clear_error();
    huffllm_status st = check_widths(widths, n_fields, nullptr);
    if (st != HUFFLLM_OK) return st;
    if (!counts_host || !entropy_bits) return fail(HUFFLLM_ERR_INVALID_ARG, "null pointer");
    const uint64_t *c = counts_host;
    for (uint32_t i = 0; i < n_fields; ++i) {
        const size_t n_bins = (size_t)1 << widths[i];
        long double total = 0;
        for (size_t b = 0; b < n_bins; ++b) total += (long double)c[b];
        double H = 0;
        if (total > 0)
            for (size_t b = 0; b < n_bins; ++b)
                if (c[b]) {
                    const double pr = (double)((long double)c[b] / total);
                    H -= pr * std::log2(pr);
                }
        entropy_bits[i] = H;
        if (huffman_bits) {
            // cost of a Huffman code = sum of the weights of the internal nodes of its tree (two-queue merge of the
            // sorted counts); a field with a single value in use is given the 1-bit code the blob format gives it
            std::vector<uint64_t> leaf;
            for (size_t b = 0; b < n_bins; ++b)
                if (c[b]) leaf.push_back(c[b]);
            std::sort(leaf.begin(), leaf.end());
            double bits = 0;
            if (leaf.size() == 1) {
                bits = 1.0;
            } else if (leaf.size() > 1) {
                std::vector<uint64_t> node;
                node.reserve(leaf.size());
                size_t li = 0, ni = 0;
                long double cost = 0;
                auto take = [&]() -> uint64_t {
                    if (li < leaf.size() && (ni >= node.size() || leaf[li] <= node[ni])) return leaf[li++];
                    return node[ni++];
                };
                for (size_t m = 0; m + 1 < leaf.size(); ++m) {
                    const uint64_t a = take(), b2 = take();
                    node.push_back(a + b2);
                    cost += (long double)(a + b2);
                }
                bits = (double)(cost / total);
            }
            huffman_bits[i] = bits;
        }
        c += n_bins;
    }
    return HUFFLLM_OK;
}
