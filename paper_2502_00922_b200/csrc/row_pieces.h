// Which weights of a row the 16-byte pieces of a decode's output hold where rows start anywhere (kernels.cu, store_piece).
// Arithmetic only, so that the host can go through column counts no test could decode.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define HUFFLLM_HD __host__ __device__ __forceinline__
#else
#define HUFFLLM_HD inline
#endif

namespace huffllm {

// Columns are counted from the first column of the chunk in hand, in front of which they are negative: a row has up to 2^31 of
// them, a chunk at most 1024, and no sum of theirs leaves 32 bits.

// Columns from `at` to the row's end, or as many as no chunk has.
HUFFLLM_HD int32_t columns_left(uint64_t cols, uint32_t at) { return (int32_t)(cols - at < (1u << 20) ? cols - at : 1u << 20); }
// The run's first column: the chunk's own, or, where the row buffers still hold columns of the chunk in front, which has at least a
// block, one in front of all that is left of it.
HUFFLLM_HD int32_t run_start(bool left_over) { return left_over ? -32 : 0; }
// First column of quad lane t's piece of block kb, in a row that starts `off` weights behind a sector's start ...
HUFFLLM_HD int32_t piece_column(uint32_t kb, uint32_t t, uint32_t off) { return (int32_t)(kb * 32u + t * 8u) - (int32_t)off; }
// ... and of the piece behind a run that ends in column `end` (lanes with 8 t < off have one).
HUFFLLM_HD int32_t last_piece_column(int32_t end, uint32_t t, uint32_t off) { return ((end + 31) & ~31) + (int32_t)(t * 8u) - (int32_t)off; }

// The weights lo .. hi - 1 of the piece in column c that lie in columns [first, end); none if lo >= hi.
struct PieceCut {
    int32_t lo, hi;
};
HUFFLLM_HD PieceCut piece_cut(int32_t c, int32_t first, int32_t end) { return {first > c ? first - c : 0, end - c < 8 ? end - c : 8}; }

}  // namespace huffllm
