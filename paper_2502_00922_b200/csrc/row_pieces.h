// Which weights of a row the 16-byte pieces of a decode's output hold where rows start anywhere (kernels.cu, store_piece).
// Arithmetic only, so that the host can go through column counts no test could decode.
#pragma once
#include <cstdint>

#include "host_device.h"

namespace huffllm {

// Columns are counted from the first one of the block in hand (32 columns), those in front of it are negative: a row has up to 2^31
// columns, and no sum of these leaves 32 bits.

// Columns from `at` to the row's end, or as many as no chunk has.
HUFFLLM_HD int32_t columns_left(uint32_t cols, uint32_t at) { return (int32_t)(cols - at < (1u << 20) ? cols - at : 1u << 20); }
// The run's first column: that of its first block, or, behind it, one in front of all that the row buffers hold.
HUFFLLM_HD int32_t run_start(bool opens) { return opens ? 0 : -32; }
// First column of quad lane t's piece, in a row that starts `off` weights behind a sector's start.
HUFFLLM_HD int32_t piece_column(uint32_t t, uint32_t off) { return (int32_t)(t * 8u) - (int32_t)off; }

// A row 8 further down starts 8 * cols weights further on: with an odd column count half a sector off, and its pieces, which are to
// lie on sectors too, start so many columns further on than those of the row that starts `off` weights behind a sector's start.
HUFFLLM_HD int32_t row_half(uint32_t off, uint32_t cols) { return cols & 1u ? (off & 8u ? 8 : -8) : 0; }

// The weights lo .. hi - 1 of the piece in column c that lie in columns [first, end); none if lo >= hi.
struct PieceCut {
    int32_t lo, hi;
};
HUFFLLM_HD PieceCut piece_cut(int32_t c, int32_t first, int32_t end) { return {first > c ? first - c : 0, end - c < 8 ? end - c : 8}; }

}  // namespace huffllm
