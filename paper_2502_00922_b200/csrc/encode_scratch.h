// The device encoder's scratch: 256 bytes for the totals, then a word per chunk for its coded bits and one for the words per sequence.
// Arithmetic only, so that the host can go through chunk counts of every remainder.
#pragma once
#include <cstddef>
#include <cstdint>

#include "host_device.h"

namespace huffllm {

constexpr uint32_t kScanThreads = 1024;      // chunks of a scan CTA, and of a group
constexpr uint64_t kScratchTotals = 256;     // bytes in front of the chunks' bits

HUFFLLM_HD uint64_t scratch_bytes(uint64_t n_chunks) { return kScratchTotals + 8 * n_chunks; }
HUFFLLM_HD uint32_t *scratch_bits(void *scratch) { return (uint32_t *)((uint8_t *)scratch + kScratchTotals); }
HUFFLLM_HD uint32_t *scratch_words(void *scratch, uint64_t n_chunks) { return scratch_bits(scratch) + n_chunks; }

// What 1024 chunks add up to, kept where their bits were.  Only whole groups have such sums: the chunks behind the last one, fewer than
// 1024 and possibly too few for their bits to make room for it (the words follow without a gap), are the last scan CTA's own.
struct EncGroup {
    unsigned long long words, bits;
    uint32_t most;
};
static_assert(sizeof(EncGroup) <= 4 * kScanThreads, "a group's sums lie where its bits were");
HUFFLLM_HD uint32_t group_count(uint64_t n_chunks) { return (uint32_t)(n_chunks / kScanThreads); }
HUFFLLM_HD EncGroup *group_at(uint32_t *bits, uint32_t g) { return (EncGroup *)(bits + (size_t)g * kScanThreads); }

}  // namespace huffllm
