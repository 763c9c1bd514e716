// Launch shape of batched queries (mips.cu): host arithmetic only, so that it can
// be checked without a GPU.
#pragma once

#include <stddef.h>
#include <stdint.h>

namespace mad {

constexpr int kDrawThreads = 256;
constexpr int kDrawMultMax = 8;              // most 256-diamond pieces of a chunk
constexpr uint32_t kMaxParts = 2048;         // (a part too full for its table splits itself)
constexpr int64_t kItemDimMax = 1024;        // longest item vectors

// Shared memory of a draw block: a chunk's records (8 bytes), their parts and
// ranks (4) and the source of each place (2); the parts' counts; the query's T2
// and TA rows and the total and bucket factor of TB's rows.
constexpr size_t draw_smem_bytes(int chunk, uint32_t parts, int64_t d) {
  return (size_t)chunk * (8 + 4 + 2) + ((size_t)parts + 1 + 4 * (size_t)d) * 4;
}

// More than the 48 KB a kernel may ask for by default (from d = 766 on at 2048
// parts, from 1,016 parts on at d = 1024), so the draw kernels opt in to this.
constexpr size_t kDrawSmemMax =
    draw_smem_bytes(kDrawThreads * kDrawMultMax, kMaxParts, kItemDimMax);
static_assert(kDrawSmemMax <= 226 * 1024, "the largest draw block fits an SM (1 KB for static words)");

}  // namespace mad
