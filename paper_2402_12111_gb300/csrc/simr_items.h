// simr_items.h -- the items of a path kernel's block: how its batches are handed to its
// warps.  Plain C++ (no CUDA headers), the kernels' and the host's one copy.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>

#ifdef __CUDACC__
#define SIMR_HD __host__ __device__ __forceinline__
#else
#define SIMR_HD inline
#endif

namespace simr {

// How the blocks of a path kernel hand their batches (a warp's paths of one pass)
// to their warps.  Block b owns a contiguous run of the launch's batches, cut into
// items by this plan alone: `levels` levels of one item per warp, each level three
// fifths of what is left, then items of tail_size batches.  A warp takes the next
// item from a counter in shared memory and leaves the item's sums in the item's
// own row (FP64; FP32 for an item of one batch, whose sums are FP32), so the
// totals do not depend on which warp took what.
constexpr int kItemLevels = 12;
struct ItemPlan {
  uint64_t batches;               // of the whole launch
  uint64_t size[kItemLevels];     // batches per item of a level
  uint64_t begin[kItemLevels];    // the level's first batch within the block
  uint64_t tail_begin, tail_size;
  int32_t levels, warps;          // items per level = warps per block
  int32_t rows64, rows32;         // most FP64 and FP32 rows a block uses
};
// Shared memory of a plan's rows and of the block's totals behind them.
inline size_t item_rows_bytes(const ItemPlan& I, size_t row) {
  const size_t wide = row > 32u * I.warps ? row : 32u * I.warps;  // sum_item_rows' columns side by side
  return (I.rows64 + 0ull) * row * 8 + wide * 8 + (I.rows32 * row + 1) / 2 * 8;
}
// Dynamic shared memory a path kernel's block may take for them.
constexpr size_t kItemBytes = 208 * 1024;

// The batches [b0, b1) of item `it` of a block that owns nb batches; false past the last.
SIMR_HD bool item_range(const ItemPlan& I, uint32_t it, uint64_t nb, uint64_t& b0, uint64_t& b1) {
  const uint32_t lvl = it / (uint32_t)I.warps;
  if (lvl < (uint32_t)I.levels) {
    b0 = I.begin[lvl] + (uint64_t)(it - lvl * I.warps) * I.size[lvl];
    b1 = b0 + I.size[lvl];
  } else {
    b0 = I.tail_begin + (uint64_t)(it - (uint32_t)(I.levels * I.warps)) * I.tail_size;
    b1 = b0 + I.tail_size;
  }
  if (b1 > nb) b1 = nb;
  return b0 < nb;
}

// The plan of `batches` on a grid of blocks of at most max_warps warps, with rows
// of `row` sums in `bytes` of shared memory (at least one FP64 row).
inline ItemPlan make_item_plan(uint64_t batches, uint64_t grid, int max_warps, size_t row, size_t bytes) {
  ItemPlan I{};
  I.batches = batches;
  const uint64_t q = batches / grid, most = (batches + grid - 1) / grid;  // batches of a block
  const uint64_t fits = (bytes - row * 8) / (row * 8);                    // FP64 rows beside the totals
  uint64_t w = std::max<uint64_t>(1, std::min<uint64_t>({(uint64_t)max_warps, fits, most}));
  // few batches a warp: as many warps as make the rounds even (31 batches on 24
  // warps: two rounds of 16, not 24 and 7: 250 steps, pricing 294 -> 270 us, 5
  // scenarios 444 -> 392; 25 batches 261 -> 253, 48 (already even) the same; at 30
  // steps within the noise of either)
  const uint64_t rounds = (most + w - 1) / w;
  if (rounds == 2) w = (most + rounds - 1) / rounds;
  while (w > 1 && (w * row + std::max<size_t>(row, 32 * w)) * 8 + 8 > bytes) --w;  // a row for every warp
  I.warps = (int)w;
  bytes -= std::max<size_t>(row, 32 * w) * 8 + 8;
  // the fewest levels after which the rest, batch by batch in FP32 rows, fits; if
  // none does, levels as long as the rows leave three wider FP64 items a warp
  uint64_t rem = q;
  while ((uint64_t)I.levels * w * row * 8 + (rem + 1) * row * 4 > bytes && I.levels < kItemLevels &&
         rem * 3 >= 5 * w && (uint64_t)(I.levels + 4) * w * row * 8 <= bytes) {
    const uint64_t size = rem * 3 / (5 * w);
    I.size[I.levels] = size;
    I.begin[I.levels] = q - rem;
    ++I.levels;
    rem -= size * w;
  }
  const uint64_t left = rem + (most - q), used = (uint64_t)I.levels * w;
  I.tail_begin = q - rem;
  I.tail_size = 1;
  I.rows64 = (int32_t)used;
  I.rows32 = (int32_t)left;
  if ((used * 8 + left * 4) * row > bytes) {
    // wider items, in FP64 rows: as many as the rows leave room for or whole rounds of
    // one item a warp, whichever lets the warps end first (the more items of those within
    // a sixteenth).  Cut by the rows alone they can leave a last round for a few warps: 5
    // scenarios x 128 strikes at 100 steps x 2^19 paths had 27 items of 4 batches on 24
    // warps, 1,211 us against 977.
    const uint64_t room = bytes / (row * 8) - used, all = room / w;
    const auto size = [&](uint64_t r) {  // r rounds; past the last: as many items as rows
      const uint64_t n = r > all ? room : std::min(room, std::max<uint64_t>(1, r) * w);
      return std::max<uint64_t>(2, (left + n - 1) / n);
    };
    const auto end = [&](uint64_t r) {  // batches of the warp with most of them
      const uint64_t full = left / size(r), part = left % size(r);
      return full % w ? (full / w + 1) * size(r) : full / w * size(r) + part;
    };
    uint64_t r = all + 1, best = end(r);
    for (uint64_t k = 1; k <= all; ++k) best = std::min(best, end(k));
    while (end(r) * 16 > best * 17) --r;
    I.tail_size = size(r);
    I.rows64 = (int32_t)(used + (left + I.tail_size - 1) / I.tail_size);
    I.rows32 = 0;
  }
  return I;
}

}  // namespace simr
