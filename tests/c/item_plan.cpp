// The item plan's two functions behind a plain C interface, for tests/test_items.py.
#include "simr_items.h"

extern "C" {

void plan(uint64_t batches, uint64_t grid, int max_warps, uint64_t row, uint64_t bytes, simr::ItemPlan* out,
          uint64_t* facts) {
  *out = simr::make_item_plan(batches, grid, max_warps, row, bytes);
  facts[0] = (uint64_t)out->warps;
  facts[1] = simr::item_rows_bytes(*out, row);
  facts[2] = (uint64_t)out->rows64 + out->rows32;
  facts[3] = (uint64_t)out->levels;
}

// The batches of items 0, 1, ... of a block of nb, one end after another into ends;
// their number, or -1 where they leave a gap or overlap, or pass max.
int64_t items(const simr::ItemPlan* I, uint64_t nb, uint64_t* ends, int64_t max) {
  uint64_t b0, b1, at = 0;
  int64_t n = 0;
  while (simr::item_range(*I, (uint32_t)n, nb, b0, b1)) {
    if (b0 != at || b1 <= b0 || n >= max) return -1;
    at = ends[n++] = b1;
  }
  return at == nb ? n : -1;
}

uint64_t plan_size(void) { return sizeof(simr::ItemPlan); }
}
