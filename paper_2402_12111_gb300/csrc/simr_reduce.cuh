// simr_reduce.cuh -- warp-level reduction helpers of the path kernels (reduction over
// paths, paper Sec. 6): FP32 sums of 32 paths, FP64 from there on.
#pragma once

#include <cstdint>

#include "simr_internal.h"

namespace simr {
namespace {

constexpr int kWarp = 32;
constexpr unsigned kFull = 0xffffffffu;

// In-place transposed butterfly: on entry vals[j] is this lane's term for strike
// j of the tile; on exit vals[0] of lane l is the sum over the 32 lanes for strike l.
__device__ __forceinline__ void butterfly32(float (&vals)[32], int lane) {
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    const bool upper = (lane & o) != 0;
#pragma unroll
    for (int j = 0; j < o; ++j) {
      const float send = upper ? vals[j] : vals[j + o];
      const float keep = upper ? vals[j + o] : vals[j];
      vals[j] = keep + __shfl_xor_sync(kFull, send, o);
    }
  }
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// An item's row: the sums of its batches, added in FP64 in batch order -- or, for
// an item of one batch, that batch's FP32 sums as they are.  It lives through the whole
// path loop, as an offset and a word or as pointers and a flag: which of the two leaves a
// kernel the better schedule is measured (path_row_pointers).
// ONE_COPY: the row's kind hidden from the compiler, which else makes a copy of the loops
// over the sums for each kind.  In a long run the warps drift out of step, and with two
// copies the path kernels of strike tiles (5 scenarios: 210 KB of code, 172 with one) then
// missed the instruction cache: 30 steps x 2.5 M paths x 32 strikes, 5 scenarios 1.60 ->
// 1.26 ms; pricing at 8 steps x 8.4 M paths x 64 strikes 0.60 -> 0.55.
template <bool POINTERS>
struct ItemRow {
  unsigned at;  // byte offset of the row in dynamic shared memory
  int kind;     // 0: FP32; 1: FP64, the item's first batch, which sets the row; 2: FP64
  template <bool ONE_COPY>
  __device__ __forceinline__ void add(unsigned char* smem, int i, float t) const {
    int k = kind;
    if (ONE_COPY) asm volatile("" : "+r"(k));
    if (k == 0) {
      reinterpret_cast<float*>(smem + at)[i] = t;
    } else {
      double* p = reinterpret_cast<double*>(smem + at) + i;
      *p = k == 1 ? (double)t : *p + (double)t;
    }
  }
  __device__ __forceinline__ void next_batch() {
    if (kind == 1) kind = 2;
  }
};
template <>
struct ItemRow<true> {
  double* wide;   // null for an FP32 row
  float* narrow;
  bool first;     // the item's first batch sets the row
  template <bool ONE_COPY>
  __device__ __forceinline__ void add(unsigned char*, int i, float t) const {
    int w = wide != nullptr;
    if (ONE_COPY) asm volatile("" : "+r"(w));
    if (!w)
      narrow[i] = t;
    else
      wide[i] = first ? (double)t : wide[i] + (double)t;
  }
  __device__ __forceinline__ void next_batch() { first = false; }
};

// The shared memory of a block's items, from byte offset `base`: FP64 rows
// [rows64][row], the block's totals, FP32 rows [rows32][row].
struct ItemRows {
  unsigned char* smem;
  unsigned base;
  int row;
  __device__ __forceinline__ unsigned acc_at(const ItemPlan& I) const { return base + (unsigned)(I.rows64 * row) * 8u; }
  __device__ __forceinline__ unsigned narrow_at(const ItemPlan& I) const {
    return acc_at(I) + (unsigned)max(row, (int)blockDim.x) * 8u;
  }
  __device__ __forceinline__ const double* wide() const { return reinterpret_cast<const double*>(smem + base); }
  __device__ __forceinline__ const float* narrow(const ItemPlan& I) const {
    return reinterpret_cast<const float*>(smem + narrow_at(I));
  }
  __device__ __forceinline__ double* acc(const ItemPlan& I) const { return reinterpret_cast<double*>(smem + acc_at(I)); }
  template <bool POINTERS = false>
  __device__ __forceinline__ ItemRow<POINTERS> at(const ItemPlan& I, uint32_t it) const {
    const uint32_t n64 = I.tail_size == 1 ? (uint32_t)(I.levels * I.warps) : 0xffffffffu;
    if constexpr (POINTERS)
      return it < n64 ? ItemRow<true>{reinterpret_cast<double*>(smem + base) + (size_t)it * row, nullptr, true}
                      : ItemRow<true>{nullptr, reinterpret_cast<float*>(smem + narrow_at(I)) + (size_t)(it - n64) * row, true};
    else
      return it < n64 ? ItemRow<false>{base + it * row * 8u, 1} : ItemRow<false>{narrow_at(I) + (it - n64) * row * 4u, 0};
  }
};

// The rows of a block that owns nb batches, summed into R.acc(I) in item order: with
// fewer columns than threads, groups of threads sum runs of rows side by side
// first.  All threads; rows complete on entry (after a barrier).
__device__ __forceinline__ void sum_item_rows(const ItemRows& R, const ItemPlan& I, uint64_t nb) {
  const int level_items = I.levels * I.warps, row = R.row;
  const int n = level_items + (int)((nb - I.tail_begin + I.tail_size - 1) / I.tail_size);
  const int n64 = I.tail_size == 1 ? level_items : n;
  const int groups = max(1, min((int)blockDim.x / row, n));
  const int per = (n + groups - 1) / groups;
  const double* wide = R.wide();
  const float* narrow = R.narrow(I);
  double* acc = R.acc(I);
  for (int i = threadIdx.x; i < row * groups; i += blockDim.x) {
    const int g = i / row, col = i - g * row;
    const int r1 = min((g + 1) * per, n);
    double s = 0.0;
    int r = g * per;
    for (; r < min(r1, n64); ++r) s += wide[(size_t)r * row + col];
    for (; r < r1; ++r) s += (double)narrow[(size_t)(r - n64) * row + col];
    acc[i] = s;
  }
  if (groups == 1) return;
  __syncthreads();
  for (int i = threadIdx.x; i < row; i += blockDim.x) {
    double s = acc[i];
    for (int g = 1; g < groups; ++g) s += acc[g * row + i];
    acc[i] = s;
  }
}

__device__ __forceinline__ double sum_rows_in_order(const double* __restrict__ p, int n, size_t row) {
  double s = 0.0;
  int b = 0;
  for (; b + 8 <= n; b += 8) {  // eight loads in flight
    double v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = __ldcg(p + (size_t)(b + k) * row);
#pragma unroll
    for (int k = 0; k < 8; ++k) s += v[k];
  }
  for (; b < n; ++b) s += __ldcg(p + (size_t)b * row);
  return s;
}

// The sum over blocks of their rows acc[0 .. row) (shared memory), in block order
// and on two levels: the last block of a group to arrive sums the group's rows,
// the last group's block the groups'.  True in every thread of the block that
// ends with the totals in acc; the tickets are zero again then.  One level over
// 608 rows took 45 us of the pricing call at 2^20 paths (one thread per column,
// each load's latency on the path), this takes about 4.
__device__ __forceinline__ bool sum_block_rows(double* acc, int row, double* __restrict__ partials,
                                               unsigned int* __restrict__ ticket, int* s_flag) {
  const int grid = gridDim.x;
  int per = 1;
  while (per * per < grid) ++per;
  per = max(per, (grid + kRowGroups - 1) / kRowGroups);  // blocks per group
  const int groups = (grid + per - 1) / per, g = blockIdx.x / per;
  const int g0 = g * per, gn = min(per, grid - g0);
  double* my_row = partials + (size_t)blockIdx.x * row;
  for (int i = threadIdx.x; i < row; i += blockDim.x) my_row[i] = acc[i];
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) *s_flag = atomicAdd(ticket + 1 + g, 1u) == (unsigned)gn - 1u;
  __syncthreads();
  if (!*s_flag) return false;
  __threadfence();
  double* g_row = partials + (size_t)(grid + g) * row;
  for (int i = threadIdx.x; i < row; i += blockDim.x)
    g_row[i] = sum_rows_in_order(partials + (size_t)g0 * row + i, gn, row);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    ticket[1 + g] = 0u;
    *s_flag = atomicAdd(ticket, 1u) == (unsigned)groups - 1u;
  }
  __syncthreads();
  if (!*s_flag) return false;
  __threadfence();
  for (int i = threadIdx.x; i < row; i += blockDim.x)
    acc[i] = sum_rows_in_order(partials + (size_t)grid * row + i, groups, row);
  if (threadIdx.x == 0) *ticket = 0u;
  __syncthreads();
  return true;
}

struct StrikeConst {
  float K, Km, Wr, pad;  // strike; K e^{-h_r T}; K e^{h_r T} - K e^{-h_r T}
};

}  // namespace
}  // namespace simr
