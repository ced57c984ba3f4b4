// simr_adjoint.cu -- pathwise adjoint (reverse-mode) Greeks of the Heston QE path, sm_103a.
//
// Per path (one lane): a forward pass of the variance recursion (Philox draws,
// QE variance step -- the paper's VariancePathQE, Sec. 4) that keeps the
// variance every `k` steps (a global [slot][resident thread] array), then a
// reverse sweep over the segments, last to first: each segment's states are
// recomputed from its checkpoint (the draws are counter-based, so the
// segment's draws are regenerated) and kept with the step's branch draw and Z_X
// -- in shared memory, or in a slab per warp in global memory (SegWarp) when the
// segment is longer than shared memory holds -- and the steps are
// differentiated backwards (LogPricePathQE's increments summed on the way),
// with the branch taken in the forward pass held fixed (pathwise derivative).
// With one segment of the whole path there is no forward pass at all: the
// recompute of that segment is the path's only simulation.  Since x' = x + (terms), the
// adjoint of x is 1 throughout; the sweep carries the adjoint of v and seven
// sums that the parameters enter through:
//   Am = sum mbar, Amv = sum mbar (v - theta), As = sum s2bar, Asv = sum s2bar v,
//   Ad = sum (theta - v), Adl = sum (v' - m), Ak3 = sum sqrt(v + v') Z_X,
// mapped once per path onto d x_T / d(v0, kappa, theta, sigma, rho) with
// FP64-derived constants.  Price sensitivities per strike (reduction over paths,
// Sec. 6): dP/dq = e^{-rT} mean[f'(S_T) S_T dx_T/dq], plus S_T/S0 for S0 and
// T - T P for r.  The terms are summed in FP32 over a warp's paths (one strike
// per lane for 32-strike tiles, a warp sum for one strike) and in FP64 on, as
// in the pricing kernel.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "simr_device.cuh"
#include "simr_internal.h"
#include "simr_reduce.cuh"
#include "simr_adjoint_path.cuh"

namespace simr {
namespace {

#ifndef SIMR_ADJ_PPT
#define SIMR_ADJ_PPT 1  // paths per thread of the per-strike adjoint kernel (2 measured slower)
#endif
// Dynamic shared memory of the per-strike kernel with segments in shared memory: strike
// constants, the last-block flag, then the segment buffers; the per-warp FP64 accumulator
// rows come first when they live in shared memory throughout (RACC false), or reuse the
// segment buffers' space once the path loop has ended (RACC true: lane l accumulates strike
// l of the one 32-strike tile in registers).
inline size_t adjoint_smem_bytes_t(const PathLaunch& L, const AdjConst& A, int tpb, int ppt, bool racc) {
  const size_t acc_bytes = (size_t)(tpb / kWarp) * kAdjAcc * L.nk_pad * sizeof(double);
  const size_t buf_bytes = adjoint_seg_floats(A, ppt) * tpb * sizeof(float);
  const size_t head = L.nk_pad * sizeof(StrikeConst) + 16;
  return racc ? head + (buf_bytes > acc_bytes ? buf_bytes : acc_bytes) : acc_bytes + head + buf_bytes;
}

// The per-strike terms of a 32-strike tile, lane l owning strike K (the
// tile's strike l): the warp's paths are broadcast one at a time -- terminal
// spot and d x_T / d(v0, kappa, theta, sigma, rho) -- and each lane adds its
// strike's payoff f, f^2, and the in-the-money weight w (S_T for a call above
// its strike, -S_T for a put below) alone and times each derivative; FP32 over
// the warp's paths.  out[0..8]: f, f^2, w, w dx/dv0 .. w dx/drho, the signed
// in-the-money indicator (the S0 column is w / S0, scaled with the totals; the r column e^{-rT} T K times the indicator's mean, see adj_term).
template <int PPT>
__device__ __forceinline__ void strike_tile_terms(bool put, float K, const float (&S)[PPT], const bool (&act)[PPT],
                                                  const float (&g)[PPT][5], float (&out)[kAdjAcc]) {
#pragma unroll
  for (int a = 0; a < kAdjAcc; ++a) out[a] = 0.0f;
#pragma unroll
  for (int j = 0; j < PPT; ++j) {
    const unsigned live = __ballot_sync(kFull, act[j]);
#pragma unroll 4
    for (int p = 0; p < kWarp; ++p) {
      const float Sp = __shfl_sync(kFull, S[j], p);
      float gp[5];
#pragma unroll
      for (int k = 0; k < 5; ++k) gp[k] = __shfl_sync(kFull, g[j][k], p);
      if ((live >> p) & 1u) {  // warp-uniform
        const float f = put ? fmaxf(K - Sp, 0.0f) : fmaxf(Sp - K, 0.0f);
        const float w = put ? (Sp < K ? -Sp : 0.0f) : (Sp > K ? Sp : 0.0f);
        out[0] += f;
        out[1] = fmaf(f, f, out[1]);
        out[2] += w;
#pragma unroll
        for (int k = 0; k < 5; ++k) out[3 + k] = fmaf(w, gp[k], out[3 + k]);
        out[8] += put ? (Sp < K ? -1.0f : 0.0f) : (Sp > K ? 1.0f : 0.0f);
      }
    }
  }
}

// Price, standard error and the seven derivatives per strike from the totals
// acc[9][nk_pad] (shared memory; s0_scale: what the S0 column's sums still lack).
__device__ __forceinline__ void write_adjoint(const PathLaunch& L, const AdjConst& A,
                                              const double* __restrict__ strikes, const double* acc, double s0_scale,
                                              const AdjOutputs& out) {
  const double inv_n = 1.0 / L.paths_total;
  const double nan = __longlong_as_double(0x7ff8000000000000ll);
  for (int kk = threadIdx.x; kk < L.n_strikes; kk += blockDim.x) {
    const double K = strikes[kk];
    const bool bad = !(K > 0.0) || !isfinite(K);
    const double mean = acc[kk] * inv_n;
    const double price = L.disc * mean;
    out.price[kk] = bad ? nan : price;
    if (out.stderr_) {
      const double n = L.paths_total;
      const double var = n > 1.0 ? (acc[L.nk_pad + kk] * inv_n - mean * mean) / (n - 1.0) : 0.0;
      out.stderr_[kk] = bad ? nan : L.disc * sqrt(var > 0.0 ? var : 0.0);
    }
    for (int c7 = 0; c7 < 7; ++c7) {
      double gsum = L.disc * acc[(size_t)(2 + c7) * L.nk_pad + kk] * inv_n;
      if (c7 == 0) gsum *= s0_scale;
      // e^{-rT} T K E[indicator] with the FP32 T and K the paths use (as the book does)
      if (c7 == 6) gsum *= (double)A.T * (double)(float)K;
      out.grad[(size_t)kk * 7 + c7] = bad ? nan : gsum;
    }
  }
}

// Minimum resident blocks per SM asked of the register allocator: 4 for strike tiles,
// whose segments (12 k bytes per thread) and rows leave room for no more from k = 16
// on (11% faster at k = 32 and 1% at k = 16 than with 5); one strike takes 5 where its
// segments leave room for them, k <= 28 (one_strike_blocks; 96 registers instead of 108:
// QE-M 9 steps x 2^22 paths 825 -> 748 us, 96 steps at k = 16 5.12 -> 4.82 ms), else 4
// (1% faster at k = 32 and 64).
#ifndef SIMR_ADJ_MINB_SMEM
#define SIMR_ADJ_MINB_SMEM 4
#endif

// Segments in shared memory (an explicit checkpoint interval).
// QEM: the QE-M log-spot step (the launch's scheme 1), differentiated one step
// at a time.
template <int TILE, int PPT, bool RACC, bool QEM, int MINB = SIMR_ADJ_MINB_SMEM>
__global__ void __launch_bounds__(128, MINB) heston_adjoint_kernel(const __grid_constant__ PathLaunch L,
                                                             const __grid_constant__ AdjConst A,
                                                             const double* __restrict__ strikes, AdjOutputs out,
                                                             double* __restrict__ partials,
                                                             unsigned int* __restrict__ ticket,
                                                             float* __restrict__ gckpt) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warps = blockDim.x / kWarp;
  const int bd = blockDim.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tid = threadIdx.x;
  const int row = kAdjAcc * L.nk_pad;
  const size_t acc_bytes = (size_t)warps * row * sizeof(double);
  const size_t ks_off = RACC ? 0 : acc_bytes;
  StrikeConst* ks = reinterpret_cast<StrikeConst*>(smem_raw + ks_off);
  int* s_last = reinterpret_cast<int*>(ks + L.nk_pad);
  float* sbuf = reinterpret_cast<float*>(s_last + 4);  // path_adjoint_ppt's segment buffers
  double* acc = RACC ? reinterpret_cast<double*>(sbuf) : reinterpret_cast<double*>(smem_raw);
  // checkpoints: this thread's column of a [slot][grid threads] global array
  float* ck = gckpt + (int)blockIdx.x * bd + tid;
  const int ck_stride = (int)(gridDim.x * blockDim.x);
  double racc[RACC ? kAdjAcc : 1];
#pragma unroll
  for (int a = 0; a < (RACC ? kAdjAcc : 1); ++a) racc[a] = 0.0;

  if (!RACC)
    for (int i = threadIdx.x; i < warps * row; i += blockDim.x) acc[i] = 0.0;
  for (int j = threadIdx.x; j < L.nk_pad; j += blockDim.x) {
    StrikeConst k{0.0f, 0.0f, 0.0f, 0.0f};
    if (j < L.n_strikes) {
      const double K = strikes[j];
      if (!(K > 0.0) || !isfinite(K)) atomicOr(out.status, 1);
      k.K = (float)K;
    }
    ks[j] = k;
  }
  __syncthreads();

  const bool put = L.is_put != 0;
  double* my_acc = acc + (size_t)warp * row;
  const uint64_t per_batch = (uint64_t)kWarp * PPT;
  const uint64_t batches = (L.path_count + per_batch - 1) / per_batch;
  const uint64_t total_warps = (uint64_t)gridDim.x * warps;
  for (uint64_t bt = (uint64_t)blockIdx.x * warps + warp; bt < batches; bt += total_warps) {
    uint64_t pth[PPT];
    bool act[PPT];
#pragma unroll
    for (int j = 0; j < PPT; ++j) {
      const uint64_t local = bt * per_batch + (uint64_t)j * kWarp + lane;
      act[j] = local < L.path_count;
      pth[j] = L.path_begin + local;
    }
    float x[PPT], comp[PPT], g[PPT][5], S[PPT];
    path_adjoint_ppt<PPT, SegShared, QEM>(L.sc[0], A, L.steps, L.option_index, L.rk, pth, ck, ck_stride,
                                                SegShared{sbuf}, x, comp, g, L.qm);
#pragma unroll
    for (int j = 0; j < PPT; ++j) S[j] = terminal_spot(L.S0, x[j], comp[j]);

    // per-strike terms, summed over the warp's paths
    if (RACC) {
      float t[kAdjAcc];
      strike_tile_terms<PPT>(put, ks[lane].K, S, act, g, t);
#pragma unroll
      for (int a = 0; a < kAdjAcc; ++a) racc[a] += (double)t[a];
    } else if (TILE == 1) {
      for (int a = 0; a < kAdjAcc; ++a) {
        float t = 0.0f;
#pragma unroll
        for (int j = 0; j < PPT; ++j) t += act[j] ? adj_term(a, put, S[j], ks[0].K, g[j], A.invS0, A.T) : 0.0f;
        t = warp_sum(t);
        if (lane == 0) my_acc[a] += (double)t;
      }
    } else {
      for (int t0 = 0; t0 < L.nk_pad; t0 += 32) {
        float t[kAdjAcc];
        strike_tile_terms<PPT>(put, ks[t0 + lane].K, S, act, g, t);
        double* row = my_acc + t0 + lane;
#pragma unroll
        for (int a = 0; a < kAdjAcc; ++a) row[(size_t)a * L.nk_pad] += (double)t[a];
      }
    }
  }
  __syncthreads();
  if (RACC) {  // the segment buffers are free now: spill the lanes' sums into the rows
#pragma unroll
    for (int a = 0; a < kAdjAcc; ++a) my_acc[(size_t)a * L.nk_pad + lane] = racc[a];
    __syncthreads();
  }

  for (int i = threadIdx.x; i < row; i += blockDim.x) {
    double s = acc[i];
    for (int w = 1; w < warps; ++w) s += acc[(size_t)w * row + i];
    acc[i] = s;
  }
  __syncthreads();
  if (!sum_block_rows(acc, row, partials, ticket, s_last)) return;
  write_adjoint(L, A, strikes, acc, TILE == 1 ? 1.0 : (double)A.invS0, out);  // (as below)
}

// Warps per SM of the kernel below (QE-M: its reverse step needs fewer registers).
#ifndef SIMR_ADJ_WARPS
#define SIMR_ADJ_WARPS 24
#endif
#ifndef SIMR_ADJ_QEM_WARPS
#define SIMR_ADJ_QEM_WARPS 28
#endif

// Segments in global memory, a slab per warp of 3 k floats a lane (a segment too long for shared
// memory, in particular one segment of the whole path: no forward pass).  One block
// per SM, its warps taking 32-path batches item by item (ItemPlan), each item's nine
// sums per strike in the item's own row.  Issue-bound (152 warp instructions per
// path-step, 33 of them packed).  252 steps x 2^20 paths x 32 strikes: 2,072 us with
// five blocks of 128 that strode over the batches (and one thread per sum over 760
// block rows at the end), 1,740 with items at 20 warps, 1,598 at 24 (80 registers;
// 28 and 32 warps spill: 2,040 and 2,080), 1,388 with the segments in warp slabs
// (SegWarp) and no selects on the common path; QE-M 948 -> 556 us at 2^18 paths.
template <int TILE, bool QEM>
__global__ void __launch_bounds__(kWarp * (QEM ? SIMR_ADJ_QEM_WARPS : SIMR_ADJ_WARPS), 1)
    heston_adjoint_seg_kernel(const __grid_constant__ PathLaunch L, const __grid_constant__ AdjConst A,
                              const __grid_constant__ ItemPlan I, const double* __restrict__ strikes, AdjOutputs out,
                              double* __restrict__ partials, unsigned int* __restrict__ ticket,
                              float* __restrict__ gckpt, float* __restrict__ gseg) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int bd = blockDim.x, lane = threadIdx.x & 31, tid = threadIdx.x;
  StrikeConst* ks = reinterpret_cast<StrikeConst*>(smem_raw);
  int* s_flag = reinterpret_cast<int*>(ks + L.nk_pad);
  unsigned* s_next = reinterpret_cast<unsigned*>(s_flag + 1);
  uint4* tab = L.pair_table ? reinterpret_cast<uint4*>(s_flag + 4) : nullptr;
  const ItemRows rows{smem_raw, (unsigned)(L.nk_pad * sizeof(StrikeConst) + 16 + L.pair_table * sizeof(uint4)), kAdjAcc * L.nk_pad};
  // checkpoints: this thread's column of a [slot][grid threads] global array
  float* ck = gckpt + (int)blockIdx.x * bd + tid;
  const int ck_stride = (int)(gridDim.x * blockDim.x);
  if (tid == 0) *s_next = 0u;
  for (int p = tid; p < L.pair_table; p += bd)
    tab[p] = philox_pair_entry(p, L.option_index, (uint32_t)(L.path_begin >> 32), L.rk);
  for (int j = tid; j < L.nk_pad; j += bd) {
    StrikeConst k{0.0f, 0.0f, 0.0f, 0.0f};
    if (j < L.n_strikes) {
      const double K = strikes[j];
      if (!(K > 0.0) || !isfinite(K)) atomicOr(out.status, 1);
      k.K = (float)K;
    }
    ks[j] = k;
  }
  __syncthreads();

  const bool put = L.is_put != 0;
  const uint64_t block0 = I.batches / gridDim.x * blockIdx.x + min((uint64_t)blockIdx.x, I.batches % gridDim.x);
  const uint64_t nb = I.batches / gridDim.x + (blockIdx.x < I.batches % gridDim.x ? 1 : 0);
  while (true) {
    unsigned it = 0;
    if (lane == 0) it = atomicAdd(s_next, 1u);
    it = __shfl_sync(kFull, it, 0);
    uint64_t b0, b1;
    if (!item_range(I, it, nb, b0, b1)) break;
    ItemRow<false> my = rows.at(I, it);
    for (uint64_t b = b0; b < b1; ++b) {
      const uint64_t local = (block0 + b) * kWarp + lane;
      const bool act[1] = {local < L.path_count};
      const uint64_t pth[1] = {L.path_begin + local};
      float x[1], comp[1], g[1][5];
      const SegWarp seg{gseg, A.ckpt_every};
      if (tab)
        path_adjoint_ppt<1, SegWarp, QEM, true>(L.sc[0], A, L.steps, L.option_index, L.rk, pth, ck, ck_stride,
                                                        seg, x, comp, g, L.qm, tab);
      else
        path_adjoint_ppt<1, SegWarp, QEM, false>(L.sc[0], A, L.steps, L.option_index, L.rk, pth, ck, ck_stride,
                                                         seg, x, comp, g, L.qm);
      const float S[1] = {terminal_spot(L.S0, x[0], comp[0])};
      if (TILE == 1) {
        for (int a = 0; a < kAdjAcc; ++a) {
          const float t = warp_sum(act[0] ? adj_term(a, put, S[0], ks[0].K, g[0], A.invS0, A.T) : 0.0f);
          if (lane == 0) my.add<false>(smem_raw, a, t);
        }
      } else {
        for (int t0 = 0; t0 < L.nk_pad; t0 += 32) {
          float t[kAdjAcc];
          strike_tile_terms<1>(put, ks[t0 + lane].K, S, act, g, t);
#pragma unroll
          for (int a = 0; a < kAdjAcc; ++a) my.add<false>(smem_raw, a * L.nk_pad + t0 + lane, t[a]);
        }
      }
      my.next_batch();
    }
  }
  __syncthreads();
  sum_item_rows(rows, I, nb);
  __syncthreads();
  if (!sum_block_rows(rows.acc(I), rows.row, partials, ticket, s_flag)) return;
  // (a tile's third sum holds the weights w: the S0 column is w / S0)
  write_adjoint(L, A, strikes, rows.acc(I), TILE == 1 ? 1.0 : (double)A.invS0, out);
}

// Per-path output: x_T and g = d x_T / d(v0, kappa, theta, sigma, rho).
template <bool QEM>
__global__ void __launch_bounds__(128) heston_paths_adjoint_kernel(const __grid_constant__ PathLaunch L,
                                                                   const __grid_constant__ AdjConst A,
                                                                   float* __restrict__ x_T, float* __restrict__ grad) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int bd = blockDim.x, tid = threadIdx.x;
  float* ckpt = reinterpret_cast<float*>(smem_raw);
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= L.path_count) return;  // no block-wide synchronisation below
  float x[1], comp[1], g[1][5];
  const uint64_t pth[1] = {L.path_begin + i};
  path_adjoint_ppt<1, SegShared, QEM>(L.sc[0], A, L.steps, L.option_index, L.rk, pth, ckpt + tid, bd,
                                            SegShared{ckpt + (A.n_seg - 1) * bd}, x, comp, g, L.qm);
  x_T[i] = x[0] - comp[0];
#pragma unroll
  for (int j = 0; j < 5; ++j) grad[i * 5 + j] = g[0][j];
}

// Blocks per SM that one strike's segments leave room for, 5 at most and 4 at least
// (an SM's shared memory less 1 KB per block).
int one_strike_blocks(const PathLaunch& L, const AdjConst& A) {
  return 5 * (adjoint_smem_bytes_t(L, A, 128, SIMR_ADJ_PPT, false) + 1024) <= 228 * 1024 ? 5 : 4;
}

template <int TILE, bool RACC, bool QEM, int MINB = SIMR_ADJ_MINB_SMEM>
cudaError_t launch_adjoint_t(const PathLaunch& L, const AdjConst& A, const double* strikes, const AdjOutputs& out,
                             const Scratch& s, int num_sms, cudaStream_t stream) {
  constexpr int PPT = SIMR_ADJ_PPT;
  const int tpb = 128, warps = tpb / kWarp;
  const size_t row = (size_t)kAdjAcc * L.nk_pad;
  const size_t smem = adjoint_smem_bytes_t(L, A, tpb, PPT, RACC);
  auto kern = heston_adjoint_kernel<TILE, PPT, RACC, QEM, MINB>;
  cudaError_t e = allow_dynamic_smem(kern);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, tpb, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const uint64_t batches = (L.path_count + (uint64_t)kWarp * PPT - 1) / ((uint64_t)kWarp * PPT);
  const uint64_t need = (batches + warps - 1) / warps;
  const uint64_t grid = std::min<uint64_t>((uint64_t)num_sms * per_sm, need);
  if ((size_t)(grid + kRowGroups) * row > s.partial_doubles) return cudaErrorMemoryAllocation;
  if ((size_t)grid * tpb * adjoint_ckpt_floats(A, PPT) > s.ckpt_floats) return cudaErrorMemoryAllocation;
  kern<<<(unsigned)grid, tpb, smem, stream>>>(L, A, strikes, out, s.partials, s.ticket, s.ckpt);
  return cudaGetLastError();
}

// The launch shape of the global-segment kernel: items, table, shared memory.
struct SegShape {
  ItemPlan I;
  uint64_t grid;
  int pair_table;
  size_t smem;
};
SegShape seg_shape(const PathLaunch& L, int num_sms, bool qem) {
  SegShape h;
  h.pair_table = pair_table_entries(L);
  const size_t row = (size_t)kAdjAcc * L.nk_pad;
  const size_t head = L.nk_pad * sizeof(StrikeConst) + 16 + h.pair_table * sizeof(uint4);
  const uint64_t batches = (L.path_count + kWarp - 1) / kWarp;
  h.grid = std::max<uint64_t>(1, std::min<uint64_t>(num_sms, batches));
  h.I = make_item_plan(batches, h.grid, qem ? SIMR_ADJ_QEM_WARPS : SIMR_ADJ_WARPS, row, kItemBytes - head);
  h.smem = head + item_rows_bytes(h.I, row);
  return h;
}

template <int TILE, bool QEM>
cudaError_t launch_adjoint_seg(const PathLaunch& L0, const AdjConst& A, const double* strikes, const AdjOutputs& out,
                               const Scratch& s, int num_sms, cudaStream_t stream) {
  const SegShape h = seg_shape(L0, num_sms, QEM);
  PathLaunch L = L0;
  L.pair_table = h.pair_table;
  const int tpb = kWarp * h.I.warps;
  const size_t row = (size_t)kAdjAcc * L.nk_pad;
  auto kern = heston_adjoint_seg_kernel<TILE, QEM>;
  cudaError_t e = allow_dynamic_smem(kern);
  if (e != cudaSuccess) return e;
  if ((size_t)(h.grid + kRowGroups) * row > s.partial_doubles) return cudaErrorMemoryAllocation;
  if ((size_t)h.grid * tpb * adjoint_ckpt_floats(A, 1) > s.ckpt_floats) return cudaErrorMemoryAllocation;
  if ((size_t)h.grid * tpb * adjoint_seg_floats(A, 1) > s.gseg_floats) return cudaErrorMemoryAllocation;
  kern<<<(unsigned)h.grid, tpb, h.smem, stream>>>(L, A, h.I, strikes, out, s.partials, s.ticket, s.ckpt, s.gseg);
  return cudaGetLastError();
}

// Whether the segment buffers go to global memory: when 3 k floats per thread
// do not fit the shared memory of a block.  (Shared-memory segments are kept
// even where they cost resident blocks: at k = 32, 4 blocks per SM with
// shared-memory segments ran 11% faster than 5 with L2-resident global ones.)
bool adjoint_gseg(const PathLaunch& L, const AdjConst& A) {
  return adjoint_smem_bytes_t(L, A, 128, SIMR_ADJ_PPT, L.nk_pad == 32) > kAdjMaxSmem;
}

template <bool QEM>
cudaError_t launch_adjoint_s(const PathLaunch& L, const AdjConst& A, const double* strikes, const AdjOutputs& out,
                             const Scratch& s, int num_sms, cudaStream_t stream) {
  if (adjoint_gseg(L, A)) {
    return L.nk_pad == 1 ? launch_adjoint_seg<1, QEM>(L, A, strikes, out, s, num_sms, stream)
                         : launch_adjoint_seg<32, QEM>(L, A, strikes, out, s, num_sms, stream);
  }
  if (L.nk_pad == 1)
    return one_strike_blocks(L, A) == 5 ? launch_adjoint_t<1, false, QEM, 5>(L, A, strikes, out, s, num_sms, stream)
                                        : launch_adjoint_t<1, false, QEM>(L, A, strikes, out, s, num_sms, stream);
  if (L.nk_pad == 32) return launch_adjoint_t<32, true, QEM>(L, A, strikes, out, s, num_sms, stream);
  return launch_adjoint_t<32, false, QEM>(L, A, strikes, out, s, num_sms, stream);
}

}  // namespace

size_t adjoint_scratch_doubles(const PathLaunch& L, int num_sms) {
  // at most 16 resident blocks of 128 threads per SM
  return ((size_t)num_sms * 16 + kRowGroups) * kAdjAcc * (size_t)L.nk_pad;
}

cudaError_t adjoint_max_ckpt_every(const PathLaunch& L, int steps_cap, int* k_max) {
  // the kernel variant launch_adjoint picks for this strike count
  const bool racc = L.nk_pad == 32;
  const void* kern = L.nk_pad == 1 ? (const void*)heston_adjoint_kernel<1, SIMR_ADJ_PPT, false, false>
                     : racc      ? (const void*)heston_adjoint_kernel<32, SIMR_ADJ_PPT, true, false>
                                 : (const void*)heston_adjoint_kernel<32, SIMR_ADJ_PPT, false, false>;
  auto blocks = [&](int k, int* n) -> cudaError_t {
    AdjConst A{};
    A.ckpt_every = k;
    const size_t smem = adjoint_smem_bytes_t(L, A, 128, SIMR_ADJ_PPT, racc);
    *n = 0;
    if (smem > kAdjMaxSmem) return cudaSuccess;
    cudaError_t e = allow_dynamic_smem(kern);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, kern, 128, smem);
  };
  int best = 0;
  cudaError_t e = blocks(2, &best);
  if (e != cudaSuccess) return e;
  if (best < 1) return cudaErrorInvalidConfiguration;
  // blocks per SM fall as k grows: the largest even k that keeps `best`
  int lo = 1, hi = (steps_cap + 1) / 2 + 1;  // k = 2 lo keeps it; k = 2 hi is past the cap
  while (hi - lo > 1) {
    const int mid = (lo + hi) / 2;
    int n = 0;
    if ((e = blocks(2 * mid, &n)) != cudaSuccess) return e;
    (n >= best ? lo : hi) = mid;
  }
  *k_max = 2 * lo;
  return cudaSuccess;
}

cudaError_t adjoint_gseg_floats(const PathLaunch& L, const AdjConst& A, int num_sms, size_t* floats) {
  *floats = 0;
  if (!adjoint_gseg(L, A)) return cudaSuccess;
  const SegShape h = seg_shape(L, num_sms, L.scheme == 1);
  *floats = (size_t)h.grid * kWarp * h.I.warps * adjoint_seg_floats(A, 1);
  return cudaSuccess;
}

size_t adjoint_ckpt_scratch_floats(const AdjConst& A, int num_sms) {
  // at most 16 resident blocks of 128 threads per SM
  return (size_t)num_sms * 16 * 128 * adjoint_ckpt_floats(A, SIMR_ADJ_PPT);
}

cudaError_t launch_paths_adjoint(const PathLaunch& L, const AdjConst& A, float* x_T, float* grad, cudaStream_t stream) {
  const int tpb = 128;
  const size_t smem = (size_t)adjoint_thread_floats(A.n_seg, A.ckpt_every, 1) * tpb * sizeof(float);
  auto kern = L.scheme == 1 ? heston_paths_adjoint_kernel<true> : heston_paths_adjoint_kernel<false>;
  cudaError_t e = allow_dynamic_smem(kern);
  if (e != cudaSuccess) return e;
  const uint64_t grid = (L.path_count + tpb - 1) / tpb;
  kern<<<(unsigned)grid, tpb, smem, stream>>>(L, A, x_T, grad);
  return cudaGetLastError();
}

cudaError_t launch_adjoint(const PathLaunch& L, const AdjConst& A, const double* strikes, const AdjOutputs& out,
                           const Scratch& s, int num_sms, cudaStream_t stream) {
  if (L.scheme == 1) return launch_adjoint_s<true>(L, A, strikes, out, s, num_sms, stream);
  return launch_adjoint_s<false>(L, A, strikes, out, s, num_sms, stream);
}

}  // namespace simr
