// simr_paths.cu -- fused Heston QE path kernels for sm_103a: pricing, bump-and-revalue
// Greeks with common random numbers, terminal states.
//
// Per path (one lane) and per time step, entirely in registers:
//   Philox4x32-10 (one call per two steps) -> two 23-bit uniforms per step ->
//   inverse normals -> QE variance step (paper Sec. 4, VariancePathQE) ->
//   log-spot step (Sec. 5, LogPricePathQE), for every simulated scenario, all
//   sharing the same draws (common random numbers).
// Per path at maturity: S_T = S0 e^{x_T} (AssetPathExponential) and the payoff
// terms of each strike.  Reduction over paths (Sec. 6): a transposed warp
// butterfly in FP32 sums 32 paths per strike in 31 shuffle-add steps for 32
// strikes at once; an item's sums go to the item's row in shared memory, the
// block's rows are summed in FP64 in item order, and the blocks' totals on two
// levels of atomic tickets, in block order, then normalised.  No path data
// touches HBM.
//
// What bounds the kernels: the issue of their arithmetic.  A packed FMA holds both
// FP32 pipes for two cycles and a Philox product the heavy one for four; with
// every warp busy an SM sub-partition spends 115 cycles on 32 path-steps of
// pricing, 88 of them on the heavy pipe.  So what counts besides the arithmetic
// itself is that all warps stay busy to the end: with a fixed share of the paths per
// warp the scheduler lets some warps run ahead, 4.5 of 6 warps were busy on
// average, and one thread per sum then added 608 rows.  Items taken from a
// counter and the two-level sums: pricing 252 steps x 2^20 paths x 32 strikes
// 885 -> 780 us, the 5-scenario Greeks 2,510 -> 2,270 us, one strike's delta,
// gamma and vega at 64 x 65,536 52.7 -> 43.5 us (warm calls back to back).  Rows too
// long for several a warp (from 128 strikes x 7 sums on, and sooner for long runs)
// leave each warp one or two long items, a fixed share in all but name.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "simr_device.cuh"
#include "simr_internal.h"
#include "simr_reduce.cuh"

// Tuning knobs (compile-time): warps per SM.  Measured at 252 steps x 2^20 paths:
// pricing 770 / 785 / 786 us at 24 / 28 / 32 warps (pipelined loops); 5 scenarios
// 2,138 / 2,170 us at 24 / 28; 11 scenarios (365 x 250,001) 1,707 / 1,728 / 1,918 us at
// 16 / 20 / 24; 3 scenarios (one strike, 64 x 65,536) 39 us at 20 and 24.  QE-M pricing x 32
// strikes at 24 / 28 / 32: 252 x 2^20 940 / 926 / 942 us on the base model and 1,595 / 1,539 /
// 1,541 at a Feller ratio of 0.04, there 252 x 2^22 5,887 / 5,774 / 5,670 and 101 x 300,007 (31
// batches a block) 265 / 265 / 233.
#ifndef SIMR_PRICE_WARPS
#define SIMR_PRICE_WARPS 24
#endif
#ifndef SIMR_QEM_WARPS
#define SIMR_QEM_WARPS 32
#endif
#ifndef SIMR_FD3_WARPS
#define SIMR_FD3_WARPS 20
#endif
#ifndef SIMR_FD11_WARPS
#define SIMR_FD11_WARPS 16
#endif
#ifndef SIMR_FD5_WARPS
#define SIMR_FD5_WARPS 24
#endif
// paths per thread of the pricing (one scenario) and bump-and-revalue kernels
#ifndef SIMR_PRICE_PPT
#define SIMR_PRICE_PPT 2
#endif
#ifndef SIMR_FD_PPT
#define SIMR_FD_PPT 1
#endif

namespace simr {
namespace {

// Per-path term of accumulator `a` for one strike (call or put), given the
// terminal spots of all scenarios.  a = 0: payoff f; 1: f^2; then per Greek bit.
template <int NS>
__device__ __forceinline__ float acc_term(const PathLaunch& L, int greek_bit, int a,
                                          const StrikeConst& k, const float (&S)[NS]) {
  const float s = S[0];
  const bool put = L.is_put != 0;
  const float f = put ? fmaxf(k.K - s, 0.0f) : fmaxf(s - k.K, 0.0f);
  if (a == 0) return f;
  if (a == 1) return f * f;
  const float h = L.h_s;
  switch (greek_bit) {
    case 0: {  // delta: f(S(1+h)) - f(S(1-h)) = min(max(S(1+h)-K, 0), 2hS) for a call
      const float w = 2.0f * h * s;
      return put ? -fminf(fmaxf(fmaf(h, s, k.K - s), 0.0f), w) : fminf(fmaxf(fmaf(h, s, s - k.K), 0.0f), w);
    }
    case 1:  // gamma: f(S(1+h)) - 2 f(S) + f(S(1-h)) = max(0, hS - |K - S|)
      return fmaxf(fmaf(h, s, -fabsf(k.K - s)), 0.0f);
    case 4:  // rho: e^{-hT} f(S e^{hT}) - e^{hT} f(S e^{-hT}) = f(S; K e^{-hT}) - f(S; K e^{hT})
      return put ? -fminf(fmaxf(k.Km + k.Wr - s, 0.0f), k.Wr) : fminf(fmaxf(s - k.Km, 0.0f), k.Wr);
    default:
      break;
  }
  return 0.0f;
}

// ratio_up f_up - ratio_dn f_dn with ratio = 1 + delta (delta exact in FP32).
template <int NS>
__device__ __forceinline__ float resim_term(const PathLaunch& L, int up, int dn, const StrikeConst& k,
                                            const float (&S)[NS]) {
  float su = 0.0f, sd = 0.0f;
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    if (s == up) su = S[s];
    if (s == dn) sd = S[s];
  }
  const bool put = L.is_put != 0;
  const float fu = put ? fmaxf(k.K - su, 0.0f) : fmaxf(su - k.K, 0.0f);
  const float fd = put ? fmaxf(k.K - sd, 0.0f) : fmaxf(sd - k.K, 0.0f);
  const float ru = up ? L.sc[up].ratio : 0.0f, rd = dn ? L.sc[dn].ratio : 0.0f;
  return fmaf(ru, fu, fmaf(-rd, fd, fu - fd));
}

// The moments of the scenario pair (2P + 1, 2P + 2): the base's constants for the
// v0 bumps (P < NV / 2), plus the pair's own deltas for the others.
template <int NV>
__device__ __forceinline__ void pair_moments(const PathLaunch& L, int P, float2 v, float2& m, float2& s2h) {
  const ScenConst& b = L.sc[0];
  if (2 * P + 2 <= NV) {
    m = p_add(p_mul(v, p_bc(b.E)), p_bc(b.thE));
    s2h = p_add(p_mul(v, p_bc(b.h1)), p_bc(b.h2));
  } else {
    const ScenConst2& d = L.pair2[P];
    m = p_add(p_fma(v, p_bc(b.E), p_fma(v, d.E, d.thE)), p_bc(b.thE));
    s2h = p_add(p_fma(v, p_bc(b.h1), p_fma(v, d.h1, d.h2)), p_bc(b.h2));
  }
}

// One QE step of the base and its scenario pairs, lane for lane step_base<true> and
// step_bumped: every chain's quadratic branch side by side, then one test for the
// exponential branch, whose lanes are redone chain by chain.  (A test per chain kept
// them apart: 252 steps x 2^20 paths x 32 strikes, 5 scenarios 2,230 -> 2,157 us; 11
// scenarios at 365 x 250,001 x 21 1,806 -> 1,707.)
// d: the step's draws; with NEXT, on return the next step's, from its words,
// computed beside the variance chains behind the same test.
struct StepDraw {
  float xv, zv, zx;  // 2 U_V - 1, Z_V, Z_X
};
template <int NS, int NV, bool NEXT>
__device__ __forceinline__ void step_merged(const PathLaunch& L, StepDraw& d, uint32_t next_v, uint32_t next_x,
                                            float (&v)[NS], float (&x)[NS], float (&c)[NS]) {
  const float xv = d.xv, zv = d.zv, zx = d.zx;
  constexpr int NP = (NS - 1) / 2;
  const ScenConst& b = L.sc[0];
  const float m0 = __fadd_rn(__fmul_rn(v[0], b.E), b.thE);
  const float s0 = __fadd_rn(__fmul_rn(v[0], b.h1), b.h2);
  const float m20 = __fmul_rn(m0, m0), t0 = qe_t(m20, s0);
  float vn0, dl0;
  qe_quad_branch(m0, t0, zv, vn0, dl0);
  bool quad = t0 > kQuadT;
  float2 vn[NP], dl[NP];
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    float2 m, s2h, m2, t;
    pair_moments<NV>(L, p, make_float2(v[2 * p + 1], v[2 * p + 2]), m, s2h);
    quad &= qe_try2(m, s2h, p_bc(zv), m2, t, vn[p], dl[p]);
  }
  float2 xu, wc, z;
  bool central = true;
  if constexpr (NEXT) {
    xu = centered_uniform2(next_v, next_x);
    central = norminv_try2(xu, wc, z);
  }
  if (!(quad && central)) {
    if constexpr (NEXT) norminv_fix2(xu, wc, z);
    if (!(t0 > kQuadT)) qe_exp_branch(m0, s0, m20, xv, vn0, dl0);
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      float2 m, s2h;
      pair_moments<NV>(L, p, make_float2(v[2 * p + 1], v[2 * p + 2]), m, s2h);
      const float2 m2 = p_mul(m, m);
      qe_fix2(m, s2h, m2, p_mul(m2, p_rcp(s2h)), p_bc(xv), vn[p], dl[p]);
    }
  }
  {
    const float s = __fadd_rn(v[0], vn0);
    float inc = __fmaf_rn(b.Cv, s, b.C0);
    inc = __fmaf_rn(-b.Cd, v[0], inc);
    inc = __fmaf_rn(b.Cdl, dl0, inc);
    inc = __fmaf_rn(__fmul_rn(b.sK3, sqrt_approx(s)), zx, inc);
    const float y = __fsub_rn(inc, c[0]);
    const float t = __fadd_rn(x[0], y);
    c[0] = __fsub_rn(__fsub_rn(t, x[0]), y);
    x[0] = t;
    v[0] = vn0;
  }
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    const float2 vv = make_float2(v[2 * p + 1], v[2 * p + 2]), xx = make_float2(x[2 * p + 1], x[2 * p + 2]),
                 cc = make_float2(c[2 * p + 1], c[2 * p + 2]);
    const float2 s = p_add(vv, vn[p]);
    const float2 q = p_sqrt(s);
    float2 inc = p_fma(p_bc(b.Cv), s, p_bc(b.C0));
    inc = p_fma(p_bc(-b.Cd), vv, inc);
    inc = p_fma(p_bc(b.Cdl), dl[p], inc);
    inc = p_fma(p_mul(p_bc(b.sK3), q), p_bc(zx), inc);
    if (2 * p + 2 > NV) {
      const ScenConst2& d = L.pair2[p];
      float2 sm = p_fma(d.Cv, s, d.C0);
      sm = p_fma(d.mCd, vv, sm);
      sm = p_fma(d.Cdl, dl[p], sm);
      sm = p_fma(p_mul(d.sK3, q), p_bc(zx), sm);
      inc = p_add(inc, sm);
    }
    const float2 y = p_sub(inc, cc);
    const float2 t = p_add(xx, y);
    const float2 cn = p_sub(p_sub(t, xx), y);
    c[2 * p + 1] = cn.x;
    c[2 * p + 2] = cn.y;
    x[2 * p + 1] = t.x;
    x[2 * p + 2] = t.y;
    v[2 * p + 1] = vn[p].x;
    v[2 * p + 2] = vn[p].y;
  }
  if constexpr (NEXT) d = StepDraw{xu.x, z.x, z.y};
}

// One time step for all NS scenarios from the two words (w_v, w_x) of the step.
// NS scenarios in registers; DYN: only the first L.n_scen of them are live.
// Scenarios 1 .. NV differ from the base only in v0 (all constant deltas zero):
// they take the base step, which is the bumped step's arithmetic with zero deltas.
// The two inverse normals run paired, and so do the scenarios after the base,
// two at a time (s, s + 1): the paired functions repeat the scalar ones lane for
// lane, so every scenario's value is the scalar step's, bit for bit.  Constants
// equal in both lanes are broadcast from the scalar ones; a bumped pair's deltas,
// which differ by lane, come pre-packed from the launch parameters (measured:
// 3.4% faster than pre-packing the broadcast constants too, 6% faster than
// packing the deltas in the kernel).
template <int NS, int NV, bool DYN, bool QEM = false>
__device__ __forceinline__ void step_all(const PathLaunch& L, uint32_t w_v, uint32_t w_x, float (&v)[NS],
                                         float (&x)[NS], float (&c)[NS]) {
  const float2 xu = centered_uniform2(w_v, w_x);  // (2 U_V - 1, 2 U_X - 1)
  const float2 z = norminv_centered2(xu);
  const float xv = xu.x, zv = z.x, zx = z.y;
  static_assert(NS % 2 == 1, "the base scenario plus up/down pairs");
  if constexpr (QEM && NS > 1) {  // QE-M with bumped scenarios: the base, then the pairs (DYN: one at a time)
    const ScenConst zero{};
    const QemConst zq{};
    step_qem_bumped(L.sc[0], zero, L.qm, zq, xv, zv, zx, v[0], x[0], c[0]);
#pragma unroll
    for (int s = 1; s < NS; ++s) {
      if constexpr (DYN) {
        if (s >= L.n_scen) break;
        step_qem_bumped(L.sc[0], L.sc[s], L.qm, L.qmd[s], xv, zv, zx, v[s], x[s], c[s]);
      } else if (s % 2 == 1) {
        float2 vv = make_float2(v[s], v[s + 1]), xx = make_float2(x[s], x[s + 1]),
               cc = make_float2(c[s], c[s + 1]);
        step_qem_bumped2(pack_const(L.sc[0], L.sc[0]), L.pair2[(s - 1) / 2], L.qm, L.qmd2[(s - 1) / 2], p_bc(xv),
                         p_bc(zv), p_bc(zx), vv, xx, cc);
        v[s] = vv.x;
        v[s + 1] = vv.y;
        x[s] = xx.x;
        x[s + 1] = xx.y;
        c[s] = cc.x;
        c[s + 1] = cc.y;
      }
    }
    return;
  }
  if constexpr (NS > 1 && !QEM && !DYN) {
    StepDraw d{xv, zv, zx};
    step_merged<NS, NV, false>(L, d, 0u, 0u, v, x, c);
    return;
  }
  step_scheme<(NS > 1), QEM>(L.sc[0], L.qm, xv, zv, zx, v[0], x[0], c[0]);
#pragma unroll
  for (int s = 1; s + 1 < NS; s += 2) {
    if (DYN && s >= L.n_scen) break;
    float2 vv = make_float2(v[s], v[s + 1]), xx = make_float2(x[s], x[s + 1]), cc = make_float2(c[s], c[s + 1]);
    if (s + 1 <= NV)
      step_base2<true>(L.sc[0], p_bc(xv), p_bc(zv), p_bc(zx), vv, xx, cc);
    else
      step_bumped2(pack_const(L.sc[0], L.sc[0]), L.pair2[(s - 1) / 2], p_bc(xv), p_bc(zv), p_bc(zx), vv, xx, cc);
    v[s] = vv.x;
    v[s + 1] = vv.y;
    x[s] = xx.x;
    x[s + 1] = xx.y;
    c[s] = cc.x;
    c[s + 1] = cc.y;
  }
}

// One time step of PPT paths, path by path.
template <int NS, int NV, bool DYN, int PPT, bool QEM>
__device__ __forceinline__ void step_paths(const PathLaunch& L, const uint32_t (&wv)[PPT], const uint32_t (&wx)[PPT],
                                           float (&v)[PPT][NS], float (&x)[PPT][NS], float (&c)[PPT][NS]) {
#pragma unroll
  for (int j = 0; j < PPT; ++j) step_all<NS, NV, DYN, QEM>(L, wv[j], wx[j], v[j], x[j], c[j]);
}

// Step 0 of every scenario of a common-random-number launch (see step0_crn).
// Under QE-M the first-step constant K0p is r dt - qa (v0 + m0) - lam(v0) (set
// on the host in FP64, where M exists at every scenario's v0), v' has no term of
// its own and dl the coefficient K2.
template <int NS, bool DYN, bool QEM = false>
__device__ __forceinline__ void step0_apply(const PathLaunch& L, float xv, float zv, float zx, float (&v)[NS],
                                            float (&x)[NS], float (&c)[NS]) {
  const float omu = one_minus_u(xv);
  const ScenConst zero{};
  FirstConst fz = L.f0[0];
  fz.a = fz.b = fz.C = fz.L = fz.m0 = fz.K0p = 0.0f;  // base: zero deltas, its own threshold
  ScenConst b0 = L.sc[0];
  if (QEM) {
    b0.Cv = 0.0f;
    b0.Cdl = L.qm.K2;
  }
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    if (DYN && s >= L.n_scen) break;
    ScenConst d0 = s == 0 ? zero : L.sc[s];
    if (QEM) {
      d0.Cv = 0.0f;
      d0.Cdl = s == 0 ? 0.0f : L.qmd[s].K2;
    }
    step0_crn(L.f0[0], s == 0 ? fz : L.f0[s], b0, d0, L.sc[s].v0, omu, zv, zx, v[s], x[s], c[s]);
  }
}

template <int NS, bool DYN, bool QEM = false>
__device__ __forceinline__ void step0_all(const PathLaunch& L, uint32_t w_v, uint32_t w_x, float (&v)[NS],
                                          float (&x)[NS], float (&c)[NS]) {
  const float xv = centered_uniform(w_v);
  step0_apply<NS, DYN, QEM>(L, xv, norminv_centered(xv), norminv_centered(centered_uniform(w_x)), v, x, c);
}

// One path of a 3- or 5-scenario launch under QE, software-pipelined: while a step's
// chains run, the next step's normals and the next pair's Philox rounds are
// computed (one strike, 64 x 65,536, 3 scenarios 41.0 -> 39.0 us; 5 scenarios at 100 x
// 20,000 73.9 -> 67.7, at 252 x 2^20 2,157 -> 2,138; with 11 scenarios, whose chains
// fill the issue by themselves, it was 7% slower).
template <bool TAB, int NS, int NV>
__device__ __forceinline__ void simulate_fd(const PathLaunch& L, const uint4* tab, uint64_t path, float (&v)[NS],
                                            float (&x)[NS], float (&c)[NS]) {
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    v[s] = L.sc[s].v0;
    x[s] = 0.0f;
    c[s] = 0.0f;
  }
  const PhiloxLane pl[1] = {philox_lane(path, L.rk)};
  uint4 w[1], n[1];
  philox_draws<TAB, 1>(tab, 0u, L.option_index, L.rk, pl, w);
  StepDraw d;
  {
    const float2 xu = centered_uniform2(w[0].x, w[0].y);
    const float2 z = norminv_centered2(xu);
    d = StepDraw{xu.x, z.x, z.y};
  }
  const uint32_t pairs = L.steps >> 1;
  uint32_t i = 0;
  if (L.first_split) {  // step 0 of every scenario from its own constants, then step 1
    step0_apply<NS, false>(L, d.xv, d.zv, d.zx, v, x, c);
    if (pairs) {
      const float2 xu = centered_uniform2(w[0].z, w[0].w);
      const float2 z = norminv_centered2(xu);
      d = StepDraw{xu.x, z.x, z.y};
      philox_draws<TAB, 1>(tab, 1u, L.option_index, L.rk, pl, w);
      step_merged<NS, NV, true>(L, d, w[0].x, w[0].y, v, x, c);
    }
    i = 1;
  }
#pragma unroll 1
  for (; i < pairs; ++i) {
    philox_draws<TAB, 1>(tab, i + 1, L.option_index, L.rk, pl, n);  // (one pair past the last step is not used)
    step_merged<NS, NV, true>(L, d, w[0].z, w[0].w, v, x, c);
    step_merged<NS, NV, true>(L, d, n[0].x, n[0].y, v, x, c);
    w[0] = n[0];
  }
  if ((L.steps & 1u) && !(L.first_split && L.steps == 1))  // odd last step
    step_merged<NS, NV, true>(L, d, 0u, 0u, v, x, c);
}

// PPT paths per thread, simulated step by step in lockstep: independent
// dependency chains the scheduler can interleave (instruction-level
// parallelism at the same occupancy).
template <bool TAB, int NS, int NV, bool DYN, int PPT, bool QEM = false, bool ROLL = false>
__device__ __forceinline__ void simulate_ppt(const PathLaunch& L, const uint4* tab, const uint64_t (&path)[PPT],
                                             float (&v)[PPT][NS], float (&x)[PPT][NS], float (&c)[PPT][NS]) {
#pragma unroll
  for (int j = 0; j < PPT; ++j) {
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      v[j][s] = (DYN && s >= L.n_scen) ? 0.0f : L.sc[s].v0;
      x[j][s] = 0.0f;
      c[j][s] = 0.0f;
    }
  }
  PhiloxLane pl[PPT];
#pragma unroll
  for (int j = 0; j < PPT; ++j) pl[j] = philox_lane(path[j], L.rk);
  if constexpr (ROLL) {  // one step per iteration (path_roll_steps)
    uint4 w[PPT];
    uint32_t n = 0;
    if (NS > 1 && L.first_split) {
      philox_draws<TAB, PPT>(tab, 0u, L.option_index, L.rk, pl, w);
#pragma unroll
      for (int j = 0; j < PPT; ++j) step0_all<NS, DYN, QEM>(L, w[j].x, w[j].y, v[j], x[j], c[j]);
      n = 1;
    }
#pragma unroll 1
    for (; n < L.steps; ++n) {
      if (!(n & 1u)) philox_draws<TAB, PPT>(tab, n >> 1, L.option_index, L.rk, pl, w);
      uint32_t wv[PPT], wx[PPT];
#pragma unroll
      for (int j = 0; j < PPT; ++j) {
        wv[j] = n & 1u ? w[j].z : w[j].x;
        wx[j] = n & 1u ? w[j].w : w[j].y;
      }
      step_paths<NS, NV, DYN, PPT, QEM>(L, wv, wx, v, x, c);
    }
    return;
  }
  const uint32_t pairs = L.steps >> 1;
  uint32_t i0 = 0;
  if (NS > 1 && L.first_split) {
    uint4 w[PPT];
    philox_draws<TAB, PPT>(tab, 0u, L.option_index, L.rk, pl, w);
#pragma unroll
    for (int j = 0; j < PPT; ++j) step0_all<NS, DYN, QEM>(L, w[j].x, w[j].y, v[j], x[j], c[j]);
    if (L.steps > 1) {
      uint32_t wv[PPT], wx[PPT];
#pragma unroll
      for (int j = 0; j < PPT; ++j) wv[j] = w[j].z, wx[j] = w[j].w;
      step_paths<NS, NV, DYN, PPT, QEM>(L, wv, wx, v, x, c);
    }
    i0 = 1;
  }
  for (uint32_t i = i0; i < pairs; ++i) {
    uint4 w[PPT];
    uint32_t wv[PPT], wx[PPT];
    philox_draws<TAB, PPT>(tab, i, L.option_index, L.rk, pl, w);
#pragma unroll
    for (int j = 0; j < PPT; ++j) wv[j] = w[j].x, wx[j] = w[j].y;
    step_paths<NS, NV, DYN, PPT, QEM>(L, wv, wx, v, x, c);
#pragma unroll
    for (int j = 0; j < PPT; ++j) wv[j] = w[j].z, wx[j] = w[j].w;
    step_paths<NS, NV, DYN, PPT, QEM>(L, wv, wx, v, x, c);
  }
  if ((L.steps & 1u) && !(NS > 1 && L.first_split && L.steps == 1)) {  // odd last step (step 0 itself when steps == 1 without the split)
    uint4 w[PPT];
    uint32_t wv[PPT], wx[PPT];
    philox_draws<TAB, PPT>(tab, pairs, L.option_index, L.rk, pl, w);
#pragma unroll
    for (int j = 0; j < PPT; ++j) wv[j] = w[j].x, wx[j] = w[j].y;
    step_paths<NS, NV, DYN, PPT, QEM>(L, wv, wx, v, x, c);
  }
}

// Results of strike k from its n_acc sums (sum_a = s[a * stride]): the price
// e^{-rT} sum f / n, its standard error, and each Greek e^{-rT} sum / (n denom);
// or, in raw mode, the sums themselves.  FP64.
// A strike flagged `bad` (not finite and > 0) gets NaN results.
__device__ __forceinline__ void write_results(const PathLaunch& L, int k, const double* s, int stride,
                                              const PathOutputs& out, bool bad) {
  const double nan = __longlong_as_double(0x7ff8000000000000ll);
  if (L.raw_sums) {
    for (int a = 0; a < L.n_acc; ++a) out.sums[(size_t)k * L.n_acc + a] = bad ? nan : s[(size_t)a * stride];
    return;
  }
  if (bad) {
    out.price[k] = nan;
    if (out.stderr_) out.stderr_[k] = nan;
    if (out.greeks)
      for (int g = 0; g < L.n_acc - 2; ++g) out.greeks[(size_t)k * (L.n_acc - 2) + g] = nan;
    return;
  }
  const double n = L.paths_total, inv_n = 1.0 / n;
  const double mean = s[0] * inv_n;
  out.price[k] = L.disc * mean;
  if (out.stderr_) {
    const double var = n > 1.0 ? (s[stride] * inv_n - mean * mean) / (n - 1.0) : 0.0;
    out.stderr_[k] = L.disc * sqrt(var > 0.0 ? var : 0.0);
  }
  if (out.greeks) {
    const int ng = L.n_acc - 2;
    for (int g = 0; g < ng; ++g)
      out.greeks[(size_t)k * ng + g] = L.disc * s[(size_t)(2 + g) * stride] * inv_n / L.denom[g];
  }
}

// Warps per block, one block per SM: the register file split by what a thread of NS
// scenarios needs.
template <int NS, bool QEM>
constexpr int path_warps() {
  return NS == 1 ? (QEM ? SIMR_QEM_WARPS : SIMR_PRICE_WARPS) : NS == 3 ? SIMR_FD3_WARPS : NS == 5 ? SIMR_FD5_WARPS : SIMR_FD11_WARPS;
}

// Whether the kernel of NS scenarios has a loop for the step pairs' counter table:
// not with 11 and more, nor the QE-M bumps, whose arithmetic hides what it saves.
template <int NS, bool QEM>
constexpr bool path_table() {
  return NS == 1 || (NS <= 5 && !QEM);
}

// The steps up to which simulate_ppt takes one step per iteration: all with strike tiles,
// where the step's code beside the tile's sums overflowed the instruction cache in a long run
// (four copies of it 208 KB a kernel, one 140 KB: 11 scenarios x 32 strikes, 30 steps x 2.5 M
// paths 3.2 -> 2.35 ms, 250 steps x 2^22 paths 18.8 -> 16.8; 13 scenarios 4% faster at 1,024
// steps still), but for 11 QE scenarios, where two steps an iteration win once the steps
// outweigh the sums (1,024 x 2^22 64.05 / 62.05 ms, 500 x 2^20 8.11 / 8.40, even near 760);
// and with 11 QE-M scenarios (one strike 5% faster).  One strike under QE keeps two steps, 4%
// faster at 200 steps with 7 and 11 scenarios, as does the terminal kernel (14%).
template <int NS, int TILE, bool QEM>
constexpr uint32_t path_roll_steps() {
  return NS == 11 && TILE > 1 && !QEM ? 760u : TILE > 1 || (QEM && NS >= 11) ? 0xffffffffu : 0u;
}

// The form of an item's row (ItemRow): pointers for QE pricing (252 steps x 2^20 paths x 32
// strikes 741 us, 748 with an offset) and 11 scenarios (365 x 250,001 x 21 1,619 / 1,667 us);
// an offset for 5 scenarios (252 x 2^20 x 32 2,160 us with pointers, 2,132 with it), 3 (64 x
// 65,536 88.9 / 86.6) and QE-M (pricing 1% slower with pointers).
template <int NS, bool QEM>
constexpr bool path_row_pointers() {
  return !QEM && (NS == 1 || NS == 11);
}

// Fused price / Greeks kernel.  TILE = 1 (single strike) or 32 (strike tiles).
// One block per SM; its warps take the block's batches item by item (ItemPlan).
// Dynamic shared memory: the strike constants [nk_pad] (StrikeConst), a flag word
// and the item counter, the step pairs' counter table, then the items' rows of n_acc x nk_pad sums (ItemRows).
template <int NS, int NV, int TILE, bool DYN, int PPT, bool QEM, bool ROLL>
__global__ void __launch_bounds__(kWarp * path_warps<NS, QEM>(), 1)
    heston_paths_kernel(const __grid_constant__ PathLaunch L, const __grid_constant__ ItemPlan I,
                        const double* __restrict__ strikes, PathOutputs out, double* __restrict__ partials,
                        unsigned int* __restrict__ ticket) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31;
  StrikeConst* ks = reinterpret_cast<StrikeConst*>(smem_raw);
  int* s_flag = reinterpret_cast<int*>(ks + L.nk_pad);
  unsigned* s_next = reinterpret_cast<unsigned*>(s_flag + 1);
  uint4* tab = L.pair_table ? reinterpret_cast<uint4*>(s_flag + 4) : nullptr;
  const ItemRows rows{smem_raw, (unsigned)(L.nk_pad * sizeof(StrikeConst) + 16 + L.pair_table * sizeof(uint4)), L.n_acc * L.nk_pad};

  if (threadIdx.x == 0) *s_next = 0u;
  for (int p = threadIdx.x; p < L.pair_table; p += blockDim.x)
    tab[p] = philox_pair_entry(p, L.option_index, (uint32_t)(L.path_begin >> 32), L.rk);
  for (int j = threadIdx.x; j < L.nk_pad; j += blockDim.x) {
    StrikeConst k{0.0f, 0.0f, 0.0f, 0.0f};
    if (j < L.n_strikes) {
      const double K = strikes[j];
      if (!(K > 0.0) || !isfinite(K)) atomicOr(out.status, 1);  // reported by simr_sync
      k.K = (float)K;
      k.Km = (float)(K * L.rho_em);
      k.Wr = (float)(K * L.rho_w);
    }
    ks[j] = k;
  }
  __syncthreads();

  constexpr bool USE_TAB = path_table<NS, QEM>();
  const uint64_t per_batch = (uint64_t)kWarp * PPT;
  const uint64_t block0 = I.batches / gridDim.x * blockIdx.x + min((uint64_t)blockIdx.x, I.batches % gridDim.x);
  const uint64_t nb = I.batches / gridDim.x + (blockIdx.x < I.batches % gridDim.x ? 1 : 0);
  while (true) {
    unsigned it = 0;
    if (lane == 0) it = atomicAdd(s_next, 1u);
    it = __shfl_sync(kFull, it, 0);
    uint64_t b0, b1;
    if (!item_range(I, it, nb, b0, b1)) break;
    auto my = rows.template at<path_row_pointers<NS, QEM>()>(I, it);
    const uint64_t end = (block0 + b1) * per_batch;
    for (uint64_t first = (block0 + b0) * per_batch; first < end; first += per_batch) {
      uint64_t pth[PPT];
      bool act[PPT];
#pragma unroll
      for (int j = 0; j < PPT; ++j) {
        const uint64_t local = first + (uint64_t)j * kWarp + lane;
        act[j] = local < L.path_count;
        pth[j] = L.path_begin + local;
      }
      float v[PPT][NS], x[PPT][NS], c[PPT][NS];
      if constexpr (NS == 1 && PPT == 2) {
        float2 v2, x2, c2;
        if (tab)
          simulate_two_pipe<QEM, true>(L.sc[0], L.steps, L.option_index, L.rk, tab, pth[0], pth[1], v2, x2, c2, L.qm,
                                       [](uint32_t) {});
        else
          simulate_two_pipe<QEM, false>(L.sc[0], L.steps, L.option_index, L.rk, tab, pth[0], pth[1], v2, x2, c2, L.qm,
                                        [](uint32_t) {});
        x[0][0] = x2.x;
        x[1][0] = x2.y;
        c[0][0] = c2.x;
        c[1][0] = c2.y;
      } else if constexpr ((NS == 3 || NS == 5) && PPT == 1 && !QEM && !DYN) {
        if (USE_TAB && tab)
          simulate_fd<USE_TAB, NS, NV>(L, tab, pth[0], v[0], x[0], c[0]);
        else
          simulate_fd<false, NS, NV>(L, nullptr, pth[0], v[0], x[0], c[0]);
      } else if (USE_TAB && tab) {
        simulate_ppt<USE_TAB, NS, NV, DYN, PPT, QEM, ROLL>(L, tab, pth, v, x, c);
      } else {
        simulate_ppt<false, NS, NV, DYN, PPT, QEM, ROLL>(L, nullptr, pth, v, x, c);
      }
      float S[PPT][NS];
#pragma unroll
      for (int j = 0; j < PPT; ++j)
#pragma unroll
        for (int s = 0; s < NS; ++s) S[j][s] = terminal_spot(L.S0, x[j][s], c[j][s]);

      // accumulator list: 0 f, 1 f^2, then set Greek bits in order
      int a = 0, r = 0;
      for (int bit = -2; bit < kMaxGreeks; ++bit) {
        if (bit >= 0 && !((L.greek_mask >> bit) & 1u)) continue;
        const bool resim = bit == 2 || bit == 3 || bit >= 5;
        const int up = resim ? L.resim_up[r] : 0, dn = resim ? L.resim_dn[r] : 0;
        if (TILE == 1) {
          float t = 0.0f;
#pragma unroll
          for (int j = 0; j < PPT; ++j) {
            const float tj = resim ? resim_term<NS>(L, up, dn, ks[0], S[j]) : acc_term<NS>(L, bit, a, ks[0], S[j]);
            t += act[j] ? tj : 0.0f;
          }
          t = warp_sum(t);
          if (lane == 0) my.add<true>(smem_raw, a, t);
        } else {
          for (int t0 = 0; t0 < L.nk_pad; t0 += 32) {
            float vals[32];
#pragma unroll
            for (int jj = 0; jj < 32; ++jj) {
              const StrikeConst k = ks[t0 + jj];
              float t = 0.0f;
#pragma unroll
              for (int j = 0; j < PPT; ++j) {
                const float tj = resim ? resim_term<NS>(L, up, dn, k, S[j]) : acc_term<NS>(L, bit, a, k, S[j]);
                t += act[j] ? tj : 0.0f;
              }
              vals[jj] = t;
            }
            butterfly32(vals, lane);
            my.add<true>(smem_raw, a * L.nk_pad + t0 + lane, vals[0]);
          }
        }
        if (resim) ++r;
        ++a;
      }
      my.next_batch();
    }
  }
  __syncthreads();
  sum_item_rows(rows, I, nb);
  __syncthreads();
  if (!sum_block_rows(rows.acc(I), rows.row, partials, ticket, s_flag)) return;
  for (int k = threadIdx.x; k < L.n_strikes; k += blockDim.x) {
    const double K = strikes[k];
    write_results(L, k, rows.acc(I) + k, L.nk_pad, out, !(K > 0.0) || !isfinite(K));
  }
}

// Normalise sums of a sharded run: sums[k][n_acc] -> outputs.
__global__ void finalize_sums_kernel(const __grid_constant__ PathLaunch L, const double* __restrict__ sums,
                                     PathOutputs out) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < L.n_strikes) write_results(L, k, sums + (size_t)k * L.n_acc, 1, out, false);
}

template <bool QEM>
__global__ void __launch_bounds__(256) heston_terminal_kernel(const __grid_constant__ PathLaunch L,
                                                              float* __restrict__ x_T, float* __restrict__ v_T) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= L.path_count) return;
  float v[1][1], x[1][1], c[1][1];
  const uint64_t pth[1] = {L.path_begin + i};
  simulate_ppt<false, 1, 0, false, 1, QEM>(L, nullptr, pth, v, x, c);
  x_T[i] = x[0][0] - c[0][0];
  if (v_T) v_T[i] = v[0][0];
}

template <int NS, int NV, int TILE, bool DYN, bool QEM = false,
          int PPT = (NS == 1 ? SIMR_PRICE_PPT : SIMR_FD_PPT)>
cudaError_t launch_t(const PathLaunch& L0, const double* strikes, const PathOutputs& out, const Scratch& s,
                     int num_sms, cudaStream_t stream, int* grid_used) {
  PathLaunch L = L0;
  L.pair_table = path_table<NS, QEM>() ? pair_table_entries(L0) : 0;
  const size_t row = (size_t)L.n_acc * L.nk_pad;
  const size_t head = L.nk_pad * sizeof(StrikeConst) + 16 + L.pair_table * sizeof(uint4);
  const uint64_t batches = (L.path_count + (uint64_t)kWarp * PPT - 1) / ((uint64_t)kWarp * PPT);
  const uint64_t grid = std::min<uint64_t>(num_sms, batches);  // one block per SM
  ItemPlan I = make_item_plan(batches, grid, path_warps<NS, QEM>(), row, kItemBytes - head);
  // rows so long that each warp has one fixed share: pricing, whose long strike loop is
  // issue-bound, with as many warps on every SM sub-partition (50 steps x 2^20 x 768 strikes
  // 747 -> 688 us at 12 warps for 15, QE-M 803 -> 736; 2^22 x 1,024 strikes 3.75 -> 3.57 ms at
  // 8 for 10; the bumps and the adjoint lose 3-10% with fewer)
  if (NS == 1 && I.levels == 0 && I.tail_size > 1 && I.warps > 8 && I.warps % 4)
    I = make_item_plan(batches, grid, I.warps & ~3, row, kItemBytes - head);
  const int tpb = kWarp * I.warps;
  const size_t smem = head + item_rows_bytes(I, row);
  constexpr uint32_t roll = path_roll_steps<NS, TILE, QEM>();
  auto kern = heston_paths_kernel<NS, NV, TILE, DYN, PPT, QEM, (roll > 0)>;
  if constexpr (roll > 0 && roll < 0xffffffffu)
    if (L.steps > roll) kern = heston_paths_kernel<NS, NV, TILE, DYN, PPT, QEM, false>;
  cudaError_t e = cudaSuccess;
  if (smem > 48 * 1024)  // (below, the default suffices)
    e = allow_dynamic_smem(kern);
  if (e != cudaSuccess) return e;
  if ((size_t)(grid + kRowGroups) * row > s.partial_doubles) return cudaErrorMemoryAllocation;
  *grid_used = (int)grid;
  kern<<<(unsigned)grid, tpb, smem, stream>>>(L, I, strikes, out, s.partials, s.ticket);
  return cudaGetLastError();
}

}  // namespace

// Entries of the shared-memory table of step-pair counters: one per pair and one
// past the last, which a pipelined loop reads; none where the paths cross a
// multiple of 2^32 (their high words differ), or past 32 KB (4,092 steps), which
// the items' rows need more.
int pair_table_entries(const PathLaunch& L) {
  const uint64_t n = (uint64_t)L.steps / 2 + 2;
  const bool one_high_word = (L.path_begin >> 32) == ((L.path_begin + L.path_count - 1) >> 32);
  return one_high_word && n <= 2048 ? (int)n : 0;
}

size_t paths_scratch_doubles(const PathLaunch& L, int num_sms) {
  return (size_t)(num_sms + kRowGroups) * (size_t)L.n_acc * L.nk_pad;
}

cudaError_t launch_paths(const PathLaunch& L, const double* strikes, const PathOutputs& out, const Scratch& s,
                         int num_sms, cudaStream_t stream, int* grid_used) {
  const bool one = L.nk_pad == 1;
  const bool v2 = L.n_v0_scen == 2;  // scenarios 1, 2 are the v0 bumps (constant deltas zero)
#define SIMR_LAUNCH(NS_, NV_, DYN_)                                                                \
  (one ? launch_t<NS_, NV_, 1, DYN_>(L, strikes, out, s, num_sms, stream, grid_used)               \
       : launch_t<NS_, NV_, 32, DYN_>(L, strikes, out, s, num_sms, stream, grid_used))
  if (L.scheme == 1) {  // QE-M: the base scenario alone, 5 or 11 scenarios in pairs, any other count dynamic
#define SIMR_LAUNCH_QEM(NS_, DYN_)                                                                     \
  (one ? launch_t<NS_, 0, 1, DYN_, true>(L, strikes, out, s, num_sms, stream, grid_used)               \
       : launch_t<NS_, 0, 32, DYN_, true>(L, strikes, out, s, num_sms, stream, grid_used))
    switch (L.n_scen) {
      case 1:
        return SIMR_LAUNCH_QEM(1, false);
      case 5:
        return SIMR_LAUNCH_QEM(5, false);
      case 11:
        return SIMR_LAUNCH_QEM(11, false);
      default:
        if (L.n_scen < 1 || L.n_scen > kMaxScen) return cudaErrorInvalidValue;
        return SIMR_LAUNCH_QEM(kMaxScen, true);
    }
#undef SIMR_LAUNCH_QEM
  }
  switch (L.n_scen) {
    case 1:
      return SIMR_LAUNCH(1, 0, false);
    case 3:
      return v2 ? SIMR_LAUNCH(3, 2, false) : SIMR_LAUNCH(3, 0, false);
    case 5:
      return v2 ? SIMR_LAUNCH(5, 2, false) : SIMR_LAUNCH(5, 0, false);
    case 11:  // all five re-simulated model-parameter Greeks
      return v2 ? SIMR_LAUNCH(11, 2, false) : SIMR_LAUNCH(11, 0, false);
    default:
      if (L.n_scen < 1 || L.n_scen > kMaxScen) return cudaErrorInvalidValue;
      return v2 ? SIMR_LAUNCH(kMaxScen, 2, true) : SIMR_LAUNCH(kMaxScen, 0, true);
  }
#undef SIMR_LAUNCH
}

cudaError_t launch_finalize(const PathLaunch& L, const double* sums, const PathOutputs& out, cudaStream_t stream) {
  const int tpb = 128;
  finalize_sums_kernel<<<(L.n_strikes + tpb - 1) / tpb, tpb, 0, stream>>>(L, sums, out);
  return cudaGetLastError();
}

cudaError_t launch_terminal(const PathLaunch& L, float* x_T, float* v_T, cudaStream_t stream) {
  const int tpb = 256;
  const uint64_t grid = (L.path_count + tpb - 1) / tpb;
  if (L.scheme == 1)
    heston_terminal_kernel<true><<<(unsigned)grid, tpb, 0, stream>>>(L, x_T, v_T);
  else
    heston_terminal_kernel<false><<<(unsigned)grid, tpb, 0, stream>>>(L, x_T, v_T);
  return cudaGetLastError();
}

}  // namespace simr
