// Element-local kernel of the 2D shallow-water cRK-FR step (sm_103a, FP64),
// shared by kernels_2d.cu (no source) and kernels_imex.cu (Chezy friction
// treated implicitly, Sec. 2 Eqs. crkfr.inner, crkfr, avg.source, with
// SSP3-IMEX(4,3,3)).
//
// One thread owns one node: an element's (N+1)^2 threads exchange the fluxes
// of a stage through shared memory and each takes its node's row of D_x and
// D_y.  All inner stages stay on chip; the kernel writes W = u^n - dt (dloc F
// + Bloc) [+ dt S] (Eqs. disc.avg.flux, local.time.avg.non.cons, avg.source)
// and, for every face node, the traces the Riemann problem needs: the
// time-averaged solution U, the time-averaged normal flux and h^n and the
// normal momentum at t^n (Eqs. time.avg.soln, combined.wave.speed,
// good.numflux.non.cons).
//
// The stage sums are FP64; the contractions with D_x, D_y and the end-point
// rows, which were 60 % of the FP64 instructions, the time averages and the
// fluxes run in block fixed point on the integer pipe (fixed_point.cuh).  D is
// applied to the time-averaged fluxes once instead of accumulating every
// stage's operator, so the last stage needs no contraction.  On a 1024 x 1024
// mesh at N = 3 the kernel takes 2.17 ms, bound by issue slots and the integer
// multiplier together (0.63 instructions per cycle and scheduler, multiplier 65
// % busy, ALU 61 %, FP64 pipe 37 %), against 6.4 ms with FP64 chains (one thread
// per element row, FP64 pipe 96 %).  One thread per row in fixed point took 4.2
// ms: 255 registers and two warps per scheduler left the latencies open, and
// 9700 instructions a warp missed the instruction cache; a thread per node takes
// a quarter of the code.  FP64 fluxes, seven FP64 instructions a stage and each
// result converted, cost another 4 to 9 % of a step (two steps on 1024 x 1024
// 5.45 against 5.22 ms, 512 x 512 with friction 2.52 against 2.28 ms).
//
// An exponent per field instead of one for hu and hv and one for all fluxes,
// and the fields of an equation aligned after their contractions, take 512 x 512
// at N = 3 from 499 to 541 us and 401 x 307 well-balanced at N = 4 from 819 to 888
// us: what a small momentum beside a large one needs to keep the precision that
// FP64 gives it.
//
// The well-balanced form (WB) has pressure-free fluxes and the
// non-conservative terms g h D_x (h + b), g h D_y (h + b).
//
// With the subcell blending limiter (LIMIT; the tensor-product extension of
// Sec. 4) the kernel ends with the first-order part of limit_2d.cuh.
#pragma once

#include <cuda_runtime.h>

#include "device_common.cuh"
#include "fixed_point.cuh"
#include "launch.h"
#include "limit_2d.cuh"

namespace crkfr {
namespace {

#ifndef CRKFR_LOCAL2D_BLOCK
#define CRKFR_LOCAL2D_BLOCK 128
#endif
constexpr int kBlockLocal = CRKFR_LOCAL2D_BLOCK;
constexpr int kTrFields = 7;
// x-face trace fields: U_h, U_hu, U_hv, F_hu, F_hv (time-averaged x fluxes of
// hu and hv), h^n, hu^n.  y-face trace fields: U_h, U_hu, U_hv, G_hu, G_hv,
// h^n, hv^n.  (The time-averaged h fluxes are U_hu and U_hv.)

// Elements per block: as many as fit (n = 2, 4: whole warps; n = 3: 14 on 126
// of 128 threads, n = 5: 5 on 125).
template <int n>
__host__ __device__ constexpr int local_elements() {
  return kBlockLocal / (n * n);
}

// Stage loop unrolled, with the earlier stages' operators and sources in
// registers (short tableaux and friction: 512 x 512 with friction 2.50 ms for
// two steps, 2.65 ms rolled), or rolled (unrolled, the kernel of N = 3 misses
// the instruction cache, hit rate 86 %: 1024 x 1024 5.67 ms for two steps, 5.47
// ms rolled; 401 x 307 at N = 4 2.25 and 2.07 ms), which also leaves room for
// 28 instead of 20 warps per SM.
template <int N, bool IMEX>
__host__ __device__ constexpr bool local_unrolled() {
  return IMEX || N <= 2;
}
template <int N, bool IMEX, bool LIMIT>
__host__ __device__ constexpr int local_min_blocks() {
  return LIMIT ? 3 : local_unrolled<N, IMEX>() ? 5 : 7;
}

// Exchange fields of the kernel: 0..5 the averages of h, hu, hv, hu hu / h
// (+ pressure), hu hv / h, hv hv / h (+ pressure), or a stage's values of
// them; 6..8 u^n.  Each of 0..5 has an exponent of its own per element (a small
// momentum beside a large one keeps its bits; two terms of one equation are
// aligned only where their derivatives are added).  The average of h enters
// the source term node by node, so it is formed in FP64, from h^n and the
// stages' operators; in the well-balanced form, whose source term has the
// stages' own h, it is for the traces only, and with GL nodes a sum as the others.
constexpr int kLocalFields = 9;
constexpr int kLocalGroups = 6;

// b~_i / b_ref of a stage counted at run time
template <class TB>
__device__ __forceinline__ int local_weight(int i) {
  unsigned long long w = 0;
#pragma unroll
  for (int k = 0; k < TB::S; ++k) w |= (unsigned long long)TB::weight(k) << (8 * k);
  return (int)(w >> (8 * i)) & 0xff;
}

// the same in FP64, from the upper halves of the weights' high words (a
// conversion is an FP64 instruction)
template <class TB>
__device__ __forceinline__ double local_weight_fp(int i) {
  unsigned long long w[2] = {0, 0};
#pragma unroll
  for (int k = 0; k < TB::S; ++k) {
    // m 2^e, m < 2: exponent 1023 + e, four bits of m - 1
    int m = TB::weight(k), e = 0;
    while (m >> (e + 1)) ++e;
    const unsigned long long h = m ? (unsigned)((1023 + e) << 4 | ((m << 4 >> e) & 15)) : 0;
    w[k / 4] |= h << (16 * (k % 4));
  }
  const unsigned long long x = TB::S > 4 && i >= 4 ? w[1] >> (16 * (i - 4)) : w[0] >> (16 * i);
  return __hiloint2double((int)(unsigned)(x << 16), 0);
}

// bit 8 i + j: a~_ij is not zero
template <class TB>
__device__ __forceinline__ unsigned long long local_nonzero() {
  unsigned long long m = 0;
#pragma unroll
  for (int i = 0; i < TB::S; ++i)
#pragma unroll
    for (int j = 0; j < i; ++j)
      if (TB::a(i, j) != 0.0) m |= 1ull << (8 * i + j);
  return m;
}

// every stage sum takes the operator of the stage before it only
template <class TB>
__host__ __device__ constexpr bool local_chain() {
  for (int i = 0; i < TB::S; ++i)
    for (int j = 0; j + 1 < i; ++j)
      if (TB::a(i, j) != 0.0) return false;
  return true;
}

// Doubles per element in shared memory, 4 modulo 16 so that the elements of a
// warp start 32 bytes apart modulo the banks.
template <int n, bool LIMIT>
__host__ __device__ constexpr int local_stride() {
  return ((LIMIT ? kLimExchange : kLocalFields) * n * n + 11) / 16 * 16 + 4;
}

template <int N, bool GLL, bool RES, bool IMEX, bool WB, bool LIMIT = false, bool STAGES = false,
          int PRE = 0>
__global__ void __launch_bounds__(kBlockLocal, local_min_blocks<N, IMEX, LIMIT>())
    k_local_2d(const Launch2D L) {
  static_assert(!(STAGES && (IMEX || WB || LIMIT)), "stages are recorded for the standard form");
  // PRE 1: only the first stage's local operator L(u^n), which needs no dt,
  // stored in L.w; PRE 2: the step, taking L(u^n) from L.w (same arithmetic)
  static_assert(PRE == 0 || !(RES || IMEX || WB || LIMIT || STAGES),
                "the first-stage pre-pass is built for the standard form");
  using TB = Tab<N, IMEX>;
  static_assert(PRE == 0 || TB::feeds(0), "the first stage feeds a later one");
  constexpr int n = N + 1;
  constexpr int nn = n * n;
  constexpr int S = TB::S;
  constexpr int EPB = local_elements<n>();
  constexpr int ES = local_stride<n, LIMIT>();
  // bits of the fixed-point operands (weighted sums up to 6 stay below 2^63;
  // the six-stage method's, up to 90, are kept in two halves), the shift that
  // brings a sum back to FB bits, and the bits by which a later stage may
  // outgrow the first before the exponents are raised
  constexpr int FB = 59;
  constexpr bool WIDE = TB::weight_sum() > 8;
  constexpr int kSumShift = WIDE ? 7 : 3;
  constexpr int kHeadroom = 1;
  // elements within whole warps need no block barrier
  constexpr bool WARP = 32 % nn == 0;
  const Tables& T = L.tab;
  __shared__ __align__(16) double sm[EPB * ES];
  __shared__ int smag[EPB][kLocalGroups];
  __shared__ StepSizes<TB> sz;

  const int le_raw = threadIdx.x / nn, node = threadIdx.x - le_raw * nn;
  const int q = node / n, p = node - q * n;
  const int64_t Ne = L.Ex * L.Ey;
  const bool lane_ok = le_raw < EPB;
  const int le = lane_ok ? le_raw : 0;
  Fx (*X)[n][n] = reinterpret_cast<Fx (*)[n][n]>(&sm[le * ES]);
  auto sync = [] {
    if (WARP)
      __syncwarp();
    else
      __syncthreads();
  };
  auto sync_or = [](bool b) -> bool {
    return WARP ? warp_barrier_or(b) : __syncthreads_or(b);
  };

  chain_begin();
  // the step size (a division) and its products by the block's first warp;
  // the others start on the first stage, which needs neither
  if (threadIdx.x < 32) {
    double dt = 0.0;
    if (threadIdx.x == 0) {
      dt = (RES || PRE == 1) ? L.ctl.dt_fixed : step_dt(L.ctl, L.st);
      if (!RES && PRE != 1 && blockIdx.x == 0 && !L.ctl.skip_bookkeeping)
        step_bookkeeping(L.ctl, L.st, dt);
    }
    dt = __shfl_sync(0xffffffffu, dt, 0);
    fill_step_sizes<TB, IMEX>(sz, dt, 1.0);
  }
  // threads past EPB n^2 and elements past the rows [row_begin, row_end)
  // compute on element 0 and store nothing to memory (the former nothing to
  // shared memory either)
  const int64_t g = L.row_begin * L.Ex + (int64_t)blockIdx.x * EPB + le;
  const bool active = lane_ok && (g < L.row_end * L.Ex);
  const int64_t ge = active ? g : 0;

  // ---- u^n, the static terms g b_x, g b_y and the node's rows of D ----------
  double u0[3];
#pragma unroll
  for (int v = 0; v < 3; ++v) u0[v] = L.u_in[(v * Ne + ge) * nn + node];
  const double gbx = L.snode[ge * nn + node], gby = L.snode[(Ne + ge) * nn + node];
  int dxh[n], dxl[n], dyh[n], dyl[n];
#pragma unroll
  for (int j = 0; j < n; ++j) {
    dxh[j] = T.fx.Dx_hi[p][j];
    dxl[j] = T.fx.Dx_lo[p][j];
    dyh[j] = T.fx.Dy_hi[q][j];
    dyl[j] = T.fx.Dy_lo[q][j];
  }
  if (lane_ok) {
    for (int k = node; k < kLocalGroups; k += nn) smag[le][k] = 0;
  }
  sync();

  // The operators L_j of earlier stages that a stage sum needs: the last one
  // only (classical RK4), or all of them, in registers or shared memory; the
  // sources of hu, hv (IMEX) in registers.
  constexpr bool UNROLL = local_unrolled<N, IMEX>(), CHAIN = !UNROLL && local_chain<TB>();
  constexpr bool SHARED = !UNROLL && !CHAIN;
  constexpr int kStageUnroll = UNROLL ? S : 1;
  static_assert(UNROLL || !IMEX, "the sources are kept in registers");
  __shared__ double sL[SHARED ? S - 1 : 1][3][SHARED ? kBlockLocal : 1];
  double rL[UNROLL ? S : 1][3], rS[IMEX ? S : 1][2];
  double Lp[3] = {0.0, 0.0, 0.0};
  if constexpr (PRE == 2) {
    // L(u^n), computed ahead by the PRE 1 instantiation; the thread
    // overwrites the same values with W at the end
#pragma unroll
    for (int v = 0; v < 3; ++v) Lp[v] = L.w[(v * Ne + ge) * nn + node];
  }
  double Sb[2] = {0.0, 0.0};     // sum_j (b_j/b_ref) s(u^(j)) (IMEX)
  double P1 = 0.0, P2 = 0.0;     // sum_j (b_j/b_ref) h g d(h + b) (WB)
  constexpr bool FIX_H = WB && !GLL;   // the average of h as field 0's sum
  double uh = 0.0;               // or sum_j (b_j/b_ref) (h^(j) - h^n), below + h^n / b_ref
  // time averages sum_j (b_j/b_ref) of the exchange fields 1..5 in the fixed
  // point of their exponents E, which only grow: the sums are shifted when
  // they do
  long long A[6] = {0, 0, 0, 0, 0, 0}, B[6] = {0, 0, 0, 0, 0, 0};
  int E[kLocalGroups] = {-1, -1, -1, -1, -1, -1};
  constexpr int k0 = WB ? 0 : 1;   // (h is contracted in the well-balanced form only)
  // row of D_x on field f (y: row of D_y)
  auto row_x = [&](int f) -> long long {
    FxAcc a;
    Fx r[n];
    fx_row<n>(X[f][q], r);
    fx_mul(a, r[0], dxh[0], dxl[0]);
#pragma unroll
    for (int j = 1; j < n; ++j) fx_mad(a, r[j], dxh[j], dxl[j]);
    return fx_sum(a);
  };
  auto row_y = [&](int f) -> long long {
    FxAcc a;
    fx_mul(a, X[f][0][p], dyh[0], dyl[0]);
#pragma unroll
    for (int j = 1; j < n; ++j) fx_mad(a, X[f][j][p], dyh[j], dyl[j]);
    return fx_sum(a);
  };
  // row of D_x on field fx plus row of D_y on field fy, in units 2^shift larger
  // (at N = 1 a row of D is a difference: equal values cancel without rounding)
  auto contract = [&](int fx, int fy, int shift) -> double {
    int e;
    const long long s =
        fx_align<N == 1>(row_x(fx), E[fx] + T.fx.kDx, row_y(fy), E[fy] + T.fx.kDy, e);
    return fx_to(s, e - FB + shift, fx_zero(max(E[fx], E[fy])));
  };
#pragma unroll kStageUnroll
  for (int i = 0; i < S; ++i) {
    if (i == (IMEX ? 0 : 1)) __syncthreads();   // the step sizes
    if (!FIX_H && i > 0) uh = fma(sz.avg[i - 1], Lp[0], uh);
    double cur[3];
#pragma unroll
    for (int v = 0; v < 3; ++v) cur[v] = u0[v];
    if constexpr (CHAIN) {
      if (i > 0) {
        const double c = sz.e[i][i - 1];
#pragma unroll
        for (int v = 0; v < 3; ++v) cur[v] = fma(c, Lp[v], cur[v]);
      }
    } else if constexpr (SHARED) {
      for (int j = 0; j < i; ++j) {
        if (!(local_nonzero<TB>() >> (8 * i + j) & 1)) continue;
        const double c = sz.e[i][j];
#pragma unroll
        for (int v = 0; v < 3; ++v) cur[v] = fma(c, sL[j][v][threadIdx.x], cur[v]);
      }
    } else {
#pragma unroll
      for (int j = 0; j < S; ++j)
        if (j < i && TB::a(i, j) != 0.0) {
#pragma unroll
          for (int v = 0; v < 3; ++v) cur[v] = fma(sz.e[i][j], rL[j][v], cur[v]);
        }
    }
    if constexpr (IMEX) {
#pragma unroll
      for (int j = 0; j < S; ++j)
        if (j < i && TB::ai(i, j) != 0.0) {
          cur[1] = fma(sz.im[i][j], rS[j][0], cur[1]);
          cur[2] = fma(sz.im[i][j], rS[j][1], cur[2]);
        }
      // Chezy friction s = -C_f |m| m / h^2 on (hu, hv), point-implicit with
      // h fixed: m is parallel to the stage sum r and
      // |m| + dt a_ii C_f |m|^2 / h^2 = |r|, so
      // m = r 2 / (1 + sqrt(1 + 4 dt a_ii C_f |r| / h^2))
      static_assert(TB::ai(0, 0) == TB::ai(S - 1, S - 1), "one diagonal coefficient");
      const double gcf = sz.im[0][0] * T.src_coef;
      const double ih = drcp(cur[0]);
      const double ih2 = ih * ih;
      const double rx = cur[1], ry = cur[2];
      double nm = dsqrt_pos(fma(rx, rx, ry * ry));
      const double qf = dsqrt_pos(fma(4.0 * gcf * ih2, nm, 1.0));
      const double f = 2.0 * drcp(1.0 + qf);
      cur[1] = rx * f;
      cur[2] = ry * f;
      nm *= f;
      const double c = -(T.src_coef * ih2) * nm;
      rS[i][0] = c * cur[1];
      rS[i][1] = c * cur[2];
      // the implicit weights b_i equal the explicit ones b~_i
      const double wd = local_weight_fp<TB>(i);
      if (wd != 0.0) {
        Sb[0] = fma(wd, rS[i][0], Sb[0]);
        Sb[1] = fma(wd, rS[i][1], Sb[1]);
      }
    }
    if constexpr (STAGES) {
      // recorded step: the adjoint reads the stage values instead of
      // recomputing them (stage 0 is u^n itself)
      if (i > 0 && active) {
        const int64_t Nr = L.stage_rows * L.Ex, gr = ge - L.stage_row0 * L.Ex;
#pragma unroll
        for (int v = 0; v < 3; ++v)
          L.stages[(((int64_t)(i - 1) * 3 + v) * Nr + gr) * nn + node] = cur[v];
      }
    }
    // (the first stage of SSP3-IMEX(4,3,3) has neither weight nor successor)
    if (IMEX && i == 0) continue;
    const int wi = local_weight<TB>(i);
    // every stage but the last feeds a later one; the last one's fluxes enter
    // the averages only
    const bool need_op = i < S - 1 && !(PRE == 2 && i == 0);
    // the exchange fields at this node: the state and the fluxes
    const FxSig sh = fx_sig(cur[0]), sx = fx_sig(cur[1]), sy = fx_sig(cur[2]);
    // one exponent per element and field: the first stage's largest
    // magnitudes with headroom, raised if a later stage exceeds them.
    // (sync_or is also the barrier after the last reads of X.)
    const int lx = fx_log(cur[1]), ly = fx_log(cur[2]), lhg = fx_log(T.half_gravity);
    // (Only the nodes that exceed them enter smag: what an element's exponents
    // become must not depend on the elements it shares a barrier with.)
    const bool over = lane_ok && fx_over<!WB>(cur[0], lx, ly, lhg, E);
    if (sync_or(over)) {
      if (over) {
        int mag[kLocalGroups];
        mag[0] = fx_mag(cur[0]);
        mag[1] = fx_mag(cur[1]);
        mag[2] = fx_mag(cur[2]);
        mag[3] = fx_flux_mag<!WB>(cur[0], lx, lx, lhg);
        mag[4] = fx_flux_mag<false>(cur[0], lx, ly, lhg);
        mag[5] = fx_flux_mag<!WB>(cur[0], ly, ly, lhg);
        if (IMEX) {
          // the traces of u^n, no stage value here, share the exponents
          mag[0] = max(mag[0], fx_mag(u0[0]));
          mag[1] = max(mag[1], fx_mag(u0[1]));
          mag[2] = max(mag[2], fx_mag(u0[2]));
        }
#pragma unroll
        for (int k = k0; k < kLocalGroups; ++k) atomicMax(&smag[le][k], mag[k]);
      }
      sync();
#pragma unroll
      for (int k = k0; k < kLocalGroups; ++k) {
        const int e = fx_exp(smag[le][k]);
        const int d = e > E[k] ? e + kHeadroom - E[k] : 0;
        E[k] += d;
        if (k > 0 || FIX_H) fx_rescale<WIDE>(A[k], B[k], d);
      }
    }
    long long f[6];
    {
      const unsigned long long R = recip_bits((unsigned)__double2hiint(cur[0]),
                                              (unsigned)__double2loint(cur[0]));
      const unsigned long long vx = fx_velocity(R, sx), vy = fx_velocity(R, sy);
      if (WB) f[0] = fx_from<FB>(sh, E[0]);
      f[1] = fx_from<FB>(sx, E[1]);
      f[2] = fx_from<FB>(sy, E[2]);
      f[3] = fx_momentum_flux<FB>(sx, vx, sx, sh, E[3]);
      f[4] = fx_momentum_flux<FB>(sx, vy, sy, sh, E[4]);
      f[5] = fx_momentum_flux<FB>(sy, vy, sy, sh, E[5]);
      if (!WB) {
        const FxSig hg = fx_sig(T.half_gravity);
        f[3] += fx_pressure<FB>(sh, hg, E[3]);
        f[5] += fx_pressure<FB>(sh, hg, E[5]);
      }
    }
#pragma unroll
    for (int k = k0; k < 6; ++k) {
      const Fx x = fx_split(f[k]);
      if (k > 0 || FIX_H) fx_accumulate<WIDE>(A[k], B[k], f[k], x, wi);
      if (lane_ok) X[k][q][p] = x;
    }
    if (need_op || WB) {
      sync();
      double ncx = 0.0, ncy = 0.0;   // well-balanced: h g (h + b)_x, _y
      if constexpr (WB) {
        const int z = fx_zero(E[0]);
        const double hx = fx_to(row_x(0), E[0] + T.fx.kDx - FB, z);
        const double hy = fx_to(row_y(0), E[0] + T.fx.kDy - FB, z);
        ncx = cur[0] * fma(T.gravity, hx, gbx);
        ncy = cur[0] * fma(T.gravity, hy, gby);
        const double wd = local_weight_fp<TB>(i);
        P1 = fma(wd, ncx, P1);
        P2 = fma(wd, ncy, P2);
      }
      if (need_op) {
        Lp[0] = contract(1, 2, 0);
        const double l1 = contract(3, 4, 0), l2 = contract(4, 5, 0);
        Lp[1] = WB ? l1 + ncx : fma(cur[0], gbx, l1);
        Lp[2] = WB ? l2 + ncy : fma(cur[0], gby, l2);
      }
    }
    if constexpr (PRE == 1) {
      if (active) {
#pragma unroll
        for (int v = 0; v < 3; ++v) L.w[(v * Ne + ge) * nn + node] = Lp[v];
      }
      return;
    }
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      if (UNROLL) rL[i][v] = Lp[v];
      if (SHARED && i < S - 1) sL[i][v][threadIdx.x] = Lp[v];
    }
  }

  // ---- W = u^n - dt (dloc F + Bloc) [+ dt S]  (or the residual's part) -------
  // The derivative of the time averages is taken once: dloc F = D (sum_j b_j
  // f_j), Bloc = g b_x (sum_j b_j h_j) (the well-balanced product is
  // accumulated stage by stage).  A, P and Sb hold time averages divided by
  // b_ref; the sums are scaled back to FB bits for the contractions.
#pragma unroll
  for (int k = FIX_H ? 0 : 1; k < 6; ++k) A[k] = fx_average<WIDE, kSumShift>(A[k], B[k]);
  const double du = uh;
  uh = fma((double)TB::weight_sum(), u0[0], du);
  if constexpr (!GLL && !FIX_H) {
    // the exponent of the traces of h: u^n and its average's increment (in sum
    // units)
    const int mu = fx_mag(du);
    const int m = max(fx_mag(u0[0]), mu >= 0x7ff00000 ? mu : mu - (kSumShift << 20));
    if (lane_ok) atomicMax(&smag[le][0], m);
  }
  sync();
  if (!GLL && !FIX_H) E[0] = fx_exp(smag[le][0]);
  if (lane_ok) {
    X[0][q][p] = FIX_H ? fx_split(A[0])
                 : GLL ? Fx{__double2hiint(uh), __double2loint(uh)}
                       : fx_split(fx_increment<WIDE, kSumShift, FB>(u0[0], TB::weight_sum(), du,
                                                                    E[0]));
#pragma unroll
    for (int k = 1; k < 6; ++k) X[k][q][p] = fx_split(A[k]);
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      if constexpr (GLL)
        X[6 + v][q][p] = Fx{__double2hiint(u0[v]), __double2loint(u0[v])};
      else
        X[6 + v][q][p] = fx_split(fx_from<FB>(u0[v], E[v]));
    }
  }
  sync();
  {
    constexpr double b0 = TB::bref();
    const double dtb0 = sz.dtb;
    double V[3];
    V[0] = contract(1, 2, kSumShift);
    V[1] = contract(3, 4, kSumShift);
    V[2] = contract(4, 5, kSumShift);
    if constexpr (WB) {
      V[1] += P1;
      V[2] += P2;
    } else {
      V[1] = fma(uh, gbx, V[1]);
      V[2] = fma(uh, gby, V[2]);
    }
    // (a record alone, without a step, has no use for W: its place may hold the
    // stage values)
    if (active && !(STAGES && RES)) {
#pragma unroll
      for (int v = 0; v < 3; ++v) {
        double o = RES ? -b0 * V[v] : fma(-dtb0, V[v], u0[v]);
        if (IMEX && v > 0) o = fma(RES ? b0 : dtb0, Sb[v - 1], o);
        L.w[(v * Ne + ge) * nn + node] = o;
      }
    }
  }

  chain_end();
  // ---- face traces: 4 n face nodes per element (side 0 / 1 of the x faces,
  //      then of the y faces), all fields of a face node by one thread --------
  if (active) {
    const int64_t tstride = Ne * n;              // one (field, side) plane of the x traces
    const int64_t plane = L.Ex * n;              // one field of a row's y traces
    const int64_t row = ge / L.Ex + 1, col = ge - (row - 1) * L.Ex;   // y-trace buffer row
#pragma unroll
    for (int j0 = 0; j0 < 4 * n; j0 += nn) {
      const int job = j0 + node;
      if (4 * n % nn != 0 && job >= 4 * n) break;
      const int dir = job / (2 * n), side = job / n & 1, r = job % n;
      // the nodes next to the face line: base + j step
      const Fx* line = &X[0][dir ? 0 : r][dir ? r : 0];
      const int step = dir ? n : 1;
      int ch[n], cl[n];
#pragma unroll
      for (int j = 0; j < n; ++j) {
        ch[j] = side ? T.fx.l1_hi[j] : T.fx.l0_hi[j];
        cl[j] = side ? T.fx.l1_lo[j] : T.fx.l0_lo[j];
      }
      double* out = dir ? L.try_ + (row * 2 + side) * kTrFields * plane + col * n + r
                        : L.trx + side * tstride + ge * n + r;
      const int64_t ostep = dir ? plane : 2 * tstride;
      // in a periodic mesh the bottom row's bottom side is also the halo
      // above the top row, and vice versa
      const bool wrap = dir && L.periodic_y && row == (side ? L.Ey : 1);
      double* halo = L.try_ + (side ? 1 : (L.Ey + 1) * 2) * kTrFields * plane + col * n + r;
#pragma unroll
      for (int fi = 0; fi < kTrFields; ++fi) {
        const int k = fi < 3 ? fi : fi < 5 ? fi + dir : fi == 5 ? 6 : 7 + dir;
        // (in y the fields after the first three are the next ones)
        const int ek = fi < 3 ? E[fi] : fi == 3 ? (dir ? E[4] : E[3])
                     : fi == 4 ? (dir ? E[5] : E[4]) : fi == 5 ? E[0] : (dir ? E[2] : E[1]);
        const Fx* x = line + k * nn;
        double t;
        if constexpr (GLL) {
          const Fx v = x[side ? N * step : 0];
          if (fi == 0 || fi >= 5)
            t = __hiloint2double(v.hi, v.lo);
          else
            t = fx_to(((long long)v.hi << 30) + v.lo, ek + 63 - FB + kSumShift, fx_zero(ek));
        } else {
          FxAcc a;
          fx_mul(a, x[0], ch[0], cl[0]);
#pragma unroll
          for (int j = 1; j < n; ++j) fx_mad(a, x[j * step], ch[j], cl[j]);
          t = fx_to(fx_sum(a), ek + T.fx.kL - FB + (fi < 5 ? kSumShift : 0), fx_zero(ek));
        }
        out[fi * ostep] = t;
        if (wrap) halo[fi * plane] = t;
      }
    }
  }
  // ---- limiter: first-order update without the element-face terms and the
  //      face data of the first-order face fluxes (limit_2d.cuh) -------------
  if constexpr (LIMIT) {
    static_assert(!RES, "the limiter needs a step");
    sync();
    limit_local_2d<N, GLL, WB>(L, u0, &sm[le * ES], node, lane_ok, active, ge, sz.dt, sync);
  }
}

template <int N, bool GLL, bool IMEX, bool WB, bool LIMIT = false>
int launch_local_t(const Launch2D& L, cudaStream_t s) {
  constexpr int per_block = local_elements<N + 1>();
  if (L.row_begin < 0 || L.row_end <= L.row_begin || L.row_end > L.Ey)
    return (int)cudaErrorInvalidValue;
  const int64_t blocks = ((L.row_end - L.row_begin) * L.Ex + per_block - 1) / per_block;
  if (blocks > 0x7fffffff) return (int)cudaErrorInvalidConfiguration;
  const dim3 grid((unsigned)blocks);
  if constexpr (LIMIT)
    return launch_chained(k_local_2d<N, GLL, false, IMEX, WB, true>, grid, kBlockLocal, s, L);
  else if (L.ctl.residual)
    return launch_chained(k_local_2d<N, GLL, true, IMEX, WB>, grid, kBlockLocal, s, L);
  else
    return launch_chained(k_local_2d<N, GLL, false, IMEX, WB>, grid, kBlockLocal, s, L);
}

template <bool IMEX, bool WB, bool LIMIT = false>
int launch_local_dispatch(const Launch2D& L, cudaStream_t s) {
  switch (L.N * 2 + (L.gll ? 1 : 0)) {
    case 2: return launch_local_t<1, false, IMEX, WB, LIMIT>(L, s);
    case 3: return launch_local_t<1, true, IMEX, WB, LIMIT>(L, s);
    case 4: return launch_local_t<2, false, IMEX, WB, LIMIT>(L, s);
    case 5: return launch_local_t<2, true, IMEX, WB, LIMIT>(L, s);
    case 6: return launch_local_t<3, false, IMEX, WB, LIMIT>(L, s);
    case 7: return launch_local_t<3, true, IMEX, WB, LIMIT>(L, s);
    case 8: return launch_local_t<4, false, IMEX, WB, LIMIT>(L, s);
    case 9: return launch_local_t<4, true, IMEX, WB, LIMIT>(L, s);
  }
  return (int)cudaErrorInvalidValue;
}

}  // namespace
}  // namespace crkfr
