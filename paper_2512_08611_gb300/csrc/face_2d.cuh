// Face kernel of the 2D shallow-water cRK-FR step (sm_103a, FP64), shared by
// kernels_2d.cu (standard form) and kernels_wb.cu (well-balanced form): the
// only inter-element coupling of a step.  Once per face node the
// time-averaged Rusanov flux (Eq. numflux.cons) with the wave-speed estimate
// of the full system at u^n, the frozen non-conservative fluctuation
// B(w^{n,+-})(W^num - W^{+-}) (Eqs. good.numflux.non.cons, total.F.non.cons),
// and the FR corrections g_L', g_R' (App. B, Eq. correction.identities)
// applied along the rows and columns of the element, added to
// W = u^n - dt (dloc F + Bloc) [+ dt S] written by the local kernel.
//
// With the subcell blending limiter (LIMIT; the tensor-product extension of
// Sec. 4) each face node's high-order flux is blended with the first-order
// flux of the nodal values next to the face (Eq. Fblend, the mean of the two
// elements' coefficients), limited by Algorithm 1 (h > 0) on the doubled-dt
// one-direction first-order updates of its two nodes, and used both in the
// corrections and in the first-order subcell update of the element; the
// update is blended (Eq. blended.scheme), the source of the first-order
// update taken point-implicitly (IMEX), and Algorithm 2 (h > 0) applied per
// element.
#pragma once

#include <cuda_runtime.h>

#include "device_common.cuh"
#include "fixed_point.cuh"
#include "launch.h"
#include "local_2d.cuh"

namespace crkfr {
namespace {

constexpr int kBlock2D = 256;
constexpr int kWarps2D = kBlock2D / 32;

// a face term converted in place
__device__ __forceinline__ Fx fx_at(const double* t) { return *reinterpret_cast<const Fx*>(t); }

// Doubled face terms of both sides of one face node, T'^- = 2 (F^num,- - F^tot,-)
// and T'^+ = 2 (F^num,+ - F^tot,+), from the two sides' traces.
// Trace fields: 0..2 U, 3..4 time-averaged normal fluxes of the two momenta,
// 5 h^n, 6 normal momentum at t^n.  `nv` (1 or 2) is the index of the normal
// momentum, whose equation carries the fluctuation; gdb = (g / b_ref)(b+ - b-).
// The well-balanced form dissipates and fluctuates eta = h + b instead of h:
// g (eta+ - eta-) in the units of the time averages is g dU_h + gdb.
template <bool WB>
__device__ __forceinline__ void face_terms(const double* tm, const double* tp, int nv, double gdb,
                                           double g, double inv_g, double sg, double Tm[3],
                                           double Tp[3]) {
  const double lam = max_nonneg(swe_speed(tm[5], tm[6], sg), swe_speed(tp[5], tp[6], sg));
  // time-averaged normal flux of h is the time-averaged normal momentum
  const double dF[3] = {tp[nv] - tm[nv], tp[3] - tm[3], tp[4] - tm[4]};
  double dU[3] = {tp[0] - tm[0], tp[1] - tm[1], tp[2] - tm[2]};
  if (WB) {
    gdb = fma(g, dU[0], gdb);
    dU[0] = gdb * inv_g;
  }
#pragma unroll
  for (int v = 0; v < 3; ++v) {
    Tm[v] = fma(-lam, dU[v], dF[v]);
    Tp[v] = -fma(lam, dU[v], dF[v]);
  }
  Tm[nv] = fma(tm[5], gdb, Tm[nv]);
  Tp[nv] = fma(-tp[5], gdb, Tp[nv]);
}

// Limited face fluxes of one face node in direction DIR (0: x, 1: y), all in
// the physical units of the first-order scheme, doubled, except the traces tm,
// tp (time averages divided by b_ref, as above).  lm, lp: limiter face data of
// the minus and plus sides (nodal u next to the face, nodal c, the doubled inner
// first-order flux of that node on its far side, trace of c).  af: blending
// coefficient of the face; c1m, c1p: dt / (w dx) of the two nodes (the doubled
// step of Algorithm 1's one-direction updates times the half of the doubled
// fluxes).  Returns the face terms F^+- / b_ref - F^tot,+- of the corrections (not
// doubled: that is one in their fixed point's exponent) and the doubled fluxes
// 2 F^-, 2 F^+ of the first-order update.
template <int DIR, bool WB>
__device__ __forceinline__ void face_limited(const double* tm, const double* tp, const double* lm,
                                             const double* lp, double af, double c1m, double c1p,
                                             const Tables& T, double Tm[3], double Tp[3],
                                             double Fm[3], double Fp[3]) {
  constexpr int nv = 1 + DIR;
  const double g = T.gravity, ib0 = T.inv_b0;
  const double cm = lm[7], cp = lp[7];
  // high-order fluxes 2 F^num,+- and totals F^tot,+- (Eqs. numflux.cons,
  // good.numflux.non.cons, total.F.non.cons), in the units of the traces
  const double lam = max_nonneg(swe_speed(tm[5], tm[6], T.sqrt_gravity),
                                swe_speed(tp[5], tp[6], T.sqrt_gravity));
  const double dUh = WB ? (tp[0] + cp * ib0) - (tm[0] + cm * ib0) : tp[0] - tm[0];
  double FHm[3], FHp[3], FTm[3], FTp[3];
  FHm[0] = fma(-lam, dUh, tm[nv] + tp[nv]);
  FHm[1] = fma(-lam, tp[1] - tm[1], tm[3] + tp[3]);
  FHm[2] = fma(-lam, tp[2] - tm[2], tm[4] + tp[4]);
  const double cn = (cm + cp) * ib0;
  const double Wn = WB ? (tm[0] + tp[0]) + cn : cn;
  const double Wm = WB ? tm[0] + cm * ib0 : cm * ib0;
  const double Wp = WB ? tp[0] + cp * ib0 : cp * ib0;
  const double ghm = g * tm[5], ghp = g * tp[5];
#pragma unroll
  for (int v = 0; v < 3; ++v) FHp[v] = FHm[v];
  FHm[nv] = fma(ghm, Wn, FHm[nv]);
  FHp[nv] = fma(ghp, Wn, FHp[nv]);
  FTm[0] = tm[nv];
  FTm[1] = tm[3];
  FTm[2] = tm[4];
  FTp[0] = tp[nv];
  FTp[1] = tp[3];
  FTp[2] = tp[4];
  FTm[nv] = fma(ghm, Wm, FTm[nv]);
  FTp[nv] = fma(ghp, Wp, FTp[nv]);
  // first-order face fluxes and Eq. Fblend
  double fLm[3], fLp[3];
  lo_flux_2d<DIR, WB>(lm, lp, lm[3], lp[3], g, fLm, fLp);
  // (af = 0, both elements unlimited, and theta = 1 below are the common
  // cases: there the blends reduce to their first terms and are skipped)
  const double b0 = T.b0;
  if (af != 0.0) {
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      Fm[v] = (1.0 - af) * (b0 * FHm[v]) + af * fLm[v];
      Fp[v] = (1.0 - af) * (b0 * FHp[v]) + af * fLp[v];
    }
  } else {
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      Fm[v] = b0 * FHm[v];
      Fp[v] = b0 * FHp[v];
    }
  }
  // Algorithm 1 (h > 0): the doubled-dt one-direction first-order updates
  // of the plus side's node 0 and the minus side's node N, in FP64 only where
  // FP32 does not show theta = 1
  if (!(theta_one(lp[0], c1p, lp[4], fLp[0], Fp[0]) &&
        theta_one(lm[0], -c1m, lm[4], fLm[0], Fm[0]))) {
    const double low0 = lp[0] - c1p * (lp[4] - fLp[0]);
    const double lowN = lm[0] - c1m * (fLm[0] - lm[4]);
    const double t0 = lp[0] - c1p * (lp[4] - Fp[0]);
    const double tN = lm[0] - c1m * (Fm[0] - lm[4]);
    const double th = fmin(theta_lin(0.1 * low0, low0, t0), theta_lin(0.1 * lowN, lowN, tN));
    if (th < 1.0) {
#pragma unroll
      for (int v = 0; v < 3; ++v) {
        Fm[v] = th * Fm[v] + (1.0 - th) * fLm[v];
        Fp[v] = th * Fp[v] + (1.0 - th) * fLp[v];
      }
    }
  }
  const double hib0 = 0.5 * ib0;
#pragma unroll
  for (int v = 0; v < 3; ++v) {
    Tm[v] = fma(Fm[v], hib0, -FTm[v]);
    Tp[v] = fma(Fp[v], hib0, -FTp[v]);
  }
}

// Tile rows (warps) of the face kernel: 8, or 4 limited (its face data takes
// twice the shared memory); 2 on meshes whose tiles of that height would leave
// SMs without a block, where the step is latency and an SM sub-partition runs
// its warps' FP64 instructions one after the other (small: 65 x 47 elements at
// N = 2 have 42 tiles of 8 rows, 168 of 2).
template <int N, bool LIMIT, bool SMALL>
struct FaceShape {
  static constexpr int TY = SMALL ? 2 : LIMIT ? 4 : kWarps2D;
  static constexpr int block = TY * 32;
  // resident blocks per SM the register allocation must allow (the plain
  // kernel: 40 warps, 32 at N = 4, to hide the barriers and the shared-memory
  // latency of the face terms)
  static constexpr int min_blocks = LIMIT ? 1 : SMALL ? 8 : N >= 4 ? 4 : 5;
};

// Face kernel on tiles of TY x TX elements (one tile row per warp).  512 x 512 at
// N = 3: 175 us, bound by the FP64 pipe (58 % busy), issue slots (0.52) and DRAM
// (38 % of its peak) together; 169 us with one exponent for both momenta and for
// W, which cut the smaller values of the state.
// Phase 1 solves every face node of the tile exactly once in a flat loop over
// the block (warps with no face left issue nothing, so only the last, partial
// warp of the loop pays for idle lanes) and keeps both sides' terms in shared
// memory; phase 2 applies them along the rows and columns of each element.

template <int N, bool GLL, bool RES, bool WB, bool LIMIT = false, bool IMEX = false,
          bool SMALL = false>
__global__ void __launch_bounds__(FaceShape<N, LIMIT, SMALL>::block,
                                  FaceShape<N, LIMIT, SMALL>::min_blocks)
    k_face_2d(const Launch2D L) {
  static_assert(!(LIMIT && RES), "the limiter needs a step");
  constexpr int n = N + 1;
  constexpr int nn = n * n;
  constexpr int TX = 32 / n;        // elements per tile row (= per warp)
  constexpr int TY = FaceShape<N, LIMIT, SMALL>::TY;
  constexpr int BT = FaceShape<N, LIMIT, SMALL>::block;
  constexpr int NX = TY * (TX + 1) * n;
  constexpr int NY = (TY + 1) * TX * n;
  // x faces to whole warps, so that no warp takes both branches of the loops
  // below (N = 3 limited: 10 passes of a warp instead of 11)
  constexpr int NXW = (NX + 31) / 32 * 32;
  constexpr int LY = LIMIT ? TY : 1, LX = LIMIT ? TX : 1;
  const Tables& T = L.tab;
  // x faces: [row][face k between elements k-1 and k][node]; y faces:
  // [face k between rows k-1 and k][column][node]; both sides, 3 variables
  // (the variable outermost: the lanes of a warp touch consecutive doubles)
  __shared__ double sxm[3][TY][TX + 1][n], sxp[3][TY][TX + 1][n];
  __shared__ double sym[3][TY + 1][TX][n], syp[3][TY + 1][TX][n];
  // limiter: the doubled face fluxes 2 F^-, 2 F^+ of the first-order update
  __shared__ double fxm[3][LY][LX + 1][n], fxp[3][LY][LX + 1][n];
  __shared__ double fym[3][LY + 1][LX][n], fyp[3][LY + 1][LX][n];

  const int64_t Ex = L.Ex, Ey = L.Ey, Ne = Ex * Ey, ts = Ne * n;
  const int64_t ex0 = (int64_t)blockIdx.x * TX, ey0 = L.row_begin + (int64_t)blockIdx.y * TY;
  chain_begin();
  // the traces hold time averages divided by b_0: so do the face terms
  const double dtp = RES ? 1.0 : L.st->dt_cur;
  // correction tables times -dt in fixed point (FB bits below 2^(ec - 1022), ec
  // of the x and of the y tables), written here, read after the barriers
  // between the phases
  constexpr int FB = 59;
  __shared__ Fx cor[4][n];
  __shared__ int cor_e[2];
  // largest magnitudes of each variable's terms on the x and the y faces of an
  // element
  __shared__ int emag[2][3][TY][TX];
  for (int k = threadIdx.x; k < 6 * TY * TX; k += BT) (&emag[0][0][0][0])[k] = 0;
  if (threadIdx.x < 4 * n) {
    const double dt = dtp * T.b0;
    const int t = threadIdx.x / n, p = threadIdx.x - t * n;
    const double g = t == 0 ? T.gRx[p] : t == 1 ? T.gLx[p] : t == 2 ? T.gRy[p] : T.gLy[p];
    const int ec = fx_exp(fx_mag(dt) + (T.fx.kG[t >> 1] << 20));
    cor[t][p] = fx_split(fx_from<FB>(-dt * g, ec));
    if (p == 0 && (t & 1) == 0) cor_e[t >> 1] = ec;
  }
  // limiter: dt / (w dx) of the nodes next to a face (0 and N), x and y
  __shared__ double cl[2][2];
  if (LIMIT && threadIdx.x < 4) {
    const int d = threadIdx.x >> 1, k = threadIdx.x & 1;
    cl[d][k] = dtp * (d ? T.inv_dy : T.inv_dx) * T.inv_w[k ? N : 0];
  }
  __syncthreads();
  // the terms of both sides of a face: to shared memory, their magnitudes to
  // the elements they belong to (minus side: r0, c0; plus side: r1, c1)
  auto keep = [&](int d, double* tm, double* tp, int vs, const double* Tm, const double* Tp,
                  int r0, int c0, int r1, int c1) {
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      tm[v * vs] = Tm[v];
      tp[v * vs] = Tp[v];
    }
    if (r0 >= 0 && c0 >= 0) {
#pragma unroll
      for (int v = 0; v < 3; ++v) atomicMax(&emag[d][v][r0][c0], fx_mag(Tm[v]));
    }
    if (r1 < TY && c1 < TX) {
#pragma unroll
      for (int v = 0; v < 3; ++v) atomicMax(&emag[d][v][r1][c1], fx_mag(Tp[v]));
    }
  };

  // ---- phase 1: every face node of the tile once --------------------------
  for (int f = threadIdx.x; f < NXW + NY; f += BT) {
    double a[kTrFields], b[kTrFields], Tm[3], Tp[3];
    if (f < NXW) {
      if (NXW != NX && f >= NX) continue;
      const int q = f % n, k = (f / n) % (TX + 1), r = f / (n * (TX + 1));
      const int64_t ey = ey0 + r;
      if (ey >= Ey || (k > 0 && ex0 + k - 1 >= Ex)) continue;
      const int64_t em = ey * Ex + (ex0 + k - 1 + Ex) % Ex;
      const int64_t ep = ey * Ex + (ex0 + k) % Ex;
#pragma unroll
      for (int fi = 0; fi < kTrFields; ++fi) {
        a[fi] = L.trx[(2 * fi + 1) * ts + em * n + q];
        b[fi] = L.trx[(2 * fi + 0) * ts + ep * n + q];
      }
      if constexpr (LIMIT) {
        double lm[kLimFields], lp[kLimFields], Fm[3], Fp[3];
#pragma unroll
        for (int fi = 0; fi < kLimFields; ++fi) {
          lm[fi] = L.lim.lx[(2 * fi + 1) * ts + em * n + q];
          lp[fi] = L.lim.lx[(2 * fi + 0) * ts + ep * n + q];
        }
        const double af = 0.5 * (L.lim.alpha[em] + L.lim.alpha[ep]);
        face_limited<0, WB>(a, b, lm, lp, af, cl[0][1], cl[0][0], T, Tm, Tp, Fm, Fp);
#pragma unroll
        for (int v = 0; v < 3; ++v) {
          fxm[v][r][k][q] = Fm[v];
          fxp[v][r][k][q] = Fp[v];
        }
      } else {
        face_terms<WB>(a, b, 1, L.sface[ep * n + q], T.gravity, T.inv_gravity, T.sqrt_gravity,
                       Tm, Tp);
      }
      keep(0, &sxm[0][r][k][q], &sxp[0][r][k][q], TY * (TX + 1) * n, Tm, Tp, r, k - 1, r, k);
    } else {
      const int g = f - NXW;
      const int p = g % n, c = (g / n) % TX, k = g / (n * TX);
      const int64_t ex = ex0 + c;
      if (ex >= Ex || (k > 0 && ey0 + k - 1 >= Ey)) continue;
      // face below element row ey0+k: minus side = buffer row ey0+k (top side),
      // plus side = buffer row ey0+k+1 (bottom side); rows 0 and Ey+1 are halos
      const int64_t plane = Ex * n;
      const int64_t rm = ey0 + k, rp = ey0 + k + 1;
#pragma unroll
      for (int fi = 0; fi < kTrFields; ++fi) {
        a[fi] = L.try_[((rm * 2 + 1) * kTrFields + fi) * plane + ex * n + p];
        b[fi] = L.try_[((rp * 2 + 0) * kTrFields + fi) * plane + ex * n + p];
      }
      if constexpr (LIMIT) {
        double lm[kLimFields], lp[kLimFields], Fm[3], Fp[3];
#pragma unroll
        for (int fi = 0; fi < kLimFields; ++fi) {
          lm[fi] = L.lim.ly[((rm * 2 + 1) * kLimFields + fi) * plane + ex * n + p];
          lp[fi] = L.lim.ly[((rp * 2 + 0) * kLimFields + fi) * plane + ex * n + p];
        }
        // the elements below and above the face: periodic in y, or on a slab
        // of a larger mesh the rows -1 and Ey from the neighbouring slabs
        double am, ap;
        if (L.lim.alpha_halo) {
          const int64_t eym = ey0 + k - 1, eyp = ey0 + k;
          am = eym < 0 ? L.lim.alpha_halo[ex] : L.lim.alpha[eym * Ex + ex];
          ap = eyp >= Ey ? L.lim.alpha_halo[Ex + ex] : L.lim.alpha[eyp * Ex + ex];
        } else {
          const int64_t eym = (ey0 + k - 1 + Ey) % Ey, eyp = (ey0 + k) % Ey;
          am = L.lim.alpha[eym * Ex + ex];
          ap = L.lim.alpha[eyp * Ex + ex];
        }
        const double af = 0.5 * (am + ap);
        face_limited<1, WB>(a, b, lm, lp, af, cl[1][1], cl[1][0], T, Tm, Tp, Fm, Fp);
#pragma unroll
        for (int v = 0; v < 3; ++v) {
          fym[v][k][c][p] = Fm[v];
          fyp[v][k][c][p] = Fp[v];
        }
      } else {
        face_terms<WB>(a, b, 2, L.sface[Ne * n + (ey0 + k) * plane + ex * n + p], T.gravity,
                       T.inv_gravity, T.sqrt_gravity, Tm, Tp);
      }
      keep(1, &sym[0][k][c][p], &syp[0][k][c][p], (TY + 1) * TX * n, Tm, Tp, k - 1, c, k, c);
    }
  }
  __syncthreads();

  // ---- the face terms in fixed point, in place: x and y terms of a variable
  //      so that their products with the correction tables have one unit per
  //      element, 2^(unit - 1022 - FB) ------------------------------------------
  auto unit = [&](int v, int r, int c, int& zero) -> int {
    const int x = fx_exp(emag[0][v][r][c]), y = fx_exp(emag[1][v][r][c]);
    zero = fx_zero(max(x, y));
    return max(x + cor_e[0], y + cor_e[1]);
  };
  for (int f = threadIdx.x; f < NXW + NY; f += BT) {
    double *tm, *tp;
    int vs, r0, c0, r1, c1;
    if (f < NXW) {
      if (NXW != NX && f >= NX) continue;
      const int q = f % n, k = (f / n) % (TX + 1), r = f / (n * (TX + 1));
      if (ey0 + r >= Ey || (k > 0 && ex0 + k - 1 >= Ex)) continue;
      tm = &sxm[0][r][k][q];
      tp = &sxp[0][r][k][q];
      vs = TY * (TX + 1) * n;
      r0 = r1 = r;
      c0 = k - 1;
      c1 = k;
    } else {
      const int g = f - NXW;
      const int p = g % n, c = (g / n) % TX, k = g / (n * TX);
      if (ex0 + c >= Ex || (k > 0 && ey0 + k - 1 >= Ey)) continue;
      tm = &sym[0][k][c][p];
      tp = &syp[0][k][c][p];
      vs = (TY + 1) * TX * n;
      r0 = k - 1;
      r1 = k;
      c0 = c1 = c;
    }
    auto convert = [&](double* t, int d, int r, int c) {
#pragma unroll
      for (int v = 0; v < 3; ++v) {
        int zero;
        *reinterpret_cast<Fx*>(t + v * vs) =
            fx_split(fx_from<FB>(t[v * vs], unit(v, r, c, zero) - cor_e[d]));
      }
    };
    if (r0 >= 0 && c0 >= 0) convert(tm, f >= NXW, r0, c0);
    if (r1 < TY && c1 < TX) convert(tp, f >= NXW, r1, c1);
  }
  __syncthreads();

  // ---- phase 2: corrections and update, one element row per thread -------
  const int lane = threadIdx.x & 31, r = threadIdx.x >> 5;
  const int c = lane / n, q = lane - c * n;
  const bool lane_ok = c < TX;
  const int cc = lane_ok ? c : 0;
  const int64_t ey = ey0 + r, ex = ex0 + cc;
  const bool active = lane_ok && ey < Ey && ex < Ex;
  const int64_t ge = active ? ey * Ex + ex : 0;
  double out[3][n];
  // largest value over the n rows of the element
  auto element_max = [&](int v) -> int {
    int m = v;
    if constexpr ((n & (n - 1)) == 0) {
#pragma unroll
      for (int o = 1; o < n; o <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    } else {
#pragma unroll
      for (int j = 1; j < n; ++j) {
        const int src = c * n + ((q + j) % n);
        m = max(m, __shfl_sync(0xffffffffu, v, src < 32 ? src : lane));
      }
    }
    return m;
  };
  // u^{n+1} = W + corrections: their sum in fixed point, W added with an
  // exponent of its own (so that a step of zero size leaves it as it is, and
  // values far below the element's largest keep their bits), rounded once.
  // Limited terms are not doubled.
#pragma unroll
  for (int v = 0; v < 3; ++v) {
    int zero;
    const int et = unit(v, r, cc, zero) - 1021 + (LIMIT ? 1 : 0);
    const Fx tr = fx_at(&sxm[v][r][cc + 1][q]), tl = fx_at(&sxp[v][r][cc][q]);
    const Fx c2 = cor[2][q], c3 = cor[3][q];
#pragma unroll
    for (int p = 0; p < n; ++p) {
      // (GLL: corrections at the end nodes only; in y by zero coefficients)
      FxAcc a;
      fx_mul(a, fx_at(&sym[v][r + 1][cc][p]), c2.hi, c2.lo);
      fx_mad(a, fx_at(&syp[v][r][cc][p]), c3.hi, c3.lo);
      if (!GLL || p == N) fx_mad(a, tr, cor[0][p].hi, cor[0][p].lo);
      if (!GLL || p == 0) fx_mad(a, tl, cor[1][p].hi, cor[1][p].lo);
      const double w = L.w[(v * Ne + ge) * nn + q * n + p];
      const int e = max(fx_exp(fx_mag(w)), et);
      out[v][p] = fx_to(fx_from<FB>(w, e) + fx_sar(fx_sum(a), e - et), e + 63 - FB,
                        fx_zero(e) | zero);
    }
  }
  if constexpr (LIMIT) {
    // first-order subcell update: the local kernel's part plus the
    // element-face fluxes of the face nodes (Eq. low.order.update), the
    // source point-implicitly; Eq. blended.scheme; Algorithm 2 (h > 0)
    // (halves of the coefficients for the doubled fluxes; in y one product of
    // the face next to the row, none inside)
    const double ax0 = 0.5 * cl[0][0], axN = 0.5 * cl[0][1];
    const double ay = q == 0 ? 0.5 * cl[1][0] : q == N ? -0.5 * cl[1][1] : 0.0;
    const double alpha = L.lim.alpha[ge];
    double lo[3][n];
#pragma unroll
    for (int p = 0; p < n; ++p) {
      double x[3];
#pragma unroll
      for (int v = 0; v < 3; ++v) {
        double o = L.lim.ulo[(v * Ne + ge) * nn + q * n + p];
        if (p == 0) o = fma(ax0, fxp[v][r][cc][q], o);
        if (p == N) o = fma(-axN, fxm[v][r][cc + 1][q], o);
        if (q == 0 || q == N) o = fma(ay, q == 0 ? fyp[v][r][cc][p] : fym[v][r + 1][cc][p], o);
        x[v] = o;
      }
      if constexpr (IMEX) {
        // backward Euler of Chezy friction, h fixed: m parallel to r,
        // m = r 2 / (1 + sqrt(1 + 4 dt C_f |r| / h^2))
        const double ih = drcp(x[0]);
        const double nm = dsqrt_pos(fma(x[1], x[1], x[2] * x[2]));
        const double qf = dsqrt_pos(fma(4.0 * dtp * T.src_coef * ih * ih, nm, 1.0));
        const double fr = 2.0 * drcp(1.0 + qf);
        x[1] *= fr;
        x[2] *= fr;
      }
#pragma unroll
      for (int v = 0; v < 3; ++v) {
        lo[v][p] = x[v];
        if (alpha != 0.0) out[v][p] = (1.0 - alpha) * out[v][p] + alpha * x[v];
      }
    }
    // Algorithm 2 over the element's n rows (lanes c*n .. c*n+n-1), in FP64
    // only where the high words of the smallest depths do not show theta = 1
    int omin = 0x7fffffff, fmn = 0x7fffffff;
#pragma unroll
    for (int p = 0; p < n; ++p) {
      omin = min(omin, __double2hiint(out[0][p]));
      fmn = min(fmn, __double2hiint(lo[0][p]));
    }
    omin = ~element_max(~omin);
    fmn = ~element_max(~fmn);
    if (__any_sync(0xffffffffu, !theta_one_element(fmn, omin))) {
      double lmin = lo[0][0];
#pragma unroll
      for (int p = 1; p < n; ++p) lmin = fmin(lmin, lo[0][p]);
#pragma unroll
      for (int k = 1; k < n; ++k) {
        const int src = c * n + ((q + k) % n);
        lmin = fmin(lmin, __shfl_sync(0xffffffffu, lmin, src < 32 ? src : lane));
      }
      const double eps = 0.1 * lmin;
      double th = 1.0;
#pragma unroll
      for (int p = 0; p < n; ++p) th = fmin(th, theta_lin(eps, lo[0][p], out[0][p]));
      double thr = th;
#pragma unroll
      for (int k = 1; k < n; ++k) {
        const int src = c * n + ((q + k) % n);
        thr = fmin(thr, __shfl_sync(0xffffffffu, th, src < 32 ? src : lane));
      }
      if (thr < 1.0) {
#pragma unroll
        for (int v = 0; v < 3; ++v)
#pragma unroll
          for (int p = 0; p < n; ++p) out[v][p] = thr * out[v][p] + (1.0 - thr) * lo[v][p];
      }
    }
  }
  chain_end();
  if (active) {
#pragma unroll
    for (int v = 0; v < 3; ++v)
#pragma unroll
      for (int p = 0; p < n; ++p) L.u_out[(v * Ne + ge) * nn + q * n + p] = out[v][p];
  }
  if (RES) return;

  bool bad = false;
#pragma unroll
  for (int p = 0; p < n; ++p)
    bad |= !positive_finite(out[0][p]) || !finite(out[1][p]) || !finite(out[2][p]);
  if (active && bad) atomicOr(&L.st->status, 1u);

  if (L.ctl.want_rate) {
    // element means (Definition admissibility.preserving.means), then
    // sigma_x/dx + sigma_y/dy (Sec. 5, Eq. time.step.2d)
    double m[3];
    // in the fixed point of each variable: the row with its weights, then the
    // rows of the element (integer sums: any order)
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      int mg = 0;
#pragma unroll
      for (int p = 0; p < n; ++p) mg = max(mg, fx_mag(out[v][p]));
      const int eo = fx_exp(element_max(mg));
      FxAcc a{0, 0};
#pragma unroll
      for (int p = 0; p < n; ++p)
        fx_mad(a, fx_split(fx_from<FB>(out[v][p], eo)), T.fx.w2_hi[q][p], T.fx.w2_lo[q][p]);
      const long long row = fx_sum(a);
      long long s = row;
      if constexpr ((n & (n - 1)) == 0) {
#pragma unroll
        for (int o = 1; o < n; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      } else {
#pragma unroll
        for (int k = 1; k < n; ++k) {
          const int src = c * n + ((q + k) % n);
          s += __shfl_sync(0xffffffffu, row, src < 32 ? src : lane);
        }
      }
      m[v] = fx_to(s, eo + 63 - FB, fx_zero(eo));
    }
    // the rates: one element per thread of the first TY * TX threads, so that
    // a warp computes 32 of them (from the n lanes of an element only one
    // would be busy)
    __shared__ double mean_s[TY][TX][3];
    if (lane_ok && q == 0) {
#pragma unroll
      for (int v = 0; v < 3; ++v) mean_s[r][c][v] = m[v];
    }
    __syncthreads();
    double rate = 0.0;
    if (threadIdx.x < TY * TX) {
      const int er = threadIdx.x / TX, ec = threadIdx.x - er * TX;
      if (ey0 + er < Ey && ex0 + ec < Ex)
        rate = swe_rate_2d(mean_s[er][ec][0], mean_s[er][ec][1], mean_s[er][ec][2],
                           T.sqrt_gravity, T.inv_dx, T.inv_dy);
    }
    block_max_atomic<BT>(rate, &L.st->rate[L.ctl.slot_write]);
  }
}

template <int N, bool GLL, bool WB, bool LIMIT, bool IMEX, bool SMALL>
int launch_face_shape(const Launch2D& L, cudaStream_t s) {
  constexpr int TX = 32 / (N + 1);
  constexpr int TY = FaceShape<N, LIMIT, SMALL>::TY, BT = FaceShape<N, LIMIT, SMALL>::block;
  const dim3 grid((unsigned)((L.Ex + TX - 1) / TX),
                  (unsigned)((L.row_end - L.row_begin + TY - 1) / TY));
  if (grid.y > 65535u) return (int)cudaErrorInvalidConfiguration;
  if constexpr (LIMIT)
    return launch_chained(k_face_2d<N, GLL, false, WB, true, IMEX, SMALL>, grid, BT, s, L);
  else if (L.ctl.residual)
    return launch_chained(k_face_2d<N, GLL, true, WB>,
                          dim3(grid.x, (grid.y * TY + kWarps2D - 1) / kWarps2D), kBlock2D, s, L);
  else
    return launch_chained(k_face_2d<N, GLL, false, WB, false, false, SMALL>, grid, BT, s, L);
}

template <int N, bool GLL, bool WB, bool LIMIT = false, bool IMEX = false>
int launch_face_t(const Launch2D& L, cudaStream_t s) {
  if (L.row_begin % 8 != 0 || L.row_end <= L.row_begin || L.row_end > L.Ey ||
      (L.row_end % 8 != 0 && L.row_end != L.Ey))
    return (int)cudaErrorInvalidValue;
  // small: fewer tiles than SMs
  constexpr int TX = 32 / (N + 1), TY = FaceShape<N, LIMIT, false>::TY;
  const int64_t tiles =
      ((L.Ex + TX - 1) / TX) * ((L.row_end - L.row_begin + TY - 1) / TY);
  return tiles < sm_count() ? launch_face_shape<N, GLL, WB, LIMIT, IMEX, true>(L, s)
                            : launch_face_shape<N, GLL, WB, LIMIT, IMEX, false>(L, s);
}

template <bool WB, bool LIMIT = false, bool IMEX = false>
int launch_face_dispatch(const Launch2D& L, cudaStream_t s) {
  switch (L.N * 2 + (L.gll ? 1 : 0)) {
    case 2: return launch_face_t<1, false, WB, LIMIT, IMEX>(L, s);
    case 3: return launch_face_t<1, true, WB, LIMIT, IMEX>(L, s);
    case 4: return launch_face_t<2, false, WB, LIMIT, IMEX>(L, s);
    case 5: return launch_face_t<2, true, WB, LIMIT, IMEX>(L, s);
    case 6: return launch_face_t<3, false, WB, LIMIT, IMEX>(L, s);
    case 7: return launch_face_t<3, true, WB, LIMIT, IMEX>(L, s);
    case 8: return launch_face_t<4, false, WB, LIMIT, IMEX>(L, s);
    case 9: return launch_face_t<4, true, WB, LIMIT, IMEX>(L, s);
  }
  return (int)cudaErrorInvalidValue;
}

}  // namespace
}  // namespace crkfr
