// The fused 1D cRK-FR step (sm_103a, FP64): the tile body shared by the
// single-mesh kernel, the ragged-ensemble kernel and their source-term (IMEX)
// instantiations, which live in different translation units.
//
// Mapping: one thread owns one node; an element's N+1 threads lie in one warp
// and exchange the fluxes of a stage through shared memory (Sec. 3,
// Eq. crkfr.non.cons.final, inner stages; Eqs. disc.avg.flux, time.avg.soln,
// local.time.avg.non.cons).  The stage sums are FP64; the products with D and
// the end-point rows, the time averages and the fluxes run in block fixed point
// on the integer pipe (fixed_point.cuh), and D is applied to the averages once
// instead of accumulating every stage's operator.  (Fluxes in fixed point
// instead of FP64: 1e5 elements at N = 4, four steps, 375 -> 302 us; the
// ensemble of 256 meshes, two steps, 4.03 -> 3.24 ms.  The average of h in FP64,
// which a shallow node needs: 311 us, 3.32 ms.)  Bound by the FP64 pipe (67 %
// busy) and issue slots (0.50) together.  A block updates all its
// elements but the first and the last, whose stages it recomputes for their
// neighbours (4 % of a 256-thread block at N = 4), so that the only
// inter-element coupling, one Riemann problem per face (Eqs. numflux.cons,
// combined.wave.speed, good.numflux.non.cons, total.F.non.cons), is solved
// from face traces exchanged through shared memory, and u is read and written
// once per step.  The step therefore reads u^n from one buffer and writes
// u^{n+1} to another.  Face terms and the next time step's rates are one
// thread per element, packed into the block's first warps (an FP64
// instruction costs the same for one lane as for 32).
//
// Face terms are carried doubled, T' = 2 (F^num,+- - F^tot,+-), and the
// correction tables hold 0.5 g'(xi_p)/dx, which saves two FP64 multiplies
// per face.  For GLL nodes the traces are the end values and g_L', g_R'
// vanish away from the end nodes (App. B, under Eq. fr.gll).
//
// With a source term (IMEX = true; Sec. 2, Eqs. crkfr.inner, crkfr,
// avg.source) the stages follow SSP3-IMEX(4,3,3): the implicit source terms
// of earlier stages join the stage sum, each stage's own source term is
// solved point by point in closed form, and the final update adds
// dt sum_i b_i s(u^(i)).  Sources: linear damping s = -K v for advection
// (the model problem of App. A), Chezy friction s = (0, -C_f |v| v) for
// shallow water (the friction term of Sec. 5.5).
//
// The well-balanced shallow-water form (SYS = CRKFR_SYS_SWE_1D_WB) drops the
// pressure from the momentum flux, adds g h D h to the local
// non-conservative term (g h D (h + b)), and dissipates and fluctuates the
// free surface eta = h + b instead of h at the faces.
//
// With the subcell blending limiter (LIMIT = true; Sec. 4) each element also
// takes a first-order finite-volume step on its N+1 subcells of widths
// w_p dx (Eqs. subcell.defn, low.order.update) with the non-conservative
// Rusanov fluxes of Eq. combined.num.flux, both schemes share the blended
// face flux of Eq. Fblend limited by Algorithm 1 so that the two adjacent
// low-order node updates keep h > 0, and the blend of Eq. blended.scheme is
// limited per element by Algorithm 2.
#pragma once

#include <cuda_runtime.h>

#include "device_common.cuh"
#include "fixed_point.cuh"
#include "launch.h"

namespace crkfr {
namespace {

constexpr int kBlock1D = kMaxBlock1D;   // of the residual and the ensemble steps
constexpr int kBlockLimit1D = 128;      // of the limited step (its shared memory)

template <int SYS>
struct Sys1D;
template <>
struct Sys1D<CRKFR_SYS_VARADV_1D> {
  static constexpr int M = 1;
  static constexpr int K = 1;       // exchange fields of a stage: v
  static constexpr int NT = 1;      // traces from nodal values: V (and then a)
  static constexpr int SV = 0;      // variable carrying the source (v)
};
template <>
struct Sys1D<CRKFR_SYS_SWE_1D> {
  static constexpr int M = 2;
  static constexpr int K = 3;       // h, hu, the momentum flux
  static constexpr int NT = 5;      // H, M (time averages), F_m, h^n, m^n (and then b)
  static constexpr int SV = 1;      // variable carrying the source (hu)
};
template <>
struct Sys1D<CRKFR_SYS_SWE_1D_WB> : Sys1D<CRKFR_SYS_SWE_1D> {};

// First-order non-conservative Rusanov fluxes (Eq. combined.num.flux) between
// the nodal states L and R: fm = f^num + B(w_L) w^num, fp = f^num + B(w_R) w^num,
// f^num = (f_L + f_R)/2 - lam/2 (jump), lam the larger spectral radius, the
// jump that of h, or of eta = h + b for the well-balanced form.
template <int SYS>
__device__ __forceinline__ void lo_flux(const double* uL, const double* uR, double cL, double cR,
                                        const Tables& T, double* fm, double* fp) {
  if constexpr (SYS == CRKFR_SYS_VARADV_1D) {
    const double lam = max_nonneg(fabs(cL), fabs(cR));
    const double f = -0.5 * lam * (uR[0] - uL[0]);
    const double un = 0.5 * (uL[0] + uR[0]);
    fm[0] = f + cL * un;
    fp[0] = f + cR * un;
  } else {
    constexpr bool WB = (SYS == CRKFR_SYS_SWE_1D_WB);
    const double g = T.gravity;
    const double hL = uL[0], mL = uL[1], hR = uR[0], mR = uR[1];
    const double lam =
        max_nonneg(swe_speed(hL, mL, T.sqrt_gravity), swe_speed(hR, mR, T.sqrt_gravity));
    const double vL = mL * drcp(hL), vR = mR * drcp(hR);
    const double fL = WB ? mL * vL : fma(0.5 * g * hL, hL, mL * vL);
    const double fR = WB ? mR * vR : fma(0.5 * g * hR, hR, mR * vR);
    const double jh = WB ? (hR + cR) - (hL + cL) : hR - hL;
    const double f0 = fma(-0.5 * lam, jh, 0.5 * (mL + mR));
    const double f1 = fma(-0.5 * lam, mR - mL, 0.5 * (fL + fR));
    const double wn = WB ? 0.5 * (hL + hR) + 0.5 * (cL + cR) : 0.5 * (cL + cR);
    fm[0] = f0;
    fp[0] = f0;
    fm[1] = f1 + g * hL * wn;
    fp[1] = f1 + g * hR * wn;
  }
}

// Per-node parts of the shallow-water first-order flux: the spectral radius
// |v| + sqrt(g h) and the momentum flux (with the pressure g h^2 / 2 in the
// standard form).
template <int SYS>
__device__ __forceinline__ void lo_node_1d(double h, double m, double g, double& s, double& f) {
  constexpr bool WB = (SYS == CRKFR_SYS_SWE_1D_WB);
  const double v = m * drcp(h);
  s = fabs(v) + dsqrt_pos(g * h);
  f = WB ? m * v : fma(0.5 * g * h, h, m * v);
}

// lo_flux for shallow water from the per-node parts of its two states
template <int SYS>
__device__ __forceinline__ void lo_flux_nodes_1d(const double* uL, const double* uR, double cL,
                                                 double cR, double sL, double sR, double fL,
                                                 double fR, double g, double* fm, double* fp) {
  constexpr bool WB = (SYS == CRKFR_SYS_SWE_1D_WB);
  const double hL = uL[0], mL = uL[1], hR = uR[0], mR = uR[1];
  const double lam = max_nonneg(sL, sR);
  const double jh = WB ? (hR + cR) - (hL + cL) : hR - hL;
  const double f0 = fma(-0.5 * lam, jh, 0.5 * (mL + mR));
  const double f1 = fma(-0.5 * lam, mR - mL, 0.5 * (fL + fR));
  const double wn = WB ? 0.5 * (hL + hR) + 0.5 * (cL + cR) : 0.5 * (cL + cR);
  fm[0] = f0;
  fp[0] = f0;
  fm[1] = f1 + g * hL * wn;
  fp[1] = f1 + g * hR * wn;
}

// Point-implicit backward-Euler source step of the low-order update
// (Eq. low.order.update): u - dt s(u) = r, in closed form.
template <int SYS>
__device__ __forceinline__ void lo_source(const Tables& T, double dt, double* u) {
  if constexpr (SYS == CRKFR_SYS_VARADV_1D) {
    u[0] *= drcp(fma(dt, T.src_coef, 1.0));
  } else {
    const double ih = drcp(u[0]);
    const double q = dsqrt_pos(fma(4.0 * dt * T.src_coef * ih * ih, fabs(u[1]), 1.0));
    u[1] *= 2.0 * drcp(1.0 + q);
  }
}

// Minimum over the n lanes of an element.
template <int n, class V>
__device__ __forceinline__ V element_min(V v, int le, int p, int lane) {
  V m = v;
#pragma unroll
  for (int k = 1; k < n; ++k) {
    const int r = p + k < n ? p + k : p + k - n, src = le * n + r;
    const V o = __shfl_sync(0xffffffffu, v, src < 32 ? src : lane);
    if constexpr (sizeof(V) == 8)
      m = fmin(m, o);
    else
      m = min(m, o);
  }
  return m;
}

// One tile (tile_elements_1d(blockDim.x, n) elements plus a halo element on
// each side) of the fused 1D step of one mesh.  T holds reference-element
// tables (dx = 1: D, l(0), l(1), 0.5 g'); xs = 1/dx scales the local operator
// and the corrections through the scalar coefficients only (stage coefficients
// dt a_ij xs, update coefficient dt b_ref xs), so one table serves meshes of
// any dx.  Every element's arithmetic is the same for any block size.  last: the
// block leaves after this tile (chain_end()).  (No __restrict__: the loads must
// not move above chain_begin().)
template <int SYS, int N, bool GLL, bool RES, bool IMEX, bool LIMIT = false>
__device__ __forceinline__ void step_1d_tile(const Tables& T, double xs,
                                             const double* u_in, double* u_out,
                                             const double* snode, const double* sface, int64_t E,
                                             int64_t tile, DevState* st, const StepCtl& ctl,
                                             bool first_tile, bool last,
                                             const LimitArgs& LA = LimitArgs{},
                                             const double* ghost = nullptr) {
  using TB = Tab<N, IMEX>;
  using SY = Sys1D<SYS>;
  constexpr int n = N + 1;
  constexpr int M = SY::M, K = SY::K, NT = SY::NT, SV = SY::SV;
  constexpr int S = TB::S;
  constexpr bool SWE = (SYS == CRKFR_SYS_SWE_1D || SYS == CRKFR_SYS_SWE_1D_WB);
  constexpr bool WB = (SYS == CRKFR_SYS_SWE_1D_WB);
  constexpr int EPW = 32 / n;                       // elements per warp
  constexpr int NE = (LIMIT ? kBlockLimit1D : kMaxBlock1D) / 32 * EPW;   // of the largest block
  constexpr int KX = SWE ? 5 : 1;                   // exchange fields per node
  // fixed point: operand bits, shift of the weighted sums back to them, and
  // the bits a later stage may outgrow the first (as in local_2d.cuh)
  constexpr int FB = 59;
  constexpr bool WIDE = TB::weight_sum() > 8;
  constexpr int kSumShift = WIDE ? 7 : 3;
  constexpr int kHeadroom = 1;

  const int t = threadIdx.x, lane = t & 31;
  const int le = lane / n, p = lane - le * n;
  const bool lane_ok = le < EPW;
  const int ne = (int)(blockDim.x >> 5) * EPW;      // elements of this block
  const int slot = (t >> 5) * EPW + (lane_ok ? le : 0);
  const int64_t e_raw = tile * (ne - 2) + slot - 1;
  int64_t e = e_raw % E;
  if (e < 0) e += E;
  const bool owner = lane_ok && slot >= 1 && slot <= ne - 2 && e_raw < E;

  __shared__ __align__(16) Fx sx[NE][KX][n];
  __shared__ double str[2][NT + 1][NE];             // traces at the left / right end
  __shared__ double sT[2][M][NE];                   // face terms: right face, left face
  __shared__ int smag[NE][K];
  __shared__ StepSizes<TB> sz;
  Fx (*X)[n] = sx[slot];

  if (t < 32) {
    // the step size (a division) and its products by the block's first warp
    double dt = 0.0;
    if (t == 0) {
      dt = RES ? ctl.dt_fixed : step_dt(ctl, st);
      if (!RES && first_tile) step_bookkeeping(ctl, st, dt);
    }
    dt = __shfl_sync(0xffffffffu, dt, 0);
    fill_step_sizes<TB, IMEX>(sz, dt, xs);
  }
  if (lane_ok) {
    // (K <= 3 entries by up to n threads)
#pragma unroll
    for (int k = 0; k < K; ++k)
      if (p == k % n) smag[slot][k] = 0;
  }

  // ---- u^n and the static coefficient terms of this node -------------------
  // (on a subdomain the elements beyond its ends are the neighbours' ghosts)
  double u0[M], sn;
  const bool from_ghost = ghost != nullptr && (e_raw < 0 || e_raw >= E);
  constexpr int GD = ghost_dyn_1d(M, n);   // static part of a ghost after GD doubles
  const double* gs = ghost + (e_raw < 0 ? 0 : ghost_stride_1d(M, n));
  if (from_ghost) {
#pragma unroll
    for (int v = 0; v < M; ++v) u0[v] = gs[v * n + p];
    sn = gs[GD + p];
  } else {
#pragma unroll
    for (int v = 0; v < M; ++v) u0[v] = u_in[((int64_t)v * E + e) * n + p];
    sn = snode[e * n + p];
  }
  if (lane_ok && p == 0) {
    str[0][NT][slot] = from_ghost ? gs[GD + n] : sface[2 * e];
    str[1][NT][slot] = from_ghost ? gs[GD + n + 1] : sface[2 * e + 1];
  }
  int dh[n], dl[n];                        // the node's row of D
#pragma unroll
  for (int j = 0; j < n; ++j) {
    dh[j] = T.fx.Dx_hi[p][j];
    dl[j] = T.fx.Dx_lo[p][j];
  }

  // ---- limiter: alpha_e, nodal c, first-order fluxes of the inner subfaces --
  static_assert(!LIMIT || (N >= 1 && !RES), "the limiter needs N >= 1 and a step");
  constexpr int LM = LIMIT ? M : 1, LE = LIMIT ? NE : 1, Ln = LIMIT ? n : 1;
  double alpha = 0.0;
  __shared__ double lu[LM][LE][Ln], lc[LE][Ln], ls[LE][Ln], lf[LE][Ln];
  __shared__ double lim[LM][LE][Ln];   // right flux of node p (B at node p), p < N
  __shared__ double lip[LM][LE][Ln];   // left flux of node p+1 (B at node p+1)
  __shared__ double lF[2][LM][LE];     // limited fluxes F^- of the right, F^+ of the left face
  __shared__ double la[LE];
  if constexpr (LIMIT) {
    const double cn = from_ghost ? gs[GD + n + 2 + p] : LA.cnode[e * n + p];
    if (LA.mode == 2) {
      alpha = LA.alpha_fixed;
    } else if (ghost) {
      // a range of a larger mesh: the raw indicator of elements -2, -1 and
      // E, E+1 comes with the ghosts (slot 0 the adjacent element, slot 1
      // the one beyond it); threads past E+1 only need in-bounds reads
      auto raw = [&](int64_t r) -> double {
        if (r < 0) return ghost[M * n + (r < -2 ? 1 : -1 - r)];
        if (r >= E) return ghost[ghost_stride_1d(M, n) + M * n + (r > E + 1 ? 1 : r - E)];
        return LA.alpha_raw[r];
      };
      const double r0 = raw(e_raw);
      const double rn = fmax(raw(e_raw - 1), raw(e_raw + 1));
      alpha = fmax(r0, 0.5 * rn);
    } else {
      const int64_t em = e == 0 ? E - 1 : e - 1, ep = e == E - 1 ? 0 : e + 1;
      const double r0 = LA.alpha_raw[e];
      const double rn = fmax(LA.alpha_raw[em], LA.alpha_raw[ep]);
      alpha = fmax(r0, 0.5 * rn);
    }
    if (lane_ok) {
#pragma unroll
      for (int v = 0; v < M; ++v) lu[v][slot][p] = u0[v];
      lc[slot][p] = cn;
      if (p == 0) la[slot] = alpha;
      // per-node parts (shallow water: one reciprocal and one root per node
      // instead of per subface side)
      if constexpr (SWE) lo_node_1d<SYS>(u0[0], u0[1], T.gravity, ls[slot][p], lf[slot][p]);
    }
    __syncwarp();
    if (lane_ok && p < N) {
      double b[M], fm_[M], fp_[M];
#pragma unroll
      for (int v = 0; v < M; ++v) b[v] = lu[v][slot][p + 1];
      if constexpr (SWE)
        lo_flux_nodes_1d<SYS>(u0, b, cn, lc[slot][p + 1], ls[slot][p], ls[slot][p + 1],
                              lf[slot][p], lf[slot][p + 1], T.gravity, fm_, fp_);
      else
        lo_flux<SYS>(u0, b, cn, lc[slot][p + 1], T, fm_, fp_);
#pragma unroll
      for (int v = 0; v < M; ++v) {
        lim[v][slot][p] = fm_[v];
        lip[v][slot][p] = fp_[v];
      }
    }
  }
  __syncwarp();

  // ---- inner stages (element-local) ----------------------------------------
  // Time averages are integer sums (h: FP64) with the weights b_j / b_ref; b_ref is
  // applied to dt in the update, and the fluctuation, the one face term that
  // is not a time average, uses g / b_ref.
  double Ls[S][M];                     // local operator at each stage
  double Ss[S];                        // source of variable SV at each stage (IMEX)
  double Sb = 0.0;                     // sum_j (b_j/b_ref) s(u^(j)) (IMEX)
  double Pb = 0.0;                     // sum_j (b_j/b_ref) h g d(h + b) (WB)
  // the average of h: field 0's sum (FIX_H), or sum_j (b_j/b_ref) (h^(j) - h^n),
  // below + h^n / b_ref, where it enters node by node (as in local_2d.cuh)
  constexpr bool FIX_H = WB && !GLL;
  double uh = 0.0;
  long long A[K], B[K];                // of the other exchange fields (WIDE: A 2^30 + B)
  int Ex[K];                           // exponents of the exchange fields
  // shallow water: h is contracted in the well-balanced form only
  constexpr int kStage0 = SWE && !WB ? 1 : 0, kAvg0 = SWE && !FIX_H ? 1 : 0;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    A[k] = B[k] = 0;
    Ex[k] = -1;
  }
  // row of D on an exchange field
  auto contract = [&](int k) -> long long {
    FxAcc a;
    Fx r[n];
    fx_row<n>(X[k], r);
    fx_mul(a, r[0], dh[0], dl[0]);
#pragma unroll
    for (int j = 1; j < n; ++j) fx_mad(a, r[j], dh[j], dl[j]);
    return fx_sum(a);
  };
  bool first = true;                   // (resolved at compile time by unrolling)
#pragma unroll
  for (int i = 0; i < S; ++i) {
    // (the step sizes: the first stage does without)
    if (i == (IMEX ? 0 : 1)) __syncthreads();
    if (SWE && !FIX_H && i > 0 && TB::feeds(i > 0 ? i - 1 : 0)) uh = fma(sz.avg[i - 1], Ls[i - 1][0], uh);
    double cur[M];
#pragma unroll
    for (int v = 0; v < M; ++v) {
      double acc = u0[v];
#pragma unroll
      for (int j = 0; j < i; ++j)
        if (TB::a(i, j) != 0.0) acc = fma(sz.e[i][j], Ls[j][v], acc);
      if (IMEX && v == SV) {
#pragma unroll
        for (int j = 0; j < i; ++j)
          if (TB::ai(i, j) != 0.0) acc = fma(sz.im[i][j], Ss[j], acc);
      }
      cur[v] = acc;
    }
    if constexpr (IMEX) {
      // point-implicit source of this stage: cur - dt a_ii s(cur) = r
      const double gam = sz.im[i][i];
      if constexpr (SWE) {
        // s = -C_f |m| m / h^2 with h fixed: |m| + gam C_f |m|^2 / h^2 = |r|
        const double gcf = gam * T.src_coef;
        const double ih = drcp(cur[0]);
        const double ih2 = ih * ih;
        if (TB::ai(i, i) != 0.0) {
          const double r = cur[1];
          const double qf = dsqrt_pos(fma(4.0 * gcf * ih2, fabs(r), 1.0));
          cur[1] = r * (2.0 * drcp(1.0 + qf));
        }
        if (TB::need_S(i)) Ss[i] = -(T.src_coef * ih2) * fabs(cur[1]) * cur[1];
      } else {
        // s = -K v
        if (TB::ai(i, i) != 0.0) cur[0] *= drcp(fma(gam, T.src_coef, 1.0));
        if (TB::need_S(i)) Ss[i] = -T.src_coef * cur[0];
      }
    }
    const int wi = TB::weight(i);
    const double wd = wi;
    const bool need_op = TB::feeds(i);
    if (need_op || wi != 0) {
      int mag[K];
      bool over = false;
#pragma unroll
      for (int k = kStage0; k < K; ++k) {
        mag[k] = k < M ? fx_mag(cur[k < M ? k : 0])
                       : fx_flux_mag<!WB>(cur[0], fx_log(cur[M - 1]), fx_log(cur[M - 1]),
                                          fx_log(T.half_gravity));
        // (IMEX: the traces of u^n, no stage value here, share the exponents)
        if (IMEX && first && k < M) mag[k] = max(mag[k], fx_mag(u0[k]));
        over = over || (lane_ok && mag[k] >> 20 > Ex[k]);
      }
      // exponents as in local_2d.cuh, after the barrier that ends the last
      // stage's reads of X
      if (warp_barrier_or(over)) {
        if (over) {
#pragma unroll
          for (int k = kStage0; k < K; ++k) atomicMax(&smag[slot][k], mag[k]);
        }
        __syncwarp();
#pragma unroll
        for (int k = kStage0; k < K; ++k) {
          const int ek = fx_exp(smag[slot][k]);
          const int d = ek > Ex[k] ? ek + kHeadroom - Ex[k] : 0;
          Ex[k] += d;
          if (!first && k >= kAvg0) fx_rescale<WIDE>(A[k], B[k], d);
        }
      }
      long long f[K];
      if constexpr (SWE) {
        const FxSig sh = fx_sig(cur[0]), sm = fx_sig(cur[1]);
        const unsigned long long R = recip_bits((unsigned)__double2hiint(cur[0]),
                                                (unsigned)__double2loint(cur[0]));
        if (WB) f[0] = fx_from<FB>(sh, Ex[0]);
        f[1] = fx_from<FB>(sm, Ex[1]);
        f[2] = fx_momentum_flux<FB>(sm, fx_velocity(R, sm), sm, sh, Ex[2]);
        if (!WB) f[2] += fx_pressure<FB>(sh, fx_sig(T.half_gravity), Ex[2]);
      } else {
        f[0] = fx_from<FB>(cur[0], Ex[0]);
      }
#pragma unroll
      for (int k = kStage0; k < K; ++k) {
        const long long v = f[k];
        const Fx x = fx_split(v);
        if (wi != 0 && k >= kAvg0) fx_accumulate<WIDE>(A[k], B[k], v, x, wi);
        if ((SWE && k == 0 ? WB : need_op) && lane_ok) X[k][p] = x;
      }
      if (need_op || WB) {
        __syncwarp();
        double nc = 0.0;
        if constexpr (WB) {
          nc = cur[0] * fma(T.gravity, fx_to(contract(0), Ex[0] + T.fx.kDx - FB, fx_zero(Ex[0])), sn);
          if (wi != 0) Pb = fma(wd, nc, Pb);
        }
        if (need_op) {
          const int k0 = SWE ? 1 : 0;
          const double l0 = fx_to(contract(k0), Ex[k0] + T.fx.kDx - FB, fx_zero(Ex[k0]));
          if constexpr (SWE) {
            const double l1 = fx_to(contract(2), Ex[2] + T.fx.kDx - FB, fx_zero(Ex[2]));
            Ls[i][0] = l0;
            Ls[i][1] = WB ? l1 + nc : fma(cur[0], sn, l1);
          } else {
            Ls[i][0] = sn * l0;
          }
        }
      }
      if (wi != 0) first = false;
    }
    if constexpr (IMEX) {
      // the implicit weights b_i equal the explicit ones b~_i
      if (wi != 0) Sb = fma(wd, Ss[i], Sb);
    }
  }

  // ---- the averages' derivative and the face traces --------------------------
#pragma unroll
  for (int k = kAvg0; k < K; ++k) A[k] = fx_average<WIDE, kSumShift>(A[k], B[k]);
  const double du = uh;
  uh = fma((double)TB::weight_sum(), u0[0], du);
  if constexpr (SWE && !GLL && !FIX_H) {
    // the exponent of the traces of h: u^n and its average's increment (in sum
    // units)
    const int mu = fx_mag(du);
    const int m = max(fx_mag(u0[0]), mu >= 0x7ff00000 ? mu : mu - (kSumShift << 20));
    if (lane_ok) atomicMax(&smag[slot][0], m);
  }
  __syncwarp();
  if (SWE && !GLL && !FIX_H) Ex[0] = fx_exp(smag[slot][0]);
  if (lane_ok) {
#pragma unroll
    for (int k = kAvg0; k < K; ++k) X[k][p] = fx_split(A[k]);
    if constexpr (SWE) {
      if (!FIX_H)
        X[0][p] = GLL ? Fx{__double2hiint(uh), __double2loint(uh)}
                      : fx_split(fx_increment<WIDE, kSumShift, FB>(u0[0], TB::weight_sum(), du,
                                                                   Ex[0]));
#pragma unroll
      for (int v = 0; v < 2; ++v)
        X[3 + v][p] = GLL ? Fx{__double2hiint(u0[v]), __double2loint(u0[v])}
                          : fx_split(fx_from<FB>(u0[v], Ex[v]));
    }
  }
  __syncwarp();
  double V[M];                         // sum_j (b_j/b_ref) L_j
  if constexpr (SWE) {
    V[0] = fx_to(contract(1), Ex[1] + T.fx.kDx - FB + kSumShift, fx_zero(Ex[1]));
    V[1] = fx_to(contract(2), Ex[2] + T.fx.kDx - FB + kSumShift, fx_zero(Ex[2]));
    if (WB)
      V[1] += Pb;
    else
      V[1] = fma(uh, sn, V[1]);
  } else {
    V[0] = sn * fx_to(contract(0), Ex[0] + T.fx.kDx - FB + kSumShift, fx_zero(Ex[0]));
  }
  // traces: 2 NT of them, shared out over the element's threads
  if (lane_ok) {
#pragma unroll
    for (int j0 = 0; j0 < 2 * NT; j0 += n) {
      const int job = j0 + p;
      if (2 * NT % n != 0 && job >= 2 * NT) break;
      const int side = job >= NT, fi = side ? job - NT : job;
      const int ex = !SWE || fi == 0 || fi == 3 ? Ex[0] : fi == 2 ? Ex[K - 1] : Ex[K > 1 ? 1 : 0];
      const int avg = fi < 3 ? kSumShift : 0;
      double tr;
      if constexpr (GLL) {
        const Fx v = X[fi][side ? N : 0];
        tr = fi >= 3 || (SWE && fi == 0) ? __hiloint2double(v.hi, v.lo)
                     : fx_to(((long long)v.hi << 30) + v.lo, ex + 63 - FB + avg, fx_zero(ex));
      } else {
        FxAcc a;
        Fx r[n];
        fx_row<n>(X[fi], r);
        fx_mul(a, r[0], side ? T.fx.l1_hi[0] : T.fx.l0_hi[0], side ? T.fx.l1_lo[0] : T.fx.l0_lo[0]);
#pragma unroll
        for (int j = 1; j < n; ++j)
          fx_mad(a, r[j], side ? T.fx.l1_hi[j] : T.fx.l0_hi[j],
                 side ? T.fx.l1_lo[j] : T.fx.l0_lo[j]);
        tr = fx_to(fx_sum(a), ex + T.fx.kL - FB + avg, fx_zero(ex));
      }
      str[side][fi][slot] = tr;
    }
  }
  __syncthreads();
  const double dt = sz.dt, dtx = dt * xs;   // (the latter for the limiter)

  // ---- Riemann problem at the right face of slot f (f | f+1), both sides ----
  for (int f = t; f < ne - 1; f += blockDim.x) {
    double tm[NT + 1], tp[NT + 1];
#pragma unroll
    for (int k = 0; k <= NT; ++k) {
      tm[k] = str[1][k][f];
      tp[k] = str[0][k][f + 1];
    }
    if constexpr (LIMIT) {
      // time-averaged numerical and total fluxes in the units of the time
      // averages (divided by b_ref), Eqs. numflux.cons, good.numflux.non.cons,
      // total.F.non.cons; the first-order face flux from the nodal values next
      // to the face; Eq. Fblend; Algorithm 1 (h > 0) for shallow water
      constexpr double b0 = TB::bref();
      double FHm[M], FHp[M], FTm[M], FTp[M];
      if constexpr (SWE) {
        const double Hm = tm[0], Mm = tm[1], Fm = tm[2], hm = tm[3], mm = tm[4], bm = tm[5];
        const double Hp = tp[0], Mp = tp[1], Fp = tp[2], hp = tp[3], mp = tp[4], bp = tp[5];
        const double g = T.gravity;
        const double lam =
            max_nonneg(swe_speed(hm, mm, T.sqrt_gravity), swe_speed(hp, mp, T.sqrt_gravity));
        const double dUh = WB ? (Hp + bp * T.inv_b0) - (Hm + bm * T.inv_b0) : Hp - Hm;
        const double Fn0 = fma(-0.5 * lam, dUh, 0.5 * (Mm + Mp));
        const double Fn1 = fma(-0.5 * lam, Mp - Mm, 0.5 * (Fm + Fp));
        const double bn = 0.5 * (bm + bp) * T.inv_b0;
        const double Wn = WB ? 0.5 * (Hm + Hp) + bn : bn;
        const double Wm = WB ? Hm + bm * T.inv_b0 : bm * T.inv_b0;
        const double Wp = WB ? Hp + bp * T.inv_b0 : bp * T.inv_b0;
        FHm[0] = Fn0;
        FHp[0] = Fn0;
        FHm[1] = Fn1 + g * hm * Wn;
        FHp[1] = Fn1 + g * hp * Wn;
        FTm[0] = Mm;
        FTp[0] = Mp;
        FTm[1] = Fm + g * hm * Wm;
        FTp[1] = Fp + g * hp * Wp;
      } else {
        const double Vm = tm[0], am = tm[1], Vp = tp[0], ap = tp[1];
        const double lam = max_nonneg(fabs(am), fabs(ap));
        const double Fn = -0.5 * lam * (Vp - Vm);
        const double Vn = 0.5 * (Vm + Vp);
        FHm[0] = Fn + am * Vn;
        FHp[0] = Fn + ap * Vn;
        FTm[0] = am * Vm;
        FTp[0] = ap * Vp;
      }
      double uN[M], u0R[M], fLm[M], fLp[M];
#pragma unroll
      for (int v = 0; v < M; ++v) {
        uN[v] = lu[v][f][N];
        u0R[v] = lu[v][f + 1][0];
      }
      lo_flux<SYS>(uN, u0R, lc[f][N], lc[f + 1][0], T, fLm, fLp);
      const double af = 0.5 * (la[f] + la[f + 1]);
      // (af = 0 and theta = 1 are the common cases: there the blends reduce
      // to their first terms and are skipped)
      double Fm_[M], Fp_[M];
#pragma unroll
      for (int v = 0; v < M; ++v) {
        Fm_[v] = b0 * FHm[v];
        Fp_[v] = b0 * FHp[v];
        if (af != 0.0) {
          Fm_[v] = (1.0 - af) * Fm_[v] + af * fLm[v];
          Fp_[v] = (1.0 - af) * Fp_[v] + af * fLp[v];
        }
      }
      if constexpr (SWE) {
        const double c0 = dtx * T.inv_w[0], cN = dtx * T.inv_w[N];
        const double fi0R = lim[0][f + 1][0], fiNL = lip[0][f][N > 0 ? N - 1 : 0];
        // (in FP64 only where FP32 does not show theta = 1)
        if (!(theta_one(u0R[0], c0, fi0R, fLp[0], Fp_[0]) &&
              theta_one(uN[0], -cN, fiNL, fLm[0], Fm_[0]))) {
          const double low0 = u0R[0] - c0 * (fi0R - fLp[0]);
          const double lowN = uN[0] - cN * (fLm[0] - fiNL);
          const double t0 = u0R[0] - c0 * (fi0R - Fp_[0]);
          const double tN = uN[0] - cN * (Fm_[0] - fiNL);
          const double th = fmin(theta_lin(0.1 * low0, low0, t0), theta_lin(0.1 * lowN, lowN, tN));
          if (th < 1.0) {
#pragma unroll
            for (int v = 0; v < M; ++v) {
              Fm_[v] = th * Fm_[v] + (1.0 - th) * fLm[v];
              Fp_[v] = th * Fp_[v] + (1.0 - th) * fLp[v];
            }
          }
        }
      }
      // face terms in the doubled units of the corrections: 2 (F - F^tot) / b_ref
#pragma unroll
      for (int v = 0; v < M; ++v) {
        lF[0][v][f] = Fm_[v];
        lF[1][v][f + 1] = Fp_[v];
        sT[0][v][f] = 2.0 * (Fm_[v] * T.inv_b0 - FTm[v]);
        sT[1][v][f + 1] = 2.0 * (Fp_[v] * T.inv_b0 - FTp[v]);
      }
    } else if constexpr (SWE) {
      const double lam =
          max_nonneg(swe_speed(tm[3], tm[4], T.sqrt_gravity), swe_speed(tp[3], tp[4], T.sqrt_gravity));
      // F_h = U_m (the h flux is the momentum)
      const double dFm = tp[2] - tm[2], dUm = tp[1] - tm[1];
      // jump of the dissipated and fluctuating state: h, or eta = h + b for
      // the well-balanced form (b is static, so in the units of the time
      // averages, divided by b_ref, its jump carries 1 / b_ref)
      const double db = tp[5] - tm[5];
      const double dUh = WB ? fma(T.inv_b0, db, tp[0] - tm[0]) : tp[0] - tm[0];
      const double gdb = WB ? T.gravity * dUh : T.face_g * db;
      sT[0][0][f] = fma(-lam, dUh, dUm);
      sT[0][M - 1][f] = fma(tm[3], gdb, fma(-lam, dUm, dFm));
      sT[1][0][f + 1] = -fma(lam, dUh, dUm);
      sT[1][M - 1][f + 1] = -fma(tp[3], gdb, fma(lam, dUm, dFm));
    } else {
      const double lam = max_nonneg(fabs(tm[1]), fabs(tp[1]));
      const double dU = tp[0] - tm[0];
      sT[0][0][f] = (tm[1] - lam) * dU;
      sT[1][0][f + 1] = -(lam + tp[1]) * dU;
    }
  }
  __syncthreads();

  if (last) chain_end();
  // ---- correction and update (owners only) --------------------------------
  constexpr double b0 = TB::bref();
  const double dtb0 = sz.dtb_x, dts = sz.dtb;
  double out[M];
#pragma unroll
  for (int v = 0; v < M; ++v) {
    double R = V[v];
    if (!GLL || p == N) R = fma(sT[0][v][slot], T.gRx[p], R);
    if (!GLL || p == 0) R = fma(sT[1][v][slot], T.gLx[p], R);
    double o = RES ? -(b0 * xs) * R : fma(-dtb0, R, u0[v]);
    if (IMEX && v == SV) o = fma(RES ? b0 : dts, Sb, o);
    out[v] = o;
  }
  if constexpr (LIMIT) {
    // first-order subcell update (Eq. low.order.update), then
    // Eq. blended.scheme and Algorithm 2 (h > 0)
    double lo[M];
    const double cw = dtx * T.inv_w[p];
#pragma unroll
    for (int v = 0; v < M; ++v) {
      const double right = p < N ? lim[v][slot][p] : lF[0][v][slot];
      const double left = p > 0 ? lip[v][slot][p > 0 ? p - 1 : 0] : lF[1][v][slot];
      lo[v] = u0[v] - cw * (right - left);
    }
    if constexpr (IMEX) lo_source<SYS>(T, dt, lo);
#pragma unroll
    for (int v = 0; v < M; ++v)
      if (alpha != 0.0) out[v] = (1.0 - alpha) * out[v] + alpha * lo[v];
    if constexpr (SWE) {
      // (in FP64 only where the high words do not show theta = 1)
      const int lmn = element_min<n>(__double2hiint(lo[0]), le, p, lane);
      const int omn = element_min<n>(__double2hiint(out[0]), le, p, lane);
      if (__any_sync(0xffffffffu, !theta_one_element(lmn, omn))) {
        const double eps = 0.1 * element_min<n>(lo[0], le, p, lane);
        const double th = element_min<n>(theta_lin(eps, lo[0], out[0]), le, p, lane);
        if (th < 1.0) {
#pragma unroll
          for (int v = 0; v < M; ++v) out[v] = th * out[v] + (1.0 - th) * lo[v];
        }
      }
    }
    if (owner && p == 0) LA.alpha_out[e] = alpha;
  }
  if (owner) {
#pragma unroll
    for (int v = 0; v < M; ++v) u_out[((int64_t)v * E + e) * n + p] = out[v];
  }
  if (RES) return;
  bool bad = false;
  if (owner) bad = SWE ? !positive_finite(out[0]) || !finite(out[M - 1]) : !finite(out[0]);
  if (bad) atomicOr(&st->status, 1u);
  if (!ctl.want_rate) return;
  // the next step's rate: element means by one thread per element (the speed
  // of advection is |a| averaged over the element)
  double* sm = reinterpret_cast<double*>(&X[0][0]);
  if (lane_ok) {
#pragma unroll
    for (int v = 0; v < M; ++v) sm[v * n + p] = SWE ? out[v] : sn;
  }
  __syncthreads();
  double rate = 0.0;
  for (int k = t; k < ne; k += blockDim.x) {
    if (k < 1 || k > ne - 2 || tile * (ne - 2) + k - 1 >= E) continue;
    const double* x = reinterpret_cast<const double*>(&sx[k][0][0]);
    double m[M];
#pragma unroll
    for (int v = 0; v < M; ++v) {
      m[v] = T.w[0] * x[v * n];
#pragma unroll
      for (int j = 1; j < n; ++j) m[v] = fma(T.w[j], x[v * n + j], m[v]);
    }
    if constexpr (SWE)
      rate = max_bits(rate, swe_speed(m[0], m[M - 1], T.sqrt_gravity) * xs);
    else
      rate = max_bits(rate, fabs(m[0]) * xs);
  }
  block_max_atomic_1d(rate, &st->rate[ctl.slot_write]);
}

// Resident blocks the register allocation must allow: 40 warps per SM (32 at N =
// 4) against 24 take the ensemble's step from 4.39 to 4.06 ms (two steps), and
// 1e5 elements at N = 4 from 389 to 382 us (four steps); the limited step, in
// 128-thread blocks, takes 16 warps.
template <int N>
__host__ __device__ constexpr int min_blocks_1d() {
  return N >= 4 ? 4 : 5;
}

template <int SYS, int N, bool GLL, bool RES, bool IMEX, bool LIMIT = false>
__global__ void __launch_bounds__(LIMIT ? kBlockLimit1D : kMaxBlock1D,
                                  LIMIT ? 4 : min_blocks_1d<N>()) k_step_1d(const Launch1D L) {
  chain_begin();
  step_1d_tile<SYS, N, GLL, RES, IMEX, LIMIT>(L.tab, L.xs, L.u_in, L.u_out, L.snode, L.sface, L.E,
                                              blockIdx.x, L.st, L.ctl, blockIdx.x == 0, true,
                                              L.lim, L.ghost);
}

// Several steps of a mesh that one cluster of blocks holds.  A step of a small
// mesh is a chain of latencies, and as a launch of its own a sixth of its time
// was the end of one kernel and the start of the next.  Here the blocks meet at
// the cluster's barrier between steps instead (release and acquire: the states,
// the rate and the time that a step writes are read by the next); the states
// alternate between two buffers as before, and every element's arithmetic is
// k_step_1d's.  Advection on 100 elements, 20 steps: 109 -> 91 us; shallow water,
// 8 steps: 150 elements at N = 4 90 -> 79 us, 490 at N = 1 60 -> 52 us (the
// largest mesh for N = 1, four warps an SM).
template <int SYS, int N, bool GLL, bool IMEX>
__global__ void __launch_bounds__(kMaxClusterThreads) k_steps_1d(const Launch1D L) {
  chain_begin();
  StepCtl ctl = L.ctl;
  const double* in = L.u_in;
  double *out = L.u_out, *next = L.u_next;
  for (int k = 0; k < L.steps; ++k) {
    if (k > 0) {
      asm volatile("barrier.cluster.arrive.release;\n\t"
                   "barrier.cluster.wait.acquire;" ::: "memory");
      in = out;
      out = next;
      next = const_cast<double*>(in);
      const int read = ctl.slot_read;
      ctl.slot_read = ctl.slot_write;
      ctl.slot_write = ctl.slot_reset;
      ctl.slot_reset = read;
      ctl.tslot ^= 1;
    }
    ctl.want_rate = k + 1 < L.steps ? !(ctl.dt_fixed > 0.0) : L.ctl.want_rate;
    step_1d_tile<SYS, N, GLL, false, IMEX>(L.tab, L.xs, in, out, L.snode, L.sface, L.E, blockIdx.x,
                                           L.st, ctl, blockIdx.x == 0, k + 1 == L.steps);
  }
}

// ragged ensembles: (instance, tile) pairs of a work list, a block taking
// items blockIdx.x, blockIdx.x + gridDim.x, ... (the grid size is a tuning
// parameter; the tile body's shared-memory phases are separated by barriers)
template <int SYS, int N, bool GLL, bool IMEX>
__global__ void __launch_bounds__(kBlock1D, min_blocks_1d<N>()) k_step_1d_batch(const LaunchBatch1D B) {
  for (int64_t wi = blockIdx.x; wi < B.nwork; wi += gridDim.x) {
    const WorkItem w = B.work[wi];
    const BatchInstance I = B.inst[w.inst];
    if (wi != blockIdx.x) __syncthreads();   // the previous tile's last reads
    step_1d_tile<SYS, N, GLL, false, IMEX>(B.tab, I.xs, B.u_in + I.u_off, B.u_out + I.u_off,
                                           B.snode + I.sn_off, B.sface + I.sf_off, I.E, w.tile,
                                           I.st, B.ctl, w.tile == 0, wi + gridDim.x >= B.nwork);
  }
}

// Threads per block of the step, chosen per mesh among kTileBlocks.  A block
// recomputes two halo elements, so large meshes take the largest block; a
// small mesh is spread over the SMs in smaller ones, since an SM sub-partition
// runs its warps' FP64 instructions one after the other: the step's time
// follows the warps of the busiest sub-partition, ceil(tiles / SMs) blocks of
// threads / 32 warps over four, and no less than one.  The larger block is
// taken among those within 2 % of the least such time.  crkfr_set_tile_1d can
// fix the size instead.
constexpr int kTileBlocks[4] = {32, 64, 128, 256};

inline int pick_tile_block(int64_t E, int n, int sms) {
  double cost[4], best = 0.0;
  for (int i = 0; i < 4; ++i) {
    const int64_t own = tile_elements_1d(kTileBlocks[i], n);
    const int64_t tiles = (E + own - 1) / own;
    const double warps = (double)((tiles + sms - 1) / sms) * (kTileBlocks[i] / 32) / 4.0;
    cost[i] = warps < 1.0 ? 1.0 : warps;
    if (i == 0 || cost[i] < best) best = cost[i];
  }
  int pick = 0;
  for (int i = 1; i < 4; ++i)
    if (cost[i] <= 1.02 * best || cost[pick] > 1.02 * best) pick = i;
  return kTileBlocks[pick];
}

// threads of the block, elements of the mesh: blocks of the launch (0: none fit)
inline unsigned tiles_1d(int64_t E, int threads, int n) {
  const int64_t own = tile_elements_1d(threads, n);
  const int64_t blocks = (E + own - 1) / own;
  return blocks > 0x7fffffff ? 0u : (unsigned)blocks;
}

template <int SYS, int N, bool GLL, bool IMEX>
int launch_steps_t(const Launch1D& L, cudaStream_t s) {
  const int threads = cluster_threads_1d(L.E, N + 1);
  if (!threads || !L.u_next || L.ghost) return (int)cudaErrorInvalidValue;
  const unsigned blocks = tiles_1d(L.E, threads, N + 1);
  return launch_chained_cluster(k_steps_1d<SYS, N, GLL, IMEX>, dim3(blocks), (unsigned)threads,
                                blocks, s, L);
}

template <int SYS, int N, bool GLL, bool IMEX>
int launch_step_t(const Launch1D& L, cudaStream_t s) {
  if (L.ctl.residual) {
    const unsigned blocks = tiles_1d(L.E, kBlock1D, N + 1);
    if (!blocks) return (int)cudaErrorInvalidConfiguration;
    return launch_chained(k_step_1d<SYS, N, GLL, true, IMEX>, dim3(blocks), kBlock1D, s, L);
  }
  if (L.steps > 1) return launch_steps_t<SYS, N, GLL, IMEX>(L, s);
  const int sms = sm_count();   // (unknown: the largest block)
  const int threads = L.tile_threads > 0 ? L.tile_threads
                      : sms > 0          ? pick_tile_block(L.E, N + 1, sms)
                                         : kBlock1D;
  const unsigned blocks = tiles_1d(L.E, threads, N + 1);
  if (!blocks) return (int)cudaErrorInvalidConfiguration;
  return launch_chained(k_step_1d<SYS, N, GLL, false, IMEX>, dim3(blocks), (unsigned)threads, s, L);
}

template <int SYS, bool IMEX>
int launch_step_sys(const Launch1D& L, cudaStream_t s) {
  switch (L.N * 2 + (L.gll ? 1 : 0)) {
    case 0: return launch_step_t<SYS, 0, false, IMEX>(L, s);
    case 2: return launch_step_t<SYS, 1, false, IMEX>(L, s);
    case 3: return launch_step_t<SYS, 1, true, IMEX>(L, s);
    case 4: return launch_step_t<SYS, 2, false, IMEX>(L, s);
    case 5: return launch_step_t<SYS, 2, true, IMEX>(L, s);
    case 6: return launch_step_t<SYS, 3, false, IMEX>(L, s);
    case 7: return launch_step_t<SYS, 3, true, IMEX>(L, s);
    case 8: return launch_step_t<SYS, 4, false, IMEX>(L, s);
    case 9: return launch_step_t<SYS, 4, true, IMEX>(L, s);
  }
  return (int)cudaErrorInvalidValue;
}

template <int SYS, int N, bool GLL, bool IMEX>
int launch_batch_t(const LaunchBatch1D& B, cudaStream_t s) {
  if (B.nwork <= 0) return 0;
  const int64_t blocks = B.grid > 0 && B.grid < B.nwork ? B.grid : B.nwork;
  k_step_1d_batch<SYS, N, GLL, IMEX><<<(unsigned)blocks, kBlock1D, 0, s>>>(B);
  return (int)cudaGetLastError();
}

template <int SYS, bool IMEX>
int launch_batch_sys(const LaunchBatch1D& B, cudaStream_t s) {
  switch (B.N * 2 + (B.gll ? 1 : 0)) {
    case 0: return launch_batch_t<SYS, 0, false, IMEX>(B, s);
    case 2: return launch_batch_t<SYS, 1, false, IMEX>(B, s);
    case 3: return launch_batch_t<SYS, 1, true, IMEX>(B, s);
    case 4: return launch_batch_t<SYS, 2, false, IMEX>(B, s);
    case 5: return launch_batch_t<SYS, 2, true, IMEX>(B, s);
    case 6: return launch_batch_t<SYS, 3, false, IMEX>(B, s);
    case 7: return launch_batch_t<SYS, 3, true, IMEX>(B, s);
    case 8: return launch_batch_t<SYS, 4, false, IMEX>(B, s);
    case 9: return launch_batch_t<SYS, 4, true, IMEX>(B, s);
  }
  return (int)cudaErrorInvalidValue;
}

}  // namespace
}  // namespace crkfr
