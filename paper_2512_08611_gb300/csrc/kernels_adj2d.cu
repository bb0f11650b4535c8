// Adjoint of one 2D shallow-water cRK-FR step (sm_103a, FP64).
//
// The forward step (kernels_2d.cu) is u^{n+1} = S(u^n; b) with a fixed dt.
// Given ubar^{n+1} = dJ/du^{n+1} this computes ubar^n = (dS/du^n)^T ubar^{n+1}
// and adds (dS/db)^T ubar^{n+1} to bbar.  It is the exact discrete adjoint of
// the kernels' arithmetic (reverse-mode differentiation written out by hand):
//
//  1. k_local_2d (forward) recomputes the face traces of u^n and its stage
//     values, unless a recorded step kept them;
//  2. k_face_adj_2d: once per face node, the adjoints of both sides' face
//     terms follow from the two elements' row (or column) sums of ubar^{n+1}
//     against the correction tables; they are pulled back through the
//     Rusanov flux, the wave-speed maximum and the frozen fluctuation
//     (Sec. 3, Eqs. numflux.cons, combined.wave.speed, good.numflux.non.cons,
//     total.F.non.cons) to adjoint traces of each side, and to the adjoint of
//     the static jump g (b+ - b-)/b_0;
//  3. k_local_adj_2d: per element, the inner stages are reversed: adjoint
//     traces -> time averages -> stage values -> local operator (transposed D_x,
//     D_y contractions) -> fluxes -> earlier stages and u^n; the bathymetry
//     enters through g b_x, g b_y and the face jumps, whose adjoints are mapped
//     back to the nodal b.
//
// Non-smooth points: |m/h| takes sign(0) = 0, and the maximum of the two wave
// speeds passes its adjoint to the side the forward kernel selected (the
// right side on a tie).
#include <cuda_runtime.h>

#include <algorithm>

#include "device_common.cuh"
#include "local_2d.cuh"

namespace crkfr {
namespace {

constexpr int kBlockAdj = 128;
constexpr int kTr = 7;

// d sigma / d h and d sigma / d m of sigma(h, m) = |m/h| + sqrt(g h), and
// sigma itself as the forward kernels compute it (so that the side of the
// maximum is the one the forward step selected).  sg = sqrt(g); with
// r1 = 1/sqrt(h): d sigma/dm = sign(m) / h, d sigma/dh = -|m|/h^2 + sg r1 / 2.
__device__ __forceinline__ void speed_grad(double h, double m, double sg, double* dh, double* dm,
                                           double* sigma) {
  const double r1 = drsqrt_pos(h);
  const double r = r1 * r1;
  const double v = m * r;
  const double s = v > 0.0 ? 1.0 : (v < 0.0 ? -1.0 : 0.0);
  *sigma = swe_speed(h, m, sg);
  *dm = s * r;
  *dh = fma(-s * v, r, 0.5 * sg * r1);
}

// Adjoint of the doubled face terms of one face node.  tm/tp: the two sides'
// traces (fields as in kernels_2d.cu); Tbm/Tbp: adjoints of T'^- and T'^+;
// outputs the adjoint traces of both sides and the adjoint of gdb.
__device__ __forceinline__ void face_terms_adj(const double* tm, const double* tp, int nv,
                                               double gdb, double sg, const double* Tbm,
                                               const double* Tbp, double* am, double* ap,
                                               double* gdb_bar) {
  double dhm, dmm, sm, dhp, dmp, sp;
  speed_grad(tm[5], tm[6], sg, &dhm, &dmm, &sm);
  speed_grad(tp[5], tp[6], sg, &dhp, &dmp, &sp);
  const bool left = sm > sp;   // the forward maximum picks the right side on a tie
  const double lam = left ? sm : sp;
#pragma unroll
  for (int f = 0; f < kTr; ++f) am[f] = ap[f] = 0.0;
  double lam_bar = 0.0;
  // Tm_v = dF_v - lam dU_v,  Tp_v = -(dF_v + lam dU_v)
#pragma unroll
  for (int v = 0; v < 3; ++v) {
    const double dU = tp[v] - tm[v];
    const double s = Tbm[v] + Tbp[v];
    const double dF_bar = Tbm[v] - Tbp[v];
    const double dU_bar = -lam * s;
    lam_bar = fma(-dU, s, lam_bar);
    ap[v] += dU_bar;
    am[v] -= dU_bar;
    const int ff = v == 0 ? nv : (v == 1 ? 3 : 4);
    ap[ff] += dF_bar;
    am[ff] -= dF_bar;
  }
  // fluctuations: Tm_nv += h^- gdb, Tp_nv -= h^+ gdb
  am[5] = fma(Tbm[nv], gdb, am[5]);
  ap[5] = fma(-Tbp[nv], gdb, ap[5]);
  *gdb_bar = fma(Tbm[nv], tm[5], -Tbp[nv] * tp[5]);
  if (left) {
    am[5] = fma(lam_bar, dhm, am[5]);
    am[6] = fma(lam_bar, dmm, am[6]);
  } else {
    ap[5] = fma(lam_bar, dhp, ap[5]);
    ap[6] = fma(lam_bar, dmp, ap[6]);
  }
}

template <int N>
__global__ void __launch_bounds__(256) k_face_adj_2d(const Launch2DAdj A) {
  constexpr int n = N + 1;
  constexpr int nn = n * n;
  const Tables& T = A.tab;
  const int64_t Ex = A.Ex, Ey = A.Ey, Ne = Ex * Ey, ts = Ne * n, plane = Ex * n;
  const double dtb0 = A.dt * Tab<N, false>::bref();
  const bool slab = A.sums_below != nullptr;
  const int64_t total = Ne * n + (slab ? Ey + 1 : Ey) * plane;   // x faces, y faces
  for (int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; f < total;
       f += (int64_t)gridDim.x * blockDim.x) {
    const bool xdir = f < Ne * n;
    const int64_t g = xdir ? f : f - Ne * n;
    const int k = (int)(g % n);                 // node along the face
    const int64_t e = g / n;                    // plus-side element
    const int64_t ey = e / Ex, ex = e - ey * Ex;
    double tm[kTr], tp[kTr], Tbm[3], Tbp[3], am[kTr], ap[kTr], gbar;
    if (xdir) {
      const int64_t em = ey * Ex + (ex == 0 ? Ex - 1 : ex - 1);
#pragma unroll
      for (int v = 0; v < 3; ++v) {
        const double* um = A.ubar1 + (v * Ne + em) * nn + k * n;   // row k of the left element
        const double* up = A.ubar1 + (v * Ne + e) * nn + k * n;
        double sm = um[0] * T.gRx[0], sp = up[0] * T.gLx[0];
#pragma unroll
        for (int p = 1; p < n; ++p) {
          sm = fma(um[p], T.gRx[p], sm);
          sp = fma(up[p], T.gLx[p], sp);
        }
        Tbm[v] = -dtb0 * sm;
        Tbp[v] = -dtb0 * sp;
      }
#pragma unroll
      for (int fi = 0; fi < kTr; ++fi) {
        tm[fi] = A.trx[(2 * fi + 1) * ts + em * n + k];
        tp[fi] = A.trx[(2 * fi + 0) * ts + e * n + k];
      }
      face_terms_adj(tm, tp, 1, A.sface[e * n + k], T.sqrt_gravity, Tbm, Tbp, am, ap, &gbar);
#pragma unroll
      for (int fi = 0; fi < kTr; ++fi) {
        A.atrx[(2 * fi + 1) * ts + em * n + k] = am[fi];
        A.atrx[(2 * fi + 0) * ts + e * n + k] = ap[fi];
      }
      A.gbar[e * n + k] = gbar;
    } else {
      // the face below element row ey (on a slab ey = 0 .. Ey: rows -1 and
      // Ey are the neighbouring slabs', whose sums came with the exchange)
      const int64_t rowm = slab ? ey - 1 : (ey == 0 ? Ey - 1 : ey - 1);
#pragma unroll
      for (int v = 0; v < 3; ++v) {
        double sm, sp;
        if (rowm >= 0) {
          const double* um = A.ubar1 + (v * Ne + rowm * Ex + ex) * nn + k;   // column k, lower
          sm = um[0] * T.gRy[0];
#pragma unroll
          for (int q = 1; q < n; ++q) sm = fma(um[q * n], T.gRy[q], sm);
        } else {
          sm = A.sums_below[(v * Ex + ex) * n + k];
        }
        if (ey < Ey) {
          const double* up = A.ubar1 + (v * Ne + ey * Ex + ex) * nn + k;     // column k, upper
          sp = up[0] * T.gLy[0];
#pragma unroll
          for (int q = 1; q < n; ++q) sp = fma(up[q * n], T.gLy[q], sp);
        } else {
          sp = A.sums_above[(v * Ex + ex) * n + k];
        }
        Tbm[v] = -dtb0 * sm;
        Tbp[v] = -dtb0 * sp;
      }
      // forward y traces: element row r in buffer row r+1 (rows 0, Ey+1 halos)
#pragma unroll
      for (int fi = 0; fi < kTr; ++fi) {
        tm[fi] = A.try_[((ey * 2 + 1) * kTr + fi) * plane + ex * n + k];
        tp[fi] = A.try_[(((ey + 1) * 2 + 0) * kTr + fi) * plane + ex * n + k];
      }
      face_terms_adj(tm, tp, 2, A.sface[Ne * n + ey * plane + ex * n + k], T.sqrt_gravity, Tbm,
                     Tbp, am, ap, &gbar);
      // adjoint y traces: [row][side][field][ex][node], no halo rows (the
      // sides of a neighbouring slab's elements are that slab's to compute)
#pragma unroll
      for (int fi = 0; fi < kTr; ++fi) {
        if (rowm >= 0) A.atry[((rowm * 2 + 1) * kTr + fi) * plane + ex * n + k] = am[fi];
        if (ey < Ey) A.atry[((ey * 2 + 0) * kTr + fi) * plane + ex * n + k] = ap[fi];
      }
      A.gbar[Ne * n + ey * plane + ex * n + k] = gbar;
    }
  }
}

// Exchange area of the adjoint local kernel per element, in doubles: the
// adjoint traces [dir][side][field][node], or a stage's operator adjoints.
template <int n>
__host__ __device__ constexpr int adjoint_stride() {
  return ((4 * kTr * n > 3 * n * n ? 4 * kTr * n : 3 * n * n) + 11) / 16 * 16 + 4;
}

// One thread per node, as k_local_2d: the pointwise reverse arithmetic in FP64
// (some 30 instructions a stage), the transposed contractions with D and the
// products with the end-point rows, more than half of the FP64 instructions
// before, in block fixed point (fixed_point.cuh).  256 x 256 at N = 3: 308 us,
// bound by the FP64 pipe (83 % busy), against 547 us with a thread per element
// row and FP64 chains (255 registers).
template <int N>
__global__ void __launch_bounds__(kBlockAdj, 5) k_local_adj_2d(const Launch2DAdj A) {
  using TB = Tab<N, false>;
  constexpr int n = N + 1;
  constexpr int nn = n * n;
  constexpr int S = TB::S;
  constexpr int EPB = kBlockAdj / nn;
  constexpr int ES = adjoint_stride<n>();
  constexpr int FB = 59, kHeadroom = 1;
  constexpr bool WARP = 32 % nn == 0;
  // as in k_local_2d: the stage loop unrolled for the short tableaux, else
  // rolled with the later stages' adjoints in a register (RK4) or shared memory
  constexpr bool UNROLL = local_unrolled<N, false>(), CHAIN = !UNROLL && local_chain<TB>();
  constexpr bool SHARED = !UNROLL && !CHAIN;
  constexpr int kStageUnroll = UNROLL ? S : 1;
  const Tables& T = A.tab;
  __shared__ __align__(16) double sm[EPB * ES];
  __shared__ int smag[EPB][2 * kTr];
  __shared__ StepSizes<TB> sz;
  __shared__ double sC[SHARED ? S : 1][3][SHARED ? kBlockAdj : 1];

  const int le_raw = threadIdx.x / nn, node = threadIdx.x - le_raw * nn;
  const int q = node / n, p = node - q * n;
  const int64_t Ex = A.Ex, Ey = A.Ey, Ne = Ex * Ey, ts = Ne * n, plane = Ex * n;
  const int64_t r0 = A.row_begin * Ex, Nr = (A.row_end - A.row_begin) * Ex;
  const bool lane_ok = le_raw < EPB;
  const int le = lane_ok ? le_raw : 0;
  const int64_t g = (int64_t)blockIdx.x * EPB + le;
  const bool active = lane_ok && g < Nr;
  const int64_t gr = active ? g : 0, ge = r0 + gr;
  const int64_t ey = ge / Ex, ex = ge - ey * Ex;
  Fx* const X = reinterpret_cast<Fx*>(&sm[le * ES]);
  auto sync = [] {
    if (WARP)
      __syncwarp();
    else
      __syncthreads();
  };
  auto sync_or = [](bool b) -> bool {
    return WARP ? warp_barrier_or(b) : __syncthreads_or(b);
  };

  if (threadIdx.x < 32) fill_step_sizes<TB, false>(sz, A.dt, 1.0);
  if (lane_ok) {
    for (int k = node; k < 2 * kTr; k += nn) smag[le][k] = 0;
  }
  const double gbx = A.snode[ge * nn + node], gby = A.snode[(Ne + ge) * nn + node];
  int dxh[n], dxl[n], dyh[n], dyl[n];   // columns p of D_x, q of D_y
#pragma unroll
  for (int j = 0; j < n; ++j) {
    dxh[j] = T.fx.Dx_hi[j][p];
    dxl[j] = T.fx.Dx_lo[j][p];
    dyh[j] = T.fx.Dy_hi[j][q];
    dyl[j] = T.fx.Dy_lo[j][q];
  }
  __syncthreads();

  // ---- adjoints of the time averages from W and the face traces ------------
  // W = u0 - dt b0 V  ->  ubar0 = Wbar,  Vbar = -dt b0 Wbar
  double ub0[3], Vb[3], Ub[3], F2b, F3b, G3b;
#pragma unroll
  for (int v = 0; v < 3; ++v) {
    ub0[v] = A.ubar1[(v * Ne + ge) * nn + node];
    Vb[v] = -sz.dtb * ub0[v];
  }
  // A trace field X gets l0[p] tbar_left + l1[p] tbar_right from the x faces
  // of its row and l0[q] tbar_bottom + l1[q] tbar_top from the y faces of its
  // column.  The 4 n face nodes of the element, 7 fields each, one thread per
  // face node; an exponent per direction and field.
  {
    constexpr int J = (4 * n + nn - 1) / nn;
    double t[J][kTr];
#pragma unroll
    for (int jj = 0; jj < J; ++jj) {
      const int job = jj * nn + node;
      if (4 * n % nn != 0 && job >= 4 * n) break;
      const int dir = job / (2 * n), side = job / n & 1, r = job % n;
      const double* in = dir ? A.atry + (ey * 2 + side) * kTr * plane + ex * n + r
                             : A.atrx + side * ts + ge * n + r;
      const int64_t step = dir ? plane : 2 * ts;
#pragma unroll
      for (int fi = 0; fi < kTr; ++fi) {
        t[jj][fi] = in[fi * step];
        if (lane_ok) atomicMax(&smag[le][dir * kTr + fi], fx_mag(t[jj][fi]));
      }
    }
    sync();
    auto E = [&](int k) { return fx_exp(smag[le][k]); };   // k = direction kTr + field
#pragma unroll
    for (int jj = 0; jj < J; ++jj) {
      const int job = jj * nn + node;
      if (4 * n % nn != 0 && job >= 4 * n) break;
      const int ds = job / n, r = job % n;   // direction and side, node of the face
#pragma unroll
      for (int fi = 0; fi < kTr; ++fi) {
        if (lane_ok)
          X[(ds * kTr + fi) * n + r] =
              fx_split(fx_from<FB>(t[jj][fi], E((ds >> 1) * kTr + fi)));
      }
    }
    sync();
    // products of field fx from the x faces, fy from the y faces (negative: none)
    auto pull = [&](int fx, int fy) -> double {
      FxAcc a{0, 0}, b{0, 0};
      const int ex = fx >= 0 ? E(fx) : 0, ey = fy >= 0 ? E(kTr + fy) : 0;
      if (fx >= 0) {
        fx_mad(a, X[fx * n + q], T.fx.l0_hi[p], T.fx.l0_lo[p]);
        fx_mad(a, X[(kTr + fx) * n + q], T.fx.l1_hi[p], T.fx.l1_lo[p]);
      }
      if (fy >= 0) {
        fx_mad(b, X[(2 * kTr + fy) * n + p], T.fx.l0_hi[q], T.fx.l0_lo[q]);
        fx_mad(b, X[(3 * kTr + fy) * n + p], T.fx.l1_hi[q], T.fx.l1_lo[q]);
      }
      int e = fx >= 0 ? ex : ey;
      const long long s = fx < 0   ? fx_sum(b)
                          : fy < 0 ? fx_sum(a)
                                   : fx_align(fx_sum(a), ex, fx_sum(b), ey, e);
      return fx_to(s, e + T.fx.kL - FB, fx_zero(max(ex, ey)));
    };
    Ub[0] = pull(0, 0);
    Ub[1] = pull(1, 1);
    Ub[2] = pull(2, 2);
    F2b = pull(3, -1);
    F3b = pull(4, 3);
    G3b = pull(-1, 4);
    ub0[0] += pull(5, 5);
    ub0[1] += pull(6, -1);
    ub0[2] += pull(-1, 6);
  }
  sync();
  if (lane_ok) {
    for (int k = node; k < 3; k += nn) smag[le][k] = 0;
  }
  sync();

  // ---- reverse through the stages -------------------------------------------
  double gbxb = 0.0, gbyb = 0.0;
  double cb[3] = {0.0, 0.0, 0.0};        // adjoint of the stage value just reversed
  double rC[UNROLL ? S : 1][3];          // of every later stage
  int E[3] = {-1, -1, -1};               // exponents of the adjoints of L
  // column p of D_x on exchange field fx plus column q of D_y on field fy
  // (negative: none)
  auto contract = [&](int fx, int fy) -> double {
    FxAcc a{0, 0}, b{0, 0};
    const int ex = fx >= 0 ? E[fx >= 0 ? fx : 0] : -1, ey = fy >= 0 ? E[fy >= 0 ? fy : 0] : -1;
    if (fx >= 0) {
#pragma unroll
      for (int j = 0; j < n; ++j) fx_mad(a, X[fx * nn + q * n + j], dxh[j], dxl[j]);
    }
    if (fy >= 0) {
#pragma unroll
      for (int j = 0; j < n; ++j) fx_mad(b, X[fy * nn + j * n + p], dyh[j], dyl[j]);
    }
    int e = fx >= 0 ? ex + T.fx.kDx : ey + T.fx.kDy;
    const long long s =
        fx < 0   ? fx_sum(b)
        : fy < 0 ? fx_sum(a)
                 : fx_align(fx_sum(a), ex + T.fx.kDx, fx_sum(b), ey + T.fx.kDy, e);
    return fx_to(s, e - FB, fx_zero(max(ex, ey)));
  };
  // fields to shared memory in the fixed point of each field and element
  auto publish = [&](const double (&f)[3]) {
    bool over = false;
#pragma unroll
    for (int k = 0; k < 3; ++k) over = over || (lane_ok && fx_mag(f[k]) >> 20 > E[k]);
    if (sync_or(over)) {
      if (over) {
#pragma unroll
        for (int k = 0; k < 3; ++k) atomicMax(&smag[le][k], fx_mag(f[k]));
      }
      sync();
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int e = fx_exp(smag[le][k]);
        E[k] = e > E[k] ? e + kHeadroom : E[k];
      }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k)
      if (lane_ok) X[k * nn + node] = fx_split(fx_from<FB>(f[k], E[k]));
    sync();
  };
#pragma unroll kStageUnroll
  for (int i = S - 1; i >= 0; --i) {
    const double wi = (double)local_weight<TB>(i);
    // adjoint of the stage's operator: cur_k = u0 - sum_j dt a_kj L_j
    double Lb[3];
#pragma unroll
    for (int v = 0; v < 3; ++v) Lb[v] = wi * Vb[v];
    if constexpr (CHAIN) {
      if (i < S - 1) {
        const double c = sz.e[i + 1][i];
#pragma unroll
        for (int v = 0; v < 3; ++v) Lb[v] = fma(c, cb[v], Lb[v]);
      }
    } else if constexpr (SHARED) {
      for (int k = S - 1; k > i; --k) {
        if (!(local_nonzero<TB>() >> (8 * k + i) & 1)) continue;
        const double c = sz.e[k][i];
#pragma unroll
        for (int v = 0; v < 3; ++v) Lb[v] = fma(c, sC[k][v][threadIdx.x], Lb[v]);
      }
    } else {
#pragma unroll
      for (int k = S - 1; k >= 0; --k)
        if (k > i && TB::a(k, i) != 0.0) {
#pragma unroll
          for (int v = 0; v < 3; ++v) Lb[v] = fma(sz.e[k][i], rC[k][v], Lb[v]);
        }
    }
    // the stage value, as the forward local kernel stored it
    const double* stage = i == 0 ? A.u + ge * nn + node
                                 : A.stages + ((int64_t)(i - 1) * 3 * Nr + gr) * nn + node;
    const int64_t vstep = (i == 0 ? Ne : Nr) * nn;
    const double h = stage[0], mx = stage[vstep], my = stage[2 * vstep];
    publish(Lb);
    // local operator L_i = Dx f + Dy g + h (g b_x, g b_y): transposed contractions
    const double mxb = contract(0, -1), myb = contract(-1, 0);
    const double f2b = fma(wi, F2b, contract(1, -1));
    const double f3b = fma(wi, F3b, contract(2, 1));
    const double g3b = fma(wi, G3b, contract(-1, 2));
    // nonconservative terms h g b_x, h g b_y and the fluxes
    // f2 = mx vx + g h^2/2, f3 = mx vy, g3 = my vy + g h^2/2
    gbxb = fma(h, Lb[1], gbxb);
    gbyb = fma(h, Lb[2], gbyb);
    const double r = drcp(h);
    const double vx = mx * r, vy = my * r;
    const double s1 = fma(vy, f3b, vx * f2b), t = vy * g3b;
    double hb = fma(gbx, Lb[1], gby * Lb[2]);
    hb = fma(T.gravity * h, f2b + g3b, hb);
    hb = fma(-vx, s1, hb);
    hb = fma(-vy, t, hb);
    cb[0] = fma(wi, Ub[0], hb);
    cb[1] = fma(wi, Ub[1], fma(vx, f2b, s1 + mxb));
    cb[2] = fma(wi, Ub[2], fma(vx, f3b, fma(2.0, t, myb)));
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      ub0[v] += cb[v];
      if (UNROLL) rC[i][v] = cb[v];
      if (SHARED) sC[i][v][threadIdx.x] = cb[v];
    }
  }

  // ---- outputs: ubar^n and the bathymetry adjoint -----------------------------
  if (active) {
#pragma unroll
    for (int v = 0; v < 3; ++v) A.ubar0[(v * Ne + ge) * nn + node] = ub0[v];
  }
  // g b_x = g sum_j Dx[p][j] b(q, j): bbar(q, j) += g sum_p Dx[p][j] gbxbar(q, p),
  // and across rows for g b_y
  const double gb2[3] = {0.0, gbxb, gbyb};
  sync();
  if (lane_ok) {
    for (int k = node; k < 3; k += nn) smag[le][k] = 0;
  }
  sync();
  E[0] = E[1] = E[2] = -1;
  publish(gb2);
  double bb = T.gravity * contract(1, 2);
  // face jumps (g / b_0)(b+ - b-): left / right x faces of row q, bottom / top
  // y faces of column p
  {
    const int64_t exr = ex == Ex - 1 ? 0 : ex + 1;
    // jump row of the top face: row Ey is the periodic top, or on a slab the
    // top face itself
    const int64_t rowt = (ey + 1 == Ey && !A.sums_below) ? 0 : ey + 1;
    double s = fma(T.l0[p], A.gbar[ge * n + q], -T.l1[p] * A.gbar[(ey * Ex + exr) * n + q]);
    s = fma(T.l0[q], A.gbar[Ne * n + ey * plane + ex * n + p], s);
    s = fma(-T.l1[q], A.gbar[Ne * n + rowt * plane + ex * n + p], s);
    bb = fma(T.face_g, s, bb);
  }
  if (active) A.bbar[ge * nn + node] += bb;
}

template <int N, bool GLL>
int launch_local_stages_t(const Launch2D& L, cudaStream_t s) {
  constexpr int per_block = local_elements<N + 1>();
  const int64_t blocks = ((L.row_end - L.row_begin) * L.Ex + per_block - 1) / per_block;
  if (blocks > 0x7fffffff) return (int)cudaErrorInvalidConfiguration;
  if (L.ctl.residual)
    k_local_2d<N, GLL, true, false, false, false, true><<<(unsigned)blocks, kBlockLocal, 0, s>>>(L);
  else
    k_local_2d<N, GLL, false, false, false, false, true><<<(unsigned)blocks, kBlockLocal, 0, s>>>(L);
  return (int)cudaGetLastError();
}

// The y-correction sums of ubar1 a neighbouring slab's face adjoint needs:
// side 0 the slab's bottom row with g_L' (for the slab below), side 1 its
// top row with g_R' (for the slab above); send [2][3][Ex][n].  The same
// products in the same order as the face adjoint kernel forms them.
__global__ void k_adjoint_sums_2d(int n, int64_t Ex, int64_t Ey, const double* __restrict__ ubar1,
                                  const Tables T, double* __restrict__ send) {
  const int64_t per = 3 * Ex * n;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 2 * per) return;
  const int side = (int)(i / per);
  const int64_t j = i - side * per;
  const int v = (int)(j / (Ex * n));
  const int64_t ex = (j / n) % Ex;
  const int k = (int)(j % n);
  const int64_t Ne = Ex * Ey, nn = (int64_t)n * n;
  const int64_t row = side ? Ey - 1 : 0;
  const double* u = ubar1 + (v * Ne + row * Ex + ex) * nn + k;
  const double* g = side ? T.gRy : T.gLy;
  double sum = u[0] * g[0];
  for (int q = 1; q < n; ++q) sum = fma(u[q * n], g[q], sum);
  send[i] = sum;
}

}  // namespace

int launch_adjoint_sums_2d(int N, int64_t Ex, int64_t Ey, const double* ubar1, const Tables& T,
                           double* send, void* stream) {
  const int64_t total = 2 * 3 * Ex * (N + 1);
  k_adjoint_sums_2d<<<(unsigned)((total + 255) / 256), 256, 0, (cudaStream_t)stream>>>(
      N + 1, Ex, Ey, ubar1, T, send);
  return (int)cudaGetLastError();
}

int launch_adjoint_faces_2d(const Launch2DAdj& A, void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
  const int n = A.N + 1;
  const int64_t faces = A.Ex * A.Ey * n + (A.sums_below ? A.Ey + 1 : A.Ey) * A.Ex * n;
  const unsigned blocks = (unsigned)std::min<int64_t>((faces + 255) / 256, 152 * 16);
  switch (A.N) {
    case 1: k_face_adj_2d<1><<<blocks, 256, 0, s>>>(A); break;
    case 2: k_face_adj_2d<2><<<blocks, 256, 0, s>>>(A); break;
    case 3: k_face_adj_2d<3><<<blocks, 256, 0, s>>>(A); break;
    case 4: k_face_adj_2d<4><<<blocks, 256, 0, s>>>(A); break;
    default: return (int)cudaErrorInvalidValue;
  }
  return (int)cudaGetLastError();
}

int launch_adjoint_local_2d(const Launch2DAdj& A, void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
  if (A.row_begin < 0 || A.row_end <= A.row_begin || A.row_end > A.Ey || !A.stages)
    return (int)cudaErrorInvalidValue;
  const int per_block = kBlockAdj / ((A.N + 1) * (A.N + 1));
  const unsigned blocks =
      (unsigned)(((A.row_end - A.row_begin) * A.Ex + per_block - 1) / per_block);
  switch (A.N) {
    case 1: k_local_adj_2d<1><<<blocks, kBlockAdj, 0, s>>>(A); break;
    case 2: k_local_adj_2d<2><<<blocks, kBlockAdj, 0, s>>>(A); break;
    case 3: k_local_adj_2d<3><<<blocks, kBlockAdj, 0, s>>>(A); break;
    case 4: k_local_adj_2d<4><<<blocks, kBlockAdj, 0, s>>>(A); break;
    default: return (int)cudaErrorInvalidValue;
  }
  return (int)cudaGetLastError();
}

int launch_local_2d_stages(const Launch2D& L, void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
  if (L.row_begin < L.stage_row0 || L.row_end <= L.row_begin ||
      L.row_end > L.stage_row0 + L.stage_rows || L.row_end > L.Ey || !L.stages)
    return (int)cudaErrorInvalidValue;
  switch (L.N * 2 + (L.gll ? 1 : 0)) {
    case 2: return launch_local_stages_t<1, false>(L, s);
    case 3: return launch_local_stages_t<1, true>(L, s);
    case 4: return launch_local_stages_t<2, false>(L, s);
    case 5: return launch_local_stages_t<2, true>(L, s);
    case 6: return launch_local_stages_t<3, false>(L, s);
    case 7: return launch_local_stages_t<3, true>(L, s);
    case 8: return launch_local_stages_t<4, false>(L, s);
    case 9: return launch_local_stages_t<4, true>(L, s);
  }
  return (int)cudaErrorInvalidValue;
}

}  // namespace crkfr
