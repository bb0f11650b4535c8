// First-order part of the subcell blending limiter of the 2D shallow-water
// step (the tensor-product extension of Sec. 4), computed by the limited
// instantiation of the element-local kernel (local_2d.cuh) after the
// high-order part.  Subcells are w_p dx x w_q dy; every inner x- and
// y-subface carries the non-conservative Rusanov fluxes of
// Eq. combined.num.flux between its two nodal states.  The kernel writes the
// first-order update of every node without its element-face terms
// (Eq. low.order.update) and, for every face node, what the face kernel
// needs for the first-order face flux and Algorithm 1: the nodal state and
// coefficient next to the face, the inner subface flux of that node on its
// far side, and the trace of the coefficient.
#pragma once

#include <cuda_runtime.h>

#include "device_common.cuh"

namespace crkfr {
namespace {

constexpr int kLimFields = 8;     // limiter face data: u (3), c, inner flux (3), trace of c
constexpr int kLimExchange = 22;  // shared-memory fields per node (limit_local_2d)
template <int D>
struct LimDir {
  static constexpr int value = D;
};

// The first-order fluxes are carried doubled, 2 f (the means without their
// halves; scaling by two is exact), with the halves in the update's
// coefficients: 12 FP64 instructions a subface instead of 23.

// Per-node parts of a first-order flux in direction DIR (0: x, 1: y): the
// spectral radius |v_n| + sqrt(g h), the normal momentum's flux (with the
// pressure g h^2 / 2 in the standard form), the tangential momentum's flux,
// and g h.
template <int DIR, bool WB>
__device__ __forceinline__ void lo_node(const double* u, double g, double& s, double& fn,
                                        double& ft, double& gh) {
  constexpr int nv = 1 + DIR, nt = 2 - DIR;
  const double h = u[0];
  const double v = u[nv] * drcp(h);
  gh = g * h;
  s = fabs(v) + dsqrt_pos(gh);
  fn = WB ? u[nv] * v : fma(0.5 * gh, h, u[nv] * v);
  ft = u[nt] * v;
}

// Doubled non-conservative Rusanov fluxes (Eq. combined.num.flux) between the
// nodal states L and R from their per-node parts: fm = 2 (f^num + B(w_L) w^num),
// fp = 2 (f^num + B(w_R) w^num); the jump of h, or of eta = h + b in the
// well-balanced form, is dissipated.
template <int DIR, bool WB>
__device__ __forceinline__ void lo_flux_nodes(const double* uL, const double* uR, double cL,
                                              double cR, double sL, double sR, double fnL,
                                              double fnR, double ftL, double ftR, double ghL,
                                              double ghR, double* fm, double* fp) {
  constexpr int nv = 1 + DIR, nt = 2 - DIR;
  const double lam = max_nonneg(sL, sR);
  const double hL = uL[0], hR = uR[0];
  const double jh = WB ? (hR + cR) - (hL + cL) : hR - hL;
  double f[3];
  f[0] = fma(-lam, jh, uL[nv] + uR[nv]);
  f[nv] = fma(-lam, uR[nv] - uL[nv], fnL + fnR);
  f[nt] = fma(-lam, uR[nt] - uL[nt], ftL + ftR);
  const double wn = WB ? (hL + hR) + (cL + cR) : cL + cR;
#pragma unroll
  for (int v = 0; v < 3; ++v) {
    fm[v] = f[v];
    fp[v] = f[v];
  }
  fm[nv] = fma(ghL, wn, f[nv]);
  fp[nv] = fma(ghR, wn, f[nv]);
}

template <int DIR, bool WB>
__device__ __forceinline__ void lo_flux_2d(const double* uL, const double* uR, double cL,
                                           double cR, double g, double* fm, double* fp) {
  double sL, sR, fnL, fnR, ftL, ftR, ghL, ghR;
  lo_node<DIR, WB>(uL, g, sL, fnL, ftL, ghL);
  lo_node<DIR, WB>(uR, g, sR, fnR, ftR, ghR);
  lo_flux_nodes<DIR, WB>(uL, uR, cL, cR, sL, sR, fnL, fnR, ftL, ftR, ghL, ghR, fm, fp);
}

// The first-order part of the local kernel, one thread per node (node = q n +
// p of element ge).  u0: u^n at the node; x: the element's exchange area
// (kLimExchange fields); sync: the element's barrier, which every thread of
// the block (or warp) reaches.  The area holds, per node: 0..2 u^n, 3 c, 4..6
// the x parts and 7..9 the y parts of the node's first-order flux; 10..12 and
// 13..15 the doubled minus- and plus-side fluxes of the x subface to its right,
// 16..18 and 19..21 of the y subface above it.
template <int N, bool GLL, bool WB, class Sync>
__device__ __forceinline__ void limit_local_2d(const Launch2D& L, const double (&u0)[3], double* x,
                                               int node, bool lane_ok, bool active, int64_t ge,
                                               double dt, Sync sync) {
  constexpr int n = N + 1;
  constexpr int nn = n * n;
  const Tables& T = L.tab;
  const double g = T.gravity;
  const int64_t Ne = L.Ex * L.Ey;
  const int64_t tstride = Ne * n;
  const int q = node / n, p = node - q * n;
  auto X = [x](int f, int k) -> double& { return x[f * nn + k]; };

  const double gh = g * u0[0];
  if (lane_ok) {
    // the per-node parts of both directions (one reciprocal, one root)
    const double ih = drcp(u0[0]), a = dsqrt_pos(gh);
    const double vx = u0[1] * ih, vy = u0[2] * ih, hgh = 0.5 * gh;
#pragma unroll
    for (int v = 0; v < 3; ++v) X(v, node) = u0[v];
    X(3, node) = L.lim.cnode[ge * nn + node];
    X(4, node) = fabs(vx) + a;
    X(5, node) = WB ? u0[1] * vx : fma(hgh, u0[0], u0[1] * vx);
    X(6, node) = u0[2] * vx;
    X(7, node) = fabs(vy) + a;
    X(8, node) = WB ? u0[2] * vy : fma(hgh, u0[0], u0[2] * vy);
    X(9, node) = u0[1] * vy;
  }
  // coefficients of the update, with the halves of the doubled fluxes, by the
  // block's first warp
  __shared__ double half_dt[2][n];
  if (threadIdx.x < 2 * n) {
    const int d = threadIdx.x >= n, k = threadIdx.x - d * n;
    half_dt[d][k] = (0.5 * dt * (d ? T.inv_dy : T.inv_dx)) * T.inv_w[k];
  }
  sync();
  // the subfaces to the right of and above the node
  auto subface = [&](auto dir, int nb) {
    constexpr int D = decltype(dir)::value;
    double a[3], b[3], fm[3], fp[3];
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      a[v] = u0[v];
      b[v] = X(v, nb);
    }
    lo_flux_nodes<D, WB>(a, b, X(3, node), X(3, nb), X(4 + 3 * D, node), X(4 + 3 * D, nb),
                         X(5 + 3 * D, node), X(5 + 3 * D, nb), X(6 + 3 * D, node),
                         X(6 + 3 * D, nb), gh, g * b[0], fm, fp);
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      X(10 + 6 * D + v, node) = fm[v];
      X(13 + 6 * D + v, node) = fp[v];
    }
  };
  if (lane_ok) {
    if (p < N) subface(LimDir<0>{}, node + 1);
    if (q < N) subface(LimDir<1>{}, node + n);
  }
  __syncthreads();
  if (!active) return;
  // first-order update of the node without the element-face terms
  const double cx = half_dt[0][p], cy = half_dt[1][q];
#pragma unroll
  for (int v = 0; v < 3; ++v) {
    const double r = p < N ? X(10 + v, node) : 0.0;
    const double l = p > 0 ? X(13 + v, node - 1) : 0.0;
    const double t = q < N ? X(16 + v, node) : 0.0;
    const double b = q > 0 ? X(19 + v, node - n) : 0.0;
    L.lim.ulo[(v * Ne + ge) * nn + node] = u0[v] - cx * (r - l) - cy * (t - b);
  }
  // face data: the nodal state and c next to the face, the doubled inner flux of that
  // node on its far side, the trace of c; the 4 n face nodes as the traces
  const int64_t plane = L.Ex * n;
  const int64_t row = ge / L.Ex + 1, col = ge - (row - 1) * L.Ex;
#pragma unroll
  for (int j0 = 0; j0 < 4 * n; j0 += nn) {
    const int job = j0 + node;
    if (4 * n % nn != 0 && job >= 4 * n) break;
    const int dir = job / (2 * n), side = job / n & 1, r = job % n;
    const int step = dir ? n : 1, base = dir ? r : r * n;
    const int at = base + (side ? N * step : 0);          // the node next to the face
    const int sub = side ? at - step : at;                // its inner subface
    double d[kLimFields];
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      d[v] = X(v, at);
      d[4 + v] = X(10 + 6 * dir + 3 * side + v, sub);
    }
    d[3] = X(3, at);
    if (GLL) {
      d[7] = d[3];
    } else {
      double c = (side ? T.l1[0] : T.l0[0]) * X(3, base);
#pragma unroll
      for (int j = 1; j < n; ++j) c = fma(side ? T.l1[j] : T.l0[j], X(3, base + j * step), c);
      d[7] = c;
    }
    // y: buffer rows as the y traces (halo rows 0 and Ey+1 filled in a
    // periodic mesh)
    double* out = dir ? L.lim.ly + (row * 2 + side) * kLimFields * plane + col * n + r
                      : L.lim.lx + side * tstride + ge * n + r;
    const int64_t ostep = dir ? plane : 2 * tstride;
    const bool wrap = dir && L.periodic_y && row == (side ? L.Ey : 1);
    double* halo = L.lim.ly + (side ? 1 : (L.Ey + 1) * 2) * kLimFields * plane + col * n + r;
#pragma unroll
    for (int f = 0; f < kLimFields; ++f) {
      out[f * ostep] = d[f];
      if (wrap) halo[f * plane] = d[f];
    }
  }
}

}  // namespace
}  // namespace crkfr
