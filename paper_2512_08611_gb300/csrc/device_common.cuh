// Device helpers shared by the 1D and 2D kernels of libcrkfr.
//
// On GB300 the FP64 pipe issues about one warp instruction per 16 SM cycles
// (two FP64 FMA lanes per SM), some 60x below FP32, and a partly masked warp
// costs the same as a full one.  These helpers therefore keep FP64
// instructions to the minimum and push everything that can be exact elsewhere
// (reciprocals and roots, comparisons, maxima of non-negative values) onto the
// FP32 and integer pipes.
#pragma once

#include <cstdint>

#include "crkfr_internal.h"
#include "tableau.h"

namespace crkfr {

// The elementary operations below work on the significand as integers: an
// FP64 instruction holds the FP64 pipe 64 cycles a warp, an IMAD.WIDE the
// integer pipe 2, so the third-order refinement of an FP32 seed costs about 30
// integer instructions (some 45 cycles) instead of 3 (reciprocal) or 5 (roots)
// FP64 ones (192, 320 cycles), and being exact up to 2^-58 it ends within 0.51
// (1/x), 0.52 (1/sqrt) and 0.58 (sqrt) ulp.

// 2^23 y for the FP32 seed y in (1/2, 1], lowered by 2^-22 so that it stays
// below 2^23
__device__ __forceinline__ unsigned seed_bits(float y) {
  return (unsigned)__float_as_int(fmaf(y, 8388606.0f, 8388608.0f)) - 0x4b000000u;
}

// (r s) 2^-32 for r < 2^23 and a signed s
__device__ __forceinline__ long long seed_times(unsigned r, long long s) {
  return (long long)(int)r * (int)(s >> 32) +
         (long long)(((unsigned long long)r * (unsigned)s) >> 32);
}

// 2^62 / m for the significand m in [1, 2) of a normal x = (hi, lo): with a
// seed r of 1/m, p = m r - 1 is formed exactly (2^75 p fits 64 bits since |p| <
// 2^-20), and 1/m = r (1 - p + p^2) up to p^3 < 2^-60.
__device__ __forceinline__ unsigned long long recip_bits(unsigned hi, unsigned lo) {
  const unsigned mh = (hi & 0xfffffu) | 0x100000u;
  float f = __int_as_float((int)((__funnelshift_l(lo, hi, 3) & 0x7fffffu) | 0x3f800000u));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"(f));
  const unsigned r = seed_bits(f);
  const long long p =
      (long long)((unsigned long long)lo * r + ((unsigned long long)(mh * r) << 32));
  const int ph = (int)(p >> 25);                              // 2^50 p
  const long long s = (((long long)ph * ph) >> 25) - p;       // 2^75 (p^2 - p)
  return ((unsigned long long)r << 39) + (unsigned long long)(seed_times(r, s) >> 4);
}

// 1/x for FP64 x.  Zero, denormal and non-finite x, and x whose reciprocal is
// not normal, take the IEEE division.
__device__ __forceinline__ double drcp(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int ex = (int)(hi >> 20) & 0x7ff;
  if ((unsigned)(ex - 1) > 2043u) return 1.0 / x;
  const unsigned long long R = recip_bits(hi, lo) + 0x100u;
  const unsigned oh = ((unsigned)(R >> 41) + ((unsigned)(2044 - ex) << 20)) | (hi & 0x80000000u);
  return __hiloint2double((int)oh, (int)(unsigned)(R >> 9));
}

// 2^58 / sqrt(m) of x = m 4^k with 1 <= m < 4, m = (mh, ml) 2^-52: with a seed
// y, p = m y^2 - 1 (2^66 p, truncated), 1/sqrt(m) = y (1 - p/2 + 3 p^2/8).
__device__ __forceinline__ unsigned long long rsqrt_bits(double x, unsigned& mh, unsigned& ml,
                                                         int& k) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int ex = (int)(hi >> 20);
  const unsigned odd = ~(unsigned)ex & 1u;                    // ex - 1023 odd
  mh = __funnelshift_l(lo, (hi & 0xfffffu) | 0x100000u, odd);
  ml = lo << odd;
  k = (ex - 1023 - (int)odd) >> 1;
  float f = __int_as_float((int)(((__funnelshift_l(lo, hi, 3) & 0x7fffffu) | 0x3f800000u) +
                                 (odd << 23)));
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"(f));
  const unsigned y = seed_bits(f);
  const unsigned long long Q = (unsigned long long)y * y;
  const unsigned qh = (unsigned)(Q >> 32), ql = (unsigned)Q;
  const long long p =
      (long long)(((unsigned long long)ml * ql >> 32) + (unsigned long long)mh * ql +
                  (unsigned long long)ml * qh + ((unsigned long long)(mh * qh) << 32));
  const int ph = (int)(p >> 17);                              // 2^49 p
  const int t = (int)(((long long)ph * ph) >> 32);            // 2^66 p^2
  const long long s = (long long)((3 * t) >> 2) - p;          // 2^67 (3 p^2/8 - p/2)
  return ((unsigned long long)y << 35) + (unsigned long long)seed_times(y, s);
}

// positive, normal and finite (the range of the two roots below)
__device__ __forceinline__ bool positive_normal(double x) {
  return (unsigned)__double2hiint(x) - 0x100000u < 0x7fe00000u;
}

// 1/sqrt(x) for FP64 x > 0; other x take the IEEE operations.
__device__ __forceinline__ double drsqrt_pos(double x) {
  if (!positive_normal(x)) return 1.0 / sqrt(x);
  unsigned mh, ml;
  int k;
  const unsigned long long q = (rsqrt_bits(x, mh, ml, k) + 0x10u) >> 5;
  return __longlong_as_double((long long)(q + ((unsigned long long)(unsigned)(1021 - k) << 52)));
}

// sqrt(x) for FP64 x > 0, as m (1/sqrt(m)); other x take the IEEE square root.
__device__ __forceinline__ double dsqrt_pos(double x) {
  if (!positive_normal(x)) return sqrt(x);
  unsigned mh, ml;
  int k;
  const unsigned long long R = rsqrt_bits(x, mh, ml, k);
  const unsigned rh = (unsigned)(R >> 32), rl = (unsigned)R;
  const unsigned long long low = ((unsigned long long)ml * rl >> 32) +
                                 (unsigned long long)mh * rl + (unsigned long long)ml * rh;
  const unsigned long long top = (unsigned long long)mh * rh + (low >> 32);   // 2^46 sqrt(m)
  const unsigned long long q = (top << 6) + ((((unsigned)low >> 25) + 1) >> 1);
  return __longlong_as_double((long long)(q + ((unsigned long long)(unsigned)(1022 + k) << 52)));
}

// sigma(f' + B) of shallow water in one direction, |m/h| + sqrt(g h), as
// r (|m| r + sqrt(g) h) with r = 1/sqrt(h): eight FP64 instructions (one
// reciprocal square root) instead of a reciprocal and a square root.
// sg = sqrt(g).
__device__ __forceinline__ double swe_speed(double h, double m, double sg) {
  const double r = drsqrt_pos(h);
  return fma(sg, h, fabs(m) * r) * r;
}

// sigma_x / dx + sigma_y / dy of the element means (h, hu, hv) (Sec. 5,
// Eq. time.step.2d) with one reciprocal square root.
__device__ __forceinline__ double swe_rate_2d(double h, double mx, double my, double sg,
                                              double inv_dx, double inv_dy) {
  const double r = drsqrt_pos(h);
  const double rr = r * r;
  const double c = (sg * h) * r;
  return fma(fma(fabs(mx), rr, c), inv_dx, fma(fabs(my), rr, c) * inv_dy);
}

// max of two non-negative doubles through their bit patterns (integer pipe)
__device__ __forceinline__ double max_nonneg(double a, double b) {
  const long long ia = __double_as_longlong(a), ib = __double_as_longlong(b);
  return __longlong_as_double(ia > ib ? ia : ib);
}

// max of the bit patterns: of non-negative values their maximum, and any NaN
// (of either sign) wins
__device__ __forceinline__ double max_bits(double a, double b) {
  const unsigned long long ia = (unsigned long long)__double_as_longlong(a);
  const unsigned long long ib = (unsigned long long)__double_as_longlong(b);
  return __longlong_as_double((long long)(ia > ib ? ia : ib));
}

// true if x > 0 and finite (integer test on the bit pattern)
__device__ __forceinline__ bool positive_finite(double x) {
  const long long ix = __double_as_longlong(x);
  return ix > 0 && ix < 0x7ff0000000000000LL;
}

__device__ __forceinline__ bool finite(double x) {
  const long long ix = __double_as_longlong(x) & 0x7fffffffffffffffLL;
  return ix < 0x7ff0000000000000LL;
}

// Step size of the step in flight (Sec. 5, Eq. time.step.2d): the fixed dt,
// or C_s CFL(N) / max rate of the current state, clipped to t_end.
__device__ __forceinline__ double step_dt(const StepCtl& c, const DevState* st) {
  if (c.dt_fixed > 0.0) return c.dt_fixed;
  const double rate = __longlong_as_double((long long)st->rate[c.slot_read]);
  if (!positive_finite(rate)) return 0.0;
  double dt = c.cs_cfl / rate;
  const double rem = c.t_end - st->time[c.tslot];
  if (rem < dt) dt = rem > 0.0 ? rem : 0.0;
  return dt;
}

// Bookkeeping done once per step by one thread of the first kernel.
__device__ __forceinline__ void step_bookkeeping(const StepCtl& c, DevState* st, double dt) {
  st->rate[c.slot_reset] = 0ull;
  st->time[c.tslot ^ 1] = st->time[c.tslot] + dt;
  st->dt_cur = dt;
  st->dt_last = dt;
  if (dt > 0.0) st->nadv += 1ull;
}

// The step size and its products with the tableau's coefficients, by the
// block's first warp (each product once, in one lane, instead of in every
// thread: an FP64 instruction costs the same for one lane as for 32): dt;
// e[i][j] = -(dt a~_ij xs); im[i][j] = dt a_ij; dt b_ref xs and dt b_ref; avg[j] =
// sum_i (b_i/b_ref) e[i][j], so that a variable without source has the time
// average (1/b_ref) u^n + sum_j avg[j] L_j in units of b_ref: one rounding of
// the size of u^n instead of one per stage.
template <class TB>
struct StepSizes {
  double dt, dtb_x, dtb;
  double e[TB::S][TB::S], avg[TB::S];   // (filled as one array)
  double im[TB::S][TB::S];
};
template <class TB, bool IMEX>
__device__ __forceinline__ void fill_step_sizes(StepSizes<TB>& s, double dt, double xs) {
  constexpr int S = TB::S;
  const int lane = threadIdx.x;
  const double dtx = dt * xs;
#pragma unroll
  for (int k0 = 0; k0 < S * S + S; k0 += 32) {
    double a = 0.0, ai = 0.0;
    const int k = k0 + lane;
#pragma unroll
    for (int i = 0; i < S; ++i)
#pragma unroll
      for (int j = 0; j <= i; ++j) {
        if (TB::a(i, j) != 0.0 && k == i * S + j) a = TB::a(i, j);
        if (IMEX && TB::ai(i, j) != 0.0 && k == i * S + j) ai = TB::ai(i, j);
      }
#pragma unroll
    for (int j = 0; j < S; ++j)
      if (k == S * S + j) a = TB::avg(j);
    if (k < S * S + S) (&s.e[0][0])[k] = -(dtx * a);
    if (IMEX && k < S * S) (&s.im[0][0])[k] = dt * ai;
  }
  if (lane == 0) {
    s.dt = dt;
    s.dtb_x = dtx * TB::bref();
    s.dtb = dt * TB::bref();
  }
}

// Weight of the candidate b in theta b + (1 - theta) a for the linear
// constraint P (Eq. theta.formula): 1 unless P(b) < eps.
__device__ __forceinline__ double theta_lin(double eps, double Pa, double Pb) {
  if (!(Pb < eps)) return 1.0;
  const double den = Pb - Pa;
  return den != 0.0 ? fmin(1.0, fabs((eps - Pa) / den)) : 1.0;
}

// x in FP32, cut to 20 fraction bits; NaN beyond the normal range but for zero
__device__ __forceinline__ float cut_f32(double x) {
  const int hi = __double2hiint(x), m = hi & 0x7fffffff;
  const int f = (int)((unsigned)(m - (896 << 20)) << 3) | (hi & (int)0x80000000);
  const bool in = (unsigned)(m - (897 << 20)) < (254u << 20);
  return __int_as_float(in ? f : (m | __double2loint(x)) == 0 ? 0 : 0x7fc00000);
}

// true only if theta_lin(0.1 low, low, t) is 1 for low = a - c (d - fl) and
// t = a - c (d - fh): t - 0.1 low in FP32 exceeds 2^-16 of the sum of the
// operands' magnitudes.  Operands are cut by 2^-20 of themselves and the handful
// of FP32 roundings are 2^-24 each, below 2^-17 of that sum together; the FP64
// evaluation rounds by 2^-50 of it.  (Six FP64 instructions a face side
// otherwise, some 400 cycles of their pipe.)
__device__ __forceinline__ bool theta_one(double a64, double c64, double d64, double fl64,
                                          double fh64) {
  const float a = cut_f32(a64), c = cut_f32(c64), d = cut_f32(d64), fl = cut_f32(fl64),
              fh = cut_f32(fh64);
  const float low = a - c * (d - fl), t = a - c * (d - fh);
  const float sum = a + fabsf(c) * (fabsf(d) + fabsf(fl) + fabsf(fh));
  return a > 1e-30f && t - 0.1f * low > 1.52587890625e-5f * sum;
}

// true only if theta_lin(0.1 lmin, ., t) is 1 for every t of an element, from the
// smallest high word of its t and of its first-order values, whose smallest is
// lmin: no t below an eighth of lmin.  (Positive doubles order as their high
// words; a negative one, or a NaN with its sign set, fails the comparison, and a
// positive NaN has theta 1.)
__device__ __forceinline__ bool theta_one_element(int lmin_hi, int tmin_hi) {
  return lmin_hi >= 0x400000 && lmin_hi < 0x7ff00000 && tmin_hi > lmin_hi - (3 << 20);
}

// True in every lane if b is in any; also the warp's barrier.  (A vote alone
// orders no shared-memory accesses: the reads of the exchange fields before it
// must not meet the writes of the next stage after it.)
__device__ __forceinline__ bool warp_barrier_or(bool b) {
  __syncwarp();
  return __any_sync(0xffffffffu, b);
}

// Max of a non-negative double over the warps that hold one above zero, then
// one atomicMax on the bit pattern per such warp.
__device__ __forceinline__ void block_max_atomic_1d(double v, unsigned long long* slot) {
  unsigned long long b = (unsigned long long)__double_as_longlong(v);
  if (!__any_sync(0xffffffffu, b != 0)) return;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    unsigned long long other = __shfl_xor_sync(0xffffffffu, b, o);
    b = other > b ? other : b;
  }
  if ((threadIdx.x & 31) == 0) atomicMax(slot, b);
}

// Block-wide max of a non-negative double, then one atomicMax on the bit
// pattern.  Every thread of the block must call it.
template <int BLOCK>
__device__ __forceinline__ void block_max_atomic(double v, unsigned long long* slot) {
  __shared__ unsigned long long red[BLOCK / 32];
  unsigned long long b = (unsigned long long)__double_as_longlong(v);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    unsigned long long other = __shfl_xor_sync(0xffffffffu, b, o);
    b = other > b ? other : b;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) red[warp] = b;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long m = red[0];
#pragma unroll
    for (int i = 1; i < BLOCK / 32; ++i) m = red[i] > m ? red[i] : m;
    atomicMax(slot, m);
  }
}

}  // namespace crkfr
