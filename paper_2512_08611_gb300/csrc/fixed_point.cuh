// Block fixed-point contractions with the constant matrices of the scheme
// (differentiation matrix, end-point interpolation) on the integer pipe.
//
// On GB300 an FP64 instruction holds its SM sub-partition's FP64 pipe for 64
// cycles per warp (two FP64 lanes per SM), an IMAD.WIDE takes 2 and a shift or
// logic instruction 2 (measured).  The steps are bound by that pipe, and more
// than half of their FP64 instructions are products with constant matrices.
// Those are done here in 60-bit block fixed point instead: the operands of a
// contraction are scaled by one power of two per element and field, split into
// two 30-bit halves, and multiplied into two 64-bit accumulators with three
// IMAD.WIDE per term (6 cycles against 64); the sum is rounded to FP64 once.
//
// Accuracy: operands are truncated 2^-59 below the power of two above the
// group's largest magnitude, coefficients are integers of a row sum up to
// 2^61, and the dropped product of the lower halves is below 2^-57 of the
// row's full scale (sum of |coefficient| times the largest operand).  An
// FP64 FMA chain rounds every partial sum, 2^-53 of the partial sums each.
//
// A group is one field of one element (a variable, a flux, an adjoint): what
// enters one sum, so that its errors are those of the sum's own terms.  A value
// far below the largest of its group loses bits, as its part of an FP64 sum over
// the element does; sums of different fields are aligned after the contraction.
// What is not summed over the element has an exponent of its own or stays FP64:
// the state in the update, the average of h in the source term, the traces of
// u^n and of that average at GLL nodes.  (The GLL traces of the averaged momenta
// and fluxes are single values in their field's fixed point: all stages but the
// first carry the rounding of a row of D on that field anyway.)  Groups whose
// largest value is below 2^-895 (1e-269) lose bits, below 2^-953 they count as
// zero; groups holding an infinity or a NaN give non-finite sums.
#pragma once

#include <cstdint>

#include "crkfr_internal.h"
#include "device_common.cuh"

namespace crkfr {
namespace {

// operand value hi * 2^30 + lo (0 <= lo < 2^30 from fx_split)
struct alignas(8) Fx {
  int hi, lo;
};

// added to the biased exponent of a group with a non-finite member: every
// member then shifts out, and fx_to returns the group's NaN for the zero sums
constexpr int kFxNonFinite = 4096;
// smallest biased exponent of a group (zeros and denormals then shift out)
constexpr int kFxMinExp = 128;

// high word of |x|: its bits 20..30 are the biased exponent, and integer
// order is magnitude order
__device__ __forceinline__ int fx_mag(double x) { return __double2hiint(x) & 0x7fffffff; }

// biased exponent of a group from the largest fx_mag of its members
__device__ __forceinline__ int fx_exp(int mag) {
  const int e = mag >> 20;
  const int m = e > kFxMinExp ? e : kFxMinExp;
  return e == 0x7ff ? m + kFxNonFinite : m;
}

// x as a signed integer of FB bits in units of 2^(E - 1022 - FB), truncated;
// E at least the biased exponent of x.  The 53-bit significand is shifted
// into place (PTX shifts of 64 or more give 0) and the sign applied.
template <int FB>
__device__ __forceinline__ long long fx_from(double x, int E) {
  const int hi = __double2hiint(x);
  const unsigned lo = (unsigned)__double2loint(x);
  const int e = (hi & 0x7fffffff) >> 20;
  long long m = (long long)(((unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 32 | lo)
                            << (FB - 53));
  // (a predicated negation: two integer adds instead of a mask, two xors and
  // two subtractions)
  asm("{\n\t.reg .pred n;\n\tshr.u64 %0, %0, %1;\n\tsetp.lt.s32 n, %2, 0;\n\t"
      "@n neg.s64 %0, %0;\n\t}"
      : "+l"(m)
      : "r"(E - e), "r"(hi));
  return m;
}

// |x| = s 2^(e - 1085), s < 2^63 (0 for zeros and denormals); neg the sign bit
struct FxSig {
  unsigned long long s;
  int e, neg;
};
__device__ __forceinline__ FxSig fx_sig(double x) {
  const int hi = __double2hiint(x);
  const int e = (hi & 0x7fffffff) >> 20;
  const unsigned mh = (unsigned)((hi & 0xfffff) | 0x100000);
  const unsigned long long m =
      ((unsigned long long)mh << 32 | (unsigned)__double2loint(x)) << 10;
  return FxSig{e == 0 ? 0 : m, e, hi};
}

// m >> sh with the sign bit of neg applied (sh >= 0; 64 or more give 0)
__device__ __forceinline__ long long fx_signed(unsigned long long m, int sh, int neg) {
  long long r;
  asm("{\n\t.reg .pred n;\n\tshr.u64 %0, %1, %2;\n\tsetp.lt.s32 n, %3, 0;\n\t"
      "@n neg.s64 %0, %0;\n\t}"
      : "=l"(r)
      : "l"(m), "r"(sh), "r"(neg));
  return r;
}

// (a b) 2^-64 less at most 2, for a and b below 2^63: three IMAD.WIDE
__device__ __forceinline__ unsigned long long fx_mulhi(unsigned long long a,
                                                       unsigned long long b) {
  const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a;
  const unsigned bh = (unsigned)(b >> 32), bl = (unsigned)b;
  const unsigned long long mid = (unsigned long long)ah * bl + (unsigned long long)al * bh;
  return (unsigned long long)ah * bh + (mid >> 32);
}
__device__ __forceinline__ unsigned long long fx_sqrhi(unsigned long long a) {
  const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a;
  return (unsigned long long)ah * ah + ((unsigned long long)ah * al >> 31);
}

// Shallow-water fluxes of a node in the fixed point of their element.  With
// FP64 products and a conversion each they cost seven FP64 instructions a
// stage (64 cycles each); the significands of h, hu, hv are at hand for the
// conversion of the state, a product of two is three IMAD.WIDE, and 1/h stays
// the integer that the reciprocal ends in.  Nothing is rounded to 53 bits on
// the way: each product is exact up to 2^-57 of itself and then truncated to
// the element's fixed point.
//
// The exponent is bounded without the products: the bits of a double read as a
// fixed-point number exceed 1023 + log2 by at most 0 and fall short by at most
// 0.087 (Mitchell's logarithm), and by another 1/16 cut to 4 fraction bits.
// fx_flux_mag adds those of the factors: m m / h lies below the sum by at most
// 2 (0.087 + 1/16) = 0.30, h h g/2 by 0.45; the sum of the two terms adds 1
// and all of it is covered by 24/16.
__device__ __forceinline__ int fx_log(double x) { return fx_mag(x) >> 16; }

// magnitude of the group (as fx_mag) of m k / h (+ h^2 g/2) with lm, lk the
// fx_log of the momenta, lhg = fx_log(g/2).  h must be normal for 1/h to be
// finite, and m, k finite: the group counts as non-finite otherwise.
template <bool PRESSURE>
__device__ __forceinline__ int fx_flux_mag(double h, int lm, int lk, int lhg) {
  const int lh = fx_log(h);
  int l = lm + lk - lh;
  if (PRESSURE) l = max(l, 2 * lh + lhg - 2 * (1023 << 4));
  l = min(max(l + 24, 0), 0x7ff0);
  return ((unsigned)((lh >> 4) - 1) > 2045u || max(lm, lk) >= 0x7ff0 ? 0x7ff0 : l) << 16;
}

// true if h (of the well-balanced form: the pressure-free one), a momentum or a
// product of a 2D node exceeds the exponents E of its element's fields h, hu,
// hv, hu hu / h, hu hv / h, hv hv / h
template <bool PRESSURE>
__device__ __forceinline__ bool fx_over(double h, int lx, int ly, int lhg, const int (&E)[6]) {
  const int lh = fx_log(h), x = lx - lh + 24, y = ly - lh + 24;
  int f3 = lx + x, f5 = ly + y;
  if (PRESSURE) {
    const int p = 2 * lh + lhg + 24 - 2 * (1023 << 4);
    f3 = max(f3, p);
    f5 = max(f5, p);
  }
  return (!PRESSURE && lh >> 4 > E[0]) || lx >> 4 > E[1] || ly >> 4 > E[2] || f3 >> 4 > E[3] ||
         ly + x >> 4 > E[4] || f5 >> 4 > E[5] || (unsigned)((lh >> 4) - 1) > 2045u;
}

// 2^61 |m| / |h| up to their exponents
__device__ __forceinline__ unsigned long long fx_velocity(unsigned long long R, const FxSig& m) {
  return fx_mulhi(m.s, R);
}
// m v for v = k / h: sign and exponent from m, k, h; FB bits at exponent E.
// (The product is in units of 2^-60 and at least 1/8 where m, k are not zero,
// so the bound above leaves the shift non-negative.)
template <int FB>
__device__ __forceinline__ long long fx_momentum_flux(const FxSig& m, unsigned long long v,
                                                      const FxSig& k, const FxSig& h, int E) {
  return fx_signed(fx_mulhi(m.s, v), 60 - FB + E - (m.e + k.e - h.e + 1), m.neg ^ k.neg ^ h.neg);
}
// h^2 g/2
template <int FB>
__device__ __forceinline__ long long fx_pressure(const FxSig& h, const FxSig& hg, int E) {
  return fx_signed(fx_mulhi(fx_sqrhi(h.s), hg.s), 61 - FB + E - (2 * h.e + hg.e - 2044), hg.neg);
}
// a value of which fx_sig is at hand
template <int FB>
__device__ __forceinline__ long long fx_from(const FxSig& x, int E) {
  return fx_signed(x.s, 63 - FB + E - x.e, x.neg);
}

__device__ __forceinline__ Fx fx_split(long long v) {
  return Fx{(int)(v >> 30), (int)v & 0x3fffffff};
}

// arithmetic shift right by s >= 0 (64 or more: the sign)
__device__ __forceinline__ long long fx_sar(long long v, int s) {
  long long r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
  return r;
}

// R1 2^(e1 - 1085) + R2 2^(e2 - 1085) in units of the larger exponent e (|R1|,
// |R2| at most 2^60).  CANCEL: of the other one's where a sum is zero, for rows
// that annihilate equal values without rounding.
template <bool CANCEL = false>
__device__ __forceinline__ long long fx_align(long long R1, int e1, long long R2, int e2,
                                              int& e) {
  if (CANCEL) {
    // (but for groups with a non-finite member, whose sums are zero too)
    if (R1 == 0 && e1 < 3000) e1 = e2;
    if (R2 == 0 && e2 < 3000) e2 = e1;
  }
  const int d = e1 - e2;
  e = max(e1, e2);
  return fx_sar(R1, max(-d, 0)) + fx_sar(R2, max(d, 0));
}

// high word of what a zero sum of a group with exponent E stands for: 0, or
// NaN for a group with a non-finite member
__device__ __forceinline__ int fx_zero(int E) { return E >= kFxNonFinite ? 0x7ff80000 : 0; }

// R * 2^(eb - 1085) rounded to FP64 (to nearest, ties away from zero); |R| <
// 2^62; zero = fx_zero of the group.  The leading bit is found by truncating
// conversions of the two halves to FP32 (2 cycles a warp each; the
// count-leading-zeros unit takes 8, the 64-bit conversion more than 60).
// Exponents above the FP64 range give a non-finite value.
__device__ __forceinline__ double fx_to(long long R, int eb, int zero) {
  const int rh = (int)(R >> 32);
  unsigned long long a = (unsigned long long)R;
  asm("{\n\t.reg .pred n;\n\tsetp.lt.s32 n, %1, 0;\n\t@n neg.s64 %0, %0;\n\t}"
      : "+l"(a)
      : "r"(rh));
  const float f = __fmaf_rz(__uint2float_rz((unsigned)(a >> 32)), 4294967296.0f,
                            __uint2float_rz((unsigned)a));
  const int ex = __float_as_int(f) >> 23;   // 127 + position of the leading bit, 0 for zero
  const int sh = 189 - ex;                  // leading bit to bit 62
  asm("shl.b64 %0, %1, %2;" : "=l"(a) : "l"(a), "r"(sh));
  a += 0x200;
  const int e = eb - sh;
  int hi = (int)(a >> 42) + (((e < 2047 ? e : 2047) - 1) << 20);
  hi |= rh & (int)0x80000000;
  return __hiloint2double(ex == 0 ? zero : hi, (int)(unsigned)(a >> 10));
}

// Weighted sums of operands: with weights up to 6 in all one 64-bit sum A holds
// them; WIDE (up to 90) keeps the halves' sums apart, A 2^30 + B.
template <bool WIDE>
__device__ __forceinline__ void fx_accumulate(long long& A, long long& B, long long v, Fx x,
                                              int w) {
  if (WIDE) {
    A += (long long)x.hi * w;
    B += (long long)x.lo * w;
  } else {
    A += (long long)((unsigned long long)(unsigned)v * (unsigned)w) +
         (long long)((unsigned long long)(unsigned)((int)(v >> 32) * w) << 32);
  }
}

// the sum in units 2^sh larger
template <bool WIDE>
__device__ __forceinline__ void fx_rescale(long long& A, long long& B, int sh) {
  if (WIDE) {
    // (the low half takes what the high one loses; from 62 on the sum is below
    // 2^-55 of the new scale)
    const long long hi = A >> (sh & 63), lost = A - (hi << (sh & 63));
    const long long low = (B >> (sh & 63)) +
                          (sh < 30 ? (lost << 30) >> (sh & 63) : lost >> ((sh - 30) & 63));
    A = sh < 62 ? hi : 0;
    B = sh < 62 ? low : 0;
  } else {
    A = sh < 62 ? A >> (sh & 63) : 0;
  }
}

// the sum shifted back to operand size
template <bool WIDE, int SHIFT>
__device__ __forceinline__ long long fx_average(long long A, long long B) {
  if (!WIDE) return A >> SHIFT;
  return ((A + (B >> 30)) << (30 - SHIFT)) + (((int)B & 0x3fffffff) >> SHIFT);
}

// The operand of the average w x + inc (inc: FP64, in units 2^SHIFT smaller than
// the result's) of a value x: what FP64 would round off the sum at x's size is
// kept.  E at least the biased exponent of x and that of inc less SHIFT.
template <bool WIDE, int SHIFT, int FB>
__device__ __forceinline__ long long fx_increment(double x, int w, double inc, int E) {
  long long A = 0, B = 0;
  const long long v = fx_from<FB>(x, E);
  fx_accumulate<WIDE>(A, B, v, fx_split(v), w);
  return fx_average<WIDE, SHIFT>(A, B) + fx_from<FB>(inc, E + SHIFT);
}

// a row of n operands in shared memory (16-byte aligned for even n)
template <int n>
__device__ __forceinline__ void fx_row(const Fx* x, Fx (&r)[n]) {
  if constexpr (n % 2 == 0) {
#pragma unroll
    for (int j = 0; j < n; j += 2) {
      const int4 v = *reinterpret_cast<const int4*>(x + j);
      r[j] = Fx{v.x, v.y};
      r[j + 1] = Fx{v.z, v.w};
    }
  } else {
#pragma unroll
    for (int j = 0; j < n; ++j) r[j] = x[j];
  }
}

// sum of products in units of operand unit x coefficient unit x 2^60
struct FxAcc {
  long long a, b;
};
__device__ __forceinline__ void fx_mul(FxAcc& s, Fx x, int ch, int cl) {
  s.a = (long long)x.hi * ch;
  s.b = (long long)x.hi * cl + (long long)x.lo * ch;
}
__device__ __forceinline__ void fx_mad(FxAcc& s, Fx x, int ch, int cl) {
  s.a += (long long)x.hi * ch;
  s.b += (long long)x.hi * cl;
  s.b += (long long)x.lo * ch;
}
__device__ __forceinline__ long long fx_sum(const FxAcc& s) { return s.a + (s.b >> 30); }

}  // namespace
}  // namespace crkfr
