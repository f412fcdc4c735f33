// fixed.cuh -- FP64 dot products and column combinations on the integer pipe.
//
// GB300 retires 2 FP64 FMA lanes per clock and multiprocessor, but 63 lanes of
// IMAD.WIDE (32 x 32 -> 64-bit multiply-add, measured) and 64 to 128 of the simple integer
// operations, so a long FP64 multiply-add stream is cheaper as integer arithmetic.  An
// operand vector is taken in fixed point relative to the largest exponent of its piece (a
// block's rows of one column) and held as two balanced 32-bit limbs, M = h 2^32 + l, l signed.
// A product of two operands is three IMAD.WIDE and, for the leading bits of l l', one 32-bit
// IMAD; integer sums are exact and do not depend on their order, so the only errors are the
// operands' cut to the piece's unit and the rounding of the total.
//
// Dots (fx_conv, fx_fma, fx_warp_sum, fx_value): |M| < 2^57 against |M'| < 2^56, sums of up to
// a super-tile's rows.  The cut is unbiased (the lowest bit of every M is set).  An error in a
// projection coefficient only touches the basis' orthogonality: the cut's is some 2^-57 of the
// largest entries, random, below what the roundings of an FP64 sum leave.
//
// Column combinations (fx_conv_near, fx_axpy_*): u = w - sum_c coef_c u_c is the Arnoldi
// relation itself, and an error with the same sign in all rows is smooth, which A^-1 amplifies
// (a plain cut to 57 bits cost a factor 20 in x against FP64 at 4.2M rows; the roundings of an
// FP64 sum are random).  So |M| < 2^61: entries within 2^8 of the piece's largest are exact,
// the rest are cut towards zero 8 bits below the FP64 spacing of the largest, the coefficients
// are rounded 54 bits below the largest term, and the sum is rounded to FP64 once.
//
// Zeros convert to exact zeros (but for the lowest bit in a dot); an infinity or a NaN in a
// piece shows in its largest exponent (2047), and the result is then NaN.
#pragma once

#include <stdint.h>

namespace gg {

struct Fx {
  int h, l;
};

// FP64 value to fixed point: e = largest biased exponent of the piece + 7 (|M| < 2^57, v = M
// 2^(e - 1086)) or + 8 (|M| < 2^56), the lowest bit set.
__device__ __forceinline__ Fx fx_conv(double v, int e) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const unsigned sh = (unsigned)(e - (int)((hi << 1) >> 21));
  // significand with its leading one at bit 63, shifted down to the common exponent
  const unsigned a = __funnelshift_l(lo, hi, 11) | 0x80000000u, b = lo << 11;
  unsigned long long x = ((unsigned long long)a << 32) | b;
  asm("shr.u64 %0, %0, %1;" : "+l"(x) : "r"(sh));  // shifts past 63 give 0
  const unsigned s = (unsigned)((int)hi >> 31);
  const unsigned l = ((unsigned)x ^ s) | 1u;
  const unsigned h = ((unsigned)(x >> 32) ^ s) + (l >> 31);
  return Fx{(int)h, (int)l};
}

// biased exponent of |v|'s largest representative, from the high word of |v|
__device__ __forceinline__ int fx_mag(double v) { return __double2hiint(v) & 0x7fffffff; }

// (hh, cr, ll) += a * b (at most 31 products): hh in units of 2^64, cr of 2^32, ll of 2^36
__device__ __forceinline__ void fx_fma(long long& hh, long long& cr, int& ll, const Fx a, int bh,
                                       int bl) {
  hh += (long long)a.h * bh;
  cr += (long long)a.h * bl;
  cr += (long long)a.l * bh;
  ll += (a.l >> 18) * (bl >> 18);
}

// A lane's total (fx_fma) summed over the warp: value s 2^64 + f 2^32, s signed, f < 2^32,
// exact but for bits below 2^37 of the unit.  Valid in every lane.
struct FxSum {
  long long s;
  unsigned f;
};
__device__ __forceinline__ FxSum fx_warp_sum(long long hh, long long cr, int ll) {
  cr += (long long)ll << 4;
  const long long t = hh + (cr >> 32);
  const unsigned t0 = (unsigned)t & 0x7ffffffu;
  const unsigned t1 = (unsigned)(t >> 27) & 0x7ffffffu;
  const int t2 = (int)(t >> 54);
  const unsigned c = (unsigned)cr >> 5;
  const unsigned r0 = __reduce_add_sync(0xffffffffu, t0);
  const unsigned r1 = __reduce_add_sync(0xffffffffu, t1);
  const int r2 = __reduce_add_sync(0xffffffffu, t2);
  const unsigned long long rc = (unsigned long long)__reduce_add_sync(0xffffffffu, c) << 5;
  FxSum o;
  o.s = ((long long)r2 << 54) + (long long)((unsigned long long)r1 << 27) + (long long)r0 +
        (long long)(rc >> 32);
  o.f = (unsigned)rc;
  return o;
}

// s 2^64 + f 2^32 in units of 2^(ea - 1079) 2^(eb - 1079) as FP64 (ea, eb: the exponents of
// the conversions, less 7); NaN when either piece holds an infinity or a NaN
__device__ __forceinline__ double fx_value(long long s, unsigned f, int ea, int eb) {
  if (ea >= 2047 || eb >= 2047) return __longlong_as_double(0x7ff8000000000000ll);
  return ldexp(fma((double)f, 0x1p-32, (double)s), ea + eb - 2094);
}

// FP64 value to fixed point, exact negation: e = largest biased exponent of the piece + 3
// (|M| < 2^61, cut towards zero)
__device__ __forceinline__ Fx fx_conv_near(double v, int e) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const unsigned sh = (unsigned)(e - (int)((hi << 1) >> 21));
  const unsigned a = __funnelshift_l(lo, hi, 11) | 0x80000000u, b = lo << 11;
  unsigned long long x = ((unsigned long long)a << 32) | b;
  asm("shr.u64 %0, %0, %1;" : "+l"(x) : "r"(sh));
  const long long s = (long long)((int)hi >> 31);
  const long long m = ((long long)x ^ s) - s;
  return Fx{(int)(m >> 32) + (int)((unsigned)m >> 31), (int)m};
}

// A coefficient times its column's unit as an integer K = kh 2^28 + kl, rounded to nearest
// (|K| <= 2^53, |kl| <= 2^27) relative to the largest of them: m = the largest of biased
// exponent + eb over the columns, eb = the column's largest biased exponent.  One unit of M K is
// 2^(m - 2158).  z: the leading bits of kl.
__device__ __forceinline__ int3 fx_coef(double coef, int m, int eb) {
  const unsigned hi = (unsigned)__double2hiint(coef), lo = (unsigned)__double2loint(coef);
  const unsigned sh = (unsigned)(m - eb + 11 - (int)((hi << 1) >> 21));  // >= 11
  const unsigned a = __funnelshift_l(lo, hi, 11) | 0x80000000u, b = lo << 11;
  const unsigned long long X = ((unsigned long long)a << 32) | b;
  const unsigned long long x = sh < 64 ? ((X >> (sh - 1)) + 1) >> 1 : 0ull;
  const long long s = (long long)((int)hi >> 31);
  const long long K = ((long long)x ^ s) - s;
  const int kl = (int)((unsigned)K << 4) >> 4;
  return make_int3((int)((K - kl) >> 28), kl, kl >> 15);
}

// Sums of at most 65 products M K: h kh (2^60), h kl (2^32), l kh (2^28), leading bits of l kl
// (2^34)
struct FxAcc {
  long long hh, hl, lh;
  int ll;
};
__device__ __forceinline__ void fx_axpy(FxAcc& a, const Fx v, const int4 k) {
  a.hh += (long long)v.h * k.x;
  a.hl += (long long)v.h * k.y;
  a.lh += (long long)v.l * k.x;
  a.ll += (v.l >> 19) * k.z;
}
// w + nscale (sum in units of 2^60): nscale = -2^(m - 2098) for w - sum; two FP64 roundings
__device__ __forceinline__ double fx_axpy_sub(const FxAcc& a, double w, double nscale) {
  const long long low = a.hl + (a.lh >> 4) + ((long long)a.ll << 2);
  const long long hi = a.hh + (low >> 28) - (1ll << 24);
  // 2^52 + the 28 low bits, times 2^-28, is 2^24 + their share
  const double r = __hiloint2double(0x43300000, (int)low & 0xfffffff);
  return fma(fma(r, 0x1p-28, (double)hi), nscale, w);
}

}  // namespace gg
