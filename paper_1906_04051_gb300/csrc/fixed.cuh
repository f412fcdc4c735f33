// fixed.cuh -- FP64 dot products and column combinations on the integer pipe.
//
// GB300 retires 2 FP64 FMA lanes per clock and multiprocessor, but 63 lanes of
// IMAD.WIDE (32 x 32 -> 64-bit multiply-add, measured) and 64 to 128 of the simple integer
// operations, so a long FP64 multiply-add stream is cheaper as integer arithmetic.  Integer
// sums are exact and do not depend on their order; the only errors are the operands' rounding
// to their fixed-point unit and the rounding of the total.
//
// A basis column is held as 64-bit integers M relative to its largest exponent E (of the whole
// column) and to a shift S of the row: v = M 2^(E - S - 1083), |M| <= 2^61, rounded to nearest.
// M = h 2^32 + l, l signed.  Converting in every pass cost some 15 integer operations per
// element, more than the multiplications, so a column is converted once, in place.
//
// The row's shift (fx_shift) is 0 where its entries come within 2^8 of their columns' largest: these
// are exact there and rounded 8 bits below the FP64 spacing of the largest elsewhere.  A row that
// stays far below its columns' largest (an uncoupled block of a system, say, whose right-hand side
// is small) gets a shift that gives its first nonzero entry all 53 bits; when a later column has a
// larger entry there, the row's shift shrinks and its earlier entries are rounded to the new unit.
// So a row's rounding errors are relative to the largest of its own entries (each in units of its
// column's largest), as those of an FP64 sum over the row are.  Without shifts, a block 2^66 below
// the rest of the system lost all but 10 digits.  A dot takes the other operand times 2^-S.
//
// Dots (fx_operand, fx_dot, fx_warp_sum, fx_value): the other operand W = wh 2^28 + wl, |W| <=
// 2^54, relative to the largest exponent of its piece.  An error in a projection coefficient
// touches the basis' orthogonality only.
//
// Column combinations (fx_coef, fx_axpy, fx_axpy_add): u = w - sum_c coef_c u_c is the Arnoldi
// relation itself, and an error with the same sign in all rows is smooth, which A^-1 amplifies
// (cutting instead of rounding to 57 bits cost a factor 20 in x against FP64 at 4.2M rows; the
// roundings of an FP64 sum are random).  The coefficients are rounded 54 bits below the largest
// term and the sum is rounded to FP64 once.  A row's result depends on that row's values and the
// column scales only: rows that hold equal values (the Dirichlet rows of an aggregate, say) keep
// equal values, as with FP64 multiply-adds.
//
// Zeros convert to zeros whatever the shift; an infinity or a NaN shows in the largest exponent (2047), and the
// result is then NaN.
#pragma once

#include <stdint.h>

namespace gg {

struct Fx {
  int h, l;
};

// high word of |v|: orders like |v|, its upper bits are the biased exponent
__device__ __forceinline__ int fx_mag(double v) { return __double2hiint(v) & 0x7fffffff; }

// |v| in units of 2^(e - 1086), to nearest (halves away from zero), signed; e - 11 is at least
// v's biased exponent
__device__ __forceinline__ long long fx_round(double v, int e) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const int ex = (int)((hi << 1) >> 21);
  const unsigned sh = (unsigned)(e - 1 - max(ex, 1));
  // significand with its leading one (a zero or subnormal value has none) at bit 63, shifted down
  // to one bit more than the result
  const unsigned a = __funnelshift_l(lo, hi, 11) | (ex ? 0x80000000u : 0u), b = lo << 11;
  unsigned long long x = ((unsigned long long)a << 32) | b;
  asm("shr.u64 %0, %0, %1;" : "+l"(x) : "r"(sh));  // shifts past 63 give 0
  const long long s = (long long)((int)hi >> 31);
  return (((long long)x ^ s) + 1) >> 1;
}

// a basis entry of a column with largest biased exponent E (less the row's shift)
__device__ __forceinline__ long long fx_basis(double v, int E) { return fx_round(v, E + 3); }

// The shift of a row: the distance of an entry's exponent ex from its column's largest, less a
// guard, so that entries up to 2^8 larger still fit later on (61 bits hold 53 and the guard).
// kFxUnset: only zeros so far.
constexpr int kFxGuard = 8;
constexpr int kFxUnset = 1000;
__device__ __forceinline__ int fx_shift(int ex, int E) {
  return min(max(E - ex - kFxGuard, 0), kFxUnset - 1);
}
// 2^-s for 0 <= s <= 1022
__device__ __forceinline__ double fx_pow2(int s) { return __hiloint2double((1023 - s) << 20, 0); }
// an integer of a row whose shift shrinks by d > 0
__device__ __forceinline__ long long fx_less_shift(long long m, int d) {
  return d > 62 ? 0 : (m + (1ll << (d - 1))) >> d;
}

__device__ __forceinline__ Fx fx_limbs(unsigned lo, unsigned hi) {
  return Fx{(int)(hi + (lo >> 31)), (int)lo};
}
__device__ __forceinline__ Fx fx_limbs(long long m) {
  return fx_limbs((unsigned)m, (unsigned)((unsigned long long)m >> 32));
}

// the other operand of a dot (wh, wl) of a piece with largest biased exponent E, plus the row's shift
__device__ __forceinline__ int2 fx_operand(double v, int E) {
  const long long m = fx_round(v, E + 10);
  const int wl = (int)((unsigned)m << 4) >> 4;
  return make_int2((int)((m - wl) >> 28), wl);
}

// Sums of at most 31 products M W: h wh (2^60), h wl (2^32), l wh (2^28), leading bits of l wl
// (2^32)
struct FxDot {
  long long hh, hl, lh;
  int ll;
};
__device__ __forceinline__ void fx_dot(FxDot& a, const Fx v, const int2 w) {
  a.hh += (long long)v.h * w.x;
  a.hl += (long long)v.h * w.y;
  a.lh += (long long)v.l * w.x;
  a.ll += (v.l >> 18) * (w.y >> 14);
}

// The lanes' totals summed over the warp: value s 2^68 + f 2^32, f < 2^36 in every lane's share
// and cut below 2^41.  Valid in every lane.
struct FxSum {
  long long s, f;
};
__device__ __forceinline__ FxSum fx_warp_sum(const FxDot& a) {
  const long long low = a.hl + (a.lh >> 4) + a.ll;
  const long long t = a.hh + (low >> 28);
  const long long s = t >> 8;
  const unsigned c = (unsigned)((((unsigned)t & 0xffu) << 19) | (((unsigned)low & 0xfffffffu) >> 9));
  const unsigned r0 = __reduce_add_sync(0xffffffffu, (unsigned)s & 0x7ffffffu);
  const int r1 = __reduce_add_sync(0xffffffffu, (int)(s >> 27));
  const unsigned rc = __reduce_add_sync(0xffffffffu, c);
  return FxSum{((long long)r1 << 27) + r0, (long long)((unsigned long long)rc << 9)};
}

// s 2^68 + f 2^32 of a column of largest exponent E against a piece of largest exponent Ew; NaN
// when either holds an infinity or a NaN
__device__ __forceinline__ double fx_value(long long s, long long f, int E, int Ew) {
  if (E >= 2047 || Ew >= 2047) return __longlong_as_double(0x7ff8000000000000ll);
  s += f >> 36;
  return ldexp(fma((double)(f & 0xfffffffffll), 0x1p-36, (double)s), E + Ew - 2091);
}

// A coefficient times its column's unit as an integer K = kh 2^28 + kl, rounded to nearest
// (|K| <= 2^53, |kl| <= 2^27) relative to the largest of them: m = the largest of biased
// exponent + E over the columns.  One unit of M K is 2^(m - 2158).  z: the leading bits of kl.
__device__ __forceinline__ int3 fx_coef(double coef, int m, int E) {
  const long long K = fx_round(coef, m - E + 11);
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
// w + scale (sum in units of 2^60): scale = +-2^(m - 2098), times 2^-S of the row; two FP64 roundings
__device__ __forceinline__ double fx_axpy_add(const FxAcc& a, double w, double scale) {
  const long long low = a.hl + (a.lh >> 4) + ((long long)a.ll << 2);
  const long long hi = a.hh + (low >> 28) - (1ll << 24);
  // 2^52 + the 28 low bits, times 2^-28, is 2^24 + their share
  const double r = __hiloint2double(0x43300000, (int)low & 0xfffffff);
  return fma(fma(r, 0x1p-28, (double)hi), scale, w);
}

// The coefficients of a column combination, by one warp: coef[c] over k columns of largest
// exponents E[c] into sK[c] = (kh, kl, leading kl bits, -), and 2^(m - 2098) in every lane (NaN
// with an infinity or a NaN among them)
__device__ __forceinline__ double fx_coefs(int k, const double* coef, const int* E, int4* sK) {
  const int lane = threadIdx.x & 31;
  int m = 0;
  bool bad = false;
  for (int c = lane; c < k; c += 32) {
    const int e = fx_mag(coef[c]) >> 20;
    bad |= e == 2047 || E[c] == 2047;
    m = max(m, e + E[c]);
  }
  m = __reduce_max_sync(0xffffffffu, m);
  bad = __any_sync(0xffffffffu, bad);
  for (int c = lane; c < k; c += 32) {
    const int3 f = fx_coef(coef[c], m, E[c]);
    sK[c] = make_int4(f.x, f.y, f.z, 0);
  }
  return bad ? __longlong_as_double(0x7ff8000000000000ll) : ldexp(1.0, m - 2098);
}

}  // namespace gg
