// Dot products of FP64 data in fixed point, on the integer pipe.
//
// This chip issues one FP64 warp instruction per 18.4 cycles and SM (measured:
// 1.056 TFLOP/s of FMA) but a 32 x 32 -> 64 bit integer multiply-add
// (IMAD.WIDE) every cycle.  A contraction sum_m P_m d_m therefore runs as
// integers: the rows P are stored as fixed point (host, once), the d_m of one
// sum are aligned to the largest of them, and every product takes three
// multiply-adds of 30-bit limbs into 64-bit accumulators instead of one FP64
// FMA, 3 cycles instead of 18.
//
// Numbers: q = hi 2^30 + lo with lo in [-2^29, 2^29), an int2 (x = hi, y = lo).
//   row entries  |q| <= 2^60, and sum_m |q_m| <= 2^60 + M over a row: P_m =
//                q_m 2^(E - 60), E the row's exponent (its sum of |P_m| < 2^E)
//   operands     |q| <= 2^B, B = 58 (57 in sums of more than 38): d = q
//                2^(e - B), |d| < 2^e for all d of the sum
//   monomials    |q| <= 2^58: x = q 2^-58, |x| <= 1
//   polynomials  coefficients as operands (B = 58, 57 at P4), aligned to the
//                largest of the cell's in coordinates scaled by powers of two,
//                one per axis, to [-1, 1]
// A product is (hi hi') 2^60 + (hi lo' + lo hi') 2^30 + lo lo'; the last term,
// at most 2^58, is dropped.  Bounds: sum |hi hi'| <= 2^30 2^28, sum |hi lo' + lo
// hi'| <= 2^30 2^29 + M 2^29 2^(B - 30) < 2^63, so no accumulator overflows for
// the M <= 68 members of a stencil.
//
// Error of a sum against the exact one, in units of max|d| sum|P|: operand rounding
// at most 2^-B, row rounding M 2^-59, dropped terms M 2^-57 (all of random sign, so
// that about sqrt(M) 2^-60 is seen).  An FP64 sum of M products rounds each partial sum
// to 2^-53 of itself.
// Measured against 128 bits on random rows and operands of one magnitude, error
// over sum|P d|, rms (largest): M = 18 fixed 1.9e-17 (9e-17), FP64 5.6e-17 (4.4e-16);
// M = 68 fixed 1.6e-17 (1.1e-16), FP64 5.7e-17 (4.8e-16).
#pragma once

#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstring>

namespace ucns {

__host__ __device__ __forceinline__ int2 fx_limbs(long long q) {
  const int hi = (int)((q + (1ll << 29)) >> 30);
  return make_int2(hi, (int)((unsigned)q - ((unsigned)hi << 30)));
}

// x rounded to an integer (host; |x| < 2^62, exact from 2^53 on)
inline long long fx_round(double x) { return (long long)(x + std::copysign(0.5, x)); }

// An exponent of kFxNan or a little below makes fx_double a NaN (a non-finite operand
// or row).  Exponents of finite sums stay below 2^13: operands and rows below 2^11
// each, and axis scales, of cells whose volume and its square are finite, below 2^10.
constexpr int kFxNan = 1 << 15;

// exponent E of a row: sum |P_m| < 2^E (a row of zeros: 0; with a NaN or an infinity: kFxNan - 1)
inline int fx_row_exponent(double l1) {
  int e = 0;
  if (!std::isfinite(l1)) return kFxNan - 1;
  if (l1 > 0.0) std::frexp(l1, &e);
  return e;
}

struct FxAcc {
  long long h = 0, m = 0;
};

// a += x y, one instruction (written as an expression, the compiler rearranges
// sums of products into trees of 64-bit additions, two more instructions each)
__host__ __device__ __forceinline__ void fx_wide(long long& a, int x, int y) {
#ifdef __CUDA_ARCH__
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(a) : "r"(x), "r"(y));
#else
  a += (long long)x * y;
#endif
}

__host__ __device__ __forceinline__ void fx_mac(FxAcc& a, int2 p, int2 d) {
  fx_wide(a.h, p.x, d.x);
  fx_wide(a.m, p.x, d.y);
  fx_wide(a.m, p.y, d.x);
}

// the sum in units of 2^58 (|h| < 2^61)
__host__ __device__ __forceinline__ long long fx_sum(const FxAcc& a) {
  return (a.h << 2) + ((a.m + (1ll << 27)) >> 28);
}

__host__ __device__ __noinline__ static double fx_double_rare(long long s, int e) {
  if (e >= kFxNan / 2) return (double)NAN;
  return ldexp((double)s, e);
}

__host__ __device__ __forceinline__ int fx_clz(unsigned long long x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return x ? __builtin_clzll(x) : 64;
#endif
}

// s 2^e rounded to nearest (ties away from zero), by integer operations; results outside
// the normal range by the library's ldexp
__host__ __device__ __forceinline__ double fx_double(long long s, int e) {
  const unsigned long long sgn = (unsigned long long)(s >> 63);
  const unsigned long long mag = ((unsigned long long)s ^ sgn) - sgn;
  const int lz = fx_clz(mag);
  const int be = 1086 + e - lz;  // biased exponent of the leading bit
  if ((unsigned)(be - 1) >= 2046u) return fx_double_rare(s, e);
  const unsigned long long m = mag << (lz & 63);
  const unsigned long long f = (m >> 11) + ((m >> 10) & 1u);  // 53 bits, a carry moves into the exponent
  unsigned long long b = (((unsigned long long)(unsigned)(be - 1) << 52) + f) | (sgn << 63);
  b = mag ? b : 0ull;
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double d;
  std::memcpy(&d, &b, 8);
  return d;
#endif
}

__host__ __device__ __forceinline__ unsigned long long fx_bits(double d) {
#ifdef __CUDA_ARCH__
  return (unsigned long long)__double_as_longlong(d);
#else
  unsigned long long b;
  std::memcpy(&b, &d, 8);
  return b;
#endif
}

// biased exponent of d
__host__ __device__ __forceinline__ int fx_exponent(double d) { return (int)((unsigned)(fx_bits(d) >> 52) & 0x7ffu); }

// bits of the operands of a sum of M
__host__ __device__ constexpr int fx_bits_of(int M) { return M <= 38 ? 58 : 57; }

// x 2^(1084 - eb) as an integer below 2^62 in magnitude, eb at least x's biased exponent
__host__ __device__ __forceinline__ long long fx_integer(double x, int eb) {
  const unsigned long long b = fx_bits(x);
  const int e = (int)((unsigned)(b >> 52) & 0x7ffu);
  const unsigned long long mant = (b & 0xfffffffffffffull) | ((unsigned long long)(e != 0) << 52);
  const int sh = eb - (e > 1 ? e : 1);
  const unsigned long long q = (mant << 9) >> (sh < 63 ? sh : 63);
  const unsigned long long sgn = (unsigned long long)((long long)b >> 63);
  return (long long)((q ^ sgn) - sgn);
}

// operand q of d, rounded to B bits, for a sum whose largest biased exponent is eb < 2047
// (d normal and at most that large, zero, or subnormal and eb at least 64)
template <int B>
__host__ __device__ __forceinline__ int2 fx_operand(double d, int eb) {
  const unsigned long long b = fx_bits(d);
  const int e = (int)((unsigned)(b >> 52) & 0x7ffu);
  const unsigned long long mant = (b & 0xfffffffffffffull) | ((unsigned long long)(e != 0) << 52);
  const unsigned sh = (unsigned)(eb - e) < 63u ? (unsigned)(eb - e) : 63u;
  const unsigned long long q = (((mant << (B - 52)) >> sh) + 1) >> 1;
  const unsigned long long sgn = (unsigned long long)((long long)b >> 63);
  return fx_limbs((long long)((q ^ sgn) - sgn));
}

// d shifted up by its lz - 1 spare leading bits and rounded to an operand of B bits.  The
// shifted value may lie within a rounding unit of 2^63 (a difference just below a power
// of two), so half a unit is added only after the shift down: |q| <= 2^B.
template <int B>
__host__ __device__ __forceinline__ int2 fx_normalised(long long d, int lz) {
  return fx_limbs((((d << (lz - 1)) >> (62 - B)) + 1) >> 1);
}

// The differences u[m] - u0, m < M, as operands q[m] of one sum: all values as
// integers aligned to the largest exponent among them, subtracted exactly, then
// shifted up by their common leading bits.  e: |u[m] - u0| < 2^e (kFxNan when a
// value is not finite).  No FP64 instruction; the error, at most 2^-61 of the
// largest value where one is 2^9 times smaller than it, else none before the
// rounding to B bits of the largest difference, is below that of FP64
// differences.  Values all below 2^-959 are scaled up first (exact).
template <int M>
__host__ __device__ __forceinline__ void fx_differences(double (&u)[M], double u0, int2 (&q)[M], int& e) {
  constexpr int B = fx_bits_of(M);
  int eb = fx_exponent(u0), low = 0;
#pragma unroll
  for (int m = 0; m < M; m++) {
    const int x = fx_exponent(u[m]);
    eb = x > eb ? x : eb;
  }
  if (eb < 64) {
    low = 512;
    u0 *= 0x1p512;
    eb = fx_exponent(u0);
#pragma unroll
    for (int m = 0; m < M; m++) {
      u[m] *= 0x1p512;
      const int x = fx_exponent(u[m]);
      eb = x > eb ? x : eb;
    }
  }
  const long long f0 = fx_integer(u0, eb);
  long long d[M];
  unsigned long long any = 0;
#pragma unroll
  for (int m = 0; m < M; m++) {
    d[m] = fx_integer(u[m], eb) - f0;
    any |= (unsigned long long)(d[m] ^ (d[m] >> 63));
  }
  const int lz = fx_clz(any | 1u);
#pragma unroll
  for (int m = 0; m < M; m++) q[m] = fx_normalised<B>(d[m], lz);
  e = eb == 2047 ? kFxNan : eb - 1020 - lz - low;
}

// The same for polynomial coefficients d[k], each to be scaled by 2^off[k]: returns eb,
// from which fx_operand(d[k], eb - off[k]) are the operands of exponent e.  Zeros take no
// part (the offset of one may lie far above the others); subnormal coefficients, which
// with a large offset need not be small, are made normal first (exact), unless one
// beside them is so large that they do not count.
template <int M>
__host__ __device__ __forceinline__ int fx_align_scaled(double (&d)[M], const int (&off)[M], int& e) {
  constexpr int none = -(1 << 14);
  int eb = none;
  bool odd = false;  // a zero, subnormal or non-finite coefficient
#pragma unroll
  for (int m = 0; m < M; m++) {
    const int x = fx_exponent(d[m]);
    odd = odd || (unsigned)(x - 1) >= 2046u;
    eb = x + off[m] > eb ? x + off[m] : eb;
  }
  e = eb - 1022;
  if (odd) {
    auto largest = [&](bool& sub, int& top) {
      int r = none;
#pragma unroll
      for (int m = 0; m < M; m++) {
        const int x = fx_exponent(d[m]);
        if (fx_bits(d[m]) << 1 == 0ull) continue;
        sub = sub || x == 0;
        top = x > top ? x : top;
        r = x + off[m] > r ? x + off[m] : r;
      }
      return r;
    };
    bool sub = false;
    int top = 0;
    eb = largest(sub, top);
    e = eb - 1022;
    if (sub && top < 1500) {
#pragma unroll
      for (int m = 0; m < M; m++) d[m] *= 0x1p512;
      eb = largest(sub, top);
      e = eb - 1022 - 512;
    }
    if (top == 2047) e = kFxNan;
  }
  return eb;
}

// product of two monomials
__host__ __device__ __forceinline__ int2 fx_mul(int2 a, int2 b) {
  FxAcc t;
  fx_mac(t, a, b);
  return fx_limbs(fx_sum(t));
}

// the integer hi 2^30 + lo
__host__ __device__ __forceinline__ long long fx_value(int2 q) { return ((long long)q.x << 30) + q.y; }

// a number s 2^e, |s| <= 2^62.2
struct FxSum {
  long long s;
  int e;
};

__host__ __device__ __forceinline__ FxSum fx_of(double x) {
  const int eb = fx_exponent(x);
  return {fx_integer(x, eb > 1 ? eb : 1), eb == 2047 ? kFxNan : (eb > 1 ? eb : 1) - 1084};
}

// a + b, the one of the smaller unit shifted to the larger (61 bits of the larger
// kept): rounded to FP64 afterwards, closer than FP64 terms added
__host__ __device__ __forceinline__ FxSum fx_add(FxSum a, FxSum b) {
  const bool swap = a.e < b.e;
  const FxSum x = swap ? b : a, y = swap ? a : b;
  const int d = x.e - y.e < 62 ? x.e - y.e : 62;
  return {(x.s >> 1) + (y.s >> (d + 1)), x.e + 1};
}

__host__ __device__ __forceinline__ double fx_double(FxSum a) { return fx_double(a.s, a.e); }

}  // namespace ucns
