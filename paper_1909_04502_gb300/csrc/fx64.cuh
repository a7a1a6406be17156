// 64-bit fixed-point arithmetic for the FP64 steps.
//
// This part issues 2 FP64 operations per clock and SM, and about 25 32 x 32 +
// 64-bit multiply-adds and 42 64-bit additions: a step whose population
// sums run on the FP64 pipe waits for it (85 % busy) while the integer pipes
// idle.  Here the populations of a cell become 64-bit integers in a unit of
// the cell's own, the long sums over them (moments, equilibrium, relaxation)
// run on the integer pipes, and only the macroscopic state of the cell, some
// hundred operations, stays in FP64.
//
// Precision.  Moments: X_i = f_i 2^(e_i) in units of 2^(E - 59) or 2^(E - 60), e_i a constant
// of the table (the exponent of p0^2, so that 2^-59 is relative to the largest
// contribution to T^00) and 2^E above them all.  Relaxation: f and f^eq of a
// run in units of 2^(u - 59), 2^u above the run's own populations and, with
// kHead spare bits, above every |term| sum of its equilibrium rows: finer than
// the rounding of an FP64 sum over the same terms.  Additions are exact.
// Products with a table constant c = h 2^32 + l (61 or 63 bits, l signed, as
// the value's lower half is) keep the partial products h xh, h xl and l xh
// exactly and drop l xl, a zero-mean 2^-61 of the full scale at most.  With one bit
// less in the relaxation and its constants a step of the order-3 and order-5 tables was up
// to 3 times as far off as one in FP64.
#pragma once
#include <cuda_runtime.h>

#include <cmath>

namespace rlbm {

constexpr int kBits = 59;        // populations in a relaxation: |X| < 2^kBits
constexpr int kBitsM = 59;       // populations in the moment sums: runs of 8 members
constexpr int kBitsM4 = 60;      // ... and of at most 4
constexpr int kHead = 4;         // results of a relaxation: below 2^(kBits + kHead)
constexpr int kCoefM = 63;       // moment constants: their sum over the runs at most 2^kCoefM
constexpr int kCoefH = 61;       // equilibrium constants (kBits + 2): a row's sum over a parity class at most four

// constant c = h 2^32 + l with l in [-2^31, 2^31)
struct Cx {
  int h, l;
};

inline Cx split_constant(double c, int bits) {   // host: c, |c| <= 1, in units of 2^-bits
  const long long i = std::llround(std::ldexp(c, bits));
  const int l = (int)(unsigned)(unsigned long long)i;
  return {(int)((i - (long long)l) >> 32), l};
}

__host__ __device__ __forceinline__ int hi32(long long v) { return (int)(v >> 32); }
__host__ __device__ __forceinline__ unsigned lo32(long long v) { return (unsigned)(unsigned long long)v; }
// a b + c in one 64-bit multiply-add: written as its two halves, since a 64-bit
// sum of a product compiles to a multiply and two additions (3 instructions).
__host__ __device__ __forceinline__ long long madw(int a, int b, long long c) {
#ifdef __CUDA_ARCH__
  unsigned l = (unsigned)(unsigned long long)c, h = (unsigned)((unsigned long long)c >> 32);
  asm("mad.lo.cc.s32 %0, %2, %3, %0;\n\tmadc.hi.s32 %1, %2, %3, %1;" : "+r"(l), "+r"(h) : "r"(a), "r"(b));
  return (long long)(((unsigned long long)h << 32) | l);
#else
  return (long long)a * b + c;
#endif
}

// Sum of products in two words: value H 2^64 + M 2^32.
struct Acc {
  long long H, M;
};

// + c V for V = vh 2^32 + vl with vl signed (split_balanced)
__host__ __device__ __forceinline__ void macs(Acc& a, Cx c, int vh, int vl) {
  a.H = madw(c.h, vh, a.H);
  a.M = madw(c.h, vl, a.M);
  a.M = madw(c.l, vh, a.M);
}

// (H 2^64 + M 2^32) 2^(j - 64), 0 <= j <= 30
__host__ __device__ __forceinline__ long long collect(const Acc& a, int j) {
  return (long long)((unsigned long long)a.H << j) + (a.M >> (32 - j));
}

__host__ __device__ __forceinline__ void split_balanced(long long V, int& h, int& l) {
  l = (int)lo32(V);
  h = hi32(V + 0x80000000LL);
}

__host__ __device__ __forceinline__ unsigned long long bits_of(double f) {
#ifdef __CUDA_ARCH__
  return (unsigned long long)__double_as_longlong(f);
#else
  unsigned long long b;
  __builtin_memcpy(&b, &f, 8);
  return b;
#endif
}
__host__ __device__ __forceinline__ double double_of(unsigned long long b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double f;
  __builtin_memcpy(&f, &b, 8);
  return f;
#endif
}

__host__ __device__ __forceinline__ int biased_exponent(double f) { return (int)((bits_of(f) >> 52) & 0x7FF); }

// f 2^(kBits - 1 - d) / 2^exponent(f), rounded to nearest (exponent(f): of f's
// leading bit): with d = u - 1 - e for a value of biased exponent e, f in units
// of 2^(u - kBits).  Subnormals and zero count as 2^-1022 (the units that
// callers take are far above).
__host__ __device__ __forceinline__ unsigned long long shift_right(unsigned long long v, int d) {
#ifdef __CUDA_ARCH__
  asm("shr.u64 %0, %0, %1;" : "+l"(v) : "r"(d));     // zero from 64 on
  return v;
#else
  return d > 63 ? 0 : v >> d;
#endif
}
__host__ __device__ __forceinline__ long long to_fixed(double f, int d) {
  const unsigned long long b = bits_of(f);
  const unsigned long long m = ((b & 0x000FFFFFFFFFFFFFULL) | 0x0010000000000000ULL) << (kBits - 52);
  const long long v = (long long)((shift_right(m, d) + 1) >> 1);
  const long long s = (long long)b >> 63;
  return (v ^ s) - s;
}
// the same for f >= 0
__host__ __device__ __forceinline__ long long to_fixed_positive(double f, int d) {
  const unsigned long long m = (bits_of(f) & 0x000FFFFFFFFFFFFFULL) | 0x0010000000000000ULL;
  return (long long)((shift_right(m << (kBits - 52), d) + 1) >> 1);
}
// |f| in units of 2^(u - BITS), the bits below the unit cut
template <int BITS>
__host__ __device__ __forceinline__ long long to_fixed_cut(double f, int d) {
  const unsigned long long m = (bits_of(f) & 0x000FFFFFFFFFFFFFULL) | 0x0010000000000000ULL;
  return (long long)shift_right(m << (BITS - 53), d);
}

// The double nearest to Y 2^(k - 1023), |Y| < 2^63, k + 62 < 2047 and k > 0.
__host__ __device__ __forceinline__ double from_fixed(long long Y, int k) {
  const unsigned long long A = Y < 0 ? 0ULL - (unsigned long long)Y : (unsigned long long)Y;
  const unsigned ah = (unsigned)(A >> 32);
  const unsigned w = ah ? ah : (unsigned)A;
#ifdef __CUDA_ARCH__
  const int lz = __clz((int)w) + (ah ? 0 : 32);          // of A
#else
  const int lz = (w ? __builtin_clz(w) : 32) + (ah ? 0 : 32);
#endif
  const unsigned long long n = ((A << (lz - 1 < 63 ? lz - 1 : 63)) + 0x200ULL) >> 10;   // leading bit at 52
  const unsigned hi = (unsigned)(n >> 32) + (unsigned)((k + 62 - lz) << 20);
  const unsigned s = (unsigned)((unsigned long long)Y >> 32) & 0x80000000U;
  const unsigned long long r = ((unsigned long long)((hi | s)) << 32) | (unsigned long long)(unsigned)n;
  return double_of(w ? r : 0ULL);
}

// the same for 2^32 <= Y
__host__ __device__ __forceinline__ double from_fixed_positive(long long Y, int k) {
#ifdef __CUDA_ARCH__
  const int lz = __clz(hi32(Y));
#else
  const int lz = __builtin_clz((unsigned)hi32(Y));
#endif
  const unsigned long long n = (((unsigned long long)Y << (lz - 1)) + 0x200ULL) >> 10;
  return double_of(n + ((unsigned long long)(unsigned)((k + 62 - lz) << 20) << 32));
}

#ifdef __CUDACC__
// FP64 <-> FP32 for values of a cell scaled to order one, on the integer
// pipe: below 2^-126 the result is zero, the significand is cut.
__device__ __forceinline__ float cut_float(double d) {
  const unsigned h = (unsigned)__double2hiint(d), l = (unsigned)__double2loint(d);
  const unsigned m = (h & 0x7FFFFFFFU) < 0x38100000U ? 0U : (__funnelshift_l(l, h, 3) - 0x40000000U) & 0x7FFFFFFFU;
  return __uint_as_float((h & 0x80000000U) | m);
}
// (a zero becomes 2^-127)
__device__ __forceinline__ double wide_double(float f) {
  const unsigned b = __float_as_uint(f);
  return __hiloint2double((int)((b & 0x80000000U) | (((b & 0x7FFFFFFFU) >> 3) + 0x38000000U)), (int)(b << 29));
}

// a / b and 1 / sqrt(x) for b, x > 0 of order one: one third-order step (Halley /
// Householder) from the part's approximation (rcp.approx, rsqrt.approx: about
// 20 bits), and for the quotient its remainder.  6 and 5 FP64 operations; the
// results are good to an ulp.
__device__ __forceinline__ double reciprocal(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ double quotient(double a, double b) {
  const double y = reciprocal(b), q = a * y;
  return fma(fma(-q, b, a), y, q);
}
__device__ __forceinline__ double reciprocal_sqrt(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x * y, y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}

// round(v 2^k) for values of a cell scaled to order one, k >= 0 and the result
// below 2^63: the exponent raised in place (a zero stays far below the unit).
__device__ __forceinline__ long long scaled_integer(double v, int k) {
  return __double2ll_rn(__hiloint2double(__double2hiint(v) + (k << 20), __double2loint(v)));
}
#endif

}  // namespace rlbm

