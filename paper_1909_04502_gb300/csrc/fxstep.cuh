// Device helpers shared by the fixed-point steps (step2x.cu, step3x.cu).
#pragma once
#include "frame64.cuh"
#include "fx64.cuh"

namespace rlbm {
namespace {

template <int N>
struct Int {
  static constexpr int value = N;
};

// exponent x with |v| < 2^x
__device__ __forceinline__ int above(float v) { return (int)((__float_as_uint(v) >> 23) & 0xFF) - 126; }

// Raises the scale 2^E of the moment sums to hold populations below 2^want, SPARE bits more.
template <int SPARE, int NM>
__device__ __forceinline__ void raise_scale(long long (&m)[NM], int& E, int want) {
  if (want <= E) return;
  const int to = want + SPARE, sh = min(to - E, 63);
#pragma unroll
  for (int k = 0; k < NM; ++k) m[k] >>= sh;
  E = to;
}

// m + c X / 2^64, rounded
__device__ __forceinline__ void add_product(long long& m, Cx c, int xh, int xl) {
  Acc a{m, 0x80000000LL};
  macs(a, c, xh, xl);
  m = a.H + (long long)hi32(a.M);
}

// The exponent that stands for an infinity or NaN: the scale of the sums then lies
// above that of every finite value.
constexpr int kNotFinite = 1 << 14;

// The largest biased exponent of a run (with CHECK kNotFinite if a member is not
// finite), and whether every member is finite and not negative.
template <bool CHECK, int L>
__device__ __forceinline__ int run_exponent(const double (&f)[L], bool& plain) {
  unsigned h = 0;
#pragma unroll
  for (int q = 0; q < L; ++q) h = max(h, (unsigned)__double2hiint(f[q]));
  plain = h < 0x7FF00000U;
  if (__builtin_expect(!plain, 0)) {
    h = 0;
#pragma unroll
    for (int q = 0; q < L; ++q) h = max(h, (unsigned)__double2hiint(f[q]) & 0x7FF00000U);
    if (CHECK && h == 0x7FF00000U) return kNotFinite;
  }
  return (int)(h >> 20);
}

// Slow relaxation, tau above kSlowTau or of a field: the unit of a run stands above
// every |term| of its equilibrium, up to 2^10 times the populations, so that a population
// that hardly changes would lose bits to it at each step.  There (SLOW) only the
// change, rate times difference, is taken in fixed point, in a unit finer by the
// rate (to 2^kSlowestRate), and added to the population in FP64: one addition more
// per population, the rounding of an FP64 step.  5 to 17 % of a step (517 x 333: 56.7
// -> 59.9 us, 2^22 cells in one dimension: 275 -> 322 us); at tau of one both forms are as
// good, at 3.9 the other had 1.0 to 1.9 times this one's error.
constexpr double kSlowTau = 2.0;
constexpr int kSlowestRate = -28;

// Signed, subnormal and non-finite values: out of line, so that the loops of
// the usual case stay short.
__device__ __noinline__ long long to_fixed_any(double f, int d) { return to_fixed(f, d - biased_exponent(f)); }
__device__ __noinline__ double from_fixed_any(long long Y, int k) { return from_fixed(Y, k); }

// the same exponent of a float
__device__ __forceinline__ int float_exponent(unsigned magnitude) {
  return magnitude < 0x7F800000U ? (int)(magnitude >> 23) + 896 : kNotFinite;
}

// g 2^ep (a float, exact) in units of 2^(E - BITS): d = E - 1 - ep - 896 + 63 - BITS.
__device__ __forceinline__ long long float_units(float g, int d) {
  const unsigned b = __float_as_uint(g);
  const int v = (int)((b & 0x7FFFFFU) | 0x800000U), s = (int)b >> 31;
  long long x = (long long)(((unsigned long long)(unsigned)(((v ^ s) - s) << 7)) << 32);
  asm("shr.s64 %0, %0, %1;" : "+l"(x) : "r"(d - (int)((b >> 23) & 0xFF)));
  return x;
}

// v 2^k, the exponent raised in place where the result is normal
__device__ __noinline__ double scaled_any(double v, int k) {
  const int k1 = k / 2;
  return v * __hiloint2double((1023 + k1) << 20, 0) * __hiloint2double((1023 + k - k1) << 20, 0);
}
__device__ __forceinline__ double scaled(double v, int k) {
  const int h = __double2hiint(v), e = (h >> 20) & 0x7FF;
  if (__builtin_expect(e > 0 && e < 0x7FF && e + k > 0 && e + k < 0x7FF, 1))
    return __hiloint2double(h + (k << 20), __double2loint(v));
  return scaled_any(v, k);
}

// 2^lo <= v < 2^hi (false for NaN)
__device__ __forceinline__ bool between(double v, int lo, int hi) {
  return (unsigned)(__double2hiint(v) - ((1023 + lo) << 20)) < (unsigned)((hi - lo) << 20);
}

// a table constant, as the integer that it stands for, times 2^k
__device__ __forceinline__ double constant_value(Cx c, int k) {
  return (double)(((long long)c.h << 32) + c.l) * __hiloint2double((1023 + k) << 20, 0);
}

// Values of a thread split for products (split_balanced), in a shared-memory
// column of its own: in registers they would hold 28 to 76 of them.
struct Column {
  int2* s;          // [][128]
  __device__ __forceinline__ void set(int k, long long v) const {
    int2 x;
    split_balanced(v, x.x, x.y);
    s[k * 128] = x;
  }
  __device__ __forceinline__ int2 get(int k) const { return s[k * 128]; }
};

}  // namespace
}  // namespace rlbm
