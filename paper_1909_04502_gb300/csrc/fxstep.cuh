// Device helpers shared by the fixed-point steps (step2x.cu, step3x.cu).
#pragma once
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

// The largest biased exponent of a run, and whether every member is finite and not negative.
template <int L>
__device__ __forceinline__ int run_exponent(const double (&f)[L], bool& plain) {
  unsigned h = 0;
#pragma unroll
  for (int q = 0; q < L; ++q) h = max(h, (unsigned)__double2hiint(f[q]));
  plain = h < 0x7FF00000U;
  if (__builtin_expect(!plain, 0)) {
    h = 0;
#pragma unroll
    for (int q = 0; q < L; ++q) h = max(h, (unsigned)__double2hiint(f[q]) & 0x7FF00000U);
  }
  return (int)(h >> 20);
}

// Signed, subnormal and non-finite values: out of line, so that the loops of
// the usual case stay short.
__device__ __noinline__ long long to_fixed_any(double f, int d) { return to_fixed(f, d - biased_exponent(f)); }
__device__ __noinline__ double from_fixed_any(long long Y, int k) { return from_fixed(Y, k); }

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
