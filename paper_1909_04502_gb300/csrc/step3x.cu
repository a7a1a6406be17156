// The (3+1)-d massless FP64 steps (orders 2 and 3) and the fields of both
// storage types with the population sums in 64-bit fixed point (fx64.cuh).
//
// The sign-orbit form: populations come in runs whose members share p0 and
// |p| componentwise, member s negating the components whose bit is set in s;
// 9 (order 2) or 33 (order 3) runs of 8 and a tail of axis pairs (order 2)
// or runs of 4 (order 3).  Per run a Walsh-Hadamard transform of the pulled
// values (exact integer additions) leaves one product per moment; the
// equilibrium's eight values come from the first row's partial sums over the
// parity classes of the basis, transformed back.  Pass 1 sums the moments,
// FP64 takes the Landau frame (Sec. 4) and the Maxwell-Juttner moments
// (App. B, d = 3, m = 0) of the cell, pass 2 pulls the populations again,
// relaxes and stores.
//
// What bounds it: latency at 24 (order 2) and 20 (order 3) warps per SM.  147 and 192
// instructions per population and step fill 49 % and 41 % of the issue slots; a warp
// waits most for the two population reads (3.4 and 3.9 cycles per issued
// instruction), then at order 2 for the instruction cache (2.0) and in either for the
// arithmetic before it (1.5 to 1.7).  The FP64 pipe, which the sums used to hold at 85 %,
// is busy 31 % and 10 %, DRAM 43 % and 35 % (96^3 and 48^3).  The basis moments and the rates lie in shared-memory columns
// so that 80 (order 2) and 96 (order 3) registers suffice; with all of them in
// registers (128, four blocks per SM) the order-2 step ran 1.3x longer.  Signed
// and non-finite populations leave the loop for functions of their own: inline
// they cost the instruction cache 1.3x; the FP64 relaxation of cells
// outside the range is out of line as well.  101 x 75 x 66, order 2: 0.38 ms per step
// and 0.13 ms for the fields against 1.6 and 1.8 ms with the sums in FP64;
// 192 x 192 x 6, order 3: 0.77 and 0.14 ms against 2.0 and 2.6 ms; the fields of
// 192^3 cells in FP32 storage: 1.2 ms against 24 ms (FP64, row by row).
#include <cuda_runtime.h>

#include "d3_impl.cuh"
#include "fxstep.cuh"
#include "step3x.h"

namespace rlbm {

namespace {

// parity class (bit 0: x odd, bit 1: y odd, bit 2: z odd) of the members of
// 1 | p0 px py pz | p0px p0py p0pz pxpx pxpy pxpz pypy pypz pzpz |
// p0 (xx xy xz yy yz zz) | xxx xxy xxz xyy xyz xzz yyy yyz yzz zzz
__device__ constexpr int kPar3[30] = {0, 0, 1, 2, 4, 1, 2, 4, 0, 3, 5, 0, 6, 0,
                                      0, 3, 5, 0, 6, 0, 1, 2, 4, 1, 7, 1, 2, 4, 2, 4};
// class of each moment sum N0 Nx Ny Nz T0x T0y T0z Txx Txy Txz Tyy Tyz Tzz
// (T00 = Txx + Tyy + Tzz on the light cone)
__device__ constexpr int kMomPar[kMom3] = {0, 1, 2, 4, 1, 2, 4, 0, 3, 5, 0, 6, 0};

// non-zero components of the tail runs: the axis pairs of order 2, the (5, 4, 0)
// patterns of order 3
template <int ORDER>
__device__ constexpr int tail_mask(int r) {
  if (ORDER == 2) return 1 << r;
  constexpr int m[6] = {3, 5, 3, 5, 6, 6};
  return m[r];
}
// class of a tail member's sign bits: the r-th set bit of mask carries bit r of c
__device__ constexpr int spread(int mask, int c) {
  int out = 0, b = 0;
  for (int k = 0; k < 3; ++k)
    if (mask >> k & 1) out |= (c >> b++ & 1) << k;
  return out;
}
__device__ constexpr int gather_bits(int mask, int par) {
  int out = 0, b = 0;
  for (int k = 0; k < 3; ++k)
    if (mask >> k & 1) out |= (par >> k & 1) << b++;
  return out;
}

// A run's populations scaled by 2^ep in units of 2^(E - kBitsM), E raised where
// they need it.
template <int L>
__device__ __forceinline__ void run_units(const double (&f)[L], int ep, long long, long long (&m)[kMom3], int& E,
                                          long long (&X)[L]) {
  bool plain;
  raise_scale<1>(m, E, run_exponent<true>(f, plain) + ep + 1);
  const int d = E - 1 - ep;
  if (__builtin_expect(plain, 1)) {
#pragma unroll
    for (int q = 0; q < L; ++q) X[q] = to_fixed_cut<kBitsM>(f[q], d - (__double2hiint(f[q]) >> 20));
  } else {
#pragma unroll
    for (int q = 0; q < L; ++q) X[q] = to_fixed_any(f[q], d) << (kBitsM - kBits);
  }
}
// FP32 storage: g = f - f_ref with the reference added (exactly); E never falls
// below ref_E, the reference's own scale.
template <int L>
__device__ __forceinline__ void run_units(const float (&g)[L], int ep, long long ref, int ref_E, long long (&m)[kMom3], int& E,
                                          long long (&X)[L]) {
  unsigned h = 0;
#pragma unroll
  for (int q = 0; q < L; ++q) h = max(h, __float_as_uint(g[q]) & 0x7FFFFFFFU);
  raise_scale<1>(m, E, float_exponent(h) + ep + 1);
  const int d = E - 1 - ep - 896 + 63 - kBitsM;
  const long long r = ref >> min(E - ref_E, 63);
#pragma unroll
  for (int q = 0; q < L; ++q) X[q] = float_units(g[q], d) + r;
}

// The macroscopic state of a cell in units of 2^E: eps U^a = T^ab U_b with
// u = U^i / U^0 and (T^ij + eps delta^ij) u_j = T^0i, eps = T^00 - T^0i u_i.
struct Cell3 {
  double L, u[3], U0, n;
  bool ok;
};

// (t = T^0i; S = Txx Txy Txz Tyy Tyz Tzz.)  The root and u in FP32 by Newton on
// g(l) = T00 - t.(S + l)^-1 t - l, g' = u.u - 1; then (l, u) together by
// iterative refinement: FP64 residuals of both equations, the correction
// through the FP32 inverse.  A pass gains about 20 bits in slow flows; two are enough
// (more run where the last still moved l by 2^-40, or u by 2^-30 of (1 - u.u)^2: a pass
// leaves about 2^-20 / (1 - u.u)^2 of its step).  The inverse's error
// grows as gamma^4: what has not settled after six passes is solved in FP64
// (frame64.cuh; from gamma of about 7 on).
__device__ __forceinline__ Cell3 landau3x(const double (&N)[4], double T00, const double (&t)[3],
                                          const double (&S)[6]) {
  const float fT = cut_float(T00), ft[3] = {cut_float(t[0]), cut_float(t[1]), cut_float(t[2])};
  float fS[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) fS[k] = cut_float(S[k]);
  const float M2 = ft[0] * ft[0] + ft[1] * ft[1] + ft[2] * ft[2], k3 = 1.f / 3.f;
  float l = (-(1.f - k3) * fT + sqrtf(fmaxf((1.f - k3) * (1.f - k3) * fT * fT + 4.f * k3 * (fT * fT - M2), 0.f))) /
            (2.f * k3);
  float A[6], v[3], w = 1.f, det = 1.f;
#pragma unroll 1
  for (int it = 0; it < 12; ++it) {
    const float xx = fS[0] + l, yy = fS[3] + l, zz = fS[5] + l;
    A[0] = yy * zz - fS[4] * fS[4];
    A[1] = fS[2] * fS[4] - fS[1] * zz;
    A[2] = fS[1] * fS[4] - fS[2] * yy;
    A[3] = xx * zz - fS[2] * fS[2];
    A[4] = fS[1] * fS[2] - xx * fS[4];
    A[5] = xx * yy - fS[1] * fS[1];
    det = xx * A[0] + fS[1] * A[1] + fS[2] * A[2];
    const float id = __fdividef(1.f, det);
#pragma unroll
    for (int k = 0; k < 6; ++k) A[k] *= id;
    v[0] = A[0] * ft[0] + A[1] * ft[1] + A[2] * ft[2];
    v[1] = A[1] * ft[0] + A[3] * ft[1] + A[4] * ft[2];
    v[2] = A[2] * ft[0] + A[4] * ft[1] + A[5] * ft[2];
    w = 1.f - v[0] * v[0] - v[1] * v[1] - v[2] * v[2];
    const float d = __fdividef(fT - ft[0] * v[0] - ft[1] * v[1] - ft[2] * v[2] - l, w);
    l += d;
    if (!(fabsf(d) > 5e-7f * l)) break;
  }
  Cell3 c;
  c.L = wide_double(l);
  c.u[0] = wide_double(v[0]);
  c.u[1] = wide_double(v[1]);
  c.u[2] = wide_double(v[2]);
  const float iw = __fdividef(1.f, w);
  bool settled = false;
#pragma unroll 1
  for (int it = 0; it < 6; ++it) {
    const double r0 = fma(-t[2], c.u[2], fma(-t[1], c.u[1], fma(-t[0], c.u[0], T00 - c.L)));
    const double rx = fma(-S[2], c.u[2], fma(-S[1], c.u[1], fma(-S[0], c.u[0], fma(-c.L, c.u[0], t[0]))));
    const double ry = fma(-S[4], c.u[2], fma(-S[3], c.u[1], fma(-S[1], c.u[0], fma(-c.L, c.u[1], t[1]))));
    const double rz = fma(-S[5], c.u[2], fma(-S[4], c.u[1], fma(-S[2], c.u[0], fma(-c.L, c.u[2], t[2]))));
    const float x = cut_float(rx), y = cut_float(ry), z = cut_float(rz);
    const float d = (cut_float(r0) - v[0] * x - v[1] * y - v[2] * z) * iw;
    const float ex = x - v[0] * d, ey = y - v[1] * d, ez = z - v[2] * d;
    const float cx = A[0] * ex + A[1] * ey + A[2] * ez, cy = A[1] * ex + A[3] * ey + A[4] * ez,
                cz = A[2] * ex + A[4] * ey + A[5] * ez;
    c.L += wide_double(d);
    c.u[0] += wide_double(cx);
    c.u[1] += wide_double(cy);
    c.u[2] += wide_double(cz);
    settled = fabsf(d) <= 1e-12f * l && fabsf(cx) + fabsf(cy) + fabsf(cz) <= 1e-9f * w * w;
    if (it >= 1 && settled) break;
  }
  bool good = true;
  if (__builtin_expect(!(settled && det > 0.f && w > 0.f), 0)) {
    const Frame64 f = frame64(T00, t, S);
    good = f.ok;
    c.L = f.l;
    c.u[0] = f.u[0];
    c.u[1] = f.u[1];
    c.u[2] = f.u[2];
  }
  const double w2 = fma(-c.u[2], c.u[2], fma(-c.u[1], c.u[1], fma(-c.u[0], c.u[0], 1.0)));
  c.U0 = reciprocal_sqrt(w2);
  c.n = c.U0 * fma(-c.u[2], N[3], fma(-c.u[1], N[2], fma(-c.u[0], N[1], N[0])));
  c.ok = good && __double2hiint(w2) > 0 && between(c.n, -100, 100) && between(c.L, -100, 100);
  return c;
}

// Pass 1: the moment sums of a cell's populations in units of 2^(E + sk - kBitsM + 64 - kCoefM).
template <int ORDER, typename S>
__device__ __forceinline__ void moment_sums(const Tables3x<ORDER>& tb, const S* __restrict__ base, long long P, bool pull,
                                            long long (&m)[kMom3], int& E) {
  using T = Tables3x<ORDER>;
  E = sizeof(S) == 4 ? tb.ref_E : -4096;
#pragma unroll
  for (int k = 0; k < kMom3; ++k) m[k] = 0;
#pragma unroll 1
  for (int r = 0; r < T::N8; ++r) {
    const S* b = base + (long long)tb.first8[r] * P;
    S f[8];
#pragma unroll
    for (int q = 0; q < 8; ++q, b += P) f[q] = __ldg(b + (pull ? tb.off8[r][q] : 0));
    long long X[8];
    if constexpr (sizeof(S) == 4) run_units(f, tb.ep8[r], tb.ref8[r], tb.ref_E, m, E, X);
    else run_units(f, tb.ep8[r], 0, m, E, X);
    fwht(X);
    int xh[8], xl[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) split_balanced(X[c], xh[c], xl[c]);
#pragma unroll
    for (int k = 0; k < kMom3; ++k) add_product(m[k], tb.M8[r][k], xh[kMomPar[k]], xl[kMomPar[k]]);
  }
#pragma unroll
  for (int r = 0; r < T::NT; ++r) {
    constexpr int L = T::LT;
    const S* b = base + (long long)tb.firstT[r] * P;
    S f[L];
#pragma unroll
    for (int q = 0; q < L; ++q, b += P) f[q] = __ldg(b + (pull ? tb.offT[r][q] : 0));
    long long X[L];
    if constexpr (sizeof(S) == 4) run_units(f, tb.epT[r], tb.refT[r], tb.ref_E, m, E, X);
    else run_units(f, tb.epT[r], 0, m, E, X);
    fwht(X);
    int xh[L], xl[L];
#pragma unroll
    for (int c = 0; c < L; ++c) split_balanced(X[c], xh[c], xl[c]);
    const int mask = tail_mask<ORDER>(r);
#pragma unroll
    for (int k = 0; k < kMom3; ++k) {
      if (kMomPar[k] & ~mask) continue;
      if (k == 7 && !(mask & 1)) continue;
      if (k == 10 && !(mask & 2)) continue;
      if (k == 12 && !(mask & 4)) continue;
      const int c = gather_bits(mask, kMomPar[k]);
      add_product(m[k], tb.MT[r][k], xh[c], xl[c]);
    }
  }
}

// the sums as doubles in units of 2^E
__device__ __forceinline__ void moment_values(const long long (&m)[kMom3], const int (&sk)[kMom3], double (&N)[4], double& T00,
                                              double (&t)[3], double (&S)[6]) {
  double v[kMom3];
#pragma unroll
  for (int k = 0; k < kMom3; ++k) v[k] = from_fixed(m[k], 1023 + sk[k] - kBitsM + 64 - kCoefM);
#pragma unroll
  for (int k = 0; k < 4; ++k) N[k] = v[k];
#pragma unroll
  for (int k = 0; k < 3; ++k) t[k] = v[4 + k];
#pragma unroll
  for (int k = 0; k < 6; ++k) S[k] = v[7 + k];
  T00 = (S[0] + S[3]) + S[5];
}

// x / 3, correctly rounded but for rare halfway cases
__device__ __forceinline__ double third(double x) {
  const double q = x * (1.0 / 3.0);
  return fma(fma(-3.0, q, x), 1.0 / 3.0, q);
}

// Maxwell-Juttner moments of the basis for (n, eps, U): <1> = n / (2T),
// <p^a> = n U^a, <p^a p^b> = n (4T U^a U^b - T eta^ab), <p^a p^b p^c> =
// n (24 T^2 U^a U^b U^c - 4 T^2 (eta^ab U^c + eta^ac U^b + eta^bc U^a)), T = eps / (3n).
template <int K>
__device__ __forceinline__ void mj_moments3x(const Cell3& c, const double (&U)[3], double (&M)[K]) {
  const double P = third(c.L), T = quotient(P, c.n);    // n T, T
  M[0] = quotient(0.5 * c.n, T);
  M[1] = c.n * c.U0;
  const double q = 4.0 * P;
  const double qU[3] = {q * U[0], q * U[1], q * U[2]};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    M[2 + i] = c.n * U[i];
    M[5 + i] = qU[i] * c.U0;
  }
  M[8] = fma(qU[0], U[0], P);
  M[9] = qU[0] * U[1];
  M[10] = qU[0] * U[2];
  M[11] = fma(qU[1], U[1], P);
  M[12] = qU[1] * U[2];
  M[13] = fma(qU[2], U[2], P);
  if constexpr (K == 30) {
    const double r3 = 4.0 * P * T, q3 = 6.0 * r3;
    const double rU[3] = {r3 * U[0], r3 * U[1], r3 * U[2]}, rU0 = r3 * c.U0;
    const double x = q3 * U[0], y = q3 * U[1], z = q3 * U[2];
    const double xx = x * U[0], xy = x * U[1], xz = x * U[2], yy = y * U[1], yz = y * U[2], zz = z * U[2];
    M[14] = fma(xx, c.U0, rU0);
    M[15] = xy * c.U0;
    M[16] = xz * c.U0;
    M[17] = fma(yy, c.U0, rU0);
    M[18] = yz * c.U0;
    M[19] = fma(zz, c.U0, rU0);
    M[20] = fma(xx, U[0], 3.0 * rU[0]);
    M[21] = fma(xx, U[1], rU[1]);
    M[22] = fma(xx, U[2], rU[2]);
    M[23] = fma(yy, U[0], rU[0]);
    M[24] = xy * U[2];
    M[25] = fma(zz, U[0], rU[0]);
    M[26] = fma(yy, U[1], 3.0 * rU[1]);
    M[27] = fma(yy, U[2], rU[2]);
    M[28] = fma(zz, U[1], rU[1]);
    M[29] = fma(zz, U[2], 3.0 * rU[2]);
  }
}

// The relaxation in FP64, for a cell whose rate or equilibrium the fixed point does
// not hold (gamma of about 64 and above), or that has no frame and keeps its populations.
// v: K basis moments in units of 2^E, then tau^-1 U0 and tau^-1 U^i / |n| (a
// column of the shared memory).
template <int ORDER>
__device__ __noinline__ void relax_plain3(const Tables3x<ORDER>& tb, const Step3Args<double>& a, const double* v, int E,
                                          bool frame, int x, int y, int z) {
  using T = Tables3x<ORDER>;
  const Scalars3& s = a.s;
  const long long si = sidx3(s, x, y, z);
  long long img[26];
  const int nimg = cell_images(s, x, y, z, img);
  // the member of a run that negates the components of neg
  auto relax = [&](int i, int off, const Cx* H, const int* n, int mask, int neg, int e) {
    double sum = 0.0, om = 0.0;
    if (frame) {
#pragma unroll 1
      for (int k = 0; k < T::K; ++k)
        if (!(kPar3[k] & ~mask))
          sum = fma((__popc(kPar3[k] & neg) & 1) ? -v[k * 128] : v[k * 128], constant_value(H[k], tb.hk[k]), sum);
      sum = scaled(sum, E - 1023 + e - kCoefH);
      om = v[T::K * 128];
      for (int c = 0; c < 3; ++c)
        if (mask >> c & 1) om = fma((neg >> c & 1) ? (double)n[c] : -(double)n[c], v[(T::K + 1 + c) * 128], om);
    }
    const long long p = (long long)i * s.plane;
    const double f = a.fin[p + si + off], g = fma(om, sum - f, f);
    a.fout[p + si] = g;
    for (int k = 0; k < nimg; ++k) a.fout[p + img[k]] = g;
  };
#pragma unroll 1
  for (int g = 0; g < T::ND; ++g)
#pragma unroll 1
    for (int r = tb.dir_first[g]; r < tb.dir_first[g + 1]; ++r)
#pragma unroll 1
      for (int m = 0; m < 8; ++m)
        relax(tb.first8[r] + m, tb.off8[r][m], tb.H8[r], tb.dir_n[g], 7, m, tb.er8[r] + tb.rho8[r]);
#pragma unroll 1
  for (int r = 0; r < T::NT; ++r) {
    const int mask = tail_mask<ORDER>(r);
#pragma unroll 1
    for (int m = 0; m < T::LT; ++m)
      relax(tb.firstT[r] + m, tb.offT[r][m], tb.HT[r], tb.nT[r], mask, spread(mask, m), tb.erT[r] + tb.rhoT[r]);
  }
}

template <int ORDER, bool SLOW>
__global__ void __launch_bounds__(128, ORDER == 2 ? 6 : 5) k_step3x(const __grid_constant__ Tables3x<ORDER> tb,
                                                                    const __grid_constant__ Step3Args<double> a) {
  using T = Tables3x<ORDER>;
  constexpr int K = T::K;
  __shared__ int2 limbs[(K + 8) * 128];
  const Scalars3& s = a.s;
  const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 4 + threadIdx.y, z = blockIdx.z;
  if (x >= s.nx || y >= s.ny || z >= s.nz) return;
  const long long si = sidx3(s, x, y, z);
  const double* __restrict__ base = a.fin + si;
  double* __restrict__ ob = a.fout + si;
  const long long P = s.plane;

  const Column M{limbs + threadIdx.y * 32 + threadIdx.x};   // basis moments in units of 2^(xg - 62) 2^E
  const Column R{M.s + K * 128};                              // the rates of a direction pattern
  int uf, ue, eo, sb = 0;    // see below
  long long O0, W[3];        // tau^-1 U0 and tau^-1 U^i / |n|, in units of 2^(eo - 62)
  {
    long long m[kMom3];
    int E;
    moment_sums<ORDER, double>(tb, base, P, true, m, E);
    double N[4], T00, t[3], S[6];
    moment_values(m, tb.sk, N, T00, t, S);
    const Cell3 c = landau3x(N, T00, t, S);
    const bool ok = c.ok && E > 128 && E < 2040;
    const double U[3] = {c.u[0] * c.U0, c.u[1] * c.U0, c.u[2] * c.U0};
    double Mk[K];
    mj_moments3x<K>(c, U, Mk);
    // sum over k of |M_k| 2^hk < 2^xg bounds every equilibrium value, om = 2 U0 / tau every rate
    float sum = 0.f;
#pragma unroll
    for (int k = 0; k < K; ++k) sum += fabsf(cut_float(Mk[k])) * __uint_as_float((unsigned)(127 + tb.hk[k]) << 23);
    const double o0 = s.inv_tau * c.U0, kl = s.inv_tau * tb.inv_len;
    const int xg = above(sum), xo = above(2.f * cut_float(o0));
    // (moments within the float range, and, as in step2x.cu, rates below 64)
    const bool fits = E > 320 && between(c.n, -28, 28) && between(c.L, -28, 28) && between(c.U0, -1, 10) && between(o0, -1000, 6);
    if (__builtin_expect(!(ok && fits && xg < 60 && xg > -60), 0)) {
      // no Landau frame: counted, left unrelaxed (a population that is not finite becomes NaN)
      if (!ok) atomicAdd(a.status, 1ULL);
      double* const v = (double*)M.s;
#pragma unroll
      for (int k = 0; k < K; ++k) v[k * 128] = Mk[k];
      v[K * 128] = o0;
#pragma unroll
      for (int i = 0; i < 3; ++i) v[(K + 1 + i) * 128] = kl * U[i];
      relax_plain3<ORDER>(tb, a, v, E, ok, x, y, z);
      return;
    }
    // the unit 2^(u - kBits) of a run: u = max(its populations' exponent + uf, rho + ue)
    uf = max(0, xo - 2);
    ue = E + xg + max(0, xo - 3);
#pragma unroll
    for (int k = 0; k < K; ++k) M.set(k, scaled_integer(Mk[k], tb.hk[k] + 62 - xg));
    eo = max(xo, SLOW ? kSlowestRate : -2);
    if constexpr (SLOW) sb = max(-eo, 0);
    O0 = scaled_integer(o0, 62 - eo);
#pragma unroll
    for (int i = 0; i < 3; ++i) W[i] = scaled_integer(kl * U[i], 62 - eo);
  }
  int img[26];
  int nimg = 0;
  {
    long long wide[26];
    nimg = cell_images(s, x, y, z, wide);
    for (int i = 0; i < nimg; ++i) img[i] = (int)(wide[i] - si);
  }
  const long long half = 1LL << (29 - eo - sb);             // half a unit of the relaxation's sum
  const int sE = ue - max(0, uf - 1);                       // E + xg
  // f^eq of a run of L members from its row, and their relaxation at the rates R
  auto relax_run = [&](auto tag, const Cx* H, const int* off, int first, int er, int rho, int mask) {
    constexpr int L = decltype(tag)::value;
    const long long p0 = (long long)first * P;
    const double* b = base + p0;
    double f[L];
#pragma unroll
    for (int q = 0; q < L; ++q, b += P) f[q] = __ldg(b + off[q]);
    // the equilibrium's sums do not wait for the populations
    long long C[L];
#pragma unroll
    for (int c = 0; c < L; ++c) {
      Acc h{0, 0x80000000LL};
#pragma unroll
      for (int k = 0; k < K; ++k)
        if (kPar3[k] == (L == 8 ? c : spread(mask, c))) {
          const int2 v = M.get(k);
          macs(h, H[k], v.x, v.y);
        }
      C[c] = h.H + (long long)hi32(h.M);
    }
    bool plain;
    const int u = max(run_exponent<false>(f, plain) + 1 - er + uf, rho + ue);
    const int j = min(u - rho - sE, 62);                    // >= 0
    const long long hj = (1LL << j) >> 1;
#pragma unroll
    for (int c = 0; c < L; ++c) C[c] = (C[c] + hj) >> j;
    fwht(C);
    const int d = u - 1 + er, k = u + er - kBits;
    long long X[L];
    if (__builtin_expect(plain, 1)) {
#pragma unroll
      for (int m = 0; m < L; ++m) X[m] = to_fixed_positive(f[m], d - (__double2hiint(f[m]) >> 20));
    } else {
#pragma unroll
      for (int m = 0; m < L; ++m) X[m] = to_fixed_any(f[m], d);
    }
    int low = 0x7FFFFFFF;
#pragma unroll
    for (int m = 0; m < L; ++m) {
      int dh, dl;
      split_balanced(C[m] - X[m], dh, dl);
      const int2 om = R.get(m);
      Acc q{0, half};
      macs(q, Cx{om.x, om.y}, dh, dl);
      const long long change = collect(q, 2 + eo + sb);
      if constexpr (SLOW) f[m] += from_fixed(change, k - sb);
      X[m] += change;
      low = min(low, hi32(X[m]));
    }
    if constexpr (SLOW) {
    } else if (__builtin_expect(low > 0, 1)) {
#pragma unroll
      for (int m = 0; m < L; ++m) f[m] = from_fixed_positive(X[m], k);
    } else {
#pragma unroll
      for (int m = 0; m < L; ++m) f[m] = from_fixed_any(X[m], k);
    }
    double* o = ob + p0;
#pragma unroll
    for (int m = 0; m < L; ++m, o += P) *o = f[m];
    if (nimg) {
#pragma unroll 1
      for (int i = 0; i < nimg; ++i) {
        o = ob + p0 + img[i];
#pragma unroll
        for (int m = 0; m < L; ++m, o += P) *o = f[m];
      }
    }
  };
#pragma unroll 1
  for (int g = 0; g < T::ND; ++g) {
    const long long X = tb.dir_n[g][0] * W[0], Y = tb.dir_n[g][1] * W[1], Z = tb.dir_n[g][2] * W[2];
    const long long r0 = O0 - X, r1 = O0 + X;
    const long long Q4[4] = {r0 - Y, r1 - Y, r0 + Y, r1 + Y};
#pragma unroll
    for (int m = 0; m < 8; ++m) R.set(m, (m & 4) ? Q4[m & 3] + Z : Q4[m & 3] - Z);
#pragma unroll 1
    for (int r = tb.dir_first[g]; r < tb.dir_first[g + 1]; ++r)
      relax_run(Int<8>{}, tb.H8[r], tb.off8[r], tb.first8[r], tb.er8[r], tb.rho8[r], 7);
  }
#pragma unroll
  for (int r = 0; r < T::NT; ++r) {
    constexpr int L = T::LT;
    const int mask = tail_mask<ORDER>(r);
#pragma unroll
    for (int m = 0; m < L; ++m) {
      const int neg = spread(mask, m);
      long long om = O0;
#pragma unroll
      for (int i = 0; i < 3; ++i)
        if (mask >> i & 1) {
          const long long w = tb.nT[r][i] * W[i];
          om += (neg >> i & 1) ? w : -w;
        }
      R.set(m, om);
    }
    relax_run(Int<L>{}, tb.HT[r], tb.offT[r], tb.firstT[r], tb.erT[r], tb.rhoT[r], mask);
  }
}

// Fields of f(t): the populations pulled from f*(t-1) (after a step) or, at
// t = 0, f*(0) = f^eq itself: n, ux, uy, uz, T, eps (n NaN without a Landau frame, all of
// them NaN where a population is not finite).
template <int ORDER, typename S>
__global__ void __launch_bounds__(128, ORDER == 2 ? 7 : 6) k_fields3x(const __grid_constant__ Tables3x<ORDER> tb,
                                                  const __grid_constant__ Fields3Args<S> a) {
  const Scalars3& s = a.s;
  const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 4 + threadIdx.y, z = blockIdx.z;
  if (x >= s.nx || y >= s.ny || z >= s.nz) return;
  long long m[kMom3];
  int E;
  moment_sums<ORDER, S>(tb, a.fin + sidx3(s, x, y, z), s.plane, a.pull != 0, m, E);
  double N[4], T00, t[3], Sm[6];
  moment_values(m, tb.sk, N, T00, t, Sm);
  const Cell3 c = landau3x(N, T00, t, Sm);
  const bool ok = c.ok && E > 128 && E < 2040;
  const double nan = __longlong_as_double(0x7ff8000000000000LL);
  const bool finite = E < kNotFinite / 2;
  const long long cell = ((long long)z * s.ny + y) * s.nx + x, nc = (long long)s.nx * s.ny * s.nz;
  a.out[cell] = ok ? scaled(c.n, E - 1023) : nan;
  a.out[nc + cell] = finite ? c.u[0] : nan;
  a.out[2 * nc + cell] = finite ? c.u[1] : nan;
  a.out[3 * nc + cell] = finite ? c.u[2] : nan;
  a.out[4 * nc + cell] = finite ? quotient(third(c.L), c.n) : nan;
  a.out[5 * nc + cell] = finite ? scaled(c.L, E - 1023) : nan;
}

dim3 grid3x(const Scalars3& s) { return dim3((s.nx + 31) / 32, (s.ny + 3) / 4, s.nz); }

}  // namespace

template <int ORDER>
cudaError_t launch_step3x(const Tables3x<ORDER>& tb, const Step3Args<double>& a, cudaStream_t st) {
  if (a.s.Q != Tables3x<ORDER>::Q) return cudaErrorInvalidValue;
  if (!(a.s.tau <= kSlowTau)) k_step3x<ORDER, true><<<grid3x(a.s), dim3(32, 4), 0, st>>>(tb, a);
  else k_step3x<ORDER, false><<<grid3x(a.s), dim3(32, 4), 0, st>>>(tb, a);
  return cudaGetLastError();
}
template <int ORDER, typename S>
cudaError_t launch_fields3x(const Tables3x<ORDER>& tb, const Fields3Args<S>& a, cudaStream_t st) {
  if (a.s.Q != Tables3x<ORDER>::Q) return cudaErrorInvalidValue;
  k_fields3x<ORDER, S><<<grid3x(a.s), dim3(32, 4), 0, st>>>(tb, a);
  return cudaGetLastError();
}

template cudaError_t launch_step3x<2>(const Tables3x<2>&, const Step3Args<double>&, cudaStream_t);
template cudaError_t launch_step3x<3>(const Tables3x<3>&, const Step3Args<double>&, cudaStream_t);
template cudaError_t launch_fields3x<2, double>(const Tables3x<2>&, const Fields3Args<double>&, cudaStream_t);
template cudaError_t launch_fields3x<2, float>(const Tables3x<2>&, const Fields3Args<float>&, cudaStream_t);
template cudaError_t launch_fields3x<3, double>(const Tables3x<3>&, const Fields3Args<double>&, cudaStream_t);
template cudaError_t launch_fields3x<3, float>(const Tables3x<3>&, const Fields3Args<float>&, cudaStream_t);

}  // namespace rlbm
