// The (2+1)-d FP64 step of the orbit-symmetric stencils (orders 2 and 3,
// massless and massive, on-lattice and bilinear) with the population sums in
// 64-bit fixed point (fx64.cuh), as step3x.cu does it in (3+1)-d.
//
// The stencil is a list of sign quartets (a, b), (-a, b), (a, -b), (-a, -b),
// axis quartets and a rest population.  Per quartet a Walsh-Hadamard transform
// of the streamed values leaves one product per moment, and the four
// equilibrium values come from its first row's partial sums over the four
// parity classes of the basis, transformed back.  The streamed values stay in
// a shared-memory column between the two passes (the bilinear pull, four FP64
// operations per population, runs once), except for the on-lattice order-3
// stencils, whose 45 to 65 doubles per thread would leave three blocks per SM:
// they are pulled again.
//
// What bounds it: latency at 20 warps per SM.  170 (order 2) and 190 (order 3)
// instructions per population and step fill 49 % and 39 % of the issue slots, the FP64
// pipe is busy 50 % and 48 % (the sums in FP64 held it at 85 % and took 540 to 980
// operations per cell of it, 80 to 160 are left); a warp waits for the arithmetic before it
// (2.2 and 2.7 cycles per issued instruction), for shared memory and the FP64 pipe (2.0
// and 2.7) and for the populations (1.5).  517 x 333, massless order 2: 56 us per
// step (chained) and 18 us for the fields against 190 and 139 us; 512 x 512, m = 5,
// order 3 (49 populations): 167 and 40 us against 445 and 300 us.
#include <cuda_runtime.h>

#include "fxstep.cuh"
#include "step2x.h"
#include "step_impl.cuh"

namespace rlbm {

namespace {

// The macroscopic state in units of 2^E (T in its own): eps U^a = T^ab U_b with
// u = U^i / U^0, (T^ij + eps delta^ij) u_j = T^0i, eps = T^00 - T^0i u_i.
struct Cell2 {
  double L, u[2], U0, n, T;
  bool ok;
};

// As landau3x: the root and u in FP32 by Newton on the secular equation, then
// (l, u) by iterative refinement with FP64 residuals, and in FP64 (frame64.cuh)
// what has not settled after six passes; T from the d = 2 EOS.
template <bool MASSLESS>
__device__ __forceinline__ Cell2 landau2x(const double (&v)[9], float k, double m) {
  const float fT = cut_float(v[3]), f0 = cut_float(v[4]), f1 = cut_float(v[5]);
  const float fxx = cut_float(v[6]), fxy = cut_float(v[7]), fyy = cut_float(v[8]);
  const float M2 = f0 * f0 + f1 * f1;
  float l = (-(1.f - k) * fT + sqrtf(fmaxf((1.f - k) * (1.f - k) * fT * fT + 4.f * k * (fT * fT - M2), 0.f))) / (2.f * k);
  float xx = 1.f, yy = 1.f, u0 = 0.f, u1 = 0.f, w = 1.f, det = 1.f, id = 1.f;
#pragma unroll 1
  for (int it = 0; it < 12; ++it) {
    xx = fxx + l;
    yy = fyy + l;
    det = xx * yy - fxy * fxy;
    id = __fdividef(1.f, det);
    u0 = (f0 * yy - fxy * f1) * id;
    u1 = (f1 * xx - fxy * f0) * id;
    w = 1.f - u0 * u0 - u1 * u1;
    const float d = __fdividef(fT - f0 * u0 - f1 * u1 - l, w);
    l += d;
    if (!(fabsf(d) > 5e-7f * l)) break;
  }
  Cell2 c;
  c.L = wide_double(l);
  c.u[0] = wide_double(u0);
  c.u[1] = wide_double(u1);
  const float iw = __fdividef(1.f, w), Axx = yy * id, Ayy = xx * id, Axy = -fxy * id;
  bool settled = false;
#pragma unroll 1
  for (int it = 0; it < 6; ++it) {
    const double r0 = fma(-v[5], c.u[1], fma(-v[4], c.u[0], v[3] - c.L));
    const double rx = fma(-v[7], c.u[1], fma(-v[6], c.u[0], fma(-c.L, c.u[0], v[4])));
    const double ry = fma(-v[8], c.u[1], fma(-v[7], c.u[0], fma(-c.L, c.u[1], v[5])));
    const float x = cut_float(rx), y = cut_float(ry);
    const float d = (cut_float(r0) - u0 * x - u1 * y) * iw;
    const float ex = x - u0 * d, ey = y - u1 * d;
    const float cx = Axx * ex + Axy * ey, cy = Axy * ex + Ayy * ey;
    c.L += wide_double(d);
    c.u[0] += wide_double(cx);
    c.u[1] += wide_double(cy);
    settled = fabsf(d) <= 1e-12f * l && fabsf(cx) + fabsf(cy) <= 1e-9f * w * w;
    if (it >= 1 && settled) break;
  }
  bool good = true;
  if (__builtin_expect(!(settled && det > 0.f && w > 0.f), 0)) {
    const double t[3] = {v[4], v[5], 0.0}, S[6] = {v[6], v[7], 0.0, v[8], 0.0, 0.0};
    const Frame64 f = frame64(v[3], t, S);
    good = f.ok;
    c.L = f.l;
    c.u[0] = f.u[0];
    c.u[1] = f.u[1];
  }
  const double w2 = fma(-c.u[1], c.u[1], fma(-c.u[0], c.u[0], 1.0));
  c.U0 = reciprocal_sqrt(w2);
  c.n = c.U0 * fma(-c.u[1], v[2], fma(-c.u[0], v[1], v[0]));
  if (MASSLESS) {
    c.T = quotient(0.5 * c.L, c.n);
  } else {
    const double e = quotient(c.L, c.n);
    const double r = fma(e, e, 4.0 * m * (e - m)), y = reciprocal_sqrt(r), q = r * y;
    c.T = 0.25 * ((e - 2.0 * m) + fma(0.5 * y, fma(-q, q, r), q));
  }
  // (NaN where the massive EOS has no real temperature: eps / n below 0.83 m)
  c.ok = good && __double2hiint(w2) > 0 && between(c.n, -100, 100) && between(c.L, -100, 100) &&
         between(c.T, -1022, 127);
  return c;
}

// Maxwell-Juttner moments of the basis of setup.h (App. B, the closed forms of
// eq_moments without a reference state).  The scalar-like members <1>, <p0 - m>,
// <pp> and <(p0 - m) pp> enter f^eq with terms up to several hundred times f (m > 0):
// their separate roundings are no change of (n, T) and made most of a step's
// error, so their leading products carry a second word lo (has_lo).
template <int K, bool MASSLESS>
__device__ constexpr bool has_lo(int k) {
  return !MASSLESS && (k == 0 || k == 6 || k == 8 || (K == 16 && (k == 1 || k == 9 || k == 11)));
}
template <int K, bool MASSLESS>
__device__ __forceinline__ void mj_moments2x(const Cell2& c, double Ux, double Uy, double m, double (&M)[K],
                                             double (&lo)[K]) {
  const double n = c.n, T = c.T, U0 = c.U0;
  double imT, iml, r2, nT, nTl;          // 1 / (m + T) and n T with their second words; (m^2 + 3mT + 3T^2) / (m + T)
  if (MASSLESS) {
    imT = iml = 0.0;                     // (unused)
    r2 = 3.0 * T;
    nT = 0.5 * c.L;
    nTl = 0.0;
    M[0] = quotient(n, T);
  } else {
    const double mT = m + T, mTl = T - (mT - m);
    imT = quotient(1.0, mT);
    iml = imT * fma(-mTl, imT, fma(-mT, imT, 1.0));
    r2 = quotient(fma(3.0 * T, mT, m * m), mT);
    nT = n * T;
    nTl = fma(n, T, -nT);
    M[0] = n * imT;
    lo[0] = fma(n, iml, fma(n, imT, -M[0]));
  }
  M[2] = n * Ux;
  M[3] = n * Uy;
  const double nr2 = n * r2, qx = nr2 * Ux, qy = nr2 * Uy;
  M[7] = qx * Uy;
  if (MASSLESS) {
    M[6] = fma(qx, Ux, nT);
    M[8] = fma(qy, Uy, nT);
  } else {
    M[6] = M[8] = nT;
    lo[6] = fma(qx, Ux, nTl);
    lo[8] = fma(qy, Uy, nTl);
  }
  if constexpr (K == 9) {
    M[1] = n * U0;
    M[4] = qx * U0;
    M[5] = qy * U0;
  } else {
    const double s2 = fma(Ux, Ux, Uy * Uy), U0m1 = quotient(s2, U0 + 1.0);
    double r3, A2, A3;                   // r2 U0 - m, r3 U0 - m r2
    if (MASSLESS) {
      r3 = 15.0 * T * T;
      A2 = fma(r2, U0m1, 3.0 * T);
      A3 = fma(r3, U0m1, r3);
      M[1] = n * (1.0 + U0m1);
    } else {
      r3 = fma(fma(fma(15.0, T, 15.0 * m), T, 6.0 * m * m), T, m * m * m) * imT;
      const double c2 = fma(3.0, T, 2.0 * m) * imT, c3 = 3.0 * fma(fma(5.0, T, 4.0 * m), T, m * m) * imT;
      A2 = fma(r2, U0m1, T * c2);
      A3 = fma(r3, U0m1, T * c3);
      // n T / (m + T) + n (U0 - 1)
      M[1] = nT * imT;
      lo[1] = fma(n, U0m1, fma(nT, iml, fma(nTl, imT, fma(nT, imT, -M[1]))));
    }
    M[4] = M[2] * A2;
    M[5] = M[3] * A2;
    const double nA3 = n * A3, ax = nA3 * Ux;
    M[10] = ax * Uy;
    if (MASSLESS) {
      const double D5 = nT * A2;
      M[9] = fma(ax, Ux, D5);
      M[11] = fma(nA3 * Uy, Uy, D5);
    } else {
      // n T A2 = 2 n T^2 + n T (T^2 / (m + T) + r2 (U0 - 1))
      const double T2 = 2.0 * T, D = nT * T2;
      const double Dl = fma(nT, fma(T * T, imT, r2 * U0m1), fma(nTl, T2, fma(nT, T2, -D)));
      M[9] = M[11] = D;
      lo[9] = fma(ax, Ux, Dl);
      lo[11] = fma(nA3 * Uy, Uy, Dl);
    }
    const double nr3 = n * r3, t = nT * r2, bx = nr3 * Ux * Ux, by = nr3 * Uy * Uy;
    M[12] = fma(bx, Ux, 3.0 * t * Ux);
    M[13] = fma(bx, Uy, t * Uy);
    M[14] = fma(by, Ux, t * Ux);
    M[15] = fma(by, Uy, 3.0 * t * Uy);
  }
}

__device__ __forceinline__ void wht4(long long (&X)[4]) {
  const long long a = X[0] + X[1], b = X[0] - X[1], c = X[2] + X[3], d = X[2] - X[3];
  X[0] = a + c;
  X[1] = b + d;
  X[2] = a - c;
  X[3] = b - d;
}

template <int MODE>
__device__ __forceinline__ double pull2x(const Tables2x& tb, const double* __restrict__ base, int i) {
  const double* p = base + tb.off[i];
  if constexpr (MODE == kOnLattice) return __ldg(p);
  double f = tb.bw[i][0] * __ldg(p);
  f = fma(tb.bw[i][1], __ldg(p + 1), f);
  f = fma(tb.bw[i][2], __ldg(p + tb.pitch), f);
  return fma(tb.bw[i][3], __ldg(p + tb.pitch + 1), f);
}

// The moments N0 Nx Ny T00 T0x T0y Txx Txy Tyy of the populations pull(i), in
// units of 2^(E + sk - kBitsM4 + 64 - kCoefM).
template <typename F>
__device__ __forceinline__ void moment_sums2x(const Tables2x& tb, F&& pull, long long (&m)[9], int& E) {
  E = -4096;
#pragma unroll
  for (int j = 0; j < 9; ++j) m[j] = 0;
  auto units = [&](auto& f, int ep, auto& X) {
    constexpr int L = sizeof(X) / sizeof(X[0]);
    bool plain;
    raise_scale<0>(m, E, run_exponent<true>(f, plain) + ep + 1);
    const int d = E - 1 - ep;
    if (__builtin_expect(plain, 1)) {
#pragma unroll
      for (int q = 0; q < L; ++q) X[q] = to_fixed_cut<kBitsM4>(f[q], d - (__double2hiint(f[q]) >> 20));
    } else {
#pragma unroll
      for (int q = 0; q < L; ++q) X[q] = to_fixed_any(f[q], d) << (kBitsM4 - kBits);
    }
  };
#pragma unroll 2
  for (int r = 0; r < tb.nq; ++r) {
    double f[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) f[q] = pull(tb.firstq[r] + q);
    long long X[4];
    units(f, tb.epq[r], X);
    wht4(X);
    int h[4], l[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) split_balanced(X[c], h[c], l[c]);
    constexpr int cls[9] = {0, 1, 2, 0, 1, 2, 0, 3, 0};
#pragma unroll
    for (int j = 0; j < 9; ++j) add_product(m[j], tb.Mq[r][j], h[cls[j]], l[cls[j]]);
  }
#pragma unroll 1
  for (int r = 0; r < tb.na; ++r) {
    double f[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) f[q] = pull(tb.firsta[r] + q);
    long long X[4];
    units(f, tb.epa[r], X);
    const long long S1 = X[0] + X[1], D1 = X[0] - X[1], S2 = X[2] + X[3], D2 = X[2] - X[3];
    int h[5], l[5];
    split_balanced(S1 + S2, h[0], l[0]);
    split_balanced(D1, h[1], l[1]);
    split_balanced(D2, h[2], l[2]);
    split_balanced(S1, h[3], l[3]);
    split_balanced(S2, h[4], l[4]);
    add_product(m[0], tb.Ma[r][0], h[0], l[0]);
    add_product(m[1], tb.Ma[r][1], h[1], l[1]);
    add_product(m[2], tb.Ma[r][1], h[2], l[2]);
    add_product(m[3], tb.Ma[r][3], h[0], l[0]);
    add_product(m[4], tb.Ma[r][4], h[1], l[1]);
    add_product(m[5], tb.Ma[r][4], h[2], l[2]);
    add_product(m[6], tb.Ma[r][6], h[3], l[3]);
    add_product(m[8], tb.Ma[r][6], h[4], l[4]);
  }
  if (tb.nr) {
    double f[1] = {pull(tb.firstr)};
    long long X[1];
    units(f, tb.epr, X);
    int h, l;
    split_balanced(X[0], h, l);
    add_product(m[0], tb.Mr[0], h, l);
    add_product(m[3], tb.Mr[1], h, l);
  }
}

// Shared memory per block: limbs of the K basis moments and of four rates, the
// streamed populations.
constexpr int kThreads2x = 128;
constexpr bool kept2x(int K, int mode) { return K == 9 || mode == kBilinear; }
constexpr size_t shared2x(int K, int mode, int Q) {
  return (size_t)(K + 4 + (kept2x(K, mode) ? Q : 0)) * kThreads2x * 8;
}

// The relaxation in FP64, for a cell whose rate or equilibrium the fixed point does
// not hold (a tau of its field that is zero, NaN or below 1/64, say), or that has no
// frame and keeps its populations.  v: K basis moments in units of 2^E, then
// tau^-1 U0 and vscale tau^-1 U^i (a column of the shared memory); kept: the
// streamed populations, or null where they are read again.
template <int K>
__device__ __noinline__ void relax_plain2(const Tables2x& tb, const StepArgs<double>& a, const double* v, const double* kept,
                                          const double* base, int E, bool frame, int x, int y) {
  const Scalars& s = a.s;
  const double o0 = v[K * kThreads2x], kx = v[(K + 1) * kThreads2x], ky = v[(K + 2) * kThreads2x];
  // sx, sy: the signs of the odd members of p^x and p^y, 0 where the row has none
  auto relax = [&](int i, const Cx* H, double sx, double sy, double om, int e) {
    double sum = 0.0;
    if (!frame) om = 0.0;
#pragma unroll 1
    for (int k = 0; frame && k < K; ++k) {
      sum = fma((mono_ax(k) ? sx : 1.0) * (mono_ay(k) ? sy : 1.0) * constant_value(H[k], tb.hk[k]), v[k * kThreads2x], sum);
    }
    const double f = kept ? kept[i * kThreads2x] : __ldg(base + tb.off[i]);
    const double g = fma(om, (frame ? scaled(sum, E - 1023 + e - kCoefH) : 0.0) - f, f);
    a.fout[(base - a.fin) + (long long)i * s.iplane] = g;
    for_each_halo_image(s, x, y, [&](long long hi) { a.fout[hi + (long long)i * s.iplane] = g; });
  };
#pragma unroll 1
  for (int q = 0; q < 4 * tb.nq; ++q) {
    const int r = q >> 2;
    const double sx = (q & 1) ? -1.0 : 1.0, sy = (q & 2) ? -1.0 : 1.0;
    relax(tb.firstq[r] + (q & 3), tb.Hq[r], sx, sy, o0 - sx * tb.nq_x[r] * kx - sy * tb.nq_y[r] * ky, tb.erq[r] + tb.rhoq[r]);
  }
#pragma unroll 1
  for (int q = 0; q < 4 * tb.na; ++q) {
    const int r = q >> 2, along = (q >> 1) & 1;
    const double sg = (q & 1) ? -1.0 : 1.0;
    relax(tb.firsta[r] + (q & 3), tb.Ha[r][along], along ? 0.0 : sg, along ? sg : 0.0,
          o0 - sg * tb.na_x[r] * (along ? ky : kx), tb.era[r] + tb.rhoa[r]);
  }
  if (tb.nr) relax(tb.firstr, tb.Hr, 0.0, 0.0, o0, tb.err + tb.rhor);
}

template <int K, int MODE, bool MASSLESS, bool SLOW>
__global__ void __launch_bounds__(kThreads2x, K == 9 || MODE == kOnLattice ? 5 : 4) k_step2x(const __grid_constant__ Tables2x tb,
                                                                        const __grid_constant__ StepArgs<double> a,
                                                                        double inv_tau) {
  extern __shared__ int2 columns[];
  const Scalars& s = a.s;
  const double* const fin = chain_begin(a.fin);
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= s.nx || y >= s.ny) return;
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  const Column M{columns + tid};                       // basis moments in units of 2^(xg - 62) 2^E
  const Column R{M.s + K * kThreads2x};                // the rates of a quartet
  double* const F = (double*)(R.s + 4 * kThreads2x);   // streamed populations
  const long long si = sidx(s, x, y);
  const double* __restrict__ base = fin + si;
  double* const ob = a.fout + si;
  const int P = s.iplane;

  auto pull = [&](int i) {
    const double f = pull2x<MODE>(tb, base, i);
    if constexpr (kept2x(K, MODE)) F[i * kThreads2x] = f;
    return f;
  };
  auto again = [&](int i) {
    if constexpr (kept2x(K, MODE)) return F[i * kThreads2x];
    else return __ldg(base + tb.off[i]);
  };

  int uf, ue, eo, sb = 0;    // the unit 2^(u - kBits) of a quartet: u = max(its exponent + uf, rho + ue)
  long long O0, W[2];        // tau^-1 U0 and vscale tau^-1 U^i in units of 2^(eo - 62)
  {
    long long m[9];
    int E;
    moment_sums2x(tb, pull, m, E);
    double v[9];
#pragma unroll
    for (int j = 0; j < 9; ++j) v[j] = from_fixed(m[j], 1023 + tb.sk[j] - kBitsM4 + 64 - kCoefM);
    const Cell2 c = landau2x<MASSLESS>(v, s.kappa_guess, s.m);
    const bool ok = c.ok && E > 128 && E < 2040;
    const double Ux = c.u[0] * c.U0, Uy = c.u[1] * c.U0;
    double Mk[K], lo[K];
    mj_moments2x<K, MASSLESS>(c, Ux, Uy, s.m, Mk, lo);
    float sum = 0.f;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      float v = fabsf(cut_float(Mk[k]));
      if (has_lo<K, MASSLESS>(k)) v += fabsf(cut_float(lo[k]));
      sum += v * __uint_as_float((unsigned)(127 + tb.hk[k]) << 23);
    }
    double it;               // 1 / tau
    if (s.tau_mode == 1) it = 1.0 / chained(a.tau_field)[y * s.nx + x];
    else if (s.tau_mode == 2) it = c.T / s.tau_coef;
    else it = inv_tau;
    const double o0 = it * c.U0, kl = it * tb.vscale;
    const int xg = above(sum), xo = above(2.f * fabsf(cut_float(o0)));
    // (a population's unit leaves room for rate times population: with rates from 64 on
    // less than FP64 would be left of it)
    const bool rate = (__double2hiint(o0) & 0x7FFFFFFF) < (1023 + 6) << 20;      // finite, |o0| < 2^6
    // (moments within the float range, whatever U and T within these)
    const bool fits = E > 320 && between(c.n, -28, 28) && between(c.L, -28, 28) && between(c.T, -30, 24) && between(c.U0, -1, 10);
    if (__builtin_expect(!(ok && rate && fits && xg < 60 && xg > -60), 0)) {
      // no Landau frame: counted, left unrelaxed (a population that is not finite becomes NaN)
      if (!ok) atomicAdd(a.status, 1ULL);
      double* const v = (double*)M.s;
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const double f = has_lo<K, MASSLESS>(k) ? Mk[k] + lo[k] : Mk[k];
        v[k * kThreads2x] = f;
      }
      v[K * kThreads2x] = o0;
      v[(K + 1) * kThreads2x] = kl * Ux;
      v[(K + 2) * kThreads2x] = kl * Uy;
      relax_plain2<K>(tb, a, v, kept2x(K, MODE) ? F : nullptr, base, E, ok, x, y);
      return;
    }
    uf = max(0, xo - 2);
    ue = E + xg + max(0, xo - 3);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      long long v = scaled_integer(Mk[k], tb.hk[k] + 62 - xg);
      if (has_lo<K, MASSLESS>(k)) v += scaled_integer(lo[k], tb.hk[k] + 62 - xg);
      M.set(k, v);
    }
    eo = max(xo, SLOW ? kSlowestRate : -2);
    if constexpr (SLOW) sb = max(-eo, 0);
    O0 = scaled_integer(o0, 62 - eo);
    W[0] = scaled_integer(kl * Ux, 62 - eo);
    W[1] = scaled_integer(kl * Uy, 62 - eo);
  }
  const bool edge = (s.boundary == 0 ? (x < s.hx || x >= s.nx - s.hx) : (x == 0 || x == s.nx - 1)) || y < s.hy ||
                    y >= s.ny - s.hy;
  const long long half = 1LL << (29 - eo - sb);             // half a unit of the relaxation's sum
  const int sE = ue - max(0, uf - 1);                       // E + xg
  // relaxation of a set of L populations from its class sums C (in units of 2^(rho + sE - 64 + ...)) and rates R
  auto relax = [&](auto tag, int first, int er, int rho, long long (&C)[decltype(tag)::value], auto&& transform) {
    constexpr int L = decltype(tag)::value;
    double f[L];
#pragma unroll
    for (int q = 0; q < L; ++q) f[q] = again(first + q);
    bool plain;
    const int u = max(run_exponent<false>(f, plain) + 1 - er + uf, rho + ue);
    const int j = min(u - rho - sE, 62);                    // >= 0
    const long long hj = (1LL << j) >> 1;
#pragma unroll
    for (int c = 0; c < L; ++c) C[c] = (C[c] + hj) >> j;
    transform(C);
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
#pragma unroll
    for (int m = 0; m < L; ++m) ob[(first + m) * P] = f[m];
    if (edge) {
      for_each_halo_image(s, x, y, [&](long long hi) {
#pragma unroll
        for (int m = 0; m < L; ++m) a.fout[hi + (long long)(first + m) * P] = f[m];
      });
    }
  };
  auto total = [&](const Acc& h) { return h.H + (long long)hi32(h.M); };
#pragma unroll 1
  for (int r = 0; r < tb.nq; ++r) {
    const long long X = tb.nq_x[r] * W[0], Y = tb.nq_y[r] * W[1];
    R.set(0, O0 - X - Y);
    R.set(1, O0 + X - Y);
    R.set(2, O0 - X + Y);
    R.set(3, O0 + X + Y);
    long long C[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      Acc h{0, 0x80000000LL};
#pragma unroll
      for (int k = 0; k < K; ++k)
        if (mono_ax(k) + 2 * mono_ay(k) == c) {
          const int2 v = M.get(k);
          macs(h, tb.Hq[r][k], v.x, v.y);
        }
      C[c] = total(h);
    }
    relax(Int<4>{}, tb.firstq[r], tb.erq[r], tb.rhoq[r], C, [](long long (&c)[4]) { wht4(c); });
  }
#pragma unroll 1
  for (int r = 0; r < tb.na; ++r) {
    const long long X = tb.na_x[r] * W[0], Y = tb.na_x[r] * W[1];
    R.set(0, O0 - X);
    R.set(1, O0 + X);
    R.set(2, O0 - Y);
    R.set(3, O0 + Y);
    long long C[4];          // even and odd sums of (p, 0), then of (0, p)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      Acc h{0, 0x80000000LL};
#pragma unroll
      for (int k = 0; k < K; ++k)
        if (mono_ax(k) + 2 * mono_ay(k) == (c == 1 ? 1 : c == 3 ? 2 : 0)) {
          const int2 v = M.get(k);
          macs(h, tb.Ha[r][c >> 1][k], v.x, v.y);
        }
      C[c] = total(h);
    }
    relax(Int<4>{}, tb.firsta[r], tb.era[r], tb.rhoa[r], C, [](long long (&c)[4]) {
      const long long e = c[0], o = c[1], g = c[2], p = c[3];
      c[0] = e + o;
      c[1] = e - o;
      c[2] = g + p;
      c[3] = g - p;
    });
  }
  if (tb.nr) {
    R.set(0, O0);
    Acc h{0, 0x80000000LL};
#pragma unroll
    for (int k = 0; k < K; ++k)
      if (!mono_ax(k) && !mono_ay(k)) {
        const int2 v = M.get(k);
        macs(h, tb.Hr[k], v.x, v.y);
      }
    long long C[1] = {total(h)};
    relax(Int<1>{}, tb.firstr, tb.err, tb.rhor, C, [](long long (&)[1]) {});
  }
}

// a warp covers a row segment; a grid of one row takes it in blocks of one row
dim3 block2x(int ny) { return ny == 1 ? dim3(kThreads2x, 1) : dim3(32, kThreads2x / 32); }
dim3 grid2x(const Scalars& s, dim3 block) { return dim3((s.nx + block.x - 1) / block.x, (s.ny + block.y - 1) / block.y); }

// Fields of f(t) (the populations streamed from f*(t-1), or f*(0) in place).
template <int MODE, bool MASSLESS>
__global__ void __launch_bounds__(kThreads2x, 8) k_fields2x(const __grid_constant__ Tables2x tb,
                                                         const __grid_constant__ MomentArgs<double> a) {
  const Scalars& s = a.s;
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= s.nx || y >= s.ny) return;
  const double* __restrict__ base = a.fin + sidx(s, x, y);
  auto pull = [&](int i) { return a.gather ? pull2x<MODE>(tb, base, i) : __ldg(base + i * s.iplane); };
  long long m[9];
  int E;
  moment_sums2x(tb, pull, m, E);
  double v[9];
#pragma unroll
  for (int j = 0; j < 9; ++j) v[j] = from_fixed(m[j], 1023 + tb.sk[j] - kBitsM4 + 64 - kCoefM);
  const Cell2 c = landau2x<MASSLESS>(v, s.kappa_guess, s.m);
  const bool ok = c.ok && E > 128 && E < 2040;
  if (!ok) atomicAdd(a.status, 1ULL);
  const int cell = y * s.nx + x;
  const int k2 = E - 1023;
  const double nan = __longlong_as_double(0x7ff8000000000000LL);
  const bool finite = E < kNotFinite / 2;                // (the populations)
  const double f[5] = {scaled(c.n, k2), c.u[0], c.u[1], c.T, scaled(c.L, k2)};
#pragma unroll
  for (int k = 0; k < 5; ++k)
    if (a.out[k]) a.out[k][cell] = finite ? f[k] : nan;
#pragma unroll
  for (int j = 0; j < 3; ++j)
    if (a.N) a.N[(size_t)j * s.ncell + cell] = finite ? scaled(v[j], k2) : nan;
#pragma unroll
  for (int j = 0; j < 6; ++j)
    if (a.Tab) a.Tab[(size_t)j * s.ncell + cell] = finite ? scaled(v[3 + j], k2) : nan;
}

template <int MODE, bool MASSLESS>
cudaError_t launch_fields(const Tables2x& tb, const MomentArgs<double>& a, cudaStream_t st) {
  const dim3 block = block2x(a.s.ny);
  k_fields2x<MODE, MASSLESS><<<grid2x(a.s, block), block, 0, st>>>(tb, a);
  return cudaGetLastError();
}

template <int K, int MODE, bool MASSLESS, bool SLOW>
cudaError_t launch2x(const Tables2x& tb, const StepArgs<double>& a, cudaStream_t st) {
  const dim3 block = block2x(a.s.ny), grid = grid2x(a.s, block);
  const size_t bytes = shared2x(K, MODE, tb.Q);
  const auto kernel = k_step2x<K, MODE, MASSLESS, SLOW>;
  if (bytes > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shared2x(K, MODE, kMaxQ));
    if (e != cudaSuccess) return e;
  }
  return launch_chained(!a.s.plain, kernel, grid, block, bytes, st, tb, a, 1.0 / a.s.tau);
}

template <int K, int MODE>
cudaError_t launch2x(const Tables2x& tb, const StepArgs<double>& a, cudaStream_t st) {
  if (a.s.tau_mode != 0 || !(a.s.tau <= kSlowTau))
    return a.s.massless ? launch2x<K, MODE, true, true>(tb, a, st) : launch2x<K, MODE, false, true>(tb, a, st);
  return a.s.massless ? launch2x<K, MODE, true, false>(tb, a, st) : launch2x<K, MODE, false, false>(tb, a, st);
}

}  // namespace

cudaError_t launch_step2x(const Tables2x& tb, const StepArgs<double>& a, int mode, cudaStream_t st) {
  if (a.s.K == 9)
    return mode == kOnLattice ? launch2x<9, kOnLattice>(tb, a, st) : launch2x<9, kBilinear>(tb, a, st);
  if (a.s.K == 16)
    return mode == kOnLattice ? launch2x<16, kOnLattice>(tb, a, st) : launch2x<16, kBilinear>(tb, a, st);
  return cudaErrorInvalidValue;
}

cudaError_t launch_fields2x(const Tables2x& tb, const MomentArgs<double>& a, int mode, cudaStream_t st) {
  if (mode == kOnLattice)
    return a.s.massless ? launch_fields<kOnLattice, true>(tb, a, st) : launch_fields<kOnLattice, false>(tb, a, st);
  return a.s.massless ? launch_fields<kBilinear, true>(tb, a, st) : launch_fields<kBilinear, false>(tb, a, st);
}

}  // namespace rlbm
