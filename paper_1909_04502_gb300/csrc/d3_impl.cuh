// Device helpers of the (3+1)-d massless steps (step3.cu: order 2; step3q.cu:
// order 3; step3x.cu: FP64): layout, periodic images, the 4 x 4 Landau frame
// (Sec. 4) in FP32 with an FP64 correction, and the Maxwell-Juttner moments of the
// bases kBasis3 / kBasis3o3 (App. B, d = 3, m = 0).
#pragma once
#include <cuda_runtime.h>

#include "d3.h"
#include "fpconv.cuh"

namespace rlbm {
namespace {

__device__ __forceinline__ long long sidx3(const Scalars3& s, int x, int y, int z) {
  return (long long)(z + s.h) * s.slab + (long long)(y + s.h) * s.pitch + (x + s.px);
}

// periodic images of coordinate c in [-h, n + h), other than c itself
__device__ __forceinline__ int images1(int c, int n, int h, int (&out)[2]) {
  int k = 0;
  if (c + n < n + h) out[k++] = c + n;
  if (c - n >= -h) out[k++] = c - n;
  return k;
}

// right null vector of B from the first column of adj(B):
// v_i = (-1)^i det(B without row 0 and column i), each 3 x 3 minor expanded
// along row 1 over the six 2 x 2 minors c_ab of rows 2 and 3; B v = det(B) e_0,
// so det(B) = sum_i B[0][i] v_i.
template <typename R>
__device__ __forceinline__ void adj_col0(const R (&B)[4][4], R (&v)[4]) {
  const R c01 = B[2][0] * B[3][1] - B[2][1] * B[3][0], c02 = B[2][0] * B[3][2] - B[2][2] * B[3][0];
  const R c03 = B[2][0] * B[3][3] - B[2][3] * B[3][0], c12 = B[2][1] * B[3][2] - B[2][2] * B[3][1];
  const R c13 = B[2][1] * B[3][3] - B[2][3] * B[3][1], c23 = B[2][2] * B[3][3] - B[2][3] * B[3][2];
  v[0] = B[1][1] * c23 - B[1][2] * c13 + B[1][3] * c12;
  v[1] = -(B[1][0] * c23 - B[1][2] * c03 + B[1][3] * c02);
  v[2] = B[1][0] * c13 - B[1][1] * c03 + B[1][3] * c01;
  v[3] = -(B[1][0] * c12 - B[1][1] * c02 + B[1][2] * c01);
}

// d v / d l for B = A - l I: each minor differentiated through the diagonal
// entries it keeps (d det / d B_rr = cofactor of B_rr).
template <typename R>
__device__ __forceinline__ void dadj_col0(const R (&B)[4][4], R (&d)[4]) {
  d[0] = -((B[2][2] * B[3][3] - B[2][3] * B[3][2]) + (B[1][1] * B[3][3] - B[1][3] * B[3][1]) +
           (B[1][1] * B[2][2] - B[1][2] * B[2][1]));
  d[1] = (B[1][0] * B[3][3] - B[1][3] * B[3][0]) + (B[1][0] * B[2][2] - B[1][2] * B[2][0]);
  d[2] = (B[2][0] * B[3][3] - B[2][3] * B[3][0]) - (B[1][0] * B[2][1] - B[1][1] * B[2][0]);
  d[3] = -((B[2][0] * B[3][2] - B[2][2] * B[3][0]) + (B[1][0] * B[3][1] - B[1][1] * B[3][0]));
}

// MJ moments of the basis 1 | p0 px py pz | p0px p0py p0pz pxpx pxpy pxpz pypy
// pypz pzpz for massless particles in d = 3 (App. B): <1> = n/(2T),
// <p^a> = n U^a, <p^a p^b> = n (4T U^a U^b - T eta^ab).
__device__ __forceinline__ void mj_moments3(double n, double T, const double (&U)[4], double (&M)[14]) {
  const double q = 4.0 * n * T;
  M[0] = n / (2.0 * T);
  M[1] = n * U[0];
  M[2] = n * U[1];
  M[3] = n * U[2];
  M[4] = n * U[3];
  M[5] = q * U[0] * U[1];
  M[6] = q * U[0] * U[2];
  M[7] = q * U[0] * U[3];
  M[8] = q * U[1] * U[1] + n * T;
  M[9] = q * U[1] * U[2];
  M[10] = q * U[1] * U[3];
  M[11] = q * U[2] * U[2] + n * T;
  M[12] = q * U[2] * U[3];
  M[13] = q * U[3] * U[3] + n * T;
}


// The root of a fast flow (landau3f) in FP32 by Newton on det(A - l I) formed from
// minors at each l: the quartic's coefficients cancel one another as gamma^6.  v: T00, T0x
// T0y T0z, Txx Txy Txz Tyy Tyz Tzz and the first guess, which becomes the root;
// returns the last slope.  Out of line, in memory.
__device__ __noinline__ float fast_root3f(float* v) {
  const float A[4][4] = {{v[0], -v[1], -v[2], -v[3]},
                         {v[1], -v[4], -v[5], -v[6]},
                         {v[2], -v[5], -v[7], -v[8]},
                         {v[3], -v[6], -v[8], -v[9]}};
  float l = v[10], dp = -1.f;
#pragma unroll 1
  for (int it = 0; it < 3; ++it) {
    const float B0 = A[0][0] - l, B1 = A[1][1] - l, B2 = A[2][2] - l, B3 = A[3][3] - l;
    // 2 x 2 minors of rows (0, 1) and (2, 3) over the column pairs
    const float s0 = B0 * B1 - A[1][0] * A[0][1], s1 = B0 * A[1][2] - A[1][0] * A[0][2];
    const float s2 = B0 * A[1][3] - A[1][0] * A[0][3], s3 = A[0][1] * A[1][2] - B1 * A[0][2];
    const float s4 = A[0][1] * A[1][3] - B1 * A[0][3], s5 = A[0][2] * A[1][3] - A[1][2] * A[0][3];
    const float c5 = B2 * B3 - A[3][2] * A[2][3], c4 = A[2][1] * B3 - A[3][1] * A[2][3];
    const float c3 = A[2][1] * A[3][2] - A[3][1] * B2, c2 = A[2][0] * B3 - A[3][0] * A[2][3];
    const float c1 = A[2][0] * A[3][2] - A[3][0] * B2, c0 = A[2][0] * A[3][1] - A[3][0] * A[2][1];
    const float det = s0 * c5 - s1 * c4 + s2 * c3 + s3 * c2 - s4 * c1 + s5 * c0;
    // the slope, minus the sum of the principal 3 x 3 minors
    auto det3 = [](float a, float b, float c, float d, float e, float f, float g, float h, float i) {
      return a * (e * i - f * h) - b * (d * i - f * g) + c * (d * h - e * g);
    };
    dp = -(det3(B1, A[1][2], A[1][3], A[2][1], B2, A[2][3], A[3][1], A[3][2], B3) +
           det3(B0, A[0][2], A[0][3], A[2][0], B2, A[2][3], A[3][0], A[3][2], B3) +
           det3(B0, A[0][1], A[0][3], A[1][0], B1, A[1][3], A[3][0], A[3][1], B3) +
           det3(B0, A[0][1], A[0][2], A[1][0], B1, A[1][2], A[2][0], A[2][1], B2));
    l -= det / dp;
  }
  v[10] = l;
  return dp;
}

// FP32 storage (g = f - f_ref, f_ref at (n_ref, rest, T_ref)): the Landau root
// in FP32 (Newton on det(A - l I) from the ideal-fluid root), then one Newton
// correction whose residual is evaluated in FP64: the cofactor vector v of
// B = A - l I at the FP32 root and p(l) = B[0] . v.  The eigenvector at the
// corrected root is v + dl dv/dl (dv/dl in FP32; the remainder is O(dl^2)),
// and from it, in FP64, nu^2 = v.v, w = v.N (n = w / nu) and the numerator
// of dn = n - n_ref = (w^2 - n_ref^2 nu^2) / (nu (w + n_ref nu)); the
// quotients, U = v / nu and dT = (d_eps - 3 T_ref dn) / (3 n) (from
// eps = 3 n T) in FP32.  About 50 FP64 operations per cell; conversions on
// the integer pipe (fpconv.cuh).
struct Macro3f {
  float U0, Ux, Uy, Uz, n, T, dn, dT;
  bool ok;
};

__device__ __forceinline__ Macro3f landau3f(const float (&N)[4], const float (&Tm)[4][4], const Scalars3& s) {
  const double nr = s.n_ref, Tr = s.T_ref, er = 3.0 * nr * Tr, Pr = nr * Tr;
  const float fnr = s.f_n_ref, fTr = s.f_T_ref;
  // T^ab = (E, s; s, P) in FP32 (reference diagonal added); the mixed tensor
  // A = T eta has det(A - l I) = (l - E) D(l) + S(l), D = det(P + l I) =
  // l^3 + a1 l^2 + a2 l + a3, S = s . adj(P + l I) s = b0 l^2 + b1 l + b2
  const float E = Tm[0][0] + s.f_e_ref, x = Tm[0][1], y = Tm[0][2], z = Tm[0][3];
  const float pxx = Tm[1][1] + s.f_P_ref, pyy = Tm[2][2] + s.f_P_ref, pzz = Tm[3][3] + s.f_P_ref;
  const float pxy = Tm[1][2], pxz = Tm[1][3], pyz = Tm[2][3];
  const float cxx = pyy * pzz - pyz * pyz, cyy = pxx * pzz - pxz * pxz, czz = pxx * pyy - pxy * pxy;
  const float cxy = pxz * pyz - pxy * pzz, cxz = pxy * pyz - pxz * pyy, cyz = pxy * pxz - pyz * pxx;
  const float a1 = pxx + pyy + pzz, a2 = cxx + cyy + czz, a3 = pxx * cxx + pxy * cxy + pxz * cxz;
  const float xx = x * x, yy = y * y, zz = z * z, xy = 2.f * x * y, xz = 2.f * x * z, yz = 2.f * y * z;
  const float b0 = xx + yy + zz;
  const float b1 = a1 * b0 - (xx * pxx + yy * pyy + zz * pzz + xy * pxy + xz * pxz + yz * pyz);
  const float b2 = xx * cxx + yy * cyy + zz * czz + xy * cxy + xz * cxz + yz * cyz;
  // FP32 root from the ideal-fluid guess (P = eps / 3)
  const float k = 1.f / 3.f;
  float lam = (-(1.f - k) * E + sqrtf(fmaxf((1.f - k) * (1.f - k) * E * E + 4.f * k * (E * E - b0), 0.f))) * 1.5f;
  float dpf = -1.f;
  const float guess = lam;
#pragma unroll
  for (int it = 0; it < 3; ++it) {
    const float D = fmaf(fmaf(lam + a1, lam, a2), lam, a3), dD = fmaf(fmaf(3.f, lam, 2.f * a1), lam, a2);
    const float S = fmaf(fmaf(b0, lam, b1), lam, b2), dS = fmaf(2.f * b0, lam, b1);
    dpf = fmaf(lam - E, dD, D + dS);
    lam -= __fdividef(fmaf(lam - E, D, S), dpf);
  }
  // The coefficients serve to T^0i of about 0.95 T^00, u = 0.9 (worst error of (n, T): 1.8e-7 with
  // either form at 0.9; 7.5e-7 against 3.6e-5 at 0.98, 7.4e-5 against 1.2e-2 at 0.99).
  if (__builtin_expect(!(b0 < 0.9f * E * E), 0)) {
    float v[11] = {E, x, y, z, pxx, pxy, pxz, pyy, pyz, pzz, guess};
    dpf = fast_root3f(v);
    lam = v[10];
  }
  // FP64 residual at the FP32 root: B = A - l I with A's entries exact from
  // the FP32 sums and the FP64 reference
  const double ld = f2d_finite(lam);
  const double d0 = ld - er, d1 = Pr + ld;
  double B[4][4];
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const double t = f2d_finite(u <= v ? Tm[u][v] : Tm[v][u]);
      B[u][v] = v == 0 ? t : -t;
    }
  B[0][0] = f2d_finite(Tm[0][0]) - d0;
#pragma unroll
  for (int u = 1; u < 4; ++u) B[u][u] = -(f2d_finite(Tm[u][u]) + d1);
  double vv[4];
  adj_col0(B, vv);
  int top = 0;
  const double p = B[0][0] * vv[0] + B[0][1] * vv[1] + B[0][2] * vv[2] + B[0][3] * vv[3];
  const float dl = -__fdividef(d2f_finite(p, top), dpf);
  // the eigenvector at l + dl to first order
  const float Bf[4][4] = {{E - lam, -x, -y, -z},
                          {x, -(pxx + lam), -pxy, -pxz},
                          {y, -pxy, -(pyy + lam), -pyz},
                          {z, -pxz, -pyz, -(pzz + lam)}};
  float dv[4];
  dadj_col0(Bf, dv);
  double vc[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) vc[u] = vv[u] + f2d_finite(dl * dv[u]);
  const double nu2 = vc[0] * vc[0] - vc[1] * vc[1] - vc[2] * vc[2] - vc[3] * vc[3];
  const double w = vc[0] * (nr + f2d_finite(N[0])) - vc[1] * f2d_finite(N[1]) - vc[2] * f2d_finite(N[2]) -
                   vc[3] * f2d_finite(N[3]);
  const double num = fma(w, w, -(nr * nr) * nu2);
  const double deps = d0 + f2d_finite(dl);
  // FP32 quotients
  const float fnu2 = d2f_finite(nu2, top);
  const float inu = rsqrtf(fnu2);
  const float fnu = fnu2 * inu;
  const float sgn = __double2hiint(vc[0]) < 0 ? -1.f : 1.f;
  const float fw = sgn * d2f_finite(w, top);
  Macro3f M;
  M.n = fw * inu;
  M.dn = __fdividef(d2f_finite(num, top), fnu * (fw + fnr * fnu));
  M.dT = __fdividef(d2f_finite(deps, top) - 3.f * fTr * M.dn, 3.f * M.n);
  M.T = fTr + M.dT;
  const float su = sgn * inu;
  M.U0 = d2f_finite(vc[0], top) * su;
  M.Ux = d2f_finite(vc[1], top) * su;
  M.Uy = d2f_finite(vc[2], top) * su;
  M.Uz = d2f_finite(vc[3], top) * su;
  // the conversions take finite values: lam and dl are not finite when a T^ab
  // or the frame is not, and the FP64 values are checked by their magnitude
  M.ok = (__double2hiint(nu2) >= kLeastFloat) && (M.n > 0.f) && (M.T > 0.f) && isfinite(M.T) && isfinite(M.dn) &&
         isfinite(M.n) && isfinite(lam) && isfinite(dl * (dv[0] + dv[1] + dv[2] + dv[3])) &&
         isfinite(N[0] + N[1] + N[2] + N[3]) && top < kNoFloat;
  return M;
}

// The rank-3 moments <p^a p^b p^c> = n (24 T^2 U^a U^b U^c - 4 T^2 (eta^ab U^c
// + eta^ac U^b + eta^bc U^a)) for the order-3 members of kBasis3o3: p0 p^i p^j
// (i <= j) and p^i p^j p^k (i <= j <= k), spatial indices 1..3.
__device__ __forceinline__ int o3_index(int k, int e) {
  // members 14-19: p0 (xx xy xz yy yz zz); 20-29: xxx xxy xxz xyy xyz xzz yyy yyz yzz zzz
  const int p2[6][2] = {{1, 1}, {1, 2}, {1, 3}, {2, 2}, {2, 3}, {3, 3}};
  const int p3[10][3] = {{1, 1, 1}, {1, 1, 2}, {1, 1, 3}, {1, 2, 2}, {1, 2, 3},
                         {1, 3, 3}, {2, 2, 2}, {2, 2, 3}, {2, 3, 3}, {3, 3, 3}};
  return k < 20 ? p2[k - 14][e] : p3[k - 20][e];
}

// Full moments of the basis (FP64 storage): K = 14 (order 2) or 30 (order 3).
template <int K>
__device__ __forceinline__ void mj_full3(double n, double T, const double (&U)[4], double (&M)[K]) {
  double M14[14];
  mj_moments3(n, T, U, M14);
#pragma unroll
  for (int k = 0; k < 14; ++k) M[k] = M14[k];
  if constexpr (K == 30) {
    const double q = 24.0 * n * T * T, r = 4.0 * n * T * T;
#pragma unroll
    for (int k = 14; k < 20; ++k) {
      const int i = o3_index(k, 0), j = o3_index(k, 1);
      M[k] = q * U[0] * U[i] * U[j] + (i == j ? r * U[0] : 0.0);
    }
#pragma unroll
    for (int k = 20; k < 30; ++k) {
      const int i = o3_index(k, 0), j = o3_index(k, 1), l = o3_index(k, 2);
      M[k] = q * U[i] * U[j] * U[l] + r * ((i == j ? U[l] : 0.0) + (i == l ? U[j] : 0.0) + (j == l ? U[i] : 0.0));
    }
  }
}

__device__ __forceinline__ float quotient32(float a, float b) {     // b normal and below 2^126
  const float r = __fdividef(1.f, b), q = a * r;
  return fmaf(fmaf(-b, q, a), r, q);
}

// Differences dM = M(n, U, T) - M(n_ref, rest, T_ref) (FP32 storage), each
// written so that it is accurate relative to itself given accurate dn, dT:
//   <1>: (dn T_ref - n_ref dT) / (2 T T_ref);  <p0>: dn U0 + n_ref (U0 - 1);
//   <p^i p^i>: 4nT (U^i)^2 + dn T + n_ref dT;
//   <p0 p^i p^i>: 24 n T^2 U0 (U^i)^2 + 4 (n T^2 (U0 - 1) + dn T^2 + n_ref dT (T + T_ref));
//   the others vanish at rest and need no rearrangement.
template <int K>
__device__ __forceinline__ void mj_delta3(const Macro3f& M, float nr, float Tr, float (&dM)[K]) {
  const float U[4] = {M.U0, M.Ux, M.Uy, M.Uz};
  const float n = M.n, T = M.T, dn = M.dn, dT = M.dT;
  const float U0m1 = quotient32(M.Ux * M.Ux + M.Uy * M.Uy + M.Uz * M.Uz, M.U0 + 1.f);
  const float q = 4.f * n * T, iso = dn * T + nr * dT;
  dM[0] = quotient32(dn * Tr - nr * dT, 2.f * T * Tr);
  dM[1] = dn * M.U0 + nr * U0m1;
  dM[2] = n * M.Ux;
  dM[3] = n * M.Uy;
  dM[4] = n * M.Uz;
  dM[5] = q * M.U0 * M.Ux;
  dM[6] = q * M.U0 * M.Uy;
  dM[7] = q * M.U0 * M.Uz;
  dM[8] = q * M.Ux * M.Ux + iso;
  dM[9] = q * M.Ux * M.Uy;
  dM[10] = q * M.Ux * M.Uz;
  dM[11] = q * M.Uy * M.Uy + iso;
  dM[12] = q * M.Uy * M.Uz;
  dM[13] = q * M.Uz * M.Uz + iso;
  if constexpr (K == 30) {
    const float q3 = 24.f * n * T * T, r3 = 4.f * n * T * T;
    const float iso3 = 4.f * (n * T * T * U0m1 + dn * T * T + nr * dT * (T + Tr));
#pragma unroll
    for (int k = 14; k < 20; ++k) {
      const int i = o3_index(k, 0), j = o3_index(k, 1);
      dM[k] = q3 * M.U0 * U[i] * U[j] + (i == j ? iso3 : 0.f);
    }
#pragma unroll
    for (int k = 20; k < 30; ++k) {
      const int i = o3_index(k, 0), j = o3_index(k, 1), l = o3_index(k, 2);
      dM[k] = q3 * U[i] * U[j] * U[l] + r3 * ((i == j ? U[l] : 0.f) + (i == l ? U[j] : 0.f) + (j == l ? U[i] : 0.f));
    }
  }
}

// The collision frame of FP32 storage from the 14 moment sums m = N0 Nx Ny Nz
// T00 T0x T0y T0z Txx Txy Txz Tyy Tyz Tzz of g = f - f_ref: the moments Mk of
// the K-member basis, as differences from the reference, and
// tau^-1 U (zero where the cell has no Landau frame, which leaves it
// unrelaxed).  Returns whether the frame exists.
// A cell without a physical Landau frame is left unrelaxed (Omega = 0); its
// frame is replaced by the reference state (rest, n_ref or 1, T_ref) so
// that the equilibrium and Omega stay finite (0 * NaN is not 0).
__device__ __forceinline__ void unphysical_to_reference3(const Scalars3& s, Macro3f& M) {
  M.n = (float)(s.n_ref > 0.0 ? s.n_ref : 1.0);
  M.T = s.f_T_ref;
  M.dn = M.dT = 0.f;
  M.U0 = 1.f;
  M.Ux = M.Uy = M.Uz = 0.f;
}

template <int K>
__device__ __forceinline__ bool frame3(const float (&m)[14], const Scalars3& s, float (&Mk)[K], float& kU0,
                                       float (&kU)[3]) {
  const float N[4] = {m[0], m[1], m[2], m[3]};
  const float Tm[4][4] = {{m[4], m[5], m[6], m[7]},
                          {m[5], m[8], m[9], m[10]},
                          {m[6], m[9], m[11], m[12]},
                          {m[7], m[10], m[12], m[13]}};
  Macro3f M = landau3f(N, Tm, s);
  if (!M.ok) unphysical_to_reference3(s, M);
  mj_delta3<K>(M, s.f_n_ref, s.f_T_ref, Mk);
  const float kt = M.ok ? s.f_inv_tau : 0.f;
  kU0 = kt * M.U0;
  kU[0] = kt * M.Ux;
  kU[1] = kt * M.Uy;
  kU[2] = kt * M.Uz;
  return M.ok;
}

// Walsh-Hadamard transform in place: v[c] <- sum_s (-1)^{popcount(c & s)} v[s]
template <typename S, int L>
__device__ __forceinline__ void fwht(S (&v)[L]) {
#pragma unroll
  for (int hb = 1; hb < L; hb <<= 1)
#pragma unroll
    for (int q = 0; q < L; ++q)
      if (!(q & hb)) {
        const S u = v[q], w = v[q | hb];
        v[q] = u + w;
        v[q | hb] = u - w;
      }
}

// the moment sums of a run of 8 from its transformed values F (F[c] = sum_s
// chi_c(s) f_s) and its first member's monomials c (Tables3::mono order)
template <typename S, typename C>
__device__ __forceinline__ void moments_run8(const S (&F)[8], const C* c, S (&m)[14]) {
  m[0] = fma((S)c[0], F[0], m[0]);
  m[1] = fma((S)c[1], F[1], m[1]);
  m[2] = fma((S)c[2], F[2], m[2]);
  m[3] = fma((S)c[3], F[4], m[3]);
  m[4] = fma((S)c[4], F[0], m[4]);
  m[5] = fma((S)c[5], F[1], m[5]);
  m[6] = fma((S)c[6], F[2], m[6]);
  m[7] = fma((S)c[7], F[4], m[7]);
  m[8] = fma((S)c[8], F[0], m[8]);
  m[9] = fma((S)c[9], F[3], m[9]);
  m[10] = fma((S)c[10], F[5], m[10]);
  m[11] = fma((S)c[11], F[0], m[11]);
  m[12] = fma((S)c[12], F[6], m[12]);
  m[13] = fma((S)c[13], F[0], m[13]);
}

// FP32 storage: the periodic images of a cell next to a face, copied from the
// values the thread has just stored for the cell itself, B populations at a
// time so that B loads are in flight (one at a time, each waits on the L2
// round trip of the one before, as the stores in between may alias them).
template <int QT, int B>
__device__ __forceinline__ void images_from_stored(const Scalars3& s, float* out, long long si, int x, int y, int z) {
  int ix[2], iy[2], iz[2];
  const int nx2 = images1(x, s.nx, s.h, ix), ny2 = images1(y, s.ny, s.h, iy), nz2 = images1(z, s.nz, s.h, iz);
  if (nx2 + ny2 + nz2 == 0) return;
  long long img[26];
  int nimg = 0;
  for (int cz = -1; cz < nz2; ++cz)
    for (int cy = -1; cy < ny2; ++cy)
      for (int cx = -1; cx < nx2; ++cx) {
        if (cx < 0 && cy < 0 && cz < 0) continue;
        img[nimg++] = sidx3(s, cx < 0 ? x : ix[cx], cy < 0 ? y : iy[cy], cz < 0 ? z : iz[cz]);
      }
  static_assert(QT % B == 0, "whole batches");
  const long long P = s.plane;
  for (int i0 = 0; i0 < QT; i0 += B) {
    float v[B];
#pragma unroll
    for (int j = 0; j < B; ++j) v[j] = out[(long long)(i0 + j) * P + si];
#pragma unroll
    for (int j = 0; j < B; ++j) {
      float* oi = out + (long long)(i0 + j) * P;
      for (int m = 0; m < nimg; ++m) oi[img[m]] = v[j];
    }
  }
}

// periodic images of a cell (every side at least h: at most 26)
__device__ __forceinline__ int cell_images(const Scalars3& s, int x, int y, int z, long long (&img)[26]) {
  int ix[2], iy[2], iz[2];
  const int nx2 = images1(x, s.nx, s.h, ix), ny2 = images1(y, s.ny, s.h, iy), nz2 = images1(z, s.nz, s.h, iz);
  int nimg = 0;
  for (int cz = -1; cz < nz2; ++cz)
    for (int cy = -1; cy < ny2; ++cy)
      for (int cx = -1; cx < nx2; ++cx) {
        if (cx < 0 && cy < 0 && cz < 0) continue;
        img[nimg++] = sidx3(s, cx < 0 ? x : ix[cx], cy < 0 ? y : iy[cy], cz < 0 ? z : iz[cz]);
      }
  return nimg;
}

}  // namespace
}  // namespace rlbm
