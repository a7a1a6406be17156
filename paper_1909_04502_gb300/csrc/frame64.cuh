// The Landau frame in FP64 throughout, for the cells where the fixed-point
// steps' FP32-started refinement (step2x.cu, step3x.cu) does not settle: fast
// flows (gamma above 7 or so: the root is what remains of T^00, gamma^2 times as
// large, and S + l has condition gamma^2), and tensors without a frame.
//
// With T^ab = (E, t; t, S) the mixed tensor A = T eta has det(A - l I) =
// (l - E) D(l) + t.adj(S + l) t, D = det(S + l).  Its root by Newton from the
// ideal-fluid root for P = eps / 3, u = U^i / U^0 = adj(S + l) t / D, and then both by
// iterative refinement of  E - t.u - l = 0,  (S + l) u = t  with FP64 residuals:
// errors of the size that the tensor's own rounding makes, gamma^4 2^-53 in l.  Inline
// behind an unlikely branch: as a call it cost the (3+1)-d order-2 step of usual flows
// 2 % (101 x 75 x 66: 382 against 375.5 us).
#pragma once
#include <cuda_runtime.h>

#include <cmath>

namespace rlbm {

struct Frame64 {
  double l, u[3];
  bool ok;               // l > 0, u timelike and the refinement settled
};

// E = T^00, t = T^0i, S = Txx Txy Txz Tyy Tyz Tzz, of order one or below.
__host__ __device__ __forceinline__ Frame64 frame64(double E, const double (&t)[3], const double (&S)[6]) {
  const double x = t[0], y = t[1], z = t[2], xx = x * x, yy = y * y, zz = z * z;
  const double xy = 2.0 * x * y, xz = 2.0 * x * z, yz = 2.0 * y * z;
  double A[6];           // adj(S + l)
  auto adjugate = [&](double l) {
    const double a = S[0] + l, b = S[3] + l, c = S[5] + l;
    A[0] = fma(b, c, -S[4] * S[4]);
    A[1] = fma(S[2], S[4], -S[1] * c);
    A[2] = fma(S[1], S[4], -S[2] * b);
    A[3] = fma(a, c, -S[2] * S[2]);
    A[4] = fma(S[1], S[2], -a * S[4]);
    A[5] = fma(a, b, -S[1] * S[1]);
    return fma(a, A[0], fma(S[1], A[1], S[2] * A[2]));
  };
  // D = l^3 + a1 l^2 + a2 l + a3 and t.adj t = b0 l^2 + b1 l + b2
  const double a3 = adjugate(0.0), a1 = S[0] + S[3] + S[5], a2 = A[0] + A[3] + A[5];
  const double b0 = xx + yy + zz;
  const double b1 = a1 * b0 - (xx * S[0] + yy * S[3] + zz * S[5] + xy * S[1] + xz * S[2] + yz * S[4]);
  const double b2 = xx * A[0] + yy * A[3] + zz * A[5] + xy * A[1] + xz * A[2] + yz * A[4];
  const double disc = 4.0 * (4.0 * E * E - 3.0 * b0);      // 9 ((2/3 E)^2 + 4/3 (E^2 - b0))
  double l = 0.5 * (sqrt(disc > 0.0 ? disc : 0.0) - 2.0 * E);
#pragma unroll 1
  for (int it = 0; it < 10; ++it) {
    const double D = fma(fma(l + a1, l, a2), l, a3), dD = fma(fma(3.0, l, 2.0 * a1), l, a2);
    const double dp = fma(l - E, dD, D + fma(2.0 * b0, l, b1));
    if (!(dp != 0.0)) break;
    const double d = fma(l - E, D, fma(fma(b0, l, b1), l, b2)) / dp;
    l -= d;
    if (fabs(d) <= 1e-15 * fabs(l)) break;
  }
  Frame64 f;
  double w = 0.0;
  bool settled = false;
  double id = 0.0, r[3];
  auto residual = [&]() {               // r = t - (S + l) u
    r[0] = fma(-S[2], f.u[2], fma(-S[1], f.u[1], fma(-S[0], f.u[0], fma(-l, f.u[0], x))));
    r[1] = fma(-S[4], f.u[2], fma(-S[3], f.u[1], fma(-S[1], f.u[0], fma(-l, f.u[1], y))));
    r[2] = fma(-S[5], f.u[2], fma(-S[4], f.u[1], fma(-S[2], f.u[0], fma(-l, f.u[2], z))));
  };
  auto inverse = [&](const double (&v)[3], double (&out)[3]) {
    out[0] = (A[0] * v[0] + A[1] * v[1] + A[2] * v[2]) * id;
    out[1] = (A[1] * v[0] + A[3] * v[1] + A[4] * v[2]) * id;
    out[2] = (A[2] * v[0] + A[4] * v[1] + A[5] * v[2]) * id;
  };
  double c[3];
  auto solve = [&]() {                  // u at l, w = 1 - u.u
    id = 1.0 / adjugate(l);
    inverse(t, f.u);
    residual();
    inverse(r, c);
    for (int i = 0; i < 3; ++i) f.u[i] += c[i];
    w = fma(-f.u[2], f.u[2], fma(-f.u[1], f.u[1], fma(-f.u[0], f.u[0], 1.0)));
  };
  auto energy = [&]() { return fma(-z, f.u[2], fma(-y, f.u[1], fma(-x, f.u[0], E - l))); };
  auto refine = [&]() {                 // l and u together; a step that leaves the neighbourhood is no frame's
    solve();
    settled = false;
#pragma unroll 1
    for (int it = 0; it < 8; ++it) {
      residual();
      const double d = (energy() - f.u[0] * r[0] - f.u[1] * r[1] - f.u[2] * r[2]) / w;
      for (int i = 0; i < 3; ++i) r[i] -= f.u[i] * d;
      inverse(r, c);
      if (!(w > 0.0 && l + d > 0.0 && fabs(d) <= l && fabs(c[0]) + fabs(c[1]) + fabs(c[2]) <= w)) {
        settled = false;
        return;
      }
      l += d;
      for (int i = 0; i < 3; ++i) f.u[i] += c[i];
      id = 1.0 / adjugate(l);
      w = fma(-f.u[2], f.u[2], fma(-f.u[1], f.u[1], fma(-f.u[0], f.u[0], 1.0)));
      const bool before = settled;
      settled = fabs(d) <= 1e-3 * l;
      if (before && settled && it > 1) return;
    }
  };
  refine();
  if (!settled) {
    // from the right: E - t.(S + l)^-1 t - l is concave and falls for l above the root while S + l is
    // positive definite, so that Newton from l = E, which is never below the root, comes down to it
    l = E;
#pragma unroll 1
    for (int it = 0; it < 40; ++it) {
      solve();
      const double d = energy() / w;
      if (!(id > 0.0 && w > 0.0 && l > 0.0)) break;
      l += d;
      if (!(fabs(d) > 1e-6 * l)) break;
    }
    refine();
  }
  f.l = l;
  f.ok = settled && w > 0.0 && l > 0.0;
  return f;
}

}  // namespace rlbm
