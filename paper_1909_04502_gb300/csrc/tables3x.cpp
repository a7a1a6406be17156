// Host side of the fixed-point tables of the (3+1)-d steps (step3x.h).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "step3x.h"

namespace rlbm {

template <int ORDER>
bool fill_tables3x(const Quadrature3& q, const int* shift, const double* fref, Tables3x<ORDER>* t) {
  using T = Tables3x<ORDER>;
  static const int kTail[6] = {ORDER == 2 ? 1 : 3, ORDER == 2 ? 2 : 5, ORDER == 2 ? 4 : 3, 5, 6, 6};
  std::memset(t, 0, sizeof(T));
  if (!q.sym || q.Q != T::Q || q.K != T::K || (int)q.orbit_mask.size() != T::N8 + T::NT) return false;
  struct Run {
    int first, size, mask, er, ep, rho;
    const int* n;
  };
  std::vector<Run> eight, tail;
  int i0 = 0;
  for (int mask : q.orbit_mask) {
    const int size = 1 << ((mask & 1) + (mask >> 1 & 1) + (mask >> 2 & 1));
    if (i0 + size > q.Q) return false;
    // the equilibrium at rest, n = T = 1: <1> = 1/2, <p0> = 1, <p^i p^i> = 1, <p0 p^i p^i> = 4
    const double* H = &q.H[(size_t)i0 * T::K];
    double f = 0.5 * H[0] + H[1] + H[8] + H[11] + H[13];
    if (T::K == 30) f += 4.0 * (H[14] + H[17] + H[19]);
    const double p0 = q.p[4 * (size_t)i0];
    if (!(f > 0.0) || !(p0 > 0.0)) return false;
    const Run run = {i0, size, mask, std::ilogb(f), std::ilogb(p0 * p0), 0, &q.n[3 * (size_t)i0]};
    if (mask == 7) eight.push_back(run);
    else if ((int)tail.size() < T::NT && size == T::LT && mask == kTail[tail.size()]) tail.push_back(run);
    else return false;
    i0 += size;
  }
  if ((int)eight.size() != T::N8 || (int)tail.size() != T::NT || i0 != q.Q) return false;
  // the runs of one pattern together
  std::stable_sort(eight.begin(), eight.end(), [](const Run& a, const Run& b) {
    return std::lexicographical_compare(a.n, a.n + 3, b.n, b.n + 3);
  });
  int nd = 0;
  for (int r = 0; r < T::N8; ++r)
    if (r == 0 || !std::equal(eight[r].n, eight[r].n + 3, eight[r - 1].n)) {
      if (nd == T::ND) return false;
      for (int k = 0; k < 3; ++k) t->dir_n[nd][k] = eight[r].n[k];
      t->dir_first[nd++] = r;
    }
  if (nd != T::ND) return false;
  t->dir_first[nd] = T::N8;
  std::vector<Run*> runs;
  for (Run& r : eight) runs.push_back(&r);
  for (Run& r : tail) runs.push_back(&r);
  auto mono = [&](int i, int k) {
    static const int kIdx[kMom3][2] = {{0, -1}, {1, -1}, {2, -1}, {3, -1}, {0, 1}, {0, 2}, {0, 3},
                                       {1, 1},  {1, 2},  {1, 3},  {2, 2},  {2, 3}, {3, 3}};
    const double* p = &q.p[4 * (size_t)i];
    return kIdx[k][1] < 0 ? p[kIdx[k][0]] : p[kIdx[k][0]] * p[kIdx[k][1]];
  };
  // column exponents: |H 2^-er| <= 2^hk; then per row |H 2^(-er - hk)| <= 2^rho (rho at least kRhoMin)
  for (int k = 0; k < T::K; ++k) {
    double big = 0.0;
    for (const Run* r : runs) big = std::fmax(big, std::fabs(std::ldexp(q.H[(size_t)r->first * T::K + k], -r->er)));
    if (!(big > 0.0)) return false;
    std::frexp(big, &t->hk[k]);
  }
  static const int kPar[30] = {0, 0, 1, 2, 4, 1, 2, 4, 0, 3, 5, 0, 6, 0,      // parity classes (step3x.cu)
                               0, 3, 5, 0, 6, 0, 1, 2, 4, 1, 7, 1, 2, 4, 2, 4};
  for (Run* r : runs) {
    double big = 0.0, sum[8] = {0.0};
    for (int k = 0; k < T::K; ++k) {
      const double c = std::fabs(std::ldexp(q.H[(size_t)r->first * T::K + k], -r->er - t->hk[k]));
      big = std::fmax(big, c);
      sum[kPar[k]] += c;
    }
    std::frexp(big, &r->rho);
    r->rho = std::max(r->rho, kRhoMin);
    for (double v : sum)
      if (!(std::ldexp(v, -r->rho) <= 4.0)) return false;
  }
  // moment constants: the sum over the runs of mono 2^-ep below 2^sk (more than one
  // run: each below it)
  for (int k = 0; k < kMom3; ++k) {
    double sum = 0.0;
    for (const Run* r : runs) {
      const double c = std::ldexp(mono(r->first, k), -r->ep);
      if (!(c >= 0.0)) return false;
      sum += c;
    }
    std::frexp(sum, &t->sk[k]);
  }
  int e = -1000;
  for (const Run* r : runs)
    if (fref[r->first] != 0.0) e = std::max(e, std::ilogb(fref[r->first]) + r->ep + 1);
  t->ref_E = 1023 + e + 1;
  auto fill = [&](const Run& r, Cx* H, Cx* M, int* off, int* ep, int* er, int* rho, int* first, long long* ref) {
    for (int k = 0; k < T::K; ++k)
      H[k] = split_constant(std::ldexp(q.H[(size_t)r.first * T::K + k], -r.er - t->hk[k] - r.rho), kCoefH);
    for (int k = 0; k < kMom3; ++k) M[k] = split_constant(std::ldexp(mono(r.first, k), -r.ep - t->sk[k]), kCoefM);
    for (int m = 0; m < r.size; ++m) off[m] = shift[r.first + m];
    *ep = r.ep;
    *er = r.er;
    *rho = r.rho;
    *first = r.first;
    *ref = fref[r.first] == 0.0 ? 0 : std::llround(std::ldexp(fref[r.first], r.ep + kBitsM - (t->ref_E - 1023)));
  };
  for (int r = 0; r < T::N8; ++r)
    fill(eight[r], t->H8[r], t->M8[r], t->off8[r], &t->ep8[r], &t->er8[r], &t->rho8[r], &t->first8[r], &t->ref8[r]);
  for (int r = 0; r < T::NT; ++r) {
    fill(tail[r], t->HT[r], t->MT[r], t->offT[r], &t->epT[r], &t->erT[r], &t->rhoT[r], &t->firstT[r], &t->refT[r]);
    for (int k = 0; k < 3; ++k) t->nT[r][k] = tail[r].n[k];
  }
  const int* n0 = &q.n[0];
  t->inv_len = 1.0 / std::sqrt((double)(n0[0] * n0[0] + n0[1] * n0[1] + n0[2] * n0[2]));
  return true;
}

template bool fill_tables3x<2>(const Quadrature3&, const int*, const double*, Tables3x<2>*);
template bool fill_tables3x<3>(const Quadrature3&, const int*, const double*, Tables3x<3>*);

}  // namespace rlbm
