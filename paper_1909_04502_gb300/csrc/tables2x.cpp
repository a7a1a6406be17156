// Host side of the fixed-point tables of the (2+1)-d FP64 step (step2x.h).
#include "step2x.h"

#include <algorithm>
#include <cmath>
#include <cstring>

namespace rlbm {

bool fill_tables2x(const Quadrature& q, const std::vector<double>& H, int K, const Scalars& s, const Tables<double>& td,
                   Tables2x* t) {
  std::memset(t, 0, sizeof(*t));
  // orbit composition in population order (the caller has checked the orbit symmetry of H)
  struct Set {
    int first, kind;    // kind 0: sign quartet, 1: axis quartet, 2: rest
    int er, ep, rho;
  };
  std::vector<Set> sets;
  for (int i = 0; i < q.Q;) {
    const bool x0 = q.px[i] == 0.0, y0 = q.py[i] == 0.0;
    const Set set = {i, x0 && y0 ? 2 : (x0 || y0 ? 1 : 0), 0, 0, 0};
    sets.push_back(set);
    i += set.kind == 2 ? 1 : 4;
    if (i > q.Q) return false;
  }
  // v_i = vscale n_i with one vscale
  double big = 0.0;
  for (int i = 0; i < q.Q; ++i)
    if (std::abs(q.nx[i]) + std::abs(q.ny[i]) > 0) {
      const int a = std::abs(q.nx[i]) >= std::abs(q.ny[i]) ? q.nx[i] : q.ny[i];
      const double p = std::abs(q.nx[i]) >= std::abs(q.ny[i]) ? q.px[i] : q.py[i];
      if (big == 0.0) big = p / q.p0[i] / a;
    }
  if (!(big > 0.0)) return false;
  t->vscale = big;
  for (int i = 0; i < q.Q; ++i)
    if (std::fabs(q.px[i] / q.p0[i] - big * q.nx[i]) > 1e-15 || std::fabs(q.py[i] / q.p0[i] - big * q.ny[i]) > 1e-15 ||
        std::abs(q.nx[i]) > 64 || std::abs(q.ny[i]) > 64)
      return false;
  std::vector<double> Mrest(K);
  const double e0[3] = {1.0, 0.0, 0.0};
  mj_moments(s.order, s.m, 1.0, e0, 1.0, Mrest.data());
  auto row = [&](int i, int k) { return H[(size_t)i * K + k]; };
  for (Set& c : sets) {
    double f = 0.0;
    for (int k = 0; k < K; ++k) f += row(c.first, k) * Mrest[k];
    if (!(f > 1e-30) || !(q.p0[c.first] > 0.0)) return false;
    c.er = std::ilogb(f);
    c.ep = std::ilogb(q.p0[c.first] * q.p0[c.first]);
  }
  // (an orbit's rows are permutations of its first: the columns of both
  // orientations, whose exponents are made equal)
  for (int k = 0; k < K; ++k) {
    double m = 0.0;
    for (const Set& c : sets)
      for (int r : {0, 2})
        if (c.kind != 2 || r == 0) m = std::fmax(m, std::fabs(std::ldexp(row(c.first + r, k), -c.er)));
    if (!(m > 0.0)) return false;
    std::frexp(m, &t->hk[k]);
  }
  for (int k = 0; k < K; ++k) t->hk[k] = std::max(t->hk[k], t->hk[mono_swap(k)]);
  for (Set& c : sets) {
    double m = 0.0, sum[4] = {0.0};
    for (int k = 0; k < K; ++k) {
      const double v = std::fabs(std::ldexp(row(c.first, k), -c.er - t->hk[k]));
      m = std::fmax(m, v);
      sum[mono_ax(k) + 2 * mono_ay(k)] += v;
    }
    int e4;
    std::frexp(std::fmax(std::fmax(sum[0], sum[1]), std::fmax(sum[2], sum[3])), &e4);
    std::frexp(m, &c.rho);
    c.rho = std::max(c.rho, e4 - 2);       // row at most one, class sums at most four
  }
  auto mono = [&](int i, int j) {
    const double p0 = q.p0[i], px = q.px[i], py = q.py[i];
    const double c[9] = {p0, px, py, p0 * p0, p0 * px, p0 * py, px * px, px * py, py * py};
    return c[j];
  };
  // every member's monomials are those of its set's first up to sign and exchange
  for (int j = 0; j < 9; ++j) {
    double sum = 0.0;
    for (const Set& c : sets) {
      const double v = mono(c.first, j);
      if (!(v >= 0.0)) return false;
      sum += std::ldexp(std::fmax(v, c.kind == 1 ? std::fmax(mono(c.first + 2, j), 0.0) : 0.0), -c.ep);
    }
    if (!(sum > 0.0)) return false;
    std::frexp(sum, &t->sk[j]);
  }
  static const int kSwap9[9] = {0, 2, 1, 3, 5, 4, 8, 7, 6};
  for (int j = 0; j < 9; ++j) t->sk[j] = std::max(t->sk[j], t->sk[kSwap9[j]]);
  auto h = [&](int i, int k, const Set& c) { return split_constant(std::ldexp(row(i, k), -c.er - t->hk[k] - c.rho), kCoefH); };
  auto m = [&](int i, int j, const Set& c) { return split_constant(std::ldexp(mono(i, j), -c.ep - t->sk[j]), kCoefM); };
  for (const Set& c : sets) {
    if (c.kind == 0) {
      if (t->nq == kQuartets) return false;
      const int r = t->nq++;
      for (int k = 0; k < K; ++k) t->Hq[r][k] = h(c.first, k, c);
      for (int j = 0; j < 9; ++j) t->Mq[r][j] = m(c.first, j, c);
      t->firstq[r] = c.first, t->nq_x[r] = q.nx[c.first], t->nq_y[r] = q.ny[c.first];
      t->epq[r] = c.ep, t->erq[r] = c.er, t->rhoq[r] = c.rho;
    } else if (c.kind == 1) {
      if (t->na == kAxes) return false;
      const int r = t->na++;
      for (int k = 0; k < K; ++k) t->Ha[r][0][k] = h(c.first, k, c), t->Ha[r][1][k] = h(c.first + 2, k, c);
      for (int j = 0; j < 9; ++j) t->Ma[r][j] = m(c.first, j, c);
      t->firsta[r] = c.first, t->na_x[r] = q.nx[c.first];
      t->epa[r] = c.ep, t->era[r] = c.er, t->rhoa[r] = c.rho;
    } else {
      if (t->nr) return false;
      t->nr = 1;
      for (int k = 0; k < K; ++k) t->Hr[k] = h(c.first, k, c);
      t->Mr[0] = m(c.first, 0, c), t->Mr[1] = m(c.first, 3, c);
      t->firstr = c.first, t->epr = c.ep, t->err = c.er, t->rhor = c.rho;
    }
  }
  t->Q = q.Q;
  for (int i = 0; i < q.Q; ++i) {
    t->off[i] = td.offp[i];
    for (int j = 0; j < 4; ++j) t->bw[i][j] = td.bw[i][j];
  }
  t->pitch = s.pitch;
  return true;
}

}  // namespace rlbm
