// Tables of the fixed-point kernels of the (3+1)-d steps (step3x.cu).
#pragma once
#include <cuda_runtime.h>

#include "d3.h"
#include "fx64.cuh"

namespace rlbm {

constexpr int kRhoMin = -4;  // smallest row exponent of the equilibrium constants
constexpr int kMom3 = 13;   // moment sums N0 Nx Ny Nz T0x T0y T0z Txx Txy Txz Tyy Tyz Tzz

// Run tables of the order-2 or order-3 table: 9 or 33 runs of 8 members, the
// runs of one direction pattern (all shells) together, and a tail of 3 axis
// pairs or 6 runs of 4.
template <int ORDER>
struct Tables3x {
  static constexpr int K = ORDER == 2 ? 14 : 30, Q = ORDER == 2 ? 78 : 288;
  static constexpr int N8 = ORDER == 2 ? 9 : 33, NT = ORDER == 2 ? 3 : 6, LT = ORDER == 2 ? 2 : 4;
  static constexpr int ND = ORDER == 2 ? 3 : 9;      // direction patterns of the runs of 8
  Cx H8[N8][K], M8[N8][kMom3];   // first rows H 2^(-er - hk - rho), moment constants mono 2^(-ep - sk)
  Cx HT[NT][K], MT[NT][kMom3];
  long long ref8[N8], refT[NT];  // f_ref 2^ep in units of 2^(ref_E - kBitsM) (FP32 storage)
  // per run: ep, the exponent of p0^2, scales its populations in the moment sums; er,
  // the exponent of its rest equilibrium, and rho, of its row's largest H 2^(-er - hk), in the relaxation
  int ep8[N8], er8[N8], rho8[N8], first8[N8], off8[N8][8];
  int epT[NT], erT[NT], rhoT[NT], firstT[NT], offT[NT][LT], nT[NT][3];
  int dir_first[ND + 1], dir_n[ND][3];   // runs of 8 by pattern: first run, stencil vector
  int hk[K], sk[kMom3];          // column exponents of H 2^-er and of the moment constants
  int ref_E;                     // biased: every |f_ref| 2^ep < 2^(ref_E - 1023 - 1)
  double inv_len;                // 1 / |n|
};

// Fills *t from the quadrature and the pull shifts (without the plane offset);
// false where the table is not in the sign-orbit layout.
template <int ORDER>
bool fill_tables3x(const Quadrature3& q, const int* shift, const double* fref, Tables3x<ORDER>* t);

// The FP64 step (order 2 or 3).
template <int ORDER>
cudaError_t launch_step3x(const Tables3x<ORDER>& tb, const Step3Args<double>& a, cudaStream_t st);
// Fields of both storage types.
template <int ORDER, typename S>
cudaError_t launch_fields3x(const Tables3x<ORDER>& tb, const Fields3Args<S>& a, cudaStream_t st);

}  // namespace rlbm
