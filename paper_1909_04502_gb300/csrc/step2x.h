// Tables and launcher of the (2+1)-d FP64 step in fixed point (step2x.cu).
#pragma once
#include <cuda_runtime.h>

#include <vector>

#include "fx64.cuh"
#include "kernels.cuh"
#include "setup.h"

namespace rlbm {

// An orbit-ordered stencil (setup.cpp) as sign quartets (a, b), (-a, b),
// (a, -b), (-a, -b) -- two per eight-member orbit, one per diagonal orbit --
// then axis quartets (p, 0), (-p, 0), (0, p), (0, -p) and a rest population.
// Scales as in Tables3x: ep, the exponent of p0^2, for the moment sums; er, of
// the rest equilibrium at n = T = 1, and rho, of the row's largest
// H 2^(-er - hk), for the relaxation.
constexpr int kQuartets = 16, kAxes = 4;
struct Tables2x {
  int Q, nq, na, nr;                 // populations, sign quartets, axis quartets, rest populations (0 or 1)
  Cx Hq[kQuartets][kMaxK], Mq[kQuartets][9];   // rows H 2^(-er - hk - rho); p0 px py p0p0 p0px p0py pxpx pxpy pypy 2^(-ep - sk)
  Cx Ha[kAxes][2][kMaxK], Ma[kAxes][9];        // rows of (p, 0) and (0, p)
  Cx Hr[kMaxK], Mr[2];                         // rest: p0, p0p0
  int firstq[kQuartets], firsta[kAxes], firstr;   // first populations
  int epq[kQuartets], erq[kQuartets], rhoq[kQuartets], nq_x[kQuartets], nq_y[kQuartets];
  int epa[kAxes], era[kAxes], rhoa[kAxes], na_x[kAxes];
  int epr, err, rhor;
  int hk[kMaxK], sk[9];
  double vscale;                     // v_i = vscale n_i
  int off[kMaxQ];                    // pull source relative to the cell, plane included (tap (0, 0))
  double bw[kMaxQ][4];               // bilinear weights
  int pitch;                         // second row of taps
};

// Fills *t for a handle's tables; false where the fixed-point step does not
// apply (velocities that are not a multiple of the stencil vectors, a rest
// equilibrium that is not positive).
bool fill_tables2x(const Quadrature& q, const std::vector<double>& H, int K, const Scalars& s, const Tables<double>& td,
                   Tables2x* t);
cudaError_t launch_step2x(const Tables2x& tb, const StepArgs<double>& a, int mode, cudaStream_t st);
cudaError_t launch_fields2x(const Tables2x& tb, const MomentArgs<double>& a, int mode, cudaStream_t st);

}  // namespace rlbm
