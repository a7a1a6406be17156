// rlbm_convert_f32_f64: the FP32 <-> FP64 conversions the FP32-storage
// kernels run on the integer pipe (fpconv.cuh), applied element-wise to
// device arrays, so that they can be compared with the hardware conversions.
// rlbm_fast_math_f64, _f32: the short quotients, square roots and conversions of the
// fixed-point steps (fx64.cuh) and of the (3+1)-d FP32 frame (d3_impl.cuh), likewise.
#include <cuda_runtime.h>

#include "../../include/rlbm.h"
#include "d3_impl.cuh"
#include "fpconv.cuh"
#include "fx64.cuh"

namespace {

__global__ void k_convert(const float* in_f, double* out_d, int nf, const double* in_d, float* out_f, int nd) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < nf) out_d[i] = rlbm::f2d(in_f[i]);
  if (i < nd) out_f[i] = rlbm::d2f(in_d[i]);
}

__global__ void k_fast_f64(const double* a, const double* b, double* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int top = 0;
  out[i] = rlbm::reciprocal(b[i]);
  out[n + i] = rlbm::quotient(a[i], b[i]);
  out[2 * n + i] = rlbm::reciprocal_sqrt(b[i]);
  out[3 * n + i] = (double)rlbm::cut_float(a[i]);
  out[4 * n + i] = (double)rlbm::d2f_finite(a[i], top);
  out[5 * n + i] = top >= rlbm::kNoFloat ? 1.0 : 0.0;
}

__global__ void k_fast_f32(const float* a, const float* b, double* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  out[i] = (double)rlbm::quotient32(a[i], b[i]);
  out[n + i] = rlbm::wide_double(a[i]);
  out[2 * n + i] = rlbm::f2d_finite(a[i]);
}

}  // namespace

extern "C" int rlbm_fast_math_f64(const double* a, const double* b, double* out, int n, void* stream) {
  if (n < 1 || n > (1 << 27) || !a || !b || !out) return RLBM_ERR_INVALID_ARG;
  k_fast_f64<<<(n + 255) / 256, 256, 0, (cudaStream_t)stream>>>(a, b, out, n);
  return cudaGetLastError() == cudaSuccess ? RLBM_OK : RLBM_ERR_CUDA;
}

extern "C" int rlbm_fast_math_f32(const float* a, const float* b, double* out, int n, void* stream) {
  if (n < 1 || n > (1 << 27) || !a || !b || !out) return RLBM_ERR_INVALID_ARG;
  k_fast_f32<<<(n + 255) / 256, 256, 0, (cudaStream_t)stream>>>(a, b, out, n);
  return cudaGetLastError() == cudaSuccess ? RLBM_OK : RLBM_ERR_CUDA;
}

extern "C" int rlbm_convert_f32_f64(const float* in_f, double* out_d, int nf, const double* in_d, float* out_f,
                                    int nd, void* stream) {
  if (nf < 0 || nd < 0 || (nf > 0 && (!in_f || !out_d)) || (nd > 0 && (!in_d || !out_f)))
    return RLBM_ERR_INVALID_ARG;
  const int n = nf > nd ? nf : nd;
  if (n == 0) return RLBM_OK;
  k_convert<<<(n + 255) / 256, 256, 0, (cudaStream_t)stream>>>(in_f, out_d, nf, in_d, out_f, nd);
  return cudaGetLastError() == cudaSuccess ? RLBM_OK : RLBM_ERR_CUDA;
}
