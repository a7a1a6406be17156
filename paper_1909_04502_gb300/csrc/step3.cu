// (3+1)-dimensional massless RLBM step, order 2 (Sec. 5-6 with d = 3):
// on-lattice pull, the moments N^a and T^ab, the Landau frame of the 4 x 4
// mixed tensor (Sec. 4), n = U.N, T = eps / (3n) (Eq. ultra-relativistic-eos,
// d = 3), f^eq = H M(n, U, T) (Eq. mj-discrete-feq), Anderson-Witting
// relaxation, store with the periodic halo images.  Here: the FP32-storage
// step k_step3fs (g = f - f_ref, the table in sign-orbit form) and the
// initialisation; the FP64 step and the fields are in step3x.cu.
//
// Layout: one plane per population, cell (x, y, z) at
//   (z + h) * slab + (y + h) * pitch + (x + px),  slab = (ny + 2h) * pitch,
// with a halo of h = 3 cells (the stencil length) on every side holding the
// periodic images, so that every pull is the cell index plus a constant.
#include <cuda_runtime.h>

#include "d3_impl.cuh"

namespace rlbm {

namespace {

// spatial exponents (x, y, z) of the order-2 basis members 1 | p0 px py pz |
// p0px p0py p0pz pxpx pxpy pxpz pypy pypz pzpz
__device__ constexpr int kBasis3Exp[14][3] = {{0, 0, 0}, {0, 0, 0}, {1, 0, 0}, {0, 1, 0}, {0, 0, 1},
                                              {1, 0, 0}, {0, 1, 0}, {0, 0, 1}, {2, 0, 0}, {1, 1, 0},
                                              {1, 0, 1}, {0, 2, 0}, {0, 1, 1}, {0, 0, 2}};

__device__ __forceinline__ void copy_async4(float* to, const void* from) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(to)), "l"(from) : "memory");
}
// all but the newest n groups have arrived
__device__ __forceinline__ void wait_copies(int n) {
  switch (n) {
#define WAIT(k) case k: asm volatile("cp.async.wait_group " #k ";" ::: "memory"); break;
    WAIT(0) WAIT(1) WAIT(2) WAIT(3) WAIT(4) WAIT(5) WAIT(6) WAIT(7) WAIT(8) WAIT(9)
#undef WAIT
  }
}

// The FP32-storage step in sign-orbit form.
// Populations come in runs whose members share p0 and |p| componentwise:
// 9 runs of 8 (member s negates the components whose bit is set in s) and
// the pairs (+-3, 0, 0), (0, +-3, 0), (0, 0, +-3).  Per run of 8, a
// Walsh-Hadamard transform of the pulled values gives the sums
// F_c = sum_s chi_c(s) f_s over the sign characters c; each moment of rank
// <= 2 needs one of them times the first member's monomial (e.g. T^xy += a b
// F_xy).  The equilibrium rows of a run are the first row with the sign
// chi_k(s) of each basis member k (checked exactly on the host), so f^eq_s =
// sum over the seven characters of chi(s) C_chi, with C_chi the first row's
// partial sums over the members of that character; the relaxation rates
// follow from v_s . U = sx vx Ux + sy vy Uy + sz vz Uz.  About 110 operations
// per run of 8 against about 270 for eight rows.
// g = f - f_ref is stored and collided in FP32; the moments are FP32 sums of g
// (the reference moments enter in FP64); the Landau root is found in FP32
// (Newton on det(A - l I)) and corrected by one Newton step whose residual,
// the eigenvector's nu^2 = v.v, w = v.N and the numerator of dn = n - n_ref
// are evaluated in FP64 (landau3f, through frame3); the equilibrium
// differences dM = M(n, U, T) - M_ref are written so that each is accurate
// relative to itself, and the equilibrium, the relaxation and the store are
// FP32.  Every run is unrolled, so each table entry (pull shift, monomial, H
// row, velocity) is an immediate constant operand rather than a load by
// run-time index (with the runs in a loop this form was slower than the
// row-by-row kernel it replaced).
// The pulled populations go to shared memory by asynchronous copies, all 78 in
// flight at once, and both passes read them there (40 KB per block of 128
// threads, five blocks per SM); the relaxed values stay there for the periodic
// images of the cells next to a face.  At 192^3: 1.39 ms per step (0.47 of the
// copy bandwidth), at 96^3 217 us, at 33^3 25 us, against 1.50 ms, 262 us and
// 44 us with the populations pulled again in the second pass by eight blocks per SM,
// the images copied from the stored values and the former frame3.  What bounds
// it: about 2870 instructions per cell at 5 warps per scheduler, whose phases
// (copies, FP64 frame, stores) overlap in part; without the images 1.28 ms.
// Half of the populations kept and eight blocks per SM: 1.48 ms.
__global__ void __launch_bounds__(128, 8) k_step3fs(const __grid_constant__ Tables3 tb,
                                                    const __grid_constant__ Step3Args<float> a) {
  const Scalars3& s = a.s;
  const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 4 + threadIdx.y, z = blockIdx.z;
  if (x >= s.nx || y >= s.ny || z >= s.nz) return;
  // (addresses: a plane's uniform one plus the cell's 32-bit offset)
  const unsigned cell = (unsigned)sidx3(s, x, y, z) * 4u;
  // the pulled populations, a column per thread: a group of copies per run
  __shared__ float columns[78 * 128];
  float* F = columns + threadIdx.y * 32 + threadIdx.x;
#pragma unroll
  for (int i = 0; i < 78; ++i) {
    copy_async4(F + i * 128, (const char*)(a.fin + tb.off[i]) + cell);
    if (i % 8 == 7 || i == 77) asm volatile("cp.async.commit_group;" ::: "memory");
  }
  // pass 1: m = N0 Nx Ny Nz T00 T0x T0y T0z Txx Txy Txz Tyy Tyz Tzz of g
  float m[14];
#pragma unroll
  for (int k = 0; k < 14; ++k) m[k] = 0.f;
#pragma unroll
  for (int r = 0; r < 9; ++r) {
    float f[8];
    wait_copies(9 - r);
#pragma unroll
    for (int q = 0; q < 8; ++q) f[q] = F[(8 * r + q) * 128];
    fwht(f);
    moments_run8(f, tb.monof[r], m);
  }
  wait_copies(0);
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) {
    const float fp = F[(72 + 2 * ax) * 128], fm = F[(73 + 2 * ax) * 128];
    const float Sm = fp + fm, D = fp - fm;
    const float* c = tb.monof[9 + ax];
    const int taa = ax == 0 ? 8 : (ax == 1 ? 11 : 13);
    m[0] = fmaf(c[0], Sm, m[0]);
    m[4] = fmaf(c[4], Sm, m[4]);
    m[1 + ax] = fmaf(c[1 + ax], D, m[1 + ax]);
    m[5 + ax] = fmaf(c[5 + ax], D, m[5 + ax]);
    m[taa] = fmaf(c[taa], Sm, m[taa]);
  }
  float Mm[14], kU0, kU[3];
  if (!frame3(m, s, Mm, kU0, kU)) atomicAdd(a.status, 1ULL);
  // pass 2: equilibrium differences, relaxation, interior store (order 2
  // keeps Q * plane below 2^31)
  int tx, ty;                          // (read again: no registers held for them meanwhile)
  asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tx));
  asm volatile("mov.u32 %0, %%tid.y;" : "=r"(ty));
  const unsigned to = (unsigned)sidx3(s, blockIdx.x * 32 + tx, blockIdx.y * 4 + ty, blockIdx.z) * 4u;
  auto plane = [&](int i) { return (char*)(a.fout + (long long)i * s.plane); };
  F = columns + ty * 32 + tx;
#pragma unroll
  for (int r = 0; r < 9; ++r) {
    const float* H0 = tb.Hf[8 * r];
    float C[8];
    C[0] = fmaf(H0[0], Mm[0], fmaf(H0[1], Mm[1], fmaf(H0[8], Mm[8], fmaf(H0[11], Mm[11], H0[13] * Mm[13]))));
    C[1] = fmaf(H0[2], Mm[2], H0[5] * Mm[5]);
    C[2] = fmaf(H0[3], Mm[3], H0[6] * Mm[6]);
    C[4] = fmaf(H0[4], Mm[4], H0[7] * Mm[7]);
    C[3] = H0[9] * Mm[9];
    C[5] = H0[10] * Mm[10];
    C[6] = H0[12] * Mm[12];
    C[7] = 0.f;
    fwht(C);
    const float* vb = tb.vf[8 * r];
    const float X = vb[0] * kU[0], Y = vb[1] * kU[1], Z = vb[2] * kU[2];
    const float r0 = kU0 - X, r1 = kU0 + X;
    const float R[4] = {r0 - Y, r1 - Y, r0 + Y, r1 + Y};
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int i = 8 * r + q;
      const float om = (q & 4) ? R[q & 3] + Z : R[q & 3] - Z;
      const float g = F[i * 128];
      *(float*)(plane(i) + to) = F[i * 128] = fmaf(om, C[q] - g, g);
    }
  }
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) {
    const int i0 = 72 + 2 * ax;
    const float* H0 = tb.Hf[i0];
    float Ce = 0.f, Co = 0.f;
#pragma unroll
    for (int k = 0; k < 14; ++k) {
      if (kBasis3Exp[k][ax] & 1) Co = fmaf(H0[k], Mm[k], Co);
      else Ce = fmaf(H0[k], Mm[k], Ce);
    }
    const float va = tb.vf[i0][ax] * kU[ax];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int i = i0 + q;
      const float feq = q ? Ce - Co : Ce + Co;
      const float om = q ? kU0 + va : kU0 - va;
      const float g = F[i * 128];
      *(float*)(plane(i) + to) = F[i * 128] = fmaf(om, feq - g, g);
    }
  }
  long long img[26];
  const int images = cell_images(s, blockIdx.x * 32 + tx, blockIdx.y * 4 + ty, blockIdx.z, img);
  for (int k = 0; k < images; ++k) {
    const unsigned at = (unsigned)img[k] * 4u;
#pragma unroll 6
    for (int i = 0; i < 78; ++i) *(float*)(plane(i) + at) = F[i * 128];
  }
}

// f*(0) = f^eq(n, U, T) of device fields (row-major [z][y][x]), stored as f
// (FP64) or f - f_ref (FP32), written to the interior and the halo images.
template <typename S>
__global__ void __launch_bounds__(128) k_init3(const __grid_constant__ Tables3 tb,
                                               const __grid_constant__ Init3Args<S> a) {
  const Scalars3& s = a.s;
  const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 4 + threadIdx.y, z = blockIdx.z;
  if (x >= s.nx || y >= s.ny || z >= s.nz) return;
  const long long c = ((long long)z * s.ny + y) * s.nx + x;
  const double ux = a.ux[c], uy = a.uy[c], uz = a.uz[c];
  const double g = 1.0 / sqrt(1.0 - ux * ux - uy * uy - uz * uz);
  const double U[4] = {g, g * ux, g * uy, g * uz};
  double Mm[14];
  mj_moments3(a.n[c], a.T[c], U, Mm);
  int ix[2], iy[2], iz[2];
  const int nx2 = images1(x, s.nx, s.h, ix), ny2 = images1(y, s.ny, s.h, iy), nz2 = images1(z, s.nz, s.h, iz);
  for (int i = 0; i < s.Q; ++i) {
    double feq = 0.0;
    for (int k = 0; k < 14; ++k) feq = fma(tb.H[i][k], Mm[k], feq);
    const S val = (S)(sizeof(S) == 4 ? feq - tb.fref[i] : feq);
    const long long pl = (long long)i * s.plane;
    for (int cz = -1; cz < nz2; ++cz)
      for (int cy = -1; cy < ny2; ++cy)
        for (int cx = -1; cx < nx2; ++cx)
          a.f[pl + sidx3(s, cx < 0 ? x : ix[cx], cy < 0 ? y : iy[cy], cz < 0 ? z : iz[cz])] = val;
  }
}

dim3 grid3(const Scalars3& s) { return dim3((s.nx + 31) / 32, (s.ny + 3) / 4, s.nz); }

}  // namespace

cudaError_t launch_step3f_sym(const Tables3& tb, const Step3Args<float>& a, cudaStream_t st) {
  if (a.s.Q != 78) return cudaErrorInvalidValue;
  k_step3fs<<<grid3(a.s), dim3(32, 4), 0, st>>>(tb, a);
  return cudaGetLastError();
}

template <typename S>
cudaError_t launch_init3(const Tables3& tb, const Init3Args<S>& a, cudaStream_t st) {
  k_init3<S><<<grid3(a.s), dim3(32, 4), 0, st>>>(tb, a);
  return cudaGetLastError();
}

template cudaError_t launch_init3<float>(const Tables3&, const Init3Args<float>&, cudaStream_t);
template cudaError_t launch_init3<double>(const Tables3&, const Init3Args<double>&, cudaStream_t);

}  // namespace rlbm
