// Steps of one-row grids (ny = 1, the one-dimensional problems) in FP32 storage.
//
// A grid of a few thousand cells is all latency: a launch with its tables
// costs 2-3 us, fetching the constants again another one, and every cell has
// 2 hy images along y (280 stores at Q = 28, hy = 5).  Here one kernel
// takes many steps: the row is shared by the blocks of one cluster, a cell per
// thread, whose hardware barrier parts the steps, and the constants stay in the
// caches.  What is left is the serial chain of one cell (20 % of the issue slots at one
// warp per scheduler) and the barrier with its fence, 2.3 of 5.1 cycles per
// instruction.  Along y the row is its own neighbour, so that the steps read
// and write it alone (row_scalars) and the images of the two buffers are written
// once at the end.  1024 cells, Q = 28, 100 steps: 2.7 us per step (a launch
// per step with the images by the cell's thread: 18 us; by eight warps: 8.7).
// Rows of more cells than the cluster has threads take a launch per step, which still
// writes the row alone.  FP64 storage, order 3 and stencils without the orbit form
// step as other grids do.
#include "dispatch.h"
#include "step_impl.cuh"

namespace rlbm {
namespace {

// Eight blocks of at most 256 threads: the portable cluster.  1024 cells are a
// warp for each scheduler of eight SMs.
constexpr int kRowBlocks = 8, kRowThreads = 256;

// nsteps steps between the two buffers; gridDim.x is one cluster unless nsteps = 1.
template <int QT, int KT, int MODE, bool FW>
__global__ void __launch_bounds__(kRowThreads) k_row_steps(const __grid_constant__ Tables<float> tb,
                                                           const __grid_constant__ StepArgs<float> a, int nsteps) {
  const float* fin = chain_begin(a.fin);
  float* fout = a.fout;
  const float* const tau_field = chained(a.tau_field);
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  for (int step = 1;; ++step) {
    if (x < a.s.nx)
      cell_update<float, QT, true, KT, MODE, true, false, true, FW>(tb, a.s, fin, fout, tau_field, a.status, x, 0);
    if (step == nsteps) return;
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    const float* const next = fout;
    fout = const_cast<float*>(fin);
    fin = next;
  }
}

// The images along y of the row's storage (with its images along x).
template <typename S>
__global__ void __launch_bounds__(256) k_row_images(S* first, S* second, const __grid_constant__ Scalars s) {
  S* const f = chain_begin(blockIdx.z ? second : first) + (long long)blockIdx.y * s.plane + (s.px - s.hx);
  const int x = blockIdx.x * 256 + threadIdx.x;
  if (x >= s.nx + 2 * s.hx) return;
  const S v = f[(long long)s.hy * s.pitch + x];
  for (int r = 0; r < 2 * s.hy + 1; ++r)
    if (r != s.hy) f[(long long)r * s.pitch + x] = v;
}

template <int QT, int KT>
cudaError_t launch_q(const Tables<float>& tb, StepArgs<float> a, int mode, int nsteps, cudaStream_t st) {
  const bool chain = !a.s.plain;
  const int nx = a.s.nx, fw = a.s.sym_fw;
  auto kernel = mode == kOnLattice ? (fw ? k_row_steps<QT, KT, kOnLattice, true> : k_row_steps<QT, KT, kOnLattice, false>)
                                   : (fw ? k_row_steps<QT, KT, kBilinear, true> : k_row_steps<QT, KT, kBilinear, false>);
  const long long row = (long long)a.s.hy * a.s.pitch;
  const Scalars full = a.s;
  a.s = row_scalars(a.s);
  float* buf[2] = {const_cast<float*>(a.fin), a.fout};
  // Wider rows: a launch per step, blocks of a warp for each scheduler.
  const bool one = nx <= kRowBlocks * kRowThreads;
  const int blocks = one ? (nx > 128 ? kRowBlocks : 1) : (nx + 127) / 128;
  const int threads = one ? ((nx + blocks - 1) / blocks + 31) / 32 * 32 : 128;
  for (int done = 0; done < nsteps;) {
    const int n = one ? min(nsteps - done, 1024) : 1;      // (a launch stays below a few ms)
    a.fin = buf[done & 1] + row;
    a.fout = buf[(done & 1) ^ 1] + row;
    const cudaError_t e = launch_chained_clusters(chain, one ? blocks : 1, kernel, dim3(blocks), dim3(threads), 0, st,
                                                  tb, a, n);
    if (e != cudaSuccess) return e;
    done += n;
  }
  // both buffers' images; the one before a single step has its own already
  float* const last = buf[nsteps & 1];
  float* const before = buf[(nsteps & 1) ^ 1];
  return launch_chained(chain, k_row_images<float>, dim3((nx + 2 * full.hx + 255) / 256, full.Q, nsteps > 1 ? 2 : 1),
                        dim3(256), 0, st, last, before, full);
}

}  // namespace

bool row_steps_supported(const Scalars& s) {
  if (s.ny != 1 || !(s.sym || s.sym_fw)) return false;
  return s.K == 9 ? (s.Q == 28 || s.Q == 25 || s.Q == 29 || s.Q == 33) : false;
}

cudaError_t launch_row_steps(const Tables<float>& tb, const StepArgs<float>& a, int mode, int nsteps, cudaStream_t st) {
  switch (a.s.Q) {
    case 28: return launch_q<28, 9>(tb, a, mode, nsteps, st);
    case 25: return launch_q<25, 9>(tb, a, mode, nsteps, st);
    case 29: return launch_q<29, 9>(tb, a, mode, nsteps, st);
    case 33: return launch_q<33, 9>(tb, a, mode, nsteps, st);
    default: return cudaErrorInvalidValue;
  }
}

template <typename S>
cudaError_t launch_row_images(S* f, const Scalars& s, cudaStream_t st) {
  return launch_chained(true, k_row_images<S>, dim3((s.nx + 2 * s.hx + 255) / 256, s.Q, 1), dim3(256), 0, st, f, f, s);
}
template cudaError_t launch_row_images<float>(float*, const Scalars&, cudaStream_t);
template cudaError_t launch_row_images<double>(double*, const Scalars&, cudaStream_t);

}  // namespace rlbm
