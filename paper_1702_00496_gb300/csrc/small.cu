// small.cu -- many steps of a small 1D problem in one launch.
//
// A small problem's step is shorter than its launch: 256 points in PEs too narrow for blocks of K steps take 3.8 us per
// step as nodes of a captured graph.  Here one thread block keeps the whole problem for a run of steps: every thread
// updates a group of four points with the step kernels' own group_step (the same bits), spare warps draw the next step's
// delays meanwhile, and a barrier separates the steps.  What bounds it is latency: the barrier, the reads of the ring
// through L1 and the step's dependent chain (1.35 us per step at order 2, 2.4 us at order 4).
//
// Measured against the graph, per step at order 2 / 4: 256 points 3.8 / 5.1 -> 1.35 / 2.4 us, 2048 points in 32 PEs 3.1 / 5.4
// -> 2.1 / 3.8 us.  Beyond one group per thread, and as a cluster of up to eight blocks with a cluster barrier between
// steps (4096 points in 64 PEs: 3.1 / 5.4 -> 3.5 / 5.8 us; 16384: 2.8 / 4.3 -> 3.5 / 5.8 us), the graph is faster, and
// blocks of K steps are where the PEs are wide enough for K >= 3 (131072 points: 1.2 / 1.5 us).
#include "stencil.cuh"

namespace {

using namespace atfd;

constexpr int kSmallThreads = 576;  // 512 groups of four points, and two warps that only draw delays

template <int H, bool AB, int KIND>
__global__ void __launch_bounds__(kSmallThreads) small_steps_kernel(const StepParams p, const int64_t n0,
                                                                    const int64_t nsteps) {
  const int tid = threadIdx.x, nthreads = blockDim.x, groups = p.n[0] >> 2;
  const int g = tid < groups ? (int)group_1d_order(p, tid) : 0;
  for (int64_t n = n0; n < n0 + nsteps; ++n) {
    const double *un = p.ring + slot_of(n, p.R) * p.ntot;
    double *out = p.ring + slot_of(n + 1, p.R) * p.ntot;
    const uint8_t *keff = p.keff + (n & 1) * p.nb;
    draw_sides(p, n + 1, nthreads - 1 - tid, nthreads, p.keff + ((n + 1) & 1) * p.nb);  // from the last thread down
    if (tid < groups) group_step<1, H, LdCoherent, AB ? 1 : 0, KIND>(p, keff, un, out, n, g << 2, 0, 0);
    __syncthreads();
  }
}

template <int H>
void launch_small_h(const StepParams &p, int threads, int64_t n, int64_t nsteps, cudaStream_t st) {
  const bool ab = p.ts > 1;
  if (p.burgers) {
    if (ab) small_steps_kernel<H, true, 1><<<1, threads, 0, st>>>(p, n, nsteps);
    else small_steps_kernel<H, false, 1><<<1, threads, 0, st>>>(p, n, nsteps);
    return;
  }
  if constexpr (H == 1) {
    if (p.scheme >= AT_AT_SPACE2) {
      small_steps_kernel<1, false, 2><<<1, threads, 0, st>>>(p, n, nsteps);
      return;
    }
  }
  if (ab) small_steps_kernel<H, true, 0><<<1, threads, 0, st>>>(p, n, nsteps);
  else small_steps_kernel<H, false, 0><<<1, threads, 0, st>>>(p, n, nsteps);
}

}  // namespace

bool small_steps_fit(const StepParams &p) {
  return p.dim == 1 && p.n[0] % 4 == 0 && p.n[0] <= 2048 && (!p.use_pe[0] || p.S[0] % 4 == 0) &&
         reinterpret_cast<uintptr_t>(p.ring) % 16 == 0 &&
         (p.frhs == nullptr || reinterpret_cast<uintptr_t>(p.frhs) % 16 == 0);
}

cudaError_t launch_small_steps(const StepParams &p, int64_t n, int64_t nsteps, cudaStream_t st) {
  const int groups = p.n[0] / 4;
  int threads = (groups + 31) / 32 * 32 + (int)(p.nb < 64 ? (p.nb + 31) / 32 * 32 : 64);
  const int64_t most = 4096;  // steps of one launch
  for (int64_t s = 0; s < nsteps; s += most) {
    const int64_t m = nsteps - s < most ? nsteps - s : most;
    if (p.h == 1) launch_small_h<1>(p, threads, n + s, m, st);
    else if (p.h == 2) launch_small_h<2>(p, threads, n + s, m, st);
    else launch_small_h<3>(p, threads, n + s, m, st);
  }
  return cudaGetLastError();
}
