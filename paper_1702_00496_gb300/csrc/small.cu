// small.cu -- many steps of a small 1D problem in one launch.
//
// A small problem's step is shorter than its launch: 256 points in PEs too narrow for blocks of K steps take 3.8 us per
// step as nodes of a captured graph.  Here one thread block keeps the whole problem for a run of steps: every thread
// updates a group of four points with the step kernels' own group_step (the same bits), spare warps draw the next step's
// delays meanwhile, and a barrier separates the steps.  What bounds it is latency: the barrier, the reads of the ring
// through L1 and the step's dependent chain (256 points: 1.14 us per step at order 2, 2.2 us at order 4).
//
// Measured against the graph, per step at order 2 / 4: 256 points 3.8 / 5.1 -> 1.14 / 2.2 us, 2048 points in 32 PEs 3.1 / 5.4
// -> 2.1 / 3.4 us.  Beyond one group per thread, and as a cluster of up to eight blocks with a cluster barrier between
// steps (4096 points in 64 PEs: 3.1 / 5.4 -> 3.5 / 5.8 us; 16384: 2.8 / 4.3 -> 3.5 / 5.8 us), the graph is faster, and
// blocks of K steps are where the PEs are wide enough for K >= 3 (131072 points: 1.2 / 1.5 us).
#include "stencil.cuh"

namespace {

using namespace atfd;

constexpr int kSmallThreads = 576;  // 512 groups of four points, and two warps that only draw delays

// GROUPED = false: shapes without aligned groups of four, point by point as the per-point kernel steps them.
template <int H, bool AB, int KIND, bool GROUPED>
__global__ void __launch_bounds__(kSmallThreads) small_steps_kernel(const StepParams p, const int64_t n0,
                                                                    const int64_t nsteps) {
  const int tid = threadIdx.x, nthreads = blockDim.x, groups = p.n[0] >> 2;
  const int g = tid < groups ? (int)group_1d_order(p, tid) : 0;
  int sn = (int)slot_of(n0, p.R);
  for (int64_t n = n0; n < n0 + nsteps; ++n) {
    const double *un = p.ring + sn * p.ntot;
    const int sout = sn + 1 == p.R ? 0 : sn + 1;
    double *out = p.ring + sout * p.ntot;
    const uint8_t *keff = p.keff + (n & 1) * p.nb;
    draw_sides(p, n + 1, nthreads - 1 - tid, nthreads, p.keff + ((n + 1) & 1) * p.nb);  // from the last thread down
    if (GROUPED) {
      if (tid < groups) group_step<1, H, LdCoherent, AB ? 1 : 0, KIND>(p, keff, un, out, n, sn, g << 2, 0, 0);
    } else {
      for (int i = tid; i < p.n[0]; i += nthreads) point_step<1, H, LdCoherent, AB, KIND>(p, keff, un, out, n, i);
    }
    __syncthreads();
    sn = sout;
  }
}

template <int H, bool AB, int KIND>
void launch_small_typed(const StepParams &p, bool grouped, int64_t n, int64_t nsteps, cudaStream_t st) {
  if (grouped) {
    const int threads = (p.n[0] / 4 + 31) / 32 * 32 + (p.nb < 64 ? (int)(p.nb + 31) / 32 * 32 : 64);
    small_steps_kernel<H, AB, KIND, true><<<1, threads, 0, st>>>(p, n, nsteps);
  } else {
    const int threads = p.n[0] < 512 ? (p.n[0] + 31) / 32 * 32 + 32 : kSmallThreads;
    small_steps_kernel<H, AB, KIND, false><<<1, threads, 0, st>>>(p, n, nsteps);
  }
}

bool small_grouped(const StepParams &p) {
  return p.n[0] % 4 == 0 && (!p.use_pe[0] || p.S[0] % 4 == 0) && reinterpret_cast<uintptr_t>(p.ring) % 16 == 0 &&
         (p.frhs == nullptr || reinterpret_cast<uintptr_t>(p.frhs) % 16 == 0);
}

template <int H>
void launch_small_h(const StepParams &p, int64_t n, int64_t nsteps, cudaStream_t st) {
  const bool ab = p.ts > 1, grouped = small_grouped(p);
  if (p.burgers) {
    if (ab) launch_small_typed<H, true, 1>(p, grouped, n, nsteps, st);
    else launch_small_typed<H, false, 1>(p, grouped, n, nsteps, st);
    return;
  }
  if constexpr (H == 1) {
    if (p.scheme >= AT_AT_SPACE2) {
      launch_small_typed<1, false, 2>(p, grouped, n, nsteps, st);
      return;
    }
  }
  if (ab) launch_small_typed<H, true, 0>(p, grouped, n, nsteps, st);
  else launch_small_typed<H, false, 0>(p, grouped, n, nsteps, st);
}

}  // namespace

bool small_steps_fit(const StepParams &p) { return p.dim == 1 && p.n[0] <= (small_grouped(p) ? 2048 : kSmallPoints); }

cudaError_t launch_small_steps(const StepParams &p, int64_t n, int64_t nsteps, cudaStream_t st) {
  const int64_t most = 4096;  // steps of one launch
  for (int64_t s = 0; s < nsteps; s += most) {
    const int64_t m = nsteps - s < most ? nsteps - s : most;
    if (p.h == 1) launch_small_h<1>(p, n + s, m, st);
    else if (p.h == 2) launch_small_h<2>(p, n + s, m, st);
    else launch_small_h<3>(p, n + s, m, st);
  }
  return cudaGetLastError();
}
