// fwd.cu -- the fused forward step of the asynchrony-tolerant (AT) scheme on sm_103a.
//
// One launch advances U^n -> U^{n+1} by forward Euler (Sec. 4.1, Eq. "time_disc" with one level):
//     U^{n+1}_i = U^n_i + dt sum_a ( -c_a D1_a U + alpha D2_a U )_i = U^n_i + dt f^n_i
// with the central differences and the AT tables folded into merged per-axis coefficients
//     s_{a,j} = dt ( -c_a cd1_j / dx_a + alpha cd2_j / dx_a^2 ),   s0 = 1 + sum_a s_{a,0},
// so an interior point costs one multiply and 2*h*dim fused multiply-adds.  With two or three time levels
// (Adams-Bashforth, Eq. "time_disc"; Eq. "time_ab2") the chain, with s0 lacking the 1, forms dt f^n; the launch
// adds the stored dt f^{n-1}, dt f^{n-2} of the previous launches with their weights and stores dt f^n.
//
// Points within h of a PE boundary (the set I_B of Sec. 2) read, for each stencil point across that
// boundary (a buffer point), the extrapolated halo value
//     u~ = sum_{m<T} w_m(k) U^{n-k-m}                                   (k = that side's delay)
// where w_m(k) are the stage-2 weights of Example 3.  Since sum_m w_m(k) CD(.. U^{n-k-m} ..) =
// CD(.. u~ ..) for the time-expanded tables ((1,2,2)b, (2,2,2)b, (1,4,2), (2,4,2), (2,6,2)), the halo value is
// formed once and shared by the first- and second-derivative taps.  The delay k of every PE side is
// drawn from Philox (Sec. 5.1) keyed by (seed, step, side) once per step -- by the launch of the previous
// step, into a double-buffered array -- and clamped so that no level before 0 is read.
//
// The FP64 pipe of GB300 does two FMAs per SM and clock, which bounded every step kernel at 9 to 25 % of the memory
// rate while the sums were FP64 chains.  They are summed in block fixed point instead (fixed.cuh), three integer
// multiply-adds of 16 lanes or more a clock per tap; windows the fixed point does not take are chains still: 1 + 2 h dim
// FMAs per point, starting with fma(s0, u_i, +0) on a runtime zero (a DMUL occupies the pipe longer than a DFMA).
//
// Kernels of 1D: forward_block_kernel (K steps in one launch), forward_group_kernel (groups of four, one step),
// forward_ragged_kernel (large shapes without aligned groups), forward_point_kernel (small ones); 3D: the marched tiles
// (brick.cu) from the size on where they are faster, groups or points below; tiny 1D problems: small.cu.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "stencil.cuh"

namespace {

using namespace atfd;

// Grouped kernel: a thread updates four consecutive x points per iteration (grid-stride); every thread
// also draws the delays of one slice of the PE sides for step n+1 into the other half of the double-buffered
// delay array, so the next launch finds them ready.
//
// 1D groups are summed in fixed point (stencil.cuh); two blocks of 512 per SM (64 registers) hide the latency of their
// integer chains: at N = 2^24 the AB2 step of order 4 takes 105 us against 133 us with the 88 registers it would use.
// The chains of 3D groups want the same but with Adams-Bashforth (160^3 in 8^3 PEs, order 2: 70.3 against 74.5 us with the 76
// registers they would use).
template <int DIM, int H, int AB, int KIND>
__global__ void __launch_bounds__(512, DIM == 1 || !AB ? 2 : 1) forward_group_kernel(const StepParams p, const int64_t n_off,
                                                            const int64_t *n_base) {
  const int64_t n = n_off + (n_base ? *n_base : 0);
  const int sn = (int)slot_of(n, p.R);
  const double *__restrict__ un = p.ring + sn * p.ntot;
  double *__restrict__ out = p.ring + slot_of(n + 1, p.R) * p.ntot;
  const uint8_t *keff = p.keff + (n & 1) * p.nb;
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, nthreads = (int64_t)gridDim.x * blockDim.x;
  draw_sides(p, n + 1, tid, nthreads, p.keff + ((n + 1) & 1) * p.nb);
  const int gx = p.n[0] >> 2;
  const int64_t groups = (int64_t)gx * p.n[1] * p.n[2];
  for (int64_t k = tid; k < groups; k += nthreads) {
    if (DIM == 1) {
      const int64_t g = group_1d_order(p, k);
      group_step<1, H, LdgNC, AB, KIND>(p, keff, un, out, n, sn, (int)(g << 2), 0, 0);
    } else {
      const int64_t g = p.order ? (int64_t)p.order[k] : k;
      const int64_t r = g / gx;
      const int x0 = (int)(g - r * gx) << 2;
      const int z = (int)(r / p.n[1]), y = (int)(r - (int64_t)z * p.n[1]);
      group_step<3, H, LdgNC, AB, KIND>(p, keff, un, out, n, sn, x0, y, z);
    }
  }
}

// Blocks of K steps (1D forward Euler, central and time-expanded rows), one launch each.  Away from PE boundaries the
// step is the same linear stencil at every point and step, so K steps of it are one stencil of half-width h K: its taps
// ck are the K-fold composition of the merged taps, and a cell whose K-step stencil stays inside its PE gets U^{n+K}
// from U^n with 2 h K + 1 taps instead of K (2 h + 1).  The cells near a PE boundary, whose buffer points take the
// delayed halo values of every step, are advanced step by step by one warp per boundary (zone_steps): steps n .. n+K-2
// on the cells within zr[j] of it (zones that shrink by at least h per step), the last step on the 4 fe cells that no
// composed stencil reaches.  The zones hold the face strips, so the intermediate levels are in the ring wherever a later
// step reads a delayed level.  A boundary's warp draws the delays of the two sides that face it for steps n+1 .. n+K,
// so the delay log and the effective delays are those of single steps.
//
// Zones and inner cells of a block do not depend on one another: both read U^n (and a zone the delayed levels of its own
// boundary's cells, before it overwrites them); a zone writes cells that only it reads; the slots of n+1 .. n+K differ
// from U^n's (K < R).  As two launches, the second waiting for the first before its edge groups, a block of a 12000-point
// problem took 17.6 us; as one it takes 6.9.

// Shared memory of a zone: levels n .. n+K-1 of the region (cells b - RR .. b + RR - 1, RR = zr[0] + h <= 27), the 2 h
// face cells at the R - 2 levels before n, and their halo values of the current step.
template <int H, int K>
struct Zone {
  static constexpr int CELLS = 2 * 27 + 2, HIST = (AT_MAX_L + AT_MAX_T) * 2 * H;
  static constexpr int BYTES = (K * CELLS + HIST + 2 * H) * 8;
};

// Steps n .. n+K-1 near the PE boundary b (a warp).  The arithmetic is the FP64 chain's: the centre tap, then the taps in
// offset order, a buffer point's value extrapolated over the delayed levels w_m(k) in the order m = 0 .. T-1.  Every
// global load is in flight before the first step.
template <int H, int K>
__device__ __forceinline__ void zone_steps(const StepParams &p, int64_t n, int sn, int b, int lane, double *sh) {
  constexpr int CELLS = Zone<H, K>::CELLS;
  double *lev = sh, *hist = sh + K * CELLS, *hv = hist + Zone<H, K>::HIST;
  const bool split = p.use_pe[0] != 0;
  const int P = p.pe[0], nx = p.n[0], RR = p.zr[0] + H, R = p.R;
  // the sides facing the boundary: the right one of the PE before it, the left one of the PE after it
  const int side = lane & 1 ? (split ? 2 * b : 1) : (split ? 2 * (b == 0 ? P - 1 : b - 1) + 1 : 0);
  const int base = b * p.S[0] - RR;  // cell of local index 0 (before wrapping)
  int k = lane < 2 ? p.keff[(n & 1) * p.nb + side] : 0;  // lanes 0, 1: delays of step n; lanes 2j, 2j+1: of step n + j
  if (split) {
    const double *un = p.ring + (int64_t)sn * p.ntot;
    for (int i = lane; i < 2 * RR; i += 32) lev[i] = un[wrap_coord(base + i, nx)];
    for (int e = lane; e < (R - 2) * 2 * H; e += 32) {
      const int d = e / (2 * H), c = e - d * (2 * H);
      hist[e] = p.ring[slot_back(sn, d + 1, R) * p.ntot + wrap_coord(base + RR - H + c, nx)];
    }
  }
  int last = 0;
  if (lane < 2 * K) {  // delays of steps n+1 .. n+K
    const int64_t st = n + 1 + (lane >> 1);
    int raw = 0;
    if (p.scheme != 0) raw = delay_draw(p.seed, (uint32_t)st, (uint32_t)side, p.L, p.use_thr ? p.thr : nullptr);
    last = delay_clamp(raw, st, p.T);
    if (p.log != nullptr && st < p.log_steps) p.log[st * p.nb + side] = (uint8_t)raw;
  }
  __syncwarp();  // for even K the delays of step n + K go where lanes 0 and 1 read those of step n; a shuffle orders no memory
  const int up = __shfl_up_sync(0xffffffffu, last, 2);
  if (lane >= 2) k = up;
  if (lane >= 2 * K - 2 && lane < 2 * K) p.keff[((n + K) & 1) * p.nb + side] = (uint8_t)last;
  if (!split) return;
  __syncwarp();
#pragma unroll
  for (int j = 0; j < K; ++j) {
    const int k_lo = __shfl_sync(0xffffffffu, k, 2 * j), k_hi = __shfl_sync(0xffffffffu, k, 2 * j + 1);
    if (lane < 2 * H) {  // halo value of face cell lane: the left ones are buffer points of the PE after the boundary
      const int ii = RR - H + lane, kk = lane < H ? k_hi : k_lo;
      double v = lev[j * CELLS + ii];
      if (kk > 0) {
#pragma unroll
        for (int m = 0; m <= H; ++m) {
          if (m >= p.T) break;
          const int q = j - kk - m;  // level relative to n
          const double u = q >= 0 ? lev[q * CELLS + ii] : hist[(-q - 1) * 2 * H + lane];
          v = m == 0 ? fma(p.w[kk][0], u, p.zero) : fma(p.w[kk][m], u, v);
        }
      }
      hv[lane] = v;
    }
    __syncwarp();
    double *out = p.ring + (int64_t)slot_back(sn, R - 1 - j, R) * p.ntot;  // slot of level n + j + 1
    const int r = j + 1 < K ? p.zr[j] : 4 * p.fe;
    for (int i = RR - r + lane; i < RR + r; i += 32) {
      const bool left = i < RR;
      double acc = fma(p.s0, lev[j * CELLS + i], p.zero);
#pragma unroll
      for (int t = -H; t <= H; ++t) {
        if (t == 0) continue;
        const int ii = i + t;
        const double v = left == (ii < RR) ? lev[j * CELLS + ii] : hv[ii - (RR - H)];
        acc = fma(p.s[0][t + H], v, acc);
      }
      if (j + 1 < K) lev[(j + 1) * CELLS + i] = acc;
      out[wrap_coord(base + i, nx)] = acc;
    }
    __syncwarp();
  }
}

// One inner cell of a block as an FP64 chain: U^{n+K}_x = sum ck_j U^n_{x+j}, the centre first, then j ascending.  The cells of
// a warp are consecutive ones, or some of them.
template <int TK>
__device__ __noinline__ double block_cell(const StepParams &p, const double *__restrict__ u0, int x) {
  const int nx = p.n[0];
  double acc = fma(p.ck[TK], LdgNC::ld(u0 + x), p.zero);
  if (x >= TK && x + TK < nx) {
#pragma unroll
    for (int j = -TK; j <= TK; ++j)
      if (j != 0) acc = fma(p.ck[j + TK], LdgNC::ld(u0 + x + j), acc);
  } else {
    for (int j = -TK; j <= TK; ++j)
      if (j != 0) acc = fma(p.ck[j + TK], LdgNC::ld(u0 + wrap_coord(x + j, nx)), acc);
  }
  return acc;
}

// Cells per lane and warp tile of the inner cells: a tile is 32 C consecutive cells of one PE.
template <int TK, int C>
struct BlockTile {
  static constexpr int CELLS = 32 * C, WIN = CELLS + 2 * TK;
  static constexpr int SLOTS = WIN + WIN / C + 1;  // one pad slot per C cells: lanes C cells apart take all banks
};
template <int H, int K, int C>
constexpr int block_warp_bytes() {  // of a warp, for a zone or a tile
  const int t = BlockTile<H * K, C>::SLOTS * 8, z = Zone<H, K>::BYTES;
  return (t > z ? t : z) + 15 & ~15;
}

// The C outputs of a lane from its window in shared memory, four at a time (independent chains for the pipe's latency).
// F32: the low parts are there as FP32 and the cross terms are summed in FP32.  Returns a bit for every four cells that are
// for the chain (fixed.cuh, kFxLeast).
template <int TK, int C, bool F32, int NT>
__device__ __forceinline__ uint32_t block_sums(const FxTaps<NT> &t, const int2 *sm, int lane, int ex, double r[C]) {
  uint32_t small = 0;
  int2 w[C + 2 * TK];
  float h[C + 2 * TK];
#pragma unroll
  for (int i = 0; i < C + 2 * TK; ++i) {
    w[i] = sm[lane * (C + 1) + i + i / C];
    if (F32) h[i] = __int2float_rn(w[i].x);
  }
#pragma unroll
  for (int q0 = 0; q0 < C; q0 += 4) {
    int64_t A[4], B[4], D[4];
    FxCross c[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      A[q] = 0; B[q] = kFxB0; D[q] = kFxC0;
      c[q] = {0.0f, 0.0f};
    }
#pragma unroll
    for (int m = 0; m <= 2 * TK; ++m) {
      const int j = fx_inward(m, 2 * TK + 1);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int i = q0 + q + j;
        A[q] = fx_mad(t.w1[j], w[i].x, A[q]);
        if (F32) {
          fx_cross(c[q], t, j, __int_as_float(w[i].y), h[i]);
        } else {
          B[q] = fx_mad(t.w1[j], w[i].y, B[q]);
          D[q] = fx_mad(t.w0[j], w[i].x, D[q]);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) A[q] = F32 ? fx_join_cross(A[q], c[q]) : fx_join(A[q], B[q], D[q]);
    if (fx_results_wide<4>(A, ex, r + q0) < (F32 ? kFxLeastNear : kFxLeast)) small |= 1u << (q0 / 4);
  }
  return small;
}

// A block: zones near the PE boundaries, inner cells U^{n+K} = ck * U^n.
//
// The inner cells are a contraction of 2 h K + 1 constant taps, which the FP64 pipe bounded (17 DFMA per cell at order
// 4 and K = 4).  They are summed in block fixed point (fixed.cuh).  A warp takes a tile of 32 C cells: it reads the tile
// and its halo once (coalesced, all loads in flight together), finds their largest exponent, converts every value once
// and lays the two 32-bit parts in shared memory; each lane then reads the window of its C cells once, sums its C
// outputs from registers, and the results go back through shared memory to coalesced stores.  What bounds it is the
// issue of the integer and FP32 pipes: per cell 17 multiply-adds of 64 bits (four cycles of a quarter each), 34 FFMA and
// about 70 other instructions at order 4 and K = 4.  The zones, bound by the FP64 pipe's latency, run beside.
template <int H, int K, int C>
__global__ void __launch_bounds__(256, 3) forward_block_kernel(const StepParams p, const int64_t n_off,
                                                               const int64_t *n_base) {
  constexpr int TK = H * K;                  // half-width of the composed stencil
  using Tile = BlockTile<TK, C>;
  extern __shared__ __align__(16) char block_smem[];
  const int64_t n = n_off + (n_base ? *n_base : 0);
  const int sn = (int)slot_of(n, p.R);
  const double *__restrict__ u0 = p.ring + (int64_t)sn * p.ntot;
  double *__restrict__ out = p.ring + slot_back(sn, p.R - K, p.R) * p.ntot;
  const int tid = blockIdx.x * blockDim.x + threadIdx.x, warps = (gridDim.x * blockDim.x) >> 5;
  const int nx = p.n[0];
  const int lane = threadIdx.x & 31;
  int2 *sm = reinterpret_cast<int2 *>(block_smem + (threadIdx.x >> 5) * block_warp_bytes<H, K, C>());
  const int S = p.use_pe[0] ? p.S[0] : nx, inner = S - 8 * p.fe;
  const int per_pe = (inner + Tile::CELLS - 1) / Tile::CELLS;
  const int tiles = (nx / S) * per_pe, zones = p.use_pe[0] ? p.pe[0] : 1;
  // Work items, one per warp at a time: the zones (long chains) first, then the tiles.
  for (int w = tid >> 5; w < zones + tiles; w += warps) {
    if (w < zones) {
      zone_steps<H, K>(p, n, sn, w, lane, reinterpret_cast<double *>(sm));
      __syncwarp();
      continue;
    }
    const int t = w - zones;
    const int pe = t / per_pe, off = (t - pe * per_pe) * Tile::CELLS;
    const int x0 = pe * S + 4 * p.fe + off, len = min(Tile::CELLS, inner - off);
    // A PE's last tile reads on past its inner cells: U^n is written nowhere meanwhile, and only the scale sees them.
    double v[C + 1];  // 2 TK <= 24 < 32: the halo takes at most one more value per lane
    const double *src = u0 + (x0 - TK + lane);
    if (x0 >= TK && x0 - TK + Tile::WIN <= nx) {
#pragma unroll
      for (int q = 0; q < C; ++q) v[q] = LdgNC::ld(src + 32 * q);
      v[C] = lane < 2 * TK ? LdgNC::ld(src + 32 * C) : v[0];
    } else {  // the window wraps around the domain, or around a small one more than once
#pragma unroll
      for (int q = 0; q <= C; ++q) {
        int i = x0 - TK + min(lane + 32 * q, Tile::WIN - 1);
        i = i < 0 ? i + nx : i;
        v[q] = LdgNC::ld(u0 + i % nx);
      }
    }
    int hi = 0, lo = 0x7fffffff;
#pragma unroll
    for (int q = 0; q <= C; ++q) {
      hi = max(hi, fx_mag(v[q]));
      lo = min(lo, fx_mag(v[q]));
    }
    const int E = __reduce_max_sync(0xffffffffu, hi) >> 20;
    const bool near = (__reduce_min_sync(0xffffffffu, lo) >> 20) >= E - kFxNear;
    const bool fixed = p.fck.ok && fx_usable(E);  // the same for the whole warp
    double r[C];
    uint32_t chain = 0;  // a bit for every four of this lane's cells that are for the chain
    __syncwarp();
    if (fixed) {
#pragma unroll
      for (int q = 0; q <= C; ++q) {
        const int i = lane + 32 * q;
        const Fx f = fx_split(fx_from(v[q], E));
        const int low = near ? __float_as_int(__int2float_rn(f.lo)) : f.lo;
        if (q < C || lane < 2 * TK) sm[i + i / C] = make_int2(f.hi, low);
      }
      __syncwarp();
      if (near) chain = block_sums<TK, C, true>(p.fck, sm, lane, E - 1023 - p.fck.sw, r);
      else chain = block_sums<TK, C, false>(p.fck, sm, lane, E - 1023 - p.fck.sw, r);
    } else {
      int low = 0;
#pragma unroll
      for (int q = 0; q <= C; ++q) low |= fx_mag(v[q]) | fx_word(v[q], 0);
      chain = __any_sync(0xffffffffu, low != 0) ? ~0u : 0u;  // sums of zeros are zero, as the chain's
#pragma unroll
      for (int q = 0; q < C; ++q) r[q] = 0.0;
    }
    __syncwarp();
    double *ro = reinterpret_cast<double *>(sm) + lane * (C + 1);
#pragma unroll
    for (int q = 0; q < C; ++q) ro[q] = r[q];
    __syncwarp();
    ro = reinterpret_cast<double *>(sm);
    double *dst = out + x0 + lane;
    if (__any_sync(0xffffffffu, chain != 0)) {
#pragma unroll 1
      for (int q = 0; q < C; ++q) {
        const int i = lane + 32 * q;
        const uint32_t owner = __shfl_sync(0xffffffffu, chain, i / C);
        if (i < len) dst[32 * q] = owner >> (i % C / 4) & 1 ? block_cell<TK>(p, u0, x0 + i) : ro[i + i / C];
      }
    } else if (len == Tile::CELLS) {
#pragma unroll
      for (int q = 0; q < C; ++q) dst[32 * q] = ro[lane + 32 * q + (lane + 32 * q) / C];
    } else {
#pragma unroll
      for (int q = 0; q < C; ++q)
        if (lane + 32 * q < len) dst[32 * q] = ro[lane + 32 * q + (lane + 32 * q) / C];
    }
  }
}

// Fallback for shapes the grouped kernel does not take (n[0] not a multiple of 4, odd slots).
template <int DIM, int H, bool AB, int KIND>
__global__ void __launch_bounds__(512) forward_point_kernel(const StepParams p, const int64_t n_off,
                                                            const int64_t *n_base) {
  const int64_t n = n_off + (n_base ? *n_base : 0);
  const double *__restrict__ un = p.ring + slot_of(n, p.R) * p.ntot;
  double *__restrict__ out = p.ring + slot_of(n + 1, p.R) * p.ntot;
  const uint8_t *keff = p.keff + (n & 1) * p.nb;
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, nthreads = (int64_t)gridDim.x * blockDim.x;
  draw_sides(p, n + 1, tid, nthreads, p.keff + ((n + 1) & 1) * p.nb);
  for (int64_t i = tid; i < p.ntot; i += nthreads) point_step<DIM, H, LdgNC, AB, KIND>(p, keff, un, out, n, i);
}

// Large 1D shapes without aligned groups of four: groups cut from each PE's first cell (750000 points in PEs of 250, order
// 4: the per-point kernel took 15.7 us per step, bound by its FP64 chains and index divisions, this one 9.8; 10 million
// points unsplit with AB2 851 against 90).
template <int H, int AB, int KIND>
__global__ void __launch_bounds__(256, 4) forward_ragged_kernel(const StepParams p, const int64_t n_off,
                                                                const int64_t *n_base) {
  const int64_t n = n_off + (n_base ? *n_base : 0);
  const int sn = (int)slot_of(n, p.R);
  const double *__restrict__ un = p.ring + sn * p.ntot;
  double *__restrict__ out = p.ring + slot_of(n + 1, p.R) * p.ntot;
  const uint8_t *keff = p.keff + (n & 1) * p.nb;
  const int tid = blockIdx.x * blockDim.x + threadIdx.x, nthreads = gridDim.x * blockDim.x;
  draw_sides(p, n + 1, tid, nthreads, p.keff + ((n + 1) & 1) * p.nb);
  const int groups = p.use_pe[0] ? p.pe[0] * ((p.S[0] + 3) >> 2) : (p.n[0] + 3) >> 2;
  for (int k = tid; k < groups; k += nthreads) group_ragged<H, LdgNC, AB, KIND>(p, keff, un, out, n, sn, k);
}

// dt f(u) with central differences everywhere (p carries no PE split and s0 without the 1): the right-hand
// sides before the first step of an Adams-Bashforth run.
template <int DIM, int H>
__global__ void __launch_bounds__(256) sync_rhs_kernel(const StepParams p, const double *__restrict__ u,
                                                       double *__restrict__ out, int grouped) {
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, nthreads = (int64_t)gridDim.x * blockDim.x;
  if (grouped) {
    const int gx = p.n[0] >> 2;
    for (int64_t g = tid; g < p.ntot / 4; g += nthreads) {
      const int64_t r = g / gx;
      const int x0 = (int)(g - r * gx) << 2;
      const int z = (int)(r / p.n[1]), y = (int)(r - (int64_t)z * p.n[1]);
      double f[4], uc[4];
      group_eval<DIM, H, LdgNC, false>(p, p.keff, u, 0, x0, y, z, f, uc);
      const int64_t i0 = (DIM == 3 ? ((int64_t)z * p.n[1] + y) * p.n[0] : 0) + x0;
      for (int q = 0; q < 4; ++q) out[i0 + q] = f[q];
    }
  } else {
    for (int64_t i = tid; i < p.ntot; i += nthreads) {
      int c[3];
      point_coords(p, DIM, i, c);
      out[i] = point_update<DIM, H, LdgNC>(p, p.keff, u, 0, i, c);
    }
  }
}

__global__ void draw_first_kernel(const StepParams p, int64_t n) {
  draw_sides(p, n, (int64_t)blockIdx.x * blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x,
             p.keff + (n & 1) * p.nb);
}

__global__ void add_steps_kernel(int64_t *n_base, int64_t v, int set) {
  if (set) *n_base = v; else *n_base += v;
}

}  // namespace

cudaError_t launch_step_counter(int64_t *n_base, int64_t v, bool set, cudaStream_t st) {
  add_steps_kernel<<<1, 1, 0, st>>>(n_base, v, set ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_draw_delays(const StepParams &p, int64_t n, cudaStream_t st) {
  const int64_t blocks = (p.nb + 255) / 256;
  draw_first_kernel<<<(int)(blocks < 1024 ? blocks : 1024), 256, 0, st>>>(p, n);
  return cudaGetLastError();
}

namespace {

// 1D shapes without aligned groups of four from this many points on are summed in fixed point (launch_typed)
constexpr int64_t kRaggedPoints = 196608;

// groups of four x points must not straddle a PE and must start on 16 bytes
bool grouped_shape(const StepParams &p, const void *base) {
  return p.n[0] % 4 == 0 && (!p.use_pe[0] || p.S[0] % 4 == 0) && (reinterpret_cast<uintptr_t>(base) % 16) == 0 &&
         (p.frhs == nullptr || (reinterpret_cast<uintptr_t>(p.frhs) % 16) == 0);
}

int sm_count() {
  int sms = 152, dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

// AB: 0 forward Euler, 1 Adams-Bashforth, 2 AB2 with both levels stored (the 1D linear grouped step only; Burgers'
// step, 3D and the per-point fallback take the general form: Burgers' AB2 step measured 462 against 406 us in it).
template <int DIM, int H, int AB>
void launch_typed(const StepParams &p, bool grouped, int blocks, int threads, int64_t n, const int64_t *n_base,
                  cudaStream_t st) {
  constexpr int ABG = AB ? 1 : 0;
  // per step, tiny / per million points more, us: the per-point kernel 2.9 / 7.5 (order 2), 3.9 / 9.3 (order 4), 5.6 / 11.7
  // (order 6), 4.3 / 22 (AB2); groups in fixed point 3.1 / 4.6, 4.6 / 5.8, 6.4 / 6.6, 5.4 / 9.5
  const bool ragged = p.ntot >= kRaggedPoints;
  const int rblocks = (int)std::min<int64_t>((p.ntot / 2 + 255) / 256, (int64_t)sm_count() * 32);
  if (DIM == 1 && p.burgers) {
    if (grouped) forward_group_kernel<1, H, ABG, 1><<<blocks, threads, 0, st>>>(p, n, n_base);
    else if (ragged) forward_ragged_kernel<H, ABG, 1><<<rblocks, 256, 0, st>>>(p, n, n_base);
    else forward_point_kernel<1, H, ABG != 0, 1><<<blocks, threads, 0, st>>>(p, n, n_base);
    return;
  }
  if constexpr (H == 1 && !AB) {
    if (p.scheme >= AT_AT_SPACE2) {  // rows expanded in space: order 2, forward Euler only
      if (grouped) forward_group_kernel<DIM, 1, false, 2><<<blocks, threads, 0, st>>>(p, n, n_base);
      else forward_point_kernel<DIM, 1, false, 2><<<blocks, threads, 0, st>>>(p, n, n_base);
      return;
    }
  }
  if (grouped) forward_group_kernel<DIM, H, DIM == 1 ? AB : ABG, 0><<<blocks, threads, 0, st>>>(p, n, n_base);
  else if (DIM == 1 && ragged) forward_ragged_kernel<H, ABG, 0><<<rblocks, 256, 0, st>>>(p, n, n_base);
  else forward_point_kernel<DIM, H, AB != 0, 0><<<blocks, threads, 0, st>>>(p, n, n_base);
}

template <int DIM, int AB>
void launch_h(const StepParams &p, bool grouped, int blocks, int threads, int64_t n, const int64_t *n_base,
              cudaStream_t st) {
  if (p.h == 1) launch_typed<DIM, 1, AB>(p, grouped, blocks, threads, n, n_base, st);
  else if (p.h == 2) launch_typed<DIM, 2, AB>(p, grouped, blocks, threads, n, n_base, st);
  else launch_typed<DIM, 3, AB>(p, grouped, blocks, threads, n, n_base, st);
}

}  // namespace

cudaError_t launch_forward_step(const StepParams &p, int64_t n, const int64_t *n_base, cudaStream_t st) {
  cudaError_t be = cudaSuccess;
  if (p.dim == 3 && launch_forward_brick(p, n, n_base, st, &be)) return be;
  const bool grouped = grouped_shape(p, p.ring);
  const bool own = p.threads <= 0 && p.dim == 1 && grouped;  // no shape set: the one below
  const int threads = p.threads > 0 ? p.threads : (own ? 128 : 256);
  const int sms = sm_count(), max_blocks = sms * (p.blocks_per_sm > 0 ? p.blocks_per_sm : (own ? 40 : 32));
  const int64_t work = grouped ? p.ntot / 4 : p.ntot;
  const int64_t b = (work + threads - 1) / threads;
  int blocks = (int)(b < max_blocks ? b : max_blocks);
  // 1D groups: blocks of 128, eight resident per SM, in whole waves -- a last wave of few blocks costs as much as a full
  // one, a second group per thread much less.  Per step, blocks of 256 capped at 32 per SM -> this: 2^22 points AB3 order 6
  // 48.5 -> 37.7 us, Burgers AB2 order 4 43.5 -> 35.8; 2^24 points AB2 103.6 -> 100.0; 2^20 points AB2 12.0 -> 10.1.
  if (p.dim == 1 && grouped && threads == 128 && blocks > 8 * sms) blocks -= blocks % (8 * sms);
  // a launch inside a captured graph (n_base set) runs only at steps at or after ab_steady
  const bool ab = p.ts > 1, steady = p.ts == 2 && (n_base != nullptr || n >= p.ab_steady);
  if (p.dim == 1) {
    if (steady) launch_h<1, 2>(p, grouped, blocks, threads, n, n_base, st);
    else if (ab) launch_h<1, 1>(p, grouped, blocks, threads, n, n_base, st);
    else launch_h<1, 0>(p, grouped, blocks, threads, n, n_base, st);
  } else {
    if (ab) launch_h<3, 1>(p, grouped, blocks, threads, n, n_base, st);
    else launch_h<3, 0>(p, grouped, blocks, threads, n, n_base, st);
  }
  return cudaGetLastError();
}

namespace {

template <int H, int K, int C>
void launch_block_tiles(const StepParams &p, int max_blocks, int64_t tiles, int threads, int64_t n_off,
                        const int64_t *n_base, cudaStream_t st) {
  const int warps = threads / 32, bytes = warps * block_warp_bytes<H, K, C>();
  auto kernel = forward_block_kernel<H, K, C>;
  if (bytes > 48 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  const int64_t items = tiles + (p.use_pe[0] ? p.pe[0] : 1), b = (items + warps - 1) / warps;
  kernel<<<(unsigned)(b < max_blocks ? b : max_blocks), threads, bytes, st>>>(p, n_off, n_base);
}

// Tiles of 32 C cells over the inner cells of every PE.
int64_t block_tiles(const StepParams &p, int C) {
  const int64_t S = p.use_pe[0] ? p.S[0] : p.n[0], inner = S - 8 * p.fe;
  return p.n[0] / S * ((inner + 32 * C - 1) / (32 * C));
}

template <int H, int K>
void launch_block_typed(const StepParams &p, int max_blocks, int threads, int64_t n_off, const int64_t *n_base,
                        cudaStream_t st) {
  // Cells per lane: 8 convert 9/8 of the values and give a PE's last tile of 256 cells to fill, 4 convert 5/4 of them
  // and fill tiles of 128; instructions per tile: C + 1 conversions and C outputs.
  const int64_t t8 = block_tiles(p, 8), t4 = block_tiles(p, 4);
  const int taps = 3 * (2 * H * K + 1) + 22;
  if (t8 >= sm_count() * 16 && t8 * (9 * 11 + 8 * taps) <= t4 * (5 * 11 + 4 * (taps + 8)))
    launch_block_tiles<H, K, 8>(p, max_blocks, t8, threads, n_off, n_base, st);
  else
    launch_block_tiles<H, K, 4>(p, max_blocks, t4, threads, n_off, n_base, st);
}

template <int H>
void launch_block_h(const StepParams &p, int blocks, int threads, int64_t n_off, const int64_t *n_base,
                    cudaStream_t st) {
  if (p.fuse_k == 2) launch_block_typed<H, 2>(p, blocks, threads, n_off, n_base, st);
  else if (p.fuse_k == 3) launch_block_typed<H, 3>(p, blocks, threads, n_off, n_base, st);
  else launch_block_typed<H, 4>(p, blocks, threads, n_off, n_base, st);
}

}  // namespace

cudaError_t launch_forward_block(const StepParams &p, int64_t n_off, const int64_t *n_base, cudaStream_t st) {
  // 80 registers give three blocks of 256 threads per SM, or six of 128, whose last wave is shorter (2^24 points, order 4:
  // 26.4 against 24.8 us per step)
  const int threads = p.threads <= 128 ? 128 : 256;
  const int max_blocks = sm_count() * (p.blocks_per_sm > 0 ? p.blocks_per_sm : 32);
  if (p.h == 1) launch_block_h<1>(p, max_blocks, threads, n_off, n_base, st);
  else if (p.h == 2) launch_block_h<2>(p, max_blocks, threads, n_off, n_base, st);
  else launch_block_h<3>(p, max_blocks, threads, n_off, n_base, st);
  return cudaGetLastError();
}

// Zone radii of a K-step block: the edge groups of the last step reach 4 ceil(h K / 4) cells in from each PE end and
// read U^{n+K-1} h cells further; each earlier step's zone reaches h cells further than the next one's (multiples
// of 4, so zones are whole groups).
static void fuse_radii(int h, int K, int *fe, int zr[]) {
  const int reach = (h * K + 3) / 4 * 4;
  *fe = reach / 4;
  int r = reach;
  for (int j = K - 2; j >= 0; --j) {
    r = (r + h + 3) / 4 * 4;
    zr[j] = r;
  }
}

int fuse_max_k(const StepParams &p, const void *ring, int kmax) {
  // The block kernel itself takes any PE width and alignment.  Shapes without aligned groups of four that run a call's
  // steps in one launch (small.cu) stay there; the others take blocks like the aligned ones (order 4, per step: 750000
  // points in PEs of 250 9.8 us in single steps, 3.7 in blocks of 4; 30030 points in PEs of 143 4.4, 1.6 in blocks of 3).
  if (p.dim != 1 || p.scheme > AT_AT || p.burgers || p.ts != 1) return 1;
  if (!grouped_shape(p, ring) && p.ntot <= kSmallPoints) return 1;
  for (int K = kmax < AT_MAX_FUSE ? kmax : AT_MAX_FUSE; K >= 2; --K) {
    if (p.R <= K) continue;  // U^n must stay in the ring while U^{n+K} is written
    int fe, zr[AT_MAX_FUSE];
    fuse_radii(p.h, K, &fe, zr);
    const int WK = (p.h * K + 1) / 2 * 2;
    if (p.n[0] < 2 * (4 + 2 * WK)) continue;  // the composed window stays within one wrap of the domain
    if (p.use_pe[0] && (2 * zr[0] > p.S[0] || p.S[0] / 4 <= 2 * fe)) continue;
    if (p.use_pe[0]) {  // FP64 operations per PE and block against K single steps: blocks must save 5 %
      const int64_t S = p.S[0], taps = 2 * p.h + 1;
      int64_t zone = 0;
      for (int j = 0; j + 1 < K; ++j) zone += 2 * zr[j];
      const int64_t block = zone * taps + (S - 8 * fe) * (2 * p.h * K + 1) + 8 * fe * taps;
      if (20 * block > 19 * K * S * taps) continue;
    }
    return K;
  }
  return 1;
}

void fuse_setup(StepParams *p, int k) {
  p->fuse_k = k > 1 ? k : 0;
  p->fe = 0;
  std::memset(p->zr, 0, sizeof(p->zr));
  std::memset(p->ck, 0, sizeof(p->ck));
  std::memset(&p->fck, 0, sizeof(p->fck));
  if (k <= 1) return;
  const int h = p->h;
  fuse_radii(h, k, &p->fe, p->zr);
  if (!p->use_pe[0]) p->fe = 0;
  // K-fold composition of the merged taps (s0 at the centre), in pairs of doubles: the fixed-point weights keep more bits
  // than a double, and the roundings of a composition in doubles would pull every block the same way
  constexpr int N = 2 * AT_MAX_H * AT_MAX_FUSE + 1;
  double s[2 * AT_MAX_H + 1], c[N] = {1.0}, cl[N] = {0.0}, t[N], tl[N];
  for (int j = -h; j <= h; ++j) s[j + h] = j == 0 ? p->s0 : p->s[0][j + h];
  int w = 0;  // c + cl holds taps -w .. w at 0 .. 2w
  for (int step = 0; step < k; ++step) {
    const int w2 = w + h;
    for (int i = 0; i <= 2 * w2; ++i) t[i] = tl[i] = 0.0;
    for (int i = 0; i <= 2 * w; ++i)
      for (int j = 0; j <= 2 * h; ++j) {
        const double m = c[i] * s[j], ml = std::fma(c[i], s[j], -m) + cl[i] * s[j];
        double &sum = t[i + j];
        const double next = sum + m, of_m = next - sum;
        tl[i + j] += ((sum - (next - of_m)) + (m - of_m)) + ml;
        sum = next;
      }
    w = w2;
    for (int i = 0; i <= 2 * w; ++i) {
      c[i] = t[i] + tl[i];
      cl[i] = (t[i] - c[i]) + tl[i];
    }
  }
  for (int i = 0; i <= 2 * w; ++i) p->ck[i] = c[i];
  fx_prepare(p->ck, 2 * w + 1, &p->fck, cl);
}

cudaError_t launch_sync_rhs(const StepParams &p, const double *u, double *out, cudaStream_t st) {
  StepParams q = p;
  q.use_pe[0] = q.use_pe[1] = q.use_pe[2] = 0;  // no PE boundary: central differences at every point
  const bool grouped = grouped_shape(q, u) && (reinterpret_cast<uintptr_t>(out) % 16) == 0;
  const int64_t work = grouped ? q.ntot / 4 : q.ntot;
  const int64_t b = (work + 255) / 256, cap = (int64_t)sm_count() * 8;
  const int blocks = (int)(b < cap ? b : cap);
  const int g = grouped ? 1 : 0;
  if (q.dim == 1) {
    if (q.h == 1) sync_rhs_kernel<1, 1><<<blocks, 256, 0, st>>>(q, u, out, g);
    else if (q.h == 2) sync_rhs_kernel<1, 2><<<blocks, 256, 0, st>>>(q, u, out, g);
    else sync_rhs_kernel<1, 3><<<blocks, 256, 0, st>>>(q, u, out, g);
  } else {
    if (q.h == 1) sync_rhs_kernel<3, 1><<<blocks, 256, 0, st>>>(q, u, out, g);
    else if (q.h == 2) sync_rhs_kernel<3, 2><<<blocks, 256, 0, st>>>(q, u, out, g);
    else sync_rhs_kernel<3, 3><<<blocks, 256, 0, st>>>(q, u, out, g);
  }
  return cudaGetLastError();
}
