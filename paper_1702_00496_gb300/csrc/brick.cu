// brick.cu -- the 3D step in block fixed point, marched along z through tiles of one PE.
//
// A 3D point is a contraction of 1 + 6 h constant taps (13 at order 4), which the FP64 pipe bounded at a tenth of the
// memory bandwidth (13 DFMA of 16 SM clocks per warp).  Here the taps are integer multiply-adds (fixed.cuh), and every
// value is converted once per tile instead of once per tap:
//
//  - A block owns a tile of up to 32 x cells by 128 / (groups of four per row) rows of one PE and marches it along z
//    through a chunk of planes.  The planes z-h .. z+h lie in shared memory as fixed-point pairs (8 bytes per cell, a
//    ring of 2 h + 2 planes), each with the h cells around the tile that its stencil reaches.
//  - Where the tile meets a face of its PE, the cells beyond are buffer points: they are extrapolated over the delayed
//    levels (FP64, as everywhere) once per tile when their plane is loaded, with that side's delay.
//  - One scale serves the planes of the ring.  A plane whose largest value exceeds it, or a ring that has fallen two
//    bits below it, rescales the ring (a shift of every entry: rare, fields change little from plane to plane).  Planes cut
//    at a scale that has fallen since lack the digits between: their values must be as much larger, and beyond kFxLift such
//    bits they are not used (fixed.cuh, FxRing).
//  - One barrier per plane: iteration i sums output plane i-2-h from planes the ring already holds (while the loads of
//    plane i are in flight), publishes plane i's largest value, and after the barrier stores plane i.
//  - A thread sums four x-consecutive points.  A group with a half more than kBrickGuard bits below the scale (where the
//    field changes sign along two axes at once, or falls steeply) is left to its FP64 chain, as is every group of a plane
//    near infinities, NaN or values at the ends of the exponent range.  The march lists them, and a second launch does them.
//
// The backward sweep of the gradient runs on the same tiles: the transposed step's level-n part (taps reversed, cells
// across a face counted only at delay 0), the alpha term (second-derivative taps of U^n times lambda, summed), and a
// small kernel for what the cells at the faces send to older levels.  256^3 in 4^3 PEs, order 4: 1.01 -> 0.63 ms per
// backward step with the alpha term, 0.52 -> 0.37 ms without.
//
// What bounds it: latency.  A block's plane is a chain of loads, the largest value, a barrier, conversions and shared-memory
// round trips, and the ring leaves 16 warps per SM to hide it: issue 42 % active, the busiest pipe 39 %, DRAM 2.2 TB/s at
// order 4.  512^3 in 8^3 PEs, L = 3 on GB300: order 4 3.51 -> 1.53 ms per step, order 2 1.83 -> 1.0 ms; 256^3 in 4^3 PEs 438 ->
// 248 and 235 -> 175 us, the second launch (10 us) included.
#include <cmath>

#include "stencil.cuh"

namespace {

using namespace atfd;

// Tiles of 32 x 16 cells in blocks of 128 threads, four blocks per SM (128 registers, 54 KB of ring at order 4): blocks of
// 256 threads on 64 x 16 cells read 5 % fewer halo cells but wait longer at their barrier (512^3, order 4: 1.70 against
// 1.62 ms; order 2: 1.12 against 1.03).
constexpr int kBrickThreads = 128;
constexpr int kBrickX = 32;
constexpr int kBrickBlocks = 4;
constexpr int kBrickWarps = kBrickThreads / 32;  // words of a plane's listed groups
constexpr int kBrickGuard = 10;  // bits below the scale that one of two x neighbours must be within
constexpr int kCore = 4;         // values of the tile's own cells a thread loads per plane
constexpr int kBrickSlots = 6;   // and with those around it

struct BrickShape {
  int32_t tx, gx, rows;            // cells and groups of four per tile row, rows per tile
  int32_t tiles_x, tiles_y;        // tiles per PE
  int32_t zc, chunks;              // planes per chunk, chunks per PE
  int32_t stride, plane;           // shared-memory slots per row (with padding) and per plane
  int32_t aligned;                 // groups start on 16 bytes and never straddle a PE: 16-byte stores, grouped chain
  int64_t blocks;
};

// What the backward step's passes read and write beside the step parameters.
struct BrickAdjoint {
  const double *src;    // MODE 1: the field the transposed taps act on (lambda^{n+1}, or mu); MODE 2: the same, as a factor
  const double *ident;  // MODE 1, Adams-Bashforth: lambda^{n+1}, which reaches lambda^n unchanged; else null
  double *cur;          // MODE 1: lambda^n
  double *fresh;        // MODE 1: the level this step initialises (zeros), or null
  double *g_blk;        // MODE 2: per-block sums of dJ/dalpha
  int32_t add;          // MODE 1: add to cur (else set it)
};

// A tile.  The march keeps it in shared memory (registers are what it has least of).
struct BrickTile {
  int32_t pidx[3], x0, y0, zs, ze, xlen, ylen;  // its PE, its first cell, its planes zs .. ze - 1, its cells per plane
  int32_t lo[3], hi[3];                         // the cells lo .. hi - 1 of its PE along each axis
  int32_t k[3][2];  // delays of the PE's sides; transposed: of the neighbours' sides that read this PE's cells
};

__device__ __forceinline__ void tile_place(const StepParams &p, const BrickShape &b, int t, BrickTile *T) {
  // x fastest, then y, then chunk, then PE
  const int tx = t % b.tiles_x; t /= b.tiles_x;
  const int ty = t % b.tiles_y; t /= b.tiles_y;
  const int ch = t % b.chunks; t /= b.chunks;
  T->pidx[0] = t % p.pe[0]; t /= p.pe[0];
  T->pidx[1] = t % p.pe[1];
  T->pidx[2] = t / p.pe[1];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    T->lo[a] = T->pidx[a] * p.S[a];
    T->hi[a] = T->lo[a] + p.S[a];
  }
  T->x0 = T->lo[0] + tx * b.tx;
  T->y0 = T->lo[1] + ty * b.rows;
  T->zs = T->lo[2] + ch * b.zc;
  T->ze = min(T->zs + b.zc, T->hi[2]);
  T->xlen = min(b.tx, T->hi[0] - T->x0);
  T->ylen = min(b.rows, T->hi[1] - T->y0);
}

template <int MODE>
__device__ __forceinline__ void tile_delays(const StepParams &p, const uint8_t *keff, BrickTile *T) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    int lo[3] = {T->pidx[0], T->pidx[1], T->pidx[2]}, hi[3] = {T->pidx[0], T->pidx[1], T->pidx[2]};
    if (MODE == 1) {
      lo[a] = lo[a] == 0 ? p.pe[a] - 1 : lo[a] - 1;
      hi[a] = hi[a] + 1 == p.pe[a] ? 0 : hi[a] + 1;
    }
    T->k[a][0] = p.use_pe[a] ? keff[side_of<3>(p, lo, a, MODE == 1 ? 1 : 0)] : 0;
    T->k[a][1] = p.use_pe[a] ? keff[side_of<3>(p, hi, a, MODE == 1 ? 0 : 1)] : 0;
  }
}

// A thread's share of a plane's cells: kCore slots of the tile's own cells, row by row, then the cells around it -- left and
// right of the rows, then below and above them -- so that the buffer points, which cost T FP64 operations each, fill few
// warps.
template <int H, int MODE>
struct TileLoad {
  int goff[kBrickSlots], code[kBrickSlots];  // cell within the plane; slot in the ring plane and delay
  bool some;                                 // the warp has buffer points with a delay beside the tile
  double v[kBrickSlots], hlev[kBrickSlots - kCore][H + 1];

  __device__ __forceinline__ void setup(const StepParams &p, const BrickShape &b, const BrickTile &T, int tid) {
    const int xlen = T.xlen, ylen = T.ylen;
    bool buffers = false;
#pragma unroll
    for (int s = 0; s < kBrickSlots; ++s) {
      int r, c, k = 0;
      bool have;
      if (s < kCore) {
        const int l = tid + s * kBrickThreads;
        have = l < ylen * xlen;
        r = l / xlen;
        c = l - r * xlen;
      } else {
        const int l = tid + (s - kCore) * kBrickThreads, side = 2 * H * ylen;
        have = l < side + 2 * H * xlen;
        if (l < side) {
          const int hi = l >= H * ylen, m = l - hi * H * ylen;
          r = m / H;
          c = m - r * H + (hi ? xlen : -H);
          if (hi ? T.x0 + c >= T.hi[0] : T.x0 + c < T.lo[0]) k = T.k[0][hi];
        } else {
          const int hi = l - side >= H * xlen, m = l - side - hi * H * xlen;
          r = m / xlen;
          c = m - r * xlen;
          r += hi ? ylen : -H;
          if (hi ? T.y0 + r >= T.hi[1] : T.y0 + r < T.lo[1]) k = T.k[1][hi];
        }
      }
      const int cc = c + 4;  // columns -4 .. : group boundaries stay multiples of four
      goff[s] = have ? wrap_coord(T.y0 + r, p.n[1]) * p.n[0] + wrap_coord(T.x0 + c, p.n[0]) : T.y0 * p.n[0] + T.x0;
      code[s] = have ? ((r + H) * b.stride + cc + (cc >> 2)) | (k << 16) : b.plane - 1;  // a pad slot nobody reads
      buffers = buffers || (have && k > 0);
    }
    some = __any_sync(0xffffffffu, buffers);
  }

  // Plane zz's values; of buffer points, levels n-k-m: fetched with the plane and combined after the sums in between.  A warp
  // with a buffer point does it for all its halo slots (delay 0: level n, not used) without branches.
  __device__ __forceinline__ void load(const StepParams &p, const double *__restrict__ un, int sn, int zz) {
    const int64_t base = (int64_t)wrap_coord(zz, p.n[2]) * ((int64_t)p.n[0] * p.n[1]);
    const double *src = un + base;
#pragma unroll
    for (int s = 0; s < kBrickSlots; ++s) v[s] = LdgNC::ld(src + goff[s]);
    if (MODE != 1 && some) {
#pragma unroll
      for (int s = kCore; s < kBrickSlots; ++s) {
        const int k = code[s] >> 16;
        const double *h = p.ring + base + goff[s];
        hlev[s - kCore][0] = LdgNC::ld(h + slot_back(sn, k, p.R) * p.ntot);
        if (p.T > 1) {  // the time-expanded rows read H + 1 levels, the others one
#pragma unroll
          for (int m = 1; m <= H; ++m) hlev[s - kCore][m] = LdgNC::ld(h + slot_back(sn, k > 0 ? k + m : 0, p.R) * p.ntot);
        }
      }
    }
  }

  __device__ __forceinline__ void extrapolate(const StepParams &p, const BrickTile &T, int sn, int zz) {
    const int kz = zz < T.lo[2] ? T.k[2][0] : (zz >= T.hi[2] ? T.k[2][1] : 0);
    if (MODE == 1) {  // what lies across a face with a delay goes to older levels (brick_faces_kernel)
#pragma unroll
      for (int s = 0; s < kBrickSlots; ++s)
        if (s < kCore ? kz > 0 : (code[s] >> 16) > 0) v[s] = 0.0;
    } else if (kz > 0) {  // a buffer plane: only the tile's own cells of it are read
      const int64_t base = (int64_t)wrap_coord(zz, p.n[2]) * ((int64_t)p.n[0] * p.n[1]);
#pragma unroll
      for (int s = 0; s < kCore; ++s) v[s] = halo_value<LdgNC>(p, base + goff[s], sn, kz);
    } else if (some) {
#pragma unroll
      for (int s = kCore; s < kBrickSlots; ++s) {
        const int k = code[s] >> 16;  // halo_value's chain
        double acc = fma(p.w[k][0], hlev[s - kCore][0], p.zero);
        if (p.T > 1) {
#pragma unroll
          for (int m = 1; m <= H; ++m) acc = fma(p.w[k][m], hlev[s - kCore][m], acc);
        }
        v[s] = k > 0 ? acc : v[s];
      }
    }
  }
};

// Four sums in fixed point: the taps in f3's order.
template <int H>
struct TileSums {
  int64_t A[4], B[4], C[4];
  __device__ __forceinline__ void centre(const FxTaps<6 * AT_MAX_H + 1> &t, int q, const int2 &f) {
    A[q] = (int64_t)t.w1[0] * f.x;
    B[q] = fx_mad(t.w1[0], f.y, kFxB0);
    C[q] = fx_mad(t.w0[0], f.x, kFxC0);
  }
  __device__ __forceinline__ void tap(const FxTaps<6 * AT_MAX_H + 1> &t, int k, int q, const int2 &f) {
    A[q] = fx_mad(t.w1[k], f.x, A[q]);
    B[q] = fx_mad(t.w1[k], f.y, B[q]);
    C[q] = fx_mad(t.w0[k], f.x, C[q]);
  }
  __device__ __forceinline__ void join() {
#pragma unroll
    for (int q = 0; q < 4; ++q) A[q] = fx_join(A[q], B[q], C[q]);
  }
};
__device__ __forceinline__ constexpr int tile_tap(int h, int a, int j) {  // f3's index of offset j != 0 of axis a
  return 1 + 2 * h * a + (j < 0 ? j + h : j + h - 1);
}

// What becomes of the `valid` sums r of the points from i0: Adams-Bashforth's combination and the store, the transposed
// step's, or (MODE 2) the sum galpha.
template <int AB, int MODE>
__device__ __forceinline__ void tile_finish(const StepParams &p, const BrickAdjoint &adj, bool aligned,
                                            const double *__restrict__ un, double *__restrict__ out, int64_t n, int64_t i0,
                                            int valid, double r[4], const AbLevels<1> old[4], double &galpha) {
  if (MODE == 2) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q < valid) galpha = fma(LdgNC::ld(adj.src + i0 + q), r[q], galpha);
    return;
  }
  if (MODE == 1 && aligned) {  // the workspace is 16-byte aligned
    double2 *o = reinterpret_cast<double2 *>(out + i0);
    double2 lo = make_double2(r[0], r[1]), hi = make_double2(r[2], r[3]);
    if (adj.ident) {
      const double2 a = LdgNC::ld2(adj.ident + i0), c = LdgNC::ld2(adj.ident + i0 + 2);
      lo.x += a.x; lo.y += a.y; hi.x += c.x; hi.y += c.y;
    }
    if (adj.add) {
      const double2 a = o[0], c = o[1];
      lo.x += a.x; lo.y += a.y; hi.x += c.x; hi.y += c.y;
    }
    o[0] = lo;
    o[1] = hi;
    if (adj.fresh) {
      double2 *z = reinterpret_cast<double2 *>(adj.fresh + i0);
      z[0] = z[1] = make_double2(0.0, 0.0);
    }
    return;
  }
  if (MODE == 1) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (q >= valid) continue;
      if (adj.ident) r[q] += LdgNC::ld(adj.ident + i0 + q);
      out[i0 + q] = adj.add ? out[i0 + q] + r[q] : r[q];
      if (adj.fresh) adj.fresh[i0 + q] = 0.0;
    }
    return;
  }
  if (AB) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (q >= valid) continue;
      const double u[1] = {LdgNC::ld(un + i0 + q)};
      ab_combine<1>(p, n, i0 + q, u, r + q, old[q]);
    }
  }
  if (aligned) {
    reinterpret_cast<double2 *>(out + i0)[0] = make_double2(r[0], r[1]);
    reinterpret_cast<double2 *>(out + i0)[1] = make_double2(r[2], r[3]);
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q < valid) out[i0 + q] = r[q];
  }
}

// The first `valid` points of a group as FMA chains: the centre, then the taps of x, y and z in offset order, across a face
// with a delay the halo value (MODE 1: nothing, such a tap goes to older levels).  An axis' values are all in flight before
// the first is used; r[q] of the points that are not there is any.
template <int H, int MODE>
__device__ __forceinline__ void tile_chain(const StepParams &p, const BrickTile &T, const double *__restrict__ un, int sn,
                                           bool aligned, const int c[3], int valid, double r[4]) {
  const int64_t nxy = (int64_t)p.n[0] * p.n[1], i = c[2] * nxy + (int64_t)c[1] * p.n[0] + c[0];
  auto four = [&](int64_t cell, double v[4]) {
    if (aligned) {
      const double2 a = LdgNC::ld2(un + cell), b = LdgNC::ld2(un + cell + 2);
      v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) v[q] = LdgNC::ld(un + cell + (q < valid ? q : 0));
    }
  };
  auto across = [&](int a, int at) { return at < T.lo[a] ? T.k[a][0] : (at >= T.hi[a] ? T.k[a][1] : 0); };
  auto halo = [&](int64_t cell, int k) { return MODE == 1 ? 0.0 : halo_value<LdgNC>(p, cell, sn, k); };
  {
    double v[4 + 2 * H];
    four(i, v + H);
#pragma unroll
    for (int m = 0; m < 2 * H; ++m) {  // the cells beside the valid points
      const int at = c[0] + (m < H ? m - H : valid + m - H), k = across(0, at);
      const int64_t cell = i + (wrap_coord(at, p.n[0]) - c[0]);
      double x = LdgNC::ld(un + cell);
      if (k > 0) x = halo(cell, k);
      if (m < H) {
        v[m] = x;
      } else {
        if (valid == 4) v[4 + m] = x;
#pragma unroll
        for (int q = 1; q < 4; ++q)
          if (q == valid) v[q + m] = x;
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      double acc = fma(p.s0, v[q + H], p.zero);
#pragma unroll
      for (int j = -H; j <= H; ++j)
        if (j != 0) acc = fma(p.s[0][j + H], v[q + j + H], acc);
      r[q] = acc;
    }
  }
#pragma unroll
  for (int a = 1; a < 3; ++a) {
    const int64_t step = a == 1 ? (int64_t)p.n[0] : nxy;
    auto cell = [&](int m) {
      const int j = m < H ? m - H : m - H + 1;
      return i + (int64_t)(wrap_coord(c[a] + j, p.n[a]) - c[a]) * step;
    };
    double v[2 * H][4];
#pragma unroll
    for (int m = 0; m < 2 * H; ++m) four(cell(m), v[m]);
    if (c[a] - H < T.lo[a] || c[a] + H >= T.hi[a]) {
#pragma unroll
      for (int m = 0; m < 2 * H; ++m) {
        const int k = across(a, c[a] + (m < H ? m - H : m - H + 1));
        if (k > 0) {
#pragma unroll
          for (int q = 0; q < 4; ++q) v[m][q] = halo(cell(m) + (q < valid ? q : 0), k);
        }
      }
    }
#pragma unroll
    for (int m = 0; m < 2 * H; ++m)
#pragma unroll
      for (int q = 0; q < 4; ++q) r[q] = fma(p.s[a][m < H ? m : m + 1], v[m][q], r[q]);
  }
}

// One point in the same way, with all of its values in flight together: few listed groups are waited for, not worked on.
template <int H, int MODE>
__device__ __forceinline__ double tile_point(const StepParams &p, const BrickTile &T, const double *__restrict__ un, int sn,
                                             const int c[3]) {
  const int64_t stride[3] = {1, (int64_t)p.n[0], (int64_t)p.n[0] * p.n[1]};
  const int64_t i = c[2] * stride[2] + c[1] * stride[1] + c[0];
  auto cell = [&](int a, int j) { return i + (int64_t)(wrap_coord(c[a] + j, p.n[a]) - c[a]) * stride[a]; };
  double v[3][2 * H];
  const double u = LdgNC::ld(un + i);
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int m = 0; m < 2 * H; ++m) v[a][m] = LdgNC::ld(un + cell(a, m < H ? m - H : m - H + 1));
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (c[a] - H >= T.lo[a] && c[a] + H < T.hi[a]) continue;
#pragma unroll
    for (int m = 0; m < 2 * H; ++m) {
      const int j = m < H ? m - H : m - H + 1;
      const int k = c[a] + j < T.lo[a] ? T.k[a][0] : (c[a] + j >= T.hi[a] ? T.k[a][1] : 0);
      if (k > 0) v[a][m] = MODE == 1 ? 0.0 : halo_value<LdgNC>(p, cell(a, j), sn, k);
    }
  }
  double acc = fma(p.s0, u, p.zero);
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int m = 0; m < 2 * H; ++m) acc = fma(p.s[a][m < H ? m : m + 1], v[a][m], acc);
  return acc;
}

// *out += the block's sum of v, in a fixed order.
template <int THREADS>
__device__ __forceinline__ void block_total(double v, double *out) {
  __shared__ double sums[THREADS / 32];
  for (int d = 16; d > 0; d >>= 1) v += __shfl_down_sync(0xffffffffu, v, d);
  if ((threadIdx.x & 31) == 0) sums[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = sums[0];
    for (int w = 1; w < THREADS / 32; ++w) t += sums[w];
    *out += t;
  }
}

// MODE 0: the forward step.  MODE 1: the part of the transposed step that stays at level n, with the taps reversed; a
// buffer point counts only where the neighbour's side that reads across has delay 0.  MODE 2: the alpha term's sum of
// lambda x (the second-derivative taps of U^n), for which p.s0, p.s and p.f3 hold those taps; each block takes the same
// tiles in the same order, so the sum is deterministic.
template <int H, int AB, int MODE>
__global__ void __launch_bounds__(kBrickThreads, kBrickBlocks) brick_kernel(const __grid_constant__ StepParams p,
                                                                            const __grid_constant__ BrickShape b,
                                                                            const __grid_constant__ BrickAdjoint adj, const int64_t n_off,
                                                                            const int64_t *n_base) {
  constexpr int NR = 2 * H + 2;  // ring planes
  extern __shared__ int2 ring[];
  __shared__ int mx[3];
  __shared__ BrickTile T;
  __shared__ FxPlanes planes;
  const int64_t n = n_off + (n_base ? *n_base : 0);
  const double *__restrict__ un = MODE == 1 ? adj.src : p.ring + slot_of(n, p.R) * p.ntot;
  double *__restrict__ out = MODE == 1 ? adj.cur : p.ring + slot_of(n + 1, p.R) * p.ntot;
  const uint8_t *keff = p.keff + (n & 1) * p.nb;
  const int tid = threadIdx.x;
  if (MODE == 0) {
    draw_sides(p, n + 1, (int64_t)blockIdx.x * kBrickThreads + tid, (int64_t)gridDim.x * kBrickThreads,
               p.keff + ((n + 1) & 1) * p.nb);
  } else if (MODE == 1 && n >= 1) {
    draw_sides(p, n - 1, (int64_t)blockIdx.x * kBrickThreads + tid, (int64_t)gridDim.x * kBrickThreads,
               p.keff + ((n - 1) & 1) * p.nb);
  }
  double galpha = 0.0;
  const int sn = (int)slot_of(n, p.R), lane = tid & 31, warp = tid >> 5;
  const bool aligned = b.aligned != 0;
  for (int tile = (int)blockIdx.x; tile < (int)b.blocks; tile += (int)gridDim.x) {
  if (tid == 0) {
    tile_place(p, b, tile, &T);
    tile_delays<MODE>(p, keff, &T);
  }
  if (tid < 3) mx[tid] = 0;
  if (tid < 8) planes.top[tid] = planes.cut[tid] = 0;
  __syncthreads();
  TileLoad<H, MODE> in;
  in.setup(p, b, T, tid);
  FxRing scale;
  // this thread's points; a thread without any sums the tile's first group along
  const int row = tid / b.gx, grp = tid - row * b.gx;
  const bool mine = row < T.ylen && 4 * grp < T.xlen;
  const int nv = min(4, mine ? T.xlen - 4 * grp : 4);
  const int col = mine ? (row + H) * b.stride + 5 * grp + 5 : H * b.stride + 5;  // its slot in a ring plane (pad slot per four)
  const int64_t cell0 = (int64_t)(T.y0 + (mine ? row : 0)) * p.n[0] + T.x0 + (mine ? 4 * grp : 0);
  const int64_t nxy = (int64_t)p.n[0] * p.n[1];
  const int zs = T.zs, ze = T.ze;
  int heavy = 0;  // planes in a row with most groups listed
  in.load(p, un, sn, zs - H);
  int wslot = 0, cslot = 0, m3 = 0;  // ring slots of plane i and of plane o - H of the output; i - (zs - H) mod 3
  for (int i = zs - H; i < ze + H + 2; ++i) {
    const int o = i - 2 - H;
    bool list = false;
    if (o >= zs) {
      const int64_t i0 = (int64_t)o * nxy + cell0;
      AbLevels<1> old[4];
      if (AB) {
#pragma unroll
        for (int q = 0; q < 4; ++q) ab_fetch<1>(p, n, i0 + (q < nv ? q : 0), old[q]);
      }
      // planes o-H .. o+H lie in ring slots cslot, cslot + 1 ..
      const int2 *pl[2 * H + 1];
#pragma unroll
      for (int d = 0; d <= 2 * H; ++d) pl[d] = ring + (cslot + d >= NR ? cslot + d - NR : cslot + d) * b.plane + col;
      const int E = scale.E, lift = fx_ring_lift(scale, planes, o, H);
      const bool usable = lift <= kFxLift;
      double r[4] = {0.0, 0.0, 0.0, 0.0};
      bool far = false;
      if (usable && E >= 0) {  // the same for the whole block; E < 0: every plane so far is zero
        const int2 *mid = pl[H];
        int2 c4[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) c4[q] = mid[q];
        {
          const uint32_t g0 = fx_upper(c4[0].x) | fx_upper(c4[1].x);
          const uint32_t g1 = nv < 3 ? g0 : fx_upper(c4[2].x) | fx_upper(c4[3].x);
          far = min(g0, g1) < fx_least(kBrickGuard, lift);
        }
        const FxTaps<6 * AT_MAX_H + 1> &t = p.f3;
        TileSums<H> sum;
#pragma unroll
        for (int q = 0; q < 4; ++q) sum.centre(t, q, c4[q]);
        // x: cells -H .. 3 + H of the row; the pad slots lie before cells 0 and 4
#pragma unroll
        for (int d = -H; d <= 3 + H; ++d) {
          const int2 f = d >= 0 && d < 4 ? c4[d & 3] : mid[d < 0 ? d - 1 : d + 1];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int j = d - q;  // tap j of point q reads cell q + j
            if (j != 0 && j >= -H && j <= H) sum.tap(t, tile_tap(H, 0, j), q, f);
          }
        }
#pragma unroll
        for (int j = -H; j <= H; ++j) {
          if (j == 0) continue;
          const int2 *s = mid + j * b.stride;
#pragma unroll
          for (int q = 0; q < 4; ++q) sum.tap(t, tile_tap(H, 1, j), q, s[q]);
        }
#pragma unroll
        for (int j = -H; j <= H; ++j) {
          if (j == 0) continue;
#pragma unroll
          for (int q = 0; q < 4; ++q) sum.tap(t, tile_tap(H, 2, j), q, pl[H + j][q]);
        }
        sum.join();
        const int ex = E - 1023 - p.f3.sw;
        if (AB) {
#pragma unroll
          for (int q = 0; q < 4; ++q) r[q] = fx_to_any(sum.A[q], ex);
        } else {
          fx_results<4>(sum.A, ex, r);
        }
      }
      list = mine && (far || !usable);
      uint32_t who = __ballot_sync(0xffffffffu, list);
      if (who != 0) {
        int top = usable ? 0 : 1;  // sums of zeros are zero (a plane that is not usable has no top either)
#pragma unroll
        for (int q = o - H; q <= o + H; ++q) top |= planes.top[q & 7];
        if (top == 0) {
          who = 0;
          list = false;
          r[0] = r[1] = r[2] = r[3] = 0.0;
        }
      }
      if (lane == 0) p.listed[(tile * b.zc + (o - zs)) * kBrickWarps + warp] = who;
      if (mine && !list) tile_finish<AB, MODE>(p, adj, aligned, un, out, n, i0, nv, r, old, galpha);
      cslot = cslot + 1 == NR ? 0 : cslot + 1;
    }
    if (i < ze + H) {
      in.extrapolate(p, T, sn, i);
      int mag = 0, low = 0;
#pragma unroll
      for (int s = 0; s < kBrickSlots; ++s) {
        mag = max(mag, fx_mag(in.v[s]));
        low |= fx_word(in.v[s], 0);
      }
      mag = __reduce_max_sync(0xffffffffu, max(mag, low != 0 ? 1 : 0));
      if ((tid & 31) == 0) atomicMax(&mx[m3], mag);
    }
    const int count = __syncthreads_count(list);
    // a steep tile, not the planes around a fall of the scale: the rest of it is listed at once
    heavy = 2 * count > T.ylen * ((T.xlen + 3) >> 2) ? heavy + (o - H > scale.until ? 3 : 1) : 0;
    if (heavy >= 9) {
      const uint32_t all = __ballot_sync(0xffffffffu, mine);
      for (int z = o + 1 + lane; z < ze; z += 32) p.listed[(tile * b.zc + (z - zs)) * kBrickWarps + warp] = all;
      break;
    }
    if (i >= ze + H) continue;
    const int m = mx[m3];
    if (tid == 0) mx[m3 == 0 ? 2 : m3 - 1] = 0;  // read by all before this barrier, used again two planes on
    const bool ok = fx_plane_usable(m);
    const int top = ok ? m >> 20 : 0, d = fx_ring_join(scale, planes, i, top, H, ok);
    if (tid == 0) fx_ring_note(planes, scale, i, top, d, ok);  // of planes that no output reads before the next barrier
    if (d != 0) {
      for (int e = tid; e < NR * b.plane; e += kBrickThreads) {
        const int2 f = ring[e];
        const Fx g = fx_split(fx_rescale((int64_t)f.x * 4294967296ll + f.y, d));
        ring[e] = make_int2(g.hi, g.lo);
      }
      __syncthreads();
    }
    if (ok) {  // a zero plane, or one before the first scale: the scale is any, the values come out 0 (-1 for -0)
      int2 *dst = ring + wslot * b.plane;
#pragma unroll
      for (int s = 0; s < kBrickSlots; ++s) {
        const Fx f = fx_split(fx_from(in.v[s], scale.E));
        dst[in.code[s] & 0xffff] = make_int2(f.hi, f.lo);
      }
    }
    wslot = wslot + 1 == NR ? 0 : wslot + 1;
    m3 = m3 == 2 ? 0 : m3 + 1;
    if (i + 1 < ze + H) in.load(p, un, sn, i + 1);
  }
  __syncthreads();
  }
  if (MODE == 2) block_total<kBrickThreads>(galpha, adj.g_blk + blockIdx.x);
}

// The groups that the march listed (a bit per group, four words per plane of a tile, every word written anew), as FMA
// chains.  A block takes up to kListWords words, every gridDim.x-th one (tiles with many listed groups are spread), makes a
// list of their groups in shared memory -- those away from the PE's faces from its front, those at a face, for which a warp
// reads delayed levels, from its end -- and shares it out.  A launch of its own, started while the march ends: the march's
// blocks have next to no L1 beside the ring and no registers to spare, a few of them hold most of a field's listed groups,
// and past what they could list they held their barriers for the chains.  256^3 in 4^3 PEs, us per step (order 4 / 2; all
// FP64 chains 438 / 235): a Gaussian of 13 cells 830 / 465 -> 637 / 372, a ball of ones in zeros 607 / 332 -> 228 / 149, noise
// with spikes 832 / 457 -> 542 / 297; a field that is zero in half of the box 645 / 357 -> 287 / 198; smooth fields, with 0.7 %
// (0.5 %) of their groups listed, pay for it (226 -> 248, 160 -> 175).
constexpr int kListThreads = 256;
constexpr int kListWords = 512;  // 32 KB of list

template <int H, int AB, int MODE>
__global__ void __launch_bounds__(kListThreads, 2) brick_listed_kernel(const StepParams p, const BrickShape b,
                                                                       const BrickAdjoint adj,
                                                                       const int64_t n_off, const int64_t *n_base) {
  __shared__ uint16_t list[kListWords * 32];
  __shared__ uint32_t sums[kListThreads / 32];
  cudaGridDependencySynchronize();
  const int64_t n = n_off + (n_base ? *n_base : 0);
  const int sn = (int)slot_of(n, p.R);
  const double *__restrict__ un = MODE == 1 ? adj.src : p.ring + sn * p.ntot;
  double *__restrict__ out = MODE == 1 ? adj.cur : p.ring + slot_of(n + 1, p.R) * p.ntot;
  const uint8_t *keff = p.keff + (n & 1) * p.nb;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, per_tile = b.zc * kBrickWarps;
  const int words = (int)b.blocks * per_tile;
  double galpha = 0.0;
  for (int w0 = (int)blockIdx.x; w0 < words; w0 += (int)gridDim.x * kListWords) {
    // this thread's words: their groups away from faces and at faces
    constexpr int W = kListWords / kListThreads;
    uint32_t inner[W], face[W], count = 0;  // count: low half away from faces, high half at faces
#pragma unroll
    for (int v = 0; v < W; ++v) {
      const int64_t at = w0 + (int64_t)(tid * W + v) * gridDim.x;
      const int w = (int)at;
      inner[v] = at < words ? p.listed[w] : 0u;
      face[v] = 0u;
      if (inner[v] != 0) {
        BrickTile T;
        tile_place(p, b, w / per_tile, &T);
        const int k = w % per_tile, z = T.zs + k / kBrickWarps;
        if (z >= T.ze) inner[v] = 0;  // planes that a PE's last chunk has not: their words are not written
        for (uint32_t left = inner[v]; left != 0; left &= left - 1) {
          const int bit = __ffs(left) - 1, t = k % kBrickWarps * 32 + bit, row = t / b.gx;
          const int x = T.x0 + 4 * (t - row * b.gx), y = T.y0 + row;
          if (x - H < T.lo[0] || x + 3 + H >= T.hi[0] || y - H < T.lo[1] || y + H >= T.hi[1] || z - H < T.lo[2] || z + H >= T.hi[2])
            face[v] |= 1u << bit;
        }
        inner[v] &= ~face[v];
      }
      count += __popc(inner[v]) | __popc(face[v]) << 16;
    }
    uint32_t upto = count;
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, upto, d);
      if (lane >= d) upto += v;
    }
    if (lane == 31) sums[warp] = upto;
    __syncthreads();
    uint32_t all = 0, before = upto - count;
    for (int q = 0; q < kListThreads / 32; ++q) {
      if (q < warp) before += sums[q];
      all += sums[q];
    }
    uint32_t front = before & 0xffff, back = kListWords * 32 - 1 - (before >> 16);
#pragma unroll
    for (int v = 0; v < W; ++v) {
      for (uint32_t left = inner[v]; left != 0; left &= left - 1)
        list[front++] = (uint16_t)((tid * W + v) << 5 | (__ffs(left) - 1));
      for (uint32_t left = face[v]; left != 0; left &= left - 1)
        list[back--] = (uint16_t)((tid * W + v) << 5 | (__ffs(left) - 1));
    }
    __syncthreads();
    // A group per thread, or, up to what keeps every thread busy once or twice, a point; those at faces, which take longest,
    // first.
    const int n_inner = (int)(all & 0xffff), n_face = (int)(all >> 16), each = n_inner + n_face <= kListThreads / 2 ? 4 : 1;
    const int from = (n_face * each + 31) / 32 * 32;
#pragma unroll 1
    for (int e = tid; e < from + n_inner * each; e += kListThreads) {
      if (e >= n_face * each && e < from) continue;
      const int at = (e < from ? e : e - from) / each, entry = list[e < from ? kListWords * 32 - 1 - at : at];
      const int w = w0 + (entry >> 5) * (int)gridDim.x, k = w % per_tile;
      BrickTile T;
      tile_place(p, b, w / per_tile, &T);
      tile_delays<MODE>(p, keff, &T);
      const int t = k % kBrickWarps * 32 + (entry & 31), row = t / b.gx, g = t - row * b.gx;
      const int c[3] = {T.x0 + 4 * g + (each == 4 ? e & 3 : 0), T.y0 + row, T.zs + k / kBrickWarps};
      const int valid = each == 4 ? min(1, T.x0 + T.xlen - c[0]) : min(4, T.xlen - 4 * g);
      if (valid < 1) continue;
      const int64_t i = ((int64_t)c[2] * p.n[1] + c[1]) * p.n[0] + c[0];
      double r[4] = {0.0, 0.0, 0.0, 0.0};
      AbLevels<1> old[4];
      if (AB) {
#pragma unroll
        for (int q = 0; q < 4; ++q) ab_fetch<1>(p, n, i + (q < valid ? q : 0), old[q]);
      }
      if (each == 4) r[0] = tile_point<H, MODE>(p, T, un, sn, c);
      else tile_chain<H, MODE>(p, T, un, sn, b.aligned != 0, c, valid, r);
      tile_finish<AB, MODE>(p, adj, each == 1 && b.aligned, un, out, n, i, valid, r, old, galpha);
    }
    __syncthreads();
  }
  if (MODE == 2) block_total<kListThreads>(galpha, adj.g_blk + blockIdx.x);
}

// The part of the transposed step that goes to older levels: a cell within h of a face whose far side's reader has delay
// k > 0 sends sum_j s_j lambda_{c-j} over the taps that cross, times w_m(k), to level n-k-m.  One thread per such cell
// (they are enumerated once each, face_cell), all its axes in turn.
// (A problem has fewer than 2^31 points: 32-bit divisions.)
struct FaceBoxes {
  uint32_t part_z, part_y, total;  // cells near a z face; near a y face but no z face; near an x face only
  uint32_t cs[3], cc[3];           // coordinates near a face and elsewhere, per axis
  int32_t hw[3];
};

__device__ __forceinline__ int near_face(const StepParams &p, int a, int hw, uint32_t t) {
  const uint32_t w = 2 * hw, pe = t / w;
  const int r = (int)(t - pe * w);
  return (int)pe * p.S[a] + (r < hw ? r : p.S[a] - (int)w + r);
}
__device__ __forceinline__ int off_face(const StepParams &p, int a, int hw, uint32_t t) {
  if (hw == 0) return (int)t;
  const uint32_t w = p.S[a] - 2 * hw, pe = t / w;
  return (int)(pe * (uint32_t)p.S[a] + hw + (t - pe * w));
}

template <int H>
__global__ void __launch_bounds__(256) brick_faces_kernel(const StepParams p, const FaceBoxes m, const double *__restrict__ src,
                                                          double *lam, const int Rl, const int64_t n) {
  const uint8_t *keff = p.keff + (n & 1) * p.nb;
  const int snl = (int)slot_of(n, Rl);
  const int64_t stride[3] = {1, (int64_t)p.n[0], (int64_t)p.n[0] * p.n[1]};
  const uint32_t nx = p.n[0], ny = p.n[1];
  for (uint32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < m.total; e += gridDim.x * blockDim.x) {
    int c[3];
    if (e < m.part_z) {
      const uint32_t row = e / nx, lay = row / ny;
      c[0] = (int)(e - row * nx);
      c[1] = (int)(row - lay * ny);
      c[2] = near_face(p, 2, m.hw[2], lay);
    } else if (e - m.part_z < m.part_y) {
      const uint32_t k = e - m.part_z, row = k / nx, lay = row / m.cs[1];
      c[0] = (int)(k - row * nx);
      c[1] = near_face(p, 1, m.hw[1], row - lay * m.cs[1]);
      c[2] = off_face(p, 2, m.hw[2], lay);
    } else {
      const uint32_t k = e - m.part_z - m.part_y, r = k / m.cs[0], lay = r / m.cc[1];
      c[0] = near_face(p, 0, m.hw[0], k - r * m.cs[0]);
      c[1] = off_face(p, 1, m.hw[1], r - lay * m.cc[1]);
      c[2] = off_face(p, 2, m.hw[2], lay);
    }
    const int64_t i = c[2] * stride[2] + c[1] * stride[1] + c[0];
    int pidx[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) pidx[a] = c[a] / p.S[a];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if (!p.use_pe[a]) continue;
      const int pos = c[a] - pidx[a] * p.S[a];
      const bool lower = pos < H;
      if (!lower && pos < p.S[a] - H) continue;
      int nb[3] = {pidx[0], pidx[1], pidx[2]};
      nb[a] = lower ? (pidx[a] == 0 ? p.pe[a] - 1 : pidx[a] - 1) : (pidx[a] + 1 == p.pe[a] ? 0 : pidx[a] + 1);
      const int k = keff[side_of<3>(p, nb, a, lower ? 1 : 0)];
      if (k == 0) continue;
      double x = 0.0;
#pragma unroll
      for (int j = -H; j <= H; ++j) {  // reversed taps: tap j reads c + j
        if (j == 0 || (pos + j >= 0 && pos + j < p.S[a])) continue;
        const int cj = wrap_coord(c[a] + j, p.n[a]);
        x = fma(p.s[a][j + H], LdgNC::ld(src + i + (int64_t)(cj - c[a]) * stride[a]), x);
      }
      for (int t = 0; t < p.T; ++t) {
        double *o = lam + slot_back(snl, k + t, Rl) * p.ntot + i;
        *o = fma(p.w[k][t], x, *o);
      }
    }
  }
}

int brick_sms() {
  int sms = 152, dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

// Tiles for the problem; false: too narrow PEs (rows of fewer than 16 cells, or tiles of fewer than 128 groups), whose
// threads would mostly idle or load halos.
bool brick_shape(const StepParams &p, BrickShape *b) {
  if (p.dim != 3 || p.scheme > AT_AT || !p.f3.ok || p.S[0] < 16) return false;
  // the tile that keeps most threads busy; among equals the one that reads fewest cells around it
  double best = 0.0;
  for (int gx = 4; gx <= kBrickX / 4; ++gx) {
    const int nt = (p.S[0] + 4 * gx - 1) / (4 * gx);
    int rows = kBrickThreads / gx;
    if (rows > p.S[1]) rows = p.S[1];
    const int ty = (p.S[1] + rows - 1) / rows;
    rows = (p.S[1] + ty - 1) / ty;
    if (2 * p.h * (rows + 4 * gx) > (kBrickSlots - kCore) * kBrickThreads) continue;
    const double busy = (double)p.S[0] * p.S[1] / ((double)nt * ty * 4 * kBrickThreads);
    const double cost = (1.0 + 0.1 * p.h * (rows + 4 * gx) / (2.0 * gx * rows)) / busy;
    if (best == 0.0 || cost < best) {
      best = cost;
      b->gx = gx;
      b->tx = 4 * gx;
      b->rows = rows;
      b->tiles_x = nt;
      b->tiles_y = ty;
    }
  }
  if (best == 0.0 || best > 2.0) return false;
  const int cols = b->tx + 8;                    // columns -4 .. tx + 3; the last slot of a row is a pad slot
  b->stride = cols + cols / 4;
  while (b->gx == 8 && b->stride % 16 != 8) ++b->stride;  // two rows of eight groups take all banks
  b->plane = (b->rows + 2 * p.h) * b->stride;
  if (b->plane >= 65536 || p.S[2] > 32767) return false;
  // Planes per chunk, and whether to take this kernel at all.  A block's iteration (one plane) takes kIter whether one or
  // four blocks share the SM -- it is a chain of shared-memory round trips, conversions and a barrier -- so a launch
  // takes as many of them as it has waves times planes, 2 h + 2 of which only fill the ring, and 5 us for the launch after
  // it.  At order 6 tiles that meet three faces, with T = 4 levels each, take 6 us per plane.  The grouped kernel (or the
  // per-point one, for shapes without groups of four) does one FP64 operation per tap and 17 % more for the halo, at 1.6
  // (1.0) lanes per SM and clock; Adams-Bashforth costs it 1.8 (1.4) times that and more, a tile's iteration 1.4 times.
  // us per step, tiles against groups or points, where the line lies: order 2, 128^3 in 2^3 PEs 37 against 35, 192 x 192 x 64
  // in 4 x 4 x 1 43 against 38, 150 x 126 x 90 in 3 x 3 x 2 (points) 43 against 43, 160^3 in 2^3 60 against 62, 200 x 168 x 140
  // in 4^3 (points) 85 against 115; order 4, 128^3 51 against 69, 100^3 in 5^3 43 in groups; order 2 with AB2, 128^3 50
  // against 65, 192 x 192 x 64 63 against 92.
  const bool grouped = p.n[0] % 4 == 0 && p.S[0] % 4 == 0, multi = p.ts > 1;
  const bool narrow = p.h == 3 && ((p.use_pe[0] && p.S[0] < 40) || (p.use_pe[1] && p.S[1] < 40));
  const double kIter[4] = {0.0, 2.7e-6, 3.4e-6, narrow ? 6e-6 : 3.0e-6}, clock = 2.07e9;
  const double iteration = kIter[p.h] * (multi ? 1.4 : 1.0), chains = !multi ? 1.0 : (grouped ? 1.8 : 1.4);
  const int sms = brick_sms(), bytes = (2 * p.h + 2) * b->plane * 8 + 4096;
  int resident = 227 * 1024 / bytes;
  if (resident > kBrickBlocks) resident = kBrickBlocks;
  if (resident < 1) return false;
  const int64_t columns = (int64_t)b->tiles_x * b->tiles_y * p.pe[0] * p.pe[1] * p.pe[2];
  double least = 0.0;
  for (int chunks = 1; chunks <= p.S[2] && chunks <= 64; ++chunks) {
    const int zc = (p.S[2] + chunks - 1) / chunks;
    const double fill = (double)(columns * ((p.S[2] + zc - 1) / zc)) / (sms * resident);
    const double waves = fill <= 3.0 ? std::ceil(fill) : fill + 0.5;
    const double t = waves * (zc + 2 * p.h + 2) * iteration;
    if (least == 0.0 || t < least) {
      least = t;
      b->zc = zc;
    }
  }
  b->chunks = (p.S[2] + b->zc - 1) / b->zc;
  b->blocks = columns * b->chunks;
  if (5e-6 + least > 0.9 * chains * (double)p.ntot * (1 + 6 * p.h) * 1.17 / ((grouped ? 1.6 : 1.0) * sms * clock)) return false;
  b->aligned = p.n[0] % 4 == 0 && p.S[0] % 4 == 0 && reinterpret_cast<uintptr_t>(p.ring) % 16 == 0;
  return b->blocks * b->zc * kBrickWarps < (1ll << 31);
}

template <int H, int AB, int MODE>
cudaError_t launch_brick_typed(const StepParams &p, const BrickShape &b, const BrickAdjoint &adj, int64_t blocks, int64_t n,
                               const int64_t *n_base, cudaStream_t st) {
  const int bytes = (2 * H + 2) * b.plane * 8;
  auto kernel = brick_kernel<H, AB, MODE>;
  if (bytes + 4096 > 48 * 1024) {  // with the static part
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
  }
  kernel<<<(unsigned)blocks, kBrickThreads, bytes, st>>>(p, b, adj, n, n_base);
  const int64_t words = b.blocks * b.zc * kBrickWarps, want = (words + 63) / 64;
  int64_t grid = 2 * brick_sms();
  if (want < grid) grid = want;
  if (MODE == 2 && blocks < grid) grid = blocks;
  if (grid > 1) grid = (grid - 1) | 1;  // odd: every block's words come from all parts of the tiles
  // launched while the march ends; it waits for the march's memory itself
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kListThreads);
  cfg.stream = st;
  cudaLaunchAttribute early = {};
  early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &early;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, brick_listed_kernel<H, AB, MODE>, p, b, adj, n, n_base);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

template <int AB, int MODE>
cudaError_t launch_brick_h(const StepParams &p, const BrickShape &b, const BrickAdjoint &adj, int64_t blocks, int64_t n,
                           const int64_t *n_base, cudaStream_t st) {
  if (p.h == 1) return launch_brick_typed<1, AB, MODE>(p, b, adj, blocks, n, n_base, st);
  if (p.h == 2) return launch_brick_typed<2, AB, MODE>(p, b, adj, blocks, n, n_base, st);
  return launch_brick_typed<3, AB, MODE>(p, b, adj, blocks, n, n_base, st);
}

// p with the taps t (centre, then each axis in offset order) in place of the step's.
void set_taps(StepParams *p, double s0, const double s[3][2 * AT_MAX_H + 1], bool reversed) {
  const int h = p->h;
  double keep[3][2 * AT_MAX_H + 1];
  for (int a = 0; a < 3; ++a)
    for (int j = 0; j <= 2 * h; ++j) keep[a][j] = s[a][reversed ? 2 * h - j : j];
  p->s0 = s0;
  for (int a = 0; a < 3; ++a)
    for (int j = 0; j <= 2 * h; ++j) p->s[a][j] = keep[a][j];
  fx_prepare_3d(p, s0, keep);
}

}  // namespace

int64_t brick_listed_words(const StepParams &p) {
  BrickShape b;
  return brick_shape(p, &b) ? b.blocks * b.zc * kBrickWarps : 0;
}

bool launch_forward_brick(const StepParams &p, int64_t n, const int64_t *n_base, cudaStream_t st, cudaError_t *e) {
  BrickShape b;
  if (!brick_shape(p, &b)) return false;
  const BrickAdjoint none = {};
  *e = p.ts > 1 ? launch_brick_h<1, 0>(p, b, none, b.blocks, n, n_base, st)
                : launch_brick_h<0, 0>(p, b, none, b.blocks, n, n_base, st);
  return true;
}

bool launch_adjoint_brick(const StepParams &f, uint8_t *akeff, double *lam, int Rl, int reach, const double *mu, bool alpha,
                          double *g_blk, int nblk, int64_t n, cudaStream_t st, cudaError_t *e) {
  BrickShape b;
  if (!brick_shape(f, &b)) return false;
  StepParams p = f;
  p.keff = akeff;
  const double *next = lam + (n + 1) % Rl * f.ntot, *src = mu ? mu : next;
  if (alpha) {
    // the second-derivative taps (no 1 in the centre), from the forward levels; before the next draws
    StepParams q = p;
    set_taps(&q, f.q0, f.q, false);
    if (!q.f3.ok) return false;
    BrickAdjoint a = {};
    a.src = src;
    a.g_blk = g_blk;
    *e = launch_brick_h<0, 2>(q, b, a, b.blocks < nblk ? b.blocks : nblk, n, nullptr, st);
    if (*e != cudaSuccess) return true;
  }
  set_taps(&p, f.s0, f.s, true);
  BrickAdjoint a = {};
  a.src = src;
  a.ident = mu ? next : nullptr;
  a.cur = lam + n % Rl * f.ntot;
  a.add = reach > 0;
  a.fresh = reach > 0 && n >= reach ? lam + (n - reach) % Rl * f.ntot : nullptr;
  if ((*e = launch_brick_h<0, 1>(p, b, a, b.blocks, n, nullptr, st)) != cudaSuccess) return true;
  FaceBoxes m;
  for (int k = 0; k < 3; ++k) {
    m.hw[k] = f.use_pe[k] ? f.h : 0;
    m.cs[k] = f.use_pe[k] ? (uint32_t)(f.pe[k] * 2 * f.h) : 0;  // a PE is at least 2 h wide
    m.cc[k] = f.n[k] - m.cs[k];
  }
  m.part_z = m.cs[2] * f.n[1] * f.n[0];
  m.part_y = m.cc[2] * m.cs[1] * f.n[0];
  m.total = m.part_z + m.part_y + m.cc[2] * m.cc[1] * m.cs[0];
  if (m.total == 0 || f.scheme == AT_SYNC || reach == 0) return true;
  const int64_t blocks = ((int64_t)m.total + 255) / 256, most = (int64_t)brick_sms() * 8;
  const unsigned g = (unsigned)(blocks < most ? blocks : most);
  if (f.h == 1) brick_faces_kernel<1><<<g, 256, 0, st>>>(p, m, src, lam, Rl, n);
  else if (f.h == 2) brick_faces_kernel<2><<<g, 256, 0, st>>>(p, m, src, lam, Rl, n);
  else brick_faces_kernel<3><<<g, 256, 0, st>>>(p, m, src, lam, Rl, n);
  *e = cudaGetLastError();
  return true;
}
