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
//    at a scale that has fallen since lack the digits between: sums over them want values as many bits larger, and beyond
//    kFxLift such bits they are not used (fixed.cuh, FxRing).
//  - One barrier per plane: iteration i sums output plane i-2-h from planes the ring already holds (while the loads of
//    plane i are in flight), publishes plane i's largest value, and after the barrier stores plane i.
//  - A thread sums four x-consecutive points.  A group with a half more than kBrickGuard bits below the scale (where the
//    field changes sign along two axes at once, or falls steeply) takes the FP64 chain, as does every group of a plane
//    near infinities, NaN or values at the ends of the exponent range.  The former are listed and done together after
//    the march: done in place, one such group held its block's barrier for 52 DFMA (256^3: 411 us per step against 242
//    without any).
//
// The backward sweep of the gradient runs on the same tiles: the transposed step's level-n part (taps reversed, cells
// across a face counted only at delay 0), the alpha term (second-derivative taps of U^n times lambda, summed), and a
// small kernel for what the cells at the faces send to older levels.  256^3 in 4^3 PEs, order 4: 1.01 -> 0.63 ms per
// backward step with the alpha term, 0.52 -> 0.37 ms without.
//
// What bounds it: the issue of the integer pipes (at order 4 39 multiply-adds per point, 22 instructions for 1.4
// conversions, 25 for the rounding, the rest addresses and control) and the barrier.  512^3 in 8^3 PEs, L = 3 on GB300:
// order 4 3.51 -> 1.43 ms per step, order 2 1.83 -> 0.96 ms; 256^3 in 4^3 PEs 453 -> 247 and 236 -> 160 us.
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
constexpr int kBrickLater = 512; // groups a block can list for the FP64 chain
constexpr int kCore = 4;         // values of the tile's own cells a thread loads per plane
constexpr int kBrickSlots = 6;   // and with those around it
constexpr int kBrickGuard = 10;  // a tile spans more cells than a 1D window: lines where the field changes sign meet in it

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

// One point of the transposed step's level-n part as an FMA chain: p.s holds the taps reversed, p.s0 the centre; a
// neighbour across a face with a delay (kn: the delays of the neighbours' sides) contributes to older levels instead.
template <int H>
__device__ __noinline__ double transposed_point(const StepParams &p, const double *__restrict__ src, const int pidx[3],
                                                const int kn[3][2], const int c[3]) {
  const int64_t stride[3] = {1, (int64_t)p.n[0], (int64_t)p.n[0] * p.n[1]};
  const int64_t i = c[2] * stride[2] + c[1] * stride[1] + c[0];
  double acc = fma(p.s0, LdgNC::ld(src + i), p.zero);
  for (int a = 0; a < 3; ++a) {
    const int pos = c[a] - pidx[a] * p.S[a];
    for (int j = -H; j <= H; ++j) {
      if (j == 0) continue;
      if (p.use_pe[a] && ((pos + j < 0 && kn[a][0] > 0) || (pos + j >= p.S[a] && kn[a][1] > 0))) continue;
      const int cj = wrap_coord(c[a] + j, p.n[a]);
      acc = fma(p.s[a][j + H], LdgNC::ld(src + i + (int64_t)(cj - c[a]) * stride[a]), acc);
    }
  }
  return acc;
}

// MODE 0: the forward step.  MODE 1: the part of the transposed step that stays at level n, with the taps reversed; a
// buffer point counts only where the neighbour's side that reads across has delay 0.  MODE 2: the alpha term's sum of
// lambda x (the second-derivative taps of U^n), for which p.s0, p.s and p.f3 hold those taps; each block takes the same
// tiles in the same order, so the sum is deterministic.
template <int H, int AB, int MODE>
__global__ void __launch_bounds__(kBrickThreads, kBrickBlocks) brick_kernel(const StepParams p, const BrickShape b,
                                                                            const BrickAdjoint adj, const int64_t n_off,
                                                                            const int64_t *n_base) {
  constexpr int NR = 2 * H + 2;  // ring planes
  extern __shared__ int2 ring[];
  __shared__ int mx[3], later[kBrickLater], n_later;
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
  const int nx = p.n[0], ny = p.n[1], nz = p.n[2], sn = (int)slot_of(n, p.R);
  const int64_t nxy = (int64_t)nx * ny;
  for (int64_t tile = blockIdx.x; tile < b.blocks; tile += gridDim.x) {
  // tile: x fastest, then y, then chunk, then PE
  int pidx[3], x0, y0, zs, ze;
  {
    int t = (int)tile;
    const int tx = t % b.tiles_x; t /= b.tiles_x;
    const int ty = t % b.tiles_y; t /= b.tiles_y;
    const int ch = t % b.chunks; t /= b.chunks;
    pidx[0] = t % p.pe[0]; t /= p.pe[0];
    pidx[1] = t % p.pe[1];
    pidx[2] = t / p.pe[1];
    x0 = pidx[0] * p.S[0] + tx * b.tx;
    y0 = pidx[1] * p.S[1] + ty * b.rows;
    zs = pidx[2] * p.S[2] + ch * b.zc;
    ze = min(zs + b.zc, (pidx[2] + 1) * p.S[2]);
  }
  const int px1 = (pidx[0] + 1) * p.S[0], py1 = (pidx[1] + 1) * p.S[1];
  const int pz0 = pidx[2] * p.S[2], pz1 = pz0 + p.S[2];
  const int xlen = min(b.tx, px1 - x0), ylen = min(b.rows, py1 - y0);
  int kside[3][2];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    // the PE's own sides; transposed: the side of the neighbour across each face that reads this PE's cells
    int lo[3] = {pidx[0], pidx[1], pidx[2]}, hi[3] = {pidx[0], pidx[1], pidx[2]};
    if (MODE == 1) {
      lo[a] = pidx[a] == 0 ? p.pe[a] - 1 : pidx[a] - 1;
      hi[a] = pidx[a] + 1 == p.pe[a] ? 0 : pidx[a] + 1;
    }
    kside[a][0] = p.use_pe[a] ? keff[side_of<3>(p, lo, a, MODE == 1 ? 1 : 0)] : 0;
    kside[a][1] = p.use_pe[a] ? keff[side_of<3>(p, hi, a, MODE == 1 ? 0 : 1)] : 0;
  }
  // This thread's share of a plane's cells: kCore slots of the tile's own cells, row by row, then the cells around it --
  // left and right of the rows, then below and above them -- so that the buffer points, which cost T FP64 operations
  // each, fill few warps.  goff: cell within the plane; code: slot in the ring plane, delay; -1: none.
  int goff[kBrickSlots], code[kBrickSlots];
  bool buffers = false;  // some of this thread's halo cells are buffer points with a delay
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
        if (hi ? x0 + c >= px1 : x0 + c < pidx[0] * p.S[0]) k = kside[0][hi];
      } else {
        const int hi = l - side >= H * xlen, m = l - side - hi * H * xlen;
        r = m / xlen;
        c = m - r * xlen;
        r += hi ? ylen : -H;
        if (hi ? y0 + r >= py1 : y0 + r < pidx[1] * p.S[1]) k = kside[1][hi];
      }
    }
    const int cc = c + 4;  // columns -4 .. : group boundaries stay multiples of four
    goff[s] = have ? wrap_coord(y0 + r, ny) * nx + wrap_coord(x0 + c, nx) : y0 * nx + x0;
    code[s] = have ? ((r + H) * b.stride + cc + (cc >> 2)) | (k << 16) : b.plane - 1;  // a pad slot nobody reads
    buffers = buffers || (have && k > 0);
  }
  // Buffer points: level n-k-m of halo slot s is hlev[s][m], fetched with the plane and combined after the sums in
  // between.  A warp with a buffer point does it for all its halo slots (delay 0: level n, not used) without branches.
  const bool some = __any_sync(0xffffffffu, buffers), deep = p.T > 1;
  double v[kBrickSlots], hlev[kBrickSlots - kCore][H + 1];
  auto load = [&](int zz) {
    const int64_t base = (int64_t)wrap_coord(zz, nz) * nxy;
    const double *src = un + base;
#pragma unroll
    for (int s = 0; s < kBrickSlots; ++s) v[s] = LdgNC::ld(src + goff[s]);
    if (MODE != 1 && some) {
#pragma unroll
      for (int s = kCore; s < kBrickSlots; ++s) {
        const int k = code[s] >> 16;
        const double *h = p.ring + base + goff[s];
        hlev[s - kCore][0] = LdgNC::ld(h + slot_back(sn, k, p.R) * p.ntot);
        if (deep) {  // the time-expanded rows read H + 1 levels, the others one
#pragma unroll
          for (int m = 1; m <= H; ++m) hlev[s - kCore][m] = LdgNC::ld(h + slot_back(sn, k > 0 ? k + m : 0, p.R) * p.ntot);
        }
      }
    }
  };
  auto extrapolate = [&](int zz) {
    const int kz = zz < pz0 ? kside[2][0] : (zz >= pz1 ? kside[2][1] : 0);
    if (MODE == 1) {  // what lies across a face with a delay goes to older levels (brick_faces_kernel)
#pragma unroll
      for (int s = 0; s < kBrickSlots; ++s)
        if (s < kCore ? kz > 0 : (code[s] >> 16) > 0) v[s] = 0.0;
    } else if (kz > 0) {  // a buffer plane: only the tile's own cells of it are read
      const int64_t base = (int64_t)wrap_coord(zz, nz) * nxy;
#pragma unroll
      for (int s = 0; s < kCore; ++s) v[s] = halo_value<LdgNC>(p, base + goff[s], sn, kz);
    } else if (some) {
#pragma unroll
      for (int s = kCore; s < kBrickSlots; ++s) {
        const int k = code[s] >> 16;  // halo_value's chain
        double acc = fma(p.w[k][0], hlev[s - kCore][0], p.zero);
        if (deep) {
#pragma unroll
          for (int m = 1; m <= H; ++m) acc = fma(p.w[k][m], hlev[s - kCore][m], acc);
        }
        v[s] = k > 0 ? acc : v[s];
      }
    }
  };
  if (tid == 0) n_later = 0;
  if (tid < 3) mx[tid] = 0;
  if (tid < 8) planes.top[tid] = planes.cut[tid] = 0;
  FxRing scale;
  // this thread's points; a thread without any sums the tile's first group along
  int row = tid / b.gx, grp = tid - row * b.gx;
  const bool mine = row < ylen && 4 * grp < xlen;
  row = mine ? row : 0;
  grp = mine ? grp : 0;
  const int nv = min(4, xlen - 4 * grp);
  const int col = (row + H) * b.stride + 4 * grp + 4 + grp + 1;  // its slot in a ring plane (pad slot per four)
  const int64_t cell0 = (int64_t)(y0 + row) * nx + x0 + 4 * grp;
  // the FP64 chain for group g of tile row rr of plane o
  auto chain = [&](int rr, int g, int o, double r[4]) {
    if (MODE == 1) {
      const int valid = min(4, xlen - 4 * g);
#pragma unroll 1
      for (int q = 0; q < valid; ++q) {
        const int c[3] = {x0 + 4 * g + q, y0 + rr, o};
        const double w = transposed_point<H>(p, un, pidx, kside, c);
        r[0] = q == 0 ? w : r[0]; r[1] = q == 1 ? w : r[1]; r[2] = q == 2 ? w : r[2]; r[3] = q == 3 ? w : r[3];
      }
    } else if (b.aligned) {
      double uc[4];
      group_eval<3, H, LdgNC, false>(p, keff, un, n, x0 + 4 * g, y0 + rr, o, r, uc);
    } else {
      const int valid = min(4, xlen - 4 * g);
      const int64_t i0 = (int64_t)o * nxy + (int64_t)(y0 + rr) * nx + x0 + 4 * g;
#pragma unroll 1
      for (int q = 0; q < valid; ++q) {
        const int c[3] = {x0 + 4 * g + q, y0 + rr, o};
        const double w = point_update<3, H, LdgNC>(p, keff, un, n, i0 + q, c);
        r[0] = q == 0 ? w : r[0]; r[1] = q == 1 ? w : r[1]; r[2] = q == 2 ? w : r[2]; r[3] = q == 3 ? w : r[3];
      }
    }
  };
  // Adams-Bashforth combination and store of `valid` points from i0
  auto finish = [&](int64_t i0, int valid, double r[4], const AbLevels<1> old[4]) {
    if (MODE == 2) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (q < valid) galpha = fma(LdgNC::ld(adj.src + i0 + q), r[q], galpha);
      return;
    }
    if (MODE == 1 && b.aligned) {  // the workspace is 16-byte aligned
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
    if (b.aligned) {
      reinterpret_cast<double2 *>(out + i0)[0] = make_double2(r[0], r[1]);
      reinterpret_cast<double2 *>(out + i0)[1] = make_double2(r[2], r[3]);
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (q < valid) out[i0 + q] = r[q];
    }
  };
  load(zs - H);
  __syncthreads();
  int wslot = 0, cslot = 0, m3 = 0;  // ring slots of plane i and of plane o - H of the output; i - (zs - H) mod 3
  for (int i = zs - H; i < ze + H + 2; ++i) {
    const int o = i - 2 - H;
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
          far = MODE != 2 && min(g0, g1) < fx_least(kBrickGuard, lift);  // a sum over all points needs no local bits
        }
        int64_t A[4], B[4], C[4];
        const FxTaps<6 * AT_MAX_H + 1> &t = p.f3;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          A[q] = (int64_t)t.w1[0] * c4[q].x;
          B[q] = fx_mad(t.w1[0], c4[q].y, kFxB0);
          C[q] = fx_mad(t.w0[0], c4[q].x, kFxC0);
        }
        auto tap = [&](int k, int q, const int2 &f) {
          A[q] = fx_mad(t.w1[k], f.x, A[q]);
          B[q] = fx_mad(t.w1[k], f.y, B[q]);
          C[q] = fx_mad(t.w0[k], f.x, C[q]);
        };
        // x: cells -H .. 3 + H of the row; the pad slots lie before cells 0 and 4
#pragma unroll
        for (int d = -H; d <= 3 + H; ++d) {
          const int2 f = d >= 0 && d < 4 ? c4[d & 3] : mid[d < 0 ? d - 1 : d + 1];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int j = d - q;  // tap j of point q reads cell q + j
            if (j != 0 && j >= -H && j <= H) tap(1 + (j < 0 ? j + H : j + H - 1), q, f);
          }
        }
#pragma unroll
        for (int j = -H; j <= H; ++j) {
          if (j == 0) continue;
          const int2 *s = mid + j * b.stride;
#pragma unroll
          for (int q = 0; q < 4; ++q) tap(1 + 2 * H + (j < 0 ? j + H : j + H - 1), q, s[q]);
        }
#pragma unroll
        for (int j = -H; j <= H; ++j) {
          if (j == 0) continue;
#pragma unroll
          for (int q = 0; q < 4; ++q) tap(1 + 4 * H + (j < 0 ? j + H : j + H - 1), q, pl[H + j][q]);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) A[q] = fx_join(A[q], B[q], C[q]);
        const int ex = E - 1023 - p.f3.sw;
        if (AB) {
#pragma unroll
          for (int q = 0; q < 4; ++q) r[q] = fx_to_any(A[q], ex);
        } else {
          fx_results<4>(A, ex, r);
        }
      }
      bool put = mine;
      if (mine && (far || !usable)) {
        const int at = usable ? atomicAdd(&n_later, 1) : kBrickLater;
        put = at >= kBrickLater;
        if (put) chain(row, grp, o, r);
        else later[at] = (o - zs) << 16 | row << 8 | grp;
      }
      if (put) finish(i0, nv, r, old);
      cslot = cslot + 1 == NR ? 0 : cslot + 1;
    }
    if (i < ze + H) {
      extrapolate(i);
      int mag = 0;
#pragma unroll
      for (int s = 0; s < kBrickSlots; ++s) mag = max(mag, fx_mag(v[s]));
      mag = __reduce_max_sync(0xffffffffu, mag);
      if ((tid & 31) == 0) atomicMax(&mx[m3], mag);
    }
    if (i >= ze + H) {
      if (i == ze + H) __syncthreads();  // the last plane stored is read in the next iteration
      continue;
    }
    __syncthreads();
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
        const Fx f = fx_split(fx_from(v[s], scale.E));
        dst[code[s] & 0xffff] = make_int2(f.hi, f.lo);
      }
    }
    wslot = wslot + 1 == NR ? 0 : wslot + 1;
    m3 = m3 == 2 ? 0 : m3 + 1;
    if (i + 1 < ze + H) load(i + 1);
  }
  __syncthreads();
#pragma unroll 1
  for (int e = tid; e < min(n_later, kBrickLater); e += kBrickThreads) {
    const int rr = (later[e] >> 8) & 0xff, g = later[e] & 0xff, o = zs + (later[e] >> 16), valid = min(4, xlen - 4 * g);
    const int64_t i0 = (int64_t)o * nxy + (int64_t)(y0 + rr) * nx + x0 + 4 * g;
    double r[4];
    AbLevels<1> old[4];
    if (AB) {
#pragma unroll
      for (int q = 0; q < 4; ++q) ab_fetch<1>(p, n, i0 + (q < valid ? q : 0), old[q]);
    }
    chain(rr, g, o, r);
    finish(i0, valid, r, old);
  }
  __syncthreads();
  }
  if (MODE == 2) {
    __shared__ double sums[kBrickThreads / 32];  // block sum in a fixed order
    for (int d = 16; d > 0; d >>= 1) galpha += __shfl_down_sync(0xffffffffu, galpha, d);
    if ((tid & 31) == 0) sums[tid >> 5] = galpha;
    __syncthreads();
    if (tid == 0) {
      double t = sums[0];
      for (int w = 1; w < kBrickThreads / 32; ++w) t += sums[w];
      adj.g_blk[blockIdx.x] += t;
    }
  }
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
  // takes as many of them as it has waves times planes, 2 h + 2 of which only fill the ring (512^3 in 8^3 PEs: 6.7 waves
  // of 70 planes, 1.43 ms at order 4; 256^3 in 8^3 PEs at order 6, where every tile meets three faces with T = 4 levels
  // each, 6 us per plane).  The grouped kernel (or the
  // per-point one, for shapes without groups of four) does one FP64 operation per tap and 8 % more for the halo, at 1.6
  // (1.0) lanes per SM and clock.
  const bool narrow = p.h == 3 && ((p.use_pe[0] && p.S[0] < 40) || (p.use_pe[1] && p.S[1] < 40));
  const double kIter[4] = {0.0, 2.1e-6, 3.1e-6, narrow ? 6e-6 : 3.0e-6}, clock = 2.07e9;
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
    const double t = waves * (zc + 2 * p.h + 2) * kIter[p.h];
    if (least == 0.0 || t < least) {
      least = t;
      b->zc = zc;
    }
  }
  b->chunks = (p.S[2] + b->zc - 1) / b->zc;
  b->blocks = columns * b->chunks;
  const bool grouped = p.n[0] % 4 == 0 && p.S[0] % 4 == 0;
  if (least > 0.95 * (double)p.ntot * (1 + 6 * p.h) * 1.08 / ((grouped ? 1.6 : 1.0) * sms * clock)) return false;
  b->aligned = p.n[0] % 4 == 0 && p.S[0] % 4 == 0 && reinterpret_cast<uintptr_t>(p.ring) % 16 == 0;
  return b->blocks < (1ll << 31);
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
  double t[6 * AT_MAX_H + 1] = {s0}, keep[3][2 * AT_MAX_H + 1];
  int c = 1;
  for (int a = 0; a < 3; ++a)
    for (int j = -h; j <= h; ++j) {
      keep[a][j + h] = s[a][reversed ? h - j : h + j];
      if (j != 0) t[c++] = keep[a][j + h];
    }
  p->s0 = s0;
  for (int a = 0; a < 3; ++a)
    for (int j = 0; j <= 2 * h; ++j) p->s[a][j] = keep[a][j];
  fx_prepare(t, c, &p->f3);
}

}  // namespace

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
