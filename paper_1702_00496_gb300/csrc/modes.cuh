// modes.cuh -- the sum over the initial-condition modes of one axis (Eq. "IC"; Eq. "ana_sol" at time t), shared by
// the single-problem kernels (wave.cu) and the ensemble engine (ensemble.cu), so both produce the same bits.
#pragma once
#include "internal.h"

namespace atfd {

// sum_q A_q sin(k_q x + phi'_q) at x = pi xpi (grid point i of n: xpi = i (2 / n), exact for n a power of two),
// each mode adding ac sin kx + as cos kx (two FMAs), from one sincospi and, over the wavenumbers k = 2 .. kmax,
//   kmax <= 16: the three-term recurrences sin (k+1)x = 2 cos x sin kx - sin (k-1)x (and the same for cos), one
//               FMA each per wavenumber.  A rounding error made at wavenumber j reaches k multiplied by
//               sin((k-j)x)/sin x, at most k - j in size: under kmax^2/2 ulp in all, 1.4e-14 at kmax = 16;
//   kmax > 16:  the rotation (cos kx, sin kx) = (cos (k-1)x, sin (k-1)x) x (cos x, sin x), two multiplies and two
//               FMAs per wavenumber, whose errors add up linearly (a few ulp per rotation).
// Requires ms.rot.
__device__ __forceinline__ double mode_sum(const ModeSet &ms, int nmodes, double xpi) {
  double sx, cx;
  sincospi(xpi, &sx, &cx);
  double sk = sx, ck = cx, s = 0.0;
  int q = 0;
  if (ms.kmax <= 16) {
    const double tc = cx + cx;
    double sp = 0.0, cp = 1.0;  // sin, cos of (k-1)x
    for (int k = 1; k <= ms.kmax; ++k) {
      if (k > 1) {
        const double ns = fma(tc, sk, -sp), nc = fma(tc, ck, -cp);
        sp = sk; cp = ck;
        sk = ns; ck = nc;
      }
      while (q < nmodes && ms.kr[q] == k) {
        s = fma(ms.as[q], ck, fma(ms.ac[q], sk, s));
        ++q;
      }
    }
    return s;
  }
  for (int k = 1; k <= ms.kmax; ++k) {
    if (k > 1) {
      const double ns = fma(sk, cx, ck * sx), nc = fma(ck, cx, -(sk * sx));
      sk = ns;
      ck = nc;
    }
    while (q < nmodes && ms.kr[q] == k) {
      s = fma(ms.as[q], ck, fma(ms.ac[q], sk, s));
      ++q;
    }
  }
  return s;
}

// The mode sums of 16 consecutive grid points, the ninth at x = pi xpi: one sincospi and the recurrences above give
// P_q = A sin(k_q x + phi'_q) and Q_q = A cos(k_q x + phi'_q) there, and the points j cells to either side are
//     sum_q P_q cos(k_q j dx) +- sum_q Q_q sin(k_q j dx),
// both sums shared by the pair: 16 FMAs per mode and run instead of a sincospi, two recurrences and two FMAs per mode
// for every point (2^24 points, 10 modes: 17 FP64 operations per point instead of about 70).  The cosines and sines of
// the offsets come from the host; an error there or in P, Q enters each point once.
//
// G threads share a run: thread `part` of them has the pairs j = part + G i (i < 8 / G; points 7 - j and 9 + j of the run, E - O
// and E + O), and s0, the ninth point, is every thread's.  The operations of a point are the same for every G, so its bits are.
// cs: the table's cosines and sines, cs[q][j] (G > 1: in shared memory, as the threads of a warp read different ones).
template <int G>
__device__ __forceinline__ void mode_pairs(const ModeSet &ms, const double (*cs)[8][2], int nmodes, double xpi, int part,
                                           double E[8 / G], double O[8 / G], double &s0) {
  double sx, cx;
  sincospi(xpi, &sx, &cx);
  double sk = sx, ck = cx;
  s0 = 0.0;
#pragma unroll
  for (int j = 0; j < 8 / G; ++j) E[j] = O[j] = 0.0;
  const double tc = cx + cx;
  double sp = 0.0, cp = 1.0;  // sin, cos of (k-1)x
  int q = 0;
  for (int k = 1; k <= ms.kmax; ++k) {
    if (k > 1) {
      double ns, nc;
      if (ms.kmax <= 16) {
        ns = fma(tc, sk, -sp);
        nc = fma(tc, ck, -cp);
        sp = sk; cp = ck;
      } else {
        ns = fma(sk, cx, ck * sx);
        nc = fma(ck, cx, -(sk * sx));
      }
      sk = ns; ck = nc;
    }
    while (q < nmodes && ms.kr[q] == k) {
      const double P = fma(ms.as[q], ck, ms.ac[q] * sk), Q = fma(ms.ac[q], ck, -(ms.as[q] * sk));
      s0 += P;
#pragma unroll
      for (int j = 0; j < 8 / G; ++j) {
        E[j] = fma(P, cs[q][part + G * j][0], E[j]);
        O[j] = fma(Q, cs[q][part + G * j][1], O[j]);
      }
      ++q;
    }
  }
}

// All 16 points by one thread.
__device__ __forceinline__ void mode_run(const ModeSet &ms, const ModeTable &mt, int nmodes, double xpi, double out[16]) {
  double E[8], O[8];
  mode_pairs<1>(ms, mt.cs, nmodes, xpi, 0, E, O, out[8]);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    out[7 - j] = E[j] - O[j];
    if (j < 7) out[9 + j] = E[j] + O[j];
  }
}

}  // namespace atfd
