// fixed.cuh -- stencil sums in block fixed point: the contractions of the step kernels on the integer pipes.
//
// GB300 retires 2 FP64 FMAs per SM and clock (measured 1.99) but about 30 multiply-adds of 32 x 32 + 64 bits with a 64-bit
// addend (and 60-126 of the logic, shift and add instructions around them), so a product of 62 by 60 bits in three of them
// takes a fifth of the time of one DFMA.  As FP64 chains the pipe bounded every step kernel at 9-20 % of the memory
// bandwidth, and a stencil sum is a contraction of values of similar size with constant weights, so it needs no exponent
// per term:
//
//   values   X = floor(v 2^(61 - e)), e the largest exponent in the window (biased: E): |X| < 2^62, 8 bits below the
//            last bit of the window's largest value.  X = hi 2^32 + lo, hi and lo signed.
//   weights  W = round(w 2^sw), sw so that sum |W| <= 1.9 2^60 (prepared on the host).  W = w1 2^29 + w0, w0 signed.
//   sum      A = sum w1 hi, B = sum w1 lo, C = sum w0 hi, in 64 bits each without overflow (|w1 hi| sums to under
//            2^62, |w1 lo| to under 2^63, |w0 hi| to under 31 2^58 for up to 31 taps); w0 lo, up to a
//            quarter of a unit of R per tap, is left out.
//            R = A + B 2^-32 + C 2^-29 = sum W X 2^-61, rounded once to the nearest FP64 value R 2^(E - 1023 - sw).
//
// R is off by a few units: at most one for the cut values and one for the joins, a quarter per tap for w0 lo and half of
// |X| 2^-61 per tap for its rounded weight.  Then there is one rounding, where an FMA chain of n terms rounds n times at 2^-53
// of its partial sums.  A cell that is small against the window's largest value loses by it, so callers look at the sum
// itself (1D; kFxLeast) or, where it is a small difference that is added to the cell's value, at that value: from 2^53 units
// on the result's own rounding is one of them.  3D tiles look at two neighbours' values (brick.cu).  Cells that are too
// small take the FMA chain, as do windows that hold an infinity or a NaN, or that lie at the ends of the exponent range
// (fx_usable).
#pragma once
#include <cstdint>
#include <cstring>

#if defined(__CUDACC__)
#define AT_FX_HD __host__ __device__ __forceinline__
#else
#define AT_FX_HD inline
#endif

namespace atfd {

// The cross terms, 2^-31 of A, can also be summed in FP32 (fx_cross: one integer multiply-add and two FFMA per tap instead
// of three multiply-adds, half the issue time).  Each of those FFMA then rounds at 2^-24 of its sum, 2^-55 of the window's
// largest value and less: before the one rounding of the result 2^-54 rms and up to 2^-51.5 for the 17 taps of four steps at
// order 4.  That is still under the FMA chain's error, rms and at worst, as long as every value of the window lies within
// kFxNear bits of the largest and the taps go from the outermost pair to the centre, in a sum for either part
// (test_fixed_cross_host.py; in one sum, in offset order, it was above the chain's from two bits on).
constexpr uint32_t kFxLeast = 1u << 21;      // upper word of a sum that is at least as exact as the chain
constexpr uint32_t kFxLeastNear = 1u << 27;  // the same with the cross terms in FP32, for windows ...
constexpr int kFxNear = 1;                   // ... whose values lie within these bits of the largest
constexpr int kFxLowBits = 29;   // bits of a weight's low part

// Can windows whose largest value has biased exponent E be summed in fixed point?  Not with infinities or NaN (2047);
// not where a result could leave the normal range (weights sum to at most 2^64 here, results reach down 2^-62).
AT_FX_HD bool fx_usable(int E) { return E >= 192 && E < 1960; }

AT_FX_HD int32_t fx_word(double v, int hi) {
#if defined(__CUDA_ARCH__)
  return hi ? __double2hiint(v) : __double2loint(v);
#else
  uint64_t b;
  std::memcpy(&b, &v, 8);
  return (int32_t)(hi ? b >> 32 : b & 0xffffffffu);
#endif
}

AT_FX_HD int64_t fx_shr(int64_t x, int s) {  // arithmetic shift right, s >= 0; from 63 on the sign
#if defined(__CUDA_ARCH__)
  int64_t r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
  return r;
#else
  return x >> (s > 63 ? 63 : s);
#endif
}

// One integer multiply-add of 32 x 32 + 64 bits (written as a product: the compiler keeps it in one instruction; as
// inline assembly it came out as a multiply and separate additions).
AT_FX_HD int64_t fx_mad(int32_t a, int32_t b, int64_t c) { return (int64_t)a * b + c; }

// |v|'s upper word: its maximum over a window, shifted down by 20, is the window's exponent E.
AT_FX_HD int32_t fx_mag(double v) { return fx_word(v, 1) & 0x7fffffff; }

// X of v as 64 bits; zero, and what lies under the window's last bit, becomes 0 or -1.
AT_FX_HD int64_t fx_from(double v, int E) {
  const uint32_t hi = (uint32_t)fx_word(v, 1), lo = (uint32_t)fx_word(v, 0);
  const uint32_t sm = (uint32_t)((int32_t)hi >> 31);
  const uint32_t m1 = ((((hi << 9) | (lo >> 23)) & 0x1fffffffu) | 0x20000000u) ^ sm, m0 = (lo << 9) ^ sm;
  const int s = E - (int)((hi + hi) >> 21);
  return fx_shr((int64_t)(((uint64_t)m1 << 32) | m0), s);
}

struct Fx {
  int32_t hi, lo;
};

AT_FX_HD Fx fx_split(int64_t x) {
  Fx f;
  f.lo = (int32_t)(uint32_t)(uint64_t)x;
  f.hi = (int32_t)((x + 0x80000000ll) >> 32);
#if defined(__CUDA_ARCH__)
  asm("" : "+r"(f.hi), "+r"(f.lo));  // plain 32-bit registers from here on: as the shifted 64-bit value they come
#endif                               // from, the compiler multiplies them in 64 x 64 bits
  return f;
}

// A + B 2^-32 + C 2^-29 (B and C carry their rounding halves from the start of the sums)
constexpr int64_t kFxB0 = 1ll << 31, kFxC0 = 1ll << (kFxLowBits - 1);
AT_FX_HD int64_t fx_join(int64_t A, int64_t B, int64_t C) { return A + (B >> 32) + (C >> kFxLowBits); }

// R 2^ex as FP64, rounded to nearest; |R| < 2^63, the result in the normal range (or zero).  fx_to_wide needs |R| >= 2^32
// (*small says when that fails): the exponent of a 32-bit integer then comes from its conversion toward zero, two
// instructions against the quarter rate of a leading-zero count.
AT_FX_HD double fx_assemble(uint64_t a, int sh, int32_t sign, int ex) {
  a = (a << sh) + 0x200;       // leading bit at 62, half of the last place added
  const uint64_t m = a >> 10;  // implicit bit at 52 (or 53 after a carry, which the sum below takes as an exponent)
  const uint32_t rh = ((uint32_t)(m >> 32) + ((uint32_t)(1023 + 62 + ex - sh - 1) << 20)) | ((uint32_t)sign & 0x80000000u);
#if defined(__CUDA_ARCH__)
  return __hiloint2double((int)rh, (int)(uint32_t)m);
#else
  const uint64_t bits = ((uint64_t)rh << 32) | (uint32_t)m;
  double v;
  std::memcpy(&v, &bits, 8);
  return v;
#endif
}

AT_FX_HD double fx_to(int64_t R, int ex) {
  const int64_t sm = R >> 63;
  const uint64_t a = (uint64_t)((R ^ sm) - sm);
  if (a == 0) return 0.0;
#if defined(__CUDA_ARCH__)
  const int sh = __clzll((long long)a) - 1;
#else
  const int sh = __builtin_clzll(a) - 1;
#endif
  return fx_assemble(a, sh, (int32_t)(sm >> 32), ex);
}

// |x|'s upper word (one less for an x below zero whose lower word is 0), given x's.
AT_FX_HD uint32_t fx_upper(int32_t hi) { return (uint32_t)(hi ^ (hi >> 31)); }

// Upper word from which on a value of an output's stencil is within `guard` bits of the largest there is, where entries
// miss `lift` bits (guard >= lift).
AT_FX_HD uint32_t fx_least(int guard, int lift) { return 1u << (30 - guard + lift); }

AT_FX_HD double fx_to_wide(int64_t R, int ex, uint32_t *small) {
#if defined(__CUDA_ARCH__)
  const int64_t sm = R >> 63;
  const uint64_t a = (uint64_t)((R ^ sm) - sm);
  const uint32_t ah = (uint32_t)(a >> 32);
  *small = ah < *small ? ah : *small;
  return fx_assemble(a, 157 - (int)(__float_as_uint(__uint2float_rz(ah)) >> 23), (int32_t)(sm >> 32), ex);
#else
  (void)small;
  return fx_to(R, ex);
#endif
}

// The same for results of any size, without a branch (differences such as dt f, which lie far below their operands).
AT_FX_HD double fx_to_any(int64_t R, int ex) {
#if defined(__CUDA_ARCH__)
  const int64_t sm = R >> 63;
  const uint64_t a = (uint64_t)((R ^ sm) - sm);
  const uint32_t ah = (uint32_t)(a >> 32), word = ah ? ah : (uint32_t)a;
  const int lead = (int)(__float_as_uint(__uint2float_rz(word)) >> 23);  // 127 + leading bit; 0 for a zero word
  const double r = fx_assemble(a, (ah ? 157 : 189) - lead, (int32_t)(sm >> 32), ex);
  return word ? r : 0.0;
#else
  return fx_to(R, ex);
#endif
}

// N results at once; returns the upper word of the smallest |R|, below 2^32 of which (0) a result is not valid.
template <int N>
AT_FX_HD uint32_t fx_results_wide(const int64_t R[N], int ex, double r[N]) {
  uint32_t small = 0xffffffffu;
#if defined(__CUDA_ARCH__)
#pragma unroll
#endif
  for (int q = 0; q < N; ++q) {
    r[q] = fx_to_wide(R[q], ex, &small);
#if !defined(__CUDA_ARCH__)
    const uint32_t up = (uint32_t)((uint64_t)(R[q] < 0 ? -R[q] : R[q]) >> 32);
    small = up < small ? up : small;
#endif
  }
  return small;
}

// The same where such results are valid too: the rare ones are done again.
template <int N>
AT_FX_HD void fx_results(const int64_t R[N], int ex, double r[N]) {
  if (fx_results_wide<N>(R, ex, r) == 0) {
#if defined(__CUDA_ARCH__)
#pragma unroll
#endif
    for (int q = 0; q < N; ++q)
      if (R[q] < (1ll << 32) && R[q] > -(1ll << 32)) r[q] = fx_to(R[q], ex);
  }
}

// The scale of a ring of planes that a march lays down one by one (brick.cu), each cut at the scale of its moment.
//
// A larger plane raises the scale: every entry is shifted down and is then cut at the new scale, like the plane itself.
// Once the ring has fallen two bits below it the scale falls and the entries are shifted up -- but the digits that were cut
// at the old scale stay lost: they are `lift` bits short of what a plane cut at the new scale holds.  Callers ask that of
// an output's planes and want values as many bits larger (fx_least), or take the FP64 chain.
constexpr int kFxLift = 6;  // planes with more missing bits than this are not used

struct FxRing {    // the same in every thread of a march
  int E = -1;      // exponent of the scale; -1: no plane but zeros so far
  int until = -8;  // planes up to this one may have been cut above it, or are not there
};
struct FxPlanes {          // of the last eight planes: plane i at i mod 8, written by one thread (fx_ring_note)
  int top[8], cut[8];      // exponent of the largest value (0: zeros, or not usable) and of the scale it was cut at
};
constexpr int kFxNever = 1 << 20;  // cut of a plane that is not usable

// Is a plane whose largest magnitude (fx_mag; 1 where that is 0 but the values are not) is mag summed in fixed point?  Zeros
// are; denormal numbers are not zeros.
AT_FX_HD bool fx_plane_usable(int mag) { return mag == 0 || fx_usable(mag >> 20); }

// Plane i joins; m: exponent of its largest value (0 as above), usable: fx_plane_usable; reach: planes on either side that
// an output reads, so the 2 reach + 1 planes before i are still in use.  Returns by how much the scale rose: entries go down
// by that, or up by its negative; 0 also for the first scale, before which every entry is 0 or -1.
AT_FX_HD int fx_ring_join(FxRing &r, const FxPlanes &p, int i, int m, int reach, bool usable) {
  int to = r.E;
  if (m != 0 && m > r.E) {
    to = m;
  } else if (m != 0 && m <= r.E - 2) {  // has the whole ring fallen?
    int most = m;
    for (int q = 1; q <= 2 * reach + 1; ++q) most = p.top[(i - q) & 7] > most ? p.top[(i - q) & 7] : most;
    if (most <= r.E - 2) to = most;
  }
  const int d = r.E < 0 ? 0 : to - r.E;
  if (d < 0) r.until = i - 1;
  if (!usable) r.until = i;
  r.E = to;
  return d;
}

AT_FX_HD void fx_ring_note(FxPlanes &p, const FxRing &r, int i, int m, int d, bool usable) {
  if (d > 0)
    for (int q = 0; q < 8; ++q) p.cut[q] = p.cut[q] > r.E ? p.cut[q] : r.E;
  p.top[i & 7] = m;
  p.cut[i & 7] = usable ? r.E : kFxNever;
}

// Bits that the planes o - reach .. o + reach of an output miss against the scale.
AT_FX_HD int fx_ring_lift(const FxRing &r, const FxPlanes &p, int o, int reach) {
  if (o - reach > r.until) return 0;
  int most = r.E;
  for (int q = o - reach; q <= o + reach; ++q) most = p.cut[q & 7] > most ? p.cut[q & 7] : most;
  return most - r.E;
}

// A ring entry after the scale rose by d (fell by -d).
AT_FX_HD int64_t fx_rescale(int64_t x, int d) {
  return d > 0 ? fx_shr(x, d) : (int64_t)((uint64_t)x << (d < -63 ? 63 : -d));
}

// Weights of up to N taps; sw = 0 with ok = 0 when they cannot be represented (not finite, all zero, out of range).
// w_low: what the weights have below their last bit (composed stencils), or null.
// f1, f0: the same parts in FP32, in units of 2^3 of R, for sums whose cross terms go through the FP32 pipe.
template <int N>
struct FxTaps {
  int32_t w1[N], w0[N];
  float f1[N], f0[N];
  int32_t sw, ok;
};

// The FP32 sums of the cross terms, of the values' lower and upper words, and what they make of A.
struct FxCross {
  float lo, hi;
};
template <int N>
AT_FX_HD void fx_cross(FxCross &c, const FxTaps<N> &t, int j, float lo, float hi) {
#if defined(__CUDA_ARCH__)
  c.lo = fmaf(t.f1[j], lo, c.lo);
  c.hi = fmaf(t.f0[j], hi, c.hi);
#else
  c.lo = __builtin_fmaf(t.f1[j], lo, c.lo);
  c.hi = __builtin_fmaf(t.f0[j], hi, c.hi);
#endif
}
AT_FX_HD int64_t fx_join_cross(int64_t A, const FxCross &c) {
#if defined(__CUDA_ARCH__)
  return A + (int64_t)(__float2int_rn(c.lo) + __float2int_rn(c.hi)) * 8;
#else
  return A + (int64_t)(__builtin_lrintf(c.lo) + __builtin_lrintf(c.hi)) * 8;
#endif
}
// Tap m of n in the order that adds the largest terms last: the outermost pair, the next one, ..., the centre (n odd).
AT_FX_HD constexpr int fx_inward(int m, int n) { return m & 1 ? n - 1 - m / 2 : m / 2; }

template <int N>
inline void fx_prepare(const double *w, int n, FxTaps<N> *t, const double *w_low = nullptr) {
  std::memset(t, 0, sizeof(*t));
  double sum = 0.0, big = 0.0;
  for (int i = 0; i < n; ++i) {
    const double a = w[i] < 0 ? -w[i] : w[i];
    if (!(a < 1e18)) return;
    sum += a;
    if (a > big) big = a;
  }
  if (!(sum > 1e-15) || n > 31) return;
  int k = 60;  // smallest k in -49..60 with sum <= 1.9 2^k and every |w| < 2^k (their upper parts fit 31 bits)
  auto fits = [&](int kk) {
    const double s = kk >= 0 ? (double)(1ull << kk) : 1.0 / (double)(1ull << -kk);
    return sum <= 1.9 * s && big <= 0.999 * s;
  };
  while (k > -49 && fits(k - 1)) --k;
  if (!fits(k)) return;
  t->sw = 60 - k;
  for (int i = 0; i < n; ++i) {
    // w 2^sw exactly: sw is in 0..109
    double v = w[i], vl = w_low ? w_low[i] : 0.0;
    int s = t->sw;
    for (; s >= 60; s -= 60) {
      v *= 1152921504606846976.0;
      vl *= 1152921504606846976.0;
    }
    v *= (double)(1ull << s);
    vl *= (double)(1ull << s);
    const int64_t whole = (int64_t)v;
    const double rest = (v - (double)whole) + vl;
    const int64_t W = whole + (int64_t)(rest < 0 ? rest - 0.5 : rest + 0.5);
    const int64_t half = 1ll << (kFxLowBits - 1), mask = (1ll << kFxLowBits) - 1;
    const int64_t lo = ((W + half) & mask) - half;
    t->w0[i] = (int32_t)lo;
    t->w1[i] = (int32_t)((W - lo) >> kFxLowBits);
    t->f1[i] = (float)t->w1[i] * (1.0f / 34359738368.0f);  // 2^-35
    t->f0[i] = (float)t->w0[i] * (1.0f / 4294967296.0f);   // 2^-32
  }
  t->ok = 1;
}

}  // namespace atfd
