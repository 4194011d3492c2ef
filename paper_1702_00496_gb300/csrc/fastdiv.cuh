// fastdiv.cuh -- division by a number that is known before the launch, as a multiplication.
#pragma once
#include <cstdint>

#if defined(__CUDACC__)
#define AT_DIV_HD __host__ __device__ __forceinline__
#else
#define AT_DIV_HD inline
#endif

namespace atfd {

// q = n / d for 0 <= n < 2^30 and 1 <= d < 2^30 without a division: n m >> (32 + s) with m = ceil(2^(32 + s) / d), s =
// ceil(log2 d) - 2 at least 0, is exact as m's rounding error times n stays under 2^(32 + s) / d.
struct FastDiv {
  uint32_t m, s;
};
inline FastDiv fast_div(uint32_t d) {
  FastDiv f = {0u, 0u};
  if (d < 1) d = 1;
  while (((uint64_t)4 << f.s) < d) ++f.s;
  const uint64_t m = (((uint64_t)1 << (32 + f.s)) + d - 1) / d;
  f.m = m > 0xffffffffull ? 0u : (uint32_t)m;  // d = 1: 2^32 does not fit; m = 0 stands for it
  return f;
}
AT_DIV_HD uint32_t fdiv(uint32_t n, const FastDiv &f) {
  return f.m == 0 ? n : (uint32_t)(((uint64_t)n * f.m) >> 32) >> f.s;
}

}  // namespace atfd
