// Integer square root of I-LayerNorm's radicands (plain C++, so that the host can run it over the whole range too).
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define IVIT_ISQRT_FN __host__ __device__ __forceinline__
#else
#define IVIT_ISQRT_FN inline
#endif

namespace ivit {

// High word of a * b, plus c.
IVIT_ISQRT_FN int isqrt_mad_hi(int a, int b, int c) {
#ifdef __CUDA_ARCH__
  int d;
  asm("mad.hi.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
#else
  return (int)(((int64_t)a * b) >> 32) + c;
#endif
}

IVIT_ISQRT_FN int isqrt_clz(unsigned n) {
#ifdef __CUDA_ARCH__
  return __clz((int)n);
#else
  return __builtin_clz(n);
#endif
}

// floor(sqrt(n)) for n < 2^26, the value the guarded iteration of Eq. (iterative) converges to, in integer arithmetic and
// without a division.  n = (1 + u) 2^e; sqrt(1 + u) on [0, 1) by the cubic of least maximal relative error (6.94e-5, from a
// linear programme on 4001 points, coefficients rounded to 32 bits), times 2^(e/2) cut to a multiple of 1/8: at
// sqrt(n) < 8192 that is off by less than 0.57 + 0.18, the integer part by at most one, which the square tells.
// A row's scalars are a chain between its loads and its stores: bit by bit the root took 13 dependent steps (calls back to back,
// bit by bit -> cubic: 25216 x 768 10.8 -> 10.5 us, 12608 x 384 4.21 -> 4.07; from the single-precision root 10.4 and 4.01).
IVIT_ISQRT_FN unsigned isqrt26(unsigned n) {
  const int z = isqrt_clz(n | 1u), e = 31 - z;
  const int u = (int)((n << z) & 0x7fffffffu);             // 31-bit fraction; a product's high word is half of u times the other
  const int k = (e & 1 ? 46341 : 1 << 15) >> (12 - (e >> 1));   // 2^(3 + e/2)
  int p = isqrt_mad_hi(u, 107103318, -231787875);          // units 2^-31
  p = isqrt_mad_hi(u, p, 533907397);                       // 2^-30
  p = isqrt_mad_hi(u, p, 536908166);                       // 2^-29: sqrt(1 + u)
  const int r = isqrt_mad_hi(p, k, 0);
  const int left = (int)n - r * r;
  return (unsigned)(r + (left > 2 * r ? 1 : 0) - (left < 0 ? 1 : 0));
}

}  // namespace ivit
