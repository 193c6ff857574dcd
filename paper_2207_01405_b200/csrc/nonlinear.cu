// I-LayerNorm (Sec. 3.5), Shiftmax (Algorithm 1) and ShiftGELU (Algorithm 2) kernels, sm_100a.
// Warps own whole rows, one or several at a time, short ones side by side; a row is read once, as coalesced words, and
// kept in registers between the reductions and the output pass (longer rows than the registers hold are read again).
#include "rowops.cuh"
#include "shiftmax.cuh"
#include <type_traits>

namespace ivit {

__device__ __forceinline__ int warp_sum(int v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ long long warp_sum_ll(long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ int warp_max(int v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Eq. (iterative): x_{i+1} = (x_i + floor(n / x_i)) >> 1 from x_0 = 2^floor(bit(n)/2); the first
// step is taken unconditionally, the following nine only while they decrease (leaving the loop
// at the first non-decrease gives the same value as holding it for the remaining steps).
__device__ __forceinline__ unsigned isqrt_u32(unsigned n) {
  if (n == 0) return 0;
  int bits = 32 - __clz(n);
  unsigned x = 1u << (bits >> 1);
  x = (x + n / x) >> 1;
#pragma unroll 1
  for (int i = 1; i < 10; ++i) {
    unsigned nx = (x + n / x) >> 1;
    if (nx >= x) break;
    x = nx;
  }
  return x;
}
__device__ __forceinline__ unsigned long long isqrt_u64(unsigned long long n) {
  if (n == 0) return 0;
  int bits = 64 - __clzll(n);
  unsigned long long x = 1ull << (bits >> 1);
  x = (x + n / x) >> 1;
#pragma unroll 1
  for (int i = 1; i < 10; ++i) {
    unsigned long long nx = (x + n / x) >> 1;
    if (nx >= x) break;
    x = nx;
  }
  return x;
}

// Four int32 values saturated to int8 and packed, x0 in the low byte.
__device__ __forceinline__ unsigned pack_sat8_u(int x0, int x1, int x2, int x3) {
  unsigned t, d;
  asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(t) : "r"(x3), "r"(x2), "r"(0));
  asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(x1), "r"(x0), "r"(t));
  return d;
}

__device__ __forceinline__ int floordiv_pos(int a, int b) {  // b > 0
  int q = a / b;
  return (a - q * b < 0) ? q - 1 : q;
}

// ------------------------------------------------------------------ I-LayerNorm, int8 input

// WPL = 32-bit words of the row held per lane (C <= 128 * WPL).
template <int WPL>
__global__ void __launch_bounds__(256) layernorm_i8_kernel(const int8_t* __restrict__ in, int64_t ldin,
                                                           ScaleDev gs, const int32_t* __restrict__ beta,
                                                           int M_ln, int8_t* __restrict__ out, int64_t ldout,
                                                           int64_t rows, int C) {
  pdl_wait();
  pdl_trigger();   // (after the wait: it may be the first kernel of a forward)
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int nwords = C >> 2;
  for (int64_t r = warp; r < rows; r += nwarps) {
    const int* src = reinterpret_cast<const int*>(in + r * ldin);
    int w[WPL];
    int s1 = 0, s2 = 0;
#pragma unroll
    for (int i = 0; i < WPL; ++i) {
      const int idx = lane + 32 * i;
      w[i] = idx < nwords ? __ldg(src + idx) : 0;
      s1 = __dp4a(w[i], 0x01010101, s1);
      s2 = __dp4a(w[i], w[i], s2);
    }
    s1 = warp_sum(s1);
    s2 = warp_sum(s2);
    const int mu = floordiv_pos(2 * s1 + C, 2 * C);
    // sum (x - mu)^2 = sum x^2 - 2 mu sum x + C mu^2, exactly
    const long long V = (long long)s2 - 2ll * mu * s1 + (long long)C * mu * mu;
    const unsigned sd = isqrt_u32((unsigned)V);
    const int F = sd == 0 ? 0 : (int)((1u << M_ln) / sd);
    int* dst = reinterpret_cast<int*>(out + r * ldout);
#pragma unroll
    for (int i = 0; i < WPL; ++i) {
      const int idx = lane + 32 * i;
      if (idx < nwords) {
        unsigned packed = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const int c = idx * 4 + b;
          const int x = (int)(int8_t)(w[i] >> (8 * b));
          int v = rq((x - mu) * F, gs.m(c), gs.s(c));
          if (beta) v += __ldg(beta + c);
          packed |= (unsigned)(sat8(v) & 0xff) << (8 * b);
        }
        dst[idx] = (int)packed;
      }
    }
  }
}

// Rows of up to 1024 channels.  L lanes share a row (G = 32 / L rows side by side in a warp), a lane holds WPL words of four
// channels of R such rows, and the constants of its channels in registers (inside a forward fetched before the wait for
// the previous kernel).  kExact: C = 4 L WPL, nothing to mask.  Rows past the end are read as the last row and not
// stored: the body has no branch but the one on the form of the constants.  What bounds it is instruction issue: byte,
// multiply-add, mad.hi, shift and half a pack per value, and about 130 instructions for the scalars of G R rows at once.
// With a branch around every word and row and one row per 32 lanes, three of four instructions were overhead.  Measured, back
// to back: 197 x 192 2.4 -> 1.5 us.  (More than 1024 rows, operator
// calls, and rows of 1536 channels: the next kernel.)
// fast: every channel of the warp has s >= 33 and a small beta (see LnConsts): m, sh = s - 32 and add = 2^(sh-1) + beta 2^sh.
template <int WPL>
struct LnLane {
  int m[WPL][4], s[WPL][4], b[WPL][4];
  bool fast;
  // words idx0, idx0 + L, ... of the row
  __device__ __forceinline__ void fetch(const ScaleDev& gs, const int32_t* beta, int nwords, int vec, int idx0, int L) {
    fast = true;
#pragma unroll
    for (int i = 0; i < WPL; ++i) {
      const int idx = idx0 + L * i;
#pragma unroll
      for (int k = 0; k < 4; ++k) { m[i][k] = 1; s[i][k] = 33; b[i][k] = 0; }
      if (idx < nwords) {
        if (vec) {
          const int4 m4 = __ldg(reinterpret_cast<const int4*>(gs.mult_c) + idx);
          const uchar4 s4 = __ldg(reinterpret_cast<const uchar4*>(gs.shift_c) + idx);
          m[i][0] = m4.x; m[i][1] = m4.y; m[i][2] = m4.z; m[i][3] = m4.w;
          s[i][0] = s4.x; s[i][1] = s4.y; s[i][2] = s4.z; s[i][3] = s4.w;
          if (beta) {
            const int4 b4 = __ldg(reinterpret_cast<const int4*>(beta) + idx);
            b[i][0] = b4.x; b[i][1] = b4.y; b[i][2] = b4.z; b[i][3] = b4.w;
          }
        } else {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            m[i][k] = gs.m(idx * 4 + k);
            s[i][k] = gs.s(idx * 4 + k);
            if (beta) b[i][k] = __ldg(beta + idx * 4 + k);
          }
        }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        s[i][k] = clamp_shift(s[i][k]);
        const int sh = s[i][k] - 32;
        fast = fast && sh >= 1 && b[i][k] > -(1 << (29 - sh)) && b[i][k] < (1 << (29 - sh));
      }
    }
    fast = __all_sync(0xffffffffu, fast);
    if (fast) {
#pragma unroll
      for (int i = 0; i < WPL; ++i)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          s[i][k] -= 32;
          b[i][k] = (1 << (s[i][k] - 1)) + b[i][k] * (1 << s[i][k]);
        }
    }
  }
};

// GA = 1: row r is row index[r] of the input (inner: inner[index[r]]), and is also copied to row r of `copy`: a window
// shift or its inverse without a pass of its own.  GA = 2: quarter k of row r is row index[4 r + k] of the input, a quarter
// as wide: the gather of a 2 x 2 patch merging.  Measured, back to back, against a gather kernel in front: a Swin-T forward of 64 images,
// 15 launches fewer, 1492 -> 1452 us.
template <int GA>
struct LnSource {
  const int32_t *index, *inner;
  int8_t* copy;
  int64_t ldcopy;
  __device__ __forceinline__ int row(int r) const {
    const int q = __ldg(index + r);
    return inner ? __ldg(inner + q) : q;
  }
};
template <>
struct LnSource<0> {};

template <int L, int WPL, int R, int PER_SM, bool kExact, int GA = 0>
__global__ void __launch_bounds__(128, PER_SM) layernorm_rows_kernel(const int8_t* __restrict__ in, int64_t ldin, ScaleDev gs,
                                                                     const int32_t* __restrict__ beta, int M_ln,
                                                                     int8_t* __restrict__ out, int64_t ldout, int rows, int C,
                                                                     unsigned mean_magic, int vec, int params, LnSource<GA> source) {
  static_assert(GA == 0 || kExact, "whole rows");
  static_assert(R <= L, "a lane per row for the scalars");
  constexpr int G = 32 / L;
  if (!params) pdl_wait();
  pdl_trigger();
  const int lane = threadIdx.x & 31, li = lane & (L - 1), grp = lane / L;
  const int nwords = kExact ? L * WPL : C >> 2;
  LnLane<WPL> k;
  k.fetch(gs, beta, nwords, vec, li, L);
  pdl_wait();
  const int warp = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int stride = (int)((gridDim.x * blockDim.x) >> 5) * (G * R);
  for (int r0 = warp * (G * R) + grp; r0 - grp < rows; r0 += stride) {
    int w[R][WPL];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int row = min(r0 + r * G, rows - 1);
      if constexpr (GA == 2) {
        constexpr int Q = L * WPL / 4;   // words of a quarter
        int q[WPL];
#pragma unroll
        for (int i = 0; i < WPL; ++i) q[i] = source.row(4 * row + (li + L * i) / Q);
#pragma unroll
        for (int i = 0; i < WPL; ++i) w[r][i] = __ldg(reinterpret_cast<const int*>(in + (int64_t)q[i] * ldin) + (li + L * i) % Q);
      } else {
        int64_t from = row;
        if constexpr (GA == 1) from = source.row(row);
        const int* src = reinterpret_cast<const int*>(in + from * ldin) + li;
#pragma unroll
        for (int i = 0; i < WPL; ++i) w[r][i] = kExact || li + L * i < nwords ? __ldg(src + L * i) : 0;
      }
    }
    if constexpr (GA == 1) {
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int i = 0; i < WPL; ++i)
          if (r0 + r * G < rows) reinterpret_cast<int*>(source.copy + (int64_t)(r0 + r * G) * source.ldcopy)[li + L * i] = w[r][i];
    }
    int my_s1 = 0, my_s2 = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      int s1 = 0, s2 = 0;
#pragma unroll
      for (int i = 0; i < WPL; ++i) {
        s1 = __dp4a(w[r][i], 0x01010101, s1);
        s2 = __dp4a(w[r][i], w[r][i], s2);
      }
      if (L == 32) {
        s1 = __reduce_add_sync(0xffffffffu, s1);
        s2 = __reduce_add_sync(0xffffffffu, s2);
      } else {
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) {
          s1 += __shfl_xor_sync(0xffffffffu, s1, o);
          s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        }
      }
      my_s1 = li == r ? s1 : my_s1;
      my_s2 = li == r ? s2 : my_s2;
    }
    // lane r < R of every group: the scalars of its r-th row (see layernorm_rows)
    const int mu = (int)__umulhi((unsigned)(2 * my_s1 + 257 * C), mean_magic) - 128;
    const unsigned V = (unsigned)(my_s2 - 2 * mu * my_s1 + C * mu * mu);
    const unsigned sd = isqrt26(V);
    const int F = sd == 0 ? 0 : (int)((1u << M_ln) / sd);
    const int muF = (int)((unsigned)mu * (unsigned)F);
    auto rows_out = [&](auto fast) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int Fr = __shfl_sync(0xffffffffu, F, grp * L + r), muFr = __shfl_sync(0xffffffffu, muF, grp * L + r);
        const int row = r0 + r * G;
        int* dst = reinterpret_cast<int*>(out + (int64_t)row * ldout) + li;
#pragma unroll
        for (int i = 0; i < WPL; ++i) {
          int v[4];
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            int xb;   // byte b, sign-extended
            asm("prmt.b32 %0, %1, %1, %2;" : "=r"(xb) : "r"(w[r][i]), "r"(0x8880 + 0x1111 * b));
            // (x - mu) * F modulo 2^32: the difference fits, |y F| <= 2^(M_ln + 1)
            const int yF = (int)((unsigned)xb * (unsigned)Fr - (unsigned)muFr);
            if (decltype(fast)::value) {
              int h;
              asm("mad.hi.s32 %0, %1, %2, %3;" : "=r"(h) : "r"(yF), "r"(k.m[i][b]), "r"(k.b[i][b]));
              v[b] = h >> k.s[i][b];
            } else {
              // (the rare form: constants from global memory, so that they do not take registers from the other)
              const int c = min((li + L * i) * 4 + b, C - 1);
              v[b] = rq(yF, gs.m(c), gs.s(c)) + (beta ? __ldg(beta + c) : 0);
            }
          }
          const int word = (int)pack_sat8_u(v[0], v[1], v[2], v[3]);
          if (row < rows && (kExact || li + L * i < nwords)) dst[L * i] = word;
        }
      }
    };
    if (k.fast) rows_out(std::true_type{});
    else rows_out(std::false_type{});
  }
}

// The same with the constants in shared memory, fetched once per word and R rows: the registers go to rows,
// so that most launches are one or two passes, and twice the warps are in flight.  Bound by issue and by the chain of the
// scalars of a pass.  Measured, back to back, against constants in registers: 18464 x 1024 12.4 -> 9.5 us, 9232 x 1024 8.4 ->
// 5.4, 25216 x 768 11.3 -> 10.6, 12608 x 768 7.1 -> 5.8, 12608 x 384 4.2 -> 3.7, 3136 x 1536 9.0 -> 4.2, 12544 x 192
// 3.65 -> 3.1, 200704 x 96 12.4 -> 11.9; with words masked 25216 x 640 17.4 -> 9.8, 25216 x 304 9.4 -> 7.0.  (As operator
// calls, whose constants are fetched behind the wait, about 0.6 us more: 25216 x 768 10.8, 2500 x 768 2.7 -> 3.3.)
template <int L, int WPL, int R, bool kExact, int GA = 0>
__global__ void __launch_bounds__(256, 2) layernorm_shared_rows_kernel(const int8_t* __restrict__ in, int64_t ldin, ScaleDev gs,
                                                                            const int32_t* __restrict__ beta, int M_ln,
                                                                            int8_t* __restrict__ out, int64_t ldout, int rows, int C,
                                                                            unsigned mean_magic, int vec, int params, LnSource<GA> source) {
  static_assert(GA == 0 || kExact, "whole rows");
  static_assert(R <= L, "a lane per row for the scalars");
  constexpr int G = 32 / L, kWords = L * WPL;
  const int nwords = kExact ? kWords : C >> 2;
  __shared__ int4 sm_m[kWords], sm_s[kWords], sm_b[kWords];
  if (!params) pdl_wait();
  pdl_trigger();
  const int lane = threadIdx.x & 31, li = lane & (L - 1), grp = lane / L;
  const bool fast = __syncthreads_and(ln_stage_consts(gs, beta, nwords, vec, sm_m, sm_s, sm_b, threadIdx.x, 256)) != 0;
  if (fast) ln_fold_consts(nwords, sm_s, sm_b, threadIdx.x, 256);
  __syncthreads();
  pdl_wait();
  const int warp = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int stride = (int)((gridDim.x * blockDim.x) >> 5) * (G * R);
  for (int r0 = warp * (G * R) + grp; r0 - grp < rows; r0 += stride) {
    int w[R][WPL];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int row = min(r0 + r * G, rows - 1);
      if constexpr (GA == 2) {
        constexpr int Q = kWords / 4;   // words of a quarter
        int q[WPL];
#pragma unroll
        for (int i = 0; i < WPL; ++i) q[i] = source.row(4 * row + (li + L * i) / Q);
#pragma unroll
        for (int i = 0; i < WPL; ++i) w[r][i] = __ldg(reinterpret_cast<const int*>(in + (int64_t)q[i] * ldin) + (li + L * i) % Q);
      } else {
        int64_t from = row;
        if constexpr (GA == 1) from = source.row(row);
        const int* src = reinterpret_cast<const int*>(in + from * ldin) + li;
#pragma unroll
        for (int i = 0; i < WPL; ++i) w[r][i] = kExact || li + L * i < nwords ? __ldg(src + L * i) : 0;
      }
    }
    if constexpr (GA == 1) {
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int i = 0; i < WPL; ++i)
          if (r0 + r * G < rows) reinterpret_cast<int*>(source.copy + (int64_t)(r0 + r * G) * source.ldcopy)[li + L * i] = w[r][i];
    }
    int my_s1 = 0, my_s2 = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      int s1 = 0, s2 = 0;
#pragma unroll
      for (int i = 0; i < WPL; ++i) {
        s1 = __dp4a(w[r][i], 0x01010101, s1);
        s2 = __dp4a(w[r][i], w[r][i], s2);
      }
      if (L == 32) {
        s1 = __reduce_add_sync(0xffffffffu, s1);
        s2 = __reduce_add_sync(0xffffffffu, s2);
      } else {
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) {
          s1 += __shfl_xor_sync(0xffffffffu, s1, o);
          s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        }
      }
      my_s1 = li == r ? s1 : my_s1;
      my_s2 = li == r ? s2 : my_s2;
    }
    const int mu = (int)__umulhi((unsigned)(2 * my_s1 + 257 * C), mean_magic) - 128;
    const unsigned V = (unsigned)(my_s2 - 2 * mu * my_s1 + C * mu * mu);
    const unsigned sd = isqrt26(V);
    const int F = sd == 0 ? 0 : (int)((1u << M_ln) / sd);
    const int muF = (int)((unsigned)mu * (unsigned)F);
    int Fr[R], muFr[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      Fr[r] = __shfl_sync(0xffffffffu, F, grp * L + r);
      muFr[r] = __shfl_sync(0xffffffffu, muF, grp * L + r);
    }
    int* dst = reinterpret_cast<int*>(out + (int64_t)r0 * ldout) + li;
    auto rows_out = [&](auto is_fast) {
#pragma unroll
      for (int i = 0; i < WPL; ++i) {
        if (!kExact && li + L * i >= nwords) break;
        const int4 m4 = sm_m[li + L * i], s4 = sm_s[li + L * i], b4 = sm_b[li + L * i];
        const int m[4] = {m4.x, m4.y, m4.z, m4.w}, sh[4] = {s4.x, s4.y, s4.z, s4.w}, be[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
        for (int r = 0; r < R; ++r) {
          int v[4];
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            int xb;   // byte b, sign-extended
            asm("prmt.b32 %0, %1, %1, %2;" : "=r"(xb) : "r"(w[r][i]), "r"(0x8880 + 0x1111 * b));
            const int yF = (int)((unsigned)xb * (unsigned)Fr[r] - (unsigned)muFr[r]);   // modulo 2^32, see layernorm_rows_kernel
            if (decltype(is_fast)::value) {
              int h;
              asm("mad.hi.s32 %0, %1, %2, %3;" : "=r"(h) : "r"(yF), "r"(m[b]), "r"(be[b]));
              v[b] = h >> sh[b];
            } else {
              v[b] = rq(yF, m[b], sh[b]) + be[b];
            }
          }
          const int word = (int)pack_sat8_u(v[0], v[1], v[2], v[3]);
          if (r0 + r * G < rows) reinterpret_cast<int*>(reinterpret_cast<int8_t*>(dst) + (int64_t)(r * G) * ldout)[L * i] = word;
        }
      }
    };
    if (fast) rows_out(std::true_type{});
    else rows_out(std::false_type{});
  }
}

// Any C (multiple of 4): the row is read again from cache for the output pass.
__global__ void __launch_bounds__(256) layernorm_i8_long_kernel(const int8_t* __restrict__ in, int64_t ldin,
                                                                ScaleDev gs, const int32_t* __restrict__ beta,
                                                                int M_ln, int8_t* __restrict__ out,
                                                                int64_t ldout, int64_t rows, int C) {
  pdl_wait();
  pdl_trigger();   // (after the wait: it may be the first kernel of a forward)
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int nwords = C >> 2;
  for (int64_t r = warp; r < rows; r += nwarps) {
    const int* src = reinterpret_cast<const int*>(in + r * ldin);
    int s1 = 0, s2 = 0;
    for (int idx = lane; idx < nwords; idx += 32) {
      const int w = __ldg(src + idx);
      s1 = __dp4a(w, 0x01010101, s1);
      s2 = __dp4a(w, w, s2);
    }
    s1 = warp_sum(s1);
    s2 = warp_sum(s2);
    const int mu = floordiv_pos(2 * s1 + C, 2 * C);
    const long long V = (long long)s2 - 2ll * mu * s1 + (long long)C * mu * mu;
    const unsigned sd = isqrt_u32((unsigned)V);
    const int F = sd == 0 ? 0 : (int)((1u << M_ln) / sd);
    int* dst = reinterpret_cast<int*>(out + r * ldout);
    for (int idx = lane; idx < nwords; idx += 32) {
      const int w = __ldg(src + idx);
      unsigned packed = 0;
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int c = idx * 4 + b;
        const int x = (int)(int8_t)(w >> (8 * b));
        int v = rq((x - mu) * F, gs.m(c), gs.s(c));
        if (beta) v += __ldg(beta + c);
        packed |= (unsigned)(sat8(v) & 0xff) << (8 * b);
      }
      dst[idx] = (int)packed;
    }
  }
}

// int32 input (|x| <= 2^20): 64-bit sums, two passes over the row.
__global__ void __launch_bounds__(256) layernorm_i32_kernel(const int32_t* __restrict__ in, int64_t ldin,
                                                            ScaleDev gs, const int32_t* __restrict__ beta,
                                                            int M_ln, int8_t* __restrict__ out, int64_t ldout,
                                                            int64_t rows, int C) {
  pdl_wait();
  pdl_trigger();   // (after the wait: it may be the first kernel of a forward)
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r = warp; r < rows; r += nwarps) {
    const int32_t* src = in + r * ldin;
    long long s1 = 0;
    for (int c = lane; c < C; c += 32) s1 += __ldg(src + c);
    s1 = warp_sum_ll(s1);
    const long long num = 2 * s1 + C, den = 2ll * C;
    long long mu = num / den;
    if (num - mu * den < 0) mu -= 1;
    long long V = 0;
    for (int c = lane; c < C; c += 32) {
      const long long y = (long long)__ldg(src + c) - mu;
      V += y * y;
    }
    V = warp_sum_ll(V);
    const unsigned long long sd = isqrt_u64((unsigned long long)V);
    const long long F = sd == 0 ? 0 : (long long)((1ull << M_ln) / sd);
    for (int c = lane; c < C; c += 32) {
      const long long y = (long long)__ldg(src + c) - mu;
      int v = rq((int)(y * F), gs.m(c), gs.s(c));
      if (beta) v += __ldg(beta + c);
      out[r * ldout + c] = (int8_t)sat8(v);
    }
  }
}

// layernorm_rows_kernel for int8 rows of C channels; false: no form for that width.
template <int GA>
static bool layernorm_rows(ivit_ctx* ctx, const int8_t* x, int64_t ldin, ScaleDev gs, const int32_t* beta, int M_ln, int8_t* out,
                           int64_t ldout, int64_t rows, int64_t C, bool params, LnSource<GA> source) {
  if (rows >= (1ll << 31) / (GA == 2 ? 4 : 1) - (1 << 20)) return false;
  const int wpl = (int)((C / 4 + 31) / 32);
  const unsigned magic = (unsigned)(0x100000000ull / (unsigned long long)(2 * C)) + 1u;
  const int vec = gs.mult_c && gs.shift_c && !(reinterpret_cast<uintptr_t>(gs.mult_c) & 15) && !(reinterpret_cast<uintptr_t>(gs.shift_c) & 3) &&
                  !(reinterpret_cast<uintptr_t>(beta) & 15);
  // (rpw: rows of a warp and pass)
  auto run = [&](auto kernel, int rpw, int per_sm) {
    const int64_t blocks = (rows + 4 * rpw - 1) / (4 * rpw), cap = (int64_t)ctx->sm_count * per_sm;
    launch_k(kernel, dim3((unsigned)(blocks < cap ? blocks : cap)), dim3(128), 0, ctx->stream, x, ldin, gs, beta, M_ln, out, ldout, (int)rows,
             (int)C, magic, vec, (int)params, source);
  };
  // Up to 1024 rows of a forward one row per group of lanes, constants in registers: with so few rows the chain of one warp
  // counts (788 x 384: 1.9 us, shared constants 2.6; 197 x 192: 1.45, four rows 1.8).  Not where the constants are
  // fetched behind the wait: every warp would wait for copies of its own (400 x 768 as an operator call 4.5 us, shared 2.6).
  const bool few = rows <= 1024 && params;
  // Beyond: constants in shared memory, two blocks per SM, and as many rows per warp
  // as make passes x (1 + rows) least, a pass costing about that (12608 x 384, 5.3 rows per warp: six rows 3.7 us, four 4.9,
  // eight 4.6; 4590 x 384, 1.9 rows per warp: two rows 2.8, six 3.3; 18464 x 1024, 7.8: four rows 9.5, six 10.9).
  const int64_t warps = (int64_t)ctx->sm_count * 16;
  auto pick = [&](std::initializer_list<int> offered, int64_t side = 1) {   // side: rows side by side in a warp
    int best = 0;
    int64_t best_cost = 0;
    for (int r : offered) {
      const int64_t cost = (rows + r * side * warps - 1) / (r * side * warps) * (1 + r);
      if (!best || cost < best_cost) { best = r; best_cost = cost; }
    }
    return best;
  };
  auto shared = [&](auto kernel, int rpw) {
    const int64_t blocks = (rows + 8 * rpw - 1) / (8 * rpw), cap = (int64_t)ctx->sm_count * 2;
    launch_k(kernel, dim3((unsigned)(blocks < cap ? blocks : cap)), dim3(256), 0, ctx->stream, x, ldin, gs, beta, M_ln, out, ldout, (int)rows,
             (int)C, magic, vec, (int)params, source);
  };
  auto up_to_six = [&](auto two, auto four, auto six, int side = 1) {
    const int r = pick({6, 4, 2}, side);
    if (r == 6) shared(six, 6 * side);
    else if (r == 4) shared(four, 4 * side);
    else shared(two, 2 * side);
  };
  switch (C) {
    case 96:
      if (GA == 2) return false;
      if constexpr (GA != 2) {
        if (few) run(layernorm_rows_kernel<8, 3, 1, 5, true, GA>, 4, 5);
        else up_to_six(layernorm_shared_rows_kernel<8, 3, 2, true, GA>, layernorm_shared_rows_kernel<8, 3, 4, true, GA>, layernorm_shared_rows_kernel<8, 3, 6, true, GA>, 4);
      }
      return true;
    case 192:
      if (GA == 2) return false;
      if constexpr (GA != 2) {
        if (few) run(layernorm_rows_kernel<16, 3, 1, 5, true, GA>, 2, 5);
        else up_to_six(layernorm_shared_rows_kernel<16, 3, 2, true, GA>, layernorm_shared_rows_kernel<16, 3, 4, true, GA>, layernorm_shared_rows_kernel<16, 3, 6, true, GA>, 2);
      }
      return true;
    case 384:
      if (few) run(layernorm_rows_kernel<32, 3, 1, 5, true, GA>, 1, 5);
      else up_to_six(layernorm_shared_rows_kernel<32, 3, 2, true, GA>, layernorm_shared_rows_kernel<32, 3, 4, true, GA>, layernorm_shared_rows_kernel<32, 3, 6, true, GA>);
      return true;
    case 512:
      if (few) run(layernorm_rows_kernel<32, 4, 1, 4, true, GA>, 1, 4);
      else up_to_six(layernorm_shared_rows_kernel<32, 4, 2, true, GA>, layernorm_shared_rows_kernel<32, 4, 4, true, GA>, layernorm_shared_rows_kernel<32, 4, 6, true, GA>);
      return true;
    case 768:
      if (few) run(layernorm_rows_kernel<32, 6, 1, 4, true, GA>, 1, 4);
      else up_to_six(layernorm_shared_rows_kernel<32, 6, 2, true, GA>, layernorm_shared_rows_kernel<32, 6, 4, true, GA>, layernorm_shared_rows_kernel<32, 6, 6, true, GA>);
      return true;
    case 1024:
      if (few) run(layernorm_rows_kernel<32, 8, 1, 3, true, GA>, 1, 3);
      else if (pick({4, 2}) == 4) shared(layernorm_shared_rows_kernel<32, 8, 4, true, GA>, 4);
      else shared(layernorm_shared_rows_kernel<32, 8, 2, true, GA>, 2);
      return true;
    case 1536: shared(layernorm_shared_rows_kernel<32, 12, 2, true, GA>, 2); return true;
  }
  if constexpr (GA == 0) {   // other widths: the words past the row masked
    if (few) {
      if (wpl <= 1) run(layernorm_rows_kernel<32, 1, 8, 10, false>, 8, 10);
      else if (wpl <= 2) run(layernorm_rows_kernel<32, 2, 4, 8, false>, 4, 8);
      else if (wpl <= 4) run(layernorm_rows_kernel<32, 4, 4, 5, false>, 4, 5);
      else if (wpl <= 8) run(layernorm_rows_kernel<32, 8, 2, 3, false>, 2, 3);
      else return false;
      return true;
    }
    auto masked = [&](auto w) {
      constexpr int W = decltype(w)::value;
      if constexpr (W <= 6) {
        up_to_six(layernorm_shared_rows_kernel<32, W, 2, false>, layernorm_shared_rows_kernel<32, W, 4, false>, layernorm_shared_rows_kernel<32, W, 6, false>);
      } else {
        if (pick({4, 2}) == 4) shared(layernorm_shared_rows_kernel<32, W, 4, false>, 4);
        else shared(layernorm_shared_rows_kernel<32, W, 2, false>, 2);
      }
      return true;
    };
    switch (wpl) {
      case 1: return masked(std::integral_constant<int, 1>{});
      case 2: return masked(std::integral_constant<int, 2>{});
      case 3: return masked(std::integral_constant<int, 3>{});
      case 4: return masked(std::integral_constant<int, 4>{});
      case 5: return masked(std::integral_constant<int, 5>{});
      case 6: return masked(std::integral_constant<int, 6>{});
      case 7: return masked(std::integral_constant<int, 7>{});
      case 8: return masked(std::integral_constant<int, 8>{});
    }
  }
  return false;
}

int launch_layernorm(ivit_ctx* ctx, const void* in, int in_dtype, int64_t ldin, ScaleDev gs,
                     const int32_t* beta, int M_ln, int8_t* out, int64_t ldout, int64_t rows, int64_t C, bool params) {
  if (rows == 0) return IVIT_OK;
  const int threads = 256, wpb = threads / 32;
  const int64_t want = (rows + wpb - 1) / wpb;
  const int grid = (int)(want < (int64_t)ctx->sm_count * 8 ? want : (int64_t)ctx->sm_count * 8);
  cudaStream_t st = ctx->stream;
  LaunchScope ls(ctx, KIND_LAYERNORM, (double)rows * (double)C * (in_dtype == IVIT_I32 ? 5.0 : 2.0));
  if (in_dtype == IVIT_I32) {
    launch_k(layernorm_i32_kernel, dim3(grid), dim3(threads), 0, st, (const int32_t*)in, ldin, gs, beta, M_ln, out, ldout, rows, (int)C);
    return ls.done();
  }
  const int8_t* x = (const int8_t*)in;
  const int wpl = (int)((C / 4 + 31) / 32);
  if (layernorm_rows<0>(ctx, x, ldin, gs, beta, M_ln, out, ldout, rows, C, params, LnSource<0>{})) return ls.done();
  if (wpl <= 12) launch_k(layernorm_i8_kernel<12>, dim3(grid), dim3(threads), 0, st, x, ldin, gs, beta, M_ln, out, ldout, rows, (int)C);
  else launch_k(layernorm_i8_long_kernel, dim3(grid), dim3(threads), 0, st, x, ldin, gs, beta, M_ln, out, ldout, rows, (int)C);
  return ls.done();
}

int launch_layernorm_gather(ivit_ctx* ctx, const int8_t* in, int64_t ldin, const int32_t* index, const int32_t* inner, bool quarters,
                            ScaleDev gs, const int32_t* beta, int M_ln, int8_t* copy, int64_t ldcopy, int8_t* out, int64_t ldout,
                            int64_t rows, int64_t C) {
  if (rows == 0) return IVIT_OK;
  LaunchScope ls(ctx, KIND_LAYERNORM, (double)rows * (double)C * (quarters ? 2.0 : 3.0));
  const bool done = quarters ? layernorm_rows<2>(ctx, in, ldin, gs, beta, M_ln, out, ldout, rows, C, true, LnSource<2>{index, inner, nullptr, 0})
                             : layernorm_rows<1>(ctx, in, ldin, gs, beta, M_ln, out, ldout, rows, C, true, LnSource<1>{index, inner, copy, ldcopy});
  return done ? ls.done() : IVIT_ERR_UNSUPPORTED;
}

bool layernorm_gathers(int64_t rows, int64_t C, bool quarters) {
  return rows < (1ll << 31) / 4 - (1 << 20) &&
         (C == 384 || C == 512 || C == 768 || C == 1024 || C == 1536 || (!quarters && (C == 96 || C == 192)));
}

// ------------------------------------------------------------------ Shiftmax

// Packed int8x4 word `idx` of row r.  I8: straight from memory.  I32: requantise four
// accumulators (+ bias) to int8 first, so both entry forms run the same row algorithm.
template <bool FROM_I32>
struct RowLoader {
  const void* in;
  int64_t ldin;
  const int32_t* bias32;
  int64_t ldbias, bias_rows;
  int pre_m, pre_s;
  __device__ __forceinline__ int load(int64_t r, int idx) const {
    if (!FROM_I32) {
      return __ldg(reinterpret_cast<const int*>((const int8_t*)in + r * ldin) + idx);
    } else {
      const int4 a = __ldg(reinterpret_cast<const int4*>((const int32_t*)in + r * ldin) + idx);
      int4 b = make_int4(0, 0, 0, 0);
      if (bias32) b = __ldg(reinterpret_cast<const int4*>(bias32 + (r % bias_rows) * ldbias) + idx);
      unsigned p = (unsigned)(sat8(rq(a.x + b.x, pre_m, pre_s)) & 0xff);
      p |= (unsigned)(sat8(rq(a.y + b.y, pre_m, pre_s)) & 0xff) << 8;
      p |= (unsigned)(sat8(rq(a.z + b.z, pre_m, pre_s)) & 0xff) << 16;
      p |= (unsigned)(sat8(rq(a.w + b.w, pre_m, pre_s)) & 0xff) << 24;
      return (int)p;
    }
  }
};

// Rows of up to 2048 values.  L lanes share a row (32 / L rows side by side in a warp); a lane holds WPL words of four
// values, their exponentials stay in registers between the row sum and the output.  Look-ups, reciprocal and
// probabilities as in the attention kernels (shiftmax.cuh).  Positions past d hold -128: they never win the maximum, their
// exponentials are taken out of the sum again, and their probabilities are masked.
// FAST: k_out = 8, I0 2^N > 2^15 and (int32 input) a shift >= 33 in front; otherwise the general arithmetic.
// What bounds it: instruction issue (about nine instructions per value, two of them multiply-highs with int32 input).
// Measured, back to back (before: a warp per row, one table, byte permutes, a 64-bit division per row): int32 18464 x 577
// 17.8 -> 9.3 us (5.7 TB/s), 75648 x 197 33.4 -> 12.6, 200000 x 49 50.4 -> 14.3; int8 75648 x 197 17.5 -> 9.5.
template <int L, int WPL, bool FROM_I32, bool FAST>
__global__ void __launch_bounds__(512, WPL > 8 ? 1 : 2) shiftmax_rows_kernel(RowLoader<FROM_I32> ld, ivit_exp_params p, int cp,
                                                               int8_t* __restrict__ out, int64_t ldout, int rows, int d) {
  extern __shared__ __align__(128) uint8_t sm_tab[];   // [256 x cp][128 seeds of the reciprocal]
  constexpr int G = 32 / L;
  pdl_trigger();
  build_exp_table(p.I0, p.N, cp, sm_tab, threadIdx.x, blockDim.x);
  unsigned* seeds = reinterpret_cast<unsigned*>(sm_tab + 1024 * cp);
  if (threadIdx.x < 128) seeds[threadIdx.x] = recip_seed(threadIdx.x);
  __syncthreads();
  const int lane = threadIdx.x & 31, li = lane & (L - 1), grp = lane / L;
  const int nwords = (d + 3) >> 2, nwords_out = ((d + 15) >> 4) << 2;
  uint32_t mask[WPL];   // bytes of this lane's words that hold values
#pragma unroll
  for (int i = 0; i < WPL; ++i) {
    const int left = d - 4 * (li + L * i);
    mask[i] = left >= 4 ? 0xffffffffu : (left <= 0 ? 0u : 0xffffffffu >> (8 * (4 - left)));
  }
  uint32_t sel[4];
#pragma unroll
  for (int b = 0; b < 4; ++b) sel[b] = exp_sel(cp, b);
  const uint32_t tab_lane = (uint32_t)__cvta_generic_to_shared(sm_tab) + 4u * (unsigned)(lane & (cp - 1));
  const unsigned top = (unsigned)p.I0 << p.N;
  const int osh = 14 - p.k_out, omax = (1 << (p.k_out - 1)) - 1;
  const int rnd = FROM_I32 && FAST ? 1 << (ld.pre_s - 33) : 0, sh = ld.pre_s - 32;
  pdl_wait();
  const int warp = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), stride = (int)((gridDim.x * blockDim.x) >> 5) * G;
  for (int r0 = warp * G; r0 < rows; r0 += stride) {
    const bool row_ok = r0 + grp < rows;
    const int r = row_ok ? r0 + grp : rows - 1;   // (a row past the end repeats the last one, not stored)
    uint32_t x[WPL];
    if (FROM_I32) {
      const int4* src = reinterpret_cast<const int4*>((const int32_t*)ld.in + (int64_t)r * ld.ldin) + li;
      int4 a[WPL];
#pragma unroll
      for (int i = 0; i < WPL; ++i) a[i] = li + L * i < nwords ? __ldg(src + L * i) : make_int4(0, 0, 0, 0);
      if (ld.bias32) {
        const int4* bs = reinterpret_cast<const int4*>(ld.bias32 + (int64_t)((unsigned)r % (unsigned)ld.bias_rows) * ld.ldbias) + li;
#pragma unroll
        for (int i = 0; i < WPL; ++i)
          if (li + L * i < nwords) {
            const int4 b = __ldg(bs + L * i);
            a[i].x += b.x; a[i].y += b.y; a[i].z += b.z; a[i].w += b.w;
          }
      }
#pragma unroll
      for (int i = 0; i < WPL; ++i) {
        int v[4] = {a[i].x, a[i].y, a[i].z, a[i].w};
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          if (FAST) {
            asm("mad.hi.s32 %0, %0, %1, %2;" : "+r"(v[b]) : "r"(ld.pre_m), "r"(rnd));
            v[b] >>= sh;
          } else {
            v[b] = rq(v[b], ld.pre_m, ld.pre_s);
          }
        }
        x[i] = pack_sat8_u(v[0], v[1], v[2], v[3]);
      }
    } else {
      const uint32_t* src = reinterpret_cast<const uint32_t*>((const int8_t*)ld.in + (int64_t)r * ld.ldin) + li;
#pragma unroll
      for (int i = 0; i < WPL; ++i) x[i] = li + L * i < nwords ? __ldg(src + L * i) : 0u;
    }
    // row maximum: pairs of 16-bit values whose upper bytes are bytes 3 and 1, or 2 and 0 (the lower bytes only break ties)
    unsigned m31 = 0x80808080u, m20 = 0x80808080u;
#pragma unroll
    for (int i = 0; i < WPL; ++i) {
      x[i] = (x[i] & mask[i]) | (0x80808080u & ~mask[i]);
      m31 = __vmaxs2(m31, x[i]);
      m20 = __vmaxs2(m20, x[i] << 8);
    }
    const unsigned m = __vmaxs2(m31, m20);
    int mx = max((int)m >> 24, (int)(m << 16) >> 24);
    if (L == 32) {
      mx = __reduce_max_sync(0xffffffffu, mx);
    } else {
#pragma unroll
      for (int o = L / 2; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    // ShiftExp(I - I_max), row sum
    const uint32_t tmx = tab_lane + (uint32_t)(4 * cp * mx);
    unsigned e[WPL][4], sum = 0;
#pragma unroll
    for (int i = 0; i < WPL; ++i) {
#pragma unroll
      for (int b = 0; b < 4; ++b) e[i][b] = exp_entry(x[i], sel[b], tmx);
      sum += (e[i][0] + e[i][1]) + (e[i][2] + e[i][3]);
    }
    if (L == 32) {
      sum = __reduce_add_sync(0xffffffffu, sum);
    } else {
#pragma unroll
      for (int o = L / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    }
    sum -= (unsigned)(4 * L * WPL - d) * exp_entry(0x80u, sel[0], tmx);
    // Eq. (IntDiv) with M = 45
    const unsigned factor = FAST ? prob_factor4(sum, top, seeds) : (unsigned)((1ull << 45) / (unsigned long long)sum);
    uint32_t* dst = reinterpret_cast<uint32_t*>(out + (int64_t)r * ldout) + li;
#pragma unroll
    for (int i = 0; i < WPL; ++i) {
      uint32_t o;
      if (FAST) {
        o = prob_word8(factor, (int)e[i][0], (int)e[i][1], (int)e[i][2], (int)e[i][3]);
      } else {
        int q[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) q[b] = min((int)(__umulhi(factor, e[i][b]) >> osh), omax);
        o = pack_sat8_u(q[0], q[1], q[2], q[3]);
      }
      if (row_ok && li + L * i < nwords_out) dst[L * i] = o & mask[i];
    }
  }
}

// Any d: the row is read again for each pass.  Bytes are handled as biased values u = x + 128 (x ^ 0x80): one byte permute
// yields the table index, ShiftExp(x - max) = tab[(max + 128) - u].  Positions past d hold u = 0 (x = -128).
template <bool FROM_I32>
__global__ void __launch_bounds__(256) shiftmax_kernel(RowLoader<FROM_I32> ld, ivit_exp_params p,
                                                       int8_t* __restrict__ out, int64_t ldout,
                                                       int64_t rows, int d) {
  pdl_trigger();
  pdl_wait();
  __shared__ unsigned exp_tab[256];  // ShiftExp(-i), i = I_max - I in [0, 255]
  for (int i = threadIdx.x; i < 256; i += blockDim.x) exp_tab[i] = shiftexp(-i, p.I0, p.N);
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int nwords = (d + 3) >> 2;
  const int nwords_out = ((d + 15) >> 4) << 2;  // zero-fill up to the next multiple of 16
  const int npad = nwords * 4 - d;              // bytes past d in the last word
  const int iters = (nwords_out + 31) / 32;
  const int osh = 14 - p.k_out, omax = (1 << (p.k_out - 1)) - 1;
  for (int64_t r = warp; r < rows; r += nwarps) {
    // biased word idx of the row: bytes past d (and whole words past the row) read as 0
    auto load_biased = [&](int idx) -> unsigned {
      if (idx >= nwords) return 0u;
      unsigned v = (unsigned)ld.load(r, idx) ^ 0x80808080u;
      if (idx == nwords - 1 && npad) v &= 0xffffffffu >> (8 * npad);
      return v;
    };
    unsigned mxu = 0;
    for (int i = 0; i < iters; ++i) {
      const unsigned v = load_biased(lane + 32 * i);
      mxu = max(max(mxu, __byte_perm(v, 0, 0x4440)), max(__byte_perm(v, 0, 0x4441), max(__byte_perm(v, 0, 0x4442), v >> 24)));
    }
    mxu = __reduce_max_sync(0xffffffffu, mxu);   // biased maximum = I_max + 128
    const uint8_t* tmx = reinterpret_cast<const uint8_t*>(exp_tab) + 4 * mxu;
    auto entries = [&](unsigned v, unsigned (&e)[4]) {
#pragma unroll
      for (int b = 0; b < 4; ++b) e[b] = *reinterpret_cast<const unsigned*>(tmx - 4 * (int)__byte_perm(v, 0, 0x4440 + b));
    };
    unsigned sum = 0;
    for (int i = 0; i < iters; ++i) {
      unsigned e[4];
      entries(load_biased(lane + 32 * i), e);
      sum += (e[0] + e[1]) + (e[2] + e[3]);
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    // every position past d of the 32 * iters words counted exp_tab[I_max + 128]: take them out
    sum -= (unsigned)(32 * iters * 4 - d) * exp_tab[mxu];
    // Eq. (IntDiv) with M = 45: (floor(2^45 / sum) * e) >> (45 - (k_out - 1)) == umulhi(factor, e) >> (14 - k_out)
    const unsigned factor = (unsigned)((1ull << 45) / (unsigned long long)sum);
    int* dst = reinterpret_cast<int*>(out + r * ldout);
    for (int i = 0; i < iters; ++i) {
      const int idx = lane + 32 * i;
      if (idx >= nwords_out) break;
      unsigned e[4];
      entries(load_biased(idx), e);
      unsigned packed = pack_sat8_u(min((int)(__umulhi(factor, e[0]) >> osh), omax), min((int)(__umulhi(factor, e[1]) >> osh), omax),
                                    min((int)(__umulhi(factor, e[2]) >> osh), omax), min((int)(__umulhi(factor, e[3]) >> osh), omax));
      if (idx >= nwords) packed = 0;
      else if (idx == nwords - 1 && npad) packed &= 0xffffffffu >> (8 * npad);
      dst[idx] = (int)packed;
    }
  }
}

template <bool FROM_I32>
static void shiftmax_dispatch(ivit_ctx* ctx, RowLoader<FROM_I32> ld, ivit_exp_params p, int8_t* out, int64_t ldout,
                              int64_t rows, int d) {
  const int words = (d + 15) / 16 * 4;
  if (words > 512 || rows >= (1ll << 31) - (1 << 20) || (FROM_I32 && ld.bias_rows >= (1ll << 31))) {
    const int64_t want = (rows + 7) / 8, cap = (int64_t)ctx->sm_count * 8;
    launch_k(shiftmax_kernel<FROM_I32>, dim3((unsigned)(want < cap ? want : cap)), dim3(256), 0, ctx->stream, ld, p, out, ldout, rows, d);
    return;
  }
  const bool fast = p.k_out == 8 && ((int64_t)p.I0 << p.N) > (1 << 15) && (!FROM_I32 || ld.pre_s >= 33);
  // G rows per warp.  Two blocks of sixteen warps per SM with a table copy per lane; few rows: small blocks on more SMs and
  // fewer copies to build.
  auto run = [&](auto kernel, int G) {
    const bool few = rows <= (int64_t)ctx->sm_count * 16 * G;
    const int threads = few ? 128 : 512, cp = few ? 8 : 32;
    const int64_t per_block = (int64_t)(threads / 32) * G, want = (rows + per_block - 1) / per_block, cap = (int64_t)ctx->sm_count * (few ? 8 : (words > 256 ? 1 : 2));
    launch_k(kernel, dim3((unsigned)(want < cap ? want : cap)), dim3(threads), (size_t)(1024 * cp + 512), ctx->stream, ld, p, cp, out, ldout,
             (int)rows, d);
  };
  auto pick = [&](auto f) {
    constexpr bool F = decltype(f)::value;
    if (words <= 16) run(shiftmax_rows_kernel<8, 2, FROM_I32, F>, 4);
    else if (words <= 32) run(shiftmax_rows_kernel<8, 4, FROM_I32, F>, 4);
    else if (words <= 56) run(shiftmax_rows_kernel<8, 7, FROM_I32, F>, 4);
    else if (words <= 96) run(shiftmax_rows_kernel<16, 6, FROM_I32, F>, 2);
    else if (words <= 160) run(shiftmax_rows_kernel<32, 5, FROM_I32, F>, 1);
    else if (words <= 256) run(shiftmax_rows_kernel<32, 8, FROM_I32, F>, 1);
    else run(shiftmax_rows_kernel<32, 16, FROM_I32, F>, 1);
  };
  if (fast) pick(std::true_type{});
  else pick(std::false_type{});
}

int launch_shiftmax(ivit_ctx* ctx, const void* in, int in_dtype, int64_t ldin, const int32_t* bias32,
                    int64_t ldbias, int64_t bias_rows, ScaleDev pre, ivit_exp_params p, int8_t* out,
                    int64_t ldout, int64_t rows, int64_t d) {
  if (rows == 0) return IVIT_OK;
  LaunchScope ls(ctx, KIND_SHIFTMAX, (double)rows * (double)d * (in_dtype == IVIT_I32 ? 5.0 : 2.0));
  if (in_dtype == IVIT_I8) {
    RowLoader<false> ld{in, ldin, nullptr, 0, 1, 0, 1};
    shiftmax_dispatch<false>(ctx, ld, p, out, ldout, rows, (int)d);
  } else {
    RowLoader<true> ld{in, ldin, bias32, ldbias, bias_rows < 1 ? 1 : bias_rows, pre.mult, clamp_shift(pre.shift)};
    shiftmax_dispatch<true>(ctx, ld, p, out, ldout, rows, (int)d);
  }
  return ls.done();
}

// ------------------------------------------------------------------ Shiftmax on int32 scores (Algorithm 1, wide form)

struct DirectConsts {
  unsigned I0;
  int N;
  int osh;                       // M - (k_out - 1)
  int omax;                      // 2^(k_out-1) - 1
  int M;
  unsigned long long magic;      // reciprocal of I0 scaled by 2^64, rounded up (unused when I0 == 1)
  unsigned long long zero_from;  // I0 * (N + 29): from here on every bit of I_b < 2^29 is shifted out
  // 32-bit form (taken when exponentials, their sum and the reciprocal all fit 32 bits and zero_from <= 2^31)
  unsigned nd_cut;               // I_max - I >= nd_cut implies -I_p >= zero_from; below it -I_p fits 32 bits
  unsigned m_hi, m_lo;           // the two words of magic
};

// ShiftExp(I - I_max) for nd = I_max - I (0 .. 2^32 - 1).  The arithmetic shifts of the negative I_delta round
// towards -inf, so -I_p = nd + ceil(nd / 2) - ceil(nd / 16).  Below zero_from the quotient by I0 is < 53 and
// (-I_p) * I0 < 2^64, which makes the multiply-high by floor(2^64 / I0) + 1 the exact floor quotient.
__device__ __forceinline__ unsigned long long shiftexp_wide(unsigned nd, const DirectConsts& c) {
  const unsigned up2 = (nd >> 1) + (nd & 1u);
  const unsigned up16 = (nd >> 4) + ((nd & 15u) != 0u);
  const unsigned long long n = (unsigned long long)nd + up2 - up16;
  if (n >= c.zero_from) return 0ull;
  const unsigned q = c.I0 == 1u ? (unsigned)n : (unsigned)__umul64hi(n, c.magic);
  const unsigned r = (unsigned)(n - (unsigned long long)q * c.I0);   // 0 <= r < I0
  const unsigned Ib = c.I0 - ((r + 1) >> 1);                         // ((-r) >> 1) + I0
  return q <= (unsigned)c.N ? (unsigned long long)Ib << (c.N - q) : (unsigned long long)(Ib >> (q - c.N));
}

// The same in 32-bit arithmetic: the quotient is the high word of n * magic, taken from two 32-bit products.
__device__ __forceinline__ unsigned shiftexp_narrow(unsigned nd, const DirectConsts& c) {
  if (nd >= c.nd_cut) return 0u;
  const unsigned n = nd + ((nd >> 1) + (nd & 1u)) - ((nd >> 4) + ((nd & 15u) != 0u));
  if (n >= (unsigned)c.zero_from) return 0u;
  const unsigned q = c.I0 == 1u ? n : (unsigned)(((unsigned long long)n * c.m_hi + __umulhi(n, c.m_lo)) >> 32);
  const unsigned r = n - q * c.I0;
  const unsigned Ib = c.I0 - ((r + 1) >> 1);
  return q <= (unsigned)c.N ? Ib << (c.N - q) : Ib >> (q - c.N);
}

__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// One warp per row.  WPL groups of four scores per lane stay in registers as their exponentials
// (d <= 128 * WPL); WPL == 0 reads the row three times instead.
// NARROW: every exponential, the row sum and the reciprocal fit 32 bits (checked by the launcher).
template <int WPL, bool NARROW>
__global__ void __launch_bounds__(256) shiftmax_direct_kernel(const int32_t* __restrict__ in, int64_t ldin,
                                                              DirectConsts c, int8_t* __restrict__ out,
                                                              int64_t ldout, int64_t rows, int d) {
  pdl_trigger();
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int ngroups = (d + 3) >> 2;                // int4 groups that hold scores
  const int nwords_out = ((d + 15) >> 4) << 2;     // output words, zero-filled up to the next multiple of 16 columns
  constexpr int W = WPL > 0 ? WPL : 1;
  const int iters = WPL > 0 ? WPL : (nwords_out + 31) / 32;
  for (int64_t r = warp; r < rows; r += nwarps) {
    const int4* src = reinterpret_cast<const int4*>(in + r * ldin);
    // pass 1: row maximum (positions past d never count)
    int mx = INT_MIN;
    int4 x[W];
#pragma unroll
    for (int i = 0; i < iters; ++i) {
      const int g = lane + 32 * i;
      int4 v = make_int4(INT_MIN, INT_MIN, INT_MIN, INT_MIN);
      if (g < ngroups) {
        v = __ldg(src + g);
        if (4 * g + 1 >= d) v.y = INT_MIN;
        if (4 * g + 2 >= d) v.z = INT_MIN;
        if (4 * g + 3 >= d) v.w = INT_MIN;
      }
      if (WPL > 0) x[i] = v;
      mx = max(max(mx, max(v.x, v.y)), max(v.z, v.w));
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    // exponentials of group g (0 for positions past d)
    using E = typename std::conditional<NARROW, unsigned, unsigned long long>::type;
    auto one = [&](int v) -> E {
      if constexpr (NARROW) return shiftexp_narrow((unsigned)mx - (unsigned)v, c);
      else return shiftexp_wide((unsigned)mx - (unsigned)v, c);
    };
    auto exps = [&](int g, const int4& v, E* e) {
      e[0] = 4 * g + 0 < d ? one(v.x) : (E)0;
      e[1] = 4 * g + 1 < d ? one(v.y) : (E)0;
      e[2] = 4 * g + 2 < d ? one(v.z) : (E)0;
      e[3] = 4 * g + 3 < d ? one(v.w) : (E)0;
    };
    // pass 2: sum
    E e[W][4];
    E sum = 0;
#pragma unroll
    for (int i = 0; i < iters; ++i) {
      const int g = lane + 32 * i;
      E t[4] = {0, 0, 0, 0};
      if (g < ngroups) exps(g, WPL > 0 ? x[i] : __ldg(src + g), t);
      if (WPL > 0) { e[i][0] = t[0]; e[i][1] = t[1]; e[i][2] = t[2]; e[i][3] = t[3]; }
      sum += (t[0] + t[1]) + (t[2] + t[3]);
    }
    // the row sum is >= I0 * 2^N: the maximum contributes exactly that
    if constexpr (NARROW) sum = __reduce_add_sync(0xffffffffu, sum);
    else sum = warp_sum_u64(sum);
    // Eq. (IntDiv); factor * e <= 2^M < 2^63.  NARROW: factor < 2^32 and M - (k_out - 1) >= 32, so the product's
    // high word shifted by the rest is the same value.
    const E factor = (E)((1ull << c.M) / (unsigned long long)sum);
    auto prob = [&](E t) -> int {
      if constexpr (NARROW) return min((int)(__umulhi(factor, t) >> (c.osh - 32)), c.omax);
      else return min((int)((factor * t) >> c.osh), c.omax);
    };
    // pass 3: outputs
    int* dst = reinterpret_cast<int*>(out + r * ldout);
#pragma unroll
    for (int i = 0; i < iters; ++i) {
      const int g = lane + 32 * i;
      if (g < nwords_out) {
        E t[4] = {0, 0, 0, 0};
        if (WPL > 0) { t[0] = e[i][0]; t[1] = e[i][1]; t[2] = e[i][2]; t[3] = e[i][3]; }
        else if (g < ngroups) exps(g, __ldg(src + g), t);
        dst[g] = (int)pack_sat8_u(prob(t[0]), prob(t[1]), prob(t[2]), prob(t[3]));
      }
    }
  }
}

int launch_shiftmax_direct(ivit_ctx* ctx, const int32_t* in, int64_t ldin, ivit_exp_params p, int8_t* out,
                           int64_t ldout, int64_t rows, int64_t d) {
  if (rows == 0) return IVIT_OK;
  DirectConsts c;
  c.I0 = (unsigned)p.I0; c.N = p.N; c.M = p.M;
  c.osh = p.M - (p.k_out - 1);
  c.omax = (1 << (p.k_out - 1)) - 1;
  // floor((2^64 - 1) / I0) + 1: floor(2^64 / I0) + 1, or exactly 2^64 / I0 when I0 is a power of two (both give the floor quotient)
  c.magic = p.I0 > 1 ? ~0ull / (unsigned long long)p.I0 + 1ull : 0ull;
  c.zero_from = (unsigned long long)p.I0 * (unsigned long long)(p.N + 29);
  c.m_hi = (unsigned)(c.magic >> 32); c.m_lo = (unsigned)c.magic;
  // -I_p >= (23 / 16) nd - 1: from nd_cut on it is at least zero_from; below it -I_p <= 1.5 nd_cut + 1 < 2^32
  c.nd_cut = (unsigned)(((c.zero_from + 1) * 16 + 22) / 23);
  const unsigned long long top = (unsigned long long)p.I0 << p.N;   // the largest exponential
  const bool narrow = c.zero_from <= (1ull << 31) && top * (unsigned long long)d < (1ull << 32) && c.osh >= 32 &&
                      (p.M <= 32 || top > (1ull << (p.M - 32)));
  const int64_t want = (rows + 7) / 8;
  const int grid = (int)(want < (int64_t)ctx->sm_count * 8 ? want : (int64_t)ctx->sm_count * 8);
  LaunchScope ls(ctx, KIND_SHIFTMAX, (double)rows * (double)d * 5.0);
  const int wpl = (int)(((d + 15) / 16 * 4 + 31) / 32);
  if (narrow) {
    if (wpl <= 2) launch_k(shiftmax_direct_kernel<2, true>, dim3(grid), dim3(256), 0, ctx->stream, in, ldin, c, out, ldout, rows, (int)d);
    else if (wpl <= 5) launch_k(shiftmax_direct_kernel<5, true>, dim3(grid), dim3(256), 0, ctx->stream, in, ldin, c, out, ldout, rows, (int)d);
    else launch_k(shiftmax_direct_kernel<0, true>, dim3(grid), dim3(256), 0, ctx->stream, in, ldin, c, out, ldout, rows, (int)d);
  } else {
    if (wpl <= 2) launch_k(shiftmax_direct_kernel<2, false>, dim3(grid), dim3(256), 0, ctx->stream, in, ldin, c, out, ldout, rows, (int)d);
    else if (wpl <= 5) launch_k(shiftmax_direct_kernel<5, false>, dim3(grid), dim3(256), 0, ctx->stream, in, ldin, c, out, ldout, rows, (int)d);
    else launch_k(shiftmax_direct_kernel<0, false>, dim3(grid), dim3(256), 0, ctx->stream, in, ldin, c, out, ldout, rows, (int)d);
  }
  return ls.done();
}

// ------------------------------------------------------------------ ShiftGELU

// ShiftGELU over an int8 row depends on two numbers only: the element x and m = max(0, row maximum of x)
// (the scaled value 1.702 x ~ (1.1011)b x of Eq. (GELU) is monotone in x, so its row maximum is that of m).
// The 128 x 256 results are produced once per parameter set; the row kernel then only looks values up.
// Entry (m, x): sigmoid(1.702 S x) as e / (e + e1) with both exponentials taken relative to the scaled maximum
// (Eq. (sigmoid)): e = exp of (scaled x - scaled m), e1 = exp of (-scaled m); quotient by Eq. (IntDiv) with
// M = 45 and k_out bits; the product x * quotient is requantised by `post` and saturated.
__global__ void shiftgelu_table_kernel(ivit_exp_params p, int post_m, int post_s, int8_t* __restrict__ table) {
  pdl_trigger();
  pdl_wait();
  const int m = blockIdx.x;            // 0..127
  const int x = (int)threadIdx.x - 128;
  int out = 0;
  if (x <= m) {                        // pairs with x above the row maximum cannot occur
    auto scaled = [](int v) { return v + (v >> 1) + (v >> 3) + (v >> 4); };
    const int top = scaled(m);
    const unsigned e1 = shiftexp(-top, p.I0, p.N);
    const unsigned e = shiftexp(scaled(x) - top, p.I0, p.N);
    const unsigned long long den = (unsigned long long)e + e1;
    int quot = 0;
    if (den != 0) {
      const unsigned long long recip = (1ull << 45) / den;
      quot = (int)((recip * e) >> (46 - p.k_out));       // recip * e <= 2^45
    }
    out = sat8(rq(x * quot, post_m, post_s));
  }
  table[m * 256 + threadIdx.x] = (int8_t)out;
}

// Rows of NV vectors of 16 values with NV R = 32 W: R rows fill the lanes of W loads (rows of 24 or 48 vectors would
// leave a quarter of them idle).  A lane's i-th vector belongs to row (lane + 32 i) / NV.
// What bounds it: instruction issue, about five instructions per four values and a look-up each.  Measured, back to back,
// against a warp per row: 200704 x 384 33.7 -> 31.6 us, 50176 x 768 15.8 -> 13.0, 197 x 768 2.4 -> 2.1.  (All 128 table
// rows in shared memory, one block of 1024 per SM, instead of a row staged per row: 31.9 and 15.1 us.)
template <int NV, int R>
__global__ void __launch_bounds__(256) shiftgelu_side_kernel(const int8_t* __restrict__ in, int64_t ldin,
                                                             const int8_t* __restrict__ table, int8_t* __restrict__ out,
                                                             int64_t ldout, int64_t rows, int fixed_max) {
  constexpr int W = NV * R / 32;
  static_assert(W * 32 == NV * R && NV >= 16, "whole loads, at most three rows in each");
  __shared__ __align__(256) unsigned tab[8][R * 64];
  pdl_trigger();
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const unsigned k256 = gelu_k256();
  int row[W], off[W];
  uint32_t t8[W];
#pragma unroll
  for (int i = 0; i < W; ++i) {
    row[i] = (lane + 32 * i) / NV;
    off[i] = (lane + 32 * i - row[i] * NV) * 16;
    t8[i] = (uint32_t)__cvta_generic_to_shared(tab[wib] + 64 * row[i]);
  }
  pdl_wait();
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r0 = warp * R; r0 < rows; r0 += nwarps * R) {
    int4 w[W];
    int m[W];
#pragma unroll
    for (int i = 0; i < W; ++i) w[i] = __ldg(reinterpret_cast<const int4*>(in + min(r0 + row[i], rows - 1) * ldin + off[i]));
#pragma unroll
    for (int i = 0; i < W; ++i) {
      ByteMax b;
      b.add(w[i]);
      m[i] = b.value();
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < R; ++r) {
      int mx = fixed_max;   // >= 0: the static-maximum variant
      if (fixed_max < 0) {
        mx = 0;
#pragma unroll
        for (int i = r * NV / 32; i <= (r * NV + NV - 1) / 32; ++i) mx = max(mx, row[i] == r ? m[i] : 0);
        mx = __reduce_max_sync(0xffffffffu, mx);
      }
      gelu_stage_row(table + mx * 256, tab[wib] + 64 * r, lane);
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < W; ++i)
      if (r0 + row[i] < rows) *reinterpret_cast<int4*>(out + (r0 + row[i]) * ldout + off[i]) = gelu_vec(w[i], t8[i], k256);
  }
}

// WPL > 0: rows of up to 512 * WPL values, R rows per warp at a time, kept in registers between the maximum and
// the look-ups (shiftgelu_rows).  WPL == 0: any width; the row is read twice.
template <int WPL, int R>
__global__ void __launch_bounds__(256) shiftgelu_kernel(const int8_t* __restrict__ in, int64_t ldin,
                                                        const int8_t* __restrict__ table,
                                                        int8_t* __restrict__ out, int64_t ldout,
                                                        int64_t rows, int cols, int fixed_max) {
  pdl_trigger();
  pdl_wait();
  __shared__ __align__(256) unsigned tab[8][(WPL > 0 ? R : 1) * 64];  // 256-byte table rows, per warp
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  if (WPL > 0) {
    constexpr int W = WPL > 0 ? WPL : 1;
    for (int64_t r0 = warp * R; r0 < rows; r0 += nwarps * R) {
      const int nrows = (int)(rows - r0 < R ? rows - r0 : R);
      shiftgelu_rows<W, R, false>(in + r0 * ldin, ldin, nrows, cols, table, tab[wib], out + r0 * ldout, ldout, lane, fixed_max);
      __syncwarp();
    }
    return;
  }
  const int nvec = cols >> 4;  // 16-byte vectors per row
  const int iters = (nvec + 31) / 32;
  const unsigned char* t8 = reinterpret_cast<const unsigned char*>(tab[wib]);
  for (int64_t r = warp; r < rows; r += nwarps) {
    const int4* src = reinterpret_cast<const int4*>(in + r * ldin);
    int mx4 = (int)0x80808080;
    for (int i = 0; i < iters; ++i) {
      const int idx = lane + 32 * i;
      int4 v = make_int4((int)0x80808080, (int)0x80808080, (int)0x80808080, (int)0x80808080);
      if (idx < nvec) v = __ldg(src + idx);
      mx4 = (int)__vmaxs4(__vmaxs4((unsigned)v.x, (unsigned)v.y), __vmaxs4(__vmaxs4((unsigned)v.z, (unsigned)v.w), (unsigned)mx4));
    }
    int mx = max(max((int)(int8_t)mx4, (int)(int8_t)(mx4 >> 8)), max((int)(int8_t)(mx4 >> 16), (int)(int8_t)(mx4 >> 24)));
    mx = fixed_max >= 0 ? fixed_max : max(0, warp_max(mx));   // fixed_max: the static-maximum variant
    __syncwarp();
    const unsigned* trow = reinterpret_cast<const unsigned*>(table + mx * 256);
    tab[wib][lane] = __ldg(trow + lane);
    tab[wib][lane + 32] = __ldg(trow + lane + 32);
    __syncwarp();
    int4* dst = reinterpret_cast<int4*>(out + r * ldout);
    for (int i = 0; i < iters; ++i) {
      const int idx = lane + 32 * i;
      if (idx < nvec) {
        const int4 v = __ldg(src + idx);
        const int vin[4] = {v.x, v.y, v.z, v.w};
        int vout[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const unsigned u = (unsigned)vin[k] ^ 0x80808080u;  // x + 128 per byte
          unsigned pk = t8[u & 0xff];
          pk |= (unsigned)t8[(u >> 8) & 0xff] << 8;
          pk |= (unsigned)t8[(u >> 16) & 0xff] << 16;
          pk |= (unsigned)t8[u >> 24] << 24;
          vout[k] = (int)pk;
        }
        dst[idx] = make_int4(vout[0], vout[1], vout[2], vout[3]);
      }
    }
  }
}

// Finds or builds the lookup table of a parameter set; *table = its 128 x 256 bytes on the device.
static int gelu_table(ivit_ctx* ctx, ivit_exp_params p, ivit_scale post, const int8_t** table) {
  const GeluKey key{p.I0, p.N, p.M, p.k_out, post.mult, post.shift};
  int slot = -1;
  for (int i = 0; i < ctx->gelu_used; ++i)
    if (ctx->gelu_keys[i] == key) { slot = i; break; }
  if (slot < 0) {
    if (ctx->gelu_used < kGeluTableSlots) {
      slot = ctx->gelu_used++;
    } else {
      slot = ctx->gelu_next;
      ctx->gelu_next = (ctx->gelu_next + 1) % kGeluTableSlots;
    }
    ctx->gelu_keys[slot] = key;
    ++ctx->gelu_gen;
    LaunchScope lt(ctx, KIND_GELU_TABLE, (double)kGeluTableBytes);
    launch_k(shiftgelu_table_kernel, dim3(128), dim3(256), 0, ctx->stream, p, post.mult, post.shift,
                                                          ctx->gelu_tables + (size_t)slot * kGeluTableBytes);
    int rc = lt.done();
    if (rc) return rc;
  }
  *table = ctx->gelu_tables + (size_t)slot * kGeluTableBytes;
  return IVIT_OK;
}

int gelu_table_for(ivit_ctx* ctx, ivit_exp_params p, ivit_scale post, const int8_t** table) {
  return gelu_table(ctx, p, post, table);
}

int gelu_static_row(ivit_ctx* ctx, ivit_exp_params p, ivit_scale post, const int8_t** row) {
  const int8_t* table = nullptr;
  const int rc = gelu_table(ctx, p, post, &table);
  if (rc) return rc;
  *row = table + 127 * 256;   // I_max = I_p(127)
  return IVIT_OK;
}

static int shiftgelu_rows(ivit_ctx* ctx, const int8_t* in, int64_t ldin, ivit_exp_params p, ivit_scale post,
                          int8_t* out, int64_t ldout, int64_t rows, int64_t cols, int fixed_max) {
  if (rows == 0) return IVIT_OK;
  const int8_t* table = nullptr;
  int rc = gelu_table(ctx, p, post, &table);
  if (rc) return rc;
  const int wpl = (int)((cols / 16 + 31) / 32);
  const int rpw = wpl <= 1 ? 4 : (wpl == 2 || wpl == 4 ? 2 : 1);            // rows a warp takes at a time
  const int64_t want = ((rows + rpw - 1) / rpw + 7) / 8;
  const int grid = (int)(want < (int64_t)ctx->sm_count * 12 ? want : (int64_t)ctx->sm_count * 12);
  cudaStream_t st = ctx->stream;
  LaunchScope ls(ctx, KIND_SHIFTGELU, 2.0 * (double)rows * (double)cols);
  if (cols == 384) launch_k(shiftgelu_side_kernel<24, 4>, dim3(grid), dim3(256), 0, st, in, ldin, table, out, ldout, rows, fixed_max);
  else if (cols == 768) launch_k(shiftgelu_side_kernel<48, 2>, dim3(grid), dim3(256), 0, st, in, ldin, table, out, ldout, rows, fixed_max);
  else if (wpl <= 1) launch_k(shiftgelu_kernel<1, 4>, dim3(grid), dim3(256), 0, st, in, ldin, table, out, ldout, rows, (int)cols, fixed_max);
  else if (wpl <= 2) launch_k(shiftgelu_kernel<2, 2>, dim3(grid), dim3(256), 0, st, in, ldin, table, out, ldout, rows, (int)cols, fixed_max);
  else if (wpl <= 3) launch_k(shiftgelu_kernel<3, 1>, dim3(grid), dim3(256), 0, st, in, ldin, table, out, ldout, rows, (int)cols, fixed_max);
  else if (wpl <= 4) launch_k(shiftgelu_kernel<4, 2>, dim3(grid), dim3(256), 0, st, in, ldin, table, out, ldout, rows, (int)cols, fixed_max);
  else if (wpl <= 6) launch_k(shiftgelu_kernel<6, 1>, dim3(grid), dim3(256), 0, st, in, ldin, table, out, ldout, rows, (int)cols, fixed_max);
  else if (wpl <= 8) launch_k(shiftgelu_kernel<8, 1>, dim3(grid), dim3(256), 0, st, in, ldin, table, out, ldout, rows, (int)cols, fixed_max);
  else launch_k(shiftgelu_kernel<0, 1>, dim3(grid), dim3(256), 0, st, in, ldin, table, out, ldout, rows, (int)cols, fixed_max);
  return ls.done();
}

int launch_shiftgelu(ivit_ctx* ctx, const int8_t* in, int64_t ldin, ivit_exp_params p, ivit_scale post,
                     int8_t* out, int64_t ldout, int64_t rows, int64_t cols) {
  return shiftgelu_rows(ctx, in, ldin, p, post, out, ldout, rows, cols, -1);
}

int launch_shiftgelu_static(ivit_ctx* ctx, const int8_t* in, int64_t ldin, ivit_exp_params p, ivit_scale post,
                            int8_t* out, int64_t ldout, int64_t rows, int64_t cols) {
  return shiftgelu_rows(ctx, in, ldin, p, post, out, ldout, rows, cols, 127);
}

}  // namespace ivit

// ---- verification aid: the square-root routine of the I-LayerNorm kernels over a range of radicands ----
namespace ivit {
__global__ void isqrt_range_kernel(unsigned n0, unsigned count, uint16_t* __restrict__ out) {
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x)
    out[i] = (uint16_t)isqrt26(n0 + i);
}
}  // namespace ivit

extern "C" int ivit_isqrt_range(ivit_ctx* ctx, uint32_t n0, uint32_t count, uint16_t* out) {
  if (!ctx || !out) return IVIT_ERR_INVALID_ARG;
  if ((uint64_t)n0 + count > (1ull << 26)) return IVIT_ERR_RANGE;
  if (count == 0) return IVIT_OK;
  ivit::isqrt_range_kernel<<<ctx->sm_count * 8, 256, 0, ctx->stream>>>(n0, count, out);
  ctx->launches += 1;
  return cudaGetLastError() == cudaSuccess ? IVIT_OK : IVIT_ERR_CUDA;
}
