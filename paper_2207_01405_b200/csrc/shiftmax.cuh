// Pieces of Algorithm 1 (Shiftmax, Sec. 3.3) shared by the attention kernels and the stand-alone row kernel.
#pragma once

#include "common.cuh"

namespace ivit {

// Eq. (IntDiv) for k_out = 8, four exponentials, packed, with factor4 = 4 floor(2^45 / sum): the probability is byte 1 of the high product word.  The one
// probability that can reach 128, and is clamped to 127, belongs to a row whose only non-zero exponential is a power of
// two; prob_factor4 takes one off the reciprocal there, which gives 127.
__device__ __forceinline__ uint32_t prob_word8(unsigned factor4, int e0, int e1, int e2, int e3) {
  return __byte_perm(__byte_perm(__umulhi(factor4, (unsigned)e0), __umulhi(factor4, (unsigned)e1), 0x0051),
                     __byte_perm(__umulhi(factor4, (unsigned)e2), __umulhi(factor4, (unsigned)e3), 0x0051), 0x5410);
}

// ShiftExp of one packed score x (int8): the table entry at t - 4 cp x, where `sel` holds -4 cp in the byte that holds x.
// (Not volatile: the table does not change once the CTA's first barrier is behind, so look-ups may be moved freely.)
__device__ __forceinline__ unsigned exp_entry(uint32_t w, uint32_t sel, uint32_t t) {
  unsigned e;
  asm("{\n\t.reg .u32 a;\n\tdp4a.s32.s32 a, %1, %2, %3;\n\tld.shared.u32 %0, [a];\n\t}" : "=r"(e) : "r"(w), "r"(sel), "r"(t));
  return e;
}

// floor(2^45 / s) for 2^15 < s < 2^32.  With d = s 2^z, 2^31 <= d < 2^32, it is floor(2^63 / d) >> (18 - z) (nested floor
// quotients).  v starts at 2^63 / (middle of the 2^24 values that share d's upper byte), relative error below 2^-8, from
// a table of 128 entries; two Newton steps square that twice; the shift (by at least 2) leaves at most one unit, which
// the exact remainder puts right.  (Checked on the CPU for every s of the range; a 64-bit division takes 700 cycles on
// the row's critical path.)
__device__ __forceinline__ unsigned recip_seed(int i) { return (unsigned)((1ull << 40) / (unsigned)(2 * (128 + i) + 1)); }
__device__ __forceinline__ unsigned recip45(unsigned s, const unsigned* seeds) {
  const int z = __clz(s);
  const unsigned d = s << z;
  unsigned v = seeds[(d >> 24) & 127u];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int e = (int)(0x80000000u - __umulhi(v, d));               // 2^31 - v d / 2^32
    v += (unsigned)__mulhi((int)(v >> 1), e << 2);
  }
  if (d == 0x80000000u) v = 0xffffffffu;   // 2^32 itself does not fit
  unsigned q = v >> (18 - z);
  long long r = (long long)((1ull << 45) - (unsigned long long)q * s);
  if (r < 0) { --q; r += s; }
  if (r >= (long long)s) ++q;
  return q;
}
// Four times the reciprocal for prob_word8; `top` = I0 2^N > 2^15, the largest exponential.
__device__ __forceinline__ unsigned prob_factor4(unsigned sum, unsigned top, const unsigned* seeds) {
  unsigned f = recip45(sum, seeds);
  if (sum == top && (sum & (sum - 1u)) == 0u) --f;
  return f << 2;
}

// Builds `cp` copies of the ShiftExp table (entry i, copy c at word i cp + c) with n threads, n a multiple of 256 or a
// divisor of it; consecutive lanes write different banks.
__device__ __forceinline__ void build_exp_table(int I0, int N, int cp, uint8_t* tab, int st, int n) {
  const int per = 32 / cp;                  // entries per 32 banks
  for (int i = st & 255; i < 256; i += n < 256 ? n : 256) {
    const unsigned e = shiftexp(-i, I0, N);
    for (int c = st >> 8; c < cp; c += n < 256 ? 1 : n >> 8)
      *reinterpret_cast<unsigned*>(tab + 4u * ((unsigned)i * cp + ((c + (st & 31) / per) & (cp - 1)))) = e;
  }
}
// -4 cp as a signed byte, in byte b (the multiplier of exp_entry).
__host__ __device__ __forceinline__ uint32_t exp_sel(int cp, int b) { return ((uint32_t)(-4 * cp) & 0xffu) << (8 * b); }

}  // namespace ivit
