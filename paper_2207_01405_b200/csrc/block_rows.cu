// Encoder blocks with few rows: one launch per block (Sec. 3.1), every CTA (or cluster of CTAs) the owner of a few token rows.
//
// With few rows the kernels of a block are a chain of launches of 3 to 4 us each in which the chip is nearly idle.  All
// steps but one work on token rows independently; only attention needs the keys and values of the other rows of the image.
// So a cluster of C CTAs takes 16 MT rows of one image through everything between two attentions,
//   scores, Shiftmax, P V, output projection + residual, LayerNorm 2, FC1, ShiftGELU, FC2 + residual,
//   LayerNorm 1 and QKV of the NEXT block,
// with the rows in shared memory all the way, and the launch boundary is the exchange of keys and values.  A forward is then
// depth + 1 such launches (the first one runs LayerNorm 1 and QKV only) instead of eight per block.
//   products   mma.sync m16n8k32 with the token rows as the M = 16 operand.  (A tcgen05 tile has 128 lanes, its operands go
//              through shared memory and its results through tensor memory: three hand-overs of a few hundred clocks each
//              for a product that takes as long as one of them.  mma.sync reaches 1950 multiply-accumulates per clock and
//              SM, which is 16 rows times the 110 bytes per clock at which weights arrive from L2.)
//   weights    from L2 straight into the B fragments: a lane of row n reads 32 bytes (ld.v8), so a warp reads whole 128-byte
//              lines of eight weight rows (105 to 115 bytes per clock and SM; with 16-byte loads 34 to 63).  Which of its
//              bytes counts as which k index of the MMA is free as long as the other operand follows the same order.
//              The loads of a step's first units are requested before the row operator and the barrier in front of it.
//   C > 1      the CTAs of a cluster share the rows: each computes 1/C of the heads or output channels and writes its piece
//              into the shared memory of all; row operators run in every CTA.  For layers whose weights would take one SM
//              longer to fetch than the cluster's barriers cost.
#include <cstdio>
#include <cstdlib>
#include "common.cuh"
#include "rowops.cuh"
#include "shiftmax.cuh"
#include "tc_ptx.cuh"

namespace ivit {
namespace {

constexpr int kRbWarps = 16, kRbThreads = 32 * kRbWarps;
constexpr int kRbCopies = 8;             // copies of the ShiftExp table (a lane uses copy lane % 8)

// Words of a LayerNorm row per lane stand for the width class: up to 256, 384, 768, 1024 channels.  NT: n-tiles (of eight
// channels) of a warp's task: the one that deals 3D, D and 4D channels out to sixteen warps more evenly.
template <int W>
struct RbWidth { static constexpr int NT = W == 3 || W == 6 ? 3 : 2, RING = NT == 3 ? 2 : 3; };

struct RbDense { const int8_t* W; const int32_t* mult; const uint8_t* shift; const int32_t* bias; };
struct RbNorm { const int32_t* mult; const uint8_t* shift; const int32_t* beta; int M; };

struct RbArgs {
  int T, D, heads, H;
  int groups;                  // groups of 16 MT rows per image
  int C;                       // CTAs per cluster
  int Tk, Tp;                  // rows of a head in K, tokens of a channel in V^T (padded)
  int first, last;             // steps: 0 attention, 1 projection, 2 FC1, 3 FC2, 4 next QKV
  int early;                   // parameters may be read ahead of the wait for the previous kernel
  const int8_t* X;             // [B T, D] input rows
  int8_t* Y;                   // [B T, D] output rows of the block
  const int8_t *Q, *K, *V;     // this block's: [B T, D], [B, heads, Tk, 64], [B, D, Tp] (values transposed)
  int8_t *Qn, *Kn, *Vn;        // the next block's
  int qk_m, qk_s, pv_m, pv_s;
  ivit_exp_params smax;
  int fast;                    // arithmetic of shiftmax.cuh's prob_word8
  uint32_t sel[4];
  const int32_t* bias;         // score bias [bias_batches, T, T] or nullptr
  int bias_batches;
  RbDense dense[4];            // projection, FC1, FC2, next QKV
  int res_m[2], res_s[2];
  RbNorm norm[2];              // LayerNorm 2, LayerNorm 1 of the next block
  unsigned mean_magic;
  const int8_t* gelu;          // ShiftGELU table
  int gelu_max;                // -1, or the fixed maximum of the static variant
  // shared memory
  uint32_t a_off, q_off, h_off, par_off[4], norm_off[2], tab_off, gelu_off, red_off;
  int q_pitch, h_pitch, s_pitch, n_pitch;
};

__device__ __forceinline__ void mma_s8(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void lds128(uint32_t addr, uint32_t* v) {
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(addr));
}
__device__ __forceinline__ void ldg128(const int8_t* p, uint32_t* v) {
  asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "l"(p));
}
__device__ __forceinline__ void ldg256(const int8_t* p, uint32_t* v) {
  asm volatile("ld.global.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]) : "l"(p));
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// Two adjacent int8 results to the same place in the shared memory of every CTA of the cluster.
__device__ __forceinline__ void store2_all(uint32_t addr, uint32_t v, int C) {
  if (C == 1) {
    asm volatile("st.shared.u16 [%0], %1;" ::"r"(addr), "h"((unsigned short)v) : "memory");
    return;
  }
  for (int r = 0; r < C; ++r) {
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(addr), "r"(r));
    asm volatile("st.shared::cluster.u16 [%0], %1;" ::"r"(remote), "h"((unsigned short)v) : "memory");
  }
}
__device__ __forceinline__ void rb_sync_all(int C) {
  if (C == 1) __syncthreads();
  else cluster_sync_all();
}

// Shiftmax of the score rows r = warp, warp + 16, ... below `rows` of the tile at S (int8, pitch bytes apart), in place;
// columns from T on become 0.  RB rows of up to 128 NW columns at a time.
template <int NW, int RB>
__device__ __forceinline__ void rb_shiftmax(uint8_t* S, int pitch, int rows, const RbArgs& a, uint32_t tab_lane, const unsigned* seeds,
                                            int warp, int lane) {
  const unsigned top = (unsigned)a.smax.I0 << a.smax.N;
  const int osh = 14 - a.smax.k_out, omax = (1 << (a.smax.k_out - 1)) - 1;
  for (int r0 = warp; r0 < rows; r0 += kRbWarps * RB) {
    uint32_t w[RB][NW];
    unsigned e[RB][NW][4];
    unsigned sum[RB], my_sum = 1;
#pragma unroll
    for (int i = 0; i < RB; ++i) {
      const int r = r0 + kRbWarps * i;
      const uint32_t* src = reinterpret_cast<const uint32_t*>(S + (size_t)r * pitch);
      ByteMax m;
#pragma unroll
      for (int k = 0; k < NW; ++k) {
        const int q = lane + 32 * k, valid = a.T - 4 * q;     // columns of this word that exist
        uint32_t x = 0x80808080u;
        if (r < rows && valid > 0) {
          x = src[q];
          if (valid < 4) {
            const uint32_t keep = 0xffffffffu >> (8 * (4 - valid));
            x = (x & keep) | (0x80808080u & ~keep);
          }
        }
        w[i][k] = x;
        m.add(x);
      }
      const int mx = __reduce_max_sync(0xffffffffu, m.value());
      const uint32_t tmx = tab_lane + (uint32_t)(4 * kRbCopies * mx);
      unsigned s = 0;
#pragma unroll
      for (int k = 0; k < NW; ++k) {
        const int valid = a.T - 4 * (lane + 32 * k);
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const unsigned v = exp_entry(w[i][k], a.sel[b], tmx);
          e[i][k][b] = b < valid ? v : 0u;
          s += e[i][k][b];
        }
      }
      sum[i] = __reduce_add_sync(0xffffffffu, s);
      if (lane == i) my_sum = sum[i];
    }
    // the reciprocals of the RB rows, one per lane (Eq. (IntDiv) with M = 45)
    const unsigned mine = a.fast ? prob_factor4(my_sum <= 32768u ? 65536u : my_sum, top, seeds)
                                 : (unsigned)((1ull << 45) / (unsigned long long)(my_sum ? my_sum : 1u));
#pragma unroll
    for (int i = 0; i < RB; ++i) {
      const unsigned factor = __shfl_sync(0xffffffffu, mine, i);
      const int r = r0 + kRbWarps * i;
      if (r >= rows) continue;
      uint32_t* dst = reinterpret_cast<uint32_t*>(S + (size_t)r * pitch);
#pragma unroll
      for (int k = 0; k < NW; ++k) {
        const int q = lane + 32 * k;
        uint32_t o;
        if (a.fast) {
          o = prob_word8(factor, (int)e[i][k][0], (int)e[i][k][1], (int)e[i][k][2], (int)e[i][k][3]);
        } else {
          int p[4];
#pragma unroll
          for (int b = 0; b < 4; ++b) p[b] = min((int)(__umulhi(factor, e[i][k][b]) >> osh), omax);
          o = pack_sat8(p[0], p[1], p[2], p[3]);
        }
        if (4 * q < a.Tp) dst[q] = o;
      }
    }
  }
}

template <int W, int MT>
__global__ void __launch_bounds__(kRbThreads, 1) block_rows_kernel(const __grid_constant__ RbArgs a) {
  constexpr int NT = RbWidth<W>::NT, RING = RbWidth<W>::RING, ROWS = 16 * MT;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 255u) & ~255u;
  uint8_t* gen = smem_raw + (base - smem_u32(smem_raw));
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int g = lane >> 2, j = lane & 3, tid = threadIdx.x;
  const int C = a.C, rank = C > 1 ? (int)cluster_ctarank() : 0;
  const int group = (int)blockIdx.x / C, b = group / a.groups, t0 = (group - b * a.groups) * ROWS;
  const int nrow = min(ROWS, a.T - t0);                 // token rows of this group that exist
  const int D = a.D, T = a.T, pitch = D + 16;
  const int h_lo = rank * a.heads / C, nh = (rank + 1) * a.heads / C - h_lo;   // heads of this CTA
  // [x rows][LayerNorm out / attention out][q rows][scores, FC1 out, QKV out][parameters][tables][partial sums]
  uint8_t* const xs = gen;
  const uint32_t as_addr = base + a.a_off, qs_addr = base + a.q_off, hs_addr = base + a.h_off;
  const uint32_t tab = base + a.tab_off, tab_lane = tab + 4u * (unsigned)(lane & (kRbCopies - 1));
  unsigned* const seeds = reinterpret_cast<unsigned*>(gen + a.tab_off + 1024 * kRbCopies);

  // ---- set-up ----
  if (a.early) pdl_trigger();
  if (a.first == 0) {
    build_exp_table(a.smax.I0, a.smax.N, kRbCopies, gen + a.tab_off, tid, kRbThreads);
    if (tid < 128) seeds[tid] = recip_seed(tid);
  }
  if (!a.early) {
    pdl_wait();
    pdl_trigger();
  }
  // per-channel parameters of this CTA's channels: [mult][bias][shift] of each Dense layer, [mult][beta][shift] of a LayerNorm
  for (int st = a.first ? a.first : 1; st < a.last; ++st) {
    const RbDense& d = a.dense[st - 1];
    const int n = (st == 2 ? a.H : (st == 4 ? 3 * D : D)) / C, n0 = rank * n;
    const uint32_t p = base + a.par_off[st - 1];
    for (int i = tid; i < n / 4; i += kRbThreads) {
      cp_async16(p + 16 * i, d.mult + n0 + 4 * i);
      if (d.bias) cp_async16(p + 4 * n + 16 * i, d.bias + n0 + 4 * i);
      else *reinterpret_cast<uint4*>(gen + a.par_off[st - 1] + 4 * n + 16 * i) = make_uint4(0u, 0u, 0u, 0u);
      if (i < n / 16) cp_async16(p + 8 * n + 16 * i, d.shift + n0 + 16 * i);
    }
  }
  for (int k = a.first ? 1 : 0; k < (a.last > 4 ? 2 : 1); ++k) {
    const RbNorm& d = a.norm[k];
    const uint32_t p = base + a.norm_off[k];
    for (int i = tid; i < D / 4; i += kRbThreads) {
      cp_async16(p + 16 * i, d.mult + 4 * i);
      if (d.beta) cp_async16(p + 4 * D + 16 * i, d.beta + 4 * i);
      else *reinterpret_cast<uint4*>(gen + a.norm_off[k] + 4 * D + 16 * i) = make_uint4(0u, 0u, 0u, 0u);
      if (i < D / 16) cp_async16(p + 12 * D + 16 * i, d.shift + 16 * i);
    }
  }
  if (a.early) pdl_wait();

  // ---- this group's rows; the first keys ----
  {
    const int8_t* x = a.X + ((int64_t)b * T + t0) * D;
    const int per = D >> 4;
    for (int i = tid; i < ROWS * per; i += kRbThreads) {
      const int r = i / per, c = i - r * per;
      if (r < nrow) cp_async16(base + r * pitch + 16 * c, x + (int64_t)r * D + 16 * c);
      else *reinterpret_cast<uint4*>(xs + r * pitch + 16 * c) = make_uint4(0u, 0u, 0u, 0u);
    }
  }
  const int ntile = (T + 7) >> 3;
  const int8_t* const kbase = a.K + ((int64_t)(b * a.heads + h_lo) * a.Tk) * 64 + lane * 16;   // (8 rows of 64 bytes)
  uint32_t kb[4][4];
  int s_h = 0, s_n = warp;            // head and key tile of the next scores
  int s_hs[4], s_ns[4];
  auto next_keys = [&]() {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      while (s_n >= ntile && s_h < nh) { s_n -= ntile; ++s_h; }
      s_hs[i] = s_h;
      s_ns[i] = s_n;
      if (s_h < nh) ldg128(kbase + ((int64_t)s_h * a.Tk + 8 * s_n) * 64, kb[i]);
      s_n += kRbWarps;
    }
  };
  if (a.first == 0) {
    const int8_t* q = a.Q + ((int64_t)b * T + t0) * D + h_lo * 64;
    const int per = 4 * nh;
    for (int i = tid; i < ROWS * per; i += kRbThreads) {
      const int r = i / per, c = i - r * per;
      if (r < nrow) cp_async16(qs_addr + r * a.q_pitch + 16 * c, q + (int64_t)r * D + 16 * c);
      else *reinterpret_cast<uint4*>(gen + a.q_off + r * a.q_pitch + 16 * c) = make_uint4(0u, 0u, 0u, 0u);
    }
    next_keys();
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  rb_sync_all(C);                      // (C > 1: every CTA of the cluster runs, its shared memory may be written)

  // LayerNorm constants into the form of rowops.cuh; agreed on by all threads
  bool ln_fast[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    if (k < (a.first ? 1 : 0) || k >= (a.last > 4 ? 2 : 1)) { ln_fast[k] = false; continue; }
    uint8_t* p = gen + a.norm_off[k];
    bool ok = true;
    int4* const sm_b = reinterpret_cast<int4*>(p + 4 * D);
    int4* const sm_s = reinterpret_cast<int4*>(p + 8 * D);
    const uchar4* raw = reinterpret_cast<const uchar4*>(p + 12 * D);
    for (int i = tid; i < D / 4; i += kRbThreads) {
      const uchar4 s4 = raw[i];
      const int4 b4 = sm_b[i];
      const int s[4] = {clamp_shift(s4.x), clamp_shift(s4.y), clamp_shift(s4.z), clamp_shift(s4.w)}, bb[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int sh = s[c] - 32;
        ok = ok && sh >= 1 && bb[c] > -(1 << (29 - sh)) && bb[c] < (1 << (29 - sh));
      }
      sm_s[i] = make_int4(s[0], s[1], s[2], s[3]);
    }
    ln_fast[k] = __syncthreads_and(ok) != 0;
    if (ln_fast[k]) ln_fold_consts(D / 4, sm_s, sm_b, tid, kRbThreads);
  }
  if (a.first) __syncthreads();        // (else the barrier behind the scores)

  // ---- scores S = Q K^T (+ bias), requantised: [head][row][token] ----
  if (a.first == 0) {
    const bool hi = a.qk_s >= 33;
    const int rnd = hi ? 1 << (a.qk_s - 33) : 0, sh = hi ? a.qk_s - 32 : 0;
    while (s_hs[0] < nh) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (s_hs[i] >= nh) break;
        const int col = 8 * s_ns[i] + 2 * j;
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
          uint32_t r0[4], r1[4];
          const uint32_t qa = qs_addr + (uint32_t)((mt * 16 + g) * a.q_pitch + s_hs[i] * 64 + 16 * j);
          lds128(qa, r0);
          lds128(qa + 8 * a.q_pitch, r1);
          int acc[4] = {0, 0, 0, 0};
          mma_s8(acc, r0[0], r1[0], r0[1], r1[1], kb[i][0], kb[i][1]);
          mma_s8(acc, r0[2], r1[2], r0[3], r1[3], kb[i][2], kb[i][3]);
          if (a.bias) {
            const int32_t* bm = a.bias + (int64_t)((unsigned)(b * a.heads + h_lo + s_hs[i]) % (unsigned)a.bias_batches) * T * T;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const int row = t0 + mt * 16 + g + 8 * (k >> 1), c = col + (k & 1);
              if (row < T && c < T) acc[k] += __ldg(bm + (int64_t)row * T + c);
            }
          }
#pragma unroll
          for (int k = 0; k < 4; ++k)
            acc[k] = hi ? mad_hi(acc[k], a.qk_m, rnd) >> sh : (int)(((long long)acc[k] * a.qk_m + (1ll << (a.qk_s - 1))) >> a.qk_s);
          const uint32_t w = pack_sat8(acc[0], acc[1], acc[2], acc[3]);
          uint8_t* o = gen + a.h_off + (size_t)(s_hs[i] * ROWS + mt * 16 + g) * a.s_pitch + col;
          *reinterpret_cast<uint16_t*>(o) = (uint16_t)w;
          *reinterpret_cast<uint16_t*>(o + 8 * a.s_pitch) = (uint16_t)(w >> 16);
        }
      }
      next_keys();
    }
    __syncthreads();
  }

  // ---- products: 0 P V, 1 projection, 2 FC1, 3 FC2, 4 QKV of the next block ----
#pragma unroll 1
  for (int st = a.first; st < a.last; ++st) {
    // B rows: channel c of segment s at W + (s nseg + c) ldw; A rows: a0 + s a_step (a segment is a head of P V)
    const int8_t* Wp;
    int ldw, K, nseg, segs = 1, a_pitch = pitch;
    uint32_t a0 = as_addr, a_step = 0;
    if (st == 0) {
      Wp = a.V + ((int64_t)b * D + h_lo * 64) * a.Tp;
      ldw = K = a.Tp; nseg = 64; segs = nh; a0 = hs_addr; a_pitch = a.s_pitch; a_step = (uint32_t)(ROWS * a.s_pitch);
    } else {
      K = st == 3 ? a.H : D;
      nseg = (st == 2 ? a.H : (st == 4 ? 3 * D : D)) / C;
      ldw = K;
      Wp = a.dense[st - 1].W + (int64_t)rank * nseg * K;
      if (st == 3) { a0 = hs_addr; a_pitch = a.h_pitch; }
    }
    const int per_seg = (nseg + 8 * NT - 1) / (8 * NT), tasks = per_seg * segs, kblocks = (K + 127) >> 7;
    // few tasks: several warps share one, each with a part of the contraction
    const int split = tasks > kRbWarps / 2 || tasks == 0 ? 1 : min(kRbWarps / tasks, kblocks);
    int task = warp, kp = 0, kb0 = 0, kb1 = kblocks;
    if (split > 1) {
      task = warp / split;
      kp = warp - task * split;
      kb0 = kp * kblocks / split;
      kb1 = (kp + 1) * kblocks / split;
    }
    uint32_t ring[RING][NT][8];
    auto load = [&](uint32_t (&v)[NT][8], int t, int k) {
      const int seg = segs == 1 ? 0 : t / per_seg, c0 = (t - seg * per_seg) * (8 * NT) + 2 * NT * (g >> 1) + (g & 1);
#pragma unroll
      for (int u = 0; u < NT; ++u) {
        const int c = min(c0 + 2 * u, nseg - 1);
        const int8_t* p = Wp + (int64_t)(seg * nseg + c) * ldw + 128 * k;
        if (K - 128 * k >= 128) ldg256(p + 32 * j, v[u]);
        else ldg128(p + 16 * j, v[u]);
      }
    };
#pragma unroll
    for (int s = 0; s < RING; ++s)
      if (task < tasks && kb0 + s < kb1) load(ring[s], task, kb0 + s);

    // ---- the row operator in front of the product ----
    if (st == 0) {
      if (a.Tp <= 256) rb_shiftmax<2, 4>(gen + a.h_off, a.s_pitch, nh * ROWS, a, tab_lane, seeds, warp, lane);
      else rb_shiftmax<5, 2>(gen + a.h_off, a.s_pitch, nh * ROWS, a, tab_lane, seeds, warp, lane);
      __syncthreads();
    } else if (st == 2 || st == 4) {
      const int k = st == 2 ? 0 : 1;
      const int4* p = reinterpret_cast<const int4*>(gen + a.norm_off[k]);
      const LnConsts c{p, p + D / 2, p + D / 4, ln_fast[k]};
      layernorm_rows<W, MT, ROWS_SHARED>(reinterpret_cast<const int8_t*>(xs + warp * MT * pitch), pitch, MT, D, a.norm[k].M, a.mean_magic, c,
                                         reinterpret_cast<int8_t*>(gen + a.a_off + warp * MT * pitch), pitch, lane);
      __syncthreads();
    } else if (st == 3) {
      unsigned* const row_tab = reinterpret_cast<unsigned*>(gen + a.gelu_off) + warp * 64;
      for (int r = 0; r < MT; ++r) {
        int8_t* row = reinterpret_cast<int8_t*>(gen + a.h_off + (size_t)(warp * MT + r) * a.h_pitch);
        shiftgelu_rows<W, 1, ROWS_SHARED>(row, 0, 1, a.H, a.gelu, row_tab, row, 0, lane, a.gelu_max);
        __syncwarp();
      }
      __syncthreads();
    }

    for (bool more = split > 1 || task < tasks; more;) {
      const bool has = task < tasks;
      const int seg = segs == 1 ? 0 : task / per_seg;
      int acc[MT][NT][4];
#pragma unroll
      for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int u = 0; u < NT; ++u)
#pragma unroll
          for (int k = 0; k < 4; ++k) acc[mt][u][k] = 0;
      if (has) {
        const uint32_t arow = a0 + (uint32_t)seg * a_step + (uint32_t)(g * a_pitch);
#pragma unroll 1
        for (int k = kb0; k < kb1; k += RING) {
#pragma unroll
          for (int s = 0; s < RING; ++s) {
            if (k + s < kb1) {
              const bool full = K - 128 * (k + s) >= 128;
#pragma unroll
              for (int mt = 0; mt < MT; ++mt) {
                uint32_t r0[8], r1[8];
                const uint32_t p = arow + (uint32_t)(mt * 16 * a_pitch + 128 * (k + s) + (full ? 32 : 16) * j);
                lds128(p, r0);
                lds128(p + 8 * a_pitch, r1);
                if (full) {
                  lds128(p + 16, r0 + 4);
                  lds128(p + 8 * a_pitch + 16, r1 + 4);
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                  if (q < 2 || full) {
#pragma unroll
                    for (int u = 0; u < NT; ++u)
                      mma_s8(acc[mt][u], r0[2 * q], r1[2 * q], r0[2 * q + 1], r1[2 * q + 1], ring[s][u][2 * q], ring[s][u][2 * q + 1]);
                  }
                }
              }
              // the unit that takes this place in the ring
              if (k + s + RING < kb1) load(ring[s], task, k + s + RING);
              else if (split == 1 && task + kRbWarps < tasks && kb0 + s < kb1) {
                // (the last unit of this task in place s)
                load(ring[s], task + kRbWarps, kb0 + s);
              }
            }
          }
        }
      }
      if (split > 1) {
        // partial sums: [warp][register][lane]
        int* const red = reinterpret_cast<int*>(gen + a.red_off) + warp * (MT * NT * 4 * 32) + lane;
        if (has && kp > 0) {
#pragma unroll
          for (int i = 0; i < MT * NT * 4; ++i) red[32 * i] = acc[i / (NT * 4)][i / 4 % NT][i % 4];
        }
        __syncthreads();
        if (has && kp == 0) {
          for (int o = 1; o < split; ++o)
#pragma unroll
            for (int i = 0; i < MT * NT * 4; ++i) acc[i / (NT * 4)][i / 4 % NT][i % 4] += red[o * (MT * NT * 4 * 32) + 32 * i];
        }
      }
      if (has && kp == 0) {
        const int c_seg = (task - seg * per_seg) * (8 * NT) + 2 * NT * j;      // this lane's first channel inside the segment
        // destination of channel 0 of the segment, row 0
        uint32_t dst;
        int d_pitch = pitch, copies = C;
        if (st == 0) dst = as_addr + (uint32_t)((h_lo + seg) * 64);
        else if (st == 2) { dst = hs_addr + (uint32_t)(rank * nseg); d_pitch = a.h_pitch; }
        else if (st == 4) { dst = hs_addr; d_pitch = a.n_pitch; copies = 1; }
        else dst = base + (uint32_t)(rank * nseg);
        const int res = st == 1 ? 0 : (st == 3 ? 1 : -1);
        // rq(x; m, s) of an int8 x on top of a word: high word of (x 2^24) m + 2^(s+23), shifted by s - 8; 0 from s = 39 on
        const int rs = res >= 0 ? a.res_s[res] : 33;
        const int rm = rs >= 39 || res < 0 ? 0 : a.res_m[res], rsh = rs >= 39 ? 31 : rs - 8, rrnd = rs >= 39 ? 0 : 1 << (rs - 9);
#pragma unroll
        for (int u = 0; u < NT; ++u) {
          const int c = c_seg + 2 * u;
          if (c >= nseg) continue;
          int m[2], s[2], bi[2];
          if (st == 0) {
            m[0] = m[1] = a.pv_m;
            s[0] = s[1] = a.pv_s;
            bi[0] = bi[1] = 0;
          } else {
            const uint8_t* par = gen + a.par_off[st - 1];
            const int2 m2 = *reinterpret_cast<const int2*>(par + 4 * c), b2 = *reinterpret_cast<const int2*>(par + 4 * nseg + 4 * c);
            const uchar2 s2 = *reinterpret_cast<const uchar2*>(par + 8 * nseg + c);
            m[0] = m2.x; m[1] = m2.y;
            bi[0] = b2.x; bi[1] = b2.y;
            s[0] = clamp_shift(s2.x); s[1] = clamp_shift(s2.y);
          }
          const bool hi = s[0] >= 33 && s[1] >= 33 && bi[0] > -(1 << 30) && bi[0] < (1 << 30) && bi[1] > -(1 << 30) && bi[1] < (1 << 30);
#pragma unroll
          for (int mt = 0; mt < MT; ++mt) {
            int v[4];
            if (hi) {
#pragma unroll
              for (int k = 0; k < 4; ++k)
                v[k] = mad_hi(acc[mt][u][k] + bi[k & 1], m[k & 1], 1 << (s[k & 1] - 33)) >> (s[k & 1] - 32);
            } else {
#pragma unroll
              for (int k = 0; k < 4; ++k)
                v[k] = (int)(mad_wide(acc[mt][u][k], m[k & 1], (long long)bi[k & 1] * m[k & 1] + (1ll << (s[k & 1] - 1))) >> s[k & 1]);
            }
            const uint32_t at = dst + (uint32_t)((mt * 16 + g) * d_pitch + c);
            if (res >= 0) {
              uint16_t x0, x1;
              asm volatile("ld.shared.u16 %0, [%1];" : "=h"(x0) : "r"(at));
              asm volatile("ld.shared.u16 %0, [%1];" : "=h"(x1) : "r"(at + 8 * d_pitch));
              v[0] += mad_hi((int)((uint32_t)x0 << 24), rm, rrnd) >> rsh;
              v[1] += mad_hi((int)((uint32_t)(x0 & 0xff00u) << 16), rm, rrnd) >> rsh;
              v[2] += mad_hi((int)((uint32_t)x1 << 24), rm, rrnd) >> rsh;
              v[3] += mad_hi((int)((uint32_t)(x1 & 0xff00u) << 16), rm, rrnd) >> rsh;
            }
            const uint32_t w = pack_sat8(v[0], v[1], v[2], v[3]);
            store2_all(at, w & 0xffffu, copies);
            store2_all(at + 8 * d_pitch, w >> 16, copies);
          }
        }
      }
      task += kRbWarps;
      more = split == 1 && task < tasks;
    }
    rb_sync_all(st == 4 ? 1 : C);

    if (st == 3) {
      // the block's output rows, shared out among the CTAs of the cluster
      int8_t* y = a.Y + ((int64_t)b * T + t0) * D;
      const int per = D >> 4;
      for (int i = tid + rank * kRbThreads; i < nrow * per; i += kRbThreads * C) {
        const int r = i / per, c = i - r * per;
        *reinterpret_cast<uint4*>(y + (int64_t)r * D + 16 * c) = *reinterpret_cast<const uint4*>(xs + r * pitch + 16 * c);
      }
    }
  }

  // ---- queries, keys and values of the next block ----
  if (a.last > 4) {
    const int n = 3 * D / C, n0 = rank * n, per = n >> 4;
    const uint8_t* hs = gen + a.h_off;
    for (int i = tid; i < nrow * per; i += kRbThreads) {
      const int r = i / per, c = n0 + 16 * (i - r * per);
      if (c >= 2 * D) continue;
      const uint4 v = *reinterpret_cast<const uint4*>(hs + r * a.n_pitch + (c - n0));
      int8_t* o = c < D ? a.Qn + ((int64_t)b * T + t0 + r) * D + c
                        : a.Kn + (((int64_t)b * a.heads + ((c - D) >> 6)) * a.Tk + t0 + r) * 64 + ((c - D) & 63);
      *reinterpret_cast<uint4*>(o) = v;
    }
    // values transposed: sixteen tokens of a channel are one store
    const int v0 = max(n0, 2 * D), nv = n0 + n - v0;
    for (int i = tid; i < MT * nv; i += kRbThreads) {
      const int mt = i / nv, c = v0 + i - mt * nv;
      if (16 * mt >= nrow) continue;
      const uint8_t* p = hs + 16 * mt * a.n_pitch + (c - n0);
      uint32_t w[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        w[k] = (uint32_t)p[4 * k * a.n_pitch] | (uint32_t)p[(4 * k + 1) * a.n_pitch] << 8 | (uint32_t)p[(4 * k + 2) * a.n_pitch] << 16 |
               (uint32_t)p[(4 * k + 3) * a.n_pitch] << 24;
      *reinterpret_cast<uint4*>(a.Vn + ((int64_t)b * D + c - 2 * D) * a.Tp + t0 + 16 * mt) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
}

constexpr size_t kRbSmem = 227 * 1024;
typedef void (*RbKernel)(RbArgs);

// One kernel per width class and number of 16-row tiles.
RbKernel rb_kernel(int64_t D, int mt) {
#define IVIT_RB(W) (mt == 1 ? block_rows_kernel<W, 1> : (mt == 2 ? block_rows_kernel<W, 2> : block_rows_kernel<W, 3>))
  return D <= 256 ? IVIT_RB(2) : (D <= 384 ? IVIT_RB(3) : (D <= 768 ? IVIT_RB(6) : IVIT_RB(8)));
#undef IVIT_RB
}
int rb_words(int64_t D) { return D <= 256 ? 2 : (D <= 384 ? 3 : (D <= 768 ? 6 : 8)); }

bool aligned32(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 31) == 0; }
bool plain_scale(const ivit_scale& s) { return s.mult_c && aligned16(s.mult_c) && aligned16(s.shift_c); }

size_t up256(size_t v) { return (v + 255) / 256 * 256; }

// Shared-memory plan; 0 when it does not fit.
size_t rb_smem(RbArgs& a, int mt, int64_t D, int64_t H, int64_t heads, int C) {
  const int rows = 16 * mt, nh = (int)((heads + C - 1) / C), words = rb_words(D), nt = words == 3 || words == 6 ? 3 : 2;
  a.q_pitch = 64 * nh + 16;
  a.h_pitch = (int)H + 16;
  a.s_pitch = a.Tp + 16;
  a.n_pitch = (int)(3 * D / C) + 16;
  size_t off = 0;
  auto take = [&](size_t bytes) { const size_t o = off; off = up256(off + bytes); return (uint32_t)o; };
  take((size_t)rows * (D + 16));
  a.a_off = take((size_t)rows * (D + 16));
  a.q_off = take((size_t)rows * a.q_pitch);
  size_t h = (size_t)rows * a.h_pitch;
  if ((size_t)nh * rows * a.s_pitch > h) h = (size_t)nh * rows * a.s_pitch;
  if ((size_t)rows * a.n_pitch > h) h = (size_t)rows * a.n_pitch;
  a.h_off = take(h);
  const int64_t n[4] = {D, H, D, 3 * D};
  for (int i = 0; i < 4; ++i) a.par_off[i] = take((size_t)(n[i] / C) * 9);
  for (int i = 0; i < 2; ++i) a.norm_off[i] = take((size_t)D * 13);
  a.tab_off = take(1024 * kRbCopies + 512);
  a.gelu_off = take(kRbWarps * 256);
  a.red_off = take((size_t)kRbWarps * mt * nt * 4 * 128);
  return off + 256 <= kRbSmem ? off + 256 : 0;
}

}  // namespace

int block_rows_prepare_device() {
  for (int D : {256, 384, 768, 1024})
    for (int mt = 1; mt <= 3; ++mt)
      if (cudaFuncSetAttribute(rb_kernel(D, mt), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRbSmem) != cudaSuccess) return IVIT_ERR_CUDA;
  return IVIT_OK;
}

size_t block_rows_scratch(const ivit_block_params* p) {
  const size_t Tk = (size_t)(p->T + 7) / 8 * 8, Tp = (size_t)(p->T + 63) / 64 * 64;
  const size_t q = up256((size_t)(p->B * p->T * p->D)), k = up256((size_t)(p->B * p->D) * Tk), v = up256((size_t)(p->B * p->D) * Tp);
  return 2 * (q + k + v);
}

// Whether a block goes this way, and how.
BlockRowsPlan block_rows_plan(const ivit_ctx* ctx, const ivit_block_params* p) {
  BlockRowsPlan plan{0, 0};
  const int64_t D = p->D, H = p->H, T = p->T;
  if (ctx->gemm_engine != 0 || ctx->row_fusion || p->B < 1 || D != 64 * p->heads || D > 1024 || H % 64 || H > 512 * rb_words(D) || T > 640) return plan;
  if (!plain_scale(p->ln1_gamma) || !plain_scale(p->qkv_scale) || !plain_scale(p->o_scale) || !plain_scale(p->ln2_gamma) ||
      !plain_scale(p->fc1_scale) || !plain_scale(p->fc2_scale))
    return plan;
  const void* p16[] = {p->bqkv, p->bo, p->b1, p->b2, p->ln1_beta, p->ln2_beta};
  for (const void* q : p16)
    if (!aligned16(q)) return plan;
  const void* p32[] = {p->Wqkv, p->Wo, p->W1, p->W2};
  for (const void* q : p32)
    if (!aligned32(q)) return plan;
  RbArgs a{};
  a.Tp = (int)((T + 63) / 64 * 64);
  if (const char* f = getenv("IVIT_RB")) {   // XXX
    int mt = 0, C = 0;
    sscanf(f, "%d,%d", &mt, &C);
    if (mt && rb_smem(a, mt, D, H, p->heads, C) && D / C % 16 == 0 && H / C % 16 == 0 && C <= p->heads) { plan.mt = mt; plan.C = C; }
    return plan;
  }
  return plan;   // XXX
  for (int mt = 1; mt <= 3; ++mt) {
    const int64_t groups = p->B * ((T + 16 * mt - 1) / (16 * mt));
    if (groups > ctx->sm_count) continue;
    for (int C = 8; C >= 1; C >>= 1) {
      if (groups * C > (C == 1 ? ctx->sm_count : ctx->sm_count / 16 * 14) || C > p->heads) continue;
      if (D / C % 16 || H / C % 16) continue;
      if (!rb_smem(a, mt, D, H, p->heads, C)) continue;
      plan.mt = mt;
      plan.C = C;
      return plan;
    }
  }
  return plan;
}

// One launch: the block `p` from its queries, keys and values on (nullptr: none) and LayerNorm 1 + QKV of `next` (nullptr:
// none) on the result (or on X when p is nullptr).  set: which of the two scratch sets holds p's queries, keys and values.
int launch_block_rows(ivit_ctx* ctx, const BlockRowsPlan& plan, const ivit_block_params* p, const ivit_block_params* next,
                      const int8_t* X, int8_t* Y, char* scratch, int set, bool early) {
  const ivit_block_params* q = p ? p : next;
  RbArgs a{};
  a.T = (int)q->T; a.D = (int)q->D; a.heads = (int)q->heads; a.H = (int)q->H;
  a.groups = (a.T + 16 * plan.mt - 1) / (16 * plan.mt);
  a.C = plan.C;
  a.Tk = (a.T + 7) / 8 * 8;
  a.Tp = (a.T + 63) / 64 * 64;
  a.first = p ? 0 : 4;
  a.last = next ? 5 : 4;
  a.early = early;
  a.X = X; a.Y = Y;
  const size_t sq = up256((size_t)(q->B * a.T) * a.D), sk = up256((size_t)(q->B * a.D) * a.Tk), sv = up256((size_t)(q->B * a.D) * a.Tp);
  int8_t* s0 = reinterpret_cast<int8_t*>(scratch) + (size_t)set * (sq + sk + sv);
  int8_t* s1 = reinterpret_cast<int8_t*>(scratch) + (size_t)(1 - set) * (sq + sk + sv);
  a.Q = s0; a.K = s0 + sq; a.V = s0 + sq + sk;
  a.Qn = s1; a.Kn = s1 + sq; a.Vn = s1 + sq + sk;
  auto dense = [](const int8_t* W, const ivit_scale& s, const int32_t* bias) { return RbDense{W, s.mult_c, s.shift_c, bias}; };
  auto norm = [](const ivit_scale& s, const int32_t* beta, int M) { return RbNorm{s.mult_c, s.shift_c, beta, M}; };
  double work = 0;
  const double rows = (double)q->B * a.T, dD = (double)a.D;
  int steps = 0;
  if (p) {
    a.qk_m = p->qk_scale.mult; a.qk_s = clamp_shift(p->qk_scale.shift);
    a.pv_m = p->pv_scale.mult; a.pv_s = clamp_shift(p->pv_scale.shift);
    a.smax = p->smax;
    a.fast = p->smax.k_out == 8 && ((int64_t)p->smax.I0 << p->smax.N) > (1 << 15);
    for (int i = 0; i < 4; ++i) a.sel[i] = exp_sel(kRbCopies, i);
    a.bias = p->attn_bias;
    a.bias_batches = p->attn_bias ? (int)p->attn_bias_batches : 1;
    a.dense[0] = dense(p->Wo, p->o_scale, p->bo);
    a.dense[1] = dense(p->W1, p->fc1_scale, p->b1);
    a.dense[2] = dense(p->W2, p->fc2_scale, p->b2);
    a.res_m[0] = p->res1_scale.mult; a.res_s[0] = clamp_shift(p->res1_scale.shift);
    a.res_m[1] = p->res2_scale.mult; a.res_s[1] = clamp_shift(p->res2_scale.shift);
    a.norm[0] = norm(p->ln2_gamma, p->ln2_beta, p->M_ln);
    if (p->gelu_static_max) {
      const int8_t* row127;
      const int rc = gelu_static_row(ctx, p->gelu, p->gelu_post, &row127);
      if (rc) return rc;
      a.gelu = row127 - 127 * 256;
      a.gelu_max = 127;
    } else {
      const int rc = gelu_table_for(ctx, p->gelu, p->gelu_post, &a.gelu);
      if (rc) return rc;
      a.gelu_max = -1;
    }
    work += 2.0 * rows * dD * (dD + 2.0 * a.H) + 4.0 * rows * a.T * dD;
    steps += p->gelu_static_max ? 5 : 6;   // attention, projection, LayerNorm, FC1, (ShiftGELU,) FC2
  }
  if (next) {
    a.dense[3] = dense(next->Wqkv, next->qkv_scale, next->bqkv);
    a.norm[1] = norm(next->ln1_gamma, next->ln1_beta, next->M_ln);
    work += 6.0 * rows * dD * dD;
    steps += 2;                            // LayerNorm, QKV
  }
  a.mean_magic = (unsigned)(0x100000000ull / (unsigned long long)(2 * a.D)) + 1u;
  const size_t smem = rb_smem(a, plan.mt, a.D, a.H, a.heads, a.C);
  if (!smem) return IVIT_ERR_UNSUPPORTED;
  LaunchScope ls(ctx, KIND_BLOCK_ROWS, work);
  launch_k_cluster(rb_kernel(a.D, plan.mt), dim3((unsigned)(q->B * a.groups * a.C)), dim3(kRbThreads), smem, ctx->stream, a.C, a);
  ctx->launches += steps - 1;
  return ls.done();
}

}  // namespace ivit
