// Fused attention core of one encoder block (Sec. 3.1 MSA equation, Sec. 3.2 and Algorithm 1):
//   S = Q_i K_i^T (+ bias)  ->  requantise to int8  ->  Shiftmax  ->  P_i V_i  ->  requantise
// for one head and 128 score rows at a time: attention_short_kernel (rows of up to 256 tokens, several short windows
// packed into the 128 rows) and attention_rows_kernel (longer rows).
//
// The int32 score tile lives in tensor memory, never in HBM.  Several threads share one score row (a TMEM lane) and
// take different columns of it, so the row maximum and the row sum of Algorithm 1 need one exchange through shared
// memory each: no shuffles.  Three passes over the scores:
//   pass A  requantise to int8, running maximum;
//   pass B  ShiftExp by look-up (256 entries, I_max - I in [0, 255]), row sum.  The table is kept `cp` times in shared
//           memory, copy (lane mod cp) serving a lane, so that look-ups do not collide on banks; dp4a with one non-zero
//           byte turns a packed score into its entry's address in one instruction;
//   pass C  one reciprocal per row (Eq. (IntDiv)), then exp * reciprocal >> shift per value; the int8 probabilities are
//           written to shared memory in the K-major 128B-swizzled layout that P V consumes as its A operand.
// V is consumed as stored ([token, d] rows, MN-major B operand).  Every wait is bounded.
// What bounds the kernels: the chain of an item (scores, pass A, exchange, pass B, exchange, pass C, P V, output), of which
// an SM has two in flight, or parts of two: on short rows issue slots are busy in 43 % of the cycles and no pipe in more than
// 28 %.  Inside a pass mad.hi / mul.hi take four cycles of a scheduler (measured), the other integer instructions two
// cycles of their pipe, a look-up one of the SM's shared-memory cycles.
#include "handover.cuh"
#include "setup.cuh"
#include "shiftmax.cuh"
#include "tc_ptx.cuh"

namespace ivit {

namespace {

constexpr int UK = 32;              // K of one tcgen05.mma.kind::i8

// Eq. (IntDiv) with M = 45 for four exponentials: (floor(2^45 / sum) * e) >> (45 - (k_out - 1)) = umulhi(factor, e) >> (14 - k_out),
// clamped to 2^(k_out-1) - 1 and packed.
__device__ __forceinline__ uint32_t prob_word(unsigned factor, int e0, int e1, int e2, int e3, int osh, int omax) {
  return pack_sat8(min((int)(__umulhi(factor, (unsigned)e0) >> osh), omax), min((int)(__umulhi(factor, (unsigned)e1) >> osh), omax),
                   min((int)(__umulhi(factor, (unsigned)e2) >> osh), omax), min((int)(__umulhi(factor, (unsigned)e3) >> osh), omax));
}
// Fields that both kernels use.
struct AttnArgs {
  int T, d, heads;
  int64_t D;                        // heads * d
  int bh;                           // images x heads
  int items;
  int kpad;                         // contraction length of P V: T rounded up to 32 (packed windows: 128)
  int kbox;                         // rows of a key box (packed windows: rows of a slot)
  int cp;                           // copies of the ShiftExp table (a power of two, at most 32)
  uint32_t sel[4];                  // -4 cp as a signed byte, in byte 0, 1, 2, 3
  int chunks;                       // 16-column chunks of a row, the last one with T & 15 columns when that is not 0
  int qk_m, qk_s, pv_m, pv_s;
  ivit_exp_params smax;
  const int32_t* bias;              // [bias_batches, T, T] or nullptr
  int bias_vec;                     // the bias starts at a 16-byte boundary
  int bias_batches;
  int8_t* O;                        // [B*T, D]
  int q_pos[3], k_pos[3], v_pos[3];
  int* status;
};

// A work item: head h of image b, 128 rows from m0 on (packed windows: head h of the windows from window b on).
struct __align__(16) AttnItem {
  int h, b, m0;
  int rot;      // row group g (32 rows) of the tile stands in lane quarter (g + rot) & 3: the quarters (and schedulers)
                // that a ragged tile leaves idle change from item to item
  // The n-th work item of a CTA.  Items are ordered tile by tile, the ragged last tiles at the end, and dealt in a snake:
  // item n gridDim + blockIdx for even n, the mirror image for odd n, so that a CTA with one item more than others has
  // it among the ragged tiles.
  __device__ __forceinline__ void init(const AttnArgs& a, uint32_t n) {
    unsigned t = n * gridDim.x + ((n & 1u) ? gridDim.x - 1 - blockIdx.x : blockIdx.x);
    m0 = 0;
    while (t >= (unsigned)a.bh) { t -= (unsigned)a.bh; m0 += 128; }
    b = (int)(t / (unsigned)a.heads);
    h = (int)t - b * a.heads;
    rot = m0 + 128 >= a.T ? (int)(t & 3u) : 0;
  }
  static __device__ __forceinline__ uint32_t count(const AttnArgs& a) {
    const uint32_t rounds = (uint32_t)a.items / gridDim.x, left = (uint32_t)a.items % gridDim.x;
    return rounds + (((rounds & 1u) ? gridDim.x - 1 - blockIdx.x : blockIdx.x) < left ? 1u : 0u);
  }
};

// Named barriers: id, number of threads that arrive or wait.
__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id, int n) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory"); }
constexpr int kBarSetup = 8, kBarTmem = 9;   // (6 and 7: handover.cuh)
template <int kThreads>
struct ShortSetup {
  __device__ __forceinline__ void arrive() const { bar_arrive(kBarSetup, kThreads); }
  __device__ __forceinline__ void sync() const { bar_sync(kBarSetup, kThreads); }
  __device__ __forceinline__ void trigger() const { pdl_trigger(); }
};
template <int kThreads>
struct BlockBarriers {
  __device__ __forceinline__ void sync(int id) const { bar_sync(id, kThreads); }
};

// Tile load by a converged warp; pos: which coordinate of the map (1..3) carries the row, the head and the image or window.
__device__ __forceinline__ void load_box(uint32_t dst, const CUtensorMap* map, uint32_t bar, const int (&pos)[3], int row, int h, int b) {
  tma_load_4d_w(dst, map, bar, 0, pos[0] == 1 ? row : (pos[1] == 1 ? h : b), pos[0] == 2 ? row : (pos[1] == 2 ? h : b),
              pos[0] == 3 ? row : (pos[1] == 3 ? h : b));
}

// Constants of the inner loops, held in registers (the compiler would fetch them again for every use).
struct PassConsts {
  uint32_t sel[4];
  int qk_m, qk_rnd, qk_sh;
  __device__ __forceinline__ void init(const AttnArgs& a) {
#pragma unroll
    for (int i = 0; i < 4; ++i) asm volatile("mov.b32 %0, %1;" : "=r"(sel[i]) : "r"(a.sel[i]));
    asm volatile("mov.b32 %0, %1;" : "=r"(qk_m) : "r"(a.qk_m));
    asm volatile("mov.b32 %0, %1;" : "=r"(qk_rnd) : "r"(a.qk_s >= 33 ? 1 << (a.qk_s - 33) : 0));
    asm volatile("mov.b32 %0, %1;" : "=r"(qk_sh) : "r"(a.qk_s - 32));
  }
};

// Pass A on W scores: requantise, columns from `valid` on (at most W) become -128 when EDGE, maximum into mx, packed
// into x.  FAST: the shift is >= 33 (high product word plus 2^(s-33), shifted by s - 32).
template <bool FAST, bool EDGE, int W>
__device__ __forceinline__ void score_piece(const AttnArgs& a, const PassConsts& k, int (&v)[W], int valid, int& mx, uint32_t* x) {
#pragma unroll
  for (int i = 0; i < W; ++i) {
    if (FAST) v[i] = mad_hi(v[i], k.qk_m, k.qk_rnd) >> k.qk_sh;
    else v[i] = (int)(((long long)v[i] * a.qk_m + (1ll << (a.qk_s - 1))) >> a.qk_s);
  }
  if (EDGE) {
#pragma unroll
    for (int i = 0; i < W; ++i)
      if (i >= valid) v[i] = -128;
  }
#pragma unroll
  for (int i = 0; i < W; i += 2) mx = __vimax3_s32(mx, v[i], v[i + 1]);
#pragma unroll
  for (int q = 0; q < W / 4; ++q) x[q] = pack_sat8(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
}
// Adds 16 entries of a bias row, p[0 .. 15], to a chunk of scores.  A lane has a row of its own, so that every load instruction
// touches 32 lines, and their number is what counts: four 16-byte loads from the boundary at or before p, and the up to three
// words behind them one by one, instead of sixteen.  (The boundary is not before the bias, see bias_vec.)  Measured with a bias:
// 8 x 197 tokens, 12 heads 24.6 -> 16.7 us, 64 x 197 85 -> 65, 32 x 400, 6 heads 149 -> 66.
template <bool VEC>
__device__ __forceinline__ void add_bias_row(int (&v)[16], const int32_t* p) {
  if (!VEC) {
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] += __ldg(p + i);
    return;
  }
  const int sh = (int)((reinterpret_cast<uintptr_t>(p) >> 2) & 3u);
  const int4* q = reinterpret_cast<const int4*>(p - sh);
  int w[19];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int4 x = __ldg(q + k);
    w[4 * k] = x.x; w[4 * k + 1] = x.y; w[4 * k + 2] = x.z; w[4 * k + 3] = x.w;
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) w[16 + i] = i < sh ? __ldg(p - sh + 16 + i) : 0;
#pragma unroll
  for (int i = 0; i < 17; ++i) w[i] = sh & 2 ? w[i + 2] : w[i];
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] += sh & 1 ? w[i + 1] : w[i];
}
// Bytes of word q of an edge chunk that hold columns below `valid`.
__device__ __forceinline__ uint32_t edge_mask(int valid, int q) {
  return valid >= 4 * q + 4 ? 0xffffffffu : (valid <= 4 * q ? 0u : 0xffffffffu >> (8 * (4 * q + 4 - valid)));
}
// O = sat8(rq(P V; pv_scale)) of 16 columns.
template <bool FAST>
__device__ __forceinline__ uint4 output_piece(const AttnArgs& a, int (&v)[16]) {
  if (FAST) {
    const int rnd = 1 << (a.pv_s - 33), sh = a.pv_s - 32;
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = mad_hi(v[i], a.pv_m, rnd) >> sh;
  } else {
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = (int)(((long long)v[i] * a.pv_m + (1ll << (a.pv_s - 1))) >> a.pv_s);
  }
  return make_uint4(pack_sat8(v[0], v[1], v[2], v[3]), pack_sat8(v[4], v[5], v[6], v[7]),
                    pack_sat8(v[8], v[9], v[10], v[11]), pack_sat8(v[12], v[13], v[14], v[15]));
}

// ------------------------------------------------------------------------------------------------------------
// Rows of up to 256 tokens.  Several CTAs per SM: they are at different points of their items, which covers the waits that
// an item cannot avoid (score MMAs, row exchanges, P V) and mixes passes that need different pipes.  Only the control
// warp polls; the others wait in hardware barriers that it releases.
//   TPR = 2        128 rows of one image; two CTAs (tensor memory holds two score tiles of 256 columns), two threads per
//                  score row, which take alternate 16-column chunks
//   TPR = 4        the same with one CTA and four threads per score row, for launches of at most one item per SM whose rows are
//                  long enough
//   TPR = 1 (kPack)  G windows of up to R = 128 / G tokens share the 128 rows (window attention): the score tile is
//                  block-diagonal and the probabilities outside a row's own window stay 0.  The int32 score bias of
//                  the tile's windows is kept in shared memory (rows padded to an odd number of words, so that the 32
//                  rows of a warp fall into different banks) and only fetched when it differs from the last item's;
//                  items are ordered so that it rarely does (per head and window position, images innermost).  Read
//                  straight from global memory, one row per lane, it took most of the kernel's time.  Four CTAs with a
//                  thread per score row: no row exchange (4096 windows of 49 tokens, 6 heads of 32, bias: 113 us; two
//                  CTAs with two threads per row 146, three 158).
// Everything of an item stays in tensor memory: the score columns hold the packed int8 scores after pass A, the
// exponentials after pass B, and O = P V at the end.
// Measured, back to back (before: one table, items drawn from a counter, bias read from global memory, every warp polling):
// 64 x 197 tokens, 6 heads of 64 29.0 -> 19.5 us; 128 x 197, 12 heads 89.1 -> 61.7; 1 x 197, 3 heads 10.1 -> 5.9.
// Threads per score row (TPR) and CTAs per SM.  Warp 0: TMA + MMA issue; TPR warps per lane quarter, the first of which owns tensor memory.
template <int TPR>
struct ShortShape {
  static constexpr int kCtas = 4 / TPR, kWorkers = 128 * TPR, kThreads = 32 + kWorkers;
  static constexpr int kPartials = (TPR > 1 ? 2 * TPR : 4) * 128 * 4;   // bytes
};

struct ShortArgs {
  AttnArgs a;
  int G, R, Btot;                   // kPack: windows per tile, rows per window slot, windows in the tensor
  unsigned t_magic;                 // floor(2^32 / T) + 1
  int units, npos;                  // kPack: tiles per head; window-position groups with a bias of their own per head
  int tmem_cols;
};

template <int TPR, bool FAST, bool BIAS>
__global__ void __launch_bounds__(ShortShape<TPR>::kThreads, ShortShape<TPR>::kCtas) attention_short_kernel(const __grid_constant__ CUtensorMap tmQ,
                                                                                       const __grid_constant__ CUtensorMap tmK,
                                                                                       const __grid_constant__ CUtensorMap tmV,
                                                                                       ShortArgs sa) {
  constexpr bool kPack = TPR == 1;
  constexpr int kShortThreads = ShortShape<TPR>::kThreads, kWorkers = ShortShape<TPR>::kWorkers;
  const AttnArgs& a = sa.a;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* gen = smem_raw + (base - smem_u32(smem_raw));
  // [Q 128 x d][K][V kpad x d][P 128 x 128B x kblocks][table 256 x cp][row partials][seeds][items][barriers][window bias]
  const uint32_t k_bytes = (uint32_t)(kPack ? 128 : a.kbox) * a.d, v_bytes = (uint32_t)a.kpad * a.d;
  const uint32_t k_off = 128u * a.d, v_off = k_off + k_bytes;
  const uint32_t p_off = (v_off + v_bytes + 1023u) & ~1023u;
  const uint32_t tab_off = p_off + (uint32_t)((a.kpad + 127) / 128) * 128 * 128;
  const uint32_t part_off = tab_off + 1024u * a.cp;      // [TPR][128 rows] partial max, then partial sum
  const uint32_t seed_off = part_off + ShortShape<TPR>::kPartials;      // [128] seeds of the reciprocal
  const uint32_t item_off = seed_off + 128 * 4;          // [2] work item of even / odd iterations, written before its scores
  const uint32_t bar_off = item_off + 2 * sizeof(AttnItem);
  const uint32_t bias_off = bar_off + 64;                // kPack && BIAS: [G][T][T | 1]
  AttnItem* const item_ring = reinterpret_cast<AttnItem*>(gen + item_off);
  // Q and K landed | V landed | scores ready | probabilities written | output ready | output read
  const uint32_t bar_qk = base + bar_off, bar_v = bar_qk + 8, bar_s = bar_qk + 16, bar_p = bar_qk + 24,
                 bar_o = bar_qk + 32, bar_e = bar_qk + 40;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gen + bar_off + 48);
  volatile uint32_t* dead = tmem_slot + 1;               // set when a wait of the control warp ran out

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  // Set-up.  The control warp initialises the barriers and goes on to its first loads; the warp behind it owns tensor memory,
  // whose address the control warp takes at a barrier of the two in front of its first MMA.
  if (threadIdx.x == 0) {
    mbar_init(bar_qk, 1);
    mbar_init(bar_v, 1);
    mbar_init(bar_s, 1);
    mbar_init(bar_p, 4 * TPR);
    mbar_init(bar_o, 1);
    mbar_init(bar_e, 4 * TPR);
    *dead = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  uint32_t tmem = 0;
  if (warp == 0) {
    __syncwarp();
    end_of_setup(ShortSetup<kShortThreads>{}, true);
    if (lane == 0) {
      prefetch_tmap(&tmQ);
      prefetch_tmap(&tmK);
      prefetch_tmap(&tmV);
    }
  } else {
    if (warp == 1) {
      tmem_alloc(smem_u32(tmem_slot), (uint32_t)sa.tmem_cols);
      tc_fence_before();
      bar_arrive(kBarTmem, 64);
    }
    end_of_setup(ShortSetup<kShortThreads>{}, false);
    tc_fence_after();
    tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
  }
  // items of this CTA: a snake over all of them, or (kPack) a contiguous range
  const uint32_t rounds = (uint32_t)a.items / gridDim.x, left = (uint32_t)a.items % gridDim.x;
  const uint32_t n_items = kPack ? rounds + (blockIdx.x < left ? 1u : 0u) : AttnItem::count(a);
  const uint32_t first = blockIdx.x * rounds + min(blockIdx.x, left);   // kPack
  const uint32_t imgs = kPack ? (uint32_t)sa.units / (uint32_t)sa.npos : 1u;   // kPack: items in a row with the same bias

  if (warp == 0) {
    if (n_items > 0) {
      auto item_at = [&](AttnItem& it, uint32_t n) {
        if (kPack) {
          const unsigned t = first + n, grp = t / imgs, img = t - grp * imgs;
          it.h = (int)(grp / (unsigned)sa.npos);
          it.b = (int)(grp - (unsigned)it.h * sa.npos + img * sa.npos) * sa.G;
          it.m0 = 0;
          it.rot = 0;
        } else {
          it.init(a, n);
        }
      };
      auto load_qk = [&](const AttnItem& it) {
        mbar_expect_tx_w(bar_qk, 128u * a.d + k_bytes);
        if (kPack) {
          load_box(base, &tmQ, bar_qk, a.q_pos, 0, it.h, it.b);
        } else {
          for (int g = 0; g < 4; ++g)
            load_box(base + (uint32_t)((g + it.rot) & 3) * 32u * a.d, &tmQ, bar_qk, a.q_pos, it.m0 + 32 * g, it.h, it.b);
        }
        load_box(base + k_off, &tmK, bar_qk, a.k_pos, 0, it.h, it.b);
      };
      auto load_v = [&](const AttnItem& it) {
        mbar_expect_tx_w(bar_v, v_bytes);
        load_box(base + v_off, &tmV, bar_v, a.v_pos, 0, it.h, it.b);
      };
      // descriptor words: rows of d bytes (Q, K, V: swizzled over their width) or 128 bytes (P)
      const uint32_t layout = a.d == 128 ? 2u : (a.d == 64 ? 4u : 6u);
      const uint32_t row_hi = desc_hi(8u * a.d, layout), p_hi = desc_hi(1024, 2);
      const uint32_t q_lo = desc_lo(base, 16), k_lo = desc_lo(base + k_off, 16), p_lo0 = desc_lo(base + p_off, 16),
                     v_lo0 = desc_lo(base + v_off, 16), v_step = (uint32_t)(UK * a.d) >> 4;
      const int s_cols = kPack ? 128 : 16 * a.chunks;
      const uint32_t idesc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(s_cols >> 3) << 17) | (8u << 24);
      const uint32_t idesc2 = (2u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(a.d >> 3) << 17) | (8u << 24);
      const int ks = a.d / UK, ks2 = a.kpad / UK;

      AttnItem cur, next;
      item_at(cur, 0);
      bool qk_flying = true, v_flying = true;   // loads issued and not yet waited for (their barrier phase = item count)
      uint32_t qk_par = 0, v_par = 0;
      pdl_wait();   // the QKV tensor comes from the previous kernel; the other warps build their table first
      load_qk(cur);
      load_v(cur);
      bar_sync(kBarTmem, 64);
      tc_fence_after();
      tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
      bool ok = true;
      bool scores_out = false;
      uint32_t done = 0;                // items whose output is there
      for (uint32_t n = 0; n < n_items; ++n) {
        const uint32_t par = n & 1u;
        ok = mbar_wait_warp(bar_qk, par, a.status);
        qk_flying = !ok;
        // the output of the previous item must have left tensor memory
        if (ok && n > 0) ok = mbar_wait_warp(bar_e, par ^ 1u, a.status);
        if (!ok) break;
        if (lane == 0) item_ring[par] = cur;
        tc_fence_after();
        for (int k = 0; k < ks; ++k)
          umma_i8_lohi_w(tmem, q_lo + k * (UK >> 4), row_hi, k_lo + k * (UK >> 4), row_hi, idesc, k != 0);
        umma_commit_w(bar_s);
        const bool more = n + 1 < n_items;
        if (more) item_at(next, n + 1);
        // Q and K may be overwritten once the score MMAs have read them
        ok = mbar_wait_warp(bar_s, par, a.status);
        if (!ok) break;
        bar_arrive(kBarScores, kShortThreads);
        scores_out = true;
        if (more) { load_qk(next); qk_flying = true; qk_par = par ^ 1u; }
        // O = P V once the probabilities are in shared memory and V has landed
        ok = mbar_wait_warp(bar_p, par, a.status);
        if (ok) { ok = mbar_wait_warp(bar_v, par, a.status); v_flying = !ok; }
        if (!ok) break;
        tc_fence_after();
        uint32_t p_lo = p_lo0, v_lo = v_lo0;
        int k = 0;
        for (; k + 4 <= ks2; k += 4, p_lo += (128 * 128) >> 4, v_lo += 4 * v_step)
          umma_i8_x4_w(tmem, p_lo, p_hi, v_lo, row_hi, idesc2, k != 0, UK >> 4, v_step);
        for (; k < ks2; ++k, p_lo += UK >> 4, v_lo += v_step)
          umma_i8_lohi_w(tmem, p_lo, p_hi, v_lo, row_hi, idesc2, k != 0);
        umma_commit_w(bar_o);
        // V may be overwritten once these MMAs have read it
        ok = mbar_wait_warp(bar_o, par, a.status);
        if (!ok) break;
        bar_arrive(kBarOutput, kShortThreads);
        ++done;
        scores_out = false;
        if (more) { load_v(next); v_flying = true; v_par = par ^ 1u; }
        cur = next;
      }
      if (!ok) {
        // a wait ran out: see walk_out
        if (lane == 0) *dead = 1;
        __syncwarp();
        walk_out(BlockBarriers<kShortThreads>{}, done, n_items, scores_out);
      }
      // nothing may be in flight at exit
      if (qk_flying) mbar_wait_warp(bar_qk, qk_par, a.status);
      if (v_flying) mbar_wait_warp(bar_v, v_par, a.status);
    }
  } else {
    // ---- Shiftmax / epilogue threads: TMEM lane quarter = warp % 4; the TPR warps of a quarter take every TPR-th chunk
    //      of the same 32 rows ----
    const int st = threadIdx.x - 32;
    const int qd = warp & 3;
    const int half = (warp - 1) >> 2;
    const int trow = qd * 32 + lane;              // row inside the tile
    build_exp_table(a.smax.I0, a.smax.N, a.cp, gen + tab_off, st, kWorkers);
    // probabilities that no item writes are 0: columns past the last chunk, other windows' columns
    for (int c = (kPack ? 0 : a.chunks) + half; c < a.kpad / 16; c += TPR)
      *reinterpret_cast<uint4*>(gen + p_off + (c >> 3) * (128 * 128) + trow * 128 + (((c & 7) ^ (trow & 7)) << 4)) = make_uint4(0u, 0u, 0u, 0u);
    unsigned* seeds = reinterpret_cast<unsigned*>(gen + seed_off);
    if (st < 128) seeds[st] = recip_seed(st);
    pdl_wait();
    PassConsts kc;
    kc.init(a);
    const uint32_t t_row = tmem + ((uint32_t)(qd * 32) << 16);
    int* part_max = reinterpret_cast<int*>(gen + part_off);
    unsigned* part_sum = reinterpret_cast<unsigned*>(gen + part_off + TPR * 128 * 4);
    const uint32_t tab_lane = base + tab_off + 4u * (unsigned)(lane & (a.cp - 1));
    const unsigned top = (unsigned)a.smax.I0 << a.smax.N;    // the largest exponential
    const int osh = 14 - a.smax.k_out, omax = (1 << (a.smax.k_out - 1)) - 1;
    // this row's whole chunks: c_lo .. c_full - 1, this thread takes every TPR-th one; rem columns remain, which the
    // thread whose turn it is takes as a piece of eight or sixteen columns
    const int slot = kPack ? trow / sa.R : 0;
    const int c_lo = kPack ? slot * (sa.R >> 4) : 0, c_full = c_lo + (a.T >> 4);
    const int rem = half == (c_full - c_lo) % TPR ? a.T & 15 : 0;
    uint8_t* const p_row = gen + p_off + trow * 128;
    auto p_addr = [&](int c) { return reinterpret_cast<uint4*>(p_row + (c >> 3) * (128 * 128) + (((c & 7) ^ (trow & 7)) << 4)); };
    const int bias_ld = a.T | 1;
    uint32_t img = kPack ? first % imgs : 0u;   // kPack: items with the present bias that are behind
    bar_sync(1, kWorkers);   // the table is complete

    bool alive = true;   // false after a wait of the control warp timed out: no more work, only the barriers
    for (uint32_t n = 0; n < n_items; ++n) {
      const uint32_t par = n & 1u;
      // The control warp alone polls the barriers of the MMAs; the others wait in hardware barriers (eight polling warps
      // per CTA issued a third of the kernel's instructions).
      bar_sync(kBarScores, kShortThreads);
      alive = *dead == 0;
      const AttnItem item = item_ring[par];
      const int b = kPack ? item.b + slot : item.b;          // image / window of this row
      const int m0 = kPack ? qd * 32 - slot * sa.R : item.m0 + ((qd - item.rot) & 3) * 32;   // first row (token) of this lane quarter
      const int r = m0 + lane;
      const bool row_ok = r < a.T && (!kPack || b < sa.Btot);
      const bool work = alive && m0 < a.T && (!kPack || b < sa.Btot);   // else the warp only keeps the barriers
      const int32_t* brow = nullptr;
      if (BIAS && kPack) {
        // (decided on the item's number alone: every thread takes the same branch)
        if (n == 0 || img == imgs) {
          if (img == imgs) img = 0;
          bar_sync(1, kWorkers);     // pass A of the last item is behind
          for (int s = 0; alive && s < sa.G; ++s) {
            const int32_t* src = a.bias + (int64_t)((unsigned)((item.b + s) * a.heads + item.h) % (unsigned)a.bias_batches) * a.T * a.T;
            int* dst = reinterpret_cast<int*>(gen + bias_off) + s * a.T * bias_ld;
            const int tt = a.T * a.T;
            for (int i0 = st; i0 < tt; i0 += kWorkers * 8) {   // eight loads in flight
              int v[8];
#pragma unroll
              for (int u = 0; u < 8; ++u) v[u] = i0 + kWorkers * u < tt ? __ldg(src + i0 + kWorkers * u) : 0;
#pragma unroll
              for (int u = 0; u < 8; ++u) {
                const unsigned i = (unsigned)(i0 + kWorkers * u), rr = __umulhi(i, sa.t_magic);   // i / T
                if (i < (unsigned)tt) dst[rr * bias_ld + (i - rr * a.T)] = v[u];
              }
            }
          }
          bar_sync(1, kWorkers);
        }
        ++img;
        brow = reinterpret_cast<const int*>(gen + bias_off) + (slot * a.T + (row_ok ? r : 0)) * bias_ld - 16 * c_lo;
      } else if (BIAS) {
        brow = a.bias + ((int64_t)((unsigned)(item.b * a.heads + item.h) % (unsigned)a.bias_batches) * a.T + (row_ok ? r : 0)) * a.T;
      }
      auto add_bias = [&](auto& v, int col, int valid) {
        if constexpr (BIAS) {
#pragma unroll
          for (int i = 0; i < (int)(sizeof(v) / sizeof(int)); ++i)
            if (i < valid) v[i] += kPack ? brow[col + i] : __ldg(brow + col + i);
        }
      };
      auto add_bias16 = [&](int (&v)[16], int col) {
        if constexpr (BIAS && kPack) add_bias(v, col, 16);
        else if constexpr (BIAS) { if (a.bias_vec) add_bias_row<true>(v, brow + col); else add_bias_row<false>(v, brow + col); }
      };

      // pass A; four packed scores to a word in the first columns of the chunk's own
      if (alive) tc_fence_after();
      int mx = -128;
      if (work) {
#pragma unroll 1
        for (int c = c_lo + half; c < c_full; c += 2 * TPR) {
          int v[2][16];
          const bool second = c + TPR < c_full;
          tmem_ld16_issue(t_row + 16 * c, v[0]);
          if (second) tmem_ld16_issue(t_row + 16 * (c + TPR), v[1]);
          uint32_t x[4];
          tmem_ld_wait16(v[0]);
          add_bias16(v[0], 16 * c);
          score_piece<FAST, false>(a, kc, v[0], 16, mx, x);
          tmem_st4(t_row + 16 * c, x);
          if (second) {
            tmem_ld_wait16(v[1]);
            add_bias16(v[1], 16 * (c + TPR));
            score_piece<FAST, false>(a, kc, v[1], 16, mx, x);
            tmem_st4(t_row + 16 * (c + TPR), x);
          }
        }
        if (rem > 8) {
          int v[16];
          uint32_t x[4];
          tmem_ld16(t_row + 16 * c_full, v);
          add_bias(v, 16 * c_full, rem);
          score_piece<FAST, true>(a, kc, v, rem, mx, x);
          tmem_st4(t_row + 16 * c_full, x);
        } else if (rem) {
          int v[8];
          uint32_t x[2];
          tmem_ld8(t_row + 16 * c_full, v);
          add_bias(v, 16 * c_full, rem);
          score_piece<FAST, true>(a, kc, v, rem, mx, x);
          tmem_st2(t_row + 16 * c_full, x);
        }
        tmem_st_wait();
        mx = max(-128, min(127, mx));
        if (TPR > 1) part_max[half * 128 + trow] = mx;
      }
      // the threads of a row exchange their partial results: a barrier of the warps that share its 32 rows
      if (TPR > 1) {
        bar_sync(2 + qd, 32 * TPR);
#pragma unroll
        for (int i = 0; i < TPR; ++i) mx = max(mx, part_max[i * 128 + trow]);
      }
      unsigned sum = 0;
      if (work) {
        // pass B: entry (I_max - I) of this lane's table copy stands at tab_lane + 4 cp (I_max - I)
        const uint32_t tmx = tab_lane + (uint32_t)(4 * a.cp * mx);
#pragma unroll 2
        for (int c = c_lo + half; c < c_full; c += TPR) {
          uint32_t x[4];
          tmem_ld4(t_row + 16 * c, x);
          int e[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) e[i] = (int)exp_entry(x[i >> 2], kc.sel[i & 3], tmx);
          tmem_st16(t_row + 16 * c, e);
#pragma unroll
          for (int i = 0; i < 16; i += 4) sum += ((unsigned)e[i] + (unsigned)e[i + 1]) + ((unsigned)e[i + 2] + (unsigned)e[i + 3]);
        }
        if (rem) {   // word by word: a class token leaves one or five columns
          uint32_t x[4];
          tmem_ld4(t_row + 16 * c_full, x);
          int e[16];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            e[4 * q] = e[4 * q + 1] = e[4 * q + 2] = e[4 * q + 3] = 0;
            if (4 * q < rem) {
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                e[4 * q + i] = 4 * q + i < rem ? (int)exp_entry(x[q], kc.sel[i], tmx) : 0;
                sum += (unsigned)e[4 * q + i];
              }
            }
          }
          tmem_st16(t_row + 16 * c_full, e);
        }
        tmem_st_wait();
        if (TPR > 1) part_sum[half * 128 + trow] = sum;
      }
      if (TPR > 1) {
        bar_sync(2 + qd, 32 * TPR);
        sum = 0;
#pragma unroll
        for (int i = 0; i < TPR; ++i) sum += part_sum[i * 128 + trow];
      }
      if (work) {
        // pass C: Eq. (IntDiv) with M = 45
        const unsigned factor = FAST ? prob_factor4(sum, top, seeds) : (unsigned)((1ull << 45) / (unsigned long long)(sum ? sum : 1u));
        auto word = [&](int e0, int e1, int e2, int e3) {
          return FAST ? prob_word8(factor, e0, e1, e2, e3) : prob_word(factor, e0, e1, e2, e3, osh, omax);
        };
        auto words = [&](const int (&e)[16]) {
          return make_uint4(word(e[0], e[1], e[2], e[3]), word(e[4], e[5], e[6], e[7]), word(e[8], e[9], e[10], e[11]),
                            word(e[12], e[13], e[14], e[15]));
        };
#pragma unroll 1
        for (int c = c_lo + half; c < c_full; c += 2 * TPR) {
          int e[2][16];
          const bool second = c + TPR < c_full;
          tmem_ld16_issue(t_row + 16 * c, e[0]);
          if (second) tmem_ld16_issue(t_row + 16 * (c + TPR), e[1]);
          tmem_ld_wait16(e[0]);
          *p_addr(c) = words(e[0]);
          if (second) {
            tmem_ld_wait16(e[1]);
            *p_addr(c + TPR) = words(e[1]);
          }
        }
        if (rem) {
          int e[16];
          tmem_ld16(t_row + 16 * c_full, e);
          uint32_t o[4] = {0u, 0u, 0u, 0u};
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (4 * q < rem) o[q] = word(e[4 * q], e[4 * q + 1], e[4 * q + 2], e[4 * q + 3]);
          *p_addr(c_full) = make_uint4(o[0], o[1], o[2], o[3]);
        }
        fence_async_smem();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_p);
      // ---- output, heads concatenated along the feature dimension ----
      bar_sync(kBarOutput, kShortThreads);
      alive = alive && *dead == 0;
      if (work && alive) {
        tc_fence_after();
        int8_t* orow = a.O + ((int64_t)b * a.T + r) * a.D + (int64_t)item.h * a.d;
#pragma unroll 1
        for (int c = half; c < a.d / 16; c += TPR) {
          int v[16];
          tmem_ld16(t_row + 16 * c, v);
          const uint4 w = output_piece<FAST>(a, v);
          if (row_ok) *reinterpret_cast<uint4*>(orow + 16 * c) = w;
        }
      }
      // tensor memory may take the next item's scores
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_e);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, (uint32_t)sa.tmem_cols);
  }
}

// ------------------------------------------------------------------------------------------------------------
// Rows of more than 256 tokens.  One CTA per SM; sixteen Shiftmax warps share a 128-row tile, four threads per score row
// (thread `part` takes the 16-column chunks part, part + 4, ...).
//   S       the score columns are taken in blocks of 192, each in one of two tensor-memory buffers; the MMA of the next
//           block, or of the next work item, runs while the Shiftmax passes work on the scores already read;
//   scores  after pass A they are parked in shared memory, where (and in the layout in which) the probabilities will
//           stand;
//   output  O = P V has tensor-memory columns of its own and is read beside the reciprocals of the NEXT item's rows.
// The chunk loops are rolled: straight-line code for all chunks waited for instructions more than for anything else.
// Measured: 32 x 577 tokens, 16 heads of 64: 282 -> 178 us (before: one table, remainders dealt to all threads, a wait
// for P V in every item).  On rows of up to 256 tokens the two CTAs per SM of the kernel above win: 19.5 against 29.6 us
// at 64 x 197, 6 heads.
// Warps 0..3: warp 0 loads, issues MMAs and owns tensor memory (the others of its warpgroup only lend their registers);
// warps 4..19: the Shiftmax threads.  The launch gives every warp 96 registers (640 threads); the first warpgroup hands
// all but 64 of its own back, which lets the other four take 104: 128 x 64 + 512 x 104 = 640 x 96.
constexpr int kRowsThreads = 640;
constexpr int kRowsFirst = 4;       // first Shiftmax warp
constexpr int kBlkChunks = 12;      // 16-column chunks per score block

struct RowsArgs {
  AttnArgs a;
  int wb;                           // columns of a score buffer in tensor memory (buffers at 0 and wb, output at 2 wb)
  int nblk;                         // score blocks per row
  int vbox, nv;                     // rows of a value box and their number
  uint32_t p_stride;                // bytes between the two probability buffers of even / odd items (0: one buffer)
};

template <bool FAST, bool BIAS>
__global__ void __launch_bounds__(kRowsThreads, 1) attention_rows_kernel(const __grid_constant__ CUtensorMap tmQ,
                                                                        const __grid_constant__ CUtensorMap tmK,
                                                                        const __grid_constant__ CUtensorMap tmV, RowsArgs ra) {
  const AttnArgs& a = ra.a;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* gen = smem_raw + (base - smem_u32(smem_raw));
  // [Q 128 x d][K block x 2][V nv vbox x d][P 128 x 128B x kblocks, x 2][table 256 x cp][row partials][seeds][items][barriers]
  const uint32_t k_off = 128u * a.d, kbuf_bytes = (uint32_t)a.kbox * a.d;
  const uint32_t v_off = k_off + 2 * kbuf_bytes, v_bytes = (uint32_t)(ra.nv * ra.vbox) * a.d;
  const uint32_t p_off = (v_off + v_bytes + 1023u) & ~1023u;
  const uint32_t tab_off = p_off + ra.p_stride + (uint32_t)((a.kpad + 127) / 128) * 128 * 128;
  const uint32_t part_off = tab_off + 1024u * a.cp;      // [4 parts][128 rows] partial max, then partial sum, [128] reciprocals
  const uint32_t seed_off = part_off + 9 * 128 * 4;      // [128] seeds of the reciprocal
  const uint32_t item_off = seed_off + 128 * 4;          // [2] work item of even / odd iterations, written before its first scores
  const uint32_t bar_off = item_off + 2 * sizeof(AttnItem);
  AttnItem* const item_ring = reinterpret_cast<AttnItem*>(gen + item_off);
  // Q landed | V landed | K block landed (x2) | scores ready (x2) | score buffer read (x2) | probabilities written |
  // output ready
  const uint32_t bar_q = base + bar_off, bar_v = bar_q + 8, bar_k = bar_q + 16, bar_s = bar_q + 32, bar_f = bar_q + 48,
                 bar_p = bar_q + 64, bar_o = bar_q + 72;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gen + bar_off + 80);

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    prefetch_tmap(&tmQ);
    prefetch_tmap(&tmK);
    prefetch_tmap(&tmV);
    mbar_init(bar_q, 1);
    mbar_init(bar_v, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar_k + 8 * i, 1);
      mbar_init(bar_s + 8 * i, 2);   // the MMAs, and the control thread (the item is in the ring)
      mbar_init(bar_f + 8 * i, 16);
    }
    mbar_init(bar_p, 16);
    mbar_init(bar_o, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  if (warp == 0) tmem_alloc(smem_u32(tmem_slot), 512u);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
  const uint32_t o_col = 2u * (uint32_t)ra.wb;
  pdl_trigger();
  const int nblk = ra.nblk;
  const uint32_t n_items = AttnItem::count(a);

  if (warp < kRowsFirst) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
    if (warp == 0) pdl_wait();   // the QKV tensor comes from the previous kernel; the other warps build their table first
    if (warp == 0 && n_items > 0) {
      auto load_q = [&](const AttnItem& it) {
        mbar_expect_tx_w(bar_q, 128u * a.d);
        for (int g = 0; g < 4; ++g)
          load_box(base + (uint32_t)((g + it.rot) & 3) * 32u * a.d, &tmQ, bar_q, a.q_pos, it.m0 + 32 * g, it.h, it.b);
      };
      auto load_v = [&](const AttnItem& it) {
        mbar_expect_tx_w(bar_v, v_bytes);
        for (int i = 0; i < ra.nv; ++i)
          load_box(base + v_off + (uint32_t)(i * ra.vbox) * a.d, &tmV, bar_v, a.v_pos, i * ra.vbox, it.h, it.b);
      };
      // descriptor words: rows of d bytes (Q, K, V: swizzled over their width) or 128 bytes (P)
      const uint32_t layout = a.d == 128 ? 2u : (a.d == 64 ? 4u : 6u);
      const uint32_t row_hi = desc_hi(8u * a.d, layout), p_hi = desc_hi(1024, 2);
      const uint32_t q_lo0 = desc_lo(base, 16), k_lo0 = desc_lo(base + k_off, 16), p_lo0 = desc_lo(base + p_off, 16),
                     v_lo0 = desc_lo(base + v_off, 16), v_step = (uint32_t)(UK * a.d) >> 4;
      const uint32_t idesc2 = (2u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(a.d >> 3) << 17) | (8u << 24);
      const int ks = a.d / UK, ks2 = a.kpad / UK;

      uint32_t g = 0, gk = 0;    // score blocks issued / key blocks requested so far, over all items of this CTA
      bool ok = true;
      bool q_fly = false, v_fly = false, k_fly[2] = {false, false};   // loads requested and not yet waited for
      uint32_t q_par = 0, v_par = 0, k_par[2] = {0, 0};
      auto load_k = [&](const AttnItem& it, int j) {
        const uint32_t buf = gk & 1u, ph = (gk >> 1) & 1u;
        // the MMAs of the block two before this one have read the buffer
        if (gk >= 2) ok = mbar_wait_warp(bar_s + 8 * buf, ph ^ 1u, a.status);
        if (!ok) return;
        mbar_expect_tx_w(bar_k + 8 * buf, kbuf_bytes);
        load_box(base + k_off + buf * kbuf_bytes, &tmK, bar_k + 8 * buf, a.k_pos, j * (16 * kBlkChunks), it.h, it.b);
        k_fly[buf] = true;
        k_par[buf] = ph;
        ++gk;
      };
      // S_buf = Q K_j^T for key block j of the n-th item of this CTA
      auto issue_block = [&](const AttnItem& it, int j, uint32_t n) {
        const uint32_t buf = g & 1u, ph = (g >> 1) & 1u;
        ok = mbar_wait_warp(bar_k + 8 * buf, ph, a.status);
        k_fly[buf] = !ok;
        if (ok && j == 0) { ok = mbar_wait_warp(bar_q, n & 1u, a.status); q_fly = !ok; }
        // pass A of the block that used this score buffer two blocks ago has read it.  (With it every Shiftmax thread is
        // past item n - 2, whose place in the ring item n takes: nblk >= 2.)
        if (ok && g >= 2) ok = mbar_wait_warp(bar_f + 8 * buf, ph ^ 1u, a.status);
        if (!ok) return;
        if (j == 0 && lane == 0) item_ring[n & 1u] = it;
        tc_fence_after();
        const int w = j == nblk - 1 ? 16 * a.chunks - j * 16 * kBlkChunks : 16 * kBlkChunks;
        const uint32_t idesc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(w >> 3) << 17) | (8u << 24);
        const uint32_t k_lo = k_lo0 + buf * (kbuf_bytes >> 4), d_tmem = tmem + buf * (uint32_t)ra.wb;
        for (int k = 0; k < ks; ++k)
          umma_i8_lohi_w(d_tmem, q_lo0 + k * (UK >> 4), row_hi, k_lo + k * (UK >> 4), row_hi, idesc, k != 0);
        umma_commit_w(bar_s + 8 * buf);
        if (lane == 0) mbar_arrive(bar_s + 8 * buf);   // releases the item written to the ring
        __syncwarp();
        ++g;
      };

      AttnItem cur, next;
      cur.init(a, 0);
      load_q(cur); q_fly = true; q_par = 0;
      load_k(cur, 0);
      load_v(cur); v_fly = true; v_par = 0;
      issue_block(cur, 0, 0);
      if (ok) load_k(cur, 1);
      for (uint32_t n = 0; ok && n < n_items; ++n) {
        // block 0 of `cur` has been issued, its block 1 requested
        const bool more = n + 1 < n_items;
        if (more) next.init(a, n + 1);
        for (int j = 1; ok && j < nblk; ++j) {
          issue_block(cur, j, n);
          if (!ok) break;
          if (j + 1 < nblk) load_k(cur, j + 1);
          else if (more) load_k(next, 0);
        }
        if (!ok) break;
        if (more) {
          // Q may be overwritten once the score MMAs of the last block have read it
          ok = mbar_wait_warp(bar_s + 8 * ((g - 1) & 1u), ((g - 1) >> 1) & 1u, a.status);
          if (!ok) break;
          load_q(next); q_fly = true; q_par = (n + 1) & 1u;
          issue_block(next, 0, n + 1);
          if (ok) load_k(next, 1);
          if (!ok) break;
        }
        // O = P V once the probabilities are in shared memory (every warp has then read the previous output too)
        // and V has landed
        ok = mbar_wait_warp(bar_p, n & 1u, a.status);
        if (ok) { ok = mbar_wait_warp(bar_v, n & 1u, a.status); v_fly = !ok; }
        if (!ok) break;
        tc_fence_after();
        uint32_t p_lo = p_lo0 + (n & 1u) * (ra.p_stride >> 4), v_lo = v_lo0;
        int k = 0;
        for (; k + 4 <= ks2; k += 4, p_lo += (128 * 128) >> 4, v_lo += 4 * v_step)
          umma_i8_x4_w(tmem + o_col, p_lo, p_hi, v_lo, row_hi, idesc2, k != 0, UK >> 4, v_step);
        for (; k < ks2; ++k, p_lo += UK >> 4, v_lo += v_step)
          umma_i8_lohi_w(tmem + o_col, p_lo, p_hi, v_lo, row_hi, idesc2, k != 0);
        umma_commit_w(bar_o);
        // V may be overwritten once these MMAs have read it
        ok = mbar_wait_warp(bar_o, n & 1u, a.status);
        if (!ok) break;
        if (more) { load_v(next); v_fly = true; v_par = (n + 1) & 1u; }
        cur = next;
      }
      // end of work (or a wait that timed out): nothing may be in flight at exit
      if (q_fly) mbar_wait_warp(bar_q, q_par, a.status);
      if (v_fly) mbar_wait_warp(bar_v, v_par, a.status);
      for (int i = 0; i < 2; ++i)
        if (k_fly[i]) mbar_wait_warp(bar_k + 8 * i, k_par[i], a.status);
    }
  } else {
    // ---- Shiftmax / epilogue threads: TMEM lane quarter = warp % 4; the four warps of a quarter share its 32 rows
    //      (and their scheduler) ----
    asm volatile("setmaxnreg.inc.sync.aligned.u32 104;");
    const int st = threadIdx.x - 32 * kRowsFirst;   // 0..511
    const int qd = warp & 3;
    const int part = (warp - kRowsFirst) >> 2;    // 0..3
    const int trow = qd * 32 + lane;              // row inside the tile
    build_exp_table(a.smax.I0, a.smax.N, a.cp, gen + tab_off, st, 512);
    // probabilities of columns past the last chunk are never written again: zero (P V contracts over kpad columns)
    for (int c = a.chunks + part; c < a.kpad / 16; c += 4)
      for (int u = 0; u < 2; ++u)
        *reinterpret_cast<uint4*>(gen + p_off + u * ra.p_stride + (c >> 3) * (128 * 128) + trow * 128 + (((c & 7) ^ (trow & 7)) << 4)) = make_uint4(0u, 0u, 0u, 0u);
    unsigned* seeds = reinterpret_cast<unsigned*>(gen + seed_off);
    if (st < 128) seeds[st] = recip_seed(st);
    pdl_wait();
    PassConsts kc;
    kc.init(a);
    const uint32_t t_row = tmem + ((uint32_t)(qd * 32) << 16);
    int* part_max = reinterpret_cast<int*>(gen + part_off);
    unsigned* part_sum = reinterpret_cast<unsigned*>(gen + part_off + 4 * 128 * 4);
    const uint32_t tab_lane = base + tab_off + 4u * (unsigned)(lane & (a.cp - 1));
    const unsigned top = (unsigned)a.smax.I0 << a.smax.N;    // the largest exponential
    const int osh = 14 - a.smax.k_out, omax = (1 << (a.smax.k_out - 1)) - 1;
    // whole chunks c = part, part + 4, ... of this thread in the A-operand layout: k-block c >> 3, 16-byte piece c & 7;
    // the remainder of rem columns belongs to part 3, whose share of whole chunks is never the larger one
    const int c_full = a.T >> 4, rem = part == 3 ? a.T & 15 : 0;
    const uint32_t sw0 = (uint32_t)((part ^ (trow & 7)) << 4), sw1 = (uint32_t)(((part + 4) ^ (trow & 7)) << 4);
    uint8_t* p_row = gen + p_off + trow * 128;
    auto p_addr = [&](int c) { return reinterpret_cast<uint4*>(p_row + (c >> 3) * (128 * 128) + ((c & 4) ? sw1 : sw0)); };
    auto p_tail = [&]() { return reinterpret_cast<uint4*>(p_row + (c_full >> 3) * (128 * 128) + (((c_full & 7) ^ (trow & 7)) << 4)); };
    asm volatile("bar.sync 1, 512;" ::: "memory");   // the table is complete

    bool alive = true;   // false after a wait that timed out: no more waits, no more work, only the barriers
    uint32_t g = 0;      // score blocks seen so far (same count as the control thread's)
    int8_t* o_prev = nullptr;          // output row of the previous item (nullptr: none, or no row of the tile)
    bool o_prev_warp = false;          // the previous item had rows in this lane quarter
    // the output of the previous item, heads concatenated along the feature dimension
    auto store_output = [&](uint32_t n_prev) {
      alive = alive && mbar_wait(bar_o, n_prev & 1u, a.status);
      if (!alive || !o_prev_warp) return;
      tc_fence_after();
#pragma unroll 1
      for (int c = part; c < a.d / 16; c += 4) {
        int v[16];
        tmem_ld16(t_row + o_col + 16 * c, v);
        const uint4 w = output_piece<FAST>(a, v);
        if (o_prev) *reinterpret_cast<uint4*>(o_prev + 16 * c) = w;
      }
      tc_fence_before();
    };

    for (uint32_t n = 0; n < n_items; ++n) {
      alive = alive && mbar_wait(bar_s + 8 * (g & 1u), (g >> 1) & 1u, a.status);
      const AttnItem item = item_ring[n & 1u];
      const int m0 = item.m0 + ((qd - item.rot) & 3) * 32;   // first row (token) of this lane quarter
      const int r = m0 + lane;
      const bool row_ok = r < a.T;
      const bool warp_ok = m0 < a.T;                // quarters whose 32 rows all lie past T only keep the barriers
      const int32_t* brow = nullptr;
      if (BIAS) brow = a.bias + ((int64_t)((unsigned)(item.b * a.heads + item.h) % (unsigned)a.bias_batches) * a.T + (row_ok ? r : 0)) * a.T;
      auto add_bias = [&](auto& v, int col, int valid) {
        if constexpr (BIAS) {
#pragma unroll
          for (int i = 0; i < (int)(sizeof(v) / sizeof(int)); ++i)
            if (i < valid) v[i] += __ldg(brow + col + i);
        }
      };
      auto add_bias16 = [&](int (&v)[16], int col) {
        if constexpr (BIAS) { if (a.bias_vec) add_bias_row<true>(v, brow + col); else add_bias_row<false>(v, brow + col); }
      };
      p_row = gen + p_off + (n & 1u) * ra.p_stride + trow * 128;
      // with one probability buffer the parked scores overwrite what the previous item's P V reads
      if (ra.p_stride == 0 && n > 0) alive = alive && mbar_wait(bar_o, (n - 1) & 1u, a.status);

      // pass A, score block by score block, two chunks at a time
      int mx = -128;
      for (int j = 0; j < nblk; ++j, ++g) {
        if (j) alive = alive && mbar_wait(bar_s + 8 * (g & 1u), (g >> 1) & 1u, a.status);
        if (alive) tc_fence_after();
        if (alive && warp_ok) {
          const uint32_t t_buf = t_row + (g & 1u) * (uint32_t)ra.wb - (uint32_t)j * (16 * kBlkChunks);
          const int c_end = j == nblk - 1 ? c_full : (j + 1) * kBlkChunks;
#pragma unroll 1
          for (int c = j * kBlkChunks + part; c < c_end; c += 8) {
            int v[2][16];
            const bool second = c + 4 < c_end;
            tmem_ld16_issue(t_buf + 16 * c, v[0]);
            if (second) tmem_ld16_issue(t_buf + 16 * c + 64, v[1]);
            uint32_t x[4];
            tmem_ld_wait16(v[0]);
            add_bias16(v[0], 16 * c);
            score_piece<FAST, false>(a, kc, v[0], 16, mx, x);
            *p_addr(c) = make_uint4(x[0], x[1], x[2], x[3]);
            if (second) {
              tmem_ld_wait16(v[1]);
              add_bias16(v[1], 16 * c + 64);
              score_piece<FAST, false>(a, kc, v[1], 16, mx, x);
              *p_addr(c + 4) = make_uint4(x[0], x[1], x[2], x[3]);
            }
          }
          if (j == nblk - 1 && rem > 8) {
            int v[16];
            uint32_t x[4];
            tmem_ld16(t_buf + 16 * c_full, v);
            add_bias(v, 16 * c_full, rem);
            score_piece<FAST, true>(a, kc, v, rem, mx, x);
            *p_tail() = make_uint4(x[0], x[1], x[2], x[3]);
          } else if (j == nblk - 1 && rem) {
            int v[8];
            uint32_t x[2];
            tmem_ld8(t_buf + 16 * c_full, v);
            add_bias(v, 16 * c_full, rem);
            score_piece<FAST, true>(a, kc, v, rem, mx, x);
            *p_tail() = make_uint4(x[0], x[1], 0u, 0u);
          }
        }
        // the score buffer may take the block after the next one
        tc_fence_before();
        if (j == nblk - 1 && alive && warp_ok) part_max[part * 128 + trow] = max(-128, min(127, mx));
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_f + 8 * (g & 1u));
      }
      // only the four warps that share these 32 rows exchange partial results: a barrier of their own
      asm volatile("bar.sync %0, 128;" ::"r"(2 + qd) : "memory");
      const bool work = alive && warp_ok;
      uint32_t tmx = 0;
      if (work) {
        mx = max(max(part_max[trow], part_max[128 + trow]), max(part_max[256 + trow], part_max[384 + trow]));
        // pass B: entry (I_max - I) of this lane's table copy stands at tab_lane + 4 cp (I_max - I)
        tmx = tab_lane + (uint32_t)(4 * a.cp * mx);
        unsigned sum = 0;
#pragma unroll 2
        for (int c = part; c < c_full; c += 4) {
          const uint4 w = *p_addr(c);
          const uint32_t x[4] = {w.x, w.y, w.z, w.w};
          unsigned e[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) e[i] = exp_entry(x[i >> 2], kc.sel[i & 3], tmx);
#pragma unroll
          for (int i = 0; i < 16; i += 4) sum += (e[i] + e[i + 1]) + (e[i + 2] + e[i + 3]);
        }
        if (rem) {
          const uint4 w = *p_tail();
          const uint32_t x[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
          for (int i = 0; i < 16; ++i) sum += i < rem ? exp_entry(x[i >> 2], kc.sel[i & 3], tmx) : 0u;
        }
        part_sum[part * 128 + trow] = sum;
      }
      asm volatile("bar.sync %0, 128;" ::"r"(2 + qd) : "memory");
      // the output of the previous item; the reciprocal (Eq. (IntDiv) with M = 45), by every thread for its row
      if (n > 0) store_output(n - 1);
      if (work) {
        const unsigned sum = (part_sum[trow] + part_sum[128 + trow]) + (part_sum[256 + trow] + part_sum[384 + trow]);
        const unsigned factor = FAST ? prob_factor4(sum, top, seeds) : (unsigned)((1ull << 45) / (unsigned long long)(sum ? sum : 1u));
        auto words = [&](const uint4& w) {
          const uint32_t x[4] = {w.x, w.y, w.z, w.w};
          uint32_t o[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            int e[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) e[i] = (int)exp_entry(x[q], kc.sel[i], tmx);
            o[q] = FAST ? prob_word8(factor, e[0], e[1], e[2], e[3]) : prob_word(factor, e[0], e[1], e[2], e[3], osh, omax);
          }
          return make_uint4(o[0], o[1], o[2], o[3]);
        };
#pragma unroll 2
        for (int c = part; c < c_full; c += 4) *p_addr(c) = words(*p_addr(c));
        if (rem) {
          uint4 o = words(*p_tail());
          o.x &= edge_mask(rem, 0); o.y &= edge_mask(rem, 1); o.z &= edge_mask(rem, 2); o.w &= edge_mask(rem, 3);
          *p_tail() = o;
        }
        fence_async_smem();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_p);
      o_prev = row_ok ? a.O + ((int64_t)item.b * a.T + r) * a.D + (int64_t)item.h * a.d : nullptr;
      o_prev_warp = warp_ok;
    }
    if (n_items > 0) store_output(n_items - 1);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, 512u);
  }
}

}  // namespace

// The shared-memory limit of a kernel is a per-device attribute: set for the current device at context creation.
int attention_prepare_device() {
  const void* kernels[] = {(const void*)attention_short_kernel<1, false, false>, (const void*)attention_short_kernel<1, false, true>,
                           (const void*)attention_short_kernel<1, true, false>, (const void*)attention_short_kernel<1, true, true>,
                           (const void*)attention_short_kernel<2, false, false>, (const void*)attention_short_kernel<2, false, true>,
                           (const void*)attention_short_kernel<2, true, false>, (const void*)attention_short_kernel<2, true, true>,
                           (const void*)attention_short_kernel<4, false, false>, (const void*)attention_short_kernel<4, false, true>,
                           (const void*)attention_short_kernel<4, true, false>, (const void*)attention_short_kernel<4, true, true>,
                           (const void*)attention_rows_kernel<true, false>, (const void*)attention_rows_kernel<true, true>,
                           (const void*)attention_rows_kernel<false, false>, (const void*)attention_rows_kernel<false, true>};
  for (const void* k : kernels)
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess) return IVIT_ERR_CUDA;
  return IVIT_OK;
}

static CUtensorMapSwizzle swizzle_of(int64_t row_bytes) {
  return row_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : (row_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
}

static void fill_args(ivit_ctx* ctx, AttnArgs& a, const ivit_block_params* p, int8_t* O) {
  a.T = (int)p->T; a.heads = (int)p->heads; a.d = (int)(p->D / p->heads); a.D = p->D;
  a.bh = (int)(p->B * p->heads);
  a.items = (int)(p->B * p->heads * ((p->T + 127) / 128));
  a.chunks = (int)((p->T + 15) / 16);
  a.kpad = (int)((p->T + 31) / 32 * 32);
  a.qk_m = p->qk_scale.mult; a.qk_s = clamp_shift(p->qk_scale.shift);
  a.pv_m = p->pv_scale.mult; a.pv_s = clamp_shift(p->pv_scale.shift);
  a.smax = p->smax;
  a.bias = p->attn_bias;
  a.bias_vec = aligned16(p->attn_bias) ? 1 : 0;
  a.bias_batches = p->attn_bias ? (int)p->attn_bias_batches : 1;
  a.O = O;
  a.status = ctx->status_dev;
}
// As many copies of the ShiftExp table (up to 32) as `limit` bytes of shared memory leave room for beside `fixed`; false: none.
static bool fit_table(AttnArgs& a, size_t fixed, size_t limit) {
  a.cp = 32;
  while (a.cp > 1 && fixed + 1024 * a.cp > limit) a.cp >>= 1;
  for (int i = 0; i < 4; ++i) a.sel[i] = exp_sel(a.cp, i);
  return fixed + 1024 * a.cp <= limit;
}
// The arithmetic forms fixed at compile time: k_out = 8, both requantisation shifts >= 33, the largest exponential (and
// with it every row sum) above 2^15.
static bool fast_form(const AttnArgs& a) {
  return a.smax.k_out == 8 && a.qk_s >= 33 && a.pv_s >= 33 && ((int64_t)a.smax.I0 << a.smax.N) > (1 << 15);
}

// IVIT_ERR_UNSUPPORTED when the row does not fit the kernel's shared memory (the probabilities of a 128-row tile and
// the whole V of a head stay resident).
static int launch_attention_rows(ivit_ctx* ctx, const ivit_block_params* p, const int8_t* QKV, int8_t* O) {
  const int64_t B = p->B, T = p->T, D = p->D, h = p->heads, d = D / h;
  if (T > 1024) return IVIT_ERR_UNSUPPORTED;
  RowsArgs ra{};
  AttnArgs& a = ra.a;
  fill_args(ctx, a, p, O);
  // two score buffers and the output share the 512 columns of tensor memory
  ra.wb = 16 * kBlkChunks;
  ra.nblk = (a.chunks + kBlkChunks - 1) / kBlkChunks;
  a.kbox = 16 * kBlkChunks;
  ra.nv = (a.kpad + 255) / 256;
  ra.vbox = ((a.kpad + ra.nv - 1) / ra.nv + 7) / 8 * 8;
  const uint32_t v_off = 128u * a.d + 2u * a.kbox * a.d;
  const uint32_t p_off = (v_off + (uint32_t)(ra.nv * ra.vbox) * a.d + 1023u) & ~1023u;
  const size_t p_bytes = (size_t)((a.kpad + 127) / 128) * 128 * 128, limit = 227 * 1024;
  size_t fixed = 1024 + p_off + p_bytes + 9 * 128 * 4 + 128 * 4 + 2 * sizeof(AttnItem) + 80 + 16;
  if (fixed + p_bytes + 1024 * 32 <= limit) {   // a second probability buffer
    ra.p_stride = (uint32_t)p_bytes;
    fixed += p_bytes;
  }
  if (!fit_table(a, fixed, limit)) return IVIT_ERR_UNSUPPORTED;
  const size_t smem = fixed + 1024 * a.cp;
  const int64_t ldq = 3 * D;
  CUtensorMap tmQ, tmK, tmV;
  if (!make_tensor_map(ctx, &tmQ, QKV, d, T, h, B, ldq, d, T * ldq, (int)d, 32, swizzle_of(d), a.q_pos) ||
      !make_tensor_map(ctx, &tmK, QKV + D, d, T, h, B, ldq, d, T * ldq, (int)d, a.kbox, swizzle_of(d), a.k_pos) ||
      !make_tensor_map(ctx, &tmV, QKV + 2 * D, d, T, h, B, ldq, d, T * ldq, (int)d, ra.vbox, swizzle_of(d), a.v_pos))
    return IVIT_ERR_UNSUPPORTED;
  const dim3 grid((unsigned)(a.items < ctx->sm_count ? a.items : ctx->sm_count)), block(kRowsThreads);
  LaunchScope ls(ctx, KIND_ATTENTION, 4.0 * (double)(B * h) * (double)T * (double)T * (double)d);
  auto run = [&](auto kernel) { launch_k(kernel, grid, block, smem, ctx->stream, tmQ, tmK, tmV, ra); };
  if (fast_form(a)) {
    if (a.bias) run(attention_rows_kernel<true, true>);
    else run(attention_rows_kernel<true, false>);
  } else {
    if (a.bias) run(attention_rows_kernel<false, true>);
    else run(attention_rows_kernel<false, false>);
  }
  return ls.done();
}

static int launch_attention_short(ivit_ctx* ctx, const ivit_block_params* p, const int8_t* QKV, int8_t* O) {
  const int64_t B = p->B, T = p->T, D = p->D, h = p->heads, d = D / h;
  ShortArgs sa{};
  AttnArgs& a = sa.a;
  fill_args(ctx, a, p, O);
  sa.Btot = (int)B;
  // several windows: 2 of up to 64 tokens, or 4 of up to 32, share one 128-row tile
  const bool pack = T <= 64 && B >= 2;
  a.kbox = 16 * a.chunks;
  size_t bias_bytes = 0;
  sa.G = sa.npos = sa.units = 1;
  sa.R = 128;
  if (pack) {
    sa.G = T <= 32 ? 4 : 2;
    sa.R = a.kbox = 128 / sa.G;
    a.kpad = 128;
    sa.units = (int)((B + sa.G - 1) / sa.G);
    a.items = (int)(sa.units * h);
    // Windows repeat their bias every `per` of them: tiles of the same positions follow one another.  Where tiles and
    // positions do not line up the matrices are fetched for every tile (imgs = 1 in the kernel).
    const int64_t per = a.bias_batches % h == 0 ? a.bias_batches / h : 0;
    if (!a.bias || a.bias_batches == 1 || per == 1) sa.npos = 1;
    else if (per > 0 && per % sa.G == 0 && B % per == 0) sa.npos = (int)(per / sa.G);
    else sa.npos = sa.units;
    if (a.bias) bias_bytes = (size_t)sa.G * T * (T | 1) * 4;
    sa.t_magic = (unsigned)(0x100000000ull / (unsigned long long)T) + 1u;
  }
  sa.tmem_cols = pack || a.chunks <= 8 ? 128 : 256;
  const uint32_t p_off = (128u * a.d + (pack ? 128u : (uint32_t)a.kbox) * a.d + (uint32_t)a.kpad * a.d + 1023u) & ~1023u;
  // Threads per score row: four where an SM has at most one item anyway and the rows are long enough to share, which with a
  // score bias (read from global memory) they are earlier.  Two -> four threads, at most 148 items, alone: 16 tokens 1.08 x the time,
  // 80 tokens 1.03 ... 1.10, 144 tokens 1.00 ... 1.07, 170 tokens 0.93 ... 1.01, 256 tokens 0.91 ... 1.02, in a block of 170 or 197 tokens
  // 0.93 ... 1.02 (mean 0.99); with bias 16 tokens 1.08, 33 ... 80 tokens 0.97 ... 1.01 on up to 74 items and 1.01 ... 1.03 on 148,
  // 129 ... 197 tokens 0.75 ... 0.97.
  const int64_t long_rows = !a.bias ? 160 : (2 * a.items <= ctx->sm_count ? 32 : 128);
  const int tpr = pack ? 1 : (a.items <= ctx->sm_count && T > long_rows ? 4 : 2);
  const size_t partials = tpr == 4 ? ShortShape<4>::kPartials : ShortShape<2>::kPartials;
  const size_t fixed = 1024 + p_off + (size_t)((a.kpad + 127) / 128) * 128 * 128 + partials + 128 * 4 + 2 * sizeof(AttnItem) + 64 + bias_bytes;
  // CTAs per SM: as many as leave room for four copies of the table.  (Four threads per row: the CTA is alone on its SM and takes all
  // of its shared memory, at d = 128 for 32 copies instead of 4: 8 x 197 tokens, two heads 7.2 -> 6.4 us, a block of that 28.0 -> 27.2.)
  int per_sm = pack ? ShortShape<1>::kCtas : (tpr == 4 ? ShortShape<4>::kCtas : ShortShape<2>::kCtas);
  auto budget = [](int n) { return n == 1 ? (size_t)(227 * 1024) : (size_t)(228 * 1024 / n - 1024); };
  while (per_sm > 1 && fixed + 4 * 1024 > budget(per_sm)) --per_sm;
  if (!fit_table(a, fixed, budget(per_sm))) return IVIT_ERR_UNSUPPORTED;
  const size_t smem = fixed + 1024 * a.cp;
  const int64_t ldq = 3 * D;
  CUtensorMap tmQ, tmK, tmV;
  // boxes: R rows of G consecutive windows; or 32 query rows / all key and value rows of one image
  if (!make_tensor_map(ctx, &tmQ, QKV, d, T, h, B, ldq, d, T * ldq, (int)d, pack ? sa.R : 32, swizzle_of(d), a.q_pos, sa.G) ||
      !make_tensor_map(ctx, &tmK, QKV + D, d, T, h, B, ldq, d, T * ldq, (int)d, a.kbox, swizzle_of(d), a.k_pos, sa.G) ||
      !make_tensor_map(ctx, &tmV, QKV + 2 * D, d, T, h, B, ldq, d, T * ldq, (int)d, pack ? sa.R : a.kpad, swizzle_of(d), a.v_pos, sa.G))
    return IVIT_ERR_UNSUPPORTED;
  const int64_t slots = (int64_t)per_sm * ctx->sm_count;
  const dim3 grid((unsigned)(a.items < slots ? a.items : slots)), block((unsigned)(32 + 128 * tpr));
  LaunchScope ls(ctx, KIND_ATTENTION, 4.0 * (double)(B * h) * (double)T * (double)T * (double)d);
  auto run = [&](auto kernel) { launch_k(kernel, grid, block, smem, ctx->stream, tmQ, tmK, tmV, sa); };
#define IVIT_SHORT(TPR) \
  (fast_form(a) ? (a.bias ? run(attention_short_kernel<TPR, true, true>) : run(attention_short_kernel<TPR, true, false>)) \
                : (a.bias ? run(attention_short_kernel<TPR, false, true>) : run(attention_short_kernel<TPR, false, false>)))
  if (tpr == 1) IVIT_SHORT(1);
  else if (tpr == 2) IVIT_SHORT(2);
  else IVIT_SHORT(4);
#undef IVIT_SHORT
  return ls.done();
}

// Returns IVIT_ERR_UNSUPPORTED when the shape is outside the fused kernels (d not 32/64/128, rows too long for
// shared memory, misaligned tensors); the caller then composes the attention from MatMul and Shiftmax kernels.
int launch_attention_fused(ivit_ctx* ctx, const ivit_block_params* p, const int8_t* QKV, int8_t* O) {
  if (!ctx->tmap_encode) return IVIT_ERR_UNSUPPORTED;
  const int64_t B = p->B, T = p->T, h = p->heads, d = p->D / h;
  if ((d != 32 && d != 64 && d != 128) || B * h > 2147483647LL / 8 || p->attn_bias_batches > 2147483647LL) return IVIT_ERR_UNSUPPORTED;
  if ((reinterpret_cast<uintptr_t>(QKV) & 15) || (reinterpret_cast<uintptr_t>(O) & 15)) return IVIT_ERR_UNSUPPORTED;
  if (B == 0) return IVIT_OK;
  return T <= 256 ? launch_attention_short(ctx, p, QKV, O) : launch_attention_rows(ctx, p, QKV, O);
}

}  // namespace ivit
