// Dense layers with few tiles (INT8 x INT8 -> INT32, dyadic requantisation of Sec. 3.2, tcgen05), optionally preceded by
// the row operator that produces their input: I-LayerNorm (Sec. 3.5) or ShiftGELU (Algorithm 2).
//
// With at most one CTA per SM a Dense layer is a chain of latencies (launch, first loads, MMAs, epilogue), and so is a
// row operator in a kernel of its own.  Here a CTA owns BN rows of the input and up to four tiles of 128 output channels:
//   warp 0      requests the weight k-blocks (TMA ring), the first ones before the wait for the previous kernel, and,
//               without a row operator, the CTA's input rows;
//   warp 1      issues the MMAs, every channel tile into tensor-memory columns of its own;
//   workers     with a row operator: compute it on the CTA's rows (rowops.cuh), straight into the swizzled shared-memory
//               operand; then the epilogue: a lane owns one channel, 4x4 byte transposes, direct 4-byte stores.
// The row operator is computed again by every CTA that shares the rows (channel groups), which costs less than a launch
// as long as the whole layer is one wave.  The split is chosen in launch_gemm_small.
#include "tc_ptx.cuh"
#include "rowops.cuh"

namespace ivit {
namespace {

constexpr int SM_BM = 128;          // channels of a tile (TMEM lanes)
constexpr int SM_BK = 128;          // bytes of K per stage
constexpr int kSmallTiles = 4;      // channel tiles per CTA at most
constexpr int kSmallStages = 8;
constexpr int NW = 16;              // worker warps (eight are as fast up to 64 rows and up to 1.4 times slower above)

struct SmallArgs {
  GemmEpilogue epi;
  int P, Q, K;                      // output channels, rows, contraction
  int BN;                           // rows of a CTA (multiple of 32, at most 128)
  int tpc;                          // channel tiles of a CTA (the last group may have fewer)
  int groups;                       // channel groups
  int stages;
  int tmem_cols;
  int p_pos[3], q_pos[3];
  const int8_t* A;                  // input rows (row operators read them directly)
  int64_t lda;
  RowOpArgs rop;                    // gs, beta, M_ln, mean_magic, vec (LayerNorm); table (ShiftGELU)
  int* status;
};

// PRO: 0 = input rows as they are, 1 = I-LayerNorm, 2 = ShiftGELU.
template <int PRO>
__global__ void __launch_bounds__(64 + 32 * NW, 1) gemm_small_kernel(const __grid_constant__ CUtensorMap tmP,
                                                                     const __grid_constant__ CUtensorMap tmQ, SmallArgs a) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* gen = smem_raw + (base - smem_u32(smem_raw));
  // [weight stages][input rows: k-blocks of BN x 128 bytes][barriers][LayerNorm constants | table rows per warp]
  const int kblocks = (a.K + SM_BK - 1) / SM_BK;
  const uint32_t q_block = (uint32_t)a.BN * SM_BK;
  const uint32_t q_off = (uint32_t)a.stages * SM_BM * SM_BK;
  const uint32_t bar_off = q_off + kblocks * q_block;
  const uint32_t full0 = base + bar_off, empty0 = full0 + 8 * kSmallStages, accf0 = empty0 + 8 * kSmallStages,
                 qready = accf0 + 8 * kSmallTiles;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gen + bar_off + 16 * kSmallStages + 8 * kSmallTiles + 8);
  uint8_t* scratch = gen + bar_off + 256;

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int q0 = (int)(blockIdx.x / (unsigned)a.groups) * a.BN;
  const int tile0 = (int)(blockIdx.x % (unsigned)a.groups) * a.tpc;            // first channel tile
  const int tiles = min(a.tpc, (a.P + SM_BM - 1) / SM_BM - tile0);
  const int nrows = min(a.BN, a.Q - q0);

  if (threadIdx.x < kSmallStages) mbar_init(full0 + 8 * threadIdx.x, 1);
  else if (threadIdx.x < 2 * kSmallStages) mbar_init(empty0 + 8 * (threadIdx.x - kSmallStages), 1);
  else if (threadIdx.x < 2 * kSmallStages + kSmallTiles) mbar_init(accf0 + 8 * (threadIdx.x - 2 * kSmallStages), 1);
  else if (threadIdx.x == 2 * kSmallStages + kSmallTiles) mbar_init(qready, NW);
  else if (threadIdx.x == 30) prefetch_tmap(&tmP);
  else if (threadIdx.x == 31 && PRO == 0) prefetch_tmap(&tmQ);
  if (threadIdx.x < 32) {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  if (warp == 1) tmem_alloc(smem_u32(tmem_slot), (uint32_t)a.tmem_cols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
  pdl_trigger();

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    const int total = tiles * kblocks;      // weight k-blocks, tile by tile
    const int pre = min(total, a.stages);
    int tile = 0, kb = 0;
    auto request = [&](int s) {
      const int p0 = (tile0 + tile) * SM_BM;
      // without a row operator the first tile's stages also bring the input rows' k-blocks (below)
      mbar_expect_tx_w(full0 + 8 * s, SM_BM * SM_BK + (PRO == 0 && tile == 0 ? q_block : 0));
      tma_load_4d_w(base + s * (SM_BM * SM_BK), &tmP, full0 + 8 * s, kb * SM_BK, a.p_pos[0] == 1 ? p0 : 0,
                    a.p_pos[0] == 2 ? p0 : 0, a.p_pos[0] == 3 ? p0 : 0);
      if (++kb == kblocks) { kb = 0; ++tile; }
    };
    auto request_q = [&](int s, int k) {
      tma_load_4d_w(base + q_off + k * q_block, &tmQ, full0 + 8 * s, k * SM_BK, a.q_pos[0] == 1 ? q0 : 0,
                    a.q_pos[0] == 2 ? q0 : 0, a.q_pos[0] == 3 ? q0 : 0);
    };
    for (int s = 0; s < pre; ++s) request(s);   // weights are parameters: before the wait for the previous kernel
    pdl_wait();
    if (PRO == 0)
      for (int s = 0; s < min(pre, kblocks); ++s) request_q(s, s);
    int s = 0;
    uint32_t par = 0;
    for (int i = pre; i < total; ++i) {
      if (!mbar_wait_warp(empty0 + 8 * s, par, a.status)) break;
      const int k = kb;
      const bool first = tile == 0;
      request(s);
      if (PRO == 0 && first) request_q(s, k);
      if (++s == a.stages) { s = 0; par ^= 1u; }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    const uint32_t idesc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(a.BN >> 3) << 17) | ((uint32_t)(SM_BM >> 4) << 24);
    const uint32_t hi = desc_hi(1024, 2), p_lo0 = desc_lo(base, 16), q_lo0 = desc_lo(base + q_off, 16);
    const int tail_steps = (a.K - (kblocks - 1) * SM_BK + 31) / 32;
    bool ok = PRO == 0 || mbar_wait_warp(qready, 0, a.status);
    int s = 0;
    uint32_t par = 0;
    for (int t = 0; ok && t < tiles; ++t) {
      const uint32_t d = tmem + (uint32_t)(t * a.BN);
      for (int kb = 0; ok && kb < kblocks; ++kb) {
        ok = mbar_wait_warp(full0 + 8 * s, par, a.status);
        tc_fence_after();
        uint32_t p_lo = p_lo0 + s * ((SM_BM * SM_BK) >> 4), q_lo = q_lo0 + kb * (q_block >> 4);
        if (kb != kblocks - 1 || tail_steps == 4) {
          umma_i8_x4_w(d, p_lo, hi, q_lo, hi, idesc, kb != 0, 2, 2);
        } else {
          for (int k = 0; k < tail_steps; ++k, p_lo += 2, q_lo += 2) umma_i8_lohi_w(d, p_lo, hi, q_lo, hi, idesc, (kb | k) != 0);
        }
        umma_commit_w(empty0 + 8 * s);
        if (++s == a.stages) { s = 0; par ^= 1u; }
      }
      umma_commit_w(accf0 + 8 * t);
    }
    if (!ok) {
      // after a timeout: nothing that was requested may be in flight at exit (waits that run out end the drain)
      for (int i = 0; i < a.stages; ++i) mbar_wait_warp(full0 + 8 * i, 0, a.status);
    }
  } else {
    // ---------------- workers ----------------
    const int ew = warp - 2, et = (int)threadIdx.x - 64;
    const GemmEpilogue& e = a.epi;
    // constants of this thread's channel (parameters: before the wait)
    const int qd = warp & 3;            // TMEM lane quarter
    int nm = 1, ns = 33, nb = 0;
    auto fetch_channel = [&](int t) {
      const int c = (tile0 + t) * SM_BM + qd * 32 + lane;
      nm = 1; ns = 33; nb = 0;
      if (c < a.P) {
        nm = e.scale.m(c);
        ns = e.scale.s(c);
        if (e.bias) nb = __ldg(e.bias + c);
      }
    };
    fetch_channel(0);
    if (PRO == 1) {
      const int nwords = a.K >> 2;
      int4* sm_m = reinterpret_cast<int4*>(scratch);
      // the form (fast / general, see LnConsts) is agreed on by all workers
      int fast = ln_stage_consts(a.rop.gs, a.rop.beta, nwords, a.rop.vec, sm_m, sm_m + nwords, sm_m + 2 * nwords, et, 32 * NW) ? 1 : 0;
      asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %0, 0;\n\tbarrier.cta.red.and.pred q, 1, %1, p;\n\tselp.s32 %0, 1, 0, q;\n\t}"
                   : "+r"(fast) : "n"(32 * NW) : "memory");
      if (fast) ln_fold_consts(nwords, sm_m + nwords, sm_m + 2 * nwords, et, 32 * NW);
      asm volatile("bar.sync 1, %0;" ::"n"(32 * NW) : "memory");
      const LnConsts lk{sm_m, sm_m + nwords, sm_m + 2 * nwords, fast != 0};
      pdl_wait();
      // word idx (channels 4 idx ..) of row r in the K-major 128-byte-swizzled operand
      auto run = [&](auto wpl, auto rr) {
        constexpr int R = decltype(rr)::value;
        for (int r0 = ew * R; r0 < nrows; r0 += NW * R)
          layernorm_rows_to<decltype(wpl)::value, R, false>(a.A + (int64_t)(q0 + r0) * a.lda, a.lda, min(R, nrows - r0), a.K,
                                                            a.rop.M_ln, a.rop.mean_magic, lk, lane, [&](int r, int idx, unsigned w) {
            const int row = r0 + r;
            *reinterpret_cast<unsigned*>(gen + q_off + (idx >> 5) * q_block + row * 128 + ((((idx >> 2) & 7) ^ (row & 7)) << 4) + (idx & 3) * 4) = w;
          });
      };
      // (rows per warp and pass: all sixteen warps have work from 32 rows on)
      if (a.K <= 256) run(Int<2>{}, Int<2>{});
      else if (a.K <= 384) run(Int<3>{}, Int<2>{});
      else if (a.K <= 512) run(Int<4>{}, Int<2>{});
      else run(Int<8>{}, Int<2>{});
    } else if (PRO == 2) {
      pdl_wait();
      auto run = [&](auto wpl, auto rr) {
        constexpr int R = decltype(rr)::value;
        unsigned* tab = reinterpret_cast<unsigned*>(scratch) + ew * (R * 64);
        for (int r0 = ew * R; r0 < nrows; r0 += NW * R)
          shiftgelu_rows_to<decltype(wpl)::value, R, false>(a.A + (int64_t)(q0 + r0) * a.lda, a.lda, min(R, nrows - r0), a.K,
                                                            a.rop.table, tab, lane, -1, [&](int r, int idx, int4 v) {
            const int row = r0 + r;
            *reinterpret_cast<int4*>(gen + q_off + (idx >> 3) * q_block + row * 128 + (((idx & 7) ^ (row & 7)) << 4)) = v;
          });
      };
      if (a.K <= 1536) run(Int<3>{}, Int<2>{});
      else run(Int<8>{}, Int<1>{});
    } else {
      pdl_wait();
    }
    if (PRO != 0) {
      fence_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(qready);
    }

    // ---- epilogue: chunks of 32 rows x this warp's 32 channels, dealt to the NW / 4 parts across the CTA's tiles ----
    constexpr int kParts = NW / 4;
    const int part = ew >> 2;
    const int nck = (nrows + 31) >> 5;
    const int li = lane & 3;
    const uint32_t sel1 = (li & 1) ? 0x3715u : 0x6240u, sel2 = (li & 2) ? 0x3276u : 0x5410u;
    // 4 x 4 byte transpose inside every group of four lanes (its own inverse)
    auto transpose4 = [&](uint32_t (&w)[4]) {
      uint32_t o[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) o[k] = __shfl_xor_sync(0xffffffffu, w[k], 1);
#pragma unroll
      for (int k = 0; k < 4; ++k) w[k] = __byte_perm(w[k], o[k], sel1);
#pragma unroll
      for (int k = 0; k < 4; ++k) o[k] = __shfl_xor_sync(0xffffffffu, w[k], 2);
#pragma unroll
      for (int k = 0; k < 4; ++k) w[k] = __byte_perm(w[k], o[k], sel2);
    };
    // rq(x; m, s) of an int8 x whose byte stands on top of a word: high word of (x 2^24) m + 2^(s+23), shifted by s - 8.
    // From s = 39 on |x m| < 2^(s-1): the result is 0.
    const int rs = clamp_shift(e.res_scale.shift);
    const int res_m = rs >= 39 ? 0 : e.res_scale.mult, res_sh = rs >= 39 ? 31 : rs - 8, res_rnd = rs >= 39 ? 0 : 1 << (rs - 9);
    const int8_t* res = e.res;
    int last_t = 0;
    bool ok = true;
    for (int g = part; g < tiles * nck; g += kParts) {
      const int t = g / nck, ck = g - t * nck;
      if (t != last_t) {
        fetch_channel(t);
        last_t = t;
      }
      const int c = (tile0 + t) * SM_BM + qd * 32 + lane, cbase = c & ~3;
      const bool cg_ok = cbase < a.P;               // P % 4 == 0: a group of four channels is valid as a whole
      const int r0 = q0 + 32 * ck;
      // residual words of the chunk, in flight while the MMAs finish: row li + 4 k of each half, four channels
      uint32_t rw[2][4];
      if (res) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int row = r0 + 16 * h + 4 * k + li;
            rw[h][k] = 0;
            if (cg_ok && row < a.Q) {
              const int64_t rr = row < e.res_rows ? row : (int64_t)((uint64_t)row % (uint64_t)e.res_rows);
              rw[h][k] = *reinterpret_cast<const uint32_t*>(res + rr * e.ldres + cbase);
            }
          }
      }
      const int m = nm, s = ns;
      const bool hi_only = __all_sync(0xffffffffu, s >= 33 && nb > -(1 << 30) && nb < (1 << 30));
      if (ok) ok = mbar_wait_warp(accf0 + 8 * t, 0, a.status);
      tc_fence_after();
      int vv[32];
      tmem_ld32(tmem + ((uint32_t)(qd * 32) << 16) + (uint32_t)(t * a.BN + 32 * ck), vv);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        int (&v)[16] = *reinterpret_cast<int (*)[16]>(&vv[16 * h]);
        if (hi_only) {
          const int rnd = 1 << (s - 33), sh = s - 32;
#pragma unroll
          for (int j = 0; j < 16; ++j) v[j] = mad_hi(v[j] + nb, m, rnd) >> sh;
        } else {
          const long long c64 = (long long)nb * m + (1ll << (s - 1));
#pragma unroll
          for (int j = 0; j < 16; ++j) v[j] = (int)(mad_wide(v[j], m, c64) >> s);
        }
        if (res) {
          transpose4(rw[h]);
#pragma unroll
          for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int b = 0; b < 4; ++b)
              v[4 * k + b] += mad_hi((int)__byte_perm(rw[h][k], 0, (b << 12) | 0x444), res_m, res_rnd) >> res_sh;
        }
        if (e.out_dtype == IVIT_I32) {
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if (c < a.P && r0 + 16 * h + j < a.Q) reinterpret_cast<int32_t*>(e.out)[(int64_t)(r0 + 16 * h + j) * e.ldo + c] = v[j];
          continue;
        }
        if (e.act_table) {   // element-wise activation of the saturated value (the static-maximum ShiftGELU variant)
#pragma unroll
          for (int j = 0; j < 16; ++j) v[j] = (int)e.act_table[sat8(v[j]) + 128];
        }
        uint32_t w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) w[k] = pack_sat8(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
        transpose4(w);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int row = r0 + 16 * h + 4 * k + li;
          int64_t ro = row;
          if (e.group_rows > 0) ro = (int64_t)((unsigned)row / (unsigned)e.group_rows) * e.group_stride + (unsigned)row % (unsigned)e.group_rows;
          if (cg_ok && row < a.Q) *reinterpret_cast<uint32_t*>(reinterpret_cast<int8_t*>(e.out) + ro * e.ldo + cbase) = w[k];
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, (uint32_t)a.tmem_cols);
  }
}

constexpr size_t kSmallSmem = 227 * 1024;

}  // namespace

int gemm_small_prepare_device() {
  const void* kernels[] = {(const void*)gemm_small_kernel<0>, (const void*)gemm_small_kernel<1>, (const void*)gemm_small_kernel<2>};
  for (const void* k : kernels)
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallSmem) != cudaSuccess) return IVIT_ERR_CUDA;
  return IVIT_OK;
}

int launch_gemm_small(ivit_ctx* ctx, const GemmProblem& g, int pro) {
  const GemmEpilogue& e = g.epi;
  if (!ctx->tmap_encode || !g.transB || g.batches_outer * g.batches_inner != 1 || e.bias32) return IVIT_ERR_UNSUPPORTED;
  if (g.M < 1 || g.M > 1 << 20 || g.N > 1 << 20 || g.N % 4 || g.lda % 16 || g.ldb % 16) return IVIT_ERR_UNSUPPORTED;
  if (e.out_dtype == IVIT_I32 ? e.group_rows > 0 : (e.ldo % 4 != 0 || (reinterpret_cast<uintptr_t>(e.out) & 3) != 0)) return IVIT_ERR_UNSUPPORTED;
  if (e.res && ((reinterpret_cast<uintptr_t>(e.res) & 3) || e.ldres % 4)) return IVIT_ERR_UNSUPPORTED;
  if (pro == 1 && (g.K > 1024 || g.K % 4)) return IVIT_ERR_UNSUPPORTED;
  if (pro == 2 && (g.K > 4096 || g.K % 16)) return IVIT_ERR_UNSUPPORTED;
  const int kblocks = (int)((g.K + SM_BK - 1) / SM_BK), tiles_p = (int)((g.N + SM_BM - 1) / SM_BM);
  const size_t scratch = pro == 1 ? (size_t)g.K * 12 : (pro == 2 ? (size_t)NW * 2 * 256 : 0);
  const size_t fixed = 1024 + 256 + scratch;
  // Rows and channel tiles per CTA, one wave of CTAs.  Without a row operator only one tile per CTA pays (with two the
  // persistent kernel is as fast: 1576 x 1536 x 384 5.4 against 4.7 us), and the fewer rows the better (197 x 384 x 384:
  // 3.6 us at 32 rows, 4.2 at 128, 5.2 in the persistent kernel).  With one: fewest rounds of epilogue chunks first, then
  // the fewest rows, which every CTA of the rows works through the operator.
  SmallArgs a{};
  int best = 0;
  for (int tpc = 1; tpc <= (pro ? kSmallTiles : 1); ++tpc) {
    const int groups = (tiles_p + tpc - 1) / tpc;
    for (int bn = 32; bn <= 128; bn += 32) {
      if (fixed + (size_t)kblocks * bn * SM_BK + 2 * SM_BM * SM_BK > kSmallSmem) break;
      if ((int64_t)groups * ((g.M + bn - 1) / bn) > ctx->sm_count) continue;
      const int cost = (tpc * bn + 127) / 128 * 40 + bn;
      if (best && cost >= best) continue;
      best = cost;
      a.BN = bn;
      a.tpc = tpc;
      a.groups = groups;
    }
  }
  if (!best) return IVIT_ERR_UNSUPPORTED;
  a.stages = (int)((kSmallSmem - fixed - (size_t)kblocks * a.BN * SM_BK) / (SM_BM * SM_BK));
  if (a.stages > kSmallStages) a.stages = kSmallStages;
  if (a.stages > a.tpc * kblocks) a.stages = a.tpc * kblocks;
  a.epi = e;
  a.P = (int)g.N; a.Q = (int)g.M; a.K = (int)g.K;
  a.A = g.A; a.lda = g.lda;
  a.rop = e.rop;
  a.rop.mean_magic = (unsigned)(0x100000000ull / (unsigned long long)(2 * g.K)) + 1u;
  a.rop.vec = e.rop.gs.mult_c && e.rop.gs.shift_c && !(reinterpret_cast<uintptr_t>(e.rop.gs.mult_c) & 15) &&
              !(reinterpret_cast<uintptr_t>(e.rop.gs.shift_c) & 3) && !(reinterpret_cast<uintptr_t>(e.rop.beta) & 15);
  a.status = ctx->status_dev;
  a.tmem_cols = 32;
  while (a.tmem_cols < a.tpc * a.BN) a.tmem_cols <<= 1;
  CUtensorMap tmP, tmQ;
  if (!make_tensor_map(ctx, &tmP, g.B, g.K, g.N, 1, 1, g.ldb, 0, 0, SM_BK, SM_BM, CU_TENSOR_MAP_SWIZZLE_128B, a.p_pos)) return IVIT_ERR_UNSUPPORTED;
  tmQ = tmP;
  if (pro == 0 && !make_tensor_map(ctx, &tmQ, g.A, g.K, g.M, 1, 1, g.lda, 0, 0, SM_BK, a.BN, CU_TENSOR_MAP_SWIZZLE_128B, a.q_pos))
    return IVIT_ERR_UNSUPPORTED;
  const size_t smem = fixed + (size_t)kblocks * a.BN * SM_BK + (size_t)a.stages * SM_BM * SM_BK;
  const dim3 grid((unsigned)(a.groups * ((g.M + a.BN - 1) / a.BN))), block(64 + 32 * NW);
  LaunchScope ls(ctx, KIND_GEMM_TC, 2.0 * (double)g.M * (double)g.N * (double)g.K);
  if (pro == 0) launch_k(gemm_small_kernel<0>, grid, block, smem, ctx->stream, tmP, tmQ, a);
  else if (pro == 1) launch_k(gemm_small_kernel<1>, grid, block, smem, ctx->stream, tmP, tmQ, a);
  else launch_k(gemm_small_kernel<2>, grid, block, smem, ctx->stream, tmP, tmQ, a);
  return ls.done();
}

}  // namespace ivit
