// Dense layers with few tiles (INT8 x INT8 -> INT32, dyadic requantisation of Sec. 3.2, tcgen05): one wave of CTAs, one
// tile of 128 output channels x 32 ... 128 rows each.
//
// Such a layer is a chain of latencies: launch, first loads, MMAs, epilogue.  Against the persistent kernel (gemm_tc.cu) the
// tiles are narrower, so that more SMs share the work and the MMAs and the epilogue of a tile are shorter; there is no
// tile loop; the output leaves with direct stores instead of staged TMA stores.
//   warp 0      requests the weight k-blocks (TMA ring), the first ones of a model's layer before the wait for the previous
//               kernel, and the input rows, which stay resident;
//   warp 1      issues the MMAs;
//   warps 2..17 epilogue: a lane owns one channel and takes 8 rows at a time; 4x4 byte transposes, direct 4-byte stores.  The
//               residual words are requested before the MMAs are awaited.
// Measured, back to back (persistent kernel -> this one): 197 x 192 x 192 with residual 4.8 -> 3.3 us, 197 x 384 x 1536
// 7.6 -> 4.6, 197 x 768 x 3072 10.7 -> 6.2, 1576 x 384 x 1536 5.6 -> 5.0.  LayerNorm and ShiftGELU computed here, in front
// of the MMAs, instead of in kernels of their own were slower on every batch size (four DeiT-T blocks of one image 154
// against 130 us): the row kernels' launches overlap their neighbours', the prologue does not.  Behind the
// MMAs, by a cluster of the CTAs of a row (totals by reductions into distributed shared memory), they were no faster either:
// DeiT-T block of one image 25.3 against 24.7 us, ViT-B 33.9 against 31.2.
#include "ring.cuh"
#include "tc_ptx.cuh"

namespace ivit {
namespace {

constexpr int SM_BM = 128;          // channels of a tile (TMEM lanes)
constexpr int SM_BK = 128;          // bytes of K per stage
constexpr int kSmallStages = 8;
constexpr int NW = 16;              // epilogue warps
constexpr int kMaxPieces = 4;       // 8-row pieces of a warp

struct SmallArgs {
  GemmEpilogue epi;
  int P, Q, K;                      // output channels, rows, contraction
  int BN;                           // rows of a CTA (multiple of 32, at most 128)
  int tiles_p;                      // channel tiles
  int stages;
  int tmem_cols;
  int p_pos[3], q_pos[3];
  int b_is_param;                   // see GemmProblem
  int* status;
};

__global__ void __launch_bounds__(64 + 32 * NW, 1) gemm_small_kernel(const __grid_constant__ CUtensorMap tmP,
                                                                     const __grid_constant__ CUtensorMap tmQ, SmallArgs a) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* gen = smem_raw + (base - smem_u32(smem_raw));
  // [weight stages][input rows: k-blocks of BN x 128 bytes][barriers]
  const int kblocks = (a.K + SM_BK - 1) / SM_BK;
  const uint32_t q_block = (uint32_t)a.BN * SM_BK;
  const uint32_t q_off = (uint32_t)a.stages * SM_BM * SM_BK;
  const uint32_t bar_off = q_off + kblocks * q_block;
  const uint32_t full0 = base + bar_off, empty0 = full0 + 8 * kSmallStages, accf = empty0 + 8 * kSmallStages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gen + bar_off + 16 * kSmallStages + 8);

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int q0 = (int)(blockIdx.x / (unsigned)a.tiles_p) * a.BN;
  const int p0 = (int)(blockIdx.x % (unsigned)a.tiles_p) * SM_BM;
  const int nrows = min(a.BN, a.Q - q0);

  if (threadIdx.x < kSmallStages) mbar_init(full0 + 8 * threadIdx.x, 1);
  else if (threadIdx.x < 2 * kSmallStages) mbar_init(empty0 + 8 * (threadIdx.x - kSmallStages), 1);
  else if (threadIdx.x == 2 * kSmallStages) mbar_init(accf, 1);
  else if (threadIdx.x == 30) prefetch_tmap(&tmP);
  else if (threadIdx.x == 31) prefetch_tmap(&tmQ);
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
    const int pre = min(kblocks, a.stages);
    auto request = [&](int s, int kb) {
      mbar_expect_tx_w(full0 + 8 * s, SM_BM * SM_BK + q_block);
      tma_load_4d_w(base + s * (SM_BM * SM_BK), &tmP, full0 + 8 * s, kb * SM_BK, a.p_pos[0] == 1 ? p0 : 0,
                    a.p_pos[0] == 2 ? p0 : 0, a.p_pos[0] == 3 ? p0 : 0);
    };
    auto request_q = [&](int s, int kb) {
      tma_load_4d_w(base + q_off + kb * q_block, &tmQ, full0 + 8 * s, kb * SM_BK, a.q_pos[0] == 1 ? q0 : 0,
                    a.q_pos[0] == 2 ? q0 : 0, a.q_pos[0] == 3 ? q0 : 0);
    };
    if (!a.b_is_param) pdl_wait();
    for (int kb = 0; kb < pre; ++kb) request(kb, kb);   // weights of a model: before the wait for the previous kernel
    pdl_wait();
    for (int kb = 0; kb < pre; ++kb) request_q(kb, kb);
    int s = 0, requested = pre;
    uint32_t par = 0;
    for (; requested < kblocks; ++requested) {
      if (!mbar_wait_warp(empty0 + 8 * s, par, a.status)) break;
      request(s, requested);
      request_q(s, requested);
      if (++s == a.stages) { s = 0; par ^= 1u; }
    }
    // nothing that was requested may be in flight at exit, also when the MMA warp gave up before it was through
    drain_ring(requested, a.stages, [&](int stage, uint32_t parity) { mbar_wait_warp(full0 + 8 * stage, parity, a.status); });
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    pdl_wait();   // the previous kernel's time does not count against the limit of the polls below
    const uint32_t idesc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(a.BN >> 3) << 17) | ((uint32_t)(SM_BM >> 4) << 24);
    const uint32_t hi = desc_hi(1024, 2), p_lo0 = desc_lo(base, 16), q_lo0 = desc_lo(base + q_off, 16);
    const int tail_steps = (a.K - (kblocks - 1) * SM_BK + 31) / 32;
    bool ok = true;
    int s = 0;
    uint32_t par = 0;
    for (int kb = 0; ok && kb < kblocks; ++kb) {
      ok = mbar_wait_warp(full0 + 8 * s, par, a.status);
      tc_fence_after();
      uint32_t p_lo = p_lo0 + s * ((SM_BM * SM_BK) >> 4), q_lo = q_lo0 + kb * (q_block >> 4);
      if (kb != kblocks - 1 || tail_steps == 4) {
        umma_i8_x4_w(tmem, p_lo, hi, q_lo, hi, idesc, kb != 0, 2, 2);
      } else {
        for (int k = 0; k < tail_steps; ++k, p_lo += 2, q_lo += 2) umma_i8_lohi_w(tmem, p_lo, hi, q_lo, hi, idesc, (kb | k) != 0);
      }
      umma_commit_w(empty0 + 8 * s);
      if (++s == a.stages) { s = 0; par ^= 1u; }
    }
    umma_commit_w(accf);
  } else {
    // ---------------- epilogue ----------------
    const GemmEpilogue& e = a.epi;
    // constants of this thread's channel (parameters of a model: before the wait)
    if (!a.b_is_param) pdl_wait();
    const int qd = warp & 3;            // TMEM lane quarter
    const int c = p0 + qd * 32 + lane, cbase = c & ~3;
    const bool cg_ok = cbase < a.P;     // P % 4 == 0: a group of four channels is valid as a whole
    int m = 1, s = 33, nb = 0;
    if (c < a.P) {
      m = e.scale.m(c);
      s = e.scale.s(c);
      if (e.bias) nb = __ldg(e.bias + c);
    }
    const bool hi_only = __all_sync(0xffffffffu, s >= 33 && nb > -(1 << 30) && nb < (1 << 30));
    pdl_wait();

    // Pieces of 8 rows x this warp's 32 channels, in a loop.  The code of a launch this short runs cold, so its length counts: a
    // piece is what the shortest tile gives each of the sixteen warps, and longer tiles run the same instructions again
    // (with 32 rows to a warp, unrolled, this part took 2500 to 4400 clocks of a launch of 6000; per block of one image DeiT-T
    // 28.1 -> 24.9 us, DeiT-S 30.0 -> 26.0, ViT-L 40.7 -> 37.2, DeiT-S of eight images 39.3 -> 37.7, of 27 50.1 -> 49.4).
    const int npieces = (nrows + 7) >> 3, part = (warp - 2) >> 2;
    static_assert(NW / 4 * 8 * kMaxPieces >= 128, "all rows");
    const int li = lane & 3;
    const uint32_t sel1 = (li & 1) ? 0x3715u : 0x6240u, sel2 = (li & 2) ? 0x3276u : 0x5410u;
    // 4 x 4 byte transpose inside every group of four lanes (its own inverse)
    auto transpose4 = [&](uint32_t w) {
      w = __byte_perm(w, __shfl_xor_sync(0xffffffffu, w, 1), sel1);
      return __byte_perm(w, __shfl_xor_sync(0xffffffffu, w, 2), sel2);
    };
    // rq(x; m, s) of an int8 x whose byte stands on top of a word: high word of (x 2^24) m + 2^(s+23), shifted by s - 8.
    // From s = 39 on |x m| < 2^(s-1): the result is 0.
    const int rs = clamp_shift(e.res_scale.shift);
    const int res_m = rs >= 39 ? 0 : e.res_scale.mult, res_sh = rs >= 39 ? 31 : rs - 8, res_rnd = rs >= 39 ? 0 : 1 << (rs - 9);
    const int8_t* res = e.res;
    // residual words of this warp's pieces, in flight while the MMAs finish: row li + 4 k of each, four channels
    uint32_t rw[kMaxPieces][2];
    if (res) {
#pragma unroll
      for (int i = 0; i < kMaxPieces; ++i)
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const int row = q0 + 8 * (part + NW / 4 * i) + 4 * k + li;
          rw[i][k] = 0;
          if (part + NW / 4 * i < npieces && cg_ok && row < a.Q) {
            const int64_t rr = row < e.res_rows ? row : (int64_t)((uint64_t)row % (uint64_t)e.res_rows);
            rw[i][k] = *reinterpret_cast<const uint32_t*>(res + rr * e.ldres + cbase);
          }
        }
    }
    mbar_wait_warp(accf, 0, a.status);   // (after a timeout the results are meaningless and the status word says so)
    tc_fence_after();
    const uint32_t t_row = tmem + ((uint32_t)(qd * 32) << 16);
#pragma unroll 1
    for (int piece = part; piece < npieces; piece += NW / 4) {
      const int r0 = q0 + 8 * piece;
      int v[8];
      tmem_ld8(t_row + (uint32_t)(8 * piece), v);
      if (hi_only) {
        const int rnd = 1 << (s - 33), sh = s - 32;
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = mad_hi(v[j] + nb, m, rnd) >> sh;
      } else {
        const long long c64 = (long long)nb * m + (1ll << (s - 1));
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = (int)(mad_wide(v[j], m, c64) >> s);
      }
      if (res) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const uint32_t w = transpose4(rw[0][k]);
#pragma unroll
          for (int b = 0; b < 4; ++b) v[4 * k + b] += mad_hi((int)__byte_perm(w, 0, (b << 12) | 0x444), res_m, res_rnd) >> res_sh;
#pragma unroll
          for (int i = 1; i < kMaxPieces; ++i) rw[i - 1][k] = rw[i][k];
        }
      }
      if (e.out_dtype == IVIT_I32) {
        int32_t* o = reinterpret_cast<int32_t*>(e.out) + (int64_t)r0 * e.ldo + c;
#pragma unroll
        for (int j = 0; j < 8; ++j, o += e.ldo)
          if (c < a.P && r0 + j < a.Q) *o = v[j];
        continue;
      }
      if (e.act_table) {   // element-wise activation of the saturated value (the static-maximum ShiftGELU variant)
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = (int)e.act_table[sat8(v[j]) + 128];
      }
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const uint32_t w = transpose4(pack_sat8(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]));
        const int row = r0 + 4 * k + li;
        int64_t ro = row;
        if (e.group_rows > 0) ro = (int64_t)((unsigned)row / (unsigned)e.group_rows) * e.group_stride + (unsigned)row % (unsigned)e.group_rows;
        if (cg_ok && row < a.Q) *reinterpret_cast<uint32_t*>(reinterpret_cast<int8_t*>(e.out) + ro * e.ldo + cbase) = w;
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
constexpr size_t kSmallSmemAlone = 116 * 1024;   // more than half of an SM's

}  // namespace

int gemm_small_prepare_device() {
  return cudaFuncSetAttribute(gemm_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallSmem) == cudaSuccess ? IVIT_OK : IVIT_ERR_CUDA;
}

int launch_gemm_small(ivit_ctx* ctx, const GemmProblem& g) {
  const GemmEpilogue& e = g.epi;
  if (!ctx->tmap_encode || !g.transB || g.batches_outer * g.batches_inner != 1 || e.bias32) return IVIT_ERR_UNSUPPORTED;
  if (g.M < 1 || g.M > 1 << 20 || g.N > 1 << 20 || g.N % 4 || g.lda % 16 || g.ldb % 16) return IVIT_ERR_UNSUPPORTED;
  if (e.out_dtype == IVIT_I32 ? e.group_rows > 0 : (e.ldo % 4 != 0 || (reinterpret_cast<uintptr_t>(e.out) & 3) != 0)) return IVIT_ERR_UNSUPPORTED;
  if (e.res && ((reinterpret_cast<uintptr_t>(e.res) & 3) || e.ldres % 4)) return IVIT_ERR_UNSUPPORTED;
  const int kblocks = (int)((g.K + SM_BK - 1) / SM_BK), tiles_p = (int)((g.N + SM_BM - 1) / SM_BM);
  const size_t fixed = 1024 + 256;
  // The narrowest tile that makes one wave (197 x 384 x 384: 3.6 us at 32 rows, 4.2 at 128, 5.2 in the persistent kernel);
  // with more than a tile per CTA the persistent kernel is as fast or faster (1576 x 1536 x 384: 4.7 against 5.4 us).
  SmallArgs a{};
  for (int bn = 32; bn <= 128 && !a.BN; bn += 32) {
    if (fixed + (size_t)kblocks * bn * SM_BK + 2 * SM_BM * SM_BK > kSmallSmem) break;
    if ((int64_t)tiles_p * ((g.M + bn - 1) / bn) <= ctx->sm_count) a.BN = bn;
  }
  if (!a.BN) return IVIT_ERR_UNSUPPORTED;
  a.tiles_p = tiles_p;
  a.stages = (int)((kSmallSmem - fixed - (size_t)kblocks * a.BN * SM_BK) / (SM_BM * SM_BK));
  if (a.stages > kSmallStages) a.stages = kSmallStages;
  if (a.stages > kblocks) a.stages = kblocks;
  a.epi = e;
  if (e.group_rows > g.M) a.epi.group_rows = g.M;   // one group (the kernel divides 32-bit row numbers)
  a.P = (int)g.N; a.Q = (int)g.M; a.K = (int)g.K;
  a.b_is_param = g.b_is_param;
  a.status = ctx->status_dev;
  a.tmem_cols = 32;
  while (a.tmem_cols < a.BN) a.tmem_cols <<= 1;
  CUtensorMap tmP, tmQ;
  if (!make_tensor_map(ctx, &tmP, g.B, g.K, g.N, 1, 1, g.ldb, 0, 0, SM_BK, SM_BM, CU_TENSOR_MAP_SWIZZLE_128B, a.p_pos) ||
      !make_tensor_map(ctx, &tmQ, g.A, g.K, g.M, 1, 1, g.lda, 0, 0, SM_BK, a.BN, CU_TENSOR_MAP_SWIZZLE_128B, a.q_pos))
    return IVIT_ERR_UNSUPPORTED;
  const dim3 grid((unsigned)(a.tiles_p * ((g.M + a.BN - 1) / a.BN))), block(64 + 32 * NW);
  // A launch of more than half of the SMs takes one CTA per SM, by its shared memory.  Two would fit otherwise (56 registers), and
  // a launch that starts while the one before it still runs then puts two of its CTAs on the SMs that are free first and leaves
  // others idle (alone, two -> one: 1576 x 1152 x 384 5.4 -> 4.2 us, with residual 6.7 -> 5.0, 394 x 1536 x 384 with residual
  // 4.5 -> 3.5; 1024 x 1152 x 384, whose 144 tiles leave no SM idle, 3.3 -> 3.5; a block of eight DeiT-S images 34.3 -> 32.6).
  size_t smem = fixed + (size_t)kblocks * a.BN * SM_BK + (size_t)a.stages * SM_BM * SM_BK;
  if (2 * grid.x > (unsigned)ctx->sm_count && smem < kSmallSmemAlone) smem = kSmallSmemAlone;
  LaunchScope ls(ctx, KIND_GEMM_TC, 2.0 * (double)g.M * (double)g.N * (double)g.K);
  launch_k(gemm_small_kernel, grid, block, smem, ctx->stream, tmP, tmQ, a);
  return ls.done();
}

}  // namespace ivit
