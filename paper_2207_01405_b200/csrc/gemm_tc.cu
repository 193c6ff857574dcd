// INT8 x INT8 -> INT32 GEMM on the sm_100a tensor cores with the dyadic requantisation of
// Sec. 3.2 fused into the epilogue.  Persistent and warp-specialised:
//
//   warp 0      TMA producer: streams the k-blocks of both operands of successive output tiles
//               through a ring of shared-memory stages (cp.async.bulk.tensor, hardware swizzle,
//               mbarrier transaction counts);
//   warp 1      owns tensor memory; one thread issues tcgen05.mma.kind::i8 (M = 128, N = BN,
//               K = 32 per instruction) into one of two accumulator buffers;
//   warps 2..17 epilogue (four per TMEM lane quarter): read the finished accumulator with tcgen05.ld (one
//               TMEM lane per thread), requantise, add the residual, saturate and store - while the tensor
//               core already works on the next tile in the other buffer.
//
// The 128 TMEM lanes of a tile hold the "P" operand's rows, the columns the "Q" operand's rows.
//   * Dense layers (per-channel scale / bias):  P = weight rows (output channels), Q = activation
//     rows.  A thread then owns ONE output channel: its multiplier, shift and bias stay in registers
//     for the whole tile (no shared-memory traffic per value).  A warp turns its 32 channels x 32 rows
//     into row-major bytes with 4x4 byte transposes (shuffles), stages them in a shared-memory slot
//     of its own and stores the slot with a TMA store of its own; the residual bytes of the same
//     32 x 32 piece arrive by TMA two chunks ahead.  No warp waits for another.
//   * Batched MatMul (per-tensor scale): P = rows of A, Q = rows of B (K-major, Q K^T) or B is
//     MN-major ([K, N] rows, P V; the V tile is consumed as stored, without a transpose).  A thread
//     owns one output row and stores 32 consecutive int8 values per chunk.
//
// One CTA per SM walks a contiguous range of tiles (channel blocks fastest, so that consecutive tiles
// share their activation rows; for short K those rows stay resident in shared memory).  Every
// device-side wait is bounded: when one runs out the thread records IVIT_ERR_DEVICE_TIMEOUT in the
// context's status word, carries on without further waits, drains its outstanding copies, and the
// CTA frees its tensor memory and returns.
#include "tc_ptx.cuh"
#include <cstring>
#include <new>
#include "residual_rows.cuh"
#include "rowops.cuh"
#include "setup.cuh"

namespace ivit {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// 4-D int8 tensor map over {inner, rows, batch_inner, batch_outer}.  The three outer dimensions are
// ordered by ascending byte stride (a head inside a token row has a smaller stride than the row);
// pos[0..2] receive the tensor-map dimension that holds the row, inner-batch and outer-batch
// coordinate.  Byte strides must be multiples of 16.
namespace {
struct TmapKey {
  const void* ptr;
  uint64_t dims[4], strides[3];
  uint32_t box[4];
  int64_t swz;   // (64 bits: the key has no padding, it is compared bytewise)
};
struct TmapSlot {
  TmapKey key;
  CUtensorMap map;
  bool used;
};
constexpr int kTmapSlots = 512;
}  // namespace

bool make_tensor_map(ivit_ctx* ctx, CUtensorMap* map, const int8_t* ptr, int64_t inner, int64_t rows, int64_t bi, int64_t bo,
              int64_t row_stride, int64_t si, int64_t so, int box_inner, int box_rows, CUtensorMapSwizzle swz,
              int pos[3], int box_bo) {
  if ((reinterpret_cast<uintptr_t>(ptr) & 15) || row_stride % 16) return false;
  struct Dim { int64_t size, stride; int box, which; };
  Dim d[3] = {{rows, row_stride, box_rows, 0}, {bi, si, 1, 1}, {bo, so, box_bo, 2}};
  // size-1 dimensions never contribute to an address: give them the largest stride so they sort last
  int64_t big = row_stride;
  for (int i = 1; i < 3; ++i)
    if (d[i].size > 1 && d[i].stride > big) big = d[i].stride;
  for (int i = 1; i < 3; ++i)
    if (d[i].size <= 1) d[i].stride = big;
  for (int i = 0; i < 3; ++i)
    for (int j = i + 1; j < 3; ++j)
      if (d[j].stride < d[i].stride) { Dim t = d[i]; d[i] = d[j]; d[j] = t; }
  cuuint64_t dims[4] = {(cuuint64_t)inner, 0, 0, 0}, strides[3];
  cuuint32_t box[4] = {(cuuint32_t)box_inner, 1, 1, 1};
  for (int i = 0; i < 3; ++i) {
    if (d[i].stride % 16 || d[i].stride <= 0 || d[i].stride >= (1ll << 40)) return false;
    dims[i + 1] = (cuuint64_t)d[i].size;
    strides[i] = (cuuint64_t)d[i].stride;
    box[i + 1] = (cuuint32_t)d[i].box;
    pos[d[i].which] = i + 1;
  }
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  // An encoded map depends on nothing but these values: a forward pass asks for the same few dozen maps again and
  // again, so they are kept (direct-mapped, the newer entry wins a slot).
  TmapKey key{};
  key.ptr = ptr;
  for (int i = 0; i < 4; ++i) { key.dims[i] = dims[i]; key.box[i] = box[i]; }
  for (int i = 0; i < 3; ++i) key.strides[i] = strides[i];
  key.swz = (int64_t)swz;
  if (!ctx->tmap_cache) ctx->tmap_cache = new (std::nothrow) TmapSlot[kTmapSlots]();
  TmapSlot* slot = nullptr;
  if (ctx->tmap_cache) {
    uint64_t h = reinterpret_cast<uintptr_t>(ptr) * 0x9E3779B97F4A7C15ull;
    h ^= (dims[1] + 31 * dims[2] + 131 * box[1] + 1031 * box[0] + 7 * (uint64_t)swz + 17 * strides[0]) * 0xC2B2AE3D27D4EB4Full;
    slot = static_cast<TmapSlot*>(ctx->tmap_cache) + (h >> 40) % kTmapSlots;
    if (slot->used && std::memcmp(&slot->key, &key, sizeof(key)) == 0) {
      *map = slot->map;
      return true;
    }
  }
  EncodeTiledFn fn = reinterpret_cast<EncodeTiledFn>(ctx->tmap_encode);
  if (fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<int8_t*>(ptr), dims, strides, box, estr,
         CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return false;
  if (slot) {
    slot->key = key;
    slot->map = *map;
    slot->used = true;
  }
  return true;
}

void tmap_cache_free(ivit_ctx* ctx) {
  delete[] static_cast<TmapSlot*>(ctx->tmap_cache);
  ctx->tmap_cache = nullptr;
}

namespace {

constexpr int BM = 128;          // TMEM lanes of a tile (UMMA M, cta_group::1)
constexpr int BK = 128;          // bytes (= int8 elements) of K per pipeline stage
constexpr int UMMA_K = 32;       // K of one tcgen05.mma.kind::i8
constexpr int kMaxStages = 8;
constexpr int kEpiWarps = 16;
constexpr int kEpiThreads = 32 * kEpiWarps;
constexpr int kFirstEpiWarp = 2;   // warp 0: TMA loads, warp 1: MMA
constexpr int kThreads = 32 * kFirstEpiWarp + kEpiThreads;

struct TcArgs {
  GemmEpilogue epi;
  int P, Q, K;       // extents along TMEM lanes / TMEM columns / contraction (32-bit: the launcher checks the sizes)
  int res_rows, group_rows;   // of the epilogue, cut to 32 bits (there are fewer output rows than that)
  int64_t sCo, sCi;
  int batches_inner;
  int total_tiles;
  int tiles_each, tiles_extra;   // every CTA walks tiles_each tiles, the first tiles_extra CTAs one more ...
  int short_tiles;               // ... of all tiles (0), or of the full ones only: then the tiles of the ragged last row
                                 // block (this many) are dealt out after them, see TileRange
  int tiles_p, tiles_q;
  int BN;            // columns of the tile (multiple of 32, <= 256)
  int stages;
  int tmem_cols;     // power of two >= 2 * BN (two accumulator buffers)
  int lanes_are_channels;  // 1: Dense orientation (lane = output channel, column = output row)
  int q_mn;          // 1: the Q operand tile is MN-major ([k, n] rows of q_row_bytes)
  int q_row_bytes;
  int q_stage_bytes;
  int q_last_bytes;  // the same for a tile of the last block: a Dense layer fetches only the chunks of 32 rows that exist
                     // there (tmL: rows past the end, which a wider box fills with zeros, take as long to arrive as others)
  int p_pos[3], q_pos[3];  // tensor-map dimension (1..3) that holds the row / inner-batch / outer-batch coordinate
  int tma_out;       // Dense orientation, int8: the output tile is staged in shared memory and stored by TMA
  int tma_res;       // ... and the residual tile of the same shape is fetched by TMA into shared memory
  int pair;          // two CTAs (a cluster) per tile of 256 channels: cta_group::2 MMAs, each CTA loads its own 128
                     // weight rows and half of the activation rows; tiles_p then counts channel PAIRS of tiles
  int q_resident;    // Dense orientation, short K: all k-blocks of the Q (activation row) tile stay in shared
                     // memory while the CTA walks the channel blocks; only weight tiles stream through the ring
  int b_is_param;    // see GemmProblem
  RowOpArgs rop;     // row operator on finished blocks of output rows (Dense orientation, staged int8 output)
  int* status;
};


struct TileCoord {
  int batch;
  int bo, bi, p0, q0;
};

// The tiles of one worker (a CTA, or a pair of them).  Tiles are ordered p-block fastest and a worker owns a contiguous range of
// them, so that those it works on in a row share their Q operand (the activation rows of a Dense layer), and, when the tiles of a
// ragged last row block are dealt out by themselves, up to two of those.  They cost a fraction of a whole tile, so the workers that have one
// whole tile less take them first (one each, then a second one), then the others take one each.  Without that a ragged
// block can add a whole round: 12608 rows are 49 blocks of 256 and one of 64, and three channel tiles of 50 blocks on 148
// workers are 150 tiles, two rounds, instead of 147 tiles and three short ones, one round and a quarter.
// Measured: 12608 x 384 x 1536 10.9 -> 10.4 us, 4728 x 1024 x 1024 9.7 -> 8.6, 12608 x 768 x 3072 24.8 -> 23.5 (all on
// single CTAs).
// (DEAL: a kernel that can do so; the others keep the shorter walk, which is worth 2 % where a tile is one or two k-blocks.)
template <bool DEAL>
struct TileRange {
  int begin, end;         // tile numbers; the short tiles are counted behind the whole ones
  int jump, jump_p;       // after this many tiles the walk goes on at channel block jump_p of the last row block
  __device__ __forceinline__ TileRange(const TcArgs& a, int worker, int workers) {
    const int lng = worker < a.tiles_extra ? 1 : 0, whole = a.tiles_each + lng;
    begin = worker * a.tiles_each + min(worker, a.tiles_extra);
    int n_short = 0;
    jump_p = 0;
    if (DEAL && a.short_tiles) {
      const int n_brief = workers - a.tiles_extra;                // workers with one whole tile less
      const int to_brief = min(a.short_tiles, 2 * n_brief), two = max(to_brief - n_brief, 0);
      if (lng) {
        n_short = worker < a.short_tiles - to_brief ? 1 : 0;
        jump_p = to_brief + worker;
      } else {
        const int i = worker - a.tiles_extra;
        n_short = (i < to_brief ? 1 : 0) + (i < two ? 1 : 0);
        jump_p = i + min(i, two);
      }
      if (whole == 0) begin = a.tiles_p * (a.tiles_q - 1) + jump_p;
    }
    end = begin + whole + n_short;
    jump = whole > 0 && n_short > 0 ? whole : 0x7fffffff;
  }
};

// Walks the tiles of a range without divisions: p-block fastest, then q-block, then batch.
template <bool DEAL>
struct TileIter {
  int left, jump_p;       // tiles before the jump, see TileRange
  int p, q, bi, bo;       // block indices
  int batch;
  int pstep, poff;        // lanes between consecutive p-blocks (two tiles when a CTA pair shares them) and this CTA's offset
  __device__ __forceinline__ void init(const TcArgs& a, const TileRange<DEAL>& range, int poff_ = 0) {
    const uint32_t t = (uint32_t)range.begin, per_batch = (uint32_t)a.tiles_p * (uint32_t)a.tiles_q;
    batch = t < per_batch ? 0 : (int)(t / per_batch);     // a Dense layer is one batch
    const uint32_t t2 = t - (uint32_t)batch * per_batch;
    if (DEAL) { left = range.jump; jump_p = range.jump_p; }
    q = (int)(t2 / (uint32_t)a.tiles_p);
    p = (int)t2 - q * a.tiles_p;
    bo = batch == 0 ? 0 : batch / a.batches_inner;
    bi = batch - bo * a.batches_inner;
    pstep = a.pair ? 2 * BM : BM;
    poff = poff_;
  }
  __device__ __forceinline__ void next(const TcArgs& a) {
    if (DEAL && --left == 0) {
      p = jump_p;
      q = a.tiles_q - 1;
    } else if (++p == a.tiles_p) {
      p = 0;
      if (++q == a.tiles_q) {
        q = 0;
        ++batch;
        if (++bi == a.batches_inner) { bi = 0; ++bo; }
      }
    }
  }
  __device__ __forceinline__ int p0() const { return p * pstep + poff; }
  __device__ __forceinline__ int q0(const TcArgs& a) const { return q * a.BN; }
  __device__ __forceinline__ bool last(const TcArgs& a) const { return DEAL && q == a.tiles_q - 1; }
  // columns of the tile that the MMAs compute (DEAL: a ragged last tile is cut to whole chunks of 32)
  __device__ __forceinline__ int cols(const TcArgs& a) const { return DEAL ? min(a.BN, (a.Q - q * a.BN + 31) & ~31) : a.BN; }
};

// The map of the last block's activation rows: only the kernels that use it carry it in their parameters.
template <bool DEAL>
struct LastMap {
  CUtensorMap map;
  __device__ __forceinline__ const CUtensorMap* get(const CUtensorMap*) const { return &map; }
};
template <>
struct LastMap<false> {
  __device__ __forceinline__ const CUtensorMap* get(const CUtensorMap* other) const { return other; }
};

// The set-up barrier of a CTA.  (A barrier of its own: the warp that goes ahead may be through with its loads, and at the barrier
// at the end, before the others are here.)  PAIR: also the other CTA's barriers are initialised behind it.
template <bool PAIR>
struct DenseSetup {
  __device__ __forceinline__ void arrive() const { asm volatile("bar.arrive 3, %0;" ::"n"(kThreads) : "memory"); }
  __device__ __forceinline__ void sync() const {
    asm volatile("bar.sync 3, %0;" ::"n"(kThreads) : "memory");
    if (PAIR) cluster_sync_all();
  }
  __device__ __forceinline__ void trigger() const { pdl_trigger(); }
};

// MODE fixes the run-time choices of the epilogue at compile time for the shapes of an encoder block, so that
// the per-chunk code carries no branches on kernel arguments: 0 = everything decided at run time (any
// orientation, output type and residual port), 1 = Dense orientation, int8 output staged for TMA stores, no
// residual, 2 = the same with the residual tile fetched by TMA, 3 = as 1 with an activation table applied to the
// saturated value (the element-wise ShiftGELU variant inside FC1), 4 = as 2 for output rows in groups with a gap between
// them and a residual that repeats (the patch embedding with its class rows and position table): the slots are filled and
// emptied by the warp itself, residual words one chunk ahead.  (As MODE 0, with byte loads of the residual and 4-byte
// stores, the embedding took as long as two such layers: 25088 x 768 x 768 39.1 us, plain 18.0.)
// ROP != 0 (MODE 1 or 2 only): a row operator on the output, run by this same kernel: 1 = I-LayerNorm into a second
// tensor (the input of the next Dense layer), 2 = ShiftGELU in place (Algorithm 2 with its row maximum).  Both need
// whole output rows, i.e. every channel tile of a block of rows, and those tiles may belong to several CTAs.  So
// every epilogue warp, once its stores of a row block are complete, adds its tiles to the block's arrival counter;
// the warp that completes the count raises the block's ready flag.  The rows are cut into slices (one batch of the
// row routine each) that are dealt to all epilogue warps of the grid in a fixed order; a warp works on its slices
// after its CTA's last tile, straight out of L2, waiting (bounded) only for the ready flag of the slice's block.
// The last CTA to finish leaves counters and flags at zero for the next launch.
// DEAL: the tiles of a ragged last block of rows are dealt out by themselves (TileRange).
template <int MODE, int ROP, bool PAIR = false, bool DEAL = PAIR>
__global__ void __launch_bounds__(kThreads, 1) gemm_tc_kernel(const __grid_constant__ CUtensorMap tmP,
                                                              const __grid_constant__ CUtensorMap tmQ,
                                                              const __grid_constant__ CUtensorMap tmO,
                                                              const __grid_constant__ CUtensorMap tmR, TcArgs a,
                                                              const __grid_constant__ LastMap<DEAL> tmL) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  // carve: [stages x (P tile | Q tile)] [barriers] [tmem address, issued count]
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* gen_base = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t stage_bytes = BM * BK + (a.q_resident ? 0 : a.q_stage_bytes);
  const int kblocks = (a.K + BK - 1) / BK;
  const uint32_t qres_bytes = a.q_resident ? kblocks * a.q_stage_bytes : 0;
  const uint32_t qres = base + a.stages * stage_bytes;         // resident Q tile: kblocks x [BN rows x 128 B]
  const uint32_t stage_out = qres + qres_bytes;                // output slots: 2 x [32 rows][32 channels] int8 per epilogue warp
  const uint32_t stage_res = stage_out + (a.tma_out ? kEpiWarps * 2048 : 0);   // residual slots, same layout
  const uint32_t bars_off = a.stages * stage_bytes + qres_bytes + (a.tma_out ? kEpiWarps * 2048 : 0) + (a.tma_res ? kEpiWarps * 2048 : 0);
  const uint32_t full0 = base + bars_off, empty0 = full0 + 8 * kMaxStages;
  const uint32_t accf0 = empty0 + 8 * kMaxStages, acce0 = accf0 + 16, resf = acce0 + 16, qrese = resf + 16 * kEpiWarps;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gen_base + bars_off + 8 * (2 * kMaxStages + 5 + 2 * kEpiWarps));
  volatile int* issued_slot = reinterpret_cast<volatile int*>(tmem_slot + 1);
  // residual port: the requantised value of every int8 residual byte (256 entries, built below), followed by the
  // 256 entries of the optional activation table
  int8_t* res_tab = reinterpret_cast<int8_t*>(tmem_slot) + 32;
  volatile uint32_t* rop_flag = tmem_slot + 2;                                // row operator: a flag the CTA agrees on
  uint8_t* rop_smem = gen_base + bars_off + 1024;   // ROP == 1: LayerNorm constants; ROP == 2: table rows, per warp

  // (read from lane 0, so that the compiler knows it to be the same in all lanes)
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  // this CTA's (with PAIR: this CTA pair's) tiles
  const uint32_t rank = PAIR ? cluster_ctarank() : 0u;      // PAIR: 0 = the CTA that issues the MMAs of the pair
  const int poff = (int)rank * BM;                          // this CTA's 128 channels inside the pair's 256
  const int worker = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
  const int workers = PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x;
  const TileRange<DEAL> range(a, worker, workers);
  const int t_begin = range.begin, t_end = range.end;

  // Set-up.  The barriers of the load ring belong to warp 0, which then goes on to its first loads without waiting for the
  // others (it only arrives at the CTA's barrier; a CTA pair's two meet first).  The previous kernel has usually left
  // the SM by the time this CTA starts, and 1300 of the 2400 clocks of the set-up stood in front of the loads: DeiT-S forward of
  // 27 images 606 -> 586 us, of 64 945 -> 929, Swin-T of 64 1405 -> 1390.
  if (warp == 0) {
    if (lane < kMaxStages) mbar_init(full0 + 8 * lane, 1);
    else if (lane < 2 * kMaxStages) mbar_init(empty0 + 8 * (lane - kMaxStages), 1);
    else if (lane < 2 * kMaxStages + 2) mbar_init(accf0 + 8 * (lane - 2 * kMaxStages), 1);
    else if (lane < 2 * kMaxStages + 4) mbar_init(acce0 + 8 * (lane - 2 * kMaxStages - 2), PAIR ? 2 * kEpiWarps : kEpiWarps);   // PAIR: both CTAs' warps
    else if (lane == 2 * kMaxStages + 4) mbar_init(qrese, 1);
    static_assert(2 * kMaxStages + 5 <= 32, "a lane per barrier");
    if (lane == 0) *issued_slot = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
    __syncwarp();
  }
  {
    const int i = (int)threadIdx.x - 64;
    if (i >= 0 && i < 2 * kEpiWarps) {
      mbar_init(resf + 8 * i, 1);   // residual slots: 2 per epilogue warp
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      fence_async_smem();
    } else if (i == 32) {
      *rop_flag = 1u;
      if (a.tma_out) prefetch_tmap(&tmO);
    } else if (i == 64) {
      if (a.tma_res) prefetch_tmap(&tmR);
    }
    if (i >= 0 && i < 256 && a.epi.res) res_tab[i] = (int8_t)rq(i - 128, a.epi.res_scale.mult, clamp_shift(a.epi.res_scale.shift));
  }
  if (warp == 1) {
    if (PAIR) tmem_alloc_pair(smem_u32(tmem_slot), (uint32_t)a.tmem_cols);
    else tmem_alloc(smem_u32(tmem_slot), (uint32_t)a.tmem_cols);
  }
  tc_fence_before();
  // Barriers, tensor memory and tables are there for the warps behind this: they let the next kernel be scheduled, then wait
  // for the previous kernel's results before touching global memory.
  end_of_setup(DenseSetup<PAIR>{}, !PAIR && warp == 0);
  tc_fence_after();
  const uint32_t tmem_base = warp == 0 ? 0u : __shfl_sync(0xffffffffu, *tmem_slot, 0);   // (warp 0 has no use for it)
  if (ROP == 1 && warp >= kFirstEpiWarp) {
    // I-LayerNorm constants of all channels into shared memory: parameters, read before the wait for the previous
    // kernel.  The form (fast / general, see LnConsts) is agreed on by all epilogue threads.
    const int et0 = (int)threadIdx.x - 32 * kFirstEpiWarp, nwords = a.P >> 2;
    int4* sm_m = reinterpret_cast<int4*>(rop_smem);
    if (!ln_stage_consts(a.rop.gs, a.rop.beta, nwords, a.rop.vec, sm_m, sm_m + nwords, sm_m + 2 * nwords, et0, kEpiThreads))
      atomicAnd(const_cast<uint32_t*>(rop_flag), 0u);
    asm volatile("bar.sync 2, %0;" ::"n"(kEpiThreads) : "memory");
    if (*rop_flag) ln_fold_consts(nwords, sm_m + nwords, sm_m + 2 * nwords, et0, kEpiThreads);
    asm volatile("bar.sync 2, %0;" ::"n"(kEpiThreads) : "memory");
  }
  if (warp != 0) pdl_wait();

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    {
      int issued = 0;            // k-blocks issued so far, over all tiles of this CTA
      int s = 0, wrap = 0;       // ring slot of the next k-block and how often the ring has wrapped
      bool ok = true;
      int pit = 0, qi = 0, cur_q = -1;
      TileIter<DEAL> ti;
      ti.init(a, range, poff);
      // which tensor-map coordinate (1..3) carries the row / inner batch / outer batch index
      const int pr = a.p_pos[0], pbi = a.p_pos[1], qr = a.q_pos[0], qbi = a.q_pos[1];
      // PAIR: both CTAs load (their 128 weight rows, their half of the activation rows); the bytes of both are
      // counted by the stage barrier of CTA rank 0, which alone arms it
      auto arm = [&](uint32_t bar, uint32_t bytes) {
        if (!PAIR) mbar_expect_tx_w(bar, bytes);
        else if (rank == 0) mbar_expect_tx_w(bar, 2u * bytes);
      };
      auto load = [&](uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2, int c3) {
        if (PAIR) tma_load_4d_pair_w(dst, map, mapa_rank0(bar), c0, c1, c2, c3);
        else tma_load_4d_w(dst, map, bar, c0, c1, c2, c3);
      };
      // Dense layer of a model: the P operand is the weight matrix, which no kernel of the forward writes.  The weight
      // k-blocks of the first tile are requested before the wait for the previous kernel (whose last CTAs may still be
      // running elsewhere); the activation k-blocks that complete the same stage barriers follow after the wait.
      int pre = 0;
      if (a.b_is_param && a.lanes_are_channels && t_begin < t_end) {
        pre = kblocks < a.stages ? kblocks : a.stages;
        for (int kb = 0; kb < pre; ++kb) {
          arm(full0 + 8 * kb, BM * BK + (ti.last(a) ? a.q_last_bytes : a.q_stage_bytes));
          load(base + kb * stage_bytes, &tmP, full0 + 8 * kb, kb * BK, pr == 1 ? ti.p0() : 0, pr == 2 ? ti.p0() : 0,
               pr == 3 ? ti.p0() : 0);
        }
      }
      pdl_wait();
      for (int t = t_begin; ok && t < t_end; ++t, ++pit, ti.next(a)) {
        const int p0 = ti.p0(), q0 = ti.q0(a) + (PAIR ? (int)rank * (ti.cols(a) >> 1) : 0);   // PAIR: this CTA's half of the rows
        const int pc1 = pr == 1 ? p0 : (pbi == 1 ? ti.bi : ti.bo), pc2 = pr == 2 ? p0 : (pbi == 2 ? ti.bi : ti.bo),
                  pc3 = pr == 3 ? p0 : (pbi == 3 ? ti.bi : ti.bo);
        const CUtensorMap* const map_q = ti.last(a) ? tmL.get(&tmQ) : &tmQ;
        const uint32_t q_bytes = ti.last(a) ? a.q_last_bytes : a.q_stage_bytes;
        bool bring_q = false;
        if (a.q_resident && q0 != cur_q) {
          // new activation row block: its k-blocks come in beside this tile's weight k-blocks, once every MMA
          // on the old block is done
          if (qi > 0 && !mbar_wait_warp(qrese, (qi - 1) & 1, a.status)) { ok = false; break; }
          bring_q = true;
          cur_q = q0;
          ++qi;
        }
        for (int kb = 0; kb < kblocks; ++kb) {
          if (wrap > 0 && !mbar_wait_warp(empty0 + 8 * s, (wrap & 1) ^ 1, a.status)) { ok = false; break; }
          const uint32_t sp = base + s * stage_bytes, sq = sp + BM * BK;
          const bool early = t == t_begin && kb < pre;   // barrier armed and weights requested before the wait
          if (!early) arm(full0 + 8 * s, BM * BK + (bring_q || !a.q_resident ? q_bytes : 0));
          if (bring_q)
            load(qres + kb * a.q_stage_bytes, map_q, full0 + 8 * s, kb * BK, qr == 1 ? q0 : 0, qr == 2 ? q0 : 0,
                 qr == 3 ? q0 : 0);
          if (!early) load(sp, &tmP, full0 + 8 * s, kb * BK, pc1, pc2, pc3);
          if (!a.q_resident) {
            const int qrow = a.q_mn ? kb * BK : q0;     // MN-major: rows of the map are k, the inner index is n
            const int qc0 = a.q_mn ? q0 : kb * BK;
            load(sq, map_q, full0 + 8 * s, qc0, qr == 1 ? qrow : (qbi == 1 ? ti.bi : ti.bo),
                 qr == 2 ? qrow : (qbi == 2 ? ti.bi : ti.bo), qr == 3 ? qrow : (qbi == 3 ? ti.bi : ti.bo));
          }
          *issued_slot = ++issued;
          if (++s == a.stages) { s = 0; ++wrap; }
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    if (rank == 0) {   // PAIR: CTA rank 0 issues for both CTAs
      // instruction descriptor: D = S32, A = B = signed 8 bit, A K-major, M = 128 (PAIR: 256 over both CTAs), no
      // saturation; N = the tile's columns is added for each tile
      const uint32_t idesc0 = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a.q_mn << 16) |
                              ((uint32_t)((PAIR ? 2 * BM : BM) >> 4) << 24);
      // P descriptors: K-major rows of 128 bytes (128B swizzle, 1024 bytes per 8 rows).  Q: the same,
      // or MN-major rows of q_row_bytes (swizzle = row width, 8 rows per group).  Along K a descriptor
      // advances by 32 bytes (K-major) or 32 rows (MN-major): an add on the low word.
      const uint32_t p_hi = desc_hi(1024, 2);
      const uint32_t q_hi = !a.q_mn ? desc_hi(1024, 2)
                                    : desc_hi(8u * a.q_row_bytes, a.q_row_bytes == 128 ? 2u : (a.q_row_bytes == 64 ? 4u : 6u));
      const uint32_t q_kstep16 = (!a.q_mn ? UMMA_K : UMMA_K * a.q_row_bytes) >> 4;
      const int k_tail = (int)(a.K - (int64_t)(kblocks - 1) * BK);            // bytes of K in the last k-block
      const int tail_steps = k_tail >= BK ? BK / UMMA_K : (k_tail + UMMA_K - 1) / UMMA_K;
      // descriptor low words: the start-address field counts 16-byte units, so stages and k-blocks are plain adds
      const uint32_t p_lo0 = desc_lo(base, 16), q_lo0 = desc_lo(qres, 16);
      const uint32_t stage16 = stage_bytes >> 4, qstage16 = (uint32_t)a.q_stage_bytes >> 4;
      int consumed = 0, s = 0, wrap = 0, it = 0;
      bool ok = true;
      int cur_q = -1;
      TileIter<DEAL> ti;
      ti.init(a, range, poff);
      for (int t = t_begin; ok && t < t_end; ++t, ++it) {
        const int buf = it & 1;
        const uint32_t idesc = idesc0 | ((uint32_t)(ti.cols(a) >> 3) << 17);
        bool last_of_q = false;
        if (DEAL || a.q_resident) {
          // q_resident: a new activation row block arrives k-block by k-block on the stage barriers of this tile
          cur_q = ti.q0(a);
          ti.next(a);
          last_of_q = a.q_resident && (t + 1 >= t_end || ti.q0(a) != cur_q);
        }
        // the epilogue must have drained this buffer (its use two tiles ago)
        if (it >= 2 && !mbar_wait_warp(acce0 + 8 * buf, ((it >> 1) & 1) ^ 1, a.status)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(buf * a.BN);
        for (int kb = 0; kb < kblocks; ++kb) {
          if (!mbar_wait_warp(full0 + 8 * s, wrap & 1, a.status)) { ok = false; break; }
          tc_fence_after();
          // low descriptor words of this stage's P tile and of the Q tile (resident, or behind P in the stage)
          const uint32_t p_lo = p_lo0 + (uint32_t)s * stage16;
          const uint32_t q_lo = a.q_resident ? q_lo0 + (uint32_t)kb * qstage16 : p_lo + ((BM * BK) >> 4);
          if (kb != kblocks - 1 || tail_steps == BK / UMMA_K) {
            if (PAIR) umma_i8_x4_pair_w(d_tmem, p_lo, p_hi, q_lo, q_hi, idesc, kb != 0, UMMA_K >> 4, q_kstep16);
            else umma_i8_x4_w(d_tmem, p_lo, p_hi, q_lo, q_hi, idesc, kb != 0, UMMA_K >> 4, q_kstep16);
          } else {
            uint32_t pl = p_lo, ql = q_lo;
            for (int k = 0; k < tail_steps; ++k) {
              if (PAIR) umma_i8_pair_w(d_tmem, pl, p_hi, ql, q_hi, idesc, (kb | k) != 0);
              else umma_i8_lohi_w(d_tmem, pl, p_hi, ql, q_hi, idesc, (kb | k) != 0);
              pl += UMMA_K >> 4;
              ql += q_kstep16;
            }
          }
          // the stage may be refilled once these MMAs have read it (PAIR: in both CTAs)
          if (PAIR) umma_commit_pair_w(empty0 + 8 * s);
          else umma_commit_w(empty0 + 8 * s);
          ++consumed;
          if (++s == a.stages) { s = 0; ++wrap; }
        }
        if (ok) {   // accumulator of this tile complete (PAIR: told to the epilogue warps of both CTAs)
          if (PAIR) umma_commit_pair_w(accf0 + 8 * buf);
          else umma_commit_w(accf0 + 8 * buf);
        }
        if (ok && last_of_q) {   // the resident tile may be replaced once these MMAs are done (PAIR: in both CTAs)
          if (PAIR) umma_commit_pair_w(qrese);
          else umma_commit_w(qrese);
        }
      }
      if (!ok) {
        // drain: copies that were issued but never consumed (only after a timeout)
        const int issued = *issued_slot;
        for (int j = consumed; j < issued; ++j) {
          mbar_wait_warp(full0 + 8 * s, wrap & 1, a.status);
          if (++s == a.stages) { s = 0; ++wrap; }
        }
      }
    }
  } else {
    // ---------------- epilogue warps; TMEM lane quarter = warp % 4, 32-column chunks dealt round-robin ----------------
    // The groups of four warps ("parts") work independently.  A wait that times out is recorded and the
    // warp carries on without further waits (its results are then meaningless and the status word says so).
    const int et = threadIdx.x - 32 * kFirstEpiWarp;
    const int ew = warp - kFirstEpiWarp;
    const int qd = warp & 3;
    const int part = ew >> 2;
    constexpr int kParts = kEpiWarps / 4;
    static_assert((kParts & (kParts - 1)) == 0, "chunk rotation");
    const GemmEpilogue& e = a.epi;
    const bool dense = MODE ? true : a.lanes_are_channels != 0;
    const bool tma_out = MODE ? true : a.tma_out != 0;
    const bool tma_res = MODE ? MODE == 2 : a.tma_res != 0;   // MODE 3 = MODE 1 + activation table
    constexpr bool kGroup = MODE == 4;
    const bool smem_res = kGroup || tma_res;
    const bool ldg_res = MODE ? false : (e.res != nullptr && !a.tma_res);
    const bool out_i32 = MODE ? false : e.out_dtype == IVIT_I32;
    const int8_t* res_tab0 = res_tab + 128;   // entry of residual byte 0
    const int8_t* act_tab0 = res_tab + 256 + 128;   // entry of value 0 of the activation table
    const bool act = MODE == 3 ? true : (MODE ? false : e.act_table != nullptr);
    constexpr bool kFrag = MODE == 1 || MODE == 3;
    if (act) {
      // the table may come from an earlier kernel of the stream: read it after the dependency wait above
      if (et < 256) res_tab[256 + et] = e.act_table[et];
      asm volatile("bar.sync 1, %0;" ::"n"(kEpiThreads) : "memory");
    }
    bool ok = true;

    // Dense orientation: constants of this thread's channel; fetched one tile ahead
    int nm = 1, ns = 32, nb = 0;
    auto fetch_channel = [&](int p0) {
      const int c = p0 + qd * 32 + lane;
      nm = 1; ns = 32; nb = 0;
      if (c < a.P) {
        nm = e.scale.m(c);
        ns = e.scale.s(c);
        if (e.bias) nb = __ldg(e.bias + c);
      }
    };
    // the first tile's coordinates, computed once (they cost integer divisions)
    TileIter<DEAL> ti_first;
    ti_first.init(a, range, poff);
    if (dense && t_begin < t_end) fetch_channel(ti_first.p0());
    // MatMul orientation: one per-tensor constant set
    const int um = e.scale.mult, us = clamp_shift(e.scale.shift);
    const long long uc = 1ll << (us - 1);

    // Staged output (and residual input) of the Dense orientation: every warp owns two slots of
    // [32 rows][32 channels] bytes for each direction and needs no other warp to move them.  Its lane 0 stores a
    // filled output slot by TMA (a box of 32 channels x 32 rows) and fetches the residual bytes two chunks
    // ahead of the arithmetic into the slot whose bytes have just been used.
    const uint32_t my_out = stage_out + (uint32_t)ew * 2048u, my_res = stage_res + (uint32_t)ew * 2048u;
    const uint32_t my_resf = resf + 16u * (uint32_t)ew;
    const int c_first = qd * 32;        // first channel of this warp inside the tile
    uint32_t g = 0;                     // chunks this warp has worked on
    uint32_t rpar = 0, rpend = 0;       // per residual slot (bit 0 / 1): parity of its next arrival; a fetch in flight
    // Chunks are dealt to the parts round-robin ACROSS tiles (chunk j of a tile goes to part (rot + j) % kParts,
    // rot = chunks of this CTA's earlier tiles), so that a tile whose chunk count is no multiple of kParts
    // does not leave the same part idle every time.
    // The warp's chunk sequence two chunks ahead (residual fetches):
    TileIter<DEAL> pf_ti;
    int pf_t = t_begin;
    int pf_ck = part;
    int pf_rot = 0;
    uint32_t pf_g = 0;
    auto pf_settle = [&]() {
      while (pf_t < t_end) {
        const int left = a.Q - pf_ti.q0(a);
        const int nck = ((left < a.BN ? left : a.BN) + 31) >> 5;
        if (pf_ck < nck) break;
        pf_ti.next(a);
        ++pf_t;
        pf_rot = (pf_rot + nck) & (kParts - 1);
        pf_ck = (part - pf_rot) & (kParts - 1);
      }
    };
    // residual bytes of the next chunk of the look-ahead into slot pf_g & 1 (a box wholly past the last channel
    // is not fetched: the arithmetic does not wait for it either)
    auto pf_fetch = [&]() {
      if (pf_t < t_end) {
        if (pf_ti.p0() + c_first < a.P) {
          const uint32_t sl = pf_g & 1u;
          mbar_expect_tx_w(my_resf + 8u * sl, 1024u);
          tma_load_4d_w(my_res + 1024u * sl, &tmR, my_resf + 8u * sl, pf_ti.p0() + c_first, pf_ti.q0(a) + 32 * pf_ck, 0, 0);
          rpend |= 1u << sl;
        }
        ++pf_g;
        pf_ck += kParts;
        pf_settle();
      }
    };
    if (tma_res && t_begin < t_end) {
      pf_ti = ti_first;
      pf_settle();
      pf_fetch();
      pf_fetch();
    }
    // MODE 4: a lane's eight words of the next chunk's residual rows (lane >> 3) + 4 k, fetched one chunk ahead
    uint32_t rw[8];
    auto group_fetch = [&]() {
      if (pf_t >= t_end) return;
      const int c = pf_ti.p0() + c_first + 4 * (lane & 7);
      const int row0 = pf_ti.q0(a) + 32 * pf_ck, first = (int)((uint32_t)row0 % (uint32_t)a.res_rows);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int rr = residual_row(row0, first, (lane >> 3) + 4 * k, a.Q, a.res_rows);
        rw[k] = c < a.P && rr >= 0 ? __ldg(reinterpret_cast<const uint32_t*>(e.res + (int64_t)rr * e.ldres + c)) : 0u;
      }
      pf_ck += kParts;
      pf_settle();
    };
    if (kGroup && t_begin < t_end) {
      pf_ti = ti_first;
      pf_settle();
      group_fetch();
    }

    int it = 0;
    int rot = 0;          // chunks of this CTA's earlier tiles, modulo kParts
    int tiles_in_q = 0;   // ROP: tiles of the current block of output rows that this CTA has finished
    TileIter<DEAL> ti = ti_first;
    for (int t = t_begin; t < t_end; ++t, ++it) {
      TileCoord tc;
      tc.batch = ti.batch; tc.bo = ti.bo; tc.bi = ti.bi; tc.p0 = ti.p0(); tc.q0 = ti.q0(a);
      ti.next(a);   // ti now describes the next tile
      const int buf = it & 1;
      const int cm = nm, cs = ns;
      const long long cc = (long long)nb * nm + (1ll << (ns - 1));   // bias * m + 2^(s-1)
      const bool hi_ok = __all_sync(0xffffffffu, cs >= 32);    // the usual case: the shift is past the low word
      // ... and when the rounding constant is past it too and acc + bias cannot leave 32 bits (|acc| <= 2^30
      // since K <= 65536), only the high word of (acc + bias) * m is needed
      const int cbias = nb;
      const bool hi_only = __all_sync(0xffffffffu, cs >= 33 && nb > -(1 << 30) && nb < (1 << 30));
      const int rnd_hi = cs >= 33 ? 1 << (cs - 33) : 0;
      // The kernels without a residual port (MODE 1, 3) read the accumulators as fragments (tmem_ld_frag16): thread l
      // then works on the four channels (l >> 2) + 8 j of its warp, whose constants it takes from the lanes that
      // fetched them.  (With the residual port the fragment form is slower: its byte look-ups lose more to bank
      // conflicts than the transposes cost.)
      int km[4], ks[4], kb[4];
      if (kFrag) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int src = (lane >> 2) + 8 * j;
          km[j] = __shfl_sync(0xffffffffu, cm, src);
          ks[j] = __shfl_sync(0xffffffffu, cs, src);
          kb[j] = __shfl_sync(0xffffffffu, cbias, src);
        }
      }
      if (dense && t + 1 < t_end) fetch_channel(ti.p0());

      if (ok) ok = mbar_wait_warp(accf0 + 8 * buf, (it >> 1) & 1, a.status);
      tc_fence_after();
      const uint32_t t_row = tmem_base + ((uint32_t)(qd * 32) << 16) + (uint32_t)(buf * a.BN);
      const int cols_left = a.Q - tc.q0;
      const int nck = ((cols_left < a.BN ? cols_left : a.BN) + 31) >> 5;   // chunks that hold output

      if (dense) {
        // lane = output channel c, TMEM column = output row
        const int c = tc.p0 + qd * 32 + lane;
        const bool c_ok = c < a.P;
        const int sh_lo = min(cs, 32), sh_hi = max(cs - 32, 0);
        const int li = lane & 3;
        const uint32_t sel1 = (li & 1) ? 0x3715u : 0x6240u;
        const uint32_t sel2 = (li & 2) ? 0x3276u : 0x5410u;
        const int cb = qd * 32 + lane;          // channel within the tile

        // One chunk = 32 output rows x this warp's 32 channels, worked through in two halves of 16 rows to keep
        // the register footprint small: the SM holds four epilogue warps per scheduler, and it is their number
        // that hides the latencies of the shuffles, the shared-memory traffic and the barrier operations.
        auto half = [&](int (&v)[16], int ck, int h, uint8_t* pe) {
          const int j0 = ck * 32 + h * 16;
          const int r0 = tc.q0 + j0;
          const int nrow = min(16, a.Q - r0);
          if (hi_only) {
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = mad_hi(v[j] + cbias, cm, rnd_hi) >> sh_hi;
          } else if (hi_ok) {
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = mad_wide_hi(v[j], cm, cc) >> sh_hi;
          } else {
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const long long tt = mad_wide(v[j], cm, cc);
              v[j] = (int)__funnelshift_rc((unsigned)tt, (unsigned)(tt >> 32), sh_lo) >> sh_hi;
            }
          }
          // residual port
          if (smem_res) {
            // residual bytes of this chunk in shared memory: [row][32 channels]
            const uint8_t* rt = gen_base + (my_res - base) + (g & 1u) * 1024 + h * 512 + lane;
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] += (int)res_tab0[(int)*reinterpret_cast<const int8_t*>(rt + j * 32)];
          } else if (ldg_res) {
            int rr = (int)((uint32_t)r0 % (uint32_t)a.res_rows);   // (the same in all lanes)
            const int8_t* rp = e.res + (int64_t)rr * e.ldres + c;
#pragma unroll
            for (int g = 0; g < 16; g += 8) {
              int xr[8];
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                xr[j] = (c_ok && g + j < nrow) ? (int)__ldg(rp) : 0;
                rp += e.ldres;
                if (++rr == a.res_rows) { rr = 0; rp = e.res + c; }
              }
#pragma unroll
              for (int j = 0; j < 8; ++j) v[g + j] += (int)res_tab0[xr[j]];
            }
          }
          if (out_i32) {
#pragma unroll
            for (int j = 0; j < 16; ++j)
              if (j < nrow && c_ok) reinterpret_cast<int32_t*>(e.out)[(int64_t)(r0 + j) * e.ldo + c] = v[j];
            return;
          }
          if (act) {
            // element-wise activation of the saturated value (the static-maximum ShiftGELU variant)
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = (int)act_tab0[max(-128, min(127, v[j]))];
          }
          // int8: pack four rows per word, transpose 4x4 bytes inside each group of four lanes so that a lane
          // ends up with four consecutive channels of one row, then store 4 bytes per lane and word
          uint32_t w[4], o[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) w[k] = pack_sat8(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
#pragma unroll
          for (int k = 0; k < 4; ++k) o[k] = __shfl_xor_sync(0xffffffffu, w[k], 1);
#pragma unroll
          for (int k = 0; k < 4; ++k) w[k] = __byte_perm(w[k], o[k], sel1);
#pragma unroll
          for (int k = 0; k < 4; ++k) o[k] = __shfl_xor_sync(0xffffffffu, w[k], 2);
#pragma unroll
          for (int k = 0; k < 4; ++k) w[k] = __byte_perm(w[k], o[k], sel2);
          if (tma_out) {
            // word k belongs to slot row 16h + li + 4k: rows of 32 bytes, one bank per lane
#pragma unroll
            for (int k = 0; k < 4; ++k) *reinterpret_cast<uint32_t*>(pe + 512 * h + 128 * k) = w[k];
          } else {
            // direct stores (grouped output rows): this lane's first word is row r0 + li, then + 4 per word
            int64_t ro = (int64_t)r0 + li;
            int grem = 0;
            if (e.group_rows > 0) {
              const uint32_t g0 = (uint32_t)r0 / (uint32_t)a.group_rows;   // (the same in all lanes)
              grem = r0 - (int)g0 * a.group_rows + li;
              ro = (int64_t)g0 * e.group_stride + grem;
              while (grem >= a.group_rows) { grem -= a.group_rows; ro += e.group_stride - a.group_rows; }
            }
            const int cbase = tc.p0 + qd * 32 + (lane & ~3);
            const bool cg_ok = cbase < a.P;   // P % 4 == 0: a group of four channels is valid as a whole
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              if (cg_ok && 4 * k + li < nrow)
                *reinterpret_cast<uint32_t*>(reinterpret_cast<int8_t*>(e.out) + ro * e.ldo + cbase) = w[k];
              ro += 4;
              if (e.group_rows > 0) {
                grem += 4;
                while (grem >= a.group_rows) { grem -= a.group_rows; ro += e.group_stride - a.group_rows; }
              }
            }
          }
        };

        const bool c_any = tc.p0 + c_first < a.P;   // else the warp's box lies wholly past the last channel
        for (int ck = (part - rot) & (kParts - 1); ck < nck; ck += kParts) {
          uint8_t* pe = nullptr;
          if (tma_out) {
            const uint32_t sl = g & 1u;
            // the store that used this slot two chunks ago must have read it; the residual bytes must be here
            if (!kGroup) tma_store_wait_read1();   // (every lane: only the one that issued the stores has any to wait for)
            if (kGroup) {
              uint32_t* rs = reinterpret_cast<uint32_t*>(gen_base + (my_res - base) + sl * 1024) + lane;
#pragma unroll
              for (int k = 0; k < 8; ++k) rs[32 * k] = rw[k];
              group_fetch();
            }
            if (tma_res && c_any) {
              if (ok) ok = mbar_wait_warp(my_resf + 8u * sl, (rpar >> sl) & 1u, a.status);
              if (ok) { rpar ^= 1u << sl; rpend &= ~(1u << sl); }
            }
            __syncwarp();
            // after the transposes a lane holds 4 consecutive channels (lane >> 2) of slot row li + 4k
            pe = gen_base + (my_out - base) + sl * 1024 + li * 32 + (lane >> 2) * 4;
          }
          if constexpr (kFrag) {
            // fragment form: 16 channels x 32 rows per step; the packed words are the fragment that one stmatrix
            // stores transposed, i.e. as rows of 16 consecutive channels, into the [32 rows][32 channels] slot
            const uint32_t out_slot = my_out + 1024u * (g & 1u) + (uint32_t)lane * 32u;
            // both halves are requested before the arithmetic on the first begins
            int vv[32];
            tmem_ld_frag16_issue<0>(t_row + (uint32_t)(32 * ck), vv);
            tmem_ld_frag16_issue<16>(t_row + (16u << 16) + (uint32_t)(32 * ck), vv);
            tmem_ld_wait(vv);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              int (&v)[16] = *reinterpret_cast<int (*)[16]>(&vv[16 * h]);
#pragma unroll
              for (int u = 0; u < 2; ++u) {       // u = 0: channel (l >> 2) + 16 h, u = 1: eight channels on
                const int m = km[2 * h + u], sft = ks[2 * h + u], bia = kb[2 * h + u];
                if (hi_only) {
                  const int add = 1 << (sft - 33), sh = sft - 32;
#pragma unroll
                  for (int i = 0; i < 4; ++i) {
                    v[4 * i + 2 * u] = mad_hi(v[4 * i + 2 * u] + bia, m, add) >> sh;
                    v[4 * i + 2 * u + 1] = mad_hi(v[4 * i + 2 * u + 1] + bia, m, add) >> sh;
                  }
                } else {
                  const long long c64 = (long long)bia * m + (1ll << (sft - 1));
#pragma unroll
                  for (int i = 0; i < 4; ++i) {
                    v[4 * i + 2 * u] = (int)(mad_wide(v[4 * i + 2 * u], m, c64) >> sft);
                    v[4 * i + 2 * u + 1] = (int)(mad_wide(v[4 * i + 2 * u + 1], m, c64) >> sft);
                  }
                }
              }
              if (act) {
#pragma unroll
                for (int j = 0; j < 16; ++j) v[j] = (int)act_tab0[max(-128, min(127, v[j]))];
              }
              uint32_t w[4];
#pragma unroll
              for (int i = 0; i < 4; ++i) w[i] = pack_sat8(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
              stmatrix_x4_trans_b8(out_slot + 16u * (uint32_t)h, w[0], w[1], w[2], w[3]);
            }
          } else {
            int v[16];
            tmem_ld16(t_row + (uint32_t)(32 * ck), v);
            half(v, ck, 0, pe);
            tmem_ld16(t_row + (uint32_t)(32 * ck + 16), v);
            half(v, ck, 1, pe);
          }
          if (kGroup) {
            // the staged rows leave as 16-byte stores, each to its place in its group
            __syncwarp();
            const int r0 = tc.q0 + 32 * ck, c = tc.p0 + c_first + 16 * (lane & 1);
            const uint32_t g0 = (uint32_t)r0 / (uint32_t)a.group_rows;
            const uint4* so = reinterpret_cast<const uint4*>(gen_base + (my_out - base) + 1024u * (g & 1u)) + lane;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int row = 16 * h + (lane >> 1);
              const int in_group = r0 - (int)g0 * a.group_rows + row;
              int64_t ro = (int64_t)g0 * e.group_stride + in_group;
              if (in_group >= a.group_rows) ro += e.group_stride - a.group_rows;   // (group_rows >= 32)
              if (r0 + row < a.Q && c < a.P) *reinterpret_cast<uint4*>(reinterpret_cast<int8_t*>(e.out) + ro * e.ldo + c) = so[32 * h];
            }
            ++g;
          } else if (tma_out) {
            fence_async_smem();
            __syncwarp();
            if (c_any) tma_store_4d_w(&tmO, my_out + 1024u * (g & 1u), tc.p0 + c_first, tc.q0 + 32 * ck, 0, 0);
            // every lane is past its reads of this slot's residual bytes: fetch those of two chunks on
            if (tma_res) pf_fetch();
            ++g;
          }
        }
      } else {
        // lane = output row, TMEM column = output column
        const int r = tc.p0 + qd * 32 + lane;
        const bool row_ok = r < a.P;
        const int64_t out_row = tc.bo * a.sCo + tc.bi * a.sCi + (int64_t)r * e.ldo;
        const int32_t* bias_row = e.bias32 ? e.bias32 + ((tc.batch % e.bias_batches) * (int64_t)a.P + r) * e.ldbias : nullptr;
        for (int ck = (part - rot) & (kParts - 1); ck < nck; ck += kParts) {
          const int j0 = ck * 32;
          const int c0 = tc.q0 + j0;
          int v[32];
          tmem_ld32(t_row + (uint32_t)j0, v);
          if (!row_ok) continue;
          const int ncol = min(32, a.Q - c0);
          if (bias_row) {
#pragma unroll
            for (int j = 0; j < 32; ++j)
              if (j < ncol) v[j] += __ldg(bias_row + c0 + j);
          }
          if (us >= 33) {   // the usual case: high product word plus 2^(s-33), shifted by s - 32
            const int u_rnd = 1 << (us - 33), u_sh = us - 32;
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = mad_hi(v[j], um, u_rnd) >> u_sh;
          } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = (int)(((long long)v[j] * um + uc) >> us);
          }
          int8_t* o = reinterpret_cast<int8_t*>(e.out) + out_row + c0;
          if (ncol == 32) {
            int4 w0, w1;
            w0.x = (int)pack_sat8(v[0], v[1], v[2], v[3]);     w0.y = (int)pack_sat8(v[4], v[5], v[6], v[7]);
            w0.z = (int)pack_sat8(v[8], v[9], v[10], v[11]);   w0.w = (int)pack_sat8(v[12], v[13], v[14], v[15]);
            w1.x = (int)pack_sat8(v[16], v[17], v[18], v[19]); w1.y = (int)pack_sat8(v[20], v[21], v[22], v[23]);
            w1.z = (int)pack_sat8(v[24], v[25], v[26], v[27]); w1.w = (int)pack_sat8(v[28], v[29], v[30], v[31]);
            reinterpret_cast<int4*>(o)[0] = w0;
            reinterpret_cast<int4*>(o)[1] = w1;
          } else {
#pragma unroll
            for (int j = 0; j < 32; ++j)
              if (j < ncol) o[j] = (int8_t)sat8(v[j]);
          }
        }
      }
      rot = (rot + nck) & (kParts - 1);
      // this warp has read everything it needs from the buffer: hand it back to the MMA warp
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (PAIR) mbar_arrive_cluster(mapa_rank0(acce0 + 8 * buf));   // the issuing CTA waits for both CTAs' warps
        else mbar_arrive(acce0 + 8 * buf);
      }
      if (ROP) {
        ++tiles_in_q;
        if (t + 1 >= t_end || ti.q0(a) != tc.q0) {
          // this warp's last tile of the row block: see the stores complete, release them, count the tiles
          tma_store_wait_all();
          asm volatile("fence.proxy.async;" ::: "memory");
          __threadfence();
          __syncwarp();
          if (lane == 0) {
            unsigned* q_state = a.rop.counters;
            const unsigned qblk = (unsigned)tc.q0 / (unsigned)a.BN;
            unsigned* cnt = q_state + 32 + qblk * kRowStateStride;
            const unsigned old = atomicAdd(cnt, (unsigned)tiles_in_q);
            if (old + (unsigned)tiles_in_q == (unsigned)(a.tiles_p * kEpiWarps)) {
              *cnt = 0u;
              __threadfence();
              asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(cnt + kRowCounters * kRowStateStride), "r"(1u) : "memory");
            }
          }
          tiles_in_q = 0;
        }
      }
    }
    if (ROP && ok) {
      // ---- row operator on this warp's slices ----
      unsigned* q_state = a.rop.counters;
      constexpr int kSlice = ROP == 1 ? 8 : 2;                       // rows of a slice: one batch of the row routine
      const unsigned spb = (unsigned)(a.BN + kSlice - 1) / kSlice;   // slices per row block
      const unsigned total = (unsigned)a.tiles_q * spb;
      const unsigned nwarps = gridDim.x * kEpiWarps;
      const int C = a.P;
      const int nwords = C >> 2;
      const int4* sm_m = reinterpret_cast<const int4*>(rop_smem);
      const LnConsts lk{sm_m, sm_m + nwords, sm_m + 2 * nwords, *rop_flag != 0u};
      unsigned* tab = reinterpret_cast<unsigned*>(rop_smem) + ew * (kGeluTailRows * 64);
      for (unsigned sl = (unsigned)ew * gridDim.x + blockIdx.x; sl < total; sl += nwarps) {
        const unsigned blk = sl / spb, j = sl - blk * spb;
        const int q0 = (int)blk * a.BN;
        const int left = a.Q - q0;
        const int in_blk = left < a.BN ? left : a.BN;
        const int r0 = (int)j * kSlice;
        if (r0 >= in_blk) continue;
        unsigned rdy = 0;
        if (lane == 0) {
          // polls back off: thousands of warps may wait for a handful of flags
          const unsigned* flag = q_state + 32 + (kRowCounters + blk) * kRowStateStride;
          unsigned pause = 64;
          for (uint32_t spin = 0; spin < kSpinLimit; ++spin) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(rdy) : "l"(flag) : "memory");
            if (rdy) break;
            __nanosleep(pause);
            if (pause < 2048) pause <<= 1;
          }
          if (!rdy) {
            *reinterpret_cast<volatile int*>(a.status) = IVIT_ERR_DEVICE_TIMEOUT;
            __threadfence_system();
          }
        }
        rdy = __shfl_sync(0xffffffffu, rdy, 0);
        if (!rdy) break;
        const int nrows = in_blk - r0 < kSlice ? in_blk - r0 : kSlice;
        int8_t* rows0 = reinterpret_cast<int8_t*>(e.out) + (int64_t)(q0 + r0) * e.ldo;
        if (ROP == 1) {
          int8_t* dst = a.rop.ln_out + (int64_t)(q0 + r0) * a.rop.ld_ln;
          if (C <= 384) {
            layernorm_rows<3, 8, true>(rows0, e.ldo, nrows, C, a.rop.M_ln, a.rop.mean_magic, lk, dst, a.rop.ld_ln, lane);
          } else if (C <= 512) {
            layernorm_rows<4, 8, true>(rows0, e.ldo, nrows, C, a.rop.M_ln, a.rop.mean_magic, lk, dst, a.rop.ld_ln, lane);
          } else {
            for (int h = 0; h < nrows; h += 4)
              layernorm_rows<8, 4, true>(rows0 + (int64_t)h * e.ldo, e.ldo, nrows - h < 4 ? nrows - h : 4, C, a.rop.M_ln,
                                         a.rop.mean_magic, lk, dst + (int64_t)h * a.rop.ld_ln, a.rop.ld_ln, lane);
          }
        } else {
          if (C <= 1536) {
            shiftgelu_rows<3, 2, true>(rows0, e.ldo, nrows, C, a.rop.table, tab, rows0, e.ldo, lane);
          } else {
            for (int h = 0; h < nrows; ++h) {
              shiftgelu_rows<8, 1, true>(rows0 + (int64_t)h * e.ldo, e.ldo, 1, C, a.rop.table, tab, rows0 + (int64_t)h * e.ldo,
                                         e.ldo, lane);
              __syncwarp();
            }
          }
          __syncwarp();
        }
      }
    }
    if (tma_out && !kGroup) tma_store_wait_all();
    // only after a timeout: residual bytes fetched for chunks that were never worked on may be in flight
    if (tma_res && !ok && lane == 0)
      for (uint32_t sl = 0; sl < 2; ++sl)
        if ((rpend >> sl) & 1u) mbar_wait(my_resf + 8u * sl, (rpar >> sl) & 1u, a.status);
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync_all();   // neither CTA leaves (or frees tensor memory) while the other may still use it
  if (warp == 1) {
    tc_fence_after();
    if (PAIR) tmem_dealloc_pair(tmem_base, (uint32_t)a.tmem_cols);
    else tmem_dealloc(tmem_base, (uint32_t)a.tmem_cols);
  }
  if (ROP) {
    // the last CTA to get here finds every other CTA out of the queue: it leaves the queue state at zero
    unsigned* q_state = a.rop.counters;
    if (threadIdx.x == 0) {
      __threadfence();
      *rop_flag = atomicAdd(q_state + 2, 1u) == gridDim.x - 1 ? 1u : 0u;
    }
    __syncthreads();
    if (*rop_flag) {
      for (int i = threadIdx.x; i < a.tiles_q; i += kThreads) q_state[32 + (kRowCounters + i) * kRowStateStride] = 0u;
      if (threadIdx.x == 0) q_state[2] = 0u;
      __threadfence();
    }
  }
}

// ---- host side ------------------------------------------------------------------------------

int pow2_at_least(int v) {
  int p = 32;
  while (p < v) p <<= 1;
  return p;
}

constexpr size_t kSmemBudget = 227 * 1024;
constexpr int64_t kPairMinK = 1024;   // contraction length from which the form with a CTA pair per tile is offered
// alignment slack + one KB of barriers, tensor-memory slot, flags and the two 256-entry tables of the residual /
// activation port; a row operator's shared memory follows it
constexpr size_t kSmemFixed = 1024 + 1024;
static_assert(8 * (2 * kMaxStages + 5 + 2 * kEpiWarps) + 32 + 512 <= 1024, "barrier block");


// Clocks that the busiest of `workers` spends when `extent` columns are cut into tiles of bn and each block of columns has
// tiles_other tiles.  A tile costs its operand traffic, (128 + columns) x K bytes (a worker that is a CTA pair: half of
// the columns' bytes per SM) at about 60 bytes per clock into an SM's shared memory, and 900 clocks; the epilogue of all
// but the last one runs beside the next tile.  *dealt: the tiles of a ragged last block are dealt out after the whole ones
// (TileRange), which a kernel that can (deal) does where there is a whole block and it is the shorter way.
// The constants are fitted to 120 measured launch times of Dense layers (4728 ... 50176 rows, 192 ... 4096 channels in and
// out): the width picked with them is 0.7 % slower than the best of the five on average.
double busiest_clocks(int64_t extent, int64_t bn, int64_t tiles_other, int64_t K, int64_t workers, bool pair,
                      bool deal, bool* dealt) {
  auto tile = [&](int64_t cols) { return (double)K * (128.0 + (double)cols * (pair ? 0.5 : 1.0)) / 60.0 + 900.0; };
  auto last = [](int64_t cols) { return 4.0 * (double)cols; };
  const int64_t tiles = tiles_other * ((extent + bn - 1) / bn);
  if (workers > tiles) workers = tiles;
  const double plain = (double)((tiles + workers - 1) / workers) * tile(bn) + last(bn);
  *dealt = false;
  const int64_t ragged = extent % bn;
  if (!deal || ragged == 0 || extent < bn) return plain;
  const int64_t whole = tiles - tiles_other, each = whole / workers, lng = whole % workers, brief = workers - lng;
  if (tiles_other > 2 * brief + lng) return plain;
  const double of_long = lng == 0 ? 0.0 : (double)(each + 1) * tile(bn) + (tiles_other > 2 * brief ? tile(ragged) + last(ragged) : last(bn));
  const double of_brief = (double)each * tile(bn) + (tiles_other > brief ? 2.0 : 1.0) * tile(ragged) + last(ragged);
  const double clocks = (of_long > of_brief ? of_long : of_brief) + 190.0 * (double)(each + 2);   // (the longer walk)
  if (clocks >= plain) return plain;
  *dealt = true;
  return clocks;
}

// Where CTA pairs are faster than single CTAs.  A single CTA fetches (128 + 256) x K bytes per tile, a CTA of a pair
// (128 + 128) x K, but a pair starts later (cluster launch, two barriers across it) and has half as many workers to
// spread the tiles over.  From 1536 on the difference shows once the activations no longer stay in the near L2, at about
// 38 MB of them, and only with enough work per launch (us, pairs / single CTAs): 18464 x 1024 x 4096 55 / 73,
// 25216 x 768 x 3072 48 / 58, 15760 x 1536 x 2048 39.7 / 40.9, but 9232 x 1024 x 3072 24.8 / 22.9,
// 4728 x 4096 x 3072 55 / 44 and 25216 x 512 x 1536 20.8 / 19.3.  Below 1536 the pair's gain is the resident activation
// tile, which with a residual port does not fit: 18464 x 4096 x 1024 59 / 61, 18464 x 3072 x 1024 44.3 / 45.1, but
// 12608 x 3072 x 1024 34.5 / 30.4 and, with the port, 18464 x 1024 x 1024 23.1 / 19.3.
bool pair_pays(int64_t M, int64_t N, int64_t K, bool res) {
  const double macs = (double)M * (double)N * (double)K;
  if (K < 1536) return !res && macs >= 52e9;
  return (double)M * (double)K >= 38e6 && macs >= (K < 3072 ? 36e9 : 29e9);
}

// Tile width along the TMEM columns: the candidate that keeps the busiest CTA the shortest time.
int pick_bn(int64_t extent, int64_t tiles_other, int64_t K, int sm_count, bool deal) {
  if (extent <= 256) return (int)((extent + 31) / 32 * 32);
  int best = 0;
  double best_clocks = 0;
  for (int bn : {256, 224, 192, 160, 128}) {
    bool dealt;
    const double clocks = busiest_clocks(extent, bn, tiles_other, K, sm_count, false, deal, &dealt);
    // ties go to the narrower tile (its MMAs, loads and stores are shorter): the loop runs from wide to narrow
    if (!best || clocks <= best_clocks) { best = bn; best_clocks = clocks; }
  }
  return best;
}

}  // namespace

// The shared-memory limit of a kernel is a per-device attribute: set for the current device at context creation.
int gemm_tc_prepare_device() {
  if (cudaFuncSetAttribute(gemm_tc_kernel<0, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget) != cudaSuccess ||
      cudaFuncSetAttribute(gemm_tc_kernel<1, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget) != cudaSuccess ||
      cudaFuncSetAttribute(gemm_tc_kernel<2, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget) != cudaSuccess ||
      cudaFuncSetAttribute(gemm_tc_kernel<3, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget) != cudaSuccess ||
      cudaFuncSetAttribute(gemm_tc_kernel<4, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget) != cudaSuccess ||
      cudaFuncSetAttribute(gemm_tc_kernel<1, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget) != cudaSuccess ||
      cudaFuncSetAttribute(gemm_tc_kernel<2, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget) != cudaSuccess ||
      cudaFuncSetAttribute(gemm_tc_kernel<1, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget) != cudaSuccess ||
      cudaFuncSetAttribute(gemm_tc_kernel<1, 0, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget) != cudaSuccess ||
      cudaFuncSetAttribute(gemm_tc_kernel<2, 0, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget) != cudaSuccess ||
      cudaFuncSetAttribute(gemm_tc_kernel<1, 0, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget) != cudaSuccess ||
      cudaFuncSetAttribute(gemm_tc_kernel<2, 0, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget) != cudaSuccess)
    return IVIT_ERR_CUDA;
  return IVIT_OK;
}

int launch_gemm_tc(ivit_ctx* ctx, const GemmProblem& g) {
  if (!ctx->tmap_encode) return IVIT_ERR_UNSUPPORTED;
  const int64_t batches = g.batches_outer * g.batches_inner;
  if (batches == 0 || g.M == 0 || g.N == 0) return IVIT_OK;
  if (g.M > 2147483647LL - 512 || g.N > 2147483647LL - 512 || g.K > 65536 || batches > 2147483647LL) return IVIT_ERR_UNSUPPORTED;
  const GemmEpilogue& e = g.epi;
  if (g.lda % 16 || g.ldb % 16 || g.sAo % 16 || g.sAi % 16 || g.sBo % 16 || g.sBi % 16) return IVIT_ERR_UNSUPPORTED;

  TcArgs a{};
  a.epi = e;
  a.res_rows = e.res_rows > 2147483647LL ? 2147483647 : (int)e.res_rows;
  a.group_rows = e.group_rows > 2147483647LL ? 2147483647 : (int)e.group_rows;
  a.K = (int)g.K; a.sCo = g.sCo; a.sCi = g.sCi; a.batches_inner = (int)g.batches_inner;
  a.b_is_param = g.b_is_param;
  a.status = ctx->status_dev;
  CUtensorMap tmP, tmQ;
  const bool dense = g.transB && batches == 1 && !e.bias32;
  bool deal = false;   // short tiles may be dealt out by themselves
  if (dense) {
    if (g.N % 4 || e.ldo % 4 || (reinterpret_cast<uintptr_t>(e.out) & 3)) return IVIT_ERR_UNSUPPORTED;
    // Dense orientation: lanes = output channels (rows of W), columns = output rows (rows of A)
    a.lanes_are_channels = 1;
    a.P = (int)g.N; a.Q = (int)g.M;
    a.tiles_p = (int)((a.P + BM - 1) / BM);
    // A pair of CTAs per tile of 256 channels (cta_group::2) halves the activation bytes per SM and the MMAs issued per
    // SM.  Possible when the layer has whole pairs of channel tiles, a tile for every pair of SMs, and one of the
    // specialised epilogues; pair_pays() says where it is the faster form.
    deal = e.out_dtype == IVIT_I8 && e.group_rows <= 0 && !(reinterpret_cast<uintptr_t>(e.out) & 15) && e.ldo % 16 == 0 &&
           (!e.res || (e.res_rows >= g.M && !(reinterpret_cast<uintptr_t>(e.res) & 15) && e.ldres % 16 == 0)) &&
           !e.act_table && !(e.rop.kind && ctx->row_fusion);   // one of the specialised epilogues (mode 1 or 2 below)
    a.pair = (deal && ctx->gemm_pairs && g.K >= kPairMinK && g.N % (2 * BM) == 0 && ctx->sm_count % 2 == 0 &&
              (g.N / (2 * BM)) * ((g.M + 255) / 256) >= ctx->sm_count / 2 &&
              (ctx->gemm_pairs == 1 || pair_pays(g.M, g.N, g.K, e.res != nullptr))) ? 1 : 0;
    if (a.pair) {
      a.tiles_p = (int)(g.N / (2 * BM));   // pairs of channel tiles
      a.BN = 256;
      a.q_stage_bytes = (a.BN / 2) * BK;   // every CTA of a pair loads half of the activation rows
    } else {
      a.BN = pick_bn(a.Q, a.tiles_p, g.K, ctx->sm_count, deal);
      a.q_stage_bytes = a.BN * BK;
    }
    if (!make_tensor_map(ctx, &tmP, g.B, g.K, g.N, 1, 1, g.ldb, 0, 0, BK, BM, CU_TENSOR_MAP_SWIZZLE_128B, a.p_pos) ||
        !make_tensor_map(ctx, &tmQ, g.A, g.K, g.M, 1, 1, g.lda, 0, 0, BK, a.pair ? a.BN / 2 : a.BN, CU_TENSOR_MAP_SWIZZLE_128B,
                         a.q_pos))
      return IVIT_ERR_UNSUPPORTED;
  } else {
    // MatMul orientation: lanes = rows of A; the epilogue's 16-byte stores need aligned output rows
    if (e.out_dtype != IVIT_I8 || e.bias || e.res || e.scale.mult_c || e.group_rows > 0 || e.act_table) return IVIT_ERR_UNSUPPORTED;
    if ((reinterpret_cast<uintptr_t>(e.out) & 15) || e.ldo % 16 || g.sCo % 16 || g.sCi % 16) return IVIT_ERR_UNSUPPORTED;
    a.P = (int)g.M; a.Q = (int)g.N;
    a.tiles_p = (int)((a.P + BM - 1) / BM);
    a.q_mn = g.transB ? 0 : 1;
    if (!make_tensor_map(ctx, &tmP, g.A, g.K, g.M, g.batches_inner, g.batches_outer, g.lda, g.sAi, g.sAo, BK, BM,
                  CU_TENSOR_MAP_SWIZZLE_128B, a.p_pos))
      return IVIT_ERR_UNSUPPORTED;
    if (a.q_mn) {
      // the whole N extent is one tile whose k rows are N bytes wide: 32, 64 or 128
      if (g.N != 32 && g.N != 64 && g.N != 128) return IVIT_ERR_UNSUPPORTED;
      a.BN = (int)g.N;
      a.q_row_bytes = (int)g.N;
      a.q_stage_bytes = BK * a.q_row_bytes;
      const CUtensorMapSwizzle swz = a.q_row_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B
                                     : (a.q_row_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
      if (!make_tensor_map(ctx, &tmQ, g.B, g.N, g.K, g.batches_inner, g.batches_outer, g.ldb, g.sBi, g.sBo, a.q_row_bytes, BK,
                    swz, a.q_pos))
        return IVIT_ERR_UNSUPPORTED;
    } else {
      a.BN = pick_bn(a.Q, (int64_t)a.tiles_p * batches, g.K, ctx->sm_count, false);
      a.q_stage_bytes = a.BN * BK;
      if (!make_tensor_map(ctx, &tmQ, g.B, g.K, g.N, g.batches_inner, g.batches_outer, g.ldb, g.sBi, g.sBo, BK, a.BN,
                    CU_TENSOR_MAP_SWIZZLE_128B, a.q_pos))
        return IVIT_ERR_UNSUPPORTED;
    }
  }
  CUtensorMap tmL = tmQ;
  a.q_last_bytes = a.q_stage_bytes;
  if (deal && a.Q % a.BN != 0) {
    const int rows = ((a.Q % a.BN + 31) & ~31) / (a.pair ? 2 : 1);
    int lpos[3];
    if (!make_tensor_map(ctx, &tmL, g.A, g.K, g.M, 1, 1, g.lda, 0, 0, BK, rows, CU_TENSOR_MAP_SWIZZLE_128B, lpos))
      return IVIT_ERR_UNSUPPORTED;
    a.q_last_bytes = rows * BK;
  }
  CUtensorMap tmO = tmP;
  if (dense && e.out_dtype == IVIT_I8 && e.group_rows <= 0 && !(reinterpret_cast<uintptr_t>(e.out) & 15) && e.ldo % 16 == 0) {
    int opos[3];
    a.tma_out = make_tensor_map(ctx, &tmO, reinterpret_cast<const int8_t*>(e.out), g.N, g.M, 1, 1, e.ldo, 0, 0, 32, 32,
                         CU_TENSOR_MAP_SWIZZLE_NONE, opos) ? 1 : 0;
  }
  CUtensorMap tmR = tmP;
  if (a.tma_out && e.res && e.res_rows >= g.M && !(reinterpret_cast<uintptr_t>(e.res) & 15) && e.ldres % 16 == 0) {
    int rpos[3];
    a.tma_res = make_tensor_map(ctx, &tmR, e.res, g.N, g.M, 1, 1, e.ldres, 0, 0, 32, 32, CU_TENSOR_MAP_SWIZZLE_NONE,
                                rpos) ? 1 : 0;
  }
  // grouped output rows: the warps fill and empty the staging slots themselves (MODE 4)
  const bool grouped = dense && e.out_dtype == IVIT_I8 && e.group_rows >= 32 && g.N % 16 == 0 && !(reinterpret_cast<uintptr_t>(e.out) & 15) &&
                       e.ldo % 16 == 0 && e.res && e.res_rows >= 32 && !(reinterpret_cast<uintptr_t>(e.res) & 3) && e.ldres % 4 == 0 && !e.act_table;
  if (grouped) a.tma_out = a.tma_res = 1;   // (the slots exist)
  // The row operator runs in this kernel when the epilogue is one of the specialised forms (staged int8 output,
  // residual absent or fetched by TMA), the rows fit the tail routines and there is a counter per row block.
  int rop = 0;
  if (e.rop.kind && !grouped && a.lanes_are_channels && a.tma_out && (!e.res || a.tma_res) && !e.act_table && ctx->row_fusion) {
    const int64_t blocks_q = (a.Q + a.BN - 1) / a.BN;
    if (blocks_q <= kRowCounters && e.rop.kind == 1 && g.N <= 1024 && (ctx->row_fusion & 1)) rop = 1;
    if (blocks_q <= kRowCounters && e.rop.kind == 2 && g.N % 16 == 0 && g.N <= 4096 && !e.res && (ctx->row_fusion & 2)) rop = 2;
  }
  a.rop = e.rop;
  a.rop.kind = rop;
  a.rop.counters = ctx->rowblk_dev;
  a.rop.mean_magic = (unsigned)(0x100000000ull / (unsigned long long)(2 * g.N)) + 1u;
  a.rop.vec = e.rop.gs.mult_c && e.rop.gs.shift_c && !(reinterpret_cast<uintptr_t>(e.rop.gs.mult_c) & 15) &&
              !(reinterpret_cast<uintptr_t>(e.rop.gs.shift_c) & 3) && !(reinterpret_cast<uintptr_t>(e.rop.beta) & 15);
  const size_t rop_bytes = rop == 1 ? ((size_t)g.N * 12 + 1023) / 1024 * 1024 : (rop == 2 ? (size_t)kGeluTailSmem : 0);
  const size_t out_stage = (a.tma_out ? (size_t)kEpiWarps * 2048 : 0) + (a.tma_res ? (size_t)kEpiWarps * 2048 : 0);
  // short K: keep the activation tile resident if that still leaves four weight stages
  const size_t kblocks = (size_t)((g.K + BK - 1) / BK);
  const size_t qres_bytes = kblocks * a.q_stage_bytes;
  a.q_resident = (dense && kSmemFixed + rop_bytes + out_stage + qres_bytes + 4 * (size_t)BM * BK <= kSmemBudget) ? 1 : 0;
  const size_t stage = (size_t)BM * BK + (a.q_resident ? 0 : a.q_stage_bytes);
  const size_t fixed = out_stage + (a.q_resident ? qres_bytes : 0);
  int stages = (int)((kSmemBudget - kSmemFixed - rop_bytes - fixed) / stage);
  a.stages = stages > kMaxStages ? kMaxStages : stages;
  if (a.stages < 2) return IVIT_ERR_UNSUPPORTED;
  a.tmem_cols = pow2_at_least(2 * a.BN);
  a.tiles_q = (int)((a.Q + a.BN - 1) / a.BN);
  const int64_t total_tiles = (int64_t)a.tiles_p * a.tiles_q * batches;
  if (total_tiles > 2147483647LL) return IVIT_ERR_UNSUPPORTED;
  a.total_tiles = (int)total_tiles;

  const size_t smem = kSmemFixed + rop_bytes + (size_t)a.stages * stage + fixed;
  const int workers_max = a.pair ? ctx->sm_count / 2 : ctx->sm_count;   // CTAs, or CTA pairs
  const int workers = a.total_tiles < workers_max ? a.total_tiles : workers_max;
  const unsigned grid = (unsigned)(a.pair ? 2 * workers : workers);
  // the encoder block's Dense layers take the specialised instantiations
  int mode = (a.lanes_are_channels && a.tma_out && (!e.res || a.tma_res)) ? (a.tma_res ? 2 : 1) : 0;
  if (e.act_table) mode = mode == 1 ? 3 : 0;
  if (grouped) mode = 4;
  bool dealt;
  busiest_clocks(a.Q, a.BN, a.tiles_p, g.K, workers_max, a.pair != 0, deal && (mode == 1 || mode == 2) && rop == 0, &dealt);
  a.short_tiles = dealt ? a.tiles_p : 0;
  const int dealt_evenly = a.total_tiles - a.short_tiles;   // all tiles, or the whole ones
  a.tiles_each = dealt_evenly / workers;
  a.tiles_extra = dealt_evenly % workers;
  const LastMap<true> last_map{tmL};
  LaunchScope ls(ctx, KIND_GEMM_TC, 2.0 * (double)batches * (double)g.M * (double)g.N * (double)g.K);
  if (a.pair && (mode != 1 && mode != 2)) return IVIT_ERR_UNSUPPORTED;   // (the conditions above imply mode 1 or 2)
  if (a.pair) ++ctx->pair_launches;
  if (a.pair && mode == 2) launch_k_pair(gemm_tc_kernel<2, 0, true>, dim3(grid), dim3(kThreads), smem, ctx->stream, tmP, tmQ, tmO, tmR, a, last_map);
  else if (a.pair) launch_k_pair(gemm_tc_kernel<1, 0, true>, dim3(grid), dim3(kThreads), smem, ctx->stream, tmP, tmQ, tmO, tmR, a, last_map);
  else if (rop == 1 && mode == 2) launch_k(gemm_tc_kernel<2, 1>, dim3(grid), dim3(kThreads), smem, ctx->stream, tmP, tmQ, tmO, tmR, a, LastMap<false>{});
  else if (rop == 1 && mode == 1) launch_k(gemm_tc_kernel<1, 1>, dim3(grid), dim3(kThreads), smem, ctx->stream, tmP, tmQ, tmO, tmR, a, LastMap<false>{});
  else if (rop == 2 && mode == 1) launch_k(gemm_tc_kernel<1, 2>, dim3(grid), dim3(kThreads), smem, ctx->stream, tmP, tmQ, tmO, tmR, a, LastMap<false>{});
  else if (dealt && mode == 2) launch_k(gemm_tc_kernel<2, 0, false, true>, dim3(grid), dim3(kThreads), smem, ctx->stream, tmP, tmQ, tmO, tmR, a, last_map);
  else if (dealt && mode == 1) launch_k(gemm_tc_kernel<1, 0, false, true>, dim3(grid), dim3(kThreads), smem, ctx->stream, tmP, tmQ, tmO, tmR, a, last_map);
  else if (mode == 4) launch_k(gemm_tc_kernel<4, 0>, dim3(grid), dim3(kThreads), smem, ctx->stream, tmP, tmQ, tmO, tmR, a, LastMap<false>{});
  else if (mode == 3) launch_k(gemm_tc_kernel<3, 0>, dim3(grid), dim3(kThreads), smem, ctx->stream, tmP, tmQ, tmO, tmR, a, LastMap<false>{});
  else if (mode == 2) launch_k(gemm_tc_kernel<2, 0>, dim3(grid), dim3(kThreads), smem, ctx->stream, tmP, tmQ, tmO, tmR, a, LastMap<false>{});
  else if (mode == 1) launch_k(gemm_tc_kernel<1, 0>, dim3(grid), dim3(kThreads), smem, ctx->stream, tmP, tmQ, tmO, tmR, a, LastMap<false>{});
  else launch_k(gemm_tc_kernel<0, 0>, dim3(grid), dim3(kThreads), smem, ctx->stream, tmP, tmQ, tmO, tmR, a, LastMap<false>{});
  ctx->rowop_fused = (rop != 0 && (mode == 1 || mode == 2)) ? 1 : 0;
  return ls.done();
}

}  // namespace ivit
