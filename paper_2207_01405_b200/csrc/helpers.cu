// Data-movement helpers around the encoder (patch extraction, row gathers, class-token rows,
// token pooling).  Pure permutations / sums; none of them is described in the paper.
#include "common.cuh"

namespace ivit {

// Quotients of n < 2^31 by a divisor that the host knows: with 2^(l-1) < d <= 2^l and m = ceil(2^(31+l) / d), the high
// product word of n m, shifted by l - 1, is the quotient (m d - 2^(31+l) < 2^l, so the error stays below 1 / d).  The
// index arithmetic of these kernels was most of their time: seven hardware-less divisions per 16 bytes moved.
struct FastDiv {
  unsigned d, m;
  int s;
  explicit FastDiv(unsigned d_) : d(d_), m(0), s(0) {
    int l = 0;
    while (l < 31 && (1u << l) < d) ++l;
    if (d > 1) { m = (unsigned)(((1ull << (31 + l)) + d - 1) / d); s = l - 1; }
  }
  __device__ __forceinline__ unsigned div(unsigned n) const { return d == 1 ? n : __umulhi(n, m) >> s; }
  __device__ __forceinline__ unsigned divmod(unsigned n, unsigned& rem) const {
    const unsigned q = div(n);
    rem = n - q * d;
    return q;
  }
};

// Row of patch (gy, gx) inside its image: raster order, or window by window.
struct PatchOrder {
  FastDiv window;
  unsigned gw, gww;   // patches per image row; windows per row of windows (0: raster order)
  PatchOrder(unsigned gw_, unsigned window_) : window(window_ ? window_ : 1u), gw(gw_), gww(window_ ? gw_ / window_ : 0u) {}
  __device__ __forceinline__ unsigned row(unsigned gy, unsigned gx) const {
    if (gww == 0) return gy * gw + gx;
    unsigned iy, ix;
    const unsigned wy = window.divmod(gy, iy), wx = window.divmod(gx, ix);
    return ((wy * gww + wx) * window.d + iy) * window.d + ix;
  }
};

// A row written once per group, 16 bytes at a time (the class token in front of every image's patches).
struct FillRows {
  const int8_t* src;
  int8_t* dst;
  int64_t group_stride;
  FastDiv per_row;
  unsigned total;   // 16-byte pieces
  __device__ __forceinline__ void run(unsigned t0, unsigned stride) const {
    for (unsigned t = t0; t < total; t += stride) {
      unsigned v;
      const unsigned g = per_row.divmod(t, v);
      reinterpret_cast<int4*>(dst + (int64_t)g * group_stride)[v] = __ldg(reinterpret_cast<const int4*>(src) + v);
    }
  }
};

// One thread per 4 output bytes (px .. px+3 of one patch row); P % 4 == 0.
__global__ void patchify_kernel(const int8_t* __restrict__ img, int64_t B, int C, int Hi, int Wi, int P,
                                int window, int8_t* __restrict__ out, int64_t ldout, int64_t total_words) {
  pdl_wait();
  pdl_trigger();   // (after the wait: the first kernel of a forward)
  const int gh = Hi / P, gw = Wi / P;
  const int kw = C * P * P / 4;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total_words;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int w = (int)(t % kw);
    const int64_t prow = t / kw;  // raster patch index over the batch
    const int gx = (int)(prow % gw), gy = (int)((prow / gw) % gh);
    const int64_t b = prow / ((int64_t)gw * gh);
    const int px = (w * 4) % P, py = ((w * 4) / P) % P, c = (w * 4) / (P * P);
    const int v = __ldg(reinterpret_cast<const int*>(img + ((b * C + c) * Hi + gy * P + py) * (int64_t)Wi + gx * P + px));
    int64_t row;
    if (window > 0) {
      const int wy = gy / window, wx = gx / window, iy = gy % window, ix = gx % window;
      row = (int64_t)(wy * (gw / window) + wx) * window * window + iy * window + ix;
    } else {
      row = (int64_t)gy * gw + gx;
    }
    *reinterpret_cast<int*>(out + (b * gh * gw + row) * ldout + w * 4) = v;
  }
}

// P % 16 == 0, aligned image rows: one thread moves 16 bytes (px .. px+15 of one patch row); `segs` = P / 16 such pieces
// per patch row.  The class rows of the token matrix, if any, are written beside it.
// Bound by the copy itself: 128 images of 224 x 224, back to back, 8.2 -> 7.6 us.
__global__ void patchify_vec_kernel(const int8_t* __restrict__ img, FastDiv per_row, FastDiv Hi, FastDiv C, FastDiv segs, FastDiv P,
                                    PatchOrder order, unsigned patches, int8_t* __restrict__ out, int64_t ldout,
                                    unsigned total_vecs, FillRows fill) {
  pdl_wait();
  pdl_trigger();   // (after the wait: the first kernel of a forward)
  const unsigned t0 = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
  for (unsigned t = t0; t < total_vecs; t += stride) {
    // t enumerates the image in memory order: consecutive threads read consecutive 16-byte pieces
    const int4 v = __ldg(reinterpret_cast<const int4*>(img) + t);
    unsigned xv, y, c, sx, py;
    const unsigned line = per_row.divmod(t, xv);                  // line = (b * C + c) * Hi + y
    const unsigned bc = Hi.divmod(line, y), b = C.divmod(bc, c);
    const unsigned gx = segs.divmod(xv, sx), gy = P.divmod(y, py);
    *reinterpret_cast<int4*>(out + ((int64_t)b * patches + order.row(gy, gx)) * ldout + (c * P.d + py) * P.d + sx * 16) = v;
  }
  fill.run(t0, stride);
}

// P = 4: one thread per patch, its C x 4 pieces of a row read as words (side by side for neighbouring threads), written as
// 16 bytes per channel.  64 images of 224 x 224 x 3, back to back: 26.5 -> 4.9 us (one word per thread, 64-bit divisions).
__global__ void patchify4_kernel(const int8_t* __restrict__ img, int C, int Hi, int Wi, FastDiv gw, FastDiv gh, PatchOrder order,
                                 int8_t* __restrict__ out, int64_t ldout, unsigned total_patches) {
  pdl_wait();
  pdl_trigger();   // (after the wait: the first kernel of a forward)
  const unsigned patches = gw.d * gh.d;
  for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < total_patches; t += gridDim.x * blockDim.x) {
    unsigned gx, gy;
    const unsigned line = gw.divmod(t, gx), b = gh.divmod(line, gy);
    const int* src = reinterpret_cast<const int*>(img + ((int64_t)b * C * Hi + 4 * gy) * Wi) + gx;
    int4* dst = reinterpret_cast<int4*>(out + ((int64_t)b * patches + order.row(gy, gx)) * ldout);
    const int wl = Wi / 4;
#pragma unroll 3
    for (int c = 0; c < C; ++c) {
      const int* s = src + (int64_t)c * Hi * wl;
      dst[c] = make_int4(__ldg(s), __ldg(s + wl), __ldg(s + 2 * wl), __ldg(s + 3 * wl));
    }
  }
}

// dst row r = src row index[r], 16 bytes per thread and step, two in flight.  Fewer than 2^31 pieces.
__global__ void gather_rows_kernel(const int8_t* __restrict__ src, int64_t ldsrc, const int32_t* __restrict__ index,
                                   FastDiv per_row, int8_t* __restrict__ dst, int64_t lddst, unsigned total) {
  pdl_trigger();
  pdl_wait();
  const unsigned stride = gridDim.x * blockDim.x;
  for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += 2 * stride) {
    const bool two = t + stride < total;
    unsigned v0, v1;
    const unsigned r0 = per_row.divmod(t, v0), r1 = per_row.divmod(two ? t + stride : t, v1);
    const int i0 = __ldg(index + r0), i1 = __ldg(index + r1);
    const int4 x0 = __ldg(reinterpret_cast<const int4*>(src + (int64_t)i0 * ldsrc) + v0);
    const int4 x1 = __ldg(reinterpret_cast<const int4*>(src + (int64_t)i1 * ldsrc) + v1);
    reinterpret_cast<int4*>(dst + (int64_t)r0 * lddst)[v0] = x0;
    if (two) reinterpret_cast<int4*>(dst + (int64_t)r1 * lddst)[v1] = x1;
  }
}

__global__ void fill_rows_kernel(FillRows fill) {
  pdl_wait();
  pdl_trigger();   // (after the wait: the first kernel of a forward)
  fill.run(blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

// Four channels per thread, the T rows of a group dealt to the eight warps of a block: fewer dependent loads per thread
// than with one channel per thread, the form below.
__global__ void __launch_bounds__(256) token_mean4_kernel(const int8_t* __restrict__ in, int64_t ldin, int T, int C4, unsigned nb,
                                                          ScaleDev scale, int8_t* __restrict__ out, int64_t ldout) {
  __shared__ int4 part[8][32];
  pdl_trigger();
  pdl_wait();
  const int64_t g = blockIdx.x / nb;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, c4 = (int)(blockIdx.x % nb) * 32 + lane;
  int4 s = make_int4(0, 0, 0, 0);
  if (c4 < C4) {
    const int* src = reinterpret_cast<const int*>(in + g * T * ldin) + c4;
#pragma unroll 8
    for (int k = w; k < T; k += 8) {
      const int x = __ldg(src + k * (ldin >> 2));
      s.x += (int)(int8_t)x; s.y += (int)(int8_t)(x >> 8); s.z += (int)(int8_t)(x >> 16); s.w += x >> 24;
    }
  }
  part[w][lane] = s;
  __syncthreads();
  if (w == 0 && c4 < C4) {
    for (int k = 1; k < 8; ++k) {
      const int4 p = part[k][lane];
      s.x += p.x; s.y += p.y; s.z += p.z; s.w += p.w;
    }
    const int m = scale.mult, sh = clamp_shift(scale.shift);
    reinterpret_cast<int*>(out + g * ldout)[c4] =
        (sat8(rq(s.x, m, sh)) & 0xff) | (sat8(rq(s.y, m, sh)) & 0xff) << 8 | (sat8(rq(s.z, m, sh)) & 0xff) << 16 | sat8(rq(s.w, m, sh)) << 24;
  }
}

__global__ void token_mean_kernel(const int8_t* __restrict__ in, int64_t ldin, int64_t groups, int T, int C,
                                  ScaleDev scale, int8_t* __restrict__ out, int64_t ldout) {
  pdl_trigger();
  pdl_wait();
  const int64_t total = groups * C;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t g = t / C;
    const int c = (int)(t % C);
    int s = 0;
    for (int k = 0; k < T; ++k) s += __ldg(in + (g * T + k) * ldin + c);
    out[g * ldout + c] = (int8_t)sat8(rq(s, scale.mult, clamp_shift(scale.shift)));
  }
}

static int grid_for(ivit_ctx* ctx, int64_t items, int threads) {
  int64_t want = (items + threads - 1) / threads;
  const int64_t cap = (int64_t)ctx->sm_count * 16;
  return (int)(want < cap ? (want < 1 ? 1 : want) : cap);
}

constexpr int64_t kMaxPieces = 0x7fffffff;   // what FastDiv divides

int launch_patchify(ivit_ctx* ctx, const int8_t* img, int64_t B, int64_t C, int64_t Hi, int64_t Wi, int64_t P, int64_t window,
                    int8_t* out, int64_t ldout, const int8_t* fill_src, int64_t fill_width, int8_t* fill_dst, int64_t fill_stride) {
  const int64_t total = B * C * Hi * Wi / 4;
  if (total == 0) return IVIT_OK;
  const bool wide = P % 16 == 0 && Wi % 16 == 0 && ldout % 16 == 0 && total / 4 < kMaxPieces && !(reinterpret_cast<uintptr_t>(img) & 15) &&
                    !(reinterpret_cast<uintptr_t>(out) & 15) && (!fill_src || B * (fill_width / 16) < kMaxPieces);
  if (fill_src && !wide) {
    const int rc = launch_fill_rows(ctx, fill_src, fill_width, fill_dst, fill_stride, B);
    if (rc) return rc;
  }
  LaunchScope ls(ctx, KIND_MOVE, 2.0 * (double)total * 4 + (fill_src && wide ? (double)B * (double)fill_width : 0.0));
  const unsigned gw = (unsigned)(Wi / P), gh = (unsigned)(Hi / P);
  if (wide) {
    const FillRows fill{fill_src, fill_dst, fill_stride, FastDiv(fill_src ? (unsigned)(fill_width / 16) : 1u),
                        fill_src ? (unsigned)(B * (fill_width / 16)) : 0u};
    launch_k(patchify_vec_kernel, dim3(grid_for(ctx, total / 4, 256)), dim3(256), 0, ctx->stream, img, FastDiv((unsigned)(Wi / 16)),
             FastDiv((unsigned)Hi), FastDiv((unsigned)C), FastDiv((unsigned)(P / 16)), FastDiv((unsigned)P), PatchOrder(gw, (unsigned)window),
             gw * gh, out, ldout, (unsigned)(total / 4), fill);
  } else if (P == 4 && ldout % 16 == 0 && !(reinterpret_cast<uintptr_t>(img) & 3) && !(reinterpret_cast<uintptr_t>(out) & 15) &&
             B * gw * gh < kMaxPieces) {
    launch_k(patchify4_kernel, dim3(grid_for(ctx, B * gw * gh, 256)), dim3(256), 0, ctx->stream, img, (int)C, (int)Hi, (int)Wi, FastDiv(gw),
             FastDiv(gh), PatchOrder(gw, (unsigned)window), out, ldout, (unsigned)(B * gw * gh));
  } else {
    launch_k(patchify_kernel, dim3(grid_for(ctx, total, 256)), dim3(256), 0, ctx->stream, img, B, (int)C, (int)Hi, (int)Wi, (int)P,
             (int)window, out, ldout, total);
  }
  return ls.done();
}

int launch_gather_rows(ivit_ctx* ctx, const int8_t* src, int64_t ldsrc, const int32_t* index,
                       int64_t n_rows, int64_t width, int8_t* dst, int64_t lddst) {
  const int64_t per_row = width / 16, slice = kMaxPieces / per_row;
  if (slice == 0) return IVIT_ERR_UNSUPPORTED;   // a row of 2^35 bytes
  for (int64_t r = 0; r < n_rows; r += slice) {
    const int64_t total = (n_rows - r < slice ? n_rows - r : slice) * per_row;
    LaunchScope ls(ctx, KIND_MOVE, 32.0 * (double)total);
    launch_k(gather_rows_kernel, dim3(grid_for(ctx, total, 256)), dim3(256), 0, ctx->stream, src, ldsrc, index + r, FastDiv((unsigned)per_row),
             dst + r * lddst, lddst, (unsigned)total);
    const int rc = ls.done();
    if (rc) return rc;
  }
  return IVIT_OK;
}

int launch_fill_rows(ivit_ctx* ctx, const int8_t* src_row, int64_t width, int8_t* dst,
                     int64_t group_stride, int64_t groups) {
  const int64_t per_row = width / 16, slice = kMaxPieces / per_row;
  if (slice == 0) return IVIT_ERR_UNSUPPORTED;   // a row of 2^35 bytes
  for (int64_t g = 0; g < groups; g += slice) {
    const int64_t total = (groups - g < slice ? groups - g : slice) * per_row;
    LaunchScope ls(ctx, KIND_MOVE, 16.0 * (double)total);
    launch_k(fill_rows_kernel, dim3(grid_for(ctx, total, 256)), dim3(256), 0, ctx->stream,
             FillRows{src_row, dst + g * group_stride, group_stride, FastDiv((unsigned)per_row), (unsigned)total});
    const int rc = ls.done();
    if (rc) return rc;
  }
  return IVIT_OK;
}

int launch_token_mean(ivit_ctx* ctx, const int8_t* in, int64_t ldin, int64_t groups, int64_t T,
                      int64_t C, ScaleDev scale, int8_t* out, int64_t ldout) {
  if (groups == 0) return IVIT_OK;
  LaunchScope ls(ctx, KIND_MOVE, (double)groups * (double)C * (double)(T + 1));
  const int64_t nb = (C / 4 + 31) / 32;
  // Many groups of few rows keep the chip busy without dealing the rows out, and a block costs more than their sums (us, four
  // channels and eight warps / one channel per thread): 64 groups of 49 x 768 3.0 / 3.6, 300 of them 6.1 / 5.9, 1000
  // 15.3 / 12.9; 300 of 4 x 384 2.1 / 2.0, 3000 10.5 / 6.9; 500 of 196 x 768 15.0 / 27.7.
  const bool deal_rows = T >= 128 || groups * nb <= (int64_t)ctx->sm_count * (T < 16 ? 3 : 8);
  if (deal_rows && C % 4 == 0 && ldin % 4 == 0 && ldout % 4 == 0 && !((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 3) &&
      groups * nb < kMaxPieces) {
    launch_k(token_mean4_kernel, dim3((unsigned)(groups * nb)), dim3(256), 0, ctx->stream, in, ldin, (int)T, (int)(C / 4), (unsigned)nb, scale,
             out, ldout);
  } else {
    launch_k(token_mean_kernel, dim3(grid_for(ctx, groups * C, 256)), dim3(256), 0, ctx->stream, in, ldin, groups, (int)T, (int)C, scale, out,
             ldout);
  }
  return ls.done();
}

}  // namespace ivit
