// ragged.cuh -- one persistent launch over a ragged batch of images (different
// sizes and filter sizes), driven by a tile table in device memory.
//
// The GigaAPI paper wanted to process a "database" of images in one go and
// gave up (Section 5, "No Batch Processing for Images"); this kernel does it:
//  * the host cuts every (image, channel) into chunks of up to 4 tiles of
//    64 x 128 pixels (1 to 32, powers of 2: the plan's autotuner times them) and
//    sorts the chunks longest first (cost K^2 per pixel);
//  * CTAs (one per SM, 16 warps) pull chunk numbers from an atomic counter,
//    stage each tile's x and dy once, and run the three ops on it: warps 0-7
//    the forward and warps 8-15 the input gradient, 8 rows each, then all 16
//    the filter gradient, split into groups of filter rows and tile rows.  The
//    three cost the same per pixel, so every warp has the same work between
//    the tile's barriers, and a scheduler has four busy warps throughout.
//    (With fixed roles -- 4 warps forward, 4 input gradient, 4 or 8 filter
//    gradient -- the warps of the slowest role run alone at a tile's end, and 4
//    of the 16 idle for K <= 9.  One 3 x 2001 x 2999 image, zero border, that ->
//    this: K = 3 155 -> 109 us, K = 11 380 -> 333, BF16 K = 3 224 -> 129, K = 11 472 ->
//    397; forward alone, clamp border, K = 3 72 -> 53, K = 11 168 -> 131.)
//  * each chunk writes one K*K vector of FP32 filter-gradient partials; the
//    CTA that completes the last chunk of an (image, channel) -- detected with
//    a per-(image, channel) atomic counter after a memory fence -- sums that
//    image-channel's partials in FP64 in a fixed order (deterministic) and, for
//    the clamp border, folds the edges of dx.  No CTA ever waits for another.
#pragma once

#include "dw_fold.cuh"
#include "dw_kernels.cuh"

namespace giga {

constexpr int kRagThreads = 512;
constexpr int kRagWarps = kRagThreads / 32;
constexpr int kRagTilesPerChunk = 4;  // the plan's default; the autotuner may pick 1 to 32
constexpr int kRagMaxK = 15;

struct RagImage {
  const void* x;
  void* y;
  const void* dy;
  void* dx;
  const float* w;
  float* dw;
  int64_t partial_base;  // float offset of this image's partials
  int H, W, C, K;
  int nch;      // chunks per channel
  int ic_base;  // completion counter of (this image, channel 0)
  int vec;  // every tensor's rows start on a chunk boundary (16 bytes FP32, 8 BF16)
  int odd_rows;  // has_odd_rows of x and dy
};

struct RagChunk {
  int image, channel, tile_begin, tile_end;
};

struct RagParams {
  const RagImage* images;
  const RagChunk* chunks;
  int* counters;  // [0]: work counter, [1 + ic]: finished chunks of (image, channel) ic
  float* partials;
  int n_chunks;
  int tpc;  // tiles per chunk
  int ops;  // GIGA_OP_* bitmask
  int border;
};

// Filter-row groups of the filter gradient: as few as keep a warp's
// accumulators (rows of the group x K) beside the forward's within the 128
// registers a thread of a 16-warp CTA has.
template <int K>
constexpr int rag_groups() {
  return K <= 5 ? 1 : (K <= 9 ? 2 : (K <= 11 ? 4 : 8));
}

template <int K, typename T>
struct RagShape {
  using G = Geo<K, sizeof(T), true>;
  static constexpr int GT = rag_groups<K>();
  static constexpr int WPG = kRagWarps / GT;
  static constexpr int AT = (K + GT - 1) / GT;
  static constexpr int DW_ROWS = kBwdTileH / WPG;
  static constexpr int DR = 4;                      // dy rows per unrolled block
  static constexpr int ROWS = kBwdTileH + 2 * G::R;
  static_assert(DW_ROWS % DR == 0, "whole row blocks");
};

// Shared memory, sized for the largest filter: two tile stages (x and dy
// tiles), two filter buffers (a chunk's filter and its rotation; indexed by
// chunk parity so the next chunk's filter can be staged while the current one
// is in use), the filter-gradient reduction rows and two ints.
template <typename T>
struct RagLayout {
  using G = Geo<kRagMaxK, sizeof(T), true>;
  static constexpr int TILE = round_up((kBwdTileH + 2 * G::R) * G::SP * (int)sizeof(T), 128);
  static constexpr int STAGE = 2 * TILE;          // x, then dy
  static constexpr int WB = G::WPAD * 4;          // one filter
  static constexpr int FILT = 2 * STAGE;          // [2][w, wf]
  static constexpr int RED = FILT + 4 * WB;       // [2 chunks][w, wf] filters
  static constexpr int RED_FLOATS = 45;           // K = 9: 5 rows x 9 taps
  // the row buffers of store_rows, one per warp, share the reduction rows'
  // space: those are used at a chunk's end, behind barriers
  static constexpr int BUF = RED;
  static constexpr int INTS = RED + kRagWarps * kRowBuf;
  static constexpr int IMAGE = INTS + 16;         // the current chunk's RagImage
  static constexpr int SM_BYTES = IMAGE + (int)sizeof(RagImage);
  static_assert(RagShape<9, T>::AT * 9 <= RED_FLOATS && RagShape<11, T>::AT * 11 <= RED_FLOATS &&
                    RagShape<15, T>::AT * 15 <= RED_FLOATS && RED_FLOATS * 4 <= kRowBuf,
                "reduction rows");
  static_assert(SM_BYTES <= 227 * 1024, "shared memory");
};

template <typename T>
constexpr size_t rag_max_smem() {
  return (size_t)RagLayout<T>::SM_BYTES;
}

// Issue the copies of tile t of chunk ch (image im) into stage sb and, for the
// first tile of a chunk, its filters into filter buffer fb (no commit).
template <typename T>
__device__ __forceinline__ void rag_stage(const RagParams& p, const RagChunk& ch,
                                          const RagImage& im, int t, char* sm, int sb, int fb,
                                          bool filters) {
  using L = RagLayout<T>;
  const int K = im.K, R = (K - 1) / 2, RP = geo_rp(K, sizeof(T));
  const int SP = geo_pitch(K, sizeof(T), true);
  const int H = im.H, W = im.W;
  const int tiles_x = (W + kTileW - 1) / kTileW;
  const int ty0 = (t / tiles_x) * kBwdTileH, tx0 = (t % tiles_x) * kTileW;
  const int64_t off = (int64_t)ch.channel * H * W;
  const bool do_fwd = p.ops & 1, do_dx = p.ops & 2, do_dw = p.ops & 4;
  T* sx = reinterpret_cast<T*>(sm + sb * L::STAGE);
  T* sdy = reinterpret_cast<T*>(sm + sb * L::STAGE + L::TILE);
  const T* x = static_cast<const T*>(im.x);
  const T* dy = static_cast<const T*>(im.dy);
  if (do_fwd || do_dw)
    stage_any<T, kRagThreads>(sx, x + off, H, W, ty0, tx0, kBwdTileH + 2 * R, R, RP, SP,
                              im.odd_rows);
  if (do_dx || do_dw)
    stage_any<T, kRagThreads>(sdy, dy + off, H, W, ty0, tx0, kBwdTileH + 2 * R, R, RP, SP,
                              im.odd_rows);
  // w may be NULL when neither the forward nor the input gradient is requested
  if (filters && (do_fwd || do_dx)) {
    const float* wc = im.w + (int64_t)ch.channel * K * K;
    float* f = reinterpret_cast<float*>(sm + L::FILT + fb * 2 * L::WB);
    stage_filter_rt<kRagThreads>(f, wc, K, false);
    stage_filter_rt<kRagThreads>(f + L::WB / 4, wc, K, true);
  }
}

// Chunk c has written its outputs and partials.  The CTA that completes the
// last chunk of an (image, channel) sums its filter gradient and, for the
// clamp border, folds the edges of dx.  It runs once per chunk, outside the
// filter sizes' bodies (K known at run time): inlined into each of them the
// sums cost the tile loops registers (seven K = 11 images 2.82 -> 2.91 ms).
// `im` is the copy in shared memory that the chunk's start left there: the fence
// empties L1, and two loads in a row from L2 are felt where a chunk is a small
// image.
template <typename T>
__device__ __forceinline__ void rag_complete(const RagParams& p, int channel, const RagImage& im,
                                             double* ps, int* s_flag) {
  const bool do_dw = p.ops & 4, folds = (p.ops & 2) && p.border == 1;
  if (do_dw || folds) {
    __threadfence();  // this thread's outputs and partials, before the count
    cta_barrier();
    if (threadIdx.x == 0)
      *s_flag = atomicAdd(p.counters + 1 + im.ic_base + channel, 1) == im.nch - 1;
    cta_barrier();
    if (*s_flag) {
      __threadfence();
      const int K = im.K, KK = K * K;
      if (do_dw) {
        // every tap's partials in FP64 by GR threads, each every GR-th chunk,
        // then their sums in order
        const float* part = p.partials + im.partial_base + (int64_t)channel * im.nch * KK;
        const int GR = min(min(kRagThreads / KK, 16), im.nch);
        const int k = threadIdx.x % KK, q = threadIdx.x / KK;
        if (q < GR) {
          double s = 0.0;
#pragma unroll 8
          for (int j = q; j < im.nch; j += GR) s += (double)__ldcg(part + (int64_t)j * KK + k);
          ps[q * KK + k] = s;
        }
        cta_barrier();
        if (threadIdx.x < KK) {
          double s = 0.0;
          for (int g = 0; g < GR; ++g) s += ps[g * KK + threadIdx.x];
          im.dw[(int64_t)channel * KK + threadIdx.x] = (float)s;
        }
      }
      if (folds) {
        const int64_t off = (int64_t)channel * im.H * im.W;
        const int64_t edges = edge_pixels(im.H, im.W);
        for (int64_t e = threadIdx.x; e < edges; e += kRagThreads)
          fold_edge_pixel<T>(static_cast<const T*>(im.dy) + off, im.w + (int64_t)channel * KK,
                             static_cast<T*>(im.dx) + off, im.H, im.W, K, e);
      }
    }
  }
  cta_barrier();  // sm_red and s_flag are reused by the next chunk
}

// One chunk: its first tile is already in stage sb (copies in flight), its
// filters in filter buffer fb.  While tile t is computed, the copies of the
// next tile -- the next of this chunk, or the first of chunk `cn` -- go to
// the other stage.  Returns the stage holding the next chunk's first tile.
template <typename T, int K>
__device__ __forceinline__ int rag_chunk(const RagParams& p, const RagChunk& ch,
                                         const RagImage& im, int cn, char* sm, int sb, int fb) {
  using G = Geo<K, sizeof(T), true>;
  using S = RagShape<K, T>;
  using L = RagLayout<T>;
  constexpr int KK = K * K;
  float* sm_red = reinterpret_cast<float*>(sm + L::RED);
  const float* sm_w = reinterpret_cast<const float*>(sm + L::FILT + fb * 2 * L::WB);
  const float* sm_wf = sm_w + L::WB / 4;

  const int H = im.H, W = im.W;
  const int tiles_x = (W + kTileW - 1) / kTileW;
  const int64_t off = (int64_t)ch.channel * H * W;
  const bool do_fwd = p.ops & 1, do_dx = p.ops & 2, do_dw = p.ops & 4;
  const bool clamp = p.border == 1, vec = im.vec != 0;
  T* yp = do_fwd ? static_cast<T*>(im.y) + off : nullptr;
  T* dxp = do_dx ? static_cast<T*>(im.dx) + off : nullptr;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = warp % S::GT;
  const int part = warp / S::GT;
  const int a_lo = group_lo(g, K, S::GT);
  const int nrows = group_lo(g + 1, K, S::GT) - a_lo;
  float acc[S::AT][K];
#pragma unroll
  for (int s = 0; s < S::AT; ++s)
#pragma unroll
    for (int b = 0; b < K; ++b) acc[s][b] = 0.f;

  for (int t = ch.tile_begin; t < ch.tile_end; ++t) {
    if (t + 1 < ch.tile_end) {
      rag_stage<T>(p, ch, im, t + 1, sm, sb ^ 1, fb, false);
    } else if (cn < p.n_chunks) {
      const RagChunk chn = p.chunks[cn];
      const RagImage imn = p.images[chn.image];
      rag_stage<T>(p, chn, imn, chn.tile_begin, sm, sb ^ 1, fb ^ 1, true);
    }
    cp_async_commit();
    cp_async_wait_group<1>();  // this tile's copies (committed one tile earlier) have landed
    T* sx = reinterpret_cast<T*>(sm + sb * L::STAGE);
    T* sdy = reinterpret_cast<T*>(sm + sb * L::STAGE + L::TILE);
    const int ty0 = (t / tiles_x) * kBwdTileH, tx0 = (t % tiles_x) * kTileW;
    if (im.odd_rows) {
      if (do_fwd || do_dw)
        shift_odd_rows<T, kRagThreads>(sx, static_cast<const T*>(im.x) + off, H, W, ty0, S::ROWS,
                                       G::R, G::RP, G::SP);
      if (do_dx || do_dw)
        shift_odd_rows<T, kRagThreads>(sdy, static_cast<const T*>(im.dy) + off, H, W, ty0,
                                       S::ROWS, G::R, G::RP, G::SP, !(do_fwd || do_dw));
    }
    cta_barrier();
    if (clamp && (do_fwd || do_dw) &&
        (ty0 - G::R < 0 || ty0 + kBwdTileH + G::R > H || tx0 - G::RP < 0 ||
         tx0 + kTileW + G::RP > W))
      clamp_fix<T, G::SP, kRagThreads>(sx, H, W, ty0, tx0, G::R, G::RP, S::ROWS);
    const int r8 = (warp & 7) * 8;
    if ((warp < 8 ? do_fwd : do_dx) && ty0 + r8 < H) {
      const T* src = warp < 8 ? sx : sdy;
      const float* f = warp < 8 ? sm_w : sm_wf;
      T* dst = warp < 8 ? yp : dxp;
      float o[8][4];
      fwd_block<K, 8, T, true>(src + r8 * G::SP + 4 * lane, f, o);
      store_tile<T, 8, kAnyPlanes>(dst, H, W, ty0 + r8, tx0, vec,
                              reinterpret_cast<float*>(sm + L::BUF + warp * kRowBuf), o);
    }
    if (do_dw) {
      const int r0 = part * S::DW_ROWS;  // dy rows below the image are zero: skipped
      const int nb = min(S::DW_ROWS / S::DR, (H - ty0 - r0 + S::DR - 1) / S::DR);
      dw_rows<K, S::AT, S::GT, G::SP, S::DR, T, true>(
          sdy + (r0 + G::R) * G::SP + G::RP + 4 * lane, sx + (r0 + a_lo) * G::SP + 4 * lane, nb,
          nrows, acc);
    }
    cta_barrier();  // stage sb is free for the copies two tiles ahead
    sb ^= 1;
  }

  // filter-gradient partial of this chunk: warp butterflies, then a fixed-order
  // sum over the group's warps
  if (do_dw) {
#pragma unroll
    for (int s = 0; s < S::AT; ++s)
#pragma unroll
      for (int b = 0; b < K; ++b) {
        float v = acc[s][b];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) sm_red[warp * L::RED_FLOATS + s * K + b] = v;
      }
  }
  cta_barrier();
  float* part_c = p.partials + im.partial_base + (int64_t)ch.channel * im.nch * KK;
  if (do_dw) {
    const int j = ch.tile_begin / p.tpc;
    for (int k = threadIdx.x; k < KK; k += kRagThreads) {
      const int a = k / K, b = k - (k / K) * K;
      int gg = 0;
      while (gg + 1 < S::GT && group_lo(gg + 1, K, S::GT) <= a) ++gg;
      const int s = a - group_lo(gg, K, S::GT);
      float sum = 0.f;
      for (int q = 0; q < S::WPG; ++q) sum += sm_red[(q * S::GT + gg) * L::RED_FLOATS + s * K + b];
      part_c[(int64_t)j * KK + k] = sum;
    }
  }
  return sb;
}

template <typename T>
__global__ void __launch_bounds__(kRagThreads, 1) rag_kernel(RagParams p) {
  extern __shared__ __align__(128) float smem[];
  using L = RagLayout<T>;
  char* sm = reinterpret_cast<char*>(smem);
  volatile int* s_next = reinterpret_cast<volatile int*>(sm + L::INTS);
  int* s_flag = reinterpret_cast<int*>(sm + L::INTS + 4);
  if (threadIdx.x == 0) *s_next = atomicAdd(p.counters, 1);
  cta_barrier();
  int c = *s_next;
  if (c >= p.n_chunks) return;
  int sb = 0, fb = 0;
  {
    const RagChunk ch = p.chunks[c];
    const RagImage im = p.images[ch.image];
    rag_stage<T>(p, ch, im, ch.tile_begin, sm, sb, fb, true);
    cp_async_commit();
  }
  for (;;) {
    cta_barrier();  // every thread has read the previous *s_next
    if (threadIdx.x == 0) *s_next = atomicAdd(p.counters, 1);  // one chunk ahead
    cta_barrier();
    const int cn = *s_next;
    const RagChunk ch = p.chunks[c];
    const RagImage im = p.images[ch.image];
    RagImage* s_im = reinterpret_cast<RagImage*>(sm + L::IMAGE);
    if (threadIdx.x == 0) *s_im = im;  // read behind rag_chunk's barriers
    switch (im.K) {
      case 1: sb = rag_chunk<T, 1>(p, ch, im, cn, sm, sb, fb); break;
      case 3: sb = rag_chunk<T, 3>(p, ch, im, cn, sm, sb, fb); break;
      case 5: sb = rag_chunk<T, 5>(p, ch, im, cn, sm, sb, fb); break;
      case 7: sb = rag_chunk<T, 7>(p, ch, im, cn, sm, sb, fb); break;
      case 9: sb = rag_chunk<T, 9>(p, ch, im, cn, sm, sb, fb); break;
      case 11: sb = rag_chunk<T, 11>(p, ch, im, cn, sm, sb, fb); break;
      case 13: sb = rag_chunk<T, 13>(p, ch, im, cn, sm, sb, fb); break;
      default: sb = rag_chunk<T, 15>(p, ch, im, cn, sm, sb, fb); break;
    }
    rag_complete<T>(p, ch.channel, *s_im, reinterpret_cast<double*>(sm + L::RED), s_flag);
    if (cn >= p.n_chunks) break;
    c = cn;
    fb ^= 1;
  }
  cp_async_wait_group<0>();
}

cudaError_t rag_launch_f32(const RagParams& p, int grid, size_t smem, cudaStream_t st);
cudaError_t rag_launch_bf16(const RagParams& p, int grid, size_t smem, cudaStream_t st);

}  // namespace giga
