// dw_misc.cu -- what follows the tile kernels of the depthwise backward pass:
//  * the clamp-border edge fold of the input gradient, and
//  * the fixed-order FP64 reduction of the per-CTA filter-gradient partials,
// in one launch (dw_finish_kernel).
#include <algorithm>
#include <cstring>

#include "dw_fold.cuh"
#include "dw_kernels.cuh"
#include "dw_launch.h"
#include "tma.cuh"

namespace giga {

// Device error word of the depthwise kernels (bounded TMA waits).
static __device__ int g_dw_err;

int* dw_error_word() {
  static int* cached[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  if (!cached[dev]) {
    int* p = nullptr;
    if (cudaGetSymbolAddress(reinterpret_cast<void**>(&p), g_dw_err) != cudaSuccess) return nullptr;
    cached[dev] = p;
  }
  return cached[dev];
}

cudaError_t dw_take_error(cudaStream_t st, int* code) {
  *code = 0;
  cudaError_t e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return e;
  int* err = dw_error_word();
  if (!err) return cudaErrorInvalidSymbol;
  e = cudaMemcpy(code, err, sizeof(int), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return e;
  const int zero = 0;
  return cudaMemcpy(err, &zero, sizeof(int), cudaMemcpyHostToDevice);
}

// One thread waits on an mbarrier that nothing ever completes: the bounded
// wait gives up after kWaitLimitNs and records kDevErrTimeout, exercising the
// same path a stalled TMA load would take.
__global__ void dw_wait_selftest_kernel(int* err) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x != 0) return;
  mbar_init(&bar, 1);
  mbar_init_fence();
  if (!mbar_wait(&bar, 0)) record_error(err, kDevErrTimeout);
}

cudaError_t dw_wait_selftest(cudaStream_t st) {
  int* err = dw_error_word();
  if (!err) return cudaErrorInvalidSymbol;
  dw_wait_selftest_kernel<<<1, 32, 0, st>>>(err);
  note_launch();
  return cudaGetLastError();
}

int64_t dw_bwd_chunks_per_plane(int64_t H, int64_t W, int tiles_per_cta) {
  const int64_t tiles = ((W + kTileW - 1) / kTileW) * ((H + kBwdTileH - 1) / kBwdTileH);
  return (tiles + tiles_per_cta - 1) / tiles_per_cta;
}

// ------------------------------------------------------------- edge fold
// BF16 planes one pixel high or wide, and very many very small ones
// (fold_by_pixel): every edge pixel recomputed from the definition.
template <typename T>
__global__ void dw_fixup_kernel(const T* __restrict__ dy, const float* __restrict__ w,
                                T* __restrict__ dx, int C, int H, int W, int K,
                                int64_t edge_per_plane, int64_t total) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t plane = e / edge_per_plane;
    const int64_t k = e - plane * edge_per_plane;
    fold_edge_pixel<T>(dy + plane * (int64_t)H * W, w + (int64_t)(plane % C) * K * K,
                       dx + plane * (int64_t)H * W, H, W, K, k);
  }
}

// ---- FP32 clamp fold as corrections on top of the zero-border values g that
// the tile pass already wrote.  With g[u][v] = sum_{a,b} w[a][b] dy[u-a+r][v-b+r]
// (dy zero outside) on the extended domain, the clamp adjoint is
// dx[p][q] = sum_{u: B(u)=p} sum_{v: B(v)=q} g[u][v], i.e. g plus the margin sums
//   top     T[q] = sum_{i<r}  sum_b Wt[i][b] dy[i][q-b+r],     Wt[i][b] = sum_{a<=r-1-i} w[a][b]
//   bottom  B[q] = sum_{d<r}  sum_b Wb[d][b] dy[H-1-d][q-b+r], Wb[d][b] = sum_{a>=r+1+d} w[a][b]
//   left    L[p] = sum_{j<r}  sum_a Wl[j][a] dy[p-a+r][j],     Wl[j][a] = sum_{b<=r-1-j} w[a][b]
//   right   R[p] = sum_{e<r}  sum_a Wr[e][a] dy[p-a+r][W-1-e], Wr[e][a] = sum_{b>=r+1+e} w[a][b]
// and at the corners the doubly-folded sums, e.g.
//   TL = sum_{i<r,j<r} (sum_{a<=r-1-i} sum_{b<=r-1-j} w[a][b]) dy[i][j]
// (i, d < H and j, e < W; dy outside the image reads zero).  BF16 results are
// rounded to storage already, so there the edge pixels are recomputed whole by
// the same sums with the taps that read the edge itself included.

// ------------------------------------------------- fold and reduction
// One launch with three kinds of blocks of NT threads (what a call does not need
// has none): the filter gradient's sums, the fold of NT / 2 pixels of the
// first and last row or column of a plane, and the fold of a plane's corner
// pixels, which both folds touch.  All are short and bound by latency, so they
// run beside each other instead of one after the other.  As launches of their
// own -> one launch with FP64 sums (this one profiled, with cold caches), us:
// 4 x 3 x 1801 x 2399, K = 3 24.9 (rows 4.4, columns 6.7, sums 13.8) -> 8.4;
// 8 x 3 x 1024^2, K = 15 52 -> 14.6; BF16 K = 9, 4 x 3 x 1800 x 2400 60 (a fold pixel
// by pixel 45 of it) -> 12.3; 4 x 3 x 257 x 251, K = 3 10.5 -> 7.6.
//
// NT is 512, or 128 (finish_small) where the planes' edges or the partial sums
// are so few that most of 512 threads would idle.
constexpr int kFinishThreads = 512, kFinishThreadsSmall = 128;

struct FinishArgs {
  const float* partials;  // filter gradient: [N * C * chunks][KK]
  float* dw;
  int N, C, KK;
  int taps, groups;  // taps per block, such groups of a filter
  int sum_blocks;   // C * groups, or 0
  FastDiv chunks;   // per plane
  const void* dy;  // fold
  const float* w;
  void* dx;
  int H, W, K;
  int row_blocks, col_blocks;  // per plane; plus one corner block
  int64_t plane0;   // first plane of this launch
};

// dw[c][k] = sum over the partial rows (image n, chunk ch) of channel c in a
// fixed order, all in FP64: a block takes p.taps taps of one channel, a thread
// every (NT / p.taps)-th row of one tap, eight loads in flight; then a butterfly
// within the warp and the warps in order.  FP64 adds and conversions run at
// about two a clock on an SM, so the taps are spread over as many blocks as fill
// the GPU (finish_taps) rather than read by few in whole sectors (4 x 3 x 1801 x
// 2399, K = 3, with the fold: 22 us with 32 taps per block, 6 us with one).
template <int NT>
__device__ __forceinline__ void finish_sums(const FinishArgs& p, double* red) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c = (int)blockIdx.x / p.groups, g = (int)blockIdx.x - c * p.groups;
  const int TB = p.taps;  // a power of two, at most 32
  const int tap = TB * g + (threadIdx.x & (TB - 1));
  const int slots = NT / TB;
  const uint32_t chunks = p.chunks.d;
  const uint32_t count = (uint32_t)p.N * chunks;
  double s = 0.0;
  if (tap < p.KK) {
    constexpr int U = 8;
    for (uint32_t i0 = threadIdx.x / TB; i0 < count; i0 += U * slots) {
      float v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint32_t i = i0 + u * slots;
        v[u] = 0.f;
        if (i < count) {
          const uint32_t n = fdiv(i, p.chunks), ch = i - n * chunks;
          v[u] = __ldg(p.partials + (((int64_t)n * p.C + c) * chunks + ch) * p.KK + tap);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (i0 + u * slots < count) s += (double)v[u];
    }
  }
  for (int o = 16; o >= TB; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane < TB) red[warp * TB + lane] = s;
  __syncthreads();
  if ((int)threadIdx.x < TB && tap < p.KK) {
    double sum = 0.0;
    // warps beyond the last row have nothing
    const int warps = min(NT / 32, ((int)min(count, (uint32_t)NT) * TB + 31) / 32);
    for (int w = 0; w < warps; ++w) sum += red[w * TB + threadIdx.x];
    p.dw[(int64_t)c * p.KK + tap] = (float)sum;
  }
}

// Taps per block: the fewest (a power of two) for which the blocks of all
// channels fit the GPU about twice over.
static int finish_taps(int64_t C, int KK) {
  int taps = 1;
  while (taps < 32 && C * ((KK + taps - 1) / taps) > 2 * (int64_t)sm_count()) taps *= 2;
  return taps;
}

__device__ __forceinline__ float dy_at(const float* g, int H, int W, int i, int j) {
  return (i >= 0 && i < H && j >= 0 && j < W) ? __ldg(g + (int64_t)i * W + j) : 0.f;
}

// Rows (columns) of dy an edge pixel's sum takes, counted from the edge, and
// the filter rows (columns) a = lo .. hi whose weights are summed for the i-th:
// FP32 adds the margin sums to the stored g, so row i < r takes the taps that
// reach outside; BF16 recomputes the whole value (one rounding), so the tap
// that reads the edge itself joins them, and row r.
template <typename T>
__device__ __forceinline__ int fold_depth(int r) { return sizeof(T) == 4 ? r : r + 1; }
template <typename T>
__device__ __forceinline__ float fold_weight(const float* f, int step, int K, int e, int i) {
  const int r = (K - 1) / 2, full = sizeof(T) == 4 ? 0 : 1;
  const int lo = e ? r + 1 + i - full : 0, hi = e ? K - 1 : r - 1 - i + full;
  float t = 0.f;
  for (int a = lo; a <= hi; ++a) t += f[a * step];
  return t;
}

// Pixels NT / 2 * blk .. of the first and last row (rows = true: sums T and B
// above, one half of the block each) or column (L and R) of a plane; its
// corner pixels are left to finish_corners.
template <typename T, int NT>
__device__ __forceinline__ void finish_edges(const FinishArgs& p, int64_t plane, int blk, bool rows,
                                             float* tab) {
  const int K = p.K, r = (K - 1) / 2, H = p.H, W = p.W, D = fold_depth<T>(r);
  constexpr int P = NT / 2;
  const int lim = rows ? W : H;    // length of the edge
  const int other = rows ? H : W;  // rows (columns) across it
  const float* f = p.w + (plane % p.C) * (int64_t)K * K;
  float* sf = tab;                // the filter
  float* wt = sf + K * K;         // [2][D][K] summed weights: first edge, last edge
  float* strip = wt + 2 * D * K;  // [2][D][SW] of dy
  const T* g = static_cast<const T*>(p.dy) + plane * (int64_t)H * W;
  const int q0 = blk * P, n = min(D, other);
  const int SW = min(P, lim - q0) + 2 * r;  // the pixels of this block and their margins
  const int e = threadIdx.x / P, t = threadIdx.x - e * P;
  const int q = q0 + t, in = e ? other - 1 : 0;
  const bool mine = q > 0 && q < lim - 1 && !(e == 1 && other == 1);
  T* d = static_cast<T*>(p.dx) + plane * (int64_t)H * W +
         (rows ? (int64_t)in * W + q : (int64_t)q * W + in);
  float s = 0.f, old = 0.f;
  if constexpr (sizeof(T) == 4)
    if (mine) old = *d;  // on its way while the strip arrives
  for (int k = threadIdx.x; k < K * K; k += NT) sf[k] = __ldg(f + k);
  // strip[k = e D + i][c]: i rows (columns) in from edge e, at position q0 - r + c.
  // Consecutive lanes run along the row (rows), or over the 2 D columns of one
  // position, a power of two of lanes for them: no index is divided.
  const int cl = rows ? 0 : 32 - __clz(2 * D - 1);  // log2 of the lanes per position
  const int c0 = rows ? threadIdx.x & 31 : threadIdx.x >> cl, cs = rows ? 32 : NT >> cl;
  const int k0 = rows ? threadIdx.x >> 5 : threadIdx.x & ((1 << cl) - 1);
  for (int k = k0; k < 2 * D; k += rows ? NT / 32 : 32) {
    const int es = k >= D, i = k - es * D, from = es ? other - 1 - i : i;
    for (int c = c0; c < SW; c += cs) {
      const int at = q0 - r + c;
      float v = 0.f;
      if (i < n && at >= 0 && at < lim)
        v = Elem<T>::load(g + (rows ? (int64_t)from * W + at : (int64_t)at * W + from));
      strip[k * SW + c] = v;
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < 2 * D * K; k += NT) {
    const int ew = k / (D * K), i = k / K - ew * D, b = k - (k / K) * K;
    wt[k] = rows ? fold_weight<T>(sf + b, K, K, ew, i) : fold_weight<T>(sf + b * K, 1, K, ew, i);
  }
  __syncthreads();
  if (q < lim)
    for (int i = 0; i < n; ++i)
      for (int b = 0; b < K; ++b)
        s = fmaf(wt[(e * D + i) * K + b], strip[(e * D + i) * SW + t + 2 * r - b], s);
  if (other == 1) {  // a single row (column) is both edges: the first half adds both sums
    __syncthreads();
    if (e == 1 && q < lim) strip[t] = s;
    __syncthreads();
    if (q < lim) s += strip[t];
  }
  if (mine) Elem<T>::store(d, old + s);
}

// BF16: the four corner pixels of a plane with H, W >= 2, recomputed:
// dx = sum_{i,j <= r} C[i][j] dy[i][j], rows and columns counted from the
// corner, C[i][j] = the sum of the taps that bring (i, j) there.
template <int NT>
__device__ __forceinline__ void finish_corners_bf16(const FinishArgs& p, int64_t plane,
                                                    float* tab) {
  const int K = p.K, r = (K - 1) / 2, H = p.H, W = p.W, D = r + 1;
  const float* f = p.w + (plane % p.C) * (int64_t)K * K;
  const __nv_bfloat16* g = static_cast<const __nv_bfloat16*>(p.dy) + plane * (int64_t)H * W;
  float* wc = tab;               // [2][D][K]: a column edge's weights of filter row a
  float* prod = wc + 2 * D * K;  // [4][D][D]
  for (int k = threadIdx.x; k < 2 * D * K; k += NT) {
    const int e = k / (D * K), j = k / K - e * D, a = k - (k / K) * K;
    wc[k] = fold_weight<__nv_bfloat16>(f + a * K, 1, K, e, j);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < 4 * D * D; k += NT) {
    const int q = k / (D * D), i = k / D - q * D, j = k - (k / D) * D;
    const int er = q >> 1, ec = q & 1;
    const float c = fold_weight<__nv_bfloat16>(wc + (ec * D + j) * K, 1, K, er, i);
    const int row = er ? H - 1 - i : i, col = ec ? W - 1 - j : j;
    const bool ok = row >= 0 && row < H && col >= 0 && col < W;
    prod[k] = ok ? c * Elem<__nv_bfloat16>::load(g + (int64_t)row * W + col) : 0.f;
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    const int er = threadIdx.x >> 1, ec = threadIdx.x & 1;
    float s = 0.f;
    for (int k = 0; k < D * D; ++k) s += prod[threadIdx.x * D * D + k];
    Elem<__nv_bfloat16>::store(static_cast<__nv_bfloat16*>(p.dx) + plane * (int64_t)H * W +
                                   (er ? (int64_t)(H - 1) * W : 0) + (ec ? W - 1 : 0),
                               s);
  }
}

// The corner pixels of a plane (one, two or four): the row sums, then the
// column sums with the doubly folded corner terms.
template <int NT>
__device__ __forceinline__ void finish_corners(const FinishArgs& p, int64_t plane, float* tab) {
  const int K = p.K, r = (K - 1) / 2, H = p.H, W = p.W;
  const float* f = p.w + (plane % p.C) * (int64_t)K * K;
  float* sf = tab;
  float* wr = sf + K * K;       // [2][r][K]: Wt, Wb
  float* wc = wr + 2 * r * K;   // [2][r][K]: Wl, Wr
  float* cw = wc + 2 * r * K;   // [2][2][r][r]: corner weights (row edge, column edge)
  float* sq = cw + 4 * r * r;   // [2][2][r + 1][r + 1]: dy counted from the corners
  float* sums = sq + 4 * (r + 1) * (r + 1);  // [8]
  const int S = r + 1;
  const float* g = static_cast<const float*>(p.dy) + plane * (int64_t)H * W;
  for (int k = threadIdx.x; k < K * K; k += NT) sf[k] = __ldg(f + k);
  for (int k = threadIdx.x; k < 4 * S * S; k += NT) {
    const int q = k / (S * S), i = k / S - q * S, j = k - (k / S) * S;
    const int row = (q >> 1) ? H - 1 - i : i, col = (q & 1) ? W - 1 - j : j;
    sq[k] = dy_at(g, H, W, row, col);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < 4 * r * K; k += NT) {
    const int rows = k < 2 * r * K, kk = rows ? k : k - 2 * r * K;
    const int e = kk / (r * K), i = kk / K - e * r, b = kk - (kk / K) * K;
    float t = 0.f;
    const int lo = e ? r + 1 + i : 0, hi = e ? K - 1 : r - 1 - i;
    for (int a = lo; a <= hi; ++a) t += rows ? sf[a * K + b] : sf[b * K + a];
    (rows ? wr : wc)[kk] = t;
  }
  __syncthreads();
  for (int k = threadIdx.x; k < 4 * r * r; k += NT) {
    const int q = k / (r * r), i = k / r - q * r, j = k - (k / r) * r;
    const int er = q >> 1, ec = q & 1;
    const int lo = er ? r + 1 + i : 0, hi = er ? K - 1 : r - 1 - i;
    float t = 0.f;
    for (int a = lo; a <= hi; ++a) t += wc[(ec * r + j) * K + a];
    cw[k] = t;
  }
  __syncthreads();
  const int nr = min(r, H), nc = min(r, W);
  if (threadIdx.x < 8) {
    // t = 0..3: sum of row edge er at column edge ec; 4..7: of column edge ec
    // at row edge er (with the corner terms)
    const int t = threadIdx.x, er = (t >> 1) & 1, ec = t & 1;
    const float* s0 = sq + (er * 2 + ec) * S * S;
    float s = 0.f;
    if (t < 4) {
      for (int i = 0; i < nr; ++i)
        for (int b = 0; b < K; ++b) {
          const int j = ec ? b - r : r - b;  // columns in from that edge
          s = fmaf(wr[(er * r + i) * K + b], j >= 0 ? s0[i * S + j] : 0.f, s);
        }
    } else {
      for (int j = 0; j < nc; ++j)
        for (int a = 0; a < K; ++a) {
          const int i = er ? a - r : r - a;
          s = fmaf(wc[(ec * r + j) * K + a], i >= 0 ? s0[i * S + j] : 0.f, s);
        }
      for (int i = 0; i < nr; ++i)
        for (int j = 0; j < nc; ++j)
          for (int q = 0; q < 2; ++q)  // a single row is both row edges
            if (q == er || H == 1)
              s = fmaf(cw[((q * 2 + ec) * r + i) * r + j], sq[((q * 2 + ec) * S + i) * S + j], s);
    }
    sums[t] = s;
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    const int er = threadIdx.x >> 1, ec = threadIdx.x & 1;
    if ((er && H == 1) || (ec && W == 1)) return;
    float* d = static_cast<float*>(p.dx) + plane * (int64_t)H * W +
               (er ? (int64_t)(H - 1) * W : 0) + (ec ? W - 1 : 0);
    float v = *d;
    v += H == 1 ? sums[ec] + sums[2 + ec] : sums[er * 2 + ec];
    v += W == 1 ? sums[4 + er * 2] + sums[4 + er * 2 + 1] : sums[4 + er * 2 + ec];
    *d = v;
  }
}

template <typename T, int NT>
__global__ void __launch_bounds__(NT, 1536 / NT) dw_finish_kernel(const FinishArgs p) {
  extern __shared__ __align__(16) float fin_smem[];
  if ((int)blockIdx.x < p.sum_blocks) {
    finish_sums<NT>(p, reinterpret_cast<double*>(fin_smem));
    return;
  }
  const uint32_t b = blockIdx.x - p.sum_blocks;
  const uint32_t per = p.row_blocks + p.col_blocks + 1;
  const int64_t plane = p.plane0 + b / per;
  const int k = (int)(b - b / per * per);
  if (k < p.row_blocks)
    finish_edges<T, NT>(p, plane, k, true, fin_smem);
  else if (k < p.row_blocks + p.col_blocks)
    finish_edges<T, NT>(p, plane, k - p.row_blocks, false, fin_smem);
  else if constexpr (sizeof(T) == 2)
    finish_corners_bf16<NT>(p, plane, fin_smem);
  else
    finish_corners<NT>(p, plane, fin_smem);
}

// Blocks of 128 threads: where the planes' edges fit two of their fold blocks, or
// without a fold where 1024 partial sums (eight per thread) are all a block adds.
static bool finish_small(const DwArgs& a, bool folds, int64_t rows, int taps) {
  return folds ? std::max(a.H, a.W) <= 128 : rows * taps <= 1024;
}

template <int NT>
static void finish_run(const DwArgs& a, const FinishArgs& p, unsigned blocks, size_t smem,
                       cudaStream_t st) {
  if (a.dtype == 0)
    dw_finish_kernel<float, NT><<<blocks, NT, smem, st>>>(p);
  else
    dw_finish_kernel<__nv_bfloat16, NT><<<blocks, NT, smem, st>>>(p);
}

// BF16 planes one pixel high or wide, where an edge pixel lies on both edges;
// and more planes than their fold blocks run at once (12 of 128 threads per SM,
// three per plane) with so few taps at their edges that a thread per edge pixel
// does less than a block spends on its tables: at most 800 per plane, from 4 x S
// planes on (4096 planes, thread per pixel against blocks, us: 7 x 7 K = 3 6 / 17,
// K = 5 15 / 19; 14 x 14 K = 3 9 / 17, K = 5 23 / 19).
static bool fold_by_pixel(const DwArgs& a) {
  return a.H == 1 || a.W == 1 ||
         (a.N * a.C >= 4 * (int64_t)sm_count() && edge_pixels(a.H, a.W) * a.K * a.K <= 800);
}

cudaError_t dw_finish_launch(const DwArgs& a, bool fold, int64_t chunks_per_plane,
                             cudaStream_t st) {
  const int r = (a.K - 1) / 2;
  const bool folds = fold && a.border == 1 && r > 0 && a.N * a.C * a.H * a.W > 0;
  const bool by_pixel = folds && a.dtype != 0 && fold_by_pixel(a);
  if (by_pixel) {
    const int64_t edge = edge_pixels(a.H, a.W);
    const int64_t total = a.N * a.C * edge;
    const int threads = 128;
    const int64_t blocks = std::min<int64_t>((total + threads - 1) / threads, 65535);
    dw_fixup_kernel<__nv_bfloat16><<<(unsigned)blocks, threads, 0, st>>>(
        static_cast<const __nv_bfloat16*>(a.dy), a.w, static_cast<__nv_bfloat16*>(a.dx),
        (int)a.C, (int)a.H, (int)a.W, a.K, edge, total);
    note_launch();
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  FinishArgs p;
  std::memset(&p, 0, sizeof(p));
  p.N = (int)a.N;
  p.C = (int)a.C;
  p.chunks = make_fastdiv(1);
  size_t smem = 0;
  int64_t blocks = 0, planes = 0, per = 0;
  const bool edges_too = folds && !by_pixel;
  const int taps = chunks_per_plane > 0 ? finish_taps(a.C, a.K * a.K) : 1;
  const bool small = finish_small(a, edges_too, a.N * chunks_per_plane, taps);
  const int nt = small ? kFinishThreadsSmall : kFinishThreads, P = nt / 2;
  if (chunks_per_plane > 0) {
    if (a.N * chunks_per_plane >= (1LL << 31)) return cudaErrorInvalidConfiguration;
    p.partials = a.partials;
    p.dw = a.dw;
    p.KK = a.K * a.K;
    p.taps = taps;
    p.groups = (p.KK + p.taps - 1) / p.taps;
    p.chunks = make_fastdiv((uint32_t)chunks_per_plane);
    blocks = a.C * p.groups;
    if (blocks >= (1LL << 31)) return cudaErrorInvalidConfiguration;
    p.sum_blocks = (int)blocks;
    smem = nt * sizeof(double);
  }
  if (edges_too) {
    p.dy = a.dy;
    p.w = a.w;
    p.dx = a.dx;
    p.H = (int)a.H;
    p.W = (int)a.W;
    p.K = a.K;
    p.row_blocks = (int)((a.W + P - 1) / P);
    p.col_blocks = (int)((a.H + P - 1) / P);
    planes = a.N * a.C;
    per = (int64_t)p.row_blocks + p.col_blocks + 1;
    const int D = a.dtype == 0 ? r : r + 1;  // fold_depth
    const size_t edges = a.K * a.K + 2 * D * a.K + 2 * D * (P + 2 * r);
    const size_t corners = a.K * a.K + 4 * D * a.K + 4 * r * r + 4 * (r + 1) * (r + 1) + 8;
    smem = std::max(smem, std::max(edges, corners) * sizeof(float));
  }
  // one launch, unless the planes' fold blocks exceed a grid
  do {
    const int64_t now = per ? std::min<int64_t>(planes - p.plane0, (0x7fffffffLL - blocks) / per) : 0;
    blocks += now * per;
    if (blocks == 0) return cudaSuccess;
    if (small)
      finish_run<kFinishThreadsSmall>(a, p, (unsigned)blocks, smem, st);
    else
      finish_run<kFinishThreads>(a, p, (unsigned)blocks, smem, st);
    note_launch();
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    p.plane0 += now;
    p.sum_blocks = 0;
    blocks = 0;
  } while (p.plane0 < planes);
  return cudaSuccess;
}

}  // namespace giga
