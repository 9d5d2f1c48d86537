// autotune.cu -- picks the launch configuration of the depthwise kernels per
// problem class by timing every candidate with CUDA events, and keeps the
// choices in memory and (optionally) in a JSON file.
//
// Candidates:
//   forward / input gradient: output rows per thread 8 (64 x 128 tiles) or
//                             4 (32 x 128 tiles: twice the CTAs, less halo reuse)
//                             x one tile per CTA or persistent CTAs x with or
//                             without an L2 prefetch of a later tile;
//   filter gradient (alone or fused): tiles per CTA = automatic, 2, 4, 8, 16
//                             (fewer partial sums vs. better load balance).
// Problem class: (op, dtype, K, border, floor(log2(N*C*H*W)), planes aligned or
// not -- they run separately compiled kernels).  A choice pinned for a
// description, or in a cache without the alignment, holds for both.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <fstream>
#include <map>
#include <mutex>
#include <sstream>
#include <string>

#include "dw_launch.h"
#include "internal.h"

namespace giga {

static std::mutex g_mu;
static std::map<std::string, int> g_cache;
static int g_mode = -1;
static bool g_loaded = false;

static int env_mode() {
  const char* e = std::getenv("GIGA_AUTOTUNE");
  if (!e) return 1;
  if (!std::strcmp(e, "off") || !std::strcmp(e, "0")) return 0;
  if (!std::strcmp(e, "full") || !std::strcmp(e, "2")) return 2;
  return 1;
}

int tune_mode() {
  std::lock_guard<std::mutex> lk(g_mu);
  if (g_mode < 0) g_mode = env_mode();
  return g_mode;
}

// Forward / input gradient: {8, 4} rows per thread x {one tile per CTA,
// persistent} x {no prefetch, L2 prefetch}; filter gradient: tiles per chunk {auto, 2, 4, 8, 16}; fused
// backward: the fused kernel with tiles per CTA {auto, 2, 4, 8, 16}, the
// two-pass split, or the persistent kernel with a tile ring (three stages where
// they fit, else two).
int tune_candidates(int op) {
  switch (op) {
    case TUNE_FWD:
    case TUNE_BWD_INPUT: return 8;
    case TUNE_BWD_FILTER: return 5;
    default: return 7;
  }
}


static int auto_tiles_per_cta(const DwArgs& a) {
  const int64_t tiles = a.N * a.C * (int64_t)((a.W + kTileW - 1) / kTileW) *
                        (int64_t)((a.H + 63) / 64);
  int64_t t = tiles / ((int64_t)sm_count() * 16);
  if (t < 1) t = 1;
  if (t > 16) t = 16;
  return (int)t;
}

// The persistent filter kernel runs one CTA per SM over chunks dealt round
// robin; a chunk ends with a reduction of the accumulators costing about a
// fifth of a tile.  Pick the chunk length (<= 16 tiles) minimising the
// busiest CTA's rounds x (tiles + 0.2), of at most max_tiles.
static int auto_filter_tiles_per_chunk(const DwArgs& a, int max_tiles = 16) {
  const int64_t tpp = (int64_t)((a.W + kTileW - 1) / kTileW) * (int64_t)((a.H + 63) / 64);
  const int64_t planes = a.N * a.C;
  const int64_t G = sm_count();
  int best = 1;
  double best_cost = 1e300;
  for (int tpc = 16; tpc >= 1; tpc /= 2) {
    if (tpc > max_tiles) continue;
    const int64_t chunks = planes * ((tpp + tpc - 1) / tpc);
    const double cost = (double)((chunks + G - 1) / G) * (tpc + 0.2);
    if (cost < best_cost * 0.999) {
      best_cost = cost;
      best = tpc;
    }
  }
  return best;
}

// Chunk length of both gradients as two passes: a lane of the filter kernel adds
// the terms of a chunk one after the other in FP32, 4 rows of every tile for K <=
// 7, 8 for K = 11, 16 else.  No more tiles than keep that as short as four warps
// of a fused kernel with the automatic chunks do: 16 rows for K <= 7, 32 for K = 9
// and 11, 64 above; half as many for BF16 K <= 7, whose short chains are almost
// exact, so that the FP32 sums over lanes and warps count (error of dw against
// FP64, 16 x 8 x 512^2 K = 7: 1.11e-7 with four tiles, 1.02e-7 with two, 0.98e-7
// the fused kernel with roles; 4 x 3 x 1024^2 67 -> 70 us).
static int split_tiles_per_chunk(const DwArgs& a) {
  const int per = a.K == 9 || (a.K <= 7 && a.dtype != 0) ? 2 : 4;
  return auto_filter_tiles_per_chunk(a, std::min(16, per * auto_tiles_per_cta(a)));
}

DwConfig tune_config(int op, int id, const DwArgs& a) {
  DwConfig c;
  c.rows_per_thread = 8;
  c.persistent = 0;
  c.prefetch = 0;
  c.split = 0;
  c.ring = 0;
  c.tiles_per_cta = op == TUNE_BWD_FILTER ? auto_filter_tiles_per_chunk(a) : auto_tiles_per_cta(a);
  static const int tpc[5] = {0, 2, 4, 8, 16};
  switch (op) {
    case TUNE_FWD:
    case TUNE_BWD_INPUT:
      c.rows_per_thread = (id & 1) ? 4 : 8;
      c.persistent = (id & 2) ? 1 : 0;
      c.prefetch = (id & 4) ? 1 : 0;
      break;
    case TUNE_BWD_FILTER:
      if (id >= 1 && id <= 4) c.tiles_per_cta = tpc[id];
      break;
    default:
      if (id >= 1 && id <= 4) c.tiles_per_cta = tpc[id];
      if (id == 5 || id == 6) {
        c.split = id == 5;
        c.ring = id == 6;
        c.tiles_per_cta = c.split ? split_tiles_per_chunk(a) : auto_filter_tiles_per_chunk(a);
      }
      break;
  }
  return c;
}

// Inputs that TMA can load: rows and bases on 16-byte boundaries (BF16 bases 8
// bytes off one still allow 8-byte accesses, DwArgs::vec, but not TMA).  Without
// pointers, as in a query, the row length decides.
static bool inputs_aligned(const DwArgs& a) {
  return a.W * (a.dtype == 0 ? 4 : 2) % 16 == 0 && reinterpret_cast<uintptr_t>(a.x) % 16 == 0 &&
         reinterpret_cast<uintptr_t>(a.dy) % 16 == 0;
}

// Candidates that the built-in rule takes beside 0 (tune_config).
constexpr int kTileRows32 = 1, kPrefetch = 4;            // forward, input gradient
constexpr int kTilePairs = 1, kTwoPasses = 5, kRing = 6;  // both gradients

// Without a stored choice the configuration follows from the filter size, the
// storage type, the inputs' alignment and the number T of 64 x 128 tiles
// against the S SMs (S = 152; times in us, candidate 0 -> the choice):
//  * forward and input gradient, T <= 2 S: 32-row tiles, because 64-row tiles
//    leave SMs with no CTA or one (512^2 K = 21: 21.2 -> 12.0, K = 31: 43 -> 24;
//    2 x 3 x 512^2 K = 15: 19 -> 16; 3 x 1080 x 1920, T = 5 S: equal), but for K >= 25,
//    whose halo costs them most, where an SM then has twice as many all the same
//    (3 x 512^2 K = 31: 43 -> 47).
//    Above: the L2 prefetch where the tile load shows -- aligned FP32 K = 7, 9
//    (16 x 3 x 2048^2: 380 -> 368, 573 -> 554) and BF16 K <= 3 (197 -> 179);
//    FP32 K = 3 loses by it (230 -> 253), the others are equal.
//  * both gradients, fused kernel -> the choice:
//    FP32 K <= 3, very many tiles: the fused kernel with two tiles per CTA, whose
//    three CTAs per SM keep HBM busier than the ring's one, and whose CTAs work
//    on nearer tiles than with the usual 8 or 16 each: K = 3 from T = 100 S (12 x 3 x
//    2048^2, ring -> pairs 297 -> 289; 8 x 3 x 4096^2 793 -> 738; unaligned 16 x 3 x
//    2048 x 2047, fused -> pairs 598 -> 556), K = 1 from 80 S (183 -> 179).
//    K <= 3, aligned planes: the tile ring, FP32 K = 3 from 32 S (4 x 3 x 1801 x 2400
//    111 -> 104; at 20 S 59.6 -> 60.8) unless a plane is one tile (32 x 128 x 56 x 56
//    59 -> 75: every chunk one tile, one reduction); BF16 from 4 S (8 x 3 x 1024^2
//    K = 1 41 -> 31). FP32 K = 1 loses (97 -> 110). Its one CTA per SM stages
//    unaligned planes with the warps that compute (160 -> 207), and its four dx
//    warps store rows at any alignment slowly (BF16 4 x 3 x 1801 x 2400, aligned
//    inputs only: 143 -> 194).
//    Two passes (planes 4 x 3 x 1801 x 2400 or 2399 unless stated).  FP32: K >= 13 from
//    4 S (3 x 1080 x 1920 K = 13 102 -> 97; 716 -> 638; K = 15 864 -> 796) but K = 15 on
//    planes of one tile (8 x 192 x 28 x 28 217 -> 226); K = 11 aligned from 4 S (86 ->
//    81, 556 -> 476), unaligned from 32 S (600 -> 575; at 20 S 291 -> 300) but planes
//    of one tile (8 x 512 x 7 x 7 346 -> 366); K = 9 aligned from 4 S (4 x 3 x 1024^2
//    111 -> 103).  BF16: K = 15, and K = 11, 13 aligned, from 32 S (904 -> 844, 540 ->
//    512, 721 -> 691; at 20 S equal; K = 11 unaligned 684 -> 708) but planes of one
//    tile (32 x 128 x 56 x 56 K = 13 433 -> 473); K = 9 aligned from 4 S (67 -> 64);
//    K = 7 aligned from 8 S (73 -> 67; 16 x 3 x 2048^2 947 -> 837) but planes of one tile
//    (174 -> 181); K = 5 aligned from 5 S (28.5 -> 26.0).
int default_choice(int op, const DwArgs& a) {
  const int64_t S = sm_count();
  const int64_t tpp = ((a.W + kTileW - 1) / kTileW) * ((a.H + 63) / 64);
  const int64_t T = a.N * a.C * tpp;
  const bool f32 = a.dtype == 0, many = tpp > 1;  // many: a plane is more than one tile
  const bool aligned = inputs_aligned(a);
  if (op == TUNE_FWD || op == TUNE_BWD_INPUT) {
    const int64_t T32 = a.N * a.C * ((a.W + kTileW - 1) / kTileW) * ((a.H + 31) / 32);
    const bool rows32 = a.K < 25 || (T32 + S - 1) / S < 2 * ((T + S - 1) / S);
    if (T <= 2 * S && rows32) return kTileRows32;
    return aligned && (f32 ? a.K == 7 || a.K == 9 : a.K <= 3) ? kPrefetch : 0;
  }
  if (op != TUNE_BWD_FUSED) return 0;
  if (f32 && a.K <= 3 && T >= (a.K == 1 ? 80 : 100) * S) return kTilePairs;
  if (a.K <= 3 && aligned && a.vec && (f32 ? a.K == 3 && many && T >= 32 * S : T >= 4 * S))
    return kRing;
  int64_t from = -1;  // two passes from this many tiles per SM on
  if (f32 && (a.K == 13 || (a.K == 15 && many) || (a.K == 11 && aligned)))
    from = 4;
  else if (a.K >= 11 && many && (aligned || f32 || a.K == 15))
    from = 32;
  else if (a.K == 9 && aligned)
    from = 4;
  else if (a.K == 7 && !f32 && aligned && many)
    from = 8;
  else if (a.K == 5 && !f32 && aligned)
    from = 5;
  return from >= 0 && T >= from * S ? kTwoPasses : 0;
}

DwConfig default_config(int op, const DwArgs& a) {
  return tune_config(op, default_choice(op, a), a);
}

static bool planes_aligned(const DwArgs& a) { return a.vec && inputs_aligned(a); }

// Key without the alignment, and with it.
static std::string pin_key(int op, const DwArgs& a) {
  const double n = (double)a.N * a.C * a.H * a.W;
  const int sc = n > 0 ? (int)std::floor(std::log2(n)) : 0;
  char buf[96];
  std::snprintf(buf, sizeof(buf), "%d:%d:%d:%d:%d", op, a.dtype, a.K, a.border, sc);
  return buf;
}
static std::string key_of(int op, const DwArgs& a) {
  return pin_key(op, a) + (planes_aligned(a) ? ":0" : ":1");
}

// A choice for a key without the alignment replaces those of both alignments.
static void put_choice(const std::string& key, int id) {
  if (std::count(key.begin(), key.end(), ':') == 4) {
    g_cache.erase(key + ":0");
    g_cache.erase(key + ":1");
  }
  g_cache[key] = id;
}

// ---- JSON persistence: {"giga_autotune": 1, "entries": {"key": id, ...}}
static bool parse_cache(const std::string& text, std::map<std::string, int>& out) {
  if (text.find("\"giga_autotune\"") == std::string::npos) return false;
  size_t p = text.find("\"entries\"");
  if (p == std::string::npos) return false;
  p = text.find('{', p);
  if (p == std::string::npos) return false;
  const size_t end = text.find('}', p);
  if (end == std::string::npos) return false;
  std::map<std::string, int> tmp;
  while (true) {
    size_t q0 = text.find('"', p);
    if (q0 == std::string::npos || q0 > end) break;
    size_t q1 = text.find('"', q0 + 1);
    if (q1 == std::string::npos || q1 > end) return false;
    std::string key = text.substr(q0 + 1, q1 - q0 - 1);
    size_t colon = text.find(':', q1);
    if (colon == std::string::npos || colon > end) return false;
    char* stop = nullptr;
    long v = std::strtol(text.c_str() + colon + 1, &stop, 10);
    if (stop == text.c_str() + colon + 1 || v < 0 || v > 64) return false;
    for (char ch : key)
      if (!(ch == ':' || ch == '-' || (ch >= '0' && ch <= '9'))) return false;
    tmp[key] = (int)v;
    p = (size_t)(stop - text.c_str());
  }
  out.swap(tmp);
  return true;
}

static bool load_file(const char* path) {
  std::ifstream f(path);
  if (!f) return false;
  std::stringstream ss;
  ss << f.rdbuf();
  std::map<std::string, int> m;
  if (!parse_cache(ss.str(), m)) return false;  // a corrupt cache is ignored
  for (auto& kv : m) put_choice(kv.first, kv.second);  // in order: a key before its longer ones
  return true;
}

static bool save_file(const char* path) {
  std::string tmp = std::string(path) + ".tmp";
  {
    std::ofstream f(tmp);
    if (!f) return false;
    f << "{\"giga_autotune\": 1, \"entries\": {";
    bool first = true;
    for (auto& kv : g_cache) {
      f << (first ? "" : ", ") << '"' << kv.first << "\": " << kv.second;
      first = false;
    }
    f << "}}\n";
  }
  return std::rename(tmp.c_str(), path) == 0;
}

static void ensure_loaded() {
  if (g_loaded) return;
  g_loaded = true;
  if (const char* p = std::getenv("GIGA_AUTOTUNE_CACHE")) load_file(p);
}

int tune_lookup(int op, const DwArgs& a) {
  std::lock_guard<std::mutex> lk(g_mu);
  ensure_loaded();
  if (g_cache.empty()) return -1;
  auto it = g_cache.find(key_of(op, a));
  if (it == g_cache.end()) it = g_cache.find(pin_key(op, a));
  if (it == g_cache.end()) return -1;
  return it->second < tune_candidates(op) ? it->second : -1;
}

void tune_store(int op, const DwArgs& a, int id, bool pin) {
  std::lock_guard<std::mutex> lk(g_mu);
  ensure_loaded();
  put_choice(pin ? pin_key(op, a) : key_of(op, a), id);
  if (const char* p = std::getenv("GIGA_AUTOTUNE_CACHE")) save_file(p);
}

// GIGA_LOG=1 (or any value but 0): each tuning decision is printed to
// standard error, one line per (op, problem class) with every candidate's time.
bool tune_log_enabled() {
  const char* e = std::getenv("GIGA_LOG");
  return e && *e && std::strcmp(e, "0") != 0;
}

static const char* op_name(int op) {
  switch (op) {
    case TUNE_FWD: return "forward";
    case TUNE_BWD_INPUT: return "input-gradient";
    case TUNE_BWD_FILTER: return "filter-gradient";
    default: return "fused-backward";
  }
}

giga_status_t tune_dw_op(int op, const DwArgs& a, cudaStream_t st) {
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess) return fail(GIGA_ERR_CUDA, "event create");
  if (cudaEventCreate(&e1) != cudaSuccess) {
    cudaEventDestroy(e0);
    return fail(GIGA_ERR_CUDA, "event create");
  }
  int best = 0;
  float best_ms = 1e30f;
  std::string times;
  giga_status_t status = GIGA_OK;
  for (int id = 0; id < tune_candidates(op) && status == GIGA_OK; ++id) {
    const DwConfig cfg = tune_config(op, id, a);
    status = run_dw_op(op, a, cfg, st);  // warm-up
    if (status != GIGA_OK) break;
    cudaEventRecord(e0, st);
    for (int rep = 0; rep < 3 && status == GIGA_OK; ++rep) status = run_dw_op(op, a, cfg, st);
    cudaEventRecord(e1, st);
    cudaError_t e = cudaEventSynchronize(e1);
    if (e != cudaSuccess) {
      status = cuda_fail(e, "autotune timing");
      break;
    }
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    char buf[48];
    std::snprintf(buf, sizeof(buf), "%s%d:%.3f", id ? " " : "", id, ms / 3.f);
    times += buf;
    if (ms < best_ms) {
      best_ms = ms;
      best = id;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (status == GIGA_OK) {
    tune_store(op, a, best, false);
    if (tune_log_enabled())
      std::fprintf(stderr,
                   "giga autotune: %s %s K=%d %s N*C*H*W=%lld (class %s) -> candidate %d "
                   "(ms per call: %s)\n",
                   op_name(op), a.dtype ? "bf16" : "f32", a.K, a.border ? "clamp" : "zero",
                   (long long)(a.N * a.C * a.H * a.W), key_of(op, a).c_str(), best,
                   times.c_str());
  }
  return status;
}

}  // namespace giga

using namespace giga;

extern "C" {

giga_status_t giga_autotune_set_mode(int32_t mode) {
  clear_error();
  if (mode < 0 || mode > 2) return fail(GIGA_ERR_INVALID_ARG, "autotune mode must be 0, 1 or 2");
  std::lock_guard<std::mutex> lk(g_mu);
  g_mode = mode;
  return GIGA_OK;
}

int32_t giga_autotune_get_mode(void) { return tune_mode(); }

giga_status_t giga_autotune_save(const char* path) {
  clear_error();
  if (!path) return fail(GIGA_ERR_INVALID_ARG, "path is NULL");
  std::lock_guard<std::mutex> lk(g_mu);
  return save_file(path) ? GIGA_OK : fail(GIGA_ERR_INVALID_ARG, "cannot write autotune cache");
}

giga_status_t giga_autotune_load(const char* path) {
  clear_error();
  if (!path) return fail(GIGA_ERR_INVALID_ARG, "path is NULL");
  std::lock_guard<std::mutex> lk(g_mu);
  g_loaded = true;
  return load_file(path) ? GIGA_OK
                         : fail(GIGA_ERR_INVALID_ARG, "autotune cache missing or corrupt (ignored)");
}

void giga_autotune_clear(void) {
  std::lock_guard<std::mutex> lk(g_mu);
  g_cache.clear();
}

}  // extern "C"
