// Host-side helpers shared by the C ABI translation units: CUDA error capture, workspace
// growth, per-phase event timing, and the tile-variant autotuner's cache.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <fstream>
#include <sstream>

#include "ozg_context.h"
#include "ozg_window.h"

namespace ozg {

long long& launch_counter() {
  static long long n = 0;
  return n;
}

namespace host {

namespace {
char g_last_cuda[256] = "no error";
std::mutex g_err_mu;
}  // namespace

const char* last_cuda_error_text() { return g_last_cuda; }

int cuda_fail(cudaError_t e) {
  std::lock_guard<std::mutex> lk(g_err_mu);
  std::snprintf(g_last_cuda, sizeof(g_last_cuda), "%s: %s", cudaGetErrorName(e), cudaGetErrorString(e));
  return OZG_ERR_CUDA;
}

char norm_trans(char t) {
  if (t >= 'a' && t <= 'z') t = (char)(t - 'a' + 'A');
  return t;
}

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

static int grow_buffer(ozg_ctx* c, void** buf, size_t* cap, size_t bytes) {
  if (bytes <= *cap) return OZG_OK;
  OZG_CUDA(cudaStreamSynchronize(c->stream));
  if (*buf) {
    cudaFree(*buf);
    *buf = nullptr;
    *cap = 0;
  }
  size_t want = workspace_size(bytes);
  if (c->fail_allocs > 0) {  // injected failure (test hook), as if cudaMalloc had failed
    --c->fail_allocs;
    return OZG_ERR_ALLOC;
  }
  cudaError_t e = cudaMalloc(buf, want);
  if (e != cudaSuccess) {
    cudaGetLastError();
    *buf = nullptr;
    return OZG_ERR_ALLOC;
  }
  *cap = want;
  return OZG_OK;
}

bool capturing(ozg_ctx* c) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(c->stream, &cs) == cudaSuccess) return cs != cudaStreamCaptureStatusNone;
  cudaGetLastError();
  return true;
}

static bool room_for(ozg_ctx* c, size_t cap, size_t lean, size_t bytes) {
  if (bytes <= cap) return true;
  if (capturing(c)) return false;  // no growing while the caller captures: keep to what was reserved
  size_t free_b = 0, total_b = 0;
  if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return layout_room(cap, lean, bytes, free_b);
}

bool ws_room(ozg_ctx* c, size_t lean, size_t bytes) { return room_for(c, c->ws_cap, lean, bytes); }
bool gws_room(ozg_ctx* c, size_t lean, size_t bytes) { return room_for(c, c->gws_cap, lean, bytes); }

int ensure_ws(ozg_ctx* c, size_t bytes) { return grow_buffer(c, &c->ws, &c->ws_cap, bytes); }
int ensure_z3ws(ozg_ctx* c, size_t bytes) { return grow_buffer(c, &c->z3ws, &c->z3ws_cap, bytes); }

int ensure_gws(ozg_ctx* c, size_t bytes) {
  if (bytes <= c->gws_cap) return OZG_OK;
  c->plan.reset();  // a captured plan points into the old buffer
  ++c->gws_epoch;
  return grow_buffer(c, &c->gws, &c->gws_cap, bytes);
}

cudaEvent_t pool_get(ozg_ctx* c) {
  if (!c->pool.empty()) {
    cudaEvent_t e = c->pool.back();
    c->pool.pop_back();
    return e;
  }
  cudaEvent_t e = nullptr;
  if (cudaEventCreate(&e) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  return e;
}

PhaseScope::PhaseScope(ozg_ctx* c_, int ph) : c(c_), phase(ph) {
  if (!c->prof) return;
  // no marks inside a graph capture (the replays are timed as a whole)
  if (capturing(c)) return;
  if ((a = pool_get(c)) != nullptr) cudaEventRecord(a, c->stream);
}

PhaseScope::~PhaseScope() {
  if (!a) return;
  cudaEvent_t b = pool_get(c);
  if (!b) {
    c->pool.push_back(a);
    return;
  }
  cudaEventRecord(b, c->stream);
  c->pending.push_back({phase, a, b});
}

// Shape bucket: rounded log2 of the stacked rows, cols and k, plus the slice count.
uint64_t shape_bucket(int64_t rows, int64_t cols, int64_t k, int s) {
  auto lg = [](int64_t x) { return (uint64_t)std::lround(std::log2((double)(x > 0 ? x : 1)) * 2.0); };
  return (lg(rows) << 40) | (lg(cols) << 24) | (lg(k) << 8) | (uint64_t)s;
}

static void tune_load(ozg_ctx* c) {
  if (c->tune_loaded) return;
  c->tune_loaded = true;
  if (c->tune_path.empty()) return;
  std::ifstream in(c->tune_path);
  std::string line;
  while (std::getline(in, line)) {
    unsigned long long b = 0;
    int v = 0;
    // single-call variants: 0 .. 3 and the stacked group pairs (no CTA pairs for single calls), or
    // difference planes where they were timed
    if (std::sscanf(line.c_str(), "%llx %d", &b, &v) == 2 &&
        ((v >= 0 && v <= 3) || v == kStackedVariant || (v == kDiffChoice && (b & kDiffBucket))))
      c->tune[b] = v;
  }
}

void tune_store(ozg_ctx* c, uint64_t bucket, int variant) {
  c->tune[bucket] = variant;
  if (c->tune_path.empty()) return;
  std::ofstream out(c->tune_path, std::ios::app);
  out << std::hex << bucket << std::dec << " " << variant << "\n";
}

// Heuristic variant: the tile width that wastes the least output area (ties -> 256 wide); for
// 256-wide tiles deferred epilogue pushes when k >= 2048 (they then overlap the next chains'
// MMAs; for short k the epilogue is the bottleneck and immediate pushes measured faster); for
// 128-wide tiles two 64-wide k sub-tiles per stage (measured faster than the deeper 6-stage
// pipeline for s = 7..12 once grouped tiles are handed out dynamically).
static int heuristic_variant(int64_t rows, int64_t cols, int64_t k, int s) {
  (void)rows;
  (void)s;
  const int64_t p256 = (cols + 255) / 256 * 256, p128 = (cols + 127) / 128 * 128;
  if (p128 < p256) return 1;
  return k >= 2048 ? 2 : 0;
}

int choose_variant(ozg_ctx* c, int64_t rows, int64_t cols, int64_t k, int s) {
  // single calls have no CTA-pair kernel: a forced pair variant runs as the 1-CTA 128-wide one
  if (c->force_variant >= 0) return c->force_variant == kPairVariant ? 1 : c->force_variant;
  tune_load(c);
  auto it = c->tune.find(shape_bucket(rows, cols, k, s));
  if (it != c->tune.end()) return it->second;
  // the stacked group pairs where they apply: on square DGEMMs of 1024 .. 8192 at s = 7 .. 10
  // they measured 0.47 - 1.06x the time of the width heuristic's choice (faster except for
  // 2048^3 and for 8192^3 at s = 10, by 6%)
  if (s <= stacked_max_slices() && !c->exact) return kStackedVariant;
  return heuristic_variant(rows, cols, k, s);
}

// How one call runs when no variant is forced: on difference planes (ozg_gemm_kd.cu) or on
// the stacked kernel, there possibly with every tile's k range cut into parts.  The times of all
// ways are estimated in microseconds from the tiles in whole waves and the costs measured per
// 64-wide k stage, per pass and per tile.
//   stacked: 128 x 128 tiles on 152 CTAs, 0.275 per stage + 18 per tile (final rounding);
//   in parts: a part adds its window sums to the tile's words in L2 instead (3 per window + 6), and
//   zeroing, reading and rounding them costs a launch and 0.1 per tile and window;
//   difference planes: 256 x 256 tiles on 76 CTA pairs, 0.30 per stage, 2 s - 1 passes and a tile
//   end of 36 (complex, whose window words stay in registers: 25); 3.3 per pass of a real tile
//   (its sums enter windows in L2; those of the first window also the second's), 1 per complex
//   one; and the split writes s^2 / 4 more planes (at 5.5 TB/s).
// Difference planes against the stacked kernel on one GB300: real 2048 x 2048 at s = 7, k = 1024 /
// 2048 / 4096: 0.95 / 1.09 / 1.21 of its speed, 8192^3 s = 7 1.41; complex 1024 x 1024 s = 7 k = 192
// / 1024: 1.10 / 1.36, 3616^3 1.51.  Parts against whole tiles (whole calls, us): 256^3 s = 7 72 ->
// 53, 148 x 100 x 4287 s = 10 705 -> 76, 1537 x 2001 x 1111 s = 10 (208 tiles: a second wave of 56)
// 455 -> 389, 1024^3 s = 8 154 -> 109; 144 complex tiles of 768^3 s = 6 103 -> 123 in two parts: whole.
SinglePlan plan_single(int num_sms, bool cplx, int64_t rows, int64_t cols, int64_t k, bool learned, int s, int s_planes) {
  SinglePlan P;
  if (s_planes > stacked_max_slices()) return P;
  const int64_t KB = (k + 63) / 64;
  auto window = [&](int x) { return window_len(x, KB * 64, cplx); };  // of the difference-plane kernel
  auto waves = [](int64_t tiles, int64_t units) { return (double)((tiles + units - 1) / units); };
  const int se = learned ? std::min(s, 8) : s;  // a learned count is 7 - 9 in practice
  int stages = 0;  // of the stacked kernel per 64-wide k sub-tile: groups in pairs from the last down
  for (int g = se + 1; g >= 2; g -= 2) stages += g - 1;
  const int64_t tiles = ((rows + 127) / 128) * ((cols + 127) / 128);
  double best = waves(tiles, num_sms) * (0.275 * stages * (double)KB + 18.0);
  const int nwin = stk_windows(se, k, cplx);
  int64_t max_parts = std::min<int64_t>(KB, 64);
  for (int64_t p = 2; p <= max_parts; ++p) {
    const int64_t kb = (KB + p - 1) / p;
    if ((KB + kb - 1) / kb != p) continue;  // the same cut as with fewer parts
    const double t = waves(tiles * p, num_sms) * (0.275 * stages * (double)kb + 3.0 * nwin + 6.0) + 8.0 +
                     0.1 * (double)(tiles * nwin);
    if (t < best) {
      best = t;
      P.parts = (int)p;
      P.part_kb = (int)kb;
    }
  }
  for (int x = 1; x <= s_planes; ++x) P.part_windows = std::max(P.part_windows, stk_windows(x, k, cplx));
  // difference planes: the exact sum must fit two windows, and R its int32
  auto fits = [&](int x) { return x <= 2 * window(x) && window(x) * k * (cplx ? 2 : 1) <= 130000; };
  int kd = std::min(s, kKdMax);
  while (kd > 0 && !fits(kd)) --kd;
  if (kd < (learned ? se : s) || kd == 0) return P;  // a fixed count runs on one kernel
  const int products = se + se * se / 4, win = window(se), len0 = se <= win ? 0 : se - win;
  const double diff = waves(kd_tiles(rows, cols), num_sms / 2) *
                          (0.30 * products * (double)KB + (cplx ? 2 * se - 1 + 25.0 : 3.3 * (2 * se - 1 + len0) + 36.0)) +
                      (double)(rows + cols) * (double)k * 2.0 * (products - se) / 5.5e6;
  if (diff < best) P.kd = kd;
  return P;
}

}  // namespace host
}  // namespace ozg

extern "C" int ozg_kernel_launches(long long* out) {
  if (!out) return OZG_ERR_INVALID;
  *out = __atomic_load_n(&ozg::launch_counter(), __ATOMIC_RELAXED);
  return OZG_OK;
}
