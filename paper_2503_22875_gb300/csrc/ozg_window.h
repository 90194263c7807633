// The epilogues' integer windows (host and device): how many slice groups one int64 word holds,
// how many words a call's sum takes, and how the difference-plane kernel's sums enter one.  The kernels and the plans that size their buffers use the same
// functions on the same padded k.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define OZG_HD __host__ __device__ __forceinline__
#else
#define OZG_HD inline
#endif

namespace ozg {

OZG_HD int bit_length(unsigned long long x) {
#ifdef __CUDA_ARCH__
  return 64 - __clzll((long long)x);
#else
  return x == 0 ? 0 : 64 - __builtin_clzll(x);
#endif
}

// The group sums enter R by Horner's rule in exact int64 arithmetic, c consecutive groups per
// window, where c is the largest count whose worst case stays below 2^63:
//   |G_g| <= (g - 1) * kpad * 127^2 (x2 for the complex combine) <= gmax < 2^L,
//   |window| <= gmax (128^c - 1) / 127 < 2^(L + 7 c) / 127 <= 2^69 / 127   with
//   c = (62 - L) / 7 + 1, i.e. L + 7 c <= 69: below 2^62 (128/127) < 2^63 - 2^57.
// Two windows form the exact 128-bit N = W0 128^len1 + W1, rounded to FP64 once with integer
// instructions only; a third and later window continue in FP64 (one rounding per window).
OZG_HD int window_len(int s, int64_t kpad, int cplx) {
  const unsigned long long gmax = (unsigned long long)s * (unsigned long long)kpad * 16129ull * (cplx ? 2ull : 1ull);
  const int c = (62 - bit_length(gmax)) / 7 + 1;
  return c < 1 ? 1 : c;
}

// The stacked kernel's windows.  Its k is padded to whole stages of this width (a call whose k
// takes an odd number of 64-wide sub-tiles has the windows of the next even one).
constexpr int kStackedK = 128;
OZG_HD int64_t stk_kpad(int64_t k) { return (k + kStackedK - 1) / kStackedK * kStackedK; }

// Length of the first window.  With three or more windows every window but the last holds win
// groups, as in the one-group kernels (their FP64 continuation rounds per window, so the split
// must be the same for the same bits).  With two windows the exact sum is rounded once and any
// split into windows of at most win groups gives the same bits: the first takes one group
// less when that makes the second window's count even (a lone group of a later window pairs
// far more planes than the lone group 2 of the first).
OZG_HD int stk_len0(int s, int win) {
  if (s <= win || s > 2 * win) return s < win ? s : win;
  return (((win - s) & 1) && s - (win - 1) <= win) ? win - 1 : win;
}

// Windows of a stacked call with s slices: the first of stk_len0 groups, then win at a time.
OZG_HD int stk_windows(int s, int64_t k, int cplx) {
  const int win = window_len(s, stk_kpad(k), cplx);
  return 1 + (s - stk_len0(s, win) + win - 1) / win;
}

// ---- weights of the difference-plane kernel's sums in a window word --------------------------
// sum_{j=0}^{n} 128^j
OZG_HD unsigned long long kd_geom(int n) {
  unsigned long long w = 1;
  for (int i = 0; i < n; ++i) w = (w << 7) + 1;
  return w;
}

// w as wh 2^32 + wl with a signed low word: v w = (int64) v wl + (v wh) 2^32 (mod 2^64)
struct KdWeight {
  int wl, wh;
};
OZG_HD KdWeight kd_weight(unsigned long long w) {
  const int wl = (int)(uint32_t)w;
  return {wl, (int)((long long)(w - (unsigned long long)(long long)wl) >> 32)};
}

// W + v w (mod 2^64); the high product counts modulo 2^32 and is formed unsigned, since v holds up to
// 64 chains (2^30) and wh several bits
OZG_HD unsigned long long kd_mac(unsigned long long W, int v, KdWeight w) {
  W += (unsigned long long)((long long)v * w.wl);
  return W + ((unsigned long long)((uint32_t)v * (uint32_t)w.wh) << 32);
}

}  // namespace ozg
