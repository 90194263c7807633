// Device code shared by the slice-product kernels (ozg_gemm.cu, ozg_gemm_kd.cu): the pipeline
// constants, the description of one output tile from either work source, and the epilogue's
// window arithmetic and final rounding of C.
#pragma once
#include <climits>

#include "ozg_device.cuh"
#include "ozg_internal.h"
#include "ozg_round.cuh"

namespace ozg {
namespace {

constexpr int BM = 128, BK = 64;  // BK: k width of one 128-byte swizzle atom (one TMA box)
constexpr int EPI_WARPS = 8;
constexpr int THREADS = 128 + EPI_WARPS * 32;
constexpr int REG_PRODUCER = 56, REG_EPILOGUE = 224;
static_assert(128 * REG_PRODUCER + EPI_WARPS * 32 * REG_EPILOGUE <= THREADS * 168, "register split");
constexpr int TRING = 4;       // tile-index ring depth (grouped launches)
constexpr int CHAIN_K = 1024;  // products per accumulation chain: 1024 * 127^2 = 16516096 < 2^24
constexpr int GROUP_M = 8;     // tile raster: GROUP_M row-tiles share a sweep over the column tiles
static_assert(CHAIN_K * 127 * 127 < (1 << 24), "FP32 chain must stay exact");

// One pipeline stage holds SUB 64-wide k sub-tiles of A and of B (SK = 64 SUB k).  With
// 128-wide tiles, two per stage (3 stages) give eight MMAs per barrier round trip instead of
// four -- one lane issuing a 128 x 128 x 64 block is slower than the tensor core executing it
// -- while one per stage (6 stages) hides more load latency (large s: bigger working sets).
//
// CTA pairs (PAIR, grouped launches, 128-wide): a 2-CTA cluster computes a 256 x BN tile with
// tcgen05.mma.cta_group::2 (M = 256) issued by the even-rank CTA.  Each CTA stages its own 128
// rows of A and BN / 2 of the B columns (the MMA reads the other half from the peer), so a stage
// is 48 KB instead of 64 KB and four stages fit; each CTA's TMEM holds its own 128 rows of the
// accumulator, drained by its own epilogue exactly as in a 1-CTA tile.
template <int BN_, int SUB_, bool PAIR_ = false>
struct Cfg {
  static constexpr int SUB = SUB_;
  static constexpr int SK = SUB * BK;
  static constexpr int SEG = CHAIN_K / SK;  // stages per chain
  static constexpr int STAGES = PAIR_ ? 4 : (BN_ == 256 ? 4 : (SUB_ == 2 ? 3 : 6));
  static constexpr uint32_t SUBA_BYTES = BM * BK * 2, SUBB_BYTES = (PAIR_ ? BN_ / 2 : BN_) * BK * 2;
  static constexpr uint32_t A_BYTES = SUB * SUBA_BYTES, B_BYTES = SUB * SUBB_BYTES, STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr uint32_t IDESC = umma_idesc_f16_f32(PAIR_ ? 2 * BM : BM, BN_);
  // two BN-column FP32 accumulators; 128-wide tiles also keep the int64 window words (two
  // columns per output) in the other half
  static constexpr uint32_t TMEM_COLS = 512;
  static constexpr int CPT = BN_ / 2;             // columns per epilogue thread
  static constexpr size_t SMEM = (size_t)STAGES * STAGE_BYTES + 1024;
};

// Everything one output tile needs, from either work source.
struct TileJob {
  const CUtensorMap* tmA;
  const CUtensorMap* tmB;
  int tm, tn, KB, s, cplx, skip, kd;
  int klast;  // 64-wide sub-tiles holding valid k in the last stage (1 .. SUB)
  int64_t rows, cols, n;  // stacked product rows / cols, output columns (complex: n)
  const int32_t* e;
  const int32_t* f;
  double* C;
  int64_t ldc;
  double a0, a1, b0, b1;
  int beta_zero;
};

__device__ __forceinline__ void tile_coords(int t, int tiles_m, int tiles_n, int& tm, int& tn) {
  int per_group = GROUP_M * tiles_n;
  int grp = t / per_group;
  int first = grp * GROUP_M;
  int gsz = min(tiles_m - first, GROUP_M);
  int r = t % per_group;
  tm = first + r % gsz;
  tn = r / gsz;
}

template <int BN_, int SUB_, bool GROUPED, bool PAIR = false, int TROWS = BM>
__device__ __forceinline__ TileJob get_job(int t, const CUtensorMap* tmA, const CUtensorMap* tmB, const GemmArgs* P,
                                           const GroupArgs* G) {
  TileJob j;
  if (!GROUPED) {
    const int tiles_m = (int)((P->rows + TROWS - 1) / TROWS), tiles_n = (int)((P->cols + BN_ - 1) / BN_);
    tile_coords(t, tiles_m, tiles_n, j.tm, j.tn);
    j.tmA = tmA;
    j.tmB = tmB;
    j.KB = (int)((P->k + Cfg<BN_, SUB_>::SK - 1) / Cfg<BN_, SUB_>::SK);
    j.klast = (int)((P->k - (int64_t)(j.KB - 1) * Cfg<BN_, SUB_>::SK + BK - 1) / BK);
    j.s = P->s_dev != nullptr ? *P->s_dev : P->s;
    j.kd = P->kd;
    j.cplx = P->cplx;
    j.skip = 0;
    j.rows = P->rows;
    j.cols = P->cols;
    j.n = P->n;
    j.e = P->e;
    j.f = P->f;
    j.C = P->C;
    j.ldc = P->ldc;
    j.a0 = P->alpha[0];
    j.a1 = P->alpha[1];
    j.b0 = P->beta[0];
    j.b1 = P->beta[1];
    j.beta_zero = P->beta_zero;
  } else {
    const GroupTile gt = G->tiles[t];
    if (gt.call < 0) {  // padding slot of the load-balanced tile list
      j.skip = 1;
      return j;
    }
    const GroupCall* c = G->calls + gt.call;
    j.tm = gt.tm;
    j.tn = gt.tn;
    j.tmA = &c->tmA;
    j.tmB = PAIR ? &c->tmBh : &c->tmB;  // CTA pairs load half of the B columns each
    j.KB = (int)((c->k + Cfg<BN_, SUB_>::SK - 1) / Cfg<BN_, SUB_>::SK);
    j.klast = (int)((c->k - (int64_t)(j.KB - 1) * Cfg<BN_, SUB_>::SK + BK - 1) / BK);
    j.s = c->s;
    j.cplx = c->cplx;
    j.skip = (c->nonfinite != nullptr && *c->nonfinite) ? 1 : 0;
    j.rows = c->rows;
    j.cols = c->cols;
    j.n = c->n;
    j.e = c->e;
    j.f = c->f;
    j.C = c->C;
    j.ldc = c->ldc;
    j.a0 = c->alpha[0];
    j.a1 = c->alpha[1];
    j.b0 = c->beta[0];
    j.b1 = c->beta[1];
    j.beta_zero = c->beta_zero;
  }
  return j;
}

__device__ __forceinline__ int nseg_of(int g, int KB, int seg) { return ((g - 1) * KB + seg - 1) / seg; }

__device__ __noinline__ double ldexp_slow(double x, int E) { return ldexp(x, E); }
// x * 2^E with one rounding (the same result as ldexp); fast path when 2^E is a normal double
__device__ __forceinline__ double scale_pow2(double x, int E) {
  if (E >= -1022 && E <= 1023) return x * __longlong_as_double((long long)(E + 1023) << 52);
  return ldexp_slow(x, E);
}

// Exact epilogue (s <= kExactMaxS): R is a 128-bit integer per output, kept as (lo, hi) in 16
// bytes of the CTA's scratch tile; the group sums enter by Horner's rule R <- 128 R + G_g, and
// the final R is rounded to FP64 once.  |R| < 2^(log2 max|G_g| + 7 (s - 1) + 1), within 127 bits
// for s <= 13 and k < 2^20.  Larger s keeps an FP64 R (one rounding per Horner step).
constexpr int kExactMaxS = 13;

__device__ __forceinline__ void horner128(const void* Rp, int g, bool first, bool group2, int64_t& hi,
                                          uint64_t& lo) {
  if (first && group2) {
    lo = (uint64_t)(int64_t)g;
    hi = g < 0 ? -1 : 0;
    return;
  }
  const longlong2 v = *reinterpret_cast<const longlong2*>(Rp);
  lo = (uint64_t)v.x;
  hi = v.y;
  if (first) {  // R <- 128 R (two's complement 128-bit shift)
    hi = (int64_t)(((uint64_t)hi << 7) | (lo >> 57));
    lo <<= 7;
  }
  const uint64_t gl = (uint64_t)(int64_t)g, nl = lo + gl;
  hi = hi + (g < 0 ? -1 : 0) + (nl < lo ? 1 : 0);
  lo = nl;
}


// One output's Horner step in either mode; returns the final value (scaled) on the last push.
__device__ __forceinline__ double horner_step(void* Rp, int g, bool exact, bool first, bool group2, bool final_push,
                                              int E) {
  if (exact) {
    int64_t hi;
    uint64_t lo;
    horner128(Rp, g, first, group2, hi, lo);
    if (final_push) return round_i128(hi, lo, E);
    *reinterpret_cast<longlong2*>(Rp) = make_longlong2((long long)lo, (long long)hi);
    return 0.0;
  }
  double* Rd = reinterpret_cast<double*>(Rp);
  const double gv = (double)g;
  const double Rv = first ? (group2 ? gv : fma(*Rd, 128.0, gv)) : (*Rd + gv);
  if (final_push) return scale_pow2(Rv, E);
  *Rd = Rv;
  return 0.0;
}

// Window-closing or final step of one output, given the first slot's word s0 (int64 W0 while
// widx == 1, FP64 bits from the second window's close on) and the active window Rw after this
// push.  Final: returns RN(N 2^E).  Closing: returns the new s0 word.
__device__ __forceinline__ double final_val(long long s0, long long Rw, int widx, int wlen, int E) {
  if (widx == 0) return rn_i128_pow2(Rw < 0 ? -1 : 0, (unsigned long long)Rw, E);
  if (widx == 1) {
    long long hi;
    unsigned long long lo;
    i128_shl_add(s0, 7 * wlen, Rw, hi, lo);
    return rn_i128_pow2(hi, lo, E);
  }
  return scale_pow2(fma(__longlong_as_double(s0), scale_pow2(1.0, 7 * wlen), (double)Rw), E);
}
__device__ __forceinline__ long long close_val(long long s0, long long Rw, int widx, int wlen) {
  if (widx == 1) {
    long long hi;
    unsigned long long lo;
    i128_shl_add(s0, 7 * wlen, Rw, hi, lo);
    return __double_as_longlong(rn_i128_pow2(hi, lo, 0));
  }
  return __double_as_longlong(fma(__longlong_as_double(s0), scale_pow2(1.0, 7 * wlen), (double)Rw));
}

enum PushKind { kPlain = 0, kSpill = 1, kClose = 2, kFinal = 3 };

// Everything a push needs besides the group sums.
struct PushArgs {
  int kind, widx, wlen;
  bool first, wstart;     // first push of its group; first push of its window
  uint32_t rtm;           // TMEM address of this thread's window words (TMEM-resident mode)
  long long* Ra;          // the active window's scratch slot (L2-resident mode)
  long long* S0;          // the first window's scratch slot
  int64_t gcol0, orow;
  bool row_ok, unit_ab, odd;
  int ebase;
};

// One push for NCH consecutive outputs o0 .. o0+NCH-1 of this thread; vals holds the chunk's
// group sums (vals[i], complex: the pair vals[2i], vals[2i+1]).  The active window lives
// in TMEM (TMR: two 32-bit columns per output, one 32x32b.x32 load and store per 16 outputs) or
// in the CTA's L2-resident scratch (loads batched NCH deep before any use, to keep that many in
// flight).  Complex: the (Re, Im) column pairs are combined exactly across the lane pair first.
// The scratch words S0 and the column exponents a closing or final push of outputs
// o0 .. o0+NCH-1 needs, loaded ahead of the push (software pipelining across chunks).
template <int NCH>
__device__ __forceinline__ void prefetch_close(const PushArgs& a, const TileJob& j, int o0, long long (&s0)[NCH],
                                               int (&fe)[NCH]) {
  if (a.widx >= 1) {
#pragma unroll
    for (int i = 0; i < NCH; ++i) s0[i] = a.S0[(size_t)(o0 + i) * BM];
  } else {
#pragma unroll
    for (int i = 0; i < NCH; ++i) s0[i] = 0;
  }
  const int64_t c0 = j.cplx ? (a.gcol0 >> 1) + o0 : a.gcol0 + o0;
  const int64_t climit = j.cplx ? j.n : j.cols;
#pragma unroll
  for (int i = 0; i < NCH; ++i) fe[i] = (a.kind == kFinal && c0 + i < climit) ? __ldg(j.f + c0 + i) : 0;
}

// RN(W 2^E) for one int64 window: one correctly rounded conversion, the power of two added to
// the exponent field.  `ok` is false when the result is not a normal double (the caller then
// takes final_val).  The same value as rn_windows(0, W, S, E) with fewer instructions.
__device__ __forceinline__ double rn_single(long long W, int E, bool& ok) {
  const long long bits = __double_as_longlong(__ll2double_rn(W));
  const int ex = (int)((bits >> 52) & 0x7ff) + E;
  ok = W == 0 || (ex >= 1 && ex <= 2046);
  return W == 0 ? 0.0 : __longlong_as_double(bits + ((long long)E << 52));
}

template <int NCH, bool TMR, bool PRE = false>
__device__ __forceinline__ void window_out(const long long* rw, int o0, const PushArgs& a, const TileJob& j,
                                           const long long* s0_pre, const int* fe_pre);

template <int NCH, bool TMR, bool PRE = false>
__device__ __forceinline__ void push_chunk(const int* vals, int o0, const PushArgs& a, const TileJob& j,
                                           const long long* s0_pre = nullptr, const int* fe_pre = nullptr) {
  static_assert(!TMR || NCH == 16, "TMEM chunks are 32 columns");
  int vv[NCH];
  if (!j.cplx) {
#pragma unroll
    for (int i = 0; i < NCH; ++i) vv[i] = vals[i];
  } else {
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
      const int other = __shfl_xor_sync(0xffffffffu, vals[2 * i + 1], 1);
      vv[i] = a.odd ? (vals[2 * i] + other) : (vals[2 * i] - other);
    }
  }
  long long rw[NCH];
  if (!(a.first && a.wstart)) {
    long long ro[NCH];
    if (TMR) {
      uint32_t t[32];
      tmem_ld32(a.rtm + 2 * o0, t);
      tmem_ld_wait();
#pragma unroll
      for (int i = 0; i < NCH; ++i) ro[i] = (long long)(((unsigned long long)t[2 * i + 1] << 32) | t[2 * i]);
    } else {
#pragma unroll
      for (int i = 0; i < NCH; ++i) ro[i] = a.Ra[(size_t)(o0 + i) * BM];
    }
#pragma unroll
    for (int i = 0; i < NCH; ++i) rw[i] = a.first ? (long long)((unsigned long long)ro[i] << 7) + vv[i] : ro[i] + vv[i];
  } else {
#pragma unroll
    for (int i = 0; i < NCH; ++i) rw[i] = vv[i];
  }
  window_out<NCH, TMR, PRE>(rw, o0, a, j, s0_pre, fe_pre);
}

// The part of a push after the window value: store the active window (plain), spill the first
// window (spill), close a later window into the FP64 partial (close), or round and write C
// (final), for outputs o0 .. o0+NCH-1 whose window values are rw.
template <int NCH, bool TMR, bool PRE>
__device__ __forceinline__ void window_out(const long long* rw, int o0, const PushArgs& a, const TileJob& j,
                                           const long long* s0_pre, const int* fe_pre) {
  if (a.kind == kPlain) {
    if (TMR) {
      uint32_t t[32];
#pragma unroll
      for (int i = 0; i < NCH; ++i) {
        t[2 * i] = (uint32_t)(unsigned long long)rw[i];
        t[2 * i + 1] = (uint32_t)((unsigned long long)rw[i] >> 32);
      }
      tmem_st32(a.rtm + 2 * o0, t);
      tmem_st_wait();
    } else {
#pragma unroll
      for (int i = 0; i < NCH; ++i) a.Ra[(size_t)(o0 + i) * BM] = rw[i];
    }
    return;
  }
  if (a.kind == kSpill) {
#pragma unroll
    for (int i = 0; i < NCH; ++i) a.S0[(size_t)(o0 + i) * BM] = rw[i];
    return;
  }
  long long s0[NCH];
  int fe[NCH];
  if (PRE) {
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
      s0[i] = s0_pre[i];
      fe[i] = fe_pre[i];
    }
  } else {
    prefetch_close<NCH>(a, j, o0, s0, fe);
  }
  // C is written with evict-first (streaming) stores: it is not read again by this launch, and
  // normal stores would displace digit-plane lines that the next groups read again from L2.
  // RN of the exact sum: for one or two windows all NCH outputs go through the branch-free
  // rounding together, and only results outside the normal range take the general path
  // (in batches of RB outputs, to bound the registers live at once)
  constexpr int RB = NCH < 8 ? NCH : 8;
  const int64_t c0 = j.cplx ? (a.gcol0 >> 1) + o0 : a.gcol0 + o0;
#pragma unroll
  for (int i0 = 0; i0 < NCH; i0 += RB) {
    double tv[RB];
    if (a.widx == 0 && a.kind == kFinal) {
      // a single window: one conversion per output
      unsigned bad = 0;
#pragma unroll
      for (int i = 0; i < RB; ++i) {
        bool ok;
        tv[i] = rn_single(rw[i0 + i], a.ebase + fe[i0 + i], ok);
        bad |= ok ? 0u : 1u << i;
      }
      if (bad != 0) {
#pragma unroll
        for (int i = 0; i < RB; ++i)
          if ((bad >> i) & 1u) tv[i] = final_val(0, rw[i0 + i], 0, a.wlen, a.ebase + fe[i0 + i]);
      }
    } else if (a.widx <= 1) {
      const bool close = a.kind == kClose;
      unsigned bad = 0;
#pragma unroll
      for (int i = 0; i < RB; ++i) {
        bool ok;
        tv[i] = rn_windows(a.widx == 0 ? 0ll : s0[i0 + i], rw[i0 + i], 7 * a.wlen, close ? 0 : a.ebase + fe[i0 + i], ok);
        bad |= ok ? 0u : 1u << i;
      }
      if (bad != 0) {
#pragma unroll
        for (int i = 0; i < RB; ++i)
          if ((bad >> i) & 1u)
            tv[i] = close ? __longlong_as_double(close_val(s0[i0 + i], rw[i0 + i], a.widx, a.wlen))
                          : final_val(s0[i0 + i], rw[i0 + i], a.widx, a.wlen, a.ebase + fe[i0 + i]);
      }
    } else {
#pragma unroll
      for (int i = 0; i < RB; ++i)
        tv[i] = a.kind == kClose ? __longlong_as_double(close_val(s0[i0 + i], rw[i0 + i], a.widx, a.wlen))
                                 : final_val(s0[i0 + i], rw[i0 + i], a.widx, a.wlen, a.ebase + fe[i0 + i]);
    }
    if (a.kind == kClose) {
#pragma unroll
      for (int i = 0; i < RB; ++i) a.S0[(size_t)(o0 + i0 + i) * BM] = __double_as_longlong(tv[i]);
      continue;
    }
    if (!j.cplx) {
      // the bound and the pointer in few instructions: 64-bit products per output cost 2%
      // (6000 x 6000 x 192 644 -> 629 us)
      const int left = a.row_ok ? (int)min((int64_t)RB, j.cols - (c0 + i0)) : 0;
      double* cp = j.C + a.orow + (c0 + i0) * j.ldc;
      if (a.unit_ab) {
#pragma unroll
        for (int i = 0; i < RB; ++i, cp += j.ldc)
          if (i < left) __stcs(cp, tv[i]);
      } else {
#pragma unroll
        for (int i = 0; i < RB; ++i, cp += j.ldc)
          if (i < left) __stcs(cp, j.beta_zero ? j.a0 * tv[i] : fma(j.a0, tv[i], j.b0 * *cp));
      }
    } else {
#pragma unroll
      for (int i = 0; i < RB; ++i) {
        const int64_t jc = c0 + i0 + i;
        const bool ok = a.row_ok && jc < j.n;
        const double part = ok ? tv[i] : 0.0;
        const double partner = __shfl_xor_sync(0xffffffffu, part, 1);
        if (ok) {
          double* cp = j.C + 2 * (a.orow + jc * j.ldc);
          if (a.unit_ab) {
            __stcs(cp + (a.odd ? 1 : 0), part);
          } else {
            const double tr = a.odd ? partner : part, ti = a.odd ? part : partner;
            double re = fma(j.a0, tr, -(j.a1 * ti));
            double im = fma(j.a0, ti, j.a1 * tr);
            if (!j.beta_zero) {
              const double cr = cp[0], ci = cp[1];
              re += fma(j.b0, cr, -(j.b1 * ci));
              im += fma(j.b0, ci, j.b1 * cr);
            }
            __stcs(cp + (a.odd ? 1 : 0), a.odd ? im : re);
          }
        }
      }
    }
  }
}

// Bounded wait used during teardown after an abort (ignores the abort flag).
__device__ __forceinline__ void drain_wait(uint64_t* bar, uint32_t parity) {
  long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (clock64() - t0 > OZG_WAIT_CYCLES) return;
  }
}

}  // namespace
}  // namespace ozg
