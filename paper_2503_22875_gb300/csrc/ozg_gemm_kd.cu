// K2 + K3 on difference planes: the slice products with one multiplication per unordered plane
// pair.  A group sum G_g = sum_{p+q=g} A_p B_q pairs (p, q) with (q, p), and
//   A_p B_q + A_q B_p = A_p B_p + A_q B_q + (A_p - A_q)(B_q - B_p),
// so with D_p = A_p B_p and M_g = sum_{p<q, p+q=g} (A_p - A_q)(B_q - B_p),
//   G_g = M_g + sum_{p=1}^{g-1} D_p          (the diagonal pair p = g/2 is D_p itself):
// s + floor(s^2 / 4) products instead of s (s + 1) / 2 (19 instead of 28 at s = 7, 29 instead of
// 45 at s = 9) for the same integers.  The digits of an entry share its sign, so a difference of
// two digits is again in [-127, 127]: the differences are exact in FP16, a chain of 1024 products
// stays below 2^24, and every bound of the plane-by-plane kernels holds unchanged.  The split
// writes the differences as planes of their own (kd_plane_base); product j multiplies plane j of A
// with plane j of B, so no plane is used twice and no tile is reused between products.
//
// That makes the operand traffic the limit of small tiles: a 128 x 128 tile needs 32 KB per 131 ns
// of MMA, and an SM receives about 125 B/ns.  So a tile is 256 x 256 on a CTA pair
// (tcgen05.mma.cta_group::2, M = 256, N = 256): each CTA stages its 128 rows of A and half of the B
// columns, 32 KB per 262 ns, and holds 128 x 256 accumulators, double buffered over all of TMEM.
// Narrower pair tiles do not pay: an N = 128 pair MMA takes 58 ns against 66 for N = 256.
//
// A window covers a run of groups.  D_p enters it with the weight sum_{g > p} 128^(gend - g) over
// the window's groups, M_g with 128^(gend - g): one 64-bit multiply-add per output and chain.  With
// two windows the second starts from R sum_g 128^(gend - g), R = the sum of the first window's D_p
// (int32, in the CTA's L2-resident scratch; the first window is kept as short as possible).
// Complex tiles have half as many outputs as accumulators, and their window words live in the
// epilogue's registers.  Real tiles need 256 KB per CTA for them: 48 of a thread's 128 outputs keep
// theirs in registers, the others collect an int32 sum per pass and add it to their words in L2 by
// reductions (red.u64; an SM sends 32 B/clk, so every word less in a push counts).  Holding them all
// on chip measured slower in four layouts, each of which costs a second N = 256 accumulator: 2048^3
// s = 8 0.36 - 0.38 ms against 0.33, 8192^3 s = 7 13.8 - 14.7 against 11.5 - 12.4.
//
// Against the stacked kernel (launch): 8192^3 s = 7 17.0 -> 11.8 ms (power limited: the clock falls
// to 1.5 GHz under digit operands, so the third fewer products is the gain), 2048^3 s = 8 0.41 ->
// 0.33 ms, complex 3616^3 s = 7 6.4 -> 4.3 ms.
#include <utility>

#include "ozg_gemm_dev.cuh"

namespace ozg {
namespace {

namespace kd {
constexpr int NE = 6;                   // stage ring: one 128 x 64 sub-tile of A and of B per entry
constexpr int TM = 2 * BM, TN = 256;    // output tile of a CTA pair
constexpr uint32_t SLOT = BM * BK * 2;  // 16 KB
constexpr uint32_t A_OFF = 0, B_OFF = NE * SLOT;
constexpr size_t SMEM = (size_t)2 * NE * SLOT + 1024;
constexpr uint32_t IDESC = umma_idesc_f16_f32(TM, TN);
constexpr int CHAIN_STAGES = CHAIN_K / BK;
constexpr int NCOL = 128;               // accumulator columns per epilogue thread
template <bool CPLX>
constexpr int NOUT = CPLX ? NCOL / 2 : NCOL;  // its outputs
template <bool CPLX>
constexpr int NREG = CPLX ? NOUT<true> : 48;  // outputs whose window words are in registers
template <bool CPLX>
constexpr int NSUM = NOUT<CPLX> - NREG<CPLX> > 0 ? NOUT<CPLX> - NREG<CPLX> : 1;  // int32 sums
constexpr uint32_t DSLOT = SLOT >> 4;
static_assert(SMEM <= 227 * 1024, "stage ring");
static_assert(SMEM < (1u << 18), "descriptor start addresses stay within their 14-bit field");
}  // namespace kd

// Chains of a pass of n stages: as many as 1024 products per chain require, of equal length (a
// short last chain would drain faster than it computes).
__device__ __forceinline__ int kd_chains(int n) { return (n + kd::CHAIN_STAGES - 1) / kd::CHAIN_STAGES; }
// Groups of the first window: all of them when they fit one, else as few as the second leaves.
__device__ __forceinline__ int kd_len0(int s, int win) { return s <= win ? s : s - win; }

// The four K = 16 MMAs of one 64-wide k sub-tile; the first overwrites the accumulator when it
// starts a chain.
__device__ __forceinline__ void kd_mma4(uint32_t dt, uint32_t da, uint32_t db, bool accumulate) {
  umma_f16_pair_lo(dt, da, db, kd::IDESC, accumulate ? 1u : 0u);
#pragma unroll
  for (int k16 = 1; k16 < BK / 16; ++k16) umma_f16_pair_lo(dt, da + 2 * k16, db + 2 * k16, kd::IDESC, 1u);
}

// One finished chain.  The thread's first NREG outputs keep their window words in registers:
// W += v w (and R += v for the D products in the first of two windows; rmode 1: first store, 2:
// add).  The others add to int32 sums (keep = 1) or start them (keep = 0; a separate reset would
// double their registers).  The accumulator is released once its values are in registers.
template <bool CPLX>
__device__ __forceinline__ void kd_drain(unsigned long long (&W)[kd::NREG<CPLX>], int (&Gr)[kd::NSUM<CPLX>],
                                         int keep, KdWeight w, uint32_t acc, bool odd, int* Rp, int rmode,
                                         uint32_t release_bar, int lane) {
  constexpr int A = CPLX ? 32 : 16, NR = kd::NREG<CPLX>;  // A: accumulator columns of 16 outputs
#pragma unroll
  for (int c = 0; c < kd::NCOL / A; ++c) {
    uint32_t a[A];
#pragma unroll
    for (int q = 0; q < A / 16; ++q) tmem_ld16(acc + A * c + 16 * q, *reinterpret_cast<uint32_t(*)[16]>(a + 16 * q));
    tmem_ld_wait();
    if (c == kd::NCOL / A - 1) {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_remote(release_bar);  // the leader's MMA warp waits on it
    }
    int v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      if (!CPLX) {
        v[i] = __float2int_rn(__uint_as_float(a[i & (A - 1)]));
      } else {  // even lanes Re = P_rr - P_ii, odd lanes Im = P_ir + P_ri
        const int x = __float2int_rn(__uint_as_float(a[(2 * i) & (A - 1)]));
        const int y = __shfl_xor_sync(0xffffffffu, __float2int_rn(__uint_as_float(a[(2 * i + 1) & (A - 1)])), 1);
        v[i] = odd ? x + y : x - y;
      }
      const int o = 16 * c + i;
      if (o < NR)
        W[o < NR ? o : 0] = kd_mac(W[o < NR ? o : 0], v[i], w);
      else
        Gr[o < NR ? 0 : o - NR] = Gr[o < NR ? 0 : o - NR] * keep + v[i];
    }
    if (16 * c < NR) {
      if (rmode == 1) {
#pragma unroll
        for (int i = 0; i < 16; ++i) Rp[(size_t)(16 * c + i) * BM] = v[i];
      } else if (rmode == 2) {
#pragma unroll
        for (int i = 0; i < 16; ++i) atomicAdd(Rp + (size_t)(16 * c + i) * BM, v[i]);
      }
    }
  }
}

// The int32 sums of a pass enter a window of the CTA's scratch: W += v w, by reductions in L2 (each
// word belongs to one thread; nothing is read back before the tile's end), or W = v w on the
// window's first pass.
template <bool FIRST, int N, int... O>
__device__ __forceinline__ void kd_push_all(const int (&Gr)[N], long long* W, KdWeight w,
                                            std::integer_sequence<int, O...>) {
  auto one = [&](int v, auto off) {
    const unsigned long long x = kd_mac(0, v, w);
    if (FIRST)
      asm volatile("st.global.cg.u64 [%0 + %2], %1;" ::"l"(W), "l"(x), "n"(decltype(off)::value * BM * 8) : "memory");
    else
      asm volatile("red.relaxed.gpu.global.add.u64 [%0 + %2], %1;" ::"l"(W), "l"(x), "n"(decltype(off)::value * BM * 8)
                   : "memory");
  };
  (one(Gr[O], std::integral_constant<int, O>()), ...);
}
template <int N>
__device__ __forceinline__ void kd_push(const int (&Gr)[N], long long* W, KdWeight w, bool first) {
  if (first)
    kd_push_all<true>(Gr, W, w, std::make_integer_sequence<int, N>());
  else
    kd_push_all<false>(Gr, W, w, std::make_integer_sequence<int, N>());
}

template <bool CPLX>
__device__ __forceinline__ void kd_body(const CUtensorMap* tmA, const CUtensorMap* tmB, const GemmArgs* P) {
  using namespace kd;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t bar_full[NE], bar_empty[NE], bar_accf[2], bar_acce[2], bar_done;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;

  int* status = P->status;
  const int ntiles = (int)(((P->rows + TM - 1) / TM) * ((P->cols + TN - 1) / TN));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // rank 0 (the leader) owns the stage-full and accumulator-empty barriers that both CTAs arrive at,
  // and issues the pair MMAs
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  const int nunits = (int)(gridDim.x / 2), unit = (int)(blockIdx.x / 2);
  if (threadIdx.x == 0) {
    for (int i = 0; i < NE; ++i) {
      mbar_init(&bar_full[i], 2);  // each CTA's producer announces its bytes
      mbar_init(&bar_empty[i], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&bar_accf[b], 1);
      mbar_init(&bar_acce[b], 2 * EPI_WARPS);
    }
    mbar_init(&bar_done, 1);
    abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(tmA);
    tma_prefetch_desc(tmB);
  }
  if (warp == 1) tmem_alloc_pair(&tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  __syncwarp();
  cluster_sync_all();  // the peer's barriers are initialised before any remote arrival
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  volatile int* abort_p = &abort_flag;

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REG_PRODUCER));
    if (warp == 0) {
      // ---------------------------------------------------------------- TMA producer
      if (lane == 0) {
        uint32_t e = 0, eph = 0;
        long long issued = 0;
        for (int t = unit; t < ntiles; t += nunits) {
          const TileJob j = get_job<256, 1, false, false, TM>(t, tmA, tmB, P, nullptr);
          // this CTA's 128 rows of A and its half of the B columns
          const int arow = j.tm * TM + (int)rank * BM, brow = j.tn * TN + (int)rank * 128;
          const int nplanes = kd_plane_base(j.s + 1);
          for (int pl = 0; pl < nplanes; ++pl)
            for (int kb = 0; kb < j.KB; ++kb) {
              if (!mbar_wait(&bar_empty[e], eph ^ 1, abort_p, status)) goto producer_done;
              // both CTAs' copies complete on the leader's stage barrier
              const uint32_t fbar = mapa_shared(&bar_full[e], 0);
              mbar_arrive_expect_tx_remote(fbar, 2 * SLOT);
              tma_load_3d_pair(j.tmA, fbar, smem + A_OFF + e * SLOT, kb * BK, arow, pl);
              tma_load_3d_pair(j.tmB, fbar, smem + B_OFF + e * SLOT, kb * BK, brow, pl);
              ++issued;
              if (++e == NE) {
                e = 0;
                eph ^= 1;
              }
            }
        }
      producer_done:
        if (*abort_p) {
          if (leader) {  // wait (bounded) for the copies still in flight
            uint32_t st = e, ph = eph;
            for (long long i = 0; i < NE && i < issued; ++i) {
              if (st == 0) {
                st = NE - 1;
                ph ^= 1;
              } else {
                --st;
              }
              drain_wait(&bar_full[st], ph);
            }
          } else {  // the follower's copies complete on the leader's barriers: give them time to land
            const long long t0 = clock64();
            while (clock64() - t0 < 2000000ll) {
            }
          }
        }
      }
    } else if (warp == 1) {
      // ---------------------------------------------------------------- MMA issuer (the leader's warp)
      // The whole warp runs the loop, so that addresses and descriptors stay in uniform registers;
      // one elected lane issues.
      if (leader) {
        const bool lead = elect_one();
        uint32_t e = 0, eph = 0;
        uint32_t acc_par = 0;  // bit b: parity of the next use of TMEM buffer b
        int buf = 0;
        const uint32_t dA0 = (uint32_t)umma_desc_sw128(smem + A_OFF), dB0 = (uint32_t)umma_desc_sw128(smem + B_OFF);
        for (int t = unit; t < ntiles; t += nunits) {
          const TileJob j = get_job<256, 1, false, false, TM>(t, tmA, tmB, P, nullptr);
          // passes: D_1, then D_t and M_{t+1} for t = 2 .. s
          for (int pass = 1; pass < 2 * j.s; ++pass) {
            const int np = (pass == 1 || !(pass & 1)) ? 1 : ((pass >> 1) + 1) / 2;
            int left = np * j.KB, nch = kd_chains(left);
            for (; nch > 0; --nch) {
              const int c = (left + nch - 1) / nch;
              left -= c;
              if (!mbar_wait_warp(&bar_acce[buf], ((acc_par >> buf) & 1) ^ 1, abort_p, status)) goto mma_done;
              const uint32_t dt = tmem + (uint32_t)(buf * TN);
              for (int i = 0; i < c; ++i) {
                if (!mbar_wait_warp(&bar_full[e], eph, abort_p, status)) goto mma_done;
                tc_fence_after();
                if (lead) {
                  kd_mma4(dt, dA0 + e * DSLOT, dB0 + e * DSLOT, i != 0);
                  umma_commit_pair_mc(&bar_empty[e], 3);  // the stage is free in both CTAs
                }
                if (++e == NE) {
                  e = 0;
                  eph ^= 1;
                }
              }
              if (lead) umma_commit_pair_mc(&bar_accf[buf], 3);  // the chain is ready in both CTAs' TMEM
              acc_par ^= 1u << buf;
              buf ^= 1;
            }
          }
        }
      mma_done:
        if (lead) {
          umma_commit_pair_mc(&bar_done, 1);
          drain_wait(&bar_done, 0);
        }
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REG_EPILOGUE));
    const int ew = warp - 4;
    const int quad = warp & 3;
    const int chalf = ew >> 2;
    const int r = quad * 32 + lane;
    uint32_t acc_par = 0;
    int buf = 0;
    // the CTA's scratch: two window words per output
    long long* scratch = reinterpret_cast<long long*>(P->Rws + (size_t)blockIdx.x * BM * TN * 2);
    const bool odd = (lane & 1) != 0;
    const uint32_t tl = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(chalf * NCOL);
    const uint32_t rel[2] = {mapa_shared(&bar_acce[0], 0), mapa_shared(&bar_acce[1], 0)};
    for (int t = unit; t < ntiles; t += nunits) {
      TileJob j = get_job<256, 1, false, false, TM>(t, tmA, tmB, P, nullptr);
      j.cplx = CPLX;
      const int s = j.s;
      const int win = window_len(s, (int64_t)j.KB * BK, CPLX);
      constexpr int N = NOUT<CPLX>, NR = NREG<CPLX>;
      // scratch words of this thread's outputs: first window, second window (R, int32, in the
      // place of the second window's for the outputs kept in registers)
      long long* W0 = scratch + (size_t)(chalf * N) * BM + r;
      long long* W1 = W0 + (size_t)BM * TN;
      int* Rp = reinterpret_cast<int*>(W1 - r) + r;
      const int len0 = kd_len0(s, win);  // groups of the first window
      const bool two = len0 < s;
      constexpr int kFold = 64;          // chains per push: the int32 sums stay below 2^31
      unsigned long long W[NR];
#pragma unroll
      for (int o = 0; o < NR; ++o) W[o] = 0;
      int Gr[NSUM<CPLX>] = {};
      int entered = 0;  // bit w: a push has entered window w
      for (int tb = 1; tb <= s; ++tb) {
        if (two && tb == len0 + 1) {  // the second window starts: spill the first, take R along
          const unsigned long long geom = kd_geom(s - tb);
#pragma unroll
          for (int o = 0; o < NR; ++o) {
            W0[(size_t)o * BM] = (long long)W[o];
            W[o] = (unsigned long long)(long long)__ldcg(Rp + (size_t)o * BM) * geom;
          }
        }
        for (int m = 0; m < (tb > 1 ? 2 : 1); ++m) {  // D_tb, then M_{tb+1}
          const int blk = tb <= len0 ? len0 : s;       // the window's last block
          const KdWeight w = kd_weight(m == 0 ? kd_geom(blk - tb) : 1ull << (7 * (blk - tb)));
          int nch = kd_chains((m == 0 ? 1 : tb / 2) * j.KB);
          for (int nf = 0, keep = 0, ch = 0; nch > 0; --nch, ++ch) {
            const int rmode = (m == 0 && two && tb <= len0) ? (tb == 1 && ch == 0 ? 1 : 2) : 0;
            if (!mbar_wait(&bar_accf[buf], (acc_par >> buf) & 1, abort_p, status)) goto epi_done;
            tc_fence_after();
            kd_drain<CPLX>(W, Gr, keep, w, tl + (uint32_t)(buf * TN), odd, Rp, rmode, buf ? rel[1] : rel[0], lane);
            acc_par ^= 1u << buf;
            buf ^= 1;
            if (NR == N) continue;
            keep = 1;
            if (nch > 1 && ++nf < kFold) continue;
            keep = nf = 0;
            // group tb + 1 and (D) the later groups of its window; a D of the first window also
            // enters every group of the second
#pragma unroll 1
            for (int wi = tb > len0 ? 1 : 0; wi <= (two && (tb > len0 || m == 0) ? 1 : 0); ++wi) {
              const KdWeight wp = wi == 1 && tb <= len0 ? kd_weight(kd_geom(s - len0 - 1)) : w;
              // a single window's words are W0's
              kd_push(Gr, (wi ? W1 : W0) + (size_t)NR * BM, wp, !((entered >> wi) & 1));
              entered |= 1 << wi;
            }
          }
        }
      }
      const int64_t grow = (int64_t)j.tm * TM + (int64_t)rank * BM + r;
      const bool row_ok = grow < j.rows;
      PushArgs pa;
      pa.gcol0 = (int64_t)j.tn * TN + chalf * NCOL;
      pa.orow = CPLX ? (grow >> 1) : grow;
      pa.row_ok = row_ok;
      pa.unit_ab = j.beta_zero && j.a0 == 1.0 && j.a1 == 0.0;
      pa.odd = odd;
      pa.ebase = (row_ok ? j.e[pa.orow] : 0) - 7 * (s + 1);
      int nfin = N;  // real tiles finish only the chunks that reach into C
      if (!CPLX) {
        int nvalid = (int)max((int64_t)0, min((int64_t)N, j.cols - pa.gcol0));
        if ((int64_t)j.tm * TM + (int64_t)rank * BM + quad * 32 >= j.rows) nvalid = 0;
        nfin = (nvalid + 7) & ~7;
      }
      // round and write C, the next chunk's window words loaded while this one is rounded
      int fcol[4];  // the column exponents of this warp's outputs, handed out by shuffles
      {
        const int64_t c0 = CPLX ? (pa.gcol0 >> 1) : pa.gcol0;
        const int64_t climit = CPLX ? j.n : j.cols;
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const int64_t c = c0 + h * 32 + lane;
          fcol[h] = (c < climit && (h < 2 || !CPLX)) ? __ldg(j.f + c) : 0;
        }
      }
      pa.widx = two ? 1 : 0;
      pa.wlen = two ? s - len0 : s;
      pa.kind = kFinal;
      auto column_exponents = [&](int o, int(&fe)[8]) {
        const int fsrc = o < 64 ? (o < 32 ? fcol[0] : fcol[1]) : (o < 96 ? fcol[2] : fcol[3]);
#pragma unroll
        for (int i = 0; i < 8; ++i) fe[i] = __shfl_sync(0xffffffffu, fsrc, (o + i) & 31);
      };
      // the outputs in registers; the array is rotated after each chunk, so that every index stays
      // a compile-time constant
      long long n0[8];  // the next chunk's first-window words, loaded while a chunk is rounded
      auto load0 = [&](int o) {
#pragma unroll
        for (int i = 0; i < 8; ++i) n0[i] = two ? __ldcg(W0 + (size_t)(o + i) * BM) : 0ll;
      };
      if (nfin > 0) load0(0);
#pragma unroll 1
      for (int o = 0; o < min(nfin, NR); o += 8) {
        long long s0c[8], rw[8];
        int fe[8];
        column_exponents(o, fe);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          s0c[i] = n0[i];
          rw[i] = (long long)W[i];
        }
        if (o + 8 < nfin) load0(o + 8);
        window_out<8, false, true>(rw, o, pa, j, s0c, fe);
#pragma unroll
        for (int c = 0; c < NR - 8; ++c) W[c] = W[c + 8];
      }
      if (NR < N) {
        const long long* Wl = two ? W1 : W0;  // the last window's words
        long long n1[8];
        auto load1 = [&](int o) {
#pragma unroll
          for (int i = 0; i < 8; ++i) n1[i] = __ldcg(Wl + (size_t)(o + i) * BM);
        };
        if (NR < nfin) load1(NR);
#pragma unroll 1
        for (int o = NR; o < nfin; o += 8) {
          long long s0c[8], rw[8];
          int fe[8];
          column_exponents(o, fe);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            s0c[i] = n0[i];
            rw[i] = n1[i];
          }
          if (o + 8 < nfin) {
            load0(o + 8);
            load1(o + 8);
          }
          window_out<8, false, true>(rw, o, pa, j, s0c, fe);
        }
      }
    }
  epi_done:;
  }

  tc_fence_before();
  __syncthreads();
  // neither CTA leaves (or frees TMEM) while the peer may still reach its shared memory or the
  // leader's MMAs its TMEM
  __syncwarp();
  cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, 512);
  }
}

// Both CTAs of a pair read the same flags, so a gated launch returns from both.
template <bool CPLX>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
    slice_gemm_kd_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                         const GemmArgs P) {
  pdl_wait();
  if (P.nonfinite != nullptr && *P.nonfinite) return;
  if (P.s_dev != nullptr && *P.s_dev > P.kd) return;  // no difference planes: the plane-by-plane launch runs
  kd_body<CPLX>(&tmA, &tmB, &P);
}

}  // namespace

int64_t kd_tiles(int64_t rows, int64_t cols) { return ((rows + kd::TM - 1) / kd::TM) * ((cols + kd::TN - 1) / kd::TN); }

cudaError_t prepare_kd_kernels() {
  const cudaError_t e =
      cudaFuncSetAttribute(slice_gemm_kd_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kd::SMEM);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(slice_gemm_kd_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kd::SMEM);
}

cudaError_t launch_slice_gemm_kd(const CUtensorMap& tmA, const CUtensorMap& tmB, const GemmArgs& a, cudaStream_t st) {
  if (a.grid <= 0) return cudaSuccess;
  if (a.grid % 2) return cudaErrorInvalidValue;  // whole clusters
  if (a.cplx)
    launch_pdl(slice_gemm_kd_kernel<true>, a.grid, THREADS, kd::SMEM, st, tmA, tmB, a);
  else
    launch_pdl(slice_gemm_kd_kernel<false>, a.grid, THREADS, kd::SMEM, st, tmA, tmB, a);
  return cudaGetLastError();
}

}  // namespace ozg
