// K1: per-row power-of-two scale and INT8-range digit planes (the split step of the Ozaki
// scheme, Sec. 2.2).  Row i of op(X) gets e_i = frexp exponent of max_l |x_il|; digit t of
// x is the t-th base-2^7 digit of |x| 2^-e_i taken by truncation, with the sign of x:
//   d_t = sign(x) * (floor(|x| 2^{7s - e_i}) >> 7(s - t)) & 127.
// Only integer bit operations are used (FP64 arithmetic is slow on this part and not
// needed: the fixed-point value is the 53-bit significand shifted).  HBM-bound: one read of
// op(X) for the maxima, one read plus s fp16 writes for the digits.
#include "../../include/ozg.h"
#include "ozg_internal.h"
#include "ozg_split_dev.cuh"

static_assert(ozg::kMaxPlanes == OZG_MAX_SLICES, "digit planes of the widest split");

namespace ozg {
namespace {

// Digit planes t_lo .. t_hi a launch writes: t_lo = *from + 1 (else 1), t_hi = *to (else s);
// nothing when *gate is non-zero.
struct PlaneRange {
  const int* from;
  const int* to;
  const int* gate;
  int kd, diff;
  __device__ __forceinline__ bool resolve(int s, int& lo, int& hi) const {
    if (gate != nullptr && *gate) return false;
    lo = from != nullptr ? *from + 1 : 1;
    hi = to != nullptr ? *to : s;
    return lo <= hi;
  }
};

// The planes lo .. hi of eight consecutive elements b (bit patterns) of a row with exponent e.
template <int KD>
__device__ __forceinline__ void store_planes8(const uint64_t (&b)[8], int e, int lo, int hi, __half* out,
                                              int64_t plane, const PlaneRange& pr) {
  DigitSrc ds[8];
  if (KD && pr.diff != 0 && hi <= pr.kd) {
    if (hi <= 9) {
#pragma unroll
      for (int j = 0; j < 8; ++j) ds[j] = digit_src_first(b[j], e);
      store_difference_planes<9>(ds, lo, hi, out, plane, pr.diff < 0);
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) ds[j] = digit_src(b[j], e);
      store_difference_planes<kKdMax>(ds, lo, hi, out, plane, pr.diff < 0);
    }
    return;
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) ds[j] = digit_src(b[j], e);
  if (KD)
    store_digit_planes_kd<kMaxPlanes>(ds, lo, hi, out, plane, pr.kd);
  else
    store_digit_planes<kMaxPlanes>(ds, lo, hi, out, plane);
}

__device__ __forceinline__ void flag_nonfinite(uint64_t absbits, int* nonfinite) {
  if (absbits >= kInfBits) atomicExch(nonfinite, 1);
}

// ---------------------------------------------------------------- row maxima, contiguous rows
// one warp per row; lanes stride along l
__global__ void rowmax_contig(const double* __restrict__ X, int64_t ld, int64_t rows, int64_t k, int cplx,
                              unsigned long long* __restrict__ maxbits, int* nonfinite) {
  pdl_entry();
  int64_t row = (int64_t)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  int lane = threadIdx.x % 32;
  if (row >= rows) return;
  unsigned long long mx = 0;
  if (!cplx) {
    const uint64_t* p = reinterpret_cast<const uint64_t*>(X) + row * ld;
    for (int64_t l = lane; l < k; l += 32) {
      uint64_t v = __ldg(p + l) & kAbsMask;
      mx = v > mx ? v : mx;
    }
  } else {
    const ulonglong2* p = reinterpret_cast<const ulonglong2*>(X) + row * ld;
    for (int64_t l = lane; l < k; l += 32) {
      ulonglong2 v = __ldg(p + l);
      uint64_t a = v.x & kAbsMask, b = v.y & kAbsMask;
      a = a > b ? a : b;
      mx = a > mx ? a : mx;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    unsigned long long t = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = t > mx ? t : mx;
  }
  if (lane == 0) {
    maxbits[row] = mx;
    flag_nonfinite(mx, nonfinite);
  }
}

// ---------------------------------------------------------------- row maxima, strided rows
// thread per row (consecutive rows are contiguous in memory), grid.y splits k; atomicMax merges
__global__ void rowmax_strided(const double* __restrict__ X, int64_t ld, int64_t rows, int64_t k, int64_t kchunk,
                               int cplx, unsigned long long* __restrict__ maxbits, int* nonfinite) {
  pdl_entry();
  int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= rows) return;
  int64_t l0 = (int64_t)blockIdx.y * kchunk, l1 = min(k, l0 + kchunk);
  unsigned long long mx = 0;
  if (!cplx) {
    const uint64_t* p = reinterpret_cast<const uint64_t*>(X);
    for (int64_t l = l0; l < l1; ++l) {
      uint64_t v = __ldg(p + row + l * ld) & kAbsMask;
      mx = v > mx ? v : mx;
    }
  } else {
    const ulonglong2* p = reinterpret_cast<const ulonglong2*>(X);
    for (int64_t l = l0; l < l1; ++l) {
      ulonglong2 v = __ldg(p + row + l * ld);
      uint64_t a = v.x & kAbsMask, b = v.y & kAbsMask;
      a = a > b ? a : b;
      mx = a > mx ? a : mx;
    }
  }
  if (mx) {
    atomicMax(&maxbits[row], mx);
    flag_nonfinite(mx, nonfinite);
  }
}

// ---------------------------------------------------------------- row maxima, both operands of a small call
// One launch whose blocks have eight loads in flight per thread: 32 rows x 64 k of a strided operand
// (lanes along the rows, the eight warps along k), 8 rows x 256 k of a contiguous one (a warp per
// row).  Latency bound: a launch per operand with one load in flight per thread took 4.1 + 3.7 us at
// 256 x 256, 9.1 + 9.1 at 768 x 768 complex.  Partial maxima merge by atomicMax.
constexpr int kRpLoads = 8, kRpStridedK = 8 * kRpLoads, kRpContigK = 32 * kRpLoads;
template <int CPLX>
__device__ __forceinline__ uint64_t abs_elem(const double* X, int64_t idx) {
  if (!CPLX) return __ldg(reinterpret_cast<const uint64_t*>(X) + idx) & kAbsMask;
  const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2*>(X) + idx);
  const uint64_t a = v.x & kAbsMask, b = v.y & kAbsMask;
  return a > b ? a : b;
}
template <int CPLX>
__global__ void __launch_bounds__(256) rowmax_pair(const SplitArgs a, const SplitArgs b, unsigned blocks_a) {
  pdl_entry();
  __shared__ unsigned long long red[8][32];
  const bool first = blockIdx.x < blocks_a;
  const SplitArgs& J = first ? a : b;
  const unsigned block = first ? blockIdx.x : blockIdx.x - blocks_a;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t rows = J.rows, k = J.k, ld = J.ld;
  uint64_t v[kRpLoads], mx = 0;
  if (J.strided) {
    const unsigned kt = (unsigned)((k + kRpStridedK - 1) / kRpStridedK);
    const int64_t row = (int64_t)(block / kt) * 32 + lane, l0 = (int64_t)(block % kt) * kRpStridedK + w;
#pragma unroll
    for (int i = 0; i < kRpLoads; ++i) {
      const int64_t l = l0 + 8 * i;
      v[i] = row < rows && l < k ? abs_elem<CPLX>(J.X, row + l * ld) : 0ull;
    }
#pragma unroll
    for (int i = 0; i < kRpLoads; ++i) mx = v[i] > mx ? v[i] : mx;
    red[w][lane] = mx;
    __syncthreads();
    if (w != 0) return;
#pragma unroll
    for (int i = 1; i < 8; ++i) mx = red[i][lane] > mx ? red[i][lane] : mx;
    if (row < rows && mx) {
      atomicMax(&J.maxbits[row], mx);
      flag_nonfinite(mx, J.nonfinite);
    }
  } else {
    const unsigned kt = (unsigned)((k + kRpContigK - 1) / kRpContigK);
    const int64_t row = (int64_t)(block / kt) * 8 + w, l0 = (int64_t)(block % kt) * kRpContigK + lane;
    if (row >= rows) return;
#pragma unroll
    for (int i = 0; i < kRpLoads; ++i) {
      const int64_t l = l0 + 32 * i;
      v[i] = l < k ? abs_elem<CPLX>(J.X, l + row * ld) : 0ull;
    }
#pragma unroll
    for (int i = 0; i < kRpLoads; ++i) mx = v[i] > mx ? v[i] : mx;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const uint64_t t = __shfl_xor_sync(0xffffffffu, mx, o);
      mx = t > mx ? t : mx;
    }
    if (lane == 0 && mx) {
      atomicMax(&J.maxbits[row], (unsigned long long)mx);
      flag_nonfinite(mx, J.nonfinite);
    }
  }
}

// ---------------------------------------------------------------- digits, contiguous rows
// thread per (row, group of 8 consecutive l); 16-byte stores per digit plane
template <int CPLX, int KD>
__device__ __forceinline__ void digits_contig(const SplitArgs& J, const PlaneRange& pr, int t_lo, int t_hi, unsigned block) {
  const double* X = J.X;
  const int64_t ld = J.ld, rows = J.rows, k = J.k, Kp = J.Kp, plane_rows = J.plane_rows;
  const int conj = J.conj;
  const unsigned long long* maxbits = J.maxbits;
  int32_t* exps = J.exps;
  __half* D = J.D;
  int64_t groups = (k + 7) / 8;
  int64_t gid = (int64_t)block * 256 + threadIdx.x;
  if (gid >= rows * groups) return;
  int64_t row = gid / groups, l0 = (gid % groups) * 8;
  int e = exponent_from_maxbits(maxbits[row]);
  if (l0 == 0 && t_lo == 1) exps[row] = e;
  const int nparts = CPLX ? 2 : 1;
  uint64_t bits[2][8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    int64_t l = l0 + j;
    if (CPLX) {
      ulonglong2 v = (l < k) ? __ldg(reinterpret_cast<const ulonglong2*>(X) + row * ld + l) : make_ulonglong2(0, 0);
      bits[0][j] = v.x;
      bits[1][j] = conj ? (v.y ^ 0x8000000000000000ull) : v.y;
    } else {
      bits[0][j] = (l < k) ? __ldg(reinterpret_cast<const uint64_t*>(X) + row * ld + l) : 0ull;
    }
  }
#pragma unroll
  for (int part = 0; part < nparts; ++part) {
    int64_t orow = CPLX ? 2 * row + part : row;
    store_planes8<KD>(bits[part], e, t_lo, t_hi, D + orow * Kp + l0, plane_rows * Kp, pr);
  }
}

// ---------------------------------------------------------------- digits, strided rows
// block: 32 rows x 64 l tile staged (transposed) through shared memory
template <int CPLX, int KD>
__device__ __forceinline__ void digits_strided(const SplitArgs& J, const PlaneRange& pr, int t_lo, int t_hi, unsigned block) {
  const double* X = J.X;
  const int64_t ld = J.ld, rows = J.rows, k = J.k, Kp = J.Kp, plane_rows = J.plane_rows;
  const int conj = J.conj;
  const unsigned long long* maxbits = J.maxbits;
  int32_t* exps = J.exps;
  __half* D = J.D;
  constexpr int TR = 32, TL = 64;
  constexpr int W = CPLX ? 2 : 1;
  __shared__ uint64_t tile[TL][TR * W + 1];
  const unsigned row_blocks = (unsigned)((rows + TR - 1) / TR);
  int64_t r0 = (int64_t)(block % row_blocks) * TR, l0 = (int64_t)(block / row_blocks) * TL;
  int tid = threadIdx.x;
  // load: thread -> (row = tid % 32, l = tid / 32 + 8 j)
  {
    int r = tid % TR;
    int64_t row = r0 + r;
    for (int j = 0; j < TL / 8; ++j) {
      int li = tid / TR + 8 * j;
      int64_t l = l0 + li;
      bool ok = row < rows && l < k;
      if (CPLX) {
        ulonglong2 v = ok ? __ldg(reinterpret_cast<const ulonglong2*>(X) + row + l * ld) : make_ulonglong2(0, 0);
        tile[li][2 * r] = v.x;
        tile[li][2 * r + 1] = conj ? (v.y ^ 0x8000000000000000ull) : v.y;
      } else {
        tile[li][r] = ok ? __ldg(reinterpret_cast<const uint64_t*>(X) + row + l * ld) : 0ull;
      }
    }
  }
  __syncthreads();
  // compute: thread -> (row = tid / 8, 8 consecutive l at (tid % 8) * 8)
  int r = tid / 8;
  int64_t row = r0 + r;
  int lg = (tid % 8) * 8;
  if (row >= rows || l0 + lg >= k) return;
  int e = exponent_from_maxbits(maxbits[row]);
  if (l0 + lg == 0 && t_lo == 1) exps[row] = e;
#pragma unroll
  for (int part = 0; part < W; ++part) {
    uint64_t b[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) b[j] = tile[lg + j][W * r + part];
    int64_t orow = CPLX ? 2 * row + part : row;
    store_planes8<KD>(b, e, t_lo, t_hi, D + orow * Kp + l0 + lg, plane_rows * Kp, pr);
  }
}

// The digits of one or both operands of a call: blocks 0 .. blocks_a - 1 work on a, the others on b.
// ROWS: the rows' layout, 0 contiguous, 1 strided, 2 either (one launch for operands of both kinds,
// which carries the registers and shared memory of the larger path).
template <int CPLX, int KD, int ROWS>
__global__ void __launch_bounds__(256) digits_kernel(const SplitArgs a, const SplitArgs b, unsigned blocks_a) {
  pdl_wait();
  const bool first = blockIdx.x < blocks_a;
  const SplitArgs& J = first ? a : b;
  const PlaneRange pr{J.plane_from, J.plane_to, J.gate, J.kd, J.diff};
  int t_lo, t_hi;
  if (!pr.resolve(J.s, t_lo, t_hi)) return;
  const unsigned block = first ? blockIdx.x : blockIdx.x - blocks_a;
  if (ROWS == 1 || (ROWS == 2 && J.strided))
    digits_strided<CPLX, KD>(J, pr, t_lo, t_hi, block);
  else
    digits_contig<CPLX, KD>(J, pr, t_lo, t_hi, block);
}

__global__ void digits_to_i8(const __half* __restrict__ D, int64_t planes_rows, int64_t k, int64_t Kp,
                             int8_t* __restrict__ out) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= planes_rows * k) return;
  int64_t r = i / k, l = i % k;
  out[i] = (int8_t)__half2int_rn(D[r * Kp + l]);
}

}  // namespace

cudaError_t launch_rowmax(const SplitArgs& a, cudaStream_t st) {
  if (a.rows <= 0) return cudaSuccess;
  if (!a.zeroed) {
    cudaError_t err = cudaMemsetAsync(a.maxbits, 0, sizeof(unsigned long long) * a.rows, st);
    if (err != cudaSuccess) return err;
  }
  if (a.k > 0) {
    if (!a.strided) {
      int wpb = 8;
      unsigned grid = (unsigned)((a.rows + wpb - 1) / wpb);
      launch_pdl(rowmax_contig, grid, 32 * wpb, 0, st, a.X, a.ld, a.rows, a.k, a.cplx, a.maxbits, a.nonfinite);
    } else {
      int64_t rb = (a.rows + 255) / 256;
      int64_t ksplit = (608 + rb - 1) / rb;  // ~4 CTAs per SM in total
      if (ksplit > a.k) ksplit = a.k;
      if (ksplit > 65535) ksplit = 65535;
      if (ksplit < 1) ksplit = 1;
      int64_t kchunk = (a.k + ksplit - 1) / ksplit;
      ksplit = (a.k + kchunk - 1) / kchunk;
      launch_pdl(rowmax_strided, dim3((unsigned)rb, (unsigned)ksplit), 256, 0, st, a.X, a.ld, a.rows, a.k, kchunk, a.cplx,
                                                                           a.maxbits, a.nonfinite);
    }
  }
  return cudaGetLastError();
}

namespace {
unsigned digit_blocks(const SplitArgs& a) {
  if (a.rows <= 0 || a.k <= 0) return 0;
  return (unsigned)(a.strided ? ((a.rows + 31) / 32) * ((a.k + 63) / 64) : (a.rows * ((a.k + 7) / 8) + 255) / 256);
}
template <int CPLX, int KD>
void digits_launch_as(const SplitArgs& a, const SplitArgs& b, unsigned blocks_a, unsigned blocks, cudaStream_t st) {
  if (a.strided != b.strided)
    launch_pdl(digits_kernel<CPLX, KD, 2>, blocks, 256, 0, st, a, b, blocks_a);
  else if (a.strided)
    launch_pdl(digits_kernel<CPLX, KD, 1>, blocks, 256, 0, st, a, b, blocks_a);
  else
    launch_pdl(digits_kernel<CPLX, KD, 0>, blocks, 256, 0, st, a, b, blocks_a);
}
cudaError_t digits_launch(const SplitArgs& a, const SplitArgs& b, unsigned blocks_a, unsigned blocks, cudaStream_t st) {
  if (blocks == 0) return cudaSuccess;
  if (a.cplx) {
    if (a.kd) digits_launch_as<1, 1>(a, b, blocks_a, blocks, st);
    else digits_launch_as<1, 0>(a, b, blocks_a, blocks, st);
  } else {
    if (a.kd) digits_launch_as<0, 1>(a, b, blocks_a, blocks, st);
    else digits_launch_as<0, 0>(a, b, blocks_a, blocks, st);
  }
  return cudaGetLastError();
}
// elements (real numbers) of both operands up to which a launch covers both at some cost per element
constexpr int64_t kPairElems = 4 << 20;
bool small_pair(const SplitArgs& a, const SplitArgs& b) { return (a.rows + b.rows) * a.k * (a.cplx ? 2 : 1) <= kPairElems; }
}  // namespace

cudaError_t launch_digits(const SplitArgs& a, cudaStream_t st) {
  return digits_launch(a, a, digit_blocks(a), digit_blocks(a), st);
}
cudaError_t launch_digits_pair(const SplitArgs& a, const SplitArgs& b, cudaStream_t st) {
  if (a.strided == b.strided || small_pair(a, b))
    return digits_launch(a, b, digit_blocks(a), digit_blocks(a) + digit_blocks(b), st);
  cudaError_t e = launch_digits(a, st);
  return e == cudaSuccess ? launch_digits(b, st) : e;
}

cudaError_t launch_split(const SplitArgs& a, cudaStream_t st) {
  cudaError_t e = launch_rowmax(a, st);
  if (e != cudaSuccess) return e;
  return launch_digits(a, st);
}

// Row maxima of both operands (maxbits zeroed): one launch for small ones; large ones, which fill the
// GPU by themselves, a streaming launch each.
cudaError_t launch_rowmax_both(const SplitArgs& a, const SplitArgs& b, cudaStream_t st) {
  if (small_pair(a, b)) {
    auto blocks = [](const SplitArgs& x) {
      return (unsigned)(x.strided ? ((x.rows + 31) / 32) * ((x.k + kRpStridedK - 1) / kRpStridedK)
                                  : ((x.rows + 7) / 8) * ((x.k + kRpContigK - 1) / kRpContigK));
    };
    const unsigned ba = blocks(a), bb = blocks(b);
    if (ba + bb == 0) return cudaSuccess;
    if (a.cplx) launch_pdl(rowmax_pair<1>, ba + bb, 256, 0, st, a, b, ba);
    else launch_pdl(rowmax_pair<0>, ba + bb, 256, 0, st, a, b, ba);
    return cudaGetLastError();
  }
  cudaError_t e = launch_rowmax(a, st);
  return e == cudaSuccess ? launch_rowmax(b, st) : e;
}

cudaError_t launch_digits_to_i8(const __half* D, int64_t planes, int64_t plane_rows, int64_t k, int64_t Kp,
                                int8_t* out, cudaStream_t st) {
  int64_t total = planes * plane_rows * k;
  if (total <= 0) return cudaSuccess;
  { digits_to_i8<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(D, planes * plane_rows, k, Kp, out); note_launch(); }
  return cudaGetLastError();
}

}  // namespace ozg
