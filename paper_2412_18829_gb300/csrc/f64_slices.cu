#include "f64_slices.h"

#include <algorithm>
#include <cmath>
#include <string>
#include <type_traits>

#include "smem_attr.h"
#include "tc_common.cuh"

namespace sox {
namespace {

// Digits are fixed point below a row's largest element, so the error of a product goes with the product
// of the two maxima; FP64 arithmetic errs by the sum S of the element's |a_k b_k|.  An element is
// taken from the digits only where S is known to be within 2^kSignif of the product of the scales: by
// kShared k at least where both rows hold elements within 2^kNear of their largest (the rows' counts of
// such elements mostly show it, one test per tile; else bit masks of the rows do), by its own size, or by
// the sum of products of 8-bit magnitudes (complex elements count by the larger part).  Any other is
// summed in FP64 from the sources.  (The checks cost an FP64 bare SOX of n = 80, N = 480, 30 times 2 %,
// 9.61 -> 9.82 ms, W of the 3 x 3 x 3 solid 2 %, the split-precision calls at most 2 %.)
constexpr int kNear = 3, kShared = 4, kSignif = 6;
static_assert(kShared << kSignif == 1 << (2 * kNear + 2), "kShared products of two such elements");

constexpr int kNonFinite = 1 << 20;

// ------------------------------------------------------------------ slicing
constexpr int kZeroRow = -kNonFinite;   // (a row maximum over nothing)
// Exponent field of x 2^sh (subnormals with the smallest normal exponent), kNonFinite for infinities
// and NaNs, kZeroRow for zeros.
__device__ __forceinline__ int exp_field(double x, int sh) {
  const int hi = __double2hiint(x), e = (hi >> 20) & 0x7ff;
  if (((hi & 0x7fffffff) | __double2loint(x)) == 0) return kZeroRow;
  return e == 0x7ff ? kNonFinite : max(e, 1) + sh;
}
// e_k of a balanced operand (SliceBalance; BAL: there is one)
template <bool BAL>
__device__ __forceinline__ int balance(const SliceBalance &bal, int b, int k) {
  if (!BAL) return 0;
  const int e = bal.kex[(long long)b * bal.stride + k];
  return e > 0 ? (e - 1023) / bal.part : 0;
}
// What is kept of a row: its largest exponent E and how many elements are within 2^kNear of the largest,
// or that it holds an infinity or a NaN.  The codes of two rows add up field by field.
constexpr int kCodeBias = 8192, kCodeNonFinite = 1 << 29;
__device__ __forceinline__ int row_code(int E, int near) {
  if (E == kZeroRow) E = 1;
  return E >= kNonFinite ? kCodeBias | kCodeNonFinite : (E + kCodeBias) | (near << 16);
}
__device__ __forceinline__ int code_near(int code) { return (code >> 16) & 0xfff; }
// x scaled by the row's exponent as an integer: x = X 2^-55 2^(E - 1022), |X| <= 2^55,
// rounded to nearest (ties up)
__device__ __forceinline__ long long fixed55(double x, int E) {
  const long long bits = __double_as_longlong(x);
  const int ef = (int)((bits >> 52) & 0x7ff);
  long long m = bits & 0xfffffffffffffll;
  if (ef) m |= 1ll << 52;
  if (m == 0) return 0;
  const int sh = E - (ef ? ef : 1) - 2;   // m 2^-sh
  if (sh <= 0)
    m <<= -sh;
  else
    m = sh > 60 ? 0 : (m + (1ll << (sh - 1))) >> sh;
  return bits < 0 ? -m : m;
}
// Eight elements of a row as its epilogue's checks see them: bits for those within 2^kNear of the row's
// largest and for those that are not zero, and magnitudes in 256ths of the scale, rounded down
// (negative values by their complement, one unit of the high word short).  pair: complex elements, by
// the larger part.
struct Sizes {
  unsigned near = 0u, nz = 0u;
  uint2 mag = make_uint2(0u, 0u);
};
__device__ __forceinline__ Sizes sizes_of(const long long (&X)[8], unsigned nz, bool pair) {
  Sizes z;
  z.nz = nz;
  unsigned a[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const int hi = (int)(X[e] >> 32);
    a[e] = (unsigned)(hi ^ (hi >> 31));
  }
  if (pair) {
#pragma unroll
    for (int e = 0; e < 8; e += 2) a[e] = a[e + 1] = max(a[e], a[e + 1]);
    z.nz |= ((nz & 0x55u) << 1) | ((nz >> 1) & 0x55u);
  }
  unsigned *m = &z.mag.x;
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    z.near |= a[e] >= (1u << (22 - kNear)) ? 1u << e : 0u;
    m[e / 4] |= min(a[e] >> 15, 255u) << (8 * (e & 3));
  }
  return z;
}
// Stores chunk c of a row's masks (two of nw words) and magnitudes (K8 bytes); the four threads of a word
// are four consecutive lanes that call this together.
__device__ __forceinline__ void put_sizes(uint32_t *mask, uint8_t *mag, int nw, int K8, int c, const Sizes &z) {
  const unsigned quad = 0xfu << (threadIdx.x & 28);
  unsigned x = (z.near | (z.nz << 16)) << (8 * (c & 1));   // two chunks of both masks
  x |= __shfl_xor_sync(quad, x, 1);
  const unsigned y = __shfl_xor_sync(quad, x, 2);           // the other two
  if ((c & 3) == 0) mask[c / 4] = (x & 0xffffu) | (y << 16);
  if ((c & 3) == 1) mask[nw + c / 4] = (x >> 16) | (y & 0xffff0000u);
  if (c * 8 < K8) *reinterpret_cast<uint2 *>(mag + c * 8) = z.mag;
}
__device__ __forceinline__ unsigned nonzero(double x) {
  return ((__double2hiint(x) & 0x7fffffff) | __double2loint(x)) != 0 ? 1u : 0u;
}
// X with the nonzero flag of its value (which may have rounded to X = 0) at bit 58, for shared memory
__device__ __forceinline__ long long flagged55(double x, int E) { return fixed55(x, E) + ((long long)nonzero(x) << 58); }
__device__ __forceinline__ unsigned take_flag(long long &X) {
  const int hi = (int)(X >> 32), f = (hi + (1 << 25)) >> 26;
  X -= (long long)f << 58;
  return (unsigned)f;
}
// Balanced base-256 digits of eight values, one 16-byte word of FP16 integers per digit.
// An integer v in [0, 1023] is the FP16 number 1024 + v with v in its low bits.
__device__ __forceinline__ void digits8(long long (&X)[8], uint4 (&w)[kSlices]) {
#pragma unroll
  for (int s = kSlices - 1; s >= 0; --s) {
    uint32_t u[4];
#pragma unroll
    for (int e = 0; e < 8; e += 2) {
      int d[2];
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        if (s > 0) {
          d[t] = (int)(signed char)(X[e + t] & 0xff);
          X[e + t] = (X[e + t] + 128) >> 8;
        } else {
          d[t] = (int)X[e + t];
        }
      }
      const uint32_t v = 0x64006400u + (uint32_t)(d[0] + 128) + ((uint32_t)(d[1] + 128) << 16);
      const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&v), __floats2half2_rn(1152.f, 1152.f));
      u[e / 2] = *reinterpret_cast<const uint32_t *>(&h);
    }
    w[s] = make_uint4(u[0], u[1], u[2], u[3]);
  }
}

// words of one of a row's two bit masks (near the largest, nonzero; zero beyond K)
__host__ __device__ inline int mask_words(int K) { return (K + 31) / 32; }

// Rows with contiguous elements (sk == 1): `lpr` lanes per row.
template <class T, bool BAL>
__global__ void __launch_bounds__(256) k_slice_rows(const T *src, long long sb, long long sr, int rows, int batch,
                                                    int batch_all, int K, int K8, int lpr, SliceBalance bal, __half *p,
                                                    int *ex, uint32_t *mask, uint8_t *mag) {
  const long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long row = g / lpr;
  const int l = (int)(g % lpr);
  const bool live = row < (long long)rows * batch;
  const int b = live ? (int)(row / rows) : 0;
  const T *x = live ? src + b * sb + (row % rows) * sr : src;
  int E = kZeroRow;
  if (live)
    for (int k = l; k < K; k += lpr) E = max(E, exp_field((double)x[k], balance<BAL>(bal, b, k)));
  for (int o = lpr / 2; o > 0; o >>= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, o));
  if (!live) return;
  const bool fin = E < kNonFinite;
  const long long plane = (long long)batch_all * rows * K8;
  const int nw = mask_words(K);
  int near = 0;
  for (int c = l; c < nw * 4; c += lpr) {   // (four lanes at least per row: a word's bytes go together)
    long long X[8];
    uint4 w[kSlices];
    unsigned nz = 0u;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int k = c * 8 + e;
      const double v = (fin && k < K) ? (double)x[k] : 0.0;
      X[e] = fixed55(v, E - (k < K ? balance<BAL>(bal, b, k) : 0));
      nz |= nonzero(v) << e;
    }
    const Sizes z = sizes_of(X, nz, false);
    near += __popc(z.near);
    put_sizes(mask + row * 2 * nw, mag + row * K8, nw, K8, c, z);
    if (c * 8 >= K8) continue;
    digits8(X, w);
#pragma unroll
    for (int s = 0; s < kSlices; ++s) *reinterpret_cast<uint4 *>(p + s * plane + row * K8 + c * 8) = w[s];
  }
  const unsigned group = lpr == 32 ? 0xffffffffu : ((1u << lpr) - 1u) << (threadIdx.x % 32 / lpr * lpr);
  for (int o = lpr / 2; o > 0; o >>= 1) near += __shfl_xor_sync(group, near, o);
  if (l == 0) ex[row] = row_code(E, near);
}

// Rows whose elements lie apart: 32 rows per block, transposed through shared memory.
template <class T, bool BAL>
__global__ void __launch_bounds__(256) k_slice_cols(const T *src, long long sb, long long sr, long long sk, int rows,
                                                    int batch_all, int K, int K8, SliceBalance bal, __half *p, int *ex,
                                                    uint32_t *mask, uint8_t *mag) {
  __shared__ long long sx[64][33];
  __shared__ int se[8][32], sE[32];
  const int b = blockIdx.y, r0 = blockIdx.x * 32, tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  const T *x = src + b * sb + (long long)(r0 + tx) * sr;
  const bool in = r0 + tx < rows;
  int E = kZeroRow;
  if (in)
    for (int k = ty; k < K; k += 8) E = max(E, exp_field((double)x[k * sk], balance<BAL>(bal, b, k)));
  se[ty][tx] = E;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 8; ++i) E = max(E, se[i][tx]);
  const bool fin = E < kNonFinite;
  if (ty == 0) sE[tx] = E;
  const long long plane = (long long)batch_all * rows * K8;
  const int row = threadIdx.x / 8, c8 = threadIdx.x % 8, nw = mask_words(K);
  int near = 0;
  for (int k0 = 0; k0 < K8; k0 += 64) {
    __syncthreads();
    for (int k = ty; k < 64; k += 8)
      sx[k][tx] = (in && fin && k0 + k < K) ? flagged55((double)x[(k0 + k) * sk], E - balance<BAL>(bal, b, k0 + k)) : 0;
    __syncthreads();
    const int c = k0 / 8 + c8;
    if (r0 + row < rows && c < nw * 4) {
      long long X[8];
      uint4 w[kSlices];
      unsigned nz = 0u;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        X[e] = sx[c8 * 8 + e][row];
        nz |= take_flag(X[e]) << e;
      }
      const long long r1 = (long long)b * rows + r0 + row;
      const Sizes z = sizes_of(X, nz, false);
      near += __popc(z.near);
      put_sizes(mask + r1 * 2 * nw, mag + r1 * K8, nw, K8, c, z);
      if (c * 8 >= K8) continue;
      digits8(X, w);
      const long long o = r1 * K8 + c * 8;
#pragma unroll
      for (int s = 0; s < kSlices; ++s) *reinterpret_cast<uint4 *>(p + s * plane + o) = w[s];
    }
  }
  if (r0 + row >= rows) return;
  for (int o = 4; o > 0; o >>= 1) near += __shfl_xor_sync(0xffu << (threadIdx.x & 24), near, o);
  if (c8 == 0) ex[(long long)b * rows + r0 + row] = row_code(sE[row], near);
}

// Complex rows (see SliceOp::kind): 32 rows per block, lanes along the index that is
// contiguous in memory, a row's eight halves (four complex values) per thread.
template <int KIND, bool BAL>
__global__ void __launch_bounds__(256) k_slice_complex(const double2 *src, long long sb, long long sr, long long sk,
                                                       int rows, int batch_all, int K, int K8, int sa, int sc,
                                                       SliceBalance bal, __half *p, int *ex, uint32_t *mask, uint8_t *mag) {
  __shared__ long long sx[2][32][33];
  __shared__ int se[32];
  const int b = blockIdx.y, r0 = blockIdx.x * 32, tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  const bool along_k = sk == 1;
  const double2 *x = src + b * sb;
  if (threadIdx.x < 32) se[threadIdx.x] = kZeroRow;
  __syncthreads();
  if (along_k) {
    for (int r = ty; r < 32; r += 8) {
      int E = kZeroRow;
      if (r0 + r < rows)
        for (int k = tx; k < K; k += 32) {
          const double2 v = x[(long long)(r0 + r) * sr + k];
          const int sh = balance<BAL>(bal, b, k);
          E = max(E, max(exp_field(v.x, sh), exp_field(v.y, sh)));
        }
      E = __reduce_max_sync(0xffffffffu, E);
      if (tx == 0) se[r] = E;
    }
  } else {
    int E = kZeroRow;
    if (r0 + tx < rows)
      for (int k = ty; k < K; k += 8) {
        const double2 v = x[(long long)(r0 + tx) * sr + k * sk];
        const int sh = balance<BAL>(bal, b, k);
        E = max(E, max(exp_field(v.x, sh), exp_field(v.y, sh)));
      }
    atomicMax(&se[tx], E);
  }
  __syncthreads();
  const int nr = KIND == 2 ? 2 : 1;   // real rows per complex row
  const long long plane = (long long)batch_all * rows * nr * K8;
  const int row = threadIdx.x / 8, c8 = threadIdx.x % 8, nw = mask_words(2 * K);
  int near = 0;
  for (int k0 = 0; 2 * k0 < K8; k0 += 32) {
    __syncthreads();
    for (int i = ty; i < 32; i += 8) {
      const int k = along_k ? tx : i, r = along_k ? i : tx, E = se[r];
      const bool in = r0 + r < rows && k0 + k < K && E < kNonFinite;
      double2 v = make_double2(0.0, 0.0);
      if (in) v = x[(long long)(r0 + r) * sr + (k0 + k) * sk];
      const int sh = in ? balance<BAL>(bal, b, k0 + k) : 0;
      sx[0][k][r] = in ? flagged55(v.x, E - sh) : 0;
      sx[1][k][r] = in ? flagged55(v.y, E - sh) : 0;
    }
    __syncthreads();
    const int c = k0 / 4 + c8;
    if (r0 + row < rows && c < nw * 4) {
      const long long r1 = ((long long)b * rows + r0 + row) * nr;
      long long re[4], im[4];
      unsigned nz = 0u;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        re[e] = sx[0][c8 * 4 + e][row];
        im[e] = sx[1][c8 * 4 + e][row];
        nz |= (take_flag(re[e]) | take_flag(im[e])) << (2 * e);
      }
      Sizes sizes;
#pragma unroll
      for (int i = 0; i < nr; ++i) {
        long long X[8];
        uint4 w[kSlices];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (KIND == 1) {
            X[2 * e] = re[e];
            X[2 * e + 1] = im[e];
          } else if (i == 0) {
            X[2 * e] = re[e];
            X[2 * e + 1] = sa * sc > 0 ? -im[e] : im[e];
          } else {
            X[2 * e] = sc > 0 ? im[e] : -im[e];
            X[2 * e + 1] = sa > 0 ? re[e] : -re[e];
          }
        }
        if (i == 0) {   // (of both parts: the same for either row)
          sizes = sizes_of(X, nz, true);
          near += __popc(sizes.near);
        }
        put_sizes(mask + (r1 + i) * 2 * nw, mag + (r1 + i) * K8, nw, K8, c, sizes);
        if (c * 8 >= K8) continue;
        digits8(X, w);
#pragma unroll
        for (int d = 0; d < kSlices; ++d) *reinterpret_cast<uint4 *>(p + d * plane + (r1 + i) * K8 + c * 8) = w[d];
      }
    }
  }
  if (r0 + row >= rows) return;
  for (int o = 4; o > 0; o >>= 1) near += __shfl_xor_sync(0xffu << (threadIdx.x & 24), near, o);
  if (c8 < nr) ex[((long long)b * rows + r0 + row) * nr + c8] = row_code(se[row], near);
}

// ------------------------------------------------------------------ product
// 128 (lane side, TMEM lanes) x 64 output tiles: the eight FP32 sums of a tile fill the 512
// TMEM columns.  K goes in chunks of 32 (64-byte swizzled rows, seven digit tiles of both
// operands, 84 KB a stage, two stages) and in windows of 128, after which the sums are
// read out; each sum's columns are handed back as soon as they are read, so the next window's
// first products run while the later sums are still being read.
// Bound by the MMAs (34 of 128 x 64 x 16 per 16 of K) and, at K <= 128, by reading the sums
// out in equal parts; the FP64 pipe (1.6 FMA a clock and SM) sees the elements that are
// summed from the sources, and no other.
// n = 120, N = 600, 160 batches: projections 2.84 ms on the FP64 pipe, 0.26 ms here with the
// slicing; final sum (K = 600) 1.74 -> 0.29 ms.  n = 250, N = 2000, 12 times: X G X^T 27.9 -> 1.7 ms.
constexpr int kL = 128, kW = 64, kKc = 32, kWin = 4;   // kWin chunks per window
constexpr int kLBytes = kL * kKc * 2, kWBytes = kW * kKc * 2;
constexpr int kStageBytes = kSlices * (kLBytes + kWBytes);
constexpr int kStages = 2;
// warp 0 TMA, warp 1 MMA, warps 2-17 epilogue: reading a sum out is a chain of dependent
// integer instructions, so four warps per scheduler take half the time of two
constexpr int kEpiWarps = 16;
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr int kGroups = 8;

struct Bars {
  uint64_t full[kStages], empty[kStages];
  uint64_t acc_full, acc_empty[kGroups];
  uint64_t drain;
  uint32_t tmem_base;
  int abort;
};

// Where an operand's elements came from
struct Plain {
  const void *x;
  int f32, kind, sa, sc;
  long long sb, sr, sk;
};

struct Args {
  int nL, nW, K, batch, tL, tW;
  int bL, bW;                // batches of the operands (1: shared)
  const int *eL, *eW;
  const uint32_t *mL, *mW;   // bit masks, twice mw words a row
  const uint8_t *gL, *gW;    // magnitudes, kw words a row
  int mw, kw;
  double *C;
  long long sC, cl, cw;
  double alpha, beta;
  const int *skip, *mirror;
  int lane_is_row;           // lane index is C's row index i (else its column index j)
  Plain xL, xW;              // sources, for rows with infinities or NaNs
  long long spin_limit;
  int *status;
};

__device__ __forceinline__ uint64_t desc_kmajor_sw64(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(512 >> 4) << 32;   // next 8-row group
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;            // 64-byte swizzle
  return d;
}

__device__ __forceinline__ long long wind_down(long long cap) { return cap > (1LL << 20) ? cap : (1LL << 20); }

// All products of one chunk with KS 16-wide steps; sum g lies at TMEM column g W.  The
// digit tiles of the W side follow one another in shared memory, and digit i of the lane side
// times digits j, j + 1, ... lands in the neighbouring sums i + j, i + j + 1, ...: one MMA takes
// as many digits as fit in N = 256 (an MMA below that width costs nearly as much as at it: with
// one MMA per pair of digits the fused kernel took 16.2 ms instead of 8.7 at n = 80).  On a window's first chunk a sum is
// overwritten by its first product, and waited for until the epilogue has read its columns.
template <int W, int KS>
__device__ __forceinline__ bool issue_chunk(uint32_t tmem, uint32_t st, bool first, uint64_t *acc_empty, uint32_t ph,
                                            long long limit, volatile int *abort, int *status) {
  constexpr int kPer = 256 / W < kSlices ? 256 / W : kSlices;   // digits per MMA
  constexpr uint32_t kWB = W * kKc * 2;
  const uint64_t dl = desc_kmajor_sw64(st), dw = desc_kmajor_sw64(st + kSlices * kLBytes);
  auto ready = [&](int g0, int g1) {   // sums g0 .. g1 - 1 may be overwritten
    for (int g = g0; g < g1; ++g)
      if (!tc::mbar_wait(&acc_empty[g], ph, limit, abort, status, 2)) return false;
    tc::tc_fence_after();
    return true;
  };
  auto mma = [&](int i, int j, int nj, int k, uint32_t acc) {
    tc::mma_f16(tmem + (i + j) * W, dl + (uint64_t)((i * kLBytes + k * 32) >> 4),
                dw + (uint64_t)((j * (int)kWB + k * 32) >> 4), tc::idesc_f16_f32(kL, nj * W), acc);
  };
#pragma unroll
  for (int k = 0; k < KS; ++k)
#pragma unroll
    for (int i = 0; i < kSlices; ++i) {
      const int J = i == 0 ? kSlices : kGroups - i;   // digits j < J
#pragma unroll
      for (int j = 0; j < J; j += kPer) {
        const int nj = J - j < kPer ? J - j : kPer;
        if (k == 0 && i == 0) {          // the first product of sums j .. j + nj - 1
          if (first && !ready(j, j + nj)) return false;
          mma(i, j, nj, k, first ? 0u : 1u);
        } else if (k == 0 && i == 1 && j + nj == J) {   // the last digit starts the last sum
          if (first) {
            if (!ready(kGroups - 1, kGroups)) return false;
            if (nj > 1) mma(i, j, nj - 1, k, 1u);
            mma(i, J - 1, 1, k, 0u);
          } else {
            mma(i, j, nj, k, 1u);
          }
        } else {
          mma(i, j, nj, k, 1u);
        }
      }
    }
  return true;
}

template <int C>
__device__ __forceinline__ void tmem_ld_cols(uint32_t taddr, float (&v)[C]) {
  if constexpr (C == 16) tc::tmem_ld_32x32b_x16(taddr, v);
  else tc::tmem_ld_32x32b_x8(taddr, v);
}
// waits for the loads issued so far; v passes through, so nothing reads it before
template <int C>
__device__ __forceinline__ void tmem_ld_wait_for(float (&v)[C]) {
  tc::tmem_ld_wait();
#pragma unroll
  for (int i = 0; i < C; i += 8)
    asm volatile("" : "+f"(v[i]), "+f"(v[i + 1]), "+f"(v[i + 2]), "+f"(v[i + 3]), "+f"(v[i + 4]), "+f"(v[i + 5]),
                 "+f"(v[i + 6]), "+f"(v[i + 7]));
}

// Adds the eight sums of C columns of a window to the integers acc (unit 2^-(62 - LK)) and
// hands each sum's columns back once they are read.
template <int LK, int C, int W>
__device__ __forceinline__ void read_window(uint32_t base, uint64_t *acc_empty, int lane, long long (&acc)[C]) {
  // sum g has the unit 2^-(8 g + 14); those with bits below the integer's unit are added
  // in FP32 first and rounded once
  constexpr int top = 62 - LK - 14, kLow = top / 8 + 1;   // first sum with such bits
  float low[C], buf[2][C];
  tmem_ld_cols(base, buf[0]);
#pragma unroll
  for (int g = 0; g < kGroups; ++g) {
    float (&v)[C] = buf[g & 1];
    tmem_ld_wait_for(v);
    if (g + 1 < kGroups) tmem_ld_cols(base + (g + 1) * W, buf[(g + 1) & 1]);   // in flight during the sums of g
    tc::tc_fence_before();
    __syncwarp();
    if (lane == 0) tc::mbar_arrive(&acc_empty[g]);
    const int sh = top - 8 * g;
#pragma unroll
    for (int j = 0; j < C; ++j) {
      if (g < kLow) {
        const int i = __float2int_rn(v[j]);
        if (sh >= 32)   // the high word alone
          acc[j] += (long long)((unsigned long long)((unsigned)i << (sh >= 32 ? sh - 32 : 0)) << 32);
        else
          acc[j] += (long long)i * (long long)(1u << (sh >= 0 && sh < 32 ? sh : 0));
      } else if (g == kLow) {
        low[j] = v[j];
      } else {
        low[j] = fmaf(v[j], 1.f / (float)(1 << (8 * (g - kLow))), low[j]);
      }
      if (g == kGroups - 1) acc[j] += (long long)__float2int_rn(low[j] * (1.f / (float)(1 << (8 * kLow - top))));
    }
  }
}

__device__ double plain_at(const Plain &p, long long b, int r, int k) {
  if (p.kind == 0) {
    const long long o = b * p.sb + r * p.sr + k * p.sk;
    return p.f32 ? (double)static_cast<const float *>(p.x)[o] : static_cast<const double *>(p.x)[o];
  }
  const double2 v = static_cast<const double2 *>(p.x)[b * p.sb + (p.kind == 2 ? r / 2 : r) * p.sr + (k / 2) * p.sk];
  if (p.kind == 1) return (k & 1) ? v.y : v.x;
  if (!(r & 1)) return (k & 1) ? -p.sa * p.sc * v.y : v.x;
  return (k & 1) ? p.sa * v.x : p.sc * v.y;
}
// Elements summed in FP64 from the sources, by a warp whose lanes hold the rows l0 + lane of the lane side
// and kC columns from w0.  A few: one at a time, the lanes over k.  Many: all columns in one pass over k,
// which the FP64 pipe bounds as it would a product that never saw digits.
constexpr int kFew = 32;
__device__ __noinline__ double plain_element(const Args &a, int b, int l, int w, int lane) {
  double acc = 0.0;
  for (int k = lane; k < a.K; k += 32)
    acc = fma(plain_at(a.xL, a.bL == 1 ? 0 : b, l, k), plain_at(a.xW, a.bW == 1 ? 0 : b, w, k), acc);
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  return acc;
}
template <int C>
__device__ __noinline__ void plain_block(const Args &a, int b, int l, int w0, double *out) {
  double acc[C] = {};
  const int bl = a.bL == 1 ? 0 : b, bw = a.bW == 1 ? 0 : b, cols = min(C, a.nW - w0);
  const bool in = l < a.nL;
  const Plain &L = a.xL, &W = a.xW;
  if (L.kind == 0 && W.kind == 0 && !L.f32 && !W.f32) {   // real FP64 rows: no index arithmetic per element
    const double *x = static_cast<const double *>(L.x) + bl * L.sb + min(l, a.nL - 1) * L.sr;
    const double *y = static_cast<const double *>(W.x) + bw * W.sb + w0 * W.sr;
#pragma unroll 2
    for (int k = 0; k < a.K; ++k, x += L.sk, y += W.sk) {
      const double v = *x;
#pragma unroll
      for (int j = 0; j < C; ++j)
        if (j < cols) acc[j] = fma(v, y[j * W.sr], acc[j]);
    }
  } else {
    for (int k = 0; k < a.K; ++k) {
      const double x = in ? plain_at(L, bl, l, k) : 0.0;
#pragma unroll
      for (int j = 0; j < C; ++j)
        if (j < cols) acc[j] = fma(x, plain_at(W, bw, w0 + j, k), acc[j]);
    }
  }
#pragma unroll
  for (int j = 0; j < C; ++j) out[j] = acc[j];
}

// Bit j: |I[j]| below 2^-kSignif of the scales
template <int LK, int C>
__device__ __forceinline__ unsigned small_sums(const long long (&I)[C]) {
  unsigned m = 0u;
#pragma unroll
  for (int j = 0; j < C; ++j) {
    const int hi = (int)(I[j] >> 32);
    m |= (unsigned)(hi ^ (hi >> 31)) < (1u << (30 - LK - kSignif)) ? 1u << j : 0u;
  }
  return m;
}
// What the checks read of a row: its masks (two of mw words) and magnitudes (words of four)
struct RowSizes {
  const uint32_t *mask, *mag;
};
__device__ __forceinline__ RowSizes row_sizes(const uint32_t *mask, const uint8_t *mag, long long row, int mw, int kw) {
  return {mask + row * 2 * mw, reinterpret_cast<const uint32_t *>(mag) + row * kw};
}
// Whether every pair of the warp's rows and columns has kShared elements at least within 2^kNear of the
// largest of both: `near` of the lane's row plus the columns' smallest, of K.
__device__ __forceinline__ bool all_settled(int near, bool in, int least, int K) {
  return __all_sync(0xffffffffu, !in || near + least >= K + kShared);
}
// The columns of `small` whose S may be small too (unsettled): none that share kShared k near both
// largest elements, none where the magnitudes' products sum to 2^-kSignif of the scales, and none where no k
// is nonzero in both rows (an exact zero).  L: the lane's row; W: column `lane`.
// Where that does not hold for all: the columns of `small` for which the lane's own pair misses it
template <int C>
__device__ __forceinline__ unsigned missed_counts(unsigned small, int near, int code_w, int K) {
#pragma unroll
  for (int j = 0; j < C; ++j)
    small &= near + code_near(__shfl_sync(0xffffffffu, code_w, j)) >= K + kShared ? ~(1u << j) : ~0u;
  return small;
}
template <int C>
__device__ __noinline__ unsigned unsettled_rest(unsigned small, RowSizes L, RowSizes W, int mw, int kw) {
  unsigned sum[C], some = 0u;
#pragma unroll
  for (int j = 0; j < C; ++j) sum[j] = 0u;
  const uint2 *l = reinterpret_cast<const uint2 *>(L.mag), *w = reinterpret_cast<const uint2 *>(W.mag);
  constexpr int kStep = 4;   // pairs of words at a time; most columns are settled by the first
  for (int i = 0; i < kw / 2; i += kStep) {
    const unsigned any = __reduce_or_sync(0xffffffffu, small);   // columns to look at, the same for all lanes
    if (any == 0u) return 0u;
    uint2 x[kStep], y[kStep];
#pragma unroll
    for (int t = 0; t < kStep; ++t) {
      x[t] = i + t < kw / 2 ? l[i + t] : make_uint2(0u, 0u);
      y[t] = i + t < kw / 2 ? w[i + t] : make_uint2(0u, 0u);
    }
#pragma unroll
    for (int j = 0; j < C; ++j) {
      if (!((any >> j) & 1u)) continue;
#pragma unroll
      for (int t = 0; t < kStep; ++t) {
        sum[j] = __dp4a(x[t].x, __shfl_sync(0xffffffffu, y[t].x, j), sum[j]);
        sum[j] = __dp4a(x[t].y, __shfl_sync(0xffffffffu, y[t].y, j), sum[j]);
      }
      if (sum[j] >= 1u << (16 - kSignif)) small &= ~(1u << j);
    }
  }
  if (!__any_sync(0xffffffffu, small != 0u)) return 0u;
  for (int i = 0; i < mw; ++i) {
    const uint32_t l = L.mask[mw + i], w = W.mask[mw + i];
#pragma unroll
    for (int j = 0; j < C; ++j) some |= (l & __shfl_sync(0xffffffffu, w, j)) ? 1u << j : 0u;
  }
  return small & some;
}
// (Not inlined: a call costs about 2 us of the warp, most of it code that is not in the cache, but one
// in hundreds of tiles makes it.)
template <int C>
__device__ __noinline__ unsigned unsettled(unsigned small, RowSizes L, RowSizes W, int mw, int kw) {
  int both[C];
#pragma unroll
  for (int j = 0; j < C; ++j) both[j] = 0;
  for (int i = 0; i < mw; ++i) {
    const uint32_t l = L.mask[i], w = W.mask[i];
#pragma unroll
    for (int j = 0; j < C; ++j) {
      both[j] += __popc(l & __shfl_sync(0xffffffffu, w, j));
      small &= both[j] >= kShared ? ~(1u << j) : ~0u;
    }
    if (!__any_sync(0xffffffffu, small != 0u)) return 0u;
  }
  return unsettled_rest<C>(small, L, W, mw, kw);
}

// I 2^x rounded to nearest even, x from the codes of the two rows, by integer instructions (a 64-bit
// conversion and a scaling would cost the FP64 pipe more than all products of the element did).
// False, and no value, for infinities or NaNs in a row and for a result outside the normal range:
// those elements are summed from the sources.
template <int LK>
__device__ __forceinline__ bool scaled_double(long long I, int code, double &v) {
  const unsigned long long u = I < 0 ? 0ull - (unsigned long long)I : (unsigned long long)I;
  const int lz = __clzll((long long)(u | 1));
  const unsigned long long m = u << lz;
  unsigned long long r = m >> 11;
  const unsigned rem = (unsigned)m & 0x7ffu;
  r += (rem + (unsigned)(r & 1)) > 0x400u ? 1u : 0u;
  const int x = (code & 0xffff) - 2 * kCodeBias - 2044 - (62 - LK);
  const int eb = 63 - lz + x + 1023;   // biased exponent of the leading bit
  const unsigned long long b =
      ((unsigned long long)(eb - 1) << 52) + r + (I < 0 ? 0x8000000000000000ull : 0ull);
  v = I == 0 ? 0.0 : __longlong_as_double((long long)b);
  return code < kCodeNonFinite && (I == 0 || (unsigned)(eb - 1) <= 2044u);
}

// What happens to an element on its way out: +-v, C +- v, or alpha v + beta C.  A template
// parameter, because a select between FP64 results computes them all, and each FP64
// instruction of a tile takes 4300 clocks of the SM's pipe (a third of the tile's time).
enum { kOutSet = 0, kOutAdd = 1, kOutGeneral = 2 };
template <int OUT>
__device__ __forceinline__ double out_value(double v, long long sign, double old, double alpha, double beta) {
  if (OUT == kOutGeneral) return beta != 0.0 ? fma(beta, old, alpha * v) : alpha * v;
  v = __longlong_as_double(__double_as_longlong(v) ^ sign);
  return OUT == kOutAdd ? old + v : v;
}

// LK: the sums of a tile stay below 2^LK (K <= 2^LK), kept as integers of 2^-(62 - LK)
template <int LK, int OUT>
__global__ void __launch_bounds__(kThreads, 1)
    k_slice_gemm(const __grid_constant__ CUtensorMap tmL, const __grid_constant__ CUtensorMap tmW, const Args a) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  Bars *bar = reinterpret_cast<Bars *>(smem + kStages * kStageBytes);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const long long per_b = (long long)a.tL * a.tW, total = per_b * a.batch;
  const int nkc = (a.K + kKc - 1) / kKc, nwin = (nkc + kWin - 1) / kWin;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      tc::mbar_init(&bar->full[s], 1);
      tc::mbar_init(&bar->empty[s], 1);
    }
    tc::mbar_init(&bar->acc_full, 1);
    for (int g = 0; g < kGroups; ++g) tc::mbar_init(&bar->acc_empty[g], kEpiWarps);
    tc::mbar_init(&bar->drain, 1);
    bar->abort = 0;
    tc::fence_barrier_init();
  }
  if (warp == 1) {
    tc::tmem_alloc(&bar->tmem_base, 512);
    tc::tmem_relinquish();
  }
  if (warp == 0 && lane == 0) {
    tc::prefetch_tmap(&tmL);
    tc::prefetch_tmap(&tmW);
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = bar->tmem_base;
  volatile int *abort = &bar->abort;
  const long long limit = a.spin_limit;

  if (warp == 0) {
    if (lane == 0) {
      long long it = 0;
      for (long long t = blockIdx.x; t < total && !*abort; t += gridDim.x) {
        const int b = (int)(t / per_b), r = (int)(t % per_b);
        if (a.skip && a.skip[b]) continue;
        const int l0 = (r % a.tL) * kL, w0 = (r / a.tL) * kW;
        const int zl = a.bL == 1 ? 0 : b, zw = a.bW == 1 ? 0 : b;
        for (int kc = 0; kc < nkc; ++kc, ++it) {
          const int s = (int)(it % kStages);
          if (!tc::mbar_wait(&bar->empty[s], (uint32_t)((it / kStages) & 1) ^ 1u, limit, abort, a.status, 1)) break;
          tc::mbar_arrive_expect_tx(&bar->full[s], kStageBytes);
          uint8_t *st = smem + (size_t)s * kStageBytes;
          for (int d = 0; d < kSlices; ++d) {
            tc::tma_load_3d(st + d * kLBytes, &tmL, &bar->full[s], kc * kKc, l0, d * a.bL + zl);
            tc::tma_load_3d(st + kSlices * kLBytes + d * kWBytes, &tmW, &bar->full[s], kc * kKc, w0, d * a.bW + zw);
          }
        }
      }
      // every stage issued has landed before the CTA exits
      for (int s = 0; s < kStages; ++s) {
        const long long n = it / kStages + ((it % kStages) > s ? 1 : 0);   // phases issued on stage s
        if (n > 0)
          for (long long i = 0; i < wind_down(limit) && !tc::mbar_try_wait(&bar->full[s], (uint32_t)((n - 1) & 1)); ++i) {
          }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      long long it = 0, win = 0;
      bool ok = true;
      for (long long t = blockIdx.x; t < total && ok && !*abort; t += gridDim.x) {
        if (a.skip && a.skip[(int)(t / per_b)]) continue;
        for (int w = 0; w < nwin && ok; ++w, ++win) {
          const int c1 = min(nkc, (w + 1) * kWin);
          for (int kc = w * kWin; kc < c1; ++kc, ++it) {
            const int s = (int)(it % kStages);
            ok = tc::mbar_wait(&bar->full[s], (uint32_t)((it / kStages) & 1), limit, abort, a.status, 4);
            if (!ok) break;
            tc::tc_fence_after();
            const uint32_t st = tc::smem_u32(smem + (size_t)s * kStageBytes);
            const bool first = kc == w * kWin;
            const uint32_t ph = (uint32_t)(win & 1) ^ 1u;
            ok = (a.K - kc * kKc > 16)
                     ? issue_chunk<kW, 2>(tmem, st, first, bar->acc_empty, ph, limit, abort, a.status)
                     : issue_chunk<kW, 1>(tmem, st, first, bar->acc_empty, ph, limit, abort, a.status);
            if (!ok) break;
            tc::mma_commit(&bar->empty[s]);
          }
          if (ok) tc::mma_commit(&bar->acc_full);
        }
      }
      tc::mma_commit(&bar->drain);
      for (long long i = 0; i < wind_down(limit) && !tc::mbar_try_wait(&bar->drain, 0); ++i) {
      }
    }
  } else {
    constexpr int kC = 4 * kW / kEpiWarps;   // columns per warp
    const int q = warp & 3, part = (warp - 2) >> 2;
    const int lr = q * 32 + lane;
    long long win = 0;
    for (long long t = blockIdx.x; t < total; t += gridDim.x) {
      const int b = (int)(t / per_b), r = (int)(t % per_b);
      if (a.skip && a.skip[b]) continue;
      const int l = (r % a.tL) * kL + lr, w0 = (r / a.tL) * kW + part * kC;
      // exponents of this lane's row and of column w0 + lane (handed round by shuffles)
      const int eL = l < a.nL ? a.eL[(a.bL == 1 ? 0LL : (long long)b * a.nL) + l] : 0;
      const int eWl = lane < kC && w0 + lane < a.nW ? a.eW[(a.bW == 1 ? 0LL : (long long)b * a.nW) + w0 + lane] : 0;
      const RowSizes sL = row_sizes(a.mL, a.gL, (a.bL == 1 ? 0LL : (long long)b * a.nL) + min(l, a.nL - 1), a.mw, a.kw);
      const RowSizes sW =
          row_sizes(a.mW, a.gW, (a.bW == 1 ? 0LL : (long long)b * a.nW) + min(w0 + lane % kC, a.nW - 1), a.mw, a.kw);
      long long acc[kC];
#pragma unroll
      for (int j = 0; j < kC; ++j) acc[j] = 0;
      bool ok = true;
      for (int w = 0; w < nwin; ++w, ++win) {
        ok = tc::mbar_wait_warp(&bar->acc_full, (uint32_t)(win & 1), limit, abort, a.status, 8);
        if (!ok) break;
        tc::tc_fence_after();
        read_window<LK, kC, kW>(tmem + ((uint32_t)(q * 32) << 16) + part * kC, bar->acc_empty, lane, acc);
      }
      if (!ok) break;
      double *C = a.C + b * a.sC + l * a.cl + w0 * a.cw;
      double *Cm = a.C + b * a.sC + w0 * a.cl + l * a.cw;   // mirror image
      const bool mir = a.mirror && a.mirror[b];
      const long long sign = a.alpha < 0.0 ? (long long)0x8000000000000000ull : 0ll;
      const int live = l < a.nL ? min(kC, a.nW - w0) : 0;
      const int least = (int)__reduce_min_sync(0xffffffffu, lane < kC && w0 + lane < a.nW ? code_near(eWl) : 0xffff);
      unsigned odd = 0u;   // columns to sum from the sources
      if (!all_settled(code_near(eL), l < a.nL, least, a.K)) {
        odd = missed_counts<kC>(small_sums<LK>(acc) & (live > 0 ? (1u << live) - 1u : 0u), code_near(eL), eWl, a.K);
        if (__any_sync(0xffffffffu, odd != 0u)) odd = unsettled<kC>(odd, sL, sW, a.mw, a.kw);
      }
      constexpr int kH = 8;   // C is read eight columns at a time, all loads before the first store
#pragma unroll
      for (int j0 = 0; j0 < kC; j0 += kH) {
        double old[kH];
        if (OUT != kOutSet && a.beta != 0.0) {
#pragma unroll
          for (int i = 0; i < kH; ++i) old[i] = (l < a.nL && w0 + j0 + i < a.nW) ? C[(j0 + i) * a.cw] : 0.0;
        }
#pragma unroll
        for (int i = 0; i < kH; ++i) {
          const int j = j0 + i, w = w0 + j;
          const int eW = __shfl_sync(0xffffffffu, eWl, j);
          double v;
          const bool fine = scaled_double<LK>(acc[j], eL + eW, v) && !((odd >> j) & 1u);
          if (l < a.nL && w < a.nW) {
            if (fine) {
              v = out_value<OUT>(v, sign, old[i], a.alpha, a.beta);
              if (!mir) {
                C[j * a.cw] = v;
              } else {
                const int ib = (a.lane_is_row ? l : w) / 32, jb = (a.lane_is_row ? w : l) / 32;
                if (ib <= jb) C[j * a.cw] = v;
                if (ib < jb) Cm[j * a.cl] = v;
              }
            } else {
              odd |= 1u << j;
            }
          }
        }
      }
      const int left = __reduce_add_sync(0xffffffffu, __popc(odd));
      if (left == 0) continue;
      auto put = [&](int j, double x) {
        const int w = w0 + j;
        double v = a.alpha * x;
        if (a.beta != 0.0) v = fma(a.beta, C[j * a.cw], v);
        const int ib = (a.lane_is_row ? l : w) / 32, jb = (a.lane_is_row ? w : l) / 32;
        if (!mir || ib <= jb) C[j * a.cw] = v;
        if (mir && ib < jb) Cm[j * a.cl] = v;
      };
      if (left > kFew) {
        double x[kC];
        plain_block<kC>(a, b, l, w0, x);
        for (int j = 0; j < kC; ++j)
          if ((odd >> j) & 1u) put(j, x[j]);
        continue;
      }
      for (unsigned who; (who = __ballot_sync(0xffffffffu, odd != 0u)) != 0u;) {
        const int from = __ffs((int)who) - 1, j = __shfl_sync(0xffffffffu, __ffs((int)odd) - 1, from);
        const double x = plain_element(a, b, l - lane + from, w0 + j, lane);
        if (lane == from) {
          put(j, x);
          odd &= odd - 1;
        }
      }
    }
  }
  __syncthreads();
  if (warp == 1) {
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, 512);
  }
}

// ------------------------------------------------------------------ fused B / C / D
// D[b][P][R] = sum_v B_v C_v with B_v = A_v GR^T and C_v = GW U2_v^T, FP64 (Sec. II C, the B,
// C and D steps): 128 P (lanes) x 32 R tiles; the eight sums of B_v and of C_v fill the 512
// TMEM columns, so one is read out while the other accumulates.  The two products become
// FP64 numbers with their own scales and D sums their product over v in FP64 registers.
// Per (tile, v) 14 MMAs (34 digit products each for B_v and C_v) per 16 of n; the FP64 pipe
// sees one FMA per element and v.  n = 80, N = 480, 30 times: 172.9 ms on the FP64 pipe, 7.5 ms
// here (tensor pipe 41 % busy; the copies of the digits into shared memory set the pace).
constexpr int kFW = 32;
constexpr int kFWBytes = kFW * kKc * 2;
constexpr int kFStageBytes = kSlices * (kLBytes + kFWBytes);
constexpr int kFStages = 3;

struct FBars {
  uint64_t full[kFStages], empty[kFStages];
  uint64_t acc_full[2], acc_empty[2][kGroups];
  uint64_t drain;
  uint32_t tmem_base;
  int abort;
};

struct FArgs {
  int n, N, batch, v0, v1, tP, tR;
  const int *eA, *eGR, *eGW, *eU;   // [b][v][P], [b][R], [b][P], [v][R]
  const uint32_t *mA, *mGR, *mGW, *mU;
  const uint8_t *gA, *gGR, *gGW, *gU;
  int mw, kw;
  double *D;
  long long sD;
  // sources, for rows with infinities or NaNs: A[b][v][P][q], GR[b][R][q], GW[b][P][w], U2[R][v][w]
  const double *xA, *xGR, *xGW, *xU;
  int nv;   // v slices of A (n)
  long long spin_limit;
  int *status;
};

// the same two ways as plain_element and plain_block, for B_v and C_v at once (contiguous sources)
__device__ __forceinline__ void plain_rows(const FArgs &a, int b, int v, int P, int R, const double *(&x)[4]) {
  x[0] = a.xA + (((long long)b * a.nv + v) * a.N + P) * a.n;
  x[1] = a.xGR + ((long long)b * a.N + R) * a.n;
  x[2] = a.xGW + ((long long)b * a.N + P) * a.n;
  x[3] = a.xU + ((long long)R * a.nv + v) * a.n;
}
__device__ __noinline__ double2 plain_bc(const FArgs &a, int b, int v, int P, int R, int lane) {
  const double *x[4];
  plain_rows(a, b, v, P, R, x);
  double2 s = make_double2(0.0, 0.0);
  for (int k = lane; k < a.n; k += 32) {
    s.x = fma(x[0][k], x[1][k], s.x);
    s.y = fma(x[2][k], x[3][k], s.y);
  }
  for (int o = 16; o > 0; o >>= 1) {
    s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
    s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
  }
  return s;
}
template <int C>
__device__ __noinline__ void plain_bc_block(const FArgs &a, int b, int v, int P, int R0, double2 *out) {
  double2 s[C];
  const double *x[4];
#pragma unroll
  for (int j = 0; j < C; ++j) s[j] = make_double2(0.0, 0.0);
  plain_rows(a, b, v, min(P, a.N - 1), 0, x);
  for (int k = 0; k < a.n; ++k) {
    const double p = x[0][k], q = x[2][k];
#pragma unroll
    for (int j = 0; j < C; ++j)
      if (R0 + j < a.N) {
        s[j].x = fma(p, x[1][(long long)(R0 + j) * a.n + k], s[j].x);
        s[j].y = fma(q, x[3][(long long)(R0 + j) * a.nv * a.n + k], s[j].y);
      }
  }
#pragma unroll
  for (int j = 0; j < C; ++j) out[j] = s[j];
}

template <int LK>
__global__ void __launch_bounds__(kThreads, 1)
    k_slice_bcd(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmGR,
                const __grid_constant__ CUtensorMap tmGW, const __grid_constant__ CUtensorMap tmU, const FArgs a) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  FBars *bar = reinterpret_cast<FBars *>(smem + kFStages * kFStageBytes);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int per_b = a.tP * a.tR;
  const long long total = (long long)per_b * a.batch;
  const int nkc = (a.n + kKc - 1) / kKc, nwin = (nkc + kWin - 1) / kWin;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kFStages; ++s) {
      tc::mbar_init(&bar->full[s], 1);
      tc::mbar_init(&bar->empty[s], 1);
    }
    for (int h = 0; h < 2; ++h) {
      tc::mbar_init(&bar->acc_full[h], 1);
      for (int g = 0; g < kGroups; ++g) tc::mbar_init(&bar->acc_empty[h][g], kEpiWarps);
    }
    tc::mbar_init(&bar->drain, 1);
    bar->abort = 0;
    tc::fence_barrier_init();
  }
  if (warp == 1) {
    tc::tmem_alloc(&bar->tmem_base, 512);
    tc::tmem_relinquish();
  }
  if (warp == 0 && lane == 0) {
    tc::prefetch_tmap(&tmA); tc::prefetch_tmap(&tmGR); tc::prefetch_tmap(&tmGW); tc::prefetch_tmap(&tmU);
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = bar->tmem_base;
  volatile int *abort = &bar->abort;
  const long long limit = a.spin_limit;

  if (warp == 0) {
    if (lane == 0) {
      long long it = 0;
      for (long long t = blockIdx.x; t < total && !*abort; t += gridDim.x) {
        const int b = (int)(t / per_b), r = (int)(t % per_b);
        const int P0 = (r / a.tR) * kL, R0 = (r % a.tR) * kFW;
        for (int v = a.v0; v < a.v1 && !*abort; ++v) {
          for (int c = 0; c < 2 * nkc; ++c, ++it) {   // the chunks of B_v, then of C_v
            const int s = (int)(it % kFStages);
            if (!tc::mbar_wait(&bar->empty[s], (uint32_t)((it / kFStages) & 1) ^ 1u, limit, abort, a.status, 1)) break;
            tc::mbar_arrive_expect_tx(&bar->full[s], kFStageBytes);
            uint8_t *st = smem + (size_t)s * kFStageBytes;
            const int x = (c % nkc) * kKc;
            for (int d = 0; d < kSlices; ++d) {
              uint8_t *sl = st + d * kLBytes, *sw = st + kSlices * kLBytes + d * kFWBytes;
              if (c < nkc) {
                tc::tma_load_3d(sl, &tmA, &bar->full[s], x, P0, (d * a.batch + b) * a.nv + v);
                tc::tma_load_3d(sw, &tmGR, &bar->full[s], x, R0, d * a.batch + b);
              } else {
                tc::tma_load_3d(sl, &tmGW, &bar->full[s], x, P0, d * a.batch + b);
                tc::tma_load_3d(sw, &tmU, &bar->full[s], x, R0, d * a.nv + v);
              }
            }
          }
        }
      }
      for (int s = 0; s < kFStages; ++s) {   // every stage issued has landed before the CTA exits
        const long long n = it / kFStages + ((it % kFStages) > s ? 1 : 0);
        if (n > 0)
          for (long long i = 0; i < wind_down(limit) && !tc::mbar_try_wait(&bar->full[s], (uint32_t)((n - 1) & 1)); ++i) {
          }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      long long it = 0, win = 0;   // win: windows done per half
      bool ok = true;
      for (long long t = blockIdx.x; t < total && ok && !*abort; t += gridDim.x)
        for (int v = a.v0; v < a.v1 && ok; ++v) {
          for (int h = 0; h < 2 && ok; ++h)
            for (int w = 0; w < nwin && ok; ++w) {
              const int c1 = min(nkc, (w + 1) * kWin);
              for (int kc = w * kWin; kc < c1; ++kc, ++it) {
                const int s = (int)(it % kFStages);
                ok = tc::mbar_wait(&bar->full[s], (uint32_t)((it / kFStages) & 1), limit, abort, a.status, 4);
                if (!ok) break;
                tc::tc_fence_after();
                const uint32_t st = tc::smem_u32(smem + (size_t)s * kFStageBytes);
                const bool first = kc == w * kWin;
                const uint32_t ph = (uint32_t)((win + w) & 1) ^ 1u;
                ok = (a.n - kc * kKc > 16) ? issue_chunk<kFW, 2>(tmem + h * 256, st, first, bar->acc_empty[h], ph, limit,
                                                                 abort, a.status)
                                           : issue_chunk<kFW, 1>(tmem + h * 256, st, first, bar->acc_empty[h], ph, limit,
                                                                 abort, a.status);
                if (!ok) break;
                tc::mma_commit(&bar->empty[s]);
              }
              if (ok) tc::mma_commit(&bar->acc_full[h]);
            }
          win += nwin;
        }
      tc::mma_commit(&bar->drain);
      for (long long i = 0; i < wind_down(limit) && !tc::mbar_try_wait(&bar->drain, 0); ++i) {
      }
    }
  } else {
    constexpr int kC = 4 * kFW / kEpiWarps;   // columns per warp
    const int q = warp & 3, part = (warp - 2) >> 2;
    const int lr = q * 32 + lane;
    long long win = 0;
    for (long long t = blockIdx.x; t < total; t += gridDim.x) {
      const int b = (int)(t / per_b), r = (int)(t % per_b);
      const int P = (r / a.tR) * kL + lr, R0 = (r % a.tR) * kFW + part * kC;
      double d[kC];
#pragma unroll
      for (int j = 0; j < kC; ++j) d[j] = 0.0;
      const bool in = P < a.N;
      const int cols = min(kC, a.N - R0);   // columns of this warp inside the tile (<= 0: none)
      const int eW = in ? a.eGW[(long long)b * a.N + P] : 0;
      const int eRl = lane < cols ? a.eGR[(long long)b * a.N + R0 + lane] : 0;
      const unsigned live = in && cols > 0 ? (1u << cols) - 1u : 0u;
      const int Pm = min(P, a.N - 1), Rm = min(R0 + lane % kC, a.N - 1);   // rows of the masks
      const int leastR = (int)__reduce_min_sync(0xffffffffu, lane < cols ? code_near(eRl) : 0xffff);
      const RowSizes sR = row_sizes(a.mGR, a.gGR, (long long)b * a.N + Rm, a.mw, a.kw);
      const RowSizes sW = row_sizes(a.mGW, a.gGW, (long long)b * a.N + Pm, a.mw, a.kw);
      bool ok = true;
      for (int v = a.v0; v < a.v1 && ok; ++v) {
        long long ib[kC], ic[kC];
#pragma unroll
        for (int j = 0; j < kC; ++j) ib[j] = ic[j] = 0;
        const int eA = in ? a.eA[((long long)b * a.nv + v) * a.N + P] : 0;
        const int eUl = lane < cols ? a.eU[(long long)v * a.N + R0 + lane] : 0;
        const RowSizes sA = row_sizes(a.mA, a.gA, ((long long)b * a.nv + v) * a.N + Pm, a.mw, a.kw);
        const RowSizes sU = row_sizes(a.mU, a.gU, (long long)v * a.N + Rm, a.mw, a.kw);
        for (int h = 0; h < 2 && ok; ++h)
          for (int w = 0; w < nwin; ++w) {
            ok = tc::mbar_wait_warp(&bar->acc_full[h], (uint32_t)((win + w) & 1), limit, abort, a.status, 8);
            if (!ok) break;
            tc::tc_fence_after();
            const uint32_t base = tmem + ((uint32_t)(q * 32) << 16) + h * 256 + part * kC;
            if (h == 0)
              read_window<LK, kC, kFW>(base, bar->acc_empty[0], lane, ib);
            else
              read_window<LK, kC, kFW>(base, bar->acc_empty[1], lane, ic);
          }
        win += nwin;
        if (!ok) break;
        unsigned odd = 0u;   // columns to sum from the sources
        if (!all_settled(code_near(eA), in, leastR, a.n)) {
          odd = missed_counts<kC>(small_sums<LK>(ib) & live, code_near(eA), eRl, a.n);
          if (__any_sync(0xffffffffu, odd != 0u)) odd = unsettled<kC>(odd, sA, sR, a.mw, a.kw);
        }
        const int leastU = (int)__reduce_min_sync(0xffffffffu, lane < cols ? code_near(eUl) : 0xffff);
        if (!all_settled(code_near(eW), in, leastU, a.n)) {
          unsigned oc = missed_counts<kC>(small_sums<LK>(ic) & live, code_near(eW), eUl, a.n);
          if (__any_sync(0xffffffffu, oc != 0u)) oc = unsettled<kC>(oc, sW, sU, a.mw, a.kw);
          odd |= oc;
        }
#pragma unroll
        for (int j = 0; j < kC; ++j) {
          const int eR = __shfl_sync(0xffffffffu, eRl, j), eU = __shfl_sync(0xffffffffu, eUl, j);
          double bv, cv;
          const bool fb = scaled_double<LK>(ib[j], eA + eR, bv);
          const bool fc = scaled_double<LK>(ic[j], eW + eU, cv);
          if (!(fb && fc))
            odd |= live & (1u << j);
          else if (!((odd >> j) & 1u))
            d[j] = fma(bv, cv, d[j]);
        }
        const int left = __reduce_add_sync(0xffffffffu, __popc(odd));
        if (left > kFew) {
          double2 x[kC];
          plain_bc_block<kC>(a, b, v, P, R0, x);
#pragma unroll
          for (int j = 0; j < kC; ++j)
            if ((odd >> j) & 1u) d[j] = fma(x[j].x, x[j].y, d[j]);
        } else if (left > 0) {
          for (unsigned who; (who = __ballot_sync(0xffffffffu, odd != 0u)) != 0u;) {
            const int from = __ffs((int)who) - 1, at = __shfl_sync(0xffffffffu, __ffs((int)odd) - 1, from);
            const double2 x = plain_bc(a, b, v, P - lane + from, R0 + at, lane);
#pragma unroll
            for (int j = 0; j < kC; ++j)
              if (lane == from && j == at) d[j] = fma(x.x, x.y, d[j]);
            if (lane == from) odd &= odd - 1;
          }
        }
      }
      if (!ok) break;
      if (!in) continue;
      double *D = a.D + b * a.sD + (long long)P * a.N;
#pragma unroll
      for (int j = 0; j < kC; ++j)
        if (R0 + j < a.N) D[R0 + j] = d[j];
    }
  }
  __syncthreads();
  if (warp == 1) {
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, 512);
  }
}

size_t fsmem_bytes() { return (size_t)kFStages * kFStageBytes + sizeof(FBars) + 1024; }

size_t smem_bytes() { return (size_t)kStages * kStageBytes + sizeof(Bars) + 1024; }

bool make_map(CUtensorMap *map, const SliceOp &op, int box_rows, std::string *err) {   // box kKc x box_rows
  static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  if (!encode) {
    cudaDriverEntryPointQueryResult q;
    void *fn = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn) {
      *err = "cuTensorMapEncodeTiled entry point not available";
      return false;
    }
    encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }
  cuuint64_t dims[3] = {(cuuint64_t)op.K8, (cuuint64_t)op.rows, (cuuint64_t)kSlices * op.batch};
  cuuint64_t strides[2] = {(cuuint64_t)op.K8 * 2, (cuuint64_t)op.K8 * op.rows * 2};
  cuuint32_t box[3] = {kKc, (cuuint32_t)box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, op.p, dims, strides, box, estr,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    *err = "cuTensorMapEncodeTiled (slices) failed with CUresult " + std::to_string((int)r);
    return false;
  }
  return true;
}

inline int round8(int x) { return (x + 7) & ~7; }
inline size_t al(size_t b) { return (b + 255) & ~size_t(255); }

}  // namespace

size_t slice_bytes(long long batch, int rows, int K) {
  return al((size_t)kSlices * batch * rows * round8(K) * 2) + al((size_t)batch * rows * 4) +
         al((size_t)batch * rows * 2 * mask_words(K) * 4) + al((size_t)batch * rows * round8(K));
}

SliceOp slice_take(Arena &ar, int batch, int rows, int K) {
  SliceOp op;
  op.batch = batch;
  op.rows = rows;
  op.K = K;
  op.K8 = round8(K);
  op.p = ar.take<__half>((size_t)kSlices * batch * rows * op.K8);
  op.ex = ar.take<int>((size_t)batch * rows);
  op.mask = ar.take<uint32_t>((size_t)batch * rows * 2 * mask_words(K));
  op.mag = ar.take<uint8_t>((size_t)batch * rows * op.K8);
  if (!op.mag) op.p = nullptr;
  return op;
}

void slice_rows(const void *src, bool f32, long long sb, long long sr, long long sk, int batch, SliceOp &op,
                cudaStream_t s, SliceBalance bal) {
  op.src = src;
  op.f32 = f32;
  op.sb = sb;
  op.sr = sr;
  op.sk = sk;
  if (batch <= 0 || op.rows <= 0) return;
  auto go = [&](auto t, auto bl) {
    using T = decltype(t);
    constexpr bool BAL = decltype(bl)::value;
    const T *x = static_cast<const T *>(src);
    if (sk == 1) {
      int lpr = 4;
      while (lpr < 32 && lpr * 8 < op.K8) lpr *= 2;
      const long long blocks = ((long long)batch * op.rows * lpr + 255) / 256;
      k_slice_rows<T, BAL><<<(unsigned)blocks, 256, 0, s>>>(x, sb, sr, op.rows, batch, op.batch, op.K, op.K8, lpr, bal, op.p,
                                                            op.ex, op.mask, op.mag);
    } else {
      k_slice_cols<T, BAL><<<dim3((op.rows + 31) / 32, batch), 256, 0, s>>>(x, sb, sr, sk, op.rows, op.batch, op.K, op.K8,
                                                                            bal, op.p, op.ex, op.mask, op.mag);
    }
  };
  if (f32)
    go(float{}, std::false_type{});   // (no FP32 operand is balanced)
  else if (bal.kex)
    go(double{}, std::true_type{});
  else
    go(double{}, std::false_type{});
}

void slice_complex_a(const double *src, long long sb, long long sr, long long sk, int batch, SliceOp &op, cudaStream_t s,
                     SliceBalance bal) {
  op.src = src;
  op.sb = sb; op.sr = sr; op.sk = sk;
  op.kind = 1;
  if (batch <= 0 || op.rows <= 0) return;
  auto *k = bal.kex ? k_slice_complex<1, true> : k_slice_complex<1, false>;
  k<<<dim3((op.rows + 31) / 32, batch), 256, 0, s>>>(reinterpret_cast<const double2 *>(src), sb, sr, sk, op.rows, op.batch,
                                                     op.K / 2, op.K8, 1, 1, bal, op.p, op.ex, op.mask, op.mag);
}

void slice_complex_b(const double *src, long long sb, long long sr, long long sk, int batch, bool conjA, bool conjB,
                     SliceOp &op, cudaStream_t s, SliceBalance bal) {
  op.src = src;
  op.sb = sb; op.sr = sr; op.sk = sk;
  op.kind = 2;
  op.sa = conjA ? -1 : 1;
  op.sc = conjB ? -1 : 1;
  if (batch <= 0 || op.rows <= 0) return;
  const int rows = op.rows / 2;
  auto *k = bal.kex ? k_slice_complex<2, true> : k_slice_complex<2, false>;
  k<<<dim3((rows + 31) / 32, batch), 256, 0, s>>>(reinterpret_cast<const double2 *>(src), sb, sr, sk, rows, op.batch,
                                                  op.K / 2, op.K8, op.sa, op.sc, bal, op.p, op.ex, op.mask, op.mag);
}

Status slice_gemm(sox_handle h, const SliceOp &A, const SliceOp &B, const SliceGemm &g, cudaStream_t s) {
  if (g.batch <= 0 || A.rows <= 0 || B.rows <= 0) return Status::ok();
  // TMEM lanes along the index that leaves less padding in the 128 x 64 tiles; equal: along
  // the one that is contiguous in C
  auto area = [](int l, int w) { return (long long)((l + kL - 1) / kL) * kL * ((w + kW - 1) / kW) * kW; };
  const long long ab = area(A.rows, B.rows), ba = area(B.rows, A.rows);
  const bool lane_a = ab != ba ? ab < ba : g.ci == 1;
  const SliceOp &L = lane_a ? A : B, &W = lane_a ? B : A;
  CUtensorMap mL, mW;
  std::string err;
  if (!make_map(&mL, L, kL, &err) || !make_map(&mW, W, kW, &err)) return {SOX_ERR_CUDA, err};
  Args a;
  a.nL = L.rows; a.nW = W.rows; a.K = A.K; a.batch = g.batch;
  a.tL = (L.rows + kL - 1) / kL;
  a.tW = (W.rows + kW - 1) / kW;
  a.bL = L.batch; a.bW = W.batch;
  a.eL = L.ex; a.eW = W.ex;
  a.mL = L.mask; a.mW = W.mask;
  a.gL = L.mag; a.gW = W.mag;
  a.mw = mask_words(A.K);
  a.kw = A.K8 / 4;
  a.C = g.C; a.sC = g.sC;
  a.cl = lane_a ? g.ci : g.cj;
  a.cw = lane_a ? g.cj : g.ci;
  a.alpha = g.alpha; a.beta = g.beta;
  a.skip = g.skip; a.mirror = g.mirror;
  a.lane_is_row = lane_a ? 1 : 0;
  a.xL = {L.src, L.f32 ? 1 : 0, L.kind, L.sa, L.sc, L.sb, L.sr, L.sk};
  a.xW = {W.src, W.f32 ? 1 : 0, W.kind, W.sa, W.sc, W.sb, W.sr, W.sk};
  a.spin_limit = h->spin_limit;
  a.status = h->d_status;
  const long long tiles = (long long)a.tL * a.tW * a.batch;
  const int grid = (int)std::max<long long>(1, std::min<long long>(tiles, h->sm_count));
  const bool unit = a.alpha == 1.0 || a.alpha == -1.0;
  const int out = unit && a.beta == 0.0 ? kOutSet : (unit && a.beta == 1.0 ? kOutAdd : kOutGeneral);
  auto go = [&](auto lk, auto o) -> cudaError_t {
    static std::atomic<unsigned long long> attr{0};
    auto *k = k_slice_gemm<decltype(lk)::value, decltype(o)::value>;
    const cudaError_t e = set_smem_once(k, (int)smem_bytes(), attr);
    if (e != cudaSuccess) return e;
    k<<<grid, kThreads, smem_bytes(), s>>>(mL, mW, a);
    return cudaGetLastError();
  };
  auto pick = [&](auto lk) {
    return out == kOutSet ? go(lk, std::integral_constant<int, kOutSet>{})
                          : (out == kOutAdd ? go(lk, std::integral_constant<int, kOutAdd>{})
                                            : go(lk, std::integral_constant<int, kOutGeneral>{}));
  };
  SOX_CUDA_TRY(a.K <= 128 ? pick(std::integral_constant<int, 7>{}) : pick(std::integral_constant<int, 10>{}));
  return Status::ok();
}

Status slice_bcd(sox_handle h, const SliceOp &A, const SliceOp &GR, const SliceOp &GW, const SliceOp &U2, int n, int N,
                 int batch, int v0, int v1, double *D, long long sD, cudaStream_t s) {
  if (batch <= 0) return Status::ok();
  v1 = (v1 <= 0 || v1 > n) ? n : v1;
  v0 = v0 < 0 ? 0 : (v0 > v1 ? v1 : v0);
  CUtensorMap mA, mGR, mGW, mU;
  std::string err;
  if (!make_map(&mA, A, kL, &err) || !make_map(&mGR, GR, kFW, &err) || !make_map(&mGW, GW, kL, &err) ||
      !make_map(&mU, U2, kFW, &err))
    return {SOX_ERR_CUDA, err};
  FArgs a;
  a.n = n; a.N = N; a.batch = GR.batch; a.v0 = v0; a.v1 = v1;
  a.tP = (N + kL - 1) / kL;
  a.tR = (N + kFW - 1) / kFW;
  a.eA = A.ex; a.eGR = GR.ex; a.eGW = GW.ex; a.eU = U2.ex;
  a.mA = A.mask; a.mGR = GR.mask; a.mGW = GW.mask; a.mU = U2.mask;
  a.gA = A.mag; a.gGR = GR.mag; a.gGW = GW.mag; a.gU = U2.mag;
  a.mw = mask_words(n);
  a.kw = A.K8 / 4;
  a.D = D; a.sD = sD;
  a.xA = static_cast<const double *>(A.src);
  a.xGR = static_cast<const double *>(GR.src);
  a.xGW = static_cast<const double *>(GW.src);
  a.xU = static_cast<const double *>(U2.src);
  a.nv = n;
  a.spin_limit = h->spin_limit;
  a.status = h->d_status;
  const long long tiles = (long long)a.tP * a.tR * a.batch;
  const int grid = (int)std::max<long long>(1, std::min<long long>(tiles, h->sm_count));
  static std::atomic<unsigned long long> attr7{0}, attr10{0};
  if (n <= 128) {
    SOX_CUDA_TRY(set_smem_once(k_slice_bcd<7>, (int)fsmem_bytes(), attr7));
    k_slice_bcd<7><<<grid, kThreads, fsmem_bytes(), s>>>(mA, mGR, mGW, mU, a);
  } else {
    SOX_CUDA_TRY(set_smem_once(k_slice_bcd<10>, (int)fsmem_bytes(), attr10));
    k_slice_bcd<10><<<grid, kThreads, fsmem_bytes(), s>>>(mA, mGR, mGW, mU, a);
  }
  SOX_CUDA_TRY(cudaGetLastError());
  return Status::ok();
}

// On the FP64 pipe a wave of 64 x 64 tiles takes 1.05 us per k (1.9 FMA a clock and SM), whatever
// part of it is valid; through slices a small product takes about 20 us, most of it the three launches.
// Both ways, us per product at K and waves of 152 tiles: 16 x 1 7 and 19; 20 x 1 14 and 20; 32 x 1
// 21 and 20; 40 x 1 42 and 22; 64 x 1 72 and 24; 80 x 4 331 and 32; 16 x 8 (600 batches of 128 x 16:
// tiles a quarter full) 39 and 47.
bool slices_pay(const sox_context *h, long long M, long long N, long long K, long long batch) {
  const double tiles = (double)((M + 63) / 64) * (double)((N + 63) / 64) * (double)batch;
  return (double)K * std::ceil(tiles / h->sm_count) >= 40.0;
}

namespace {
// A product runs in passes whose digits stay below slice_pass_bytes per operand: over batches, and
// over the columns of a single large one.
struct Passes {
  bool sharedA, sharedB;   // one block for every batch
  int k, nb, rows;         // K, batches and columns of a pass
};
Passes passes_of(sox_handle h, const GemmF64 &g) {
  const size_t most = slice_pass_bytes(h);
  Passes p;
  p.sharedA = g.batch == 1 || g.sA == 0;
  p.sharedB = g.batch == 1 || g.sB == 0;
  p.k = std::min(g.K, kSliceMaxK);
  const size_t per = std::max(p.sharedA ? 0 : slice_bytes(1, g.M, p.k), p.sharedB ? 0 : slice_bytes(1, g.Nc, p.k));
  p.nb = per == 0 ? g.batch : (int)std::max<size_t>(1, std::min<size_t>(g.batch, most / per));
  const size_t row = slice_bytes(1, 1024, p.k) / 1024 + 1;
  p.rows = (int)std::max<size_t>(1024, std::min<size_t>(g.Nc, most / row / (p.sharedB ? 1 : p.nb)));
  p.rows = std::min(p.rows, g.Nc);
  return p;
}
}  // namespace

size_t gemm_f64_bytes(sox_handle h, const GemmF64 &g) {
  if (!slices_pay(h, g.M, g.Nc, g.K, g.batch)) return 0;
  const Passes p = passes_of(h, g);
  return slice_bytes(p.sharedA ? 1 : p.nb, g.M, p.k) + slice_bytes(p.sharedB ? 1 : p.nb, p.rows, p.k);
}

Status gemm_f64(sox_handle h, const GemmF64 &g, Arena scratch, cudaStream_t s) {
  if (g.M <= 0 || g.Nc <= 0 || g.batch <= 0) return Status::ok();
  if (!slices_pay(h, g.M, g.Nc, g.K, g.batch)) {
    launch_gemm_f64(g, s);
    return Status::ok();
  }
  const Passes p = passes_of(h, g);
  for (int k0 = 0; k0 < g.K; k0 += p.k)
    for (int b0 = 0; b0 < g.batch; b0 += p.nb) {
      const int k = std::min(p.k, g.K - k0), nb = std::min(p.nb, g.batch - b0);
      Arena ar = scratch;
      SliceOp A = slice_take(ar, p.sharedA ? 1 : nb, g.M, k);
      if (!A.p) return {SOX_ERR_OOM, "workspace too small (internal sizing error)"};
      slice_rows(g.A + b0 * g.sA + k0 * g.ak, false, g.sA, g.ai, g.ak, A.batch, A, s);
      for (int j0 = 0; j0 < g.Nc; j0 += p.rows) {
        Arena br = ar;
        SliceOp B = slice_take(br, p.sharedB ? 1 : nb, std::min(p.rows, g.Nc - j0), k);
        if (!B.p) return {SOX_ERR_OOM, "workspace too small (internal sizing error)"};
        slice_rows(g.B + b0 * g.sB + k0 * g.bk + j0 * g.bj, false, g.sB, g.bj, g.bk, B.batch, B, s);
        SliceGemm sg;
        sg.C = g.C + b0 * g.sC + j0 * g.cj;
        sg.sC = g.sC; sg.ci = g.ci; sg.cj = g.cj;
        sg.alpha = g.alpha;
        sg.beta = k0 == 0 ? g.beta : 1.0;
        sg.batch = nb;
        sg.skip = g.skip ? g.skip + b0 : nullptr;
        SOX_TRY(slice_gemm(h, A, B, sg, s));
        h->launches += 2;   // the slicings; callers count the product
      }
    }
  return Status::ok();
}

}  // namespace sox
