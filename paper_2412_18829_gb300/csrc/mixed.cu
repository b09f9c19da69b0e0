// FP32 CUDA-core contractions of the split-precision chain: the mixed THC tensor
// U_Pqs = sum_Q U_PQ X_qQ X_sQ (Eq. U_contraction at k = 0) and the half transform of the
// back-projection, both in round-to-nearest FP32 over one ascending sum per element.
#include <algorithm>

#include "sgemm.cuh"
#include "tc_kernels.h"

namespace sox {
namespace {

// The pair columns (q, s) are symmetric in their indices (X_qQ X_sQ is one product either
// way), so only q >= s is computed, in column tiles of 8 q by 16 s:
// tile t of row block qt = q / 8 has s block st = s / 16 in [0, qt / 2].
constexpr int kQB = 8, kSB = 16;
__host__ __device__ inline int tiles_before(int qt) {   // tiles of the row blocks below qt
  const int m = qt / 2;
  return (qt & 1) ? (m + 1) * (m + 1) : m * (m + 1);
}
int pair_tiles(int n) { return tiles_before((n + kQB - 1) / kQB); }

__device__ __forceinline__ void decode_tile(int t, int &qt, int &st) {
  int m = (int)((sqrtf(4.f * (float)t + 1.f) - 1.f) * 0.5f);
  while (m > 0 && m * (m + 1) > t) --m;
  while ((m + 1) * (m + 2) <= t) ++m;
  const int odd = (m + 1) * (m + 1);
  qt = t >= odd ? 2 * m + 1 : 2 * m;
  st = t >= odd ? t - odd : t - m * (m + 1);
}

// Y[Q][t * 128 + c] = float(X_qQ X_sQ) for the columns of tile t (zero for q >= n or s >= n):
// formed once in FP64 and rounded once, outside the GEMM's loop (in the loop the FP64
// products and conversions took as long as the FP32 FMAs they fed).
__global__ void __launch_bounds__(128) k_pair_columns(const double *X, int N, int n, int ncols, float *Y) {
  int qt, st;
  decode_tile(blockIdx.x, qt, st);
  const int q = qt * kQB + threadIdx.x / kSB, s = st * kSB + threadIdx.x % kSB;
  const bool in = q < n && s < n;
  for (int Q = blockIdx.y; Q < N; Q += gridDim.y) {
    const double *x = X + (long long)Q * n;
    Y[(long long)Q * ncols + blockIdx.x * sg::kBN + threadIdx.x] = in ? (float)(x[q] * x[s]) : 0.f;
  }
}

// dst[c][r] = float(src[r][c]) for a square N x N source, rows of ld >= N elements (pad zero)
__global__ void __launch_bounds__(256) k_transpose_f32(const double *src, int N, int ld, float *dst) {
  __shared__ float t[32][33];
  const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32, tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  for (int i = ty; i < 32; i += 8)
    t[i][tx] = (r0 + i < N && c0 + tx < N) ? (float)src[(long long)(r0 + i) * N + c0 + tx] : 0.f;
  __syncthreads();
  for (int i = ty; i < 32; i += 8)
    if (c0 + i < N && r0 + tx < ld) dst[(long long)(c0 + i) * ld + r0 + tx] = t[tx][i];
}

// dst[r][c] = float(src[r][c]), rows of ld >= cols elements (pad zero)
__global__ void k_rows_f32(const double *src, int rows, int cols, int ld, float *dst) {
  const long long total = (long long)rows * ld;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int r = (int)(e / ld), c = (int)(e % ld);
    dst[e] = c < cols ? (float)src[(long long)r * cols + c] : 0.f;
  }
}

// U[P][q][s] and its mirror U[P][s][q] for one BM x 128 tile; entries with q or s >= n are
// not written.  The row tiles run fastest, so a column tile of Y leaves DRAM once.
// Bound by the FP32 pipe: n = 298, N = 1788 (2.9e11 flops after the symmetry) 5.0 ms, 57 of
// the pipe's 80 TFLOP/s; a 64 x 64 tile that formed the products in its loop, over all
// (q, s), took 32.0 ms.
template <int BM>
__global__ void __launch_bounds__(sg::kThreads, 2) k_mixed_f32(const float *VT, int ldv, const float *Y, int ncols,
                                                               int N, int n, int Kp, float *U) {
  constexpr int kStages = 3;
  __shared__ __align__(16) float sa[kStages][sg::kBK * BM];
  __shared__ __align__(16) float sb[kStages][sg::kBK * sg::kBN];
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  const int P0 = blockIdx.x * BM;
  const long long c0 = (long long)blockIdx.y * sg::kBN;
  const int nkb = (N + sg::kBK - 1) / sg::kBK;
  auto load = [&](int kb, int st) {
#pragma unroll
    for (int e = tid; e < sg::kBK * BM / 4; e += sg::kThreads) {
      const int k = e / (BM / 4), r = (e % (BM / 4)) * 4, Q = kb * sg::kBK + k;
      const bool ok = Q < N && P0 + r < ldv;   // ldv is a multiple of 4: a chunk is all in or all out
      sg::cp16(&sa[st][k * BM + r], ok ? VT + (long long)Q * ldv + P0 + r : VT, ok ? 16 : 0);
    }
#pragma unroll
    for (int e = tid; e < sg::kBK * sg::kBN / 4; e += sg::kThreads) {
      const int k = e / (sg::kBN / 4), c = (e % (sg::kBN / 4)) * 4, Q = kb * sg::kBK + k;
      const bool ok = Q < N;
      sg::cp16(&sb[st][k * sg::kBN + c], ok ? Y + (long long)Q * ncols + c0 + c : Y, ok ? 16 : 0);
    }
  };
  sg::Acc<BM> acc;
  acc.zero();
#pragma unroll
  for (int p = 0; p < kStages - 1; ++p) {
    if (p < nkb) load(p, p);
    sg::cp_commit();
  }
  for (int kb = 0; kb < nkb; ++kb) {
    sg::cp_wait<kStages - 2>();
    __syncthreads();
    if (kb + kStages - 1 < nkb) load(kb + kStages - 1, (kb + kStages - 1) % kStages);
    sg::cp_commit();
    acc.step(sa[kb % kStages], BM, sb[kb % kStages], tx, ty);
  }
  int qt, st;
  decode_tile(blockIdx.y, qt, st);
  const long long blk = (long long)Kp * Kp;
#pragma unroll
  for (int i = 0; i < sg::Acc<BM>::R; ++i) {
    const int P = P0 + sg::Acc<BM>::row(i, ty);
    if (P >= N) continue;
    float *u = U + (long long)P * blk;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c = h * 64 + tx * 4;
      const int q = qt * kQB + c / kSB, s0 = st * kSB + c % kSB;
      if (q >= n || s0 > q) continue;
      float v[4];
      sg::unpack2(acc.v[i][2 * h], v[0], v[1]);
      sg::unpack2(acc.v[i][2 * h + 1], v[2], v[3]);
      if (s0 + 3 <= q) {
        *reinterpret_cast<float4 *>(u + (long long)q * Kp + s0) = make_float4(v[0], v[1], v[2], v[3]);
#pragma unroll
        for (int e = 0; e < 4; ++e) u[(long long)(s0 + e) * Kp + q] = v[e];
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (s0 + e <= q) {
            u[(long long)q * Kp + s0 + e] = v[e];
            u[(long long)(s0 + e) * Kp + q] = v[e];
          }
      }
    }
  }
}

// T[b][R][r] = sum_P Dt[b][R][P] X[P][r], BM rows R x 128 columns r per block.  Dt's rows
// run along the sum, so its tile is transposed on the way into shared memory (registers
// hold the next one while this one is used).  n = 120, N = 600, 160 batches: 0.31 ms (45
// TFLOP/s) against 0.76 ms for 64 x 64 tiles that converted X in their loop.
template <int BM>
__global__ void __launch_bounds__(sg::kThreads, 2) k_backproject_T(const float *Dt, long long ldD, const float *Xf,
                                                                   int ldx, int N, int n, float *T) {
  constexpr int kLda = BM + 4, kPer = sg::kBK * BM / sg::kThreads;
  __shared__ __align__(16) float sa[2][sg::kBK * kLda];
  __shared__ __align__(16) float sb[2][sg::kBK * sg::kBN];
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  const int R0 = blockIdx.y * BM, r0 = blockIdx.x * sg::kBN;
  const float *D = Dt + (long long)blockIdx.z * N * ldD;
  const int nkb = (N + sg::kBK - 1) / sg::kBK;
  float ra[kPer];
  const int kk = tid % sg::kBK, rr = tid / sg::kBK;
  auto load_a = [&](int kb) {
    const int P = kb * sg::kBK + kk;
#pragma unroll
    for (int e = 0; e < kPer; ++e) {
      const int R = R0 + rr + e * 16;
      ra[e] = (R < N && P < N) ? D[(long long)R * ldD + P] : 0.f;
    }
  };
  auto load_b = [&](int kb, int st) {
#pragma unroll
    for (int e = tid; e < sg::kBK * sg::kBN / 4; e += sg::kThreads) {
      const int k = e / (sg::kBN / 4), c = (e % (sg::kBN / 4)) * 4, P = kb * sg::kBK + k;
      const bool ok = P < N && r0 + c < ldx;
      sg::cp16(&sb[st][k * sg::kBN + c], ok ? Xf + (long long)P * ldx + r0 + c : Xf, ok ? 16 : 0);
    }
    sg::cp_commit();
  };
  sg::Acc<BM> acc;
  acc.zero();
  load_a(0);
  load_b(0, 0);
  for (int kb = 0; kb < nkb; ++kb) {
    const int st = kb & 1;
#pragma unroll
    for (int e = 0; e < kPer; ++e) sa[st][kk * kLda + rr + e * 16] = ra[e];
    sg::cp_wait<0>();
    __syncthreads();   // also: every thread is done with the other stage (read one step ago)
    if (kb + 1 < nkb) {
      load_b(kb + 1, st ^ 1);
      load_a(kb + 1);
    }
    acc.step(sa[st], kLda, sb[st], tx, ty);
  }
#pragma unroll
  for (int i = 0; i < sg::Acc<BM>::R; ++i) {
    const int R = R0 + sg::Acc<BM>::row(i, ty);
    if (R >= N) continue;
    float *t = T + ((long long)blockIdx.z * N + R) * n;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float v[4];
      sg::unpack2(acc.v[i][2 * h], v[0], v[1]);
      sg::unpack2(acc.v[i][2 * h + 1], v[2], v[3]);
      const int c = r0 + h * 64 + tx * 4;
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (c + e < n) t[c + e] = v[e];
    }
  }
}

inline int round4(int x) { return (x + 3) & ~3; }

}  // namespace

size_t mixed_f32_scratch(int N, int n) {
  const size_t vt = ((size_t)N * round4(N) * 4 + 255) & ~size_t(255);
  return vt + (size_t)N * pair_tiles(n) * sg::kBN * 4;
}

void launch_mixed_f32(int sms, const double *V, const double *X, int N, int n, int Kp, float *U, void *scratch,
                      cudaStream_t s) {
  const int ldv = round4(N), tiles = pair_tiles(n), ncols = tiles * sg::kBN;
  float *VT = static_cast<float *>(scratch);
  float *Y = reinterpret_cast<float *>(static_cast<char *>(scratch) + (((size_t)N * ldv * 4 + 255) & ~size_t(255)));
  k_transpose_f32<<<dim3((N + 31) / 32, (N + 31) / 32), 256, 0, s>>>(V, N, ldv, VT);
  k_pair_columns<<<dim3(tiles, std::min(N, 64)), 128, 0, s>>>(X, N, n, ncols, Y);
  // 64-row tiles while 128-row tiles would leave SMs idle (fewer than two tiles per SM)
  if ((long long)((N + 127) / 128) * tiles < 2LL * sms)
    k_mixed_f32<64><<<dim3((N + 63) / 64, tiles), sg::kThreads, 0, s>>>(VT, ldv, Y, ncols, N, n, Kp, U);
  else
    k_mixed_f32<128><<<dim3((N + 127) / 128, tiles), sg::kThreads, 0, s>>>(VT, ldv, Y, ncols, N, n, Kp, U);
}

size_t rows_f32_bytes(int N, int n) { return (size_t)N * round4(n) * 4; }

void launch_rows_f32(const double *X, int N, int n, float *Xf, cudaStream_t s) {
  const long long total = (long long)N * round4(n);
  k_rows_f32<<<(int)std::min<long long>((total + 255) / 256, 65535), 256, 0, s>>>(X, N, n, round4(n), Xf);
}

void launch_backproject_T(int sms, const float *Dt, long long ldD, const float *Xf, int N, int n, int batch, float *T,
                          cudaStream_t s) {
  const int tn = (n + sg::kBN - 1) / sg::kBN;
  if ((long long)((N + 127) / 128) * tn * batch < 2LL * sms)
    k_backproject_T<64><<<dim3(tn, (N + 63) / 64, batch), sg::kThreads, 0, s>>>(Dt, ldD, Xf, round4(n), N, n, T);
  else
    k_backproject_T<128><<<dim3(tn, (N + 127) / 128, batch), sg::kThreads, 0, s>>>(Dt, ldD, Xf, round4(n), N, n, T);
}

}  // namespace sox
