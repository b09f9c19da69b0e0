// Block Gauss-Jordan with partial pivoting on [K | B], batched.
//
// Column blocks of kNb: the block's columns are factored by LU with partial pivoting over the
// rows not yet used (which fixes the row exchanges), the exchanges are applied to the whole
// rows, and with the pivot block A11 the remaining columns change by two products,
//   R = A11^-1 A_blk,   A_i -= A_i,blk R   for every row i outside the block,
// both through digit slices on the tensor cores (f64_slices.h).  A column at a time, the same
// elimination is two launches per column and runs on the FP64 pipe: 228 ms for 810 complex
// systems of N = 300, 43.5 ms for one real system of N = 2000.  In blocks 45 and 19 ms: half
// the products (bound by reading and writing the N x 2N matrix and its sums once per block),
// then the factorisation of a block's columns on one SM's FP64 pipe per system.
#include "gj.h"

#include <algorithm>

#include "f64_slices.h"
#include "smem_attr.h"

namespace sox {
namespace {

constexpr int kNb = 32;        // columns of a block
constexpr int kInner = 8;      // columns factored at once when the whole block does not fit
constexpr int kPanelThreads = 512;
constexpr size_t kPanelSmem = 200 * 1024;

using z = double2;
__device__ __forceinline__ double mul(double a, double b) { return a * b; }
__device__ __forceinline__ z mul(z a, z b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
// c - a b
__device__ __forceinline__ double nfma(double a, double b, double c) { return fma(-a, b, c); }
__device__ __forceinline__ z nfma(z a, z b, z c) {
  return make_double2(fma(-a.x, b.x, fma(a.y, b.y, c.x)), fma(-a.x, b.y, fma(-a.y, b.x, c.y)));
}
// size of a pivot candidate: |a|, and |re| + |im| (no product on the FP64 pipe)
// as an integer that orders like it (-1 for a NaN, below every candidate)
__device__ __forceinline__ long long bits_of(double m) { return m >= 0.0 ? __double_as_longlong(m) : -1ll; }
__device__ __forceinline__ long long size_of(double a) {
  const long long b = __double_as_longlong(a) & 0x7fffffffffffffffll;
  return b > 0x7ff0000000000000ll ? -1ll : b;
}
__device__ __forceinline__ long long size_of(z a) { return bits_of(fabs(a.x) + fabs(a.y)); }
__device__ __forceinline__ double recip(double a) { return 1.0 / a; }
__device__ __forceinline__ z recip(z a) {
  const double d = 1.0 / (a.x * a.x + a.y * a.y);
  return make_double2(a.x * d, -a.y * d);
}
template <class T> __device__ __forceinline__ T zero();
template <> __device__ __forceinline__ double zero<double>() { return 0.0; }
template <> __device__ __forceinline__ z zero<z>() { return make_double2(0.0, 0.0); }
template <class T> __device__ __forceinline__ T minus_one();
template <> __device__ __forceinline__ double minus_one<double>() { return -1.0; }
template <> __device__ __forceinline__ z minus_one<z>() { return make_double2(-1.0, 0.0); }

// P[b][j][i] = Aug[b][i][k0 + j] for rows i >= k0 (column by column, for coalesced scans)
template <class T>
__global__ void __launch_bounds__(256) k_gj_panel(const T *Aug, int N, int k0, int nb, T *P) {
  __shared__ T t[32][33];
  const int b = blockIdx.y, i0 = k0 + blockIdx.x * 32, tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  const T *A = Aug + (long long)b * N * 2 * N;
  for (int i = ty; i < 32; i += 8)
    if (i0 + i < N && tx < nb) t[i][tx] = A[(long long)(i0 + i) * 2 * N + k0 + tx];
  __syncthreads();
  for (int j = ty; j < nb; j += 8)
    if (i0 + tx < N) P[((long long)b * kNb + j) * N + i0 + tx] = t[tx][j];
}

// LU with partial pivoting of columns j0 .. j1 - 1 of the block, rows k0 + j0 .. N - 1, one
// block per system; a thread owns rows, so scaling, update and the next column's pivot
// candidates need no barrier between them.  piv[b][j]: the row exchanged with row k0 + j.
// SMEM: the columns are held in shared memory (else in P itself).
template <class T, bool SMEM>
__global__ void __launch_bounds__(kPanelThreads) k_gj_lu(T *P, int N, int k0, int j0, int j1, int *piv, int *info) {
  extern __shared__ __align__(16) unsigned char raw[];
  __shared__ long long wbest[kPanelThreads / 32];
  __shared__ int wrow[kPanelThreads / 32];
  __shared__ T urow[kNb];
  __shared__ int s_p;
  __shared__ T s_inv;
  const int b = blockIdx.x, tid = threadIdx.x, r0 = k0 + j0, m = N - r0, nc = j1 - j0;
  T *G = P + ((long long)b * kNb + j0) * N + r0;   // column c at G + c N
  T *A = SMEM ? reinterpret_cast<T *>(raw) : G;
  const int ld = SMEM ? m : N;
  if (SMEM) {
    for (int c = 0; c < nc; ++c)
      for (int i = tid; i < m; i += kPanelThreads) A[(long long)c * ld + i] = G[(long long)c * N + i];
    __syncthreads();
  }
  long long bv = -1;
  int bi = 0;
  for (int i = tid; i < m; i += kPanelThreads) {
    const long long v = size_of(A[i]);
    if (v > bv) {
      bv = v;
      bi = i;
    }
  }
  for (int c = 0; c < nc; ++c) {
    for (int o = 16; o > 0; o >>= 1) {
      const long long ov = __shfl_xor_sync(0xffffffffu, bv, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ov > bv || (ov == bv && oi < bi)) {
        bv = ov;
        bi = oi;
      }
    }
    if (tid % 32 == 0) {
      wbest[tid / 32] = bv;
      wrow[tid / 32] = bi;
    }
    __syncthreads();
    if (tid < 32) {
      bv = tid < kPanelThreads / 32 ? wbest[tid] : -1;
      bi = tid < kPanelThreads / 32 ? wrow[tid] : 0;
      for (int o = 8; o > 0; o >>= 1) {
        const long long ov = __shfl_xor_sync(0xffffffffu, bv, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov > bv || (ov == bv && oi < bi)) {
          bv = ov;
          bi = oi;
        }
      }
      const int p = __shfl_sync(0xffffffffu, bi, 0);
      const long long best = __shfl_sync(0xffffffffu, bv, 0);
      // exchange rows c and p of the factored columns, keep the pivot row in urow
      if (tid < nc) {
        T *col = A + (long long)tid * ld;
        const T v = col[p];
        if (p != c) {
          col[p] = col[c];
          col[c] = v;
        }
        urow[tid] = v;
      }
      if (tid == 0) {
        s_p = best > 0 ? p : -1;
        piv[(long long)b * kNb + j0 + c] = r0 + (best > 0 ? p : c);
      }
      __syncwarp();
      if (tid == 0) s_inv = recip(urow[c]);
    }
    __syncthreads();
    if (s_p < 0) {   // a zero column (or NaNs): uniform for the block
      if (tid == 0) atomicExch(&info[1], 1);
      for (int c2 = c + 1 + tid; c2 < nc; c2 += kPanelThreads) piv[(long long)b * kNb + j0 + c2] = r0 + c2;
      break;
    }
    const T inv = s_inv;
    bv = -1;
    bi = c + 1;
    for (int i = tid; i < m; i += kPanelThreads) {
      if (i <= c) continue;
      const T l = mul(A[(long long)c * ld + i], inv);
      A[(long long)c * ld + i] = l;
      for (int j = c + 1; j < nc; ++j) {
        const T v = nfma(l, urow[j], A[(long long)j * ld + i]);
        A[(long long)j * ld + i] = v;
        if (j == c + 1) {
          const long long q = size_of(v);
          if (q > bv) {
            bv = q;
            bi = i;
          }
        }
      }
    }
    __syncthreads();
  }
  if (SMEM) {
    __syncthreads();
    for (int c = 0; c < nc; ++c)
      for (int i = tid; i < m; i += kPanelThreads) G[(long long)c * N + i] = A[(long long)c * ld + i];
  }
}

// The row exchanges of columns j0 .. j1 - 1 and the unit-lower solve on the block's later
// columns (one thread per column), before k_gj_inner_update.
template <class T>
__global__ void k_gj_inner_rows(T *P, int N, int k0, int j0, int j1, int nb, const int *piv) {
  const int b = blockIdx.x, j = j1 + threadIdx.x;
  if (j >= nb) return;
  T *col = P + ((long long)b * kNb + j) * N;
  const T *L = P + ((long long)b * kNb + j0) * N;
  for (int c = j0; c < j1; ++c) {
    const int p = piv[(long long)b * kNb + c], r = k0 + c;
    const T v = col[p];
    if (p != r) {
      col[p] = col[r];
      col[r] = v;
    }
  }
  T u[kInner];
#pragma unroll
  for (int c = 0; c < kInner; ++c) {
    if (c >= j1 - j0) break;
    T v = col[k0 + j0 + c];
#pragma unroll
    for (int d = 0; d < c; ++d) v = nfma(L[(long long)d * N + k0 + j0 + c], u[d], v);
    u[c] = v;
    col[k0 + j0 + c] = v;
  }
}

// A_ij -= sum_c L_ic u_cj for the block's later columns and the rows below
template <class T>
__global__ void __launch_bounds__(256) k_gj_inner_update(T *P, int N, int k0, int j0, int j1, int nb) {
  __shared__ T u[kInner][kNb];
  const int b = blockIdx.y, i = k0 + j1 + blockIdx.x * 256 + threadIdx.x;
  T *Pb = P + (long long)b * kNb * N;
  for (int e = threadIdx.x; e < (j1 - j0) * (nb - j1); e += 256) {
    const int c = e / (nb - j1), j = j1 + e % (nb - j1);
    u[c][j] = Pb[(long long)j * N + k0 + j0 + c];
  }
  __syncthreads();
  if (i >= N) return;
  T l[kInner];
#pragma unroll
  for (int c = 0; c < kInner; ++c) l[c] = c < j1 - j0 ? Pb[(long long)(j0 + c) * N + i] : zero<T>();
  for (int j = j1; j < nb; ++j) {
    T v = Pb[(long long)j * N + i];
#pragma unroll
    for (int c = 0; c < kInner; ++c)
      if (c < j1 - j0) v = nfma(l[c], u[c][j], v);
    Pb[(long long)j * N + i] = v;
  }
}

// The block's row exchanges on columns k0 .. 2N - 1 of [K | B], one thread per column.
template <class T>
__global__ void __launch_bounds__(128) k_gj_swap(T *Aug, int N, int k0, int nb, const int *piv) {
  __shared__ int sp[kNb];
  const int b = blockIdx.y;
  const long long j = k0 + blockIdx.x * 128 + threadIdx.x;
  if (threadIdx.x < nb) sp[threadIdx.x] = piv[(long long)b * kNb + threadIdx.x];
  __syncthreads();
  if (j >= 2LL * N) return;
  T *A = Aug + (long long)b * N * 2 * N + j;
  for (int c = 0; c < nb; ++c) {
    const int p = sp[c];
    if (p == k0 + c) continue;
    const T v = A[(long long)p * 2 * N], w = A[(long long)(k0 + c) * 2 * N];
    A[(long long)p * 2 * N] = w;
    A[(long long)(k0 + c) * 2 * N] = v;
  }
}

// F[b][i][c] = Aug[b][i][k0 + c] outside the block's rows, zero inside (columns c >= nb zero)
template <class T>
__global__ void __launch_bounds__(256) k_gj_factor(const T *Aug, int N, int k0, int nb, T *F) {
  const int b = blockIdx.y, c = threadIdx.x % kNb, i = blockIdx.x * 8 + threadIdx.x / kNb;
  if (i >= N) return;
  const bool in = c < nb && !(i >= k0 && i < k0 + nb);
  F[((long long)b * N + i) * kNb + c] = in ? Aug[((long long)b * N + i) * 2 * N + k0 + c] : zero<T>();
}

// Inv[b] = A11^-1 (rows of kNb, zero beyond nb): in-place Gauss-Jordan with partial pivoting in
// shared memory (the rows are in pivot order already; the search guards A11 itself)
template <class T>
__global__ void __launch_bounds__(256) k_gj_block_inverse(const T *Aug, int N, int k0, int nb, T *Inv, int *info) {
  __shared__ T A[kNb * kNb];
  __shared__ T rk[kNb], fk[kNb];
  __shared__ int piv[kNb];
  const int b = blockIdx.x, tid = threadIdx.x;
  for (int e = tid; e < nb * nb; e += 256)
    A[e] = Aug[((long long)b * N + k0 + e / nb) * 2 * N + k0 + e % nb];
  for (int k = 0; k < nb; ++k) {
    __syncthreads();
    if (tid < 32) {
      long long bv = (tid >= k && tid < nb) ? size_of(A[tid * nb + k]) : -1;
      int p = tid;
      for (int o = 16; o > 0; o >>= 1) {
        const long long ov = __shfl_xor_sync(0xffffffffu, bv, o);
        const int oi = __shfl_xor_sync(0xffffffffu, p, o);
        if (ov > bv || (ov == bv && oi < p)) {
          bv = ov;
          p = oi;
        }
      }
      if (bv > 0) {
        const T inv = recip(A[p * nb + k]), akk = A[k * nb + k];
        if (tid < nb) {
          rk[tid] = tid == k ? inv : mul(A[p * nb + tid], inv);
          fk[tid] = tid == k ? minus_one<T>() : (tid == p ? akk : A[tid * nb + k]);
        }
        __syncwarp();
        if (p != k && tid < nb) A[p * nb + tid] = A[k * nb + tid];
      }
      if (tid == 0) piv[k] = bv > 0 ? p : -1;
    }
    __syncthreads();
    if (piv[k] < 0) {
      if (tid == 0) atomicExch(&info[1], 1);
      return;
    }
    for (int e = tid; e < nb * nb; e += 256) {
      const int i = e / nb, j = e % nb;
      A[e] = nfma(fk[i], rk[j], (i == k || j == k) ? zero<T>() : A[e]);
    }
  }
  __syncthreads();
  if (tid < nb)
    for (int k = nb - 1; k >= 0; --k) {
      const int p = piv[k];
      if (p != k) {
        const T t = A[tid * nb + k];
        A[tid * nb + k] = A[tid * nb + p];
        A[tid * nb + p] = t;
      }
    }
  __syncthreads();
  for (int e = tid; e < kNb * kNb; e += 256) {
    const int i = e / kNb, j = e % kNb;
    Inv[(long long)b * kNb * kNb + e] = (i < nb && j < nb) ? A[i * nb + j] : zero<T>();
  }
}

// The block's rows, columns k0 + nb ..: Aug = R[b][c][j] (rows of ldr)
template <class T>
__global__ void __launch_bounds__(256) k_gj_put_rows(const T *R, long long ldr, int N, int k0, int nb, T *Aug) {
  const int b = blockIdx.z, c = blockIdx.y;
  const long long j = blockIdx.x * 256 + threadIdx.x, rest = 2LL * N - k0 - nb;
  if (j < rest) Aug[((long long)b * N + k0 + c) * 2 * N + k0 + nb + j] = R[((long long)b * kNb + c) * ldr + j];
}

// bytes of scratch per system of a pass
size_t per_system(int N, bool cplx) {
  const int c = cplx ? 2 : 1;
  const size_t e = 8 * c;
  return 4 * (size_t)kNb * N * e + kNb * kNb * e + kNb * 4 + slice_bytes(1, kNb, kNb * c) + slice_bytes(1, N, kNb * c) +
         slice_bytes(1, 2 * N * c, kNb * c) + 2048;
}
// the most systems of a pass: its scratch stays near 1 GiB.  (Passes are of equal size, so a smaller
// batch can have larger passes than a larger one: scratch is sized by this, which grows with the batch.)
size_t most_systems(int N, int batch, bool cplx) {
  return std::max<size_t>(1, std::min<size_t>(batch, (size_t(1) << 30) / per_system(N, cplx)));
}
int pass_systems(int N, int batch, bool cplx) {
  const size_t most = most_systems(N, batch, cplx);
  const size_t passes = ((size_t)batch + most - 1) / most;
  return (int)(((size_t)batch + passes - 1) / passes);
}

template <class T>
Status solve(sox_handle h, T *Aug, int N, int batch, int *info, Arena scratch, cudaStream_t s) {
  constexpr bool cplx = sizeof(T) == 16;
  constexpr int c = cplx ? 2 : 1;
  T *P = scratch.take<T>((size_t)batch * kNb * N), *F = scratch.take<T>((size_t)batch * N * kNb);
  T *Inv = scratch.take<T>((size_t)batch * kNb * kNb), *Rs = scratch.take<T>((size_t)batch * kNb * 2 * N);
  int *piv = scratch.take<int>((size_t)batch * kNb);
  if (!piv) return {SOX_ERR_OOM, "workspace too small (internal sizing error)"};
  static std::atomic<unsigned long long> attr{0};
  SOX_CUDA_TRY(set_smem_once(k_gj_lu<T, true>, (int)kPanelSmem, attr));
  const long long ld = 2LL * N, sys = (long long)N * ld;
  for (int k0 = 0; k0 < N; k0 += kNb) {
    const int nb = std::min(kNb, N - k0), m = N - k0;
    k_gj_panel<T><<<dim3((m + 31) / 32, batch), 256, 0, s>>>(Aug, N, k0, nb, P);
    // the whole block in one kernel when it fits in shared memory and there are systems
    // enough for the SMs (one SM's FP64 pipe factors a block); else kInner columns at a time
    // with the later columns updated by the whole device
    const bool whole = (size_t)m * nb * sizeof(T) <= kPanelSmem && (batch >= 64 || m <= 256);
    const int step = whole ? nb : kInner;
    for (int j0 = 0; j0 < nb; j0 += step) {
      const int j1 = std::min(nb, j0 + step);
      const size_t shm = (size_t)(m - j0) * (j1 - j0) * sizeof(T);
      if (shm <= kPanelSmem)
        k_gj_lu<T, true><<<batch, kPanelThreads, shm, s>>>(P, N, k0, j0, j1, piv, info);
      else
        k_gj_lu<T, false><<<batch, kPanelThreads, 0, s>>>(P, N, k0, j0, j1, piv, info);
      h->launches += 1;
      if (j1 < nb) {
        k_gj_inner_rows<T><<<batch, 32, 0, s>>>(P, N, k0, j0, j1, nb, piv);
        if (k0 + j1 < N)
          k_gj_inner_update<T><<<dim3((N - k0 - j1 + 255) / 256, batch), 256, 0, s>>>(P, N, k0, j0, j1, nb);
        h->launches += 2;
      }
    }
    k_gj_swap<T><<<dim3((unsigned)((ld - k0 + 127) / 128), batch), 128, 0, s>>>(Aug, N, k0, nb, piv);
    k_gj_block_inverse<T><<<batch, 256, 0, s>>>(Aug, N, k0, nb, Inv, info);
    k_gj_factor<T><<<dim3((N + 7) / 8, batch), 256, 0, s>>>(Aug, N, k0, nb, F);
    h->launches += 4;
    const int rest = 2 * N - k0 - nb;
    const double *blk = reinterpret_cast<const double *>(Aug + (long long)k0 * ld + k0 + nb);
    const double *rs = reinterpret_cast<const double *>(Rs);
    const double *inv = reinterpret_cast<const double *>(Inv), *f = reinterpret_cast<const double *>(F);
    Arena ar = scratch;
    SliceOp I = slice_take(ar, batch, nb, nb * c), Fs = slice_take(ar, batch, N, nb * c),
            R = slice_take(ar, batch, rest * c, nb * c);
    if (!I.p || !Fs.p || !R.p) return {SOX_ERR_OOM, "workspace too small (internal sizing error)"};
    // R = A11^-1 A_blk into scratch (a product may read its sources again until it is done: it may
    // not write over them), then A -= F R, then R into the block's rows
    SliceGemm g;
    g.batch = batch;
    g.C = reinterpret_cast<double *>(Rs);
    g.sC = c * kNb * ld; g.ci = c * ld; g.cj = 1;
    if (cplx) {
      slice_complex_a(inv, kNb * kNb, kNb, 1, batch, I, s);
      slice_complex_b(blk, sys, 1, ld, batch, false, false, R, s);
    } else {
      slice_rows(inv, false, kNb * kNb, kNb, 1, batch, I, s);
      slice_rows(blk, false, sys, 1, ld, batch, R, s);
    }
    SOX_TRY(slice_gemm(h, I, R, g, s));
    if (cplx) {
      slice_complex_a(f, (long long)N * kNb, kNb, 1, batch, Fs, s);
      slice_complex_b(rs, kNb * ld, 1, ld, batch, false, false, R, s);
    } else {
      slice_rows(f, false, (long long)N * kNb, kNb, 1, batch, Fs, s);
      slice_rows(rs, false, kNb * ld, 1, ld, batch, R, s);
    }
    g.C = reinterpret_cast<double *>(Aug + k0 + nb);
    g.sC = c * sys;
    g.alpha = -1.0;
    g.beta = 1.0;
    SOX_TRY(slice_gemm(h, Fs, R, g, s));
    k_gj_put_rows<T><<<dim3((rest + 255) / 256, nb, batch), 256, 0, s>>>(Rs, ld, N, k0, nb, Aug);
    h->launches += 7;
  }
  SOX_CUDA_TRY(cudaGetLastError());
  return Status::ok();
}

}  // namespace

// Below, two launches per column cost less than the twenty of a block.
bool gj_pays(int N) { return N >= 64; }

size_t gj_bytes(int N, int batch, bool cplx) {
  return gj_pays(N) ? per_system(N, cplx) * most_systems(N, batch, cplx) : 0;
}

Status gj_solve(sox_handle h, double *Aug, int N, int batch, bool cplx, int *info, Arena scratch, cudaStream_t s) {
  const int per = pass_systems(N, batch, cplx);
  for (int b0 = 0; b0 < batch; b0 += per) {
    const int nb = std::min(per, batch - b0);
    if (cplx)
      SOX_TRY(solve(h, reinterpret_cast<z *>(Aug) + (long long)b0 * N * 2 * N, N, nb, info, scratch, s));
    else
      SOX_TRY(solve(h, Aug + (long long)b0 * N * 2 * N, N, nb, info, scratch, s));
  }
  return Status::ok();
}

}  // namespace sox
