// Solve of K W = B by block LU with partial pivoting on [K | B], batched.
//
// Column blocks of kNb: the block's columns are factored over the rows not yet used (which fixes the
// row exchanges), the exchanges and L11^-1 are applied to the block's rows of the remaining columns,
// U12 = L11^-1 A12, and the rows below change by one product, A22 -= L21 U12.  Then, from the last
// block up, X = U11^-1 U1B for the right half and one product for the rows above, B -= U01 X.
// The products run through digit slices on the tensor cores (f64_slices.h), balanced along their
// inner index; the triangular systems are solved by substitution on the FP64 pipe, one column per thread.
// Neither L11^-1, U11^-1 nor A11^-1 is formed: a product with A11^-1 passes through numbers as
// large as its condition, and lost two to four digits where V Pi is large (V of norm 1e6, N = 64 to
// 200: 5e-11 to 3e-10 of the largest element against 3e-13 to 7e-13 here and by single columns).  The
// substitutions cost 25 ms for 810 complex systems of N = 300, where products with A11^-1 took 5.
// A column at a time, the elimination is two launches per column and runs on the FP64 pipe: 228 ms for
// 810 complex systems of N = 300, 43.5 ms for one real system of N = 2000.  In blocks 64 and 20 ms.
#include "block_lu.h"

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
// whether recip has a number to divide by (a modulus whose square underflows is none)
__device__ __forceinline__ bool divisible(double) { return true; }
__device__ __forceinline__ bool divisible(z a) { return a.x * a.x + a.y * a.y > 0.0; }
template <class T> __device__ __forceinline__ T zero();
template <> __device__ __forceinline__ double zero<double>() { return 0.0; }
template <> __device__ __forceinline__ z zero<z>() { return make_double2(0.0, 0.0); }

// P[b][j][i] = Aug[b][i][k0 + j] for rows i >= k0 (column by column, for coalesced scans)
template <class T>
__global__ void __launch_bounds__(256) k_lu_panel(const T *Aug, int N, int k0, int nb, T *P) {
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
__global__ void __launch_bounds__(kPanelThreads) k_lu_factor(T *P, int N, int k0, int j0, int j1, int *piv, int *info) {
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
      if (tid == 0) piv[(long long)b * kNb + j0 + c] = r0 + (best > 0 ? p : c);
      __syncwarp();
      if (tid == 0) {
        s_p = best > 0 && divisible(urow[c]) ? p : -1;
        s_inv = recip(urow[c]);
      }
    }
    __syncthreads();
    if (s_p < 0) {   // a zero column (or NaNs, or no number to divide by): uniform for the block
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

// The row exchanges of columns j0 .. j1 - 1 on the block's other columns, and the unit-lower solve on
// the later ones (one thread per column), before k_lu_inner_update.
template <class T>
__global__ void k_lu_inner_rows(T *P, int N, int k0, int j0, int j1, int nb, const int *piv) {
  const int b = blockIdx.x, j = threadIdx.x;
  if (j >= nb || (j >= j0 && j < j1)) return;
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
  if (j < j0) return;
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
__global__ void __launch_bounds__(256) k_lu_inner_update(T *P, int N, int k0, int j0, int j1, int nb) {
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

template <class T> __device__ __forceinline__ T one();
template <> __device__ __forceinline__ double one<double>() { return 1.0; }
template <> __device__ __forceinline__ z one<z>() { return make_double2(1.0, 0.0); }
__device__ __forceinline__ int exponent_of(double a) { return balance_exponent(a); }
__device__ __forceinline__ int exponent_of(z a) { return max(balance_exponent(a.x), balance_exponent(a.y)); }

// kex[b][c] = max over the warp's columns of the exponent of row c: what the product that
// follows balances its inner index by
template <class T>
__device__ __forceinline__ void row_exponents(const T (&x)[kNb], bool live, int *kex) {
  int mine = 0;
#pragma unroll
  for (int c = 0; c < kNb; ++c) {
    const int e = (int)__reduce_max_sync(0xffffffffu, (unsigned)(live ? exponent_of(x[c]) : 0));
    if ((int)(threadIdx.x % 32) == c) mine = e;
  }
  if (mine > 0) atomicMax(kex + threadIdx.x % 32, mine);
}

// The block's row exchanges as one permutation, found by a warp: block row c takes the content of row
// src[c], and the rows out[t] below the block that of the block's rows out_src[t], t < count (a row
// below the block only ever receives what was in the block: contents move down at a later exchange, but
// what came up stays).  Lane c follows block row c, and the t-th row below.
__device__ __forceinline__ void exchanges(const int *piv, int k0, int nb, int lane, int *src, int *out, int *out_src,
                                          int *count) {
  int cont = k0 + lane, row = -1, rcont = -1, n = 0;
  const int mine = lane < nb ? piv[lane] : 0;
  for (int c = 0; c < nb; ++c) {
    const int p = __shfl_sync(0xffffffffu, mine, c), cc = __shfl_sync(0xffffffffu, cont, c);
    int up;
    if (p < k0 + nb) {
      up = __shfl_sync(0xffffffffu, cont, p - k0);
      if (lane == p - k0) cont = cc;
    } else {
      const unsigned has = __ballot_sync(0xffffffffu, row == p);
      const int t = has ? __ffs((int)has) - 1 : n;
      up = has ? __shfl_sync(0xffffffffu, rcont, t) : p;
      if (lane == t) {
        row = p;
        rcont = cc;
      }
      n += has ? 0 : 1;
    }
    if (lane == c) cont = up;
  }
  src[lane] = cont;
  out[lane] = row;
  out_src[lane] = rcont;
  if (lane == 0) *count = n;
}

// The block's row exchanges on columns k0 + nb .. 2N - 1 of [K | B] and U12 = L11^-1 A12 by forward
// substitution, one thread per column; U11 into its place in K (the first block of a system).
// Bound by the FP64 pipe (kNb^2 / 2 multiply-adds per column): 810 complex systems of N = 300, ten
// steps, 13.8 ms for 6.8e9 real ones.  A single system has few columns and waits for memory instead: the
// exchanges are one permutation, so that its loads do not wait for one another.
template <class T>
__global__ void __launch_bounds__(128) k_lu_lower(T *Aug, int N, int k0, int nb, const T *P, const int *piv, int *kex) {
  __shared__ T L[kNb][kNb];   // L[c][i], i > c
  __shared__ int src[kNb], out[kNb], out_src[kNb], count;
  const int b = blockIdx.y, tid = threadIdx.x;
  const long long ld = 2LL * N, j = k0 + nb + (long long)blockIdx.x * blockDim.x + tid;
  T *A = Aug + (long long)b * N * ld;
  const T *Pb = P + (long long)b * kNb * N + k0;
  if (tid < 32) exchanges(piv + (long long)b * kNb, k0, nb, tid, src, out, out_src, &count);
#pragma unroll 8
  for (int e = tid; e < kNb * kNb; e += blockDim.x) {
    const int c = e / kNb, i = e % kNb;
    L[c][i] = (c < nb && i < nb) ? Pb[(long long)c * N + i] : zero<T>();
  }
  __syncthreads();
  if (blockIdx.x == 0)
    for (int e = tid; e < nb * kNb; e += blockDim.x) {
      const int c = e / kNb, i = e % kNb;
      if (i <= c) A[(k0 + i) * ld + k0 + c] = L[c][i];
    }
  const bool live = j < ld;
  T x[kNb];
#pragma unroll
  for (int c = 0; c < kNb; ++c) x[c] = (live && c < nb) ? A[src[c] * ld + j] : zero<T>();
  if (live) {
    for (int t0 = 0; t0 < count; t0 += 8) {   // (the block's rows are still as they were)
      T v[8];
#pragma unroll
      for (int t = 0; t < 8; ++t)
        if (t0 + t < count) v[t] = A[out_src[t0 + t] * ld + j];
#pragma unroll
      for (int t = 0; t < 8; ++t)
        if (t0 + t < count) A[out[t0 + t] * ld + j] = v[t];
    }
  }
#pragma unroll
  for (int c = 0; c < kNb; ++c)
#pragma unroll
    for (int i = c + 1; i < kNb; ++i) x[i] = nfma(L[c][i], x[c], x[i]);
  if (live) {
#pragma unroll
    for (int c = 0; c < kNb; ++c)
      if (c < nb) A[(k0 + c) * ld + j] = x[c];
  }
  row_exponents(x, live, kex + (long long)b * kNb);
}

// X = U11^-1 B in the block's rows of the right half by back substitution, one thread per column (the
// same systems: 11.5 ms for 5.1e9)
template <class T>
__global__ void __launch_bounds__(128) k_lu_upper(T *Aug, int N, int k0, int nb, int *kex) {
  __shared__ T U[kNb][kNb];   // U[c][i], i < c; the diagonal's reciprocals in inv
  __shared__ T inv[kNb];
  const int b = blockIdx.y, tid = threadIdx.x;
  const long long ld = 2LL * N, j = N + (long long)blockIdx.x * blockDim.x + tid;
  T *A = Aug + (long long)b * N * ld;
#pragma unroll 8
  for (int e = tid; e < kNb * kNb; e += blockDim.x) {
    const int i = e / kNb, c = e % kNb;
    U[c][i] = (i <= c && c < nb) ? A[(k0 + i) * ld + k0 + c] : zero<T>();
  }
  __syncthreads();
  if (tid < kNb) inv[tid] = tid < nb ? recip(U[tid][tid]) : one<T>();
  __syncthreads();
  const bool live = j < ld;
  T x[kNb];
#pragma unroll
  for (int c = 0; c < kNb; ++c) x[c] = (live && c < nb) ? A[(k0 + c) * ld + j] : zero<T>();
#pragma unroll
  for (int c = kNb - 1; c >= 0; --c) {
    x[c] = mul(x[c], inv[c]);
#pragma unroll
    for (int i = 0; i < c; ++i) x[i] = nfma(U[c][i], x[c], x[i]);
  }
  if (live) {
#pragma unroll
    for (int c = 0; c < kNb; ++c)
      if (c < nb) A[(k0 + c) * ld + j] = x[c];
  }
  row_exponents(x, live, kex + (long long)b * kNb);
}

inline int blocks_of(int N) { return (N + kNb - 1) / kNb; }

// bytes of scratch per system of a pass
size_t per_system(int N, bool cplx) {
  const int c = cplx ? 2 : 1;
  return (size_t)kNb * N * 8 * c + kNb * 4 + (size_t)2 * blocks_of(N) * kNb * 4 + slice_bytes(1, N, kNb * c) +
         slice_bytes(1, 2 * N * c, kNb * c) + 2048;
}
// the most systems of a pass: its scratch stays below slice_pass_bytes (one system at least).  (Passes are of equal size, so a smaller
// batch can have larger passes than a larger one: scratch is sized by this, which grows with the batch.)
size_t most_systems(sox_handle h, int N, int batch, bool cplx) {
  return std::max<size_t>(1, std::min<size_t>(batch, slice_pass_bytes(h) / per_system(N, cplx)));
}
int pass_systems(sox_handle h, int N, int batch, bool cplx) {
  const size_t most = most_systems(h, N, batch, cplx);
  const size_t passes = ((size_t)batch + most - 1) / most;
  return (int)(((size_t)batch + passes - 1) / passes);
}

// C -= A B of one step for every system: A rows of `rows` and B rows of `cols` (complex) elements, K = nb,
// digits balanced by kex (SliceBalance)
template <class T>
Status update(sox_handle h, int batch, const T *A, long long sA, long long ai, long long ak, const T *B, long long sys,
              long long ld, T *C, int rows, int cols, int nb, const int *kex, Arena scratch, cudaStream_t s) {
  constexpr bool cplx = sizeof(T) == 16;
  constexpr int c = cplx ? 2 : 1;
  SliceOp As = slice_take(scratch, batch, rows, nb * c), Bs = slice_take(scratch, batch, cols * c, nb * c);
  if (!As.p || !Bs.p) return {SOX_ERR_OOM, "workspace too small (internal sizing error)"};
  const double *a = reinterpret_cast<const double *>(A), *b = reinterpret_cast<const double *>(B);
  const SliceBalance up{kex, kNb, 1}, down{kex, kNb, -1};
  if (cplx) {
    slice_complex_a(a, sA, ai, ak, batch, As, s, up);
    slice_complex_b(b, sys, 1, ld, batch, false, false, Bs, s, down);
  } else {
    slice_rows(a, false, sA, ai, ak, batch, As, s, up);
    slice_rows(b, false, sys, 1, ld, batch, Bs, s, down);
  }
  SliceGemm g;
  g.batch = batch;
  g.C = reinterpret_cast<double *>(C);
  g.sC = c * sys; g.ci = c * ld; g.cj = 1;
  g.alpha = -1.0;
  g.beta = 1.0;
  h->launches += 3;
  return slice_gemm(h, As, Bs, g, s);
}

template <class T>
Status solve(sox_handle h, T *Aug, int N, int batch, int *info, Arena scratch, cudaStream_t s) {
  const int nblk = blocks_of(N);
  T *P = scratch.take<T>((size_t)batch * kNb * N);
  int *piv = scratch.take<int>((size_t)batch * kNb);
  int *kex = scratch.take<int>((size_t)2 * nblk * batch * kNb);   // [step][system][k]
  if (!kex) return {SOX_ERR_OOM, "workspace too small (internal sizing error)"};
  static std::atomic<unsigned long long> attr{0};
  SOX_CUDA_TRY(set_smem_once(k_lu_factor<T, true>, (int)kPanelSmem, attr));
  SOX_CUDA_TRY(cudaMemsetAsync(kex, 0, sizeof(int) * 2 * (size_t)nblk * batch * kNb, s));
  const long long ld = 2LL * N, sys = (long long)N * ld;
  // columns per block of the substitutions: fewer where 128 would leave SMs idle
  auto threads_for = [&](long long cols) { return cols * batch < 2LL * 128 * h->sm_count ? 32 : 128; };
  for (int k0 = 0; k0 < N; k0 += kNb) {
    const int nb = std::min(kNb, N - k0), m = N - k0;
    k_lu_panel<T><<<dim3((m + 31) / 32, batch), 256, 0, s>>>(Aug, N, k0, nb, P);
    // the whole block in one kernel when it fits in shared memory and there are systems
    // enough for the SMs (one SM's FP64 pipe factors a block); else kInner columns at a time
    // with the later columns updated by the whole device
    const bool whole = (size_t)m * nb * sizeof(T) <= kPanelSmem && (batch >= 64 || m <= 256);
    const int step = whole ? nb : kInner;
    for (int j0 = 0; j0 < nb; j0 += step) {
      const int j1 = std::min(nb, j0 + step);
      const size_t shm = (size_t)(m - j0) * (j1 - j0) * sizeof(T);
      if (shm <= kPanelSmem)
        k_lu_factor<T, true><<<batch, kPanelThreads, shm, s>>>(P, N, k0, j0, j1, piv, info);
      else
        k_lu_factor<T, false><<<batch, kPanelThreads, 0, s>>>(P, N, k0, j0, j1, piv, info);
      h->launches += 1;
      if (j1 - j0 < nb) {
        k_lu_inner_rows<T><<<batch, kNb, 0, s>>>(P, N, k0, j0, j1, nb, piv);
        h->launches += 1;
        if (j1 < nb) {
          k_lu_inner_update<T><<<dim3((N - k0 - j1 + 255) / 256, batch), 256, 0, s>>>(P, N, k0, j0, j1, nb);
          h->launches += 1;
        }
      }
    }
    const int cols = 2 * N - k0 - nb, below = N - k0 - nb, nt = threads_for(cols);
    int *ke = kex + (size_t)(k0 / kNb) * batch * kNb;
    k_lu_lower<T><<<dim3((cols + nt - 1) / nt, batch), nt, 0, s>>>(Aug, N, k0, nb, P, piv, ke);
    h->launches += 2;
    if (below > 0)
      SOX_TRY(update(h, batch, P + k0 + nb, (long long)kNb * N, 1, N, Aug + (long long)k0 * ld + k0 + nb, sys, ld,
                     Aug + (long long)(k0 + nb) * ld + k0 + nb, below, cols, nb, ke, scratch, s));
  }
  for (int k0 = (nblk - 1) * kNb; k0 >= 0; k0 -= kNb) {
    const int nb = std::min(kNb, N - k0), nt = threads_for(N);
    int *ke = kex + (size_t)(nblk + k0 / kNb) * batch * kNb;
    k_lu_upper<T><<<dim3((N + nt - 1) / nt, batch), nt, 0, s>>>(Aug, N, k0, nb, ke);
    h->launches += 1;
    if (k0 > 0)
      SOX_TRY(update(h, batch, Aug + k0, sys, ld, 1, Aug + (long long)k0 * ld + N, sys, ld, Aug + N, k0, N, nb, ke,
                     scratch, s));
  }
  SOX_CUDA_TRY(cudaGetLastError());
  return Status::ok();
}

}  // namespace

// Below, two launches per column cost less than the twenty of a block.
bool lu_pays(int N) { return N >= 64; }

size_t lu_bytes(sox_handle h, int N, int batch, bool cplx) {
  return lu_pays(N) ? per_system(N, cplx) * most_systems(h, N, batch, cplx) : 0;
}

Status lu_solve(sox_handle h, double *Aug, int N, int batch, bool cplx, int *info, Arena scratch, cudaStream_t s) {
  const int per = pass_systems(h, N, batch, cplx);
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
