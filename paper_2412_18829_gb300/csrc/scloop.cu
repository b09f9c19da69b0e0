// The self-consistent loop around Sigma for molecules (Sec. II A) on the GPU: the Dyson
// equation on fermionic Matsubara frequencies (Eqs. Dyson and G0 with S = 1), the
// high-frequency tails of G, the transforms between imaginary time and frequency, the
// electron count for the chemical-potential update, the Hartree-Fock self-energy in THC
// form and the Galitskii-Migdal energies (Eqs. E1b, E2b).  FP64 throughout.
#include <algorithm>

#include "scloop.h"
#include "smem_attr.h"

namespace sox {
namespace {

using z = double2;
__device__ __forceinline__ z zmul(z a, z b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ __forceinline__ z zfma(z a, z b, z c) {
  return make_double2(fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y)));
}

int grid_of(long long total) { return (int)std::max<long long>(1, std::min<long long>((total + 255) / 256, 65535 * 4)); }

// Aug[b] = [ (i w + mu) 1 - F[s] - Sigma[s][w]  |  1 ]  for system b = s * n_w + w  (n x 2n)
__global__ void k_dyson_build(const double *omegas, double mu, const double *F, const z *Sig, int n, int n_w,
                              int n_spin, z *Aug) {
  const long long nn = (long long)n * n, total = nn * n_w * n_spin;
  for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < total;
       g += (long long)gridDim.x * blockDim.x) {
    const long long b = g / nn, e = g % nn;
    const int s = (int)(b / n_w), w = (int)(b % n_w);
    const int i = (int)(e / n), j = (int)(e % n);
    z a = make_double2(-F[(long long)s * nn + e], 0.0);
    if (Sig) {
      const z sg = Sig[b * nn + e];
      a.x -= sg.x;
      a.y -= sg.y;
    }
    if (i == j) {
      a.x += mu;
      a.y += omegas[w];
    }
    z *row = Aug + b * 2 * nn + (long long)i * 2 * n;
    row[j] = a;
    row[n + j] = make_double2(i == j ? 1.0 : 0.0, 0.0);
  }
}

// Gauss-Jordan with partial pivoting on each n x 2n system (one block per system); the
// right half becomes the inverse.  singular[0] is set for a zero pivot column.
__global__ void __launch_bounds__(256) k_gj_block(z *Aug, int n, int *singular) {
  extern __shared__ z fk[];   // column k of the system (n entries)
  __shared__ double best[256];
  __shared__ int bidx[256];
  const long long W = 2LL * n;
  z *A = Aug + (long long)blockIdx.x * n * W;
  for (int k = 0; k < n; ++k) {
    double bv = -1.0;
    int bi = k;
    for (int i = k + threadIdx.x; i < n; i += blockDim.x) {
      const z a = A[(long long)i * W + k];
      const double m2 = a.x * a.x + a.y * a.y;
      if (m2 > bv) {
        bv = m2;
        bi = i;
      }
    }
    best[threadIdx.x] = bv;
    bidx[threadIdx.x] = bi;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
      if (threadIdx.x < o) {
        const double ov = best[threadIdx.x + o];
        const int oi = bidx[threadIdx.x + o];
        if (ov > best[threadIdx.x] || (ov == best[threadIdx.x] && oi < bidx[threadIdx.x])) {
          best[threadIdx.x] = ov;
          bidx[threadIdx.x] = oi;
        }
      }
      __syncthreads();
    }
    if (!(best[0] > 0.0)) {
      if (threadIdx.x == 0) atomicExch(singular, 1);
      return;   // uniform: every thread sees best[0]
    }
    const int p = bidx[0];
    const z pv = A[(long long)p * W + k];
    const double d = pv.x * pv.x + pv.y * pv.y;
    const z inv = make_double2(pv.x / d, -pv.y / d);
    __syncthreads();
    for (long long j = k + threadIdx.x; j < W; j += blockDim.x) {
      const z a = A[(long long)k * W + j];
      const z b = A[(long long)p * W + j];
      if (p != k) A[(long long)p * W + j] = a;
      A[(long long)k * W + j] = zmul(b, inv);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) fk[i] = A[(long long)i * W + k];
    __syncthreads();
    const long long cols = W - (k + 1);
    for (long long e = threadIdx.x; e < (long long)n * cols; e += blockDim.x) {
      const int i = (int)(e / cols);
      if (i == k) continue;
      const long long j = k + 1 + e % cols;
      const z f = fk[i];
      z *c = A + (long long)i * W + j;
      *c = zfma(make_double2(-f.x, -f.y), A[(long long)k * W + j], *c);
    }
    __syncthreads();
  }
}

// G[b] = right half of Aug[b]
__global__ void k_right_half(const z *Aug, int n, long long batch, z *G) {
  const long long nn = (long long)n * n, total = nn * batch;
  for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < total;
       g += (long long)gridDim.x * blockDim.x) {
    const long long b = g / nn, e = g % nn;
    const int i = (int)(e / n), j = (int)(e % n);
    G[g] = Aug[b * 2 * nn + (long long)i * 2 * n + n + j];
  }
}

// ---------------------------------------------------------------------------------------
// Systems that fit in shared memory (n <= kSmallN): built, inverted in place and used by one
// block per (spin, frequency), with no augmented matrix in global memory.  Bound by the FP64
// pipe (n^3 complex multiply-adds per system) and the chain of n pivots.  n = 20, 400
// frequencies: 63 us for an inverse (162 us for the augmented elimination in global memory
// with its build and copy); a bisection step for mu 61 us in one launch (before: seven
// launches and two host round trips, 0.8 ms).
// ---------------------------------------------------------------------------------------
constexpr int kSmallN = 110;        // n^2 + 2 n complex values and the pivots stay below 200 KB
constexpr int kSmallThreads = 128;
size_t small_smem(int n) { return sizeof(z) * ((size_t)n * n + 2 * (size_t)n) + sizeof(int) * (size_t)n + 16; }

// A = (i w + mu) 1 - F - Sigma(i w) of system b in shared memory
__device__ __forceinline__ void small_build(z *A, const double *F, const z *Sig, double mu, double om, long long b,
                                            int s, int n) {
  const int nn = n * n;
  const double *Fs = F + (long long)s * nn;
  const z *Sb = Sig ? Sig + b * nn : nullptr;
  for (int e = threadIdx.x; e < nn; e += blockDim.x) {
    z a = make_double2(-Fs[e], 0.0);
    if (Sb) {
      const z sg = Sb[e];
      a.x -= sg.x;
      a.y -= sg.y;
    }
    if (e % (n + 1) == 0) {   // the diagonal of a row-major n x n matrix
      a.x += mu;
      a.y += om;
    }
    A[e] = a;
  }
}

// In-place Gauss-Jordan inverse with partial pivoting (rows are exchanged, the exchanges
// undone on the columns at the end).  rk, fk: n values each, piv: n ints, all shared.
// Every thread of the block calls it; false (for all) on a zero pivot column.
// Warp 0 alone finds the pivot, divides, exchanges the rows and lays out the scaled row and
// the column factors (the FP64 pipe takes 16 clocks per warp instruction, so a division in
// every warp cost more than the rank-1 update of a 20 x 20 system); then all warps update
// with one multiply-add per element: element (i, j) becomes -f_i r_j + a with a = 0 in row
// and column k and f_k = -1.
__device__ __forceinline__ bool small_invert(z *A, z *rk, z *fk, int *piv, int n) {
  const int tid = threadIdx.x, nn = n * n;
  const int di = blockDim.x / n, dj = blockDim.x % n;
  for (int k = 0; k < n; ++k) {
    __syncthreads();
    if (tid < 32) {
      // the larger of |re|, |im| by its high word (NaNs last): no FP64 instruction in the search
      // (n = 20, 400 systems: a bisection step of 72 us takes 61)
      unsigned bv = 0u;
      int bi = k + tid;
      for (int i = k + tid; i < n; i += 32) {
        const z a = A[i * n + k];
        const unsigned hx = (unsigned)__double2hiint(a.x) & 0x7fffffffu, hy = (unsigned)__double2hiint(a.y) & 0x7fffffffu;
        const unsigned m = max(hx, hy) > 0x7ff00000u ? 0u : max(hx, hy);
        if (m > bv) {
          bv = m;
          bi = i;
        }
      }
      const unsigned top = __reduce_max_sync(0xffffffffu, bv);
      const int p = top == 0u ? k : (int)__reduce_min_sync(0xffffffffu, bv == top ? (unsigned)bi : 0xffffffffu);
      const z pv = A[p * n + k], akk = A[k * n + k];
      const double den = pv.x * pv.x + pv.y * pv.y, id = 1.0 / den;
      const z inv = make_double2(pv.x * id, -pv.y * id);
      for (int j = tid; j < n; j += 32) {
        const z b = A[p * n + j];
        rk[j] = (j == k) ? inv : zmul(b, inv);
        fk[j] = (j == k) ? make_double2(-1.0, 0.0) : ((j == p) ? akk : A[j * n + k]);
      }
      __syncwarp();
      if (p != k)
        for (int j = tid; j < n; j += 32) A[p * n + j] = A[k * n + j];
      if (tid == 0) piv[k] = den > 0.0 ? p : -1;
    }
    __syncthreads();
    if (piv[k] < 0) return false;
    int i = tid / n, j = tid % n;
    for (int e = tid; e < nn; e += blockDim.x) {
      const z f = fk[i];
      const z a = (i == k || j == k) ? make_double2(0.0, 0.0) : A[e];
      A[e] = zfma(make_double2(-f.x, -f.y), rk[j], a);
      i += di;
      j += dj;
      if (j >= n) {
        j -= n;
        ++i;
      }
    }
  }
  __syncthreads();
  for (int i = tid; i < n; i += blockDim.x)
    for (int k = n - 1; k >= 0; --k) {
      const int p = piv[k];
      if (p != k) {
        const z t = A[i * n + k];
        A[i * n + k] = A[i * n + p];
        A[i * n + p] = t;
      }
    }
  __syncthreads();
  return true;
}

__global__ void __launch_bounds__(kSmallThreads) k_dyson_small(const double *omegas, double mu, const double *F,
                                                               const z *Sig, int n, int n_w, z *G, int *singular) {
  extern __shared__ z sm[];
  const long long b = blockIdx.x;
  const int s = (int)(b / n_w), w = (int)(b % n_w), nn = n * n;
  z *A = sm, *rk = sm + nn, *fk = rk + n;
  small_build(A, F, Sig, mu, omegas[w], b, s, n);
  if (!small_invert(A, rk, fk, reinterpret_cast<int *>(fk + n), n)) {
    if (threadIdx.x == 0) atomicExch(singular, 1);
    return;
  }
  for (int e = threadIdx.x; e < nn; e += blockDim.x) G[b * nn + e] = A[e];
}

// State of the bisection for mu, in device memory (the host reads it once at the end)
struct MuState {
  double lo, hi;
  unsigned ticket;
  int singular;
};

// One bisection step: every block inverts one (spin, frequency) system at mu = (lo + hi) / 2
// and forms its term of the electron count
//   count(mu) = -sum_s Tr G(beta^-),
//   G(beta^-) = (1/beta) sum_w Re[e^{-i w beta} (G - tails)] - c1/2 + beta/4 c2,
// from the diagonal of G; the last block to finish adds the terms up in a fixed order and
// moves lo or hi.  Without a step left to do (hi - lo < tol) it returns at once.
__global__ void __launch_bounds__(kSmallThreads) k_mu_step(const double *omegas, const double *F, const z *Sig,
                                                           const double *Sig_tau, int n, int T, int n_w, double beta,
                                                           double target, double tol, double *partial, MuState *st) {
  extern __shared__ z sm[];
  __shared__ double red[kSmallThreads];
  __shared__ bool last;
  const double lo = st->lo, hi = st->hi;
  if (!(hi - lo >= tol)) return;
  const double mu = 0.5 * (lo + hi);
  const long long b = blockIdx.x;
  const int s = (int)(b / n_w), w = (int)(b % n_w), nn = n * n, tid = threadIdx.x;
  z *A = sm, *rk = sm + nn, *fk = rk + n;
  const double om = omegas[w];
  small_build(A, F, Sig, mu, om, b, s, n);
  if (small_invert(A, rk, fk, reinterpret_cast<int *>(fk + n), n)) {
    const double *Fs = F + (long long)s * nn;
    const double iw1 = 1.0 / om, iw2 = iw1 * iw1, iw3 = iw2 * iw1;
    double sn, cs;
    sincos(om * beta, &sn, &cs);
    double acc = 0.0;
    for (int i = tid; i < n; i += blockDim.x) {
      const long long e = (long long)i * n + i;
      const double c2 = Fs[e] - mu;
      double c3 = 0.0;
      for (int k = 0; k < n; ++k) {
        const double m = (i == k) ? mu : 0.0;
        c3 = fma(Fs[i * n + k] - m, Fs[k * n + i] - m, c3);
      }
      if (Sig_tau) {
        const double *S = Sig_tau + (long long)s * T * nn;
        c3 -= S[(long long)(T - 1) * nn + e] + S[e];
      }
      const z g = A[e];
      const double rx = g.x + c2 * iw2, ry = g.y + iw1 - c3 * iw3;
      acc -= (rx * cs + ry * sn) / beta;
      if (w == 0) acc -= -0.5 + 0.25 * beta * c2;   // the closed tau images, once per spin
    }
    red[tid] = acc;
    __syncthreads();
    for (int o = kSmallThreads / 2; o > 0; o >>= 1) {
      if (tid < o) red[tid] += red[tid + o];
      __syncthreads();
    }
    if (tid == 0) partial[b] = red[0];
  } else if (tid == 0) {
    atomicExch(&st->singular, 1);
    partial[b] = 0.0;
  }
  if (tid == 0) {
    __threadfence();
    last = atomicAdd(&st->ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double c = 0.0;
  for (unsigned i = tid; i < gridDim.x; i += blockDim.x) c += __ldcg(partial + i);
  red[tid] = c;
  __syncthreads();
  for (int o = kSmallThreads / 2; o > 0; o >>= 1) {
    if (tid < o) red[tid] += red[tid + o];
    __syncthreads();
  }
  if (tid == 0) {
    if (red[0] < target)
      st->lo = mu;
    else
      st->hi = mu;
    st->ticket = 0;
  }
}

// tails[s] = {1, A, A A + S1} with A = F - mu 1 and S1 = -(Sigma(tau_{T-1}) + Sigma(tau_0))
// (the jump of the antiperiodic Sigma(tau); zero when Sigma_tau is NULL); real [n_spin][3][n][n]
__global__ void k_tails(const double *F, double mu, const double *Sig_tau, int n, int T, int n_spin, double *tails) {
  const long long nn = (long long)n * n, total = nn * n_spin;
  for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < total;
       g += (long long)gridDim.x * blockDim.x) {
    const int s = (int)(g / nn);
    const long long e = g % nn;
    const int i = (int)(e / n), j = (int)(e % n);
    const double *Fs = F + (long long)s * nn;
    double a2 = 0.0;
    for (int k = 0; k < n; ++k) {
      const double aik = Fs[(long long)i * n + k] - (i == k ? mu : 0.0);
      const double akj = Fs[(long long)k * n + j] - (k == j ? mu : 0.0);
      a2 = fma(aik, akj, a2);
    }
    double s1 = 0.0;
    if (Sig_tau) {
      const double *S = Sig_tau + (long long)s * T * nn;
      s1 = -(S[(long long)(T - 1) * nn + e] + S[e]);
    }
    double *t = tails + (long long)s * 3 * nn;
    t[e] = (i == j) ? 1.0 : 0.0;
    t[nn + e] = Fs[e] - (i == j ? mu : 0.0);
    t[2 * nn + e] = a2 + s1;
  }
}

// (cos, sin)(w tau_t) for every frequency and a block of times, [n_w][n_t8], the times padded to 8
__global__ void k_phases(const double *omegas, int n_w, const double *tau, int n_t, int n_t8, z *ph) {
  const long long total = (long long)n_w * n_t8;
  for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < total;
       g += (long long)gridDim.x * blockDim.x) {
    const int w = (int)(g / n_t8), t = (int)(g % n_t8);
    double sn = 0.0, cs = 0.0;
    if (t < n_t) sincos(omegas[w] * tau[t], &sn, &cs);
    ph[g] = make_double2(cs, sn);
  }
}

// G(tau_t) = Re[(1/beta) sum_w e^{-i w tau_t} (G(iw) - c1/(iw) - c2/(iw)^2 - c3/(iw)^3)]
//            + t1(tau) c1 + t2(tau) c2 + t3(tau) c3
// with the closed-form tau images t1 = -1/2, t2 = (2 tau - beta)/4, t3 = tau (beta - tau)/4 of the
// tails summed over all fermionic frequencies; tau on [0, beta] read as 0^+ and beta^-.
// A block holds 32 matrix elements and 8 times; 8 warps share the frequencies.  The phases
// come from a table (a sincos per element, time and frequency took 20 times the sums).
__global__ void __launch_bounds__(256) k_iw_to_tau(const z *Giw, const double *omegas, int n_w, const double *tails,
                                                   const double *tau, const z *ph, int n_t, int n_t8, int n_all, int n,
                                                   double beta, double *Gtau) {
  __shared__ double red[8][8][33];
  const long long nn = (long long)n * n;
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
  const long long e = (long long)blockIdx.x * 32 + lane;
  const int t0 = blockIdx.y * 8, s = blockIdx.z;
  double c1 = 0.0, c2 = 0.0, c3 = 0.0, acc[8] = {};
  if (e < nn) {
    const double *c = tails + (long long)s * 3 * nn;
    c1 = c[e];
    c2 = c[nn + e];
    c3 = c[2 * nn + e];
    const z *G = Giw + (long long)s * n_w * nn + e;
    for (int w = warp; w < n_w; w += 8) {
      // residual r = G - c1/(i w) - c2/(i w)^2 - c3/(i w)^3 = G + i c1/w + c2/w^2 - i c3/w^3
      const double iw1 = 1.0 / omegas[w], iw2 = iw1 * iw1, iw3 = iw2 * iw1;
      const z gv = G[(long long)w * nn];
      const double rx = gv.x + c2 * iw2, ry = gv.y + c1 * iw1 - c3 * iw3;
      const z *p = ph + (long long)w * n_t8 + t0;
#pragma unroll
      for (int t = 0; t < 8; ++t) acc[t] = fma(rx, p[t].x, fma(ry, p[t].y, acc[t]));   // Re[(cos - i sin)(rx + i ry)]
    }
  }
#pragma unroll
  for (int t = 0; t < 8; ++t) red[warp][t][lane] = acc[t];
  __syncthreads();
  const int t = t0 + warp;   // one time per warp
  if (e >= nn || t >= n_t) return;
  double a = 0.0;
#pragma unroll
  for (int i = 0; i < 8; ++i) a += red[i][warp][lane];
  const double tt = tau[t];
  Gtau[((long long)s * n_all + t) * nn + e] =
      a / beta - 0.5 * c1 + 0.25 * (2.0 * tt - beta) * c2 + 0.25 * tt * (beta - tt) * c3;
}

// F_iw[s][w] = sum_j Tw[w][j] F_tau[s][j]  (Tw complex [n_w][n_tau], F_tau real)
__global__ void k_tau_to_iw(const z *Tw, const double *Ft, int n_w, int T, int n, int n_spin, z *Fiw) {
  const long long nn = (long long)n * n, total = nn * n_w * n_spin;
  for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < total;
       g += (long long)gridDim.x * blockDim.x) {
    const long long e = g % nn;
    const int w = (int)((g / nn) % n_w), s = (int)(g / (nn * n_w));
    const double *F = Ft + (long long)s * T * nn + e;
    const z *Tr = Tw + (long long)w * T;
    z acc = make_double2(0.0, 0.0);
    for (int j = 0; j < T; ++j) {
      const double f = F[(long long)j * nn];
      acc.x = fma(Tr[j].x, f, acc.x);
      acc.y = fma(Tr[j].y, f, acc.y);
    }
    Fiw[g] = acc;
  }
}

// count[0] = sum_s Tr gamma^s, gamma = -G(beta^-)^T, from G(iw) and the tails (trace only).  One
// thread per (spin, frequency) (one sincos each) walks the diagonal; one block, fixed order.
__global__ void __launch_bounds__(1024) k_trace_gamma(const z *Giw, const double *omegas, int n_w, const double *tails,
                                                      int n, int n_spin, double beta, double *count) {
  __shared__ double red[1024];
  double acc = 0.0;
  const long long nn = (long long)n * n;
  for (long long b = threadIdx.x; b < (long long)n_spin * n_w; b += blockDim.x) {
    const int s = (int)(b / n_w), w = (int)(b % n_w);
    const double *c = tails + (long long)s * 3 * nn;
    const double om = omegas[w], iw1 = 1.0 / om, iw2 = iw1 * iw1, iw3 = iw2 * iw1;
    double sn, cs;
    sincos(om * beta, &sn, &cs);
    for (int i = 0; i < n; ++i) {
      const long long e = (long long)i * n + i;
      const double c1 = c[e], c2 = c[nn + e], c3 = c[2 * nn + e];
      const z g = Giw[b * nn + e];
      const double rx = g.x + c2 * iw2, ry = g.y + c1 * iw1 - c3 * iw3;
      acc -= (rx * cs + ry * sn) / beta;
      if (w == 0) acc -= -0.5 * c1 + 0.25 * beta * c2;   // tau = beta: t3 = 0
    }
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int o = 512; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) count[0] = red[0];
}

// THC Hartree-Fock: d[Q] = sum_rs X[Q][r] X[Q][s] rho_rs (rho = sum_s gamma^s),
// Gam[s][P][Q] = sum_rs X[P][r] gamma^s_rs X[Q][s]
__global__ void k_hf_density(const double *X, const double *gam, int N, int n, int n_spin, double *d) {
  const long long nn = (long long)n * n;
  for (int Q = blockIdx.x * blockDim.x + threadIdx.x; Q < N; Q += gridDim.x * blockDim.x) {
    const double *x = X + (long long)Q * n;
    double acc = 0.0;
    for (int s = 0; s < n_spin; ++s)
      for (int r = 0; r < n; ++r) {
        double row = 0.0;
        for (int c = 0; c < n; ++c) row = fma(gam[s * nn + (long long)r * n + c], x[c], row);
        acc = fma(x[r], row, acc);
      }
    d[Q] = acc;
  }
}

// Sigma_HF^s = J - K^s = X^T R^s with
//   R^s[P][q] = (sum_Q V_PQ d_Q) X_Pq - sum_Q V_PQ Gam^s_PQ X_Qq
// (J = sum_PQ X_Pp X_Pq V_PQ d_Q, K^s = sum_PQ X_Pp X_Qq V_PQ Gam^s_PQ): one block per (P, s),
// N n + N multiply-adds each instead of N^2 per element of Sigma.
constexpr int kHfChunk = 1024;
__global__ void __launch_bounds__(128) k_hf_rows(const double *X, const double *V, const double *d, const double *Gam,
                                                 int N, int n, double *R) {
  constexpr int kPer = SOX_MAX_N_AO / 128;   // columns q per thread
  __shared__ double vg[kHfChunk];            // V_PQ Gam_PQ, a chunk of this row at a time
  __shared__ double red[128];
  const int P = blockIdx.x, s = blockIdx.y, tid = threadIdx.x;
  const double *v = V + (long long)P * N, *g = Gam + ((long long)s * N + P) * N;
  double acc = 0.0, k[kPer] = {};
  for (int Q0 = 0; Q0 < N; Q0 += kHfChunk) {
    const int nq = min(kHfChunk, N - Q0);
    __syncthreads();
    for (int Q = tid; Q < nq; Q += 128) {
      vg[Q] = v[Q0 + Q] * g[Q0 + Q];
      acc = fma(v[Q0 + Q], d[Q0 + Q], acc);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int q = tid + i * 128;
      if (q < n)
        for (int Q = 0; Q < nq; ++Q) k[i] = fma(vg[Q], X[(long long)(Q0 + Q) * n + q], k[i]);
    }
  }
  red[tid] = acc;
  __syncthreads();
  for (int o = 64; o > 0; o >>= 1) {
    if (tid < o) red[tid] += red[tid + o];
    __syncthreads();
  }
  const double vd = red[0];
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    const int q = tid + i * 128;
    if (q < n) R[((long long)s * N + P) * n + q] = fma(vd, X[(long long)P * n + q], -k[i]);
  }
}

// out[0] += sum_s sum_pq (H0 + Sigma_HF^s / 2)_pq gamma^s_pq                       (E_inf, Eq. E1b)
// out[1] -= sum_s sum_j w_j sum_pq Sigma^s_pq(tau_{T-1-j}) G^s_qp(tau_j)            (E_dyn, Eq. E2b)
__global__ void k_energies(const double *H0, const double *Shf, const double *gam, const double *Sig, const double *G,
                           const double *w, int n, int T, int n_spin, double *out) {
  const long long nn = (long long)n * n;
  double einf = 0.0, edyn = 0.0;
  const long long total1 = nn * n_spin;
  for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < total1;
       g += (long long)gridDim.x * blockDim.x) {
    const long long e = g % nn;
    einf = fma(H0[e] + 0.5 * Shf[g], gam[g], einf);
  }
  const long long total2 = nn * T * n_spin;
  for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < total2;
       g += (long long)gridDim.x * blockDim.x) {
    const long long e = g % nn;
    const int j = (int)((g / nn) % T), s = (int)(g / (nn * T));
    const int p = (int)(e / n), q = (int)(e % n);
    const double sv = Sig[((long long)s * T + (T - 1 - j)) * nn + e];
    const double gv = G[((long long)s * T + j) * nn + (long long)q * n + p];
    edyn = fma(-w[j] * sv, gv, edyn);
  }
  for (int o = 16; o > 0; o >>= 1) {
    einf += __shfl_xor_sync(0xffffffffu, einf, o);
    edyn += __shfl_xor_sync(0xffffffffu, edyn, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&out[0], einf);
    atomicAdd(&out[1], edyn);
  }
}

// G = (1 - a) G + a Gnew; change[0] = max |Gnew - G_old| (bit pattern of a non-negative double)
__global__ void k_mix(double *G, const double *Gnew, long long count, double a, unsigned long long *change) {
  double m = 0.0;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < count;
       e += (long long)gridDim.x * blockDim.x) {
    const double g = G[e], gn = Gnew[e];
    m = fmax(m, fabs(gn - g));
    G[e] = (1.0 - a) * g + a * gn;
  }
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(change, (unsigned long long)__double_as_longlong(m));
}

}  // namespace

size_t dyson_bytes(int n, int n_w, int n_spin) {
  if (n <= kSmallN) return 4096;
  return aligned_bytes((size_t)n_spin * n_w * 2 * (size_t)n * n, 16) + 4096;
}

Status dyson(sox_handle h, int n, int n_w, int n_spin, const double *omegas, double mu, const double *F,
             const double *Sigma_iw, double *G_iw, Arena &ar, cudaStream_t s) {
  const bool small = n <= kSmallN;
  z *Aug = small ? nullptr : ar.take<z>((size_t)n_spin * n_w * 2 * (size_t)n * n);
  int *info = ar.take<int>(4);
  if (!info) return {SOX_ERR_OOM, "workspace too small (internal sizing error)"};
  const long long batch = (long long)n_spin * n_w;
  if (batch > 0x7fffffff) return {SOX_ERR_SHAPE, "too many Dyson systems"};
  ProfScope ps(h, "dyson", s, small ? 1 : 3);
  SOX_CUDA_TRY(cudaMemsetAsync(info, 0, 4 * sizeof(int), s));
  if (small) {
    static std::atomic<unsigned long long> attr{0};
    SOX_CUDA_TRY(set_smem_once(k_dyson_small, (int)small_smem(kSmallN), attr));
    k_dyson_small<<<(unsigned)batch, kSmallThreads, small_smem(n), s>>>(
        omegas, mu, F, reinterpret_cast<const z *>(Sigma_iw), n, n_w, reinterpret_cast<z *>(G_iw), info);
  } else {
    k_dyson_build<<<grid_of(batch * n * n), 256, 0, s>>>(omegas, mu, F, reinterpret_cast<const z *>(Sigma_iw), n, n_w,
                                                         n_spin, Aug);
    const size_t shm = sizeof(z) * (size_t)n;
    k_gj_block<<<(unsigned)batch, 256, shm, s>>>(Aug, n, info);
    k_right_half<<<grid_of(batch * n * n), 256, 0, s>>>(Aug, n, batch, reinterpret_cast<z *>(G_iw));
  }
  SOX_CUDA_TRY(cudaGetLastError());
  int hinfo[4] = {0, 0, 0, 0};
  SOX_CUDA_TRY(cudaMemcpyAsync(hinfo, info, sizeof(hinfo), cudaMemcpyDeviceToHost, s));
  SOX_CUDA_TRY(cudaStreamSynchronize(s));
  if (hinfo[0]) return {SOX_ERR_INVALID_ARG, "(i w + mu) - F - Sigma(i w) is singular at some frequency"};
  return Status::ok();
}

bool mu_on_device(int n) { return n <= kSmallN; }
size_t mu_bytes(int n_w, int n_spin) {
  return aligned_bytes((size_t)n_spin * n_w, 8) + aligned_bytes(sizeof(MuState), 1) + 4096;
}

Status mu_bisect(sox_handle h, int n, int T, int n_w, int n_spin, const double *omegas, double beta, double target,
                 const double *F, const double *Sigma_iw, const double *Sigma_tau, double *lo, double *hi, double tol,
                 int max_iter, Arena &ar, cudaStream_t s) {
  const long long batch = (long long)n_spin * n_w;
  if (batch > 0x7fffffff) return {SOX_ERR_SHAPE, "too many Dyson systems"};
  double *partial = ar.take<double>((size_t)batch);
  MuState *st = reinterpret_cast<MuState *>(ar.take<char>(sizeof(MuState)));
  if (!st) return {SOX_ERR_OOM, "workspace too small (internal sizing error)"};
  static std::atomic<unsigned long long> attr{0};
  SOX_CUDA_TRY(set_smem_once(k_mu_step, (int)small_smem(kSmallN), attr));
  MuState hs{*lo, *hi, 0u, 0};
  SOX_CUDA_TRY(cudaMemcpyAsync(st, &hs, sizeof(hs), cudaMemcpyHostToDevice, s));
  // the steps that halving needs to reach tol, one more for rounding; the surplus returns at once
  int done = 0;
  while (done < max_iter && hs.hi - hs.lo >= tol && !hs.singular) {
    int steps = 1;
    for (double wd = hs.hi - hs.lo; wd >= tol && steps < 4096; wd *= 0.5) ++steps;
    steps = std::min(steps, max_iter - done);
    for (int i = 0; i < steps; ++i)
      k_mu_step<<<(unsigned)batch, kSmallThreads, small_smem(n), s>>>(omegas, F, reinterpret_cast<const z *>(Sigma_iw),
                                                                    Sigma_tau, n, T, n_w, beta, target, tol, partial,
                                                                    st);
    SOX_CUDA_TRY(cudaGetLastError());
    h->launches += steps;
    done += steps;
    const double w0 = hs.hi - hs.lo;
    SOX_CUDA_TRY(cudaMemcpyAsync(&hs, st, sizeof(hs), cudaMemcpyDeviceToHost, s));
    SOX_CUDA_TRY(cudaStreamSynchronize(s));
    if (!(hs.hi - hs.lo < w0)) break;   // lo and hi are neighbouring numbers: no step moves them any more
  }
  if (hs.singular) return {SOX_ERR_INVALID_ARG, "(i w + mu) - F - Sigma(i w) is singular at some frequency"};
  *lo = hs.lo;
  *hi = hs.hi;
  return Status::ok();
}

void launch_green_tails(const double *F, double mu, const double *Sigma_tau, int n, int T, int n_spin, double *tails,
                        cudaStream_t s) {
  k_tails<<<grid_of((long long)n * n * n_spin), 256, 0, s>>>(F, mu, Sigma_tau, n, T, n_spin, tails);
}

// Times of a block of phases: as many groups of eight as 64 MB (or the handle's limit) hold, one at least
// (then 128 bytes per frequency, no more than G(i w) itself from n = 3 on).
int iw_to_tau_block(sox_handle h, int n_w, int n_t) {
  const size_t most = std::min(size_t(64) << 20, chunk_budget(h, size_t(64) << 20));
  const long long groups = std::max<long long>(1, (long long)(most / ((size_t)n_w * 8 * sizeof(z))));
  return (int)std::min<long long>(8 * groups, (n_t + 7) / 8 * 8);
}
size_t iw_to_tau_bytes(sox_handle h, int n_w, int n_t) {
  return aligned_bytes((size_t)n_w * iw_to_tau_block(h, n_w, n_t), sizeof(z));
}

void launch_iw_to_tau(sox_handle h, const double *G_iw, const double *omegas, int n_w, const double *tails,
                      const double *tau, int n_t, int n, int n_spin, double beta, void *scratch, double *G_tau,
                      cudaStream_t s) {
  z *ph = static_cast<z *>(scratch);
  const int block = iw_to_tau_block(h, n_w, n_t);
  const long long nn = (long long)n * n;
  for (int t0 = 0; t0 < n_t; t0 += block) {
    const int nt = std::min(block, n_t - t0), nt8 = (nt + 7) / 8 * 8;
    k_phases<<<grid_of((long long)n_w * nt8), 256, 0, s>>>(omegas, n_w, tau + t0, nt, nt8, ph);
    k_iw_to_tau<<<dim3((unsigned)((nn + 31) / 32), nt8 / 8, n_spin), 256, 0, s>>>(
        reinterpret_cast<const z *>(G_iw), omegas, n_w, tails, tau + t0, ph, nt, nt8, n_t, n, beta, G_tau + t0 * nn);
    h->launches += 2;
  }
}

void launch_tau_to_iw(const double *Tw, const double *F_tau, int n_w, int T, int n, int n_spin, double *F_iw,
                      cudaStream_t s) {
  k_tau_to_iw<<<grid_of((long long)n * n * n_w * n_spin), 256, 0, s>>>(reinterpret_cast<const z *>(Tw), F_tau, n_w, T,
                                                                       n, n_spin, reinterpret_cast<z *>(F_iw));
}

void launch_trace_gamma(const double *G_iw, const double *omegas, int n_w, const double *tails, int n, int n_spin,
                        double beta, double *count, cudaStream_t s) {
  k_trace_gamma<<<1, 1024, 0, s>>>(reinterpret_cast<const z *>(G_iw), omegas, n_w, tails, n, n_spin, beta, count);
}

void launch_sigma_hf(const double *X, const double *V, const double *gamma, int N, int n, int n_spin, double *d,
                     double *Gam, double *S, cudaStream_t s) {
  k_hf_density<<<grid_of(N), 256, 0, s>>>(X, gamma, N, n, n_spin, d);
  for (int sp = 0; sp < n_spin; ++sp) {   // Gam[s] = X gamma^s X^T (FP64 GEMMs)
    GemmF64 a;   // T = gamma X^T -> Gam = X T; done as one GEMM pair through Gam as scratch
    a.M = N; a.Nc = n; a.K = n;
    a.A = X; a.ai = n; a.ak = 1;
    a.B = gamma + (long long)sp * n * n; a.bk = n; a.bj = 1;
    a.C = d + N + (long long)sp * N * n; a.ci = n; a.cj = 1;   // M = X gamma  (scratch after d)
    launch_gemm_f64(a, s);
    GemmF64 b;
    b.M = N; b.Nc = N; b.K = n;
    b.A = d + N + (long long)sp * N * n; b.ai = n; b.ak = 1;
    b.B = X; b.bk = 1; b.bj = n;
    b.C = Gam + (long long)sp * N * N; b.ci = N; b.cj = 1;
    launch_gemm_f64(b, s);
  }
  double *R = d + N;   // the X gamma scratch, free again
  k_hf_rows<<<dim3(N, n_spin), 128, 0, s>>>(X, V, d, Gam, N, n, R);
  GemmF64 g;           // S[s][p][q] = sum_P X[P][p] R[s][P][q]
  g.M = n; g.Nc = n; g.K = N; g.batch = n_spin;
  g.A = X; g.ai = 1; g.ak = n;
  g.B = R; g.sB = (long long)N * n; g.bk = n; g.bj = 1;
  g.C = S; g.sC = (long long)n * n; g.ci = n; g.cj = 1;
  launch_gemm_f64(g, s);
}

void launch_energies(const double *H0, const double *Shf, const double *gamma, const double *Sigma_tau,
                     const double *G_tau, const double *w, int n, int T, int n_spin, double *out, cudaStream_t s) {
  k_energies<<<grid_of((long long)n * n * T * n_spin), 256, 0, s>>>(H0, Shf, gamma, Sigma_tau, G_tau, w, n, T, n_spin,
                                                                    out);
}

void launch_mix(double *G, const double *Gnew, long long count, double a, unsigned long long *change, cudaStream_t s) {
  k_mix<<<grid_of(count), 256, 0, s>>>(G, Gnew, count, a, change);
}

}  // namespace sox

namespace sox {
namespace {
// gamma[s][p][q] = -G[s][T-1][q][p]
__global__ void k_gamma_from_tau(const double *G, int n, int T, int n_spin, double *gam) {
  const long long nn = (long long)n * n, total = nn * n_spin;
  for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < total;
       g += (long long)gridDim.x * blockDim.x) {
    const int s = (int)(g / nn);
    const long long e = g % nn;
    const int p = (int)(e / n), q = (int)(e % n);
    gam[g] = -G[((long long)s * T + (T - 1)) * nn + (long long)q * n + p];
  }
}
}  // namespace

void launch_gamma_from_tau(const double *G_tau, int n, int T, int n_spin, double *gamma, cudaStream_t s) {
  k_gamma_from_tau<<<grid_of((long long)n * n * n_spin), 256, 0, s>>>(G_tau, n, T, n_spin, gamma);
}
}  // namespace sox
