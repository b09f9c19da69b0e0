// sm_103a building blocks for the tensor-core path: mbarriers with bounded
// waits, TMA tiled loads, tcgen05 MMA / commit / TMEM load, shared-memory and
// instruction descriptors, and host-side tensor-map encoding.
#pragma once

#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <cstdint>

namespace sox {
namespace tc {

// ----------------------------- device side --------------------------------

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_barrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait on phase `parity`.  On exhaustion sets *abort (shared) and the
// global status word, and returns false; the caller then winds down.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, long long limit,
                                          volatile int *abort, int *status, int code) {
  for (long long i = 0; i < limit; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if (*abort) return false;
  }
  *abort = 1;
  atomicOr(status, code);
  return false;
}

// The same for a whole warp: its lanes go on together or leave together.  (A lane that alone sees
// the wait run out, or the abort flag, must not leave the others in warp-wide loads, shuffles and
// barriers.)
__device__ __forceinline__ bool mbar_wait_warp(uint64_t *bar, uint32_t parity, long long limit,
                                               volatile int *abort, int *status, int code) {
  const bool got = mbar_wait(bar, parity, limit, abort, status, code);
  return __all_sync(0xffffffffu, got && !*abort);
}

// Phase bookkeeping for a stage ring whose full barriers come in two sets, one per MMA
// issuer (full[q][s]), fed by one TMA producer.  Bit 16q + s of `par` is the parity of the
// next phase the holder expects on full[q][s]; bit 16q + s of `used` marks a barrier the
// producer has issued on.  Registers only: the set index is a runtime value.
struct RingPhases {
  uint32_t par = 0u, used = 0u;
  __device__ __forceinline__ uint32_t next(int q, int s) const { return (par >> (16 * q + s)) & 1u; }
  // takes the next phase of full[q][s] and returns its parity
  __device__ __forceinline__ uint32_t take(int q, int s) {
    const uint32_t m = 1u << (16 * q + s);
    const uint32_t ph = (par & m) ? 1u : 0u;
    par ^= m;
    used |= m;
    return ph;
  }
};

// Order of one v's 2 nk chunks in a fused kernel's stage ring (nk chunks each for the B_v
// and the C_v products, issued by two MMA threads): groups of g chunks of B_v and g of C_v
// alternate, so ring positions [2gj, 2gj + g) hold B chunks gj .. gj + g - 1 and the next
// g positions the same C chunks (the last group may be shorter).  g = 1 alternates single
// chunks, g = nk runs all of B_v's chunks, then all of C_v's.
// chunk kc and half h (0: B_v, 1: C_v) at position p of the v's chunks
__device__ __forceinline__ void bc_decode(int p, int nk, int g, int &kc, int &h) {
  const int j = p / (2 * g);
  const int gl = min(g, nk - j * g);
  const int w = p - 2 * g * j;
  h = w >= gl ? 1 : 0;
  kc = j * g + w - h * gl;
}
// position of chunk kc of half h
__device__ __forceinline__ int bc_pos(int kc, int h, int nk, int g) {
  const int j = kc / g, w = kc - j * g;
  const int gl = min(g, nk - j * g);
  return 2 * g * j + h * gl + w;
}

// Producer wind-down: waits (at most `limit` polls each) until the last phase issued on
// every barrier of both sets has completed, so no TMA write is in flight when the CTA
// leaves.
template <int S>
__device__ __forceinline__ void ring_wind_down(uint64_t (&full)[2][S], const RingPhases &r, long long limit) {
  static_assert(S <= 16, "RingPhases keeps 16 stages per set");
  for (int q = 0; q < 2; ++q)
    for (int s = 0; s < S; ++s)
      if ((r.used >> (16 * q + s)) & 1u) {
        const uint32_t ph = r.next(q, s) ^ 1u;
        for (long long i = 0; i < limit && !mbar_try_wait(&full[q][s], ph); ++i) {
        }
      }
}

// 3-D tiled TMA load into shared memory, completion counted on `bar`.
__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, uint64_t *bar, int x,
                                            int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z)
      : "memory");
}

__device__ __forceinline__ void prefetch_tmap(const CUtensorMap *map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

// --- tcgen05 ---
__device__ __forceinline__ void tmem_alloc(uint32_t *dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
               "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// D[tmem] (+)= A[smem] * B[smem]^T, kind::f16 (FP16 inputs, FP32 accumulate), cta_group::1.
__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                        uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Arrive once on `bar` when every tcgen05.mma issued so far by this thread has completed.
__device__ __forceinline__ void mma_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_u32(bar))
               : "memory");
}

// 32 lanes x 32 consecutive 32-bit columns: thread i of the warp gets lane (base lane + i).
__device__ __forceinline__ void tmem_ld_32x32b_x32(uint32_t taddr, float (&r)[32]) {
  uint32_t u[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
      "%13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, "
      "[%32];"
      : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]),
        "=r"(u[8]), "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]),
        "=r"(u[15]), "=r"(u[16]), "=r"(u[17]), "=r"(u[18]), "=r"(u[19]), "=r"(u[20]), "=r"(u[21]),
        "=r"(u[22]), "=r"(u[23]), "=r"(u[24]), "=r"(u[25]), "=r"(u[26]), "=r"(u[27]), "=r"(u[28]),
        "=r"(u[29]), "=r"(u[30]), "=r"(u[31])
      : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 32; ++i) r[i] = __uint_as_float(u[i]);
}
// 32 lanes x 16 consecutive 32-bit columns.
__device__ __forceinline__ void tmem_ld_32x32b_x16(uint32_t taddr, float (&r)[16]) {
  uint32_t u[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
      "%13, %14, %15}, [%16];"
      : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]),
        "=r"(u[8]), "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]),
        "=r"(u[15])
      : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 16; ++i) r[i] = __uint_as_float(u[i]);
}
// 32 lanes x 8 consecutive 32-bit columns.
__device__ __forceinline__ void tmem_ld_32x32b_x8(uint32_t taddr, float (&r)[8]) {
  uint32_t u[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7])
               : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 8; ++i) r[i] = __uint_as_float(u[i]);
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor for a K-major tile written by TMA with
// 128-byte swizzle: rows of 128 bytes, 8-row atoms 1024 bytes apart.
__device__ __forceinline__ uint64_t desc_kmajor_sw128(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);   // start address
  d |= (uint64_t)1 << 16;                      // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;            // stride byte offset: next 8-row group
  d |= (uint64_t)1 << 46;                      // descriptor version (tcgen05)
  d |= (uint64_t)2 << 61;                      // layout: 128-byte swizzle
  return d;
}

// Instruction descriptor: kind::f16, A = B = FP16, D = FP32, both K-major, M x N.
__host__ __device__ constexpr uint32_t idesc_f16_f32(int M, int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// --- CTA pairs (cluster of two CTAs on neighbouring SMs, cta_group::2) ---
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// shared::cluster address of the variable at shared::cta address `saddr` in CTA `rank`
__device__ __forceinline__ uint32_t mapa_shared(uint32_t saddr, uint32_t rank) {
  uint32_t d;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(saddr), "r"(rank));
  return d;
}
// arrive (release at cluster scope) on an mbarrier given by its shared::cluster address
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t caddr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(caddr) : "memory");
}
// every thread of both CTAs: arrive (release) then wait (acquire) on the cluster barrier
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// 3-D tiled TMA load into this CTA's shared memory whose completion is counted on an
// mbarrier of either CTA of the pair (`bar_caddr`: shared::cluster address)
__device__ __forceinline__ void tma_load_3d_pair(void *dst, const CUtensorMap *map, uint32_t bar_caddr, int x, int y,
                                                 int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar_caddr), "r"(x), "r"(y), "r"(z)
      : "memory");
}
// TMEM of both CTAs of the pair: one warp of each CTA executes these
__device__ __forceinline__ void tmem_alloc_pair(uint32_t *dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
               "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// Pair MMA issued by one thread of the even CTA: A rows [0, M/2) from the even CTA's shared
// memory and [M/2, M) from the odd one's (same offsets), B rows [0, N/2) and [N/2, N)
// likewise; each CTA's TMEM receives its own M/2 rows of D.
__device__ __forceinline__ void mma_f16_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                             uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrive once on the mbarrier at `bar`'s offset in every CTA of `mask` when the pair MMAs
// issued so far by this thread have completed.
__device__ __forceinline__ void mma_commit_pair_mc(uint64_t *bar, uint16_t mask) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
                   smem_u32(bar)),
               "h"(mask)
               : "memory");
}
__device__ __forceinline__ void mma_commit_pair(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

// power-of-two helpers for the split scales
__device__ __forceinline__ float pow2_floor_inv(float m) {
  // 2^-floor(log2 m) for m > 0 (exact power of two), 1 for m == 0.  The exponent
  // is clamped to [-120, 120] so the scale and its inverse stay normal FP32
  // numbers; rows below 2^-120 then split to zero (far below any tolerance).
  if (!(m > 0.f)) return 1.f;
  int e;
  frexpf(m, &e);              // m = f * 2^e, f in [0.5, 1)
  int k = 1 - e;              // 2^-(e-1) = 2^-floor(log2 m)
  k = k < -120 ? -120 : (k > 120 ? 120 : k);
  return ldexpf(1.f, k);
}

// 2^(14 - floor(log2 m)) for m > 0 (m in [2^e, 2^(e+1)) -> scaled max in [2^14, 2^15)), 1 for
// m == 0; clamped to normal FP32 powers of two
__device__ __forceinline__ float big_scale(float m) {
  if (!(m > 0.f)) return 1.f;
  int e;
  frexpf(m, &e);   // m = f 2^e, f in [0.5, 1): floor(log2 m) = e - 1
  int k = 15 - e;
  k = k < -120 ? -120 : (k > 120 ? 120 : k);
  return ldexpf(1.f, k);
}

// x = hi + lo (FP16 pair) after scaling; hi rounds to nearest.
__device__ __forceinline__ void split_f16(float x, __half &hi, __half &lo) {
  hi = __float2half_rn(x);
  lo = __float2half_rn(x - __half2float(hi));
}

// The FP16 pairs of x0 and x1 packed two to a word (x0 in the low half): the same values
// as split_f16 on each, from two packed conversions instead of four single ones.
__device__ __forceinline__ void split_f16x2(float x0, float x1, uint32_t &hi, uint32_t &lo) {
  const __half2 h = __floats2half2_rn(x0, x1);
  const float2 hf = __half22float2(h);
  const __half2 l = __floats2half2_rn(x0 - hf.x, x1 - hf.y);
  hi = *reinterpret_cast<const uint32_t *>(&h);
  lo = *reinterpret_cast<const uint32_t *>(&l);
}

// FP64 values into FP32 and FP16 pairs without the FP64 pipe (1.9 lanes a clock and SM: a
// conversion or a subtraction there costs as much as forty other instructions).

// (float)x, round to nearest even
__device__ __forceinline__ float f32_of(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const int ef = (int)((hi >> 20) & 0x7ffu);
  if (ef == 0) return __uint_as_float(hi & 0x80000000u);      // FP64 subnormals lie below FP32's
  if (ef < 898 || ef > 1149) return (float)x;                 // FP32 subnormals, overflow, infinities, NaNs
  uint32_t u = ((uint32_t)(ef - 896) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
  const uint32_t rem = lo & 0x1fffffffu;
  u += (rem + (u & 1u)) > 0x10000000u ? 1u : 0u;
  return __uint_as_float(u | (hi & 0x80000000u));
}
__device__ __forceinline__ float f32_abs(double x) {
  return f32_of(__hiloint2double(__double2hiint(x) & 0x7fffffff, __double2loint(x)));
}

// exponent k of a power of two s = 2^k (normal)
__device__ __forceinline__ int log2_of(float s) { return (int)((__float_as_uint(s) >> 23) & 0xffu) - 127; }

// FP16 pair of x 2^k: h = RN16(RN32(x 2^k)), l = RN16(RN32(x 2^k - h)).  With f = RN32(x 2^k) and
// the 29 bits g = x 2^k - f that FP32 drops, f - h is exact in FP32 and l = RN16(RN32(f - h + g)).
// g has up to 28 bits: it enters with its last four as a sticky bit, far below the rounding of
// the sum, or rounded by itself where f = h.  (Rounded to FP32 in every case one value in 10^9 came
// out a bit off, and one value of a long operand shows in the last digits of a whole output row.)
__device__ __forceinline__ void split_f16_f64(double x, int k, __half &h, __half &l) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const int ef = (int)((hi >> 20) & 0x7ffu), e = ef + k - 1023;   // exponent of x 2^k
  if (e < -30 || e > 15 || ef == 0 || ef == 0x7ff) {
    if (ef == 0 || e < -30) {   // rounds to zero in both halves
      h = l = __ushort_as_half(0);
    } else {                    // infinities, NaNs, values above the range of the scale
      const double xs = x * scalbn(1.0, k);
      h = __float2half_rn((float)xs);
      l = __float2half_rn((float)(xs - (double)__half2float(h)));
    }
    return;
  }
  uint32_t u = ((uint32_t)(e + 127) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
  const uint32_t rem = lo & 0x1fffffffu;
  const bool up = (rem + (u & 1u)) > 0x10000000u;
  u += up ? 1u : 0u;
  const int g = (int)rem - (up ? 0x20000000 : 0);
  const uint32_t sgn = hi & 0x80000000u;
  const float f = __uint_as_float(u | sgn);
  h = __float2half_rn(f);
  // 2^(e - 52) with the sign of x
  const float unit = __uint_as_float(((uint32_t)(e - 52 + 127) << 23) | sgn);
  const float d = f - __half2float(h);
  const int gs = d == 0.f ? g : ((g & ~15) | ((g & 15) ? 16 : 0));
  l = __float2half_rn(fmaf((float)gs, unit, d));
}

}  // namespace tc

// ------------------------------ host side ----------------------------------

// Encodes a 3-D FP16 tensor map [d2][d1][d0] (d0 innermost, contiguous) with a
// box of {64, 128, 1} and 128-byte swizzle.  Out-of-range reads return zero.
bool make_tmap_f16_3d(CUtensorMap *map, const void *base, uint64_t d0, uint64_t d1, uint64_t d2,
                      uint32_t box0, uint32_t box1, std::string *err);

}  // namespace sox
