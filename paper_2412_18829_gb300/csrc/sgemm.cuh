// FP32 CUDA-core GEMM tile shared by the mixed-tensor and back-projection kernels.
//
// Every output element is one chain acc = fma(a_k, b_k, acc) over k = 0, 1, 2, ... in FP32,
// round to nearest: the tile shape and the pipelining change the speed only, never a bit of
// the result.  Bound: the FP32 pipe (128 FMA a clock and SM).  256 threads hold an 8 x 8
// (or 4 x 8) block each; the FMAs go out in packed pairs (fma.rn.f32x2, two columns per
// instruction), which leaves issue slots for the shared-memory loads.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace sox {
namespace sg {

constexpr int kBN = 128, kBK = 16, kThreads = 256;

__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ void unpack2(uint64_t v, float &lo, float &hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

// 16-byte asynchronous copy; bytes = 0 fills with zeros (src is then not read)
__device__ __forceinline__ void cp16(void *dst, const void *src, int bytes) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Columns of a thread: tx * 4 + (0..3) and 64 + tx * 4 + (0..3); rows ty * 4 + (0..3) and,
// for BM = 128, 64 + ty * 4 + (0..3).  acc[i][j]: row i, column pair j.
template <int BM>
struct Acc {
  static constexpr int R = BM / 16;
  uint64_t v[R][4];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) v[i][j] = 0ull;   // (+0, +0)
  }
  // one staged K block: sa[kBK][lda] (k-major rows), sb[kBK][kBN]
  __device__ __forceinline__ void step(const float *sa, int lda, const float *sb, int tx, int ty) {
#pragma unroll
    for (int k = 0; k < kBK; ++k) {
      float a[R];
      const float4 a0 = *reinterpret_cast<const float4 *>(sa + k * lda + ty * 4);
      a[0] = a0.x; a[1] = a0.y; a[2] = a0.z; a[3] = a0.w;
      if (R == 8) {
        const float4 a1 = *reinterpret_cast<const float4 *>(sa + k * lda + 64 + ty * 4);
        a[R - 4] = a1.x; a[R - 3] = a1.y; a[R - 2] = a1.z; a[R - 1] = a1.w;
      }
      uint64_t b[4];
      const ulonglong2 b0 = *reinterpret_cast<const ulonglong2 *>(sb + k * kBN + tx * 4);
      const ulonglong2 b1 = *reinterpret_cast<const ulonglong2 *>(sb + k * kBN + 64 + tx * 4);
      b[0] = b0.x; b[1] = b0.y; b[2] = b1.x; b[3] = b1.y;
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const uint64_t aa = pack2(a[i], a[i]);
#pragma unroll
        for (int j = 0; j < 4; ++j) v[i][j] = fma2(aa, b[j], v[i][j]);
      }
    }
  }
  __device__ static __forceinline__ int row(int i, int ty) { return (i < 4 ? 0 : 64) + ty * 4 + (i & 3); }
};

}  // namespace sg
}  // namespace sox
