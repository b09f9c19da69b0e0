// FP64 matrix products on the FP16 tensor cores (f64_slices.cu).
//
// Each row of an operand (its K elements) is scaled by a power of two and written as seven
// 8-bit signed digits, x = 2^e sum_i d_i 2^-(8 i + 7), |d_i| <= 128, each digit an FP16
// integer: fixed point to 2^-55 of the row's largest element.  Digit products d_i d_j are exact in the
// tensor core, and so are their FP32 sums over 128 elements (at most 7 * 128 * 2^14 < 2^24).  Products
// with equal i + j share one accumulator; i + j <= 7 are kept (34 of 49).  The eight sums are added as
// 64-bit integers and rounded to FP64 once.  An element's error is below (1.1 K + 9) 2^-54 of the product
// of the two rows' largest elements: for rows of similar elements less than a chain of FP64 FMAs makes.
// Elements whose terms may all be far smaller than that product (their magnitudes' sum S below 2^-6 of
// it) are summed in FP64 from the sources, so the error is also below (1.1 K + 9) 2^-48 S.
// This is the Ozaki splitting (error-free transformation of a matrix product into exact
// lower-precision ones; Ozaki, Ogita, Oishi and Rump, 2012), with the digits on the K-major
// operand layout of tcgen05.
#pragma once
#include <cuda_fp16.h>

#include "internal.h"

namespace sox {

constexpr int kSlices = 7;

// A sliced operand: `batch` blocks of `rows` rows of K elements, digit s of (b, r, k) at
// p[((s * batch + b) * rows + r) * K8 + k]; ex[b * rows + r] the row's exponent
// (f64_slices.cu, row_code), mask and mag the elements' sizes within it.  src stays readable,
// and unchanged, until the products that use the operand are done: they sum some elements from it.
struct SliceOp {
  __half *p = nullptr;
  int *ex = nullptr;
  uint32_t *mask = nullptr;
  uint8_t *mag = nullptr;
  int batch = 0, rows = 0, K = 0, K8 = 0;
  const void *src = nullptr;
  bool f32 = false;
  long long sb = 0, sr = 0, sk = 0;
  // complex operands (strides in complex elements): kind 1 is the A side, a complex row as one
  // row of 2 K interleaved reals; kind 2 the B side, a complex row as the two rows
  // (b_r, -sa sc b_i) and (sc b_i, sa b_r), sa, sc = -1 for the conjugate of A, of B
  int kind = 0, sa = 1, sc = 1;
};
size_t slice_bytes(long long batch, int rows, int K);
SliceOp slice_take(Arena &ar, int batch, int rows, int K);
// Powers of two along the inner index: operand A of a product times 2^e_k, B times 2^-e_k, with e_k =
// (kex[b * stride + k] - 1023) / part from exponent fields (0: none); part > 0 for A, the negative for
// B.  The product is the same; a K index that is large in one operand and small in the other keeps its
// digits in both.  kex holds B's largest exponents: part 1 where A's elements fall as B's rise (rows of a
// factored system), 2 where they do not depend on them (the range is then shared).
struct SliceBalance {
  const int *kex = nullptr;
  int stride = 0, part = 1;
};
// what goes into kex: the exponent field of a finite value, 0 for zeros, infinities and NaNs (the
// greatest one along index k of B, by atomicMax on zeroed memory)
__device__ __forceinline__ int balance_exponent(double a) {
  const int hi = __double2hiint(a), e = (hi >> 20) & 0x7ff;
  if (e == 0x7ff || (((hi & 0x7fffffff) | __double2loint(a)) == 0)) return 0;
  return max(e, 1);
}
// digits of element (b, r, k) = src[b * sb + r * sr + k * sk], FP64 or FP32; `batch` blocks
// (at most op's)
void slice_rows(const void *src, bool f32, long long sb, long long sr, long long sk, int batch, SliceOp &op,
                cudaStream_t s, SliceBalance bal = {});

// The same for complex rows (FP64, interleaved): op taken with rows (A) or 2 rows (B) and 2 K
// (bal: over the K complex indices)
void slice_complex_a(const double *src, long long sb, long long sr, long long sk, int batch, SliceOp &op, cudaStream_t s,
                     SliceBalance bal = {});
void slice_complex_b(const double *src, long long sb, long long sr, long long sk, int batch, bool conjA, bool conjB,
                     SliceOp &op, cudaStream_t s, SliceBalance bal = {});

// C[b](i, j) = alpha sum_k A(b, i, k) B(b, j, k) + beta C[b](i, j); an operand of batch 1 is
// shared.  Element (i, j) at C + b * sC + i * ci + j * cj.
struct SliceGemm {
  double *C = nullptr;
  long long sC = 0, ci = 0, cj = 0;
  double alpha = 1.0, beta = 0.0;
  int batch = 1;
  const int *skip = nullptr;     // batch b is left out when skip[b] != 0
  const int *mirror = nullptr;   // mirror[b] != 0: square C, only the 32 x 32 blocks with i / 32 <= j / 32
                                 // are computed and the others are their mirror images
};
// K <= kSliceMaxK per call
constexpr int kSliceMaxK = 1024;
Status slice_gemm(sox_handle h, const SliceOp &A, const SliceOp &B, const SliceGemm &g, cudaStream_t s);

// D[b][P][R] = sum_{v0 <= v < v1} (sum_q A[b][v][P][q] GR[b][R][q]) (sum_w GW[b][P][w] U2[R][v][w]) (v1 <= 0: all n):
// A sliced as batch (b, v), rows P; GR and GW as batch b; U2 as batch v, rows R, with src
// strides of the contiguous arrays named here.  n <= kSliceMaxK.
Status slice_bcd(sox_handle h, const SliceOp &A, const SliceOp &GR, const SliceOp &GW, const SliceOp &U2, int n, int N,
                 int batch, int v0, int v1, double *D, long long sD, cudaStream_t s);

// Whether a product of these sizes is faster through slices than on the FP64 pipe of the handle's device.
bool slices_pay(const sox_context *h, long long M, long long N, long long K, long long batch);

// Any GemmF64 through slices (operands sliced into `scratch`, K in blocks of kSliceMaxK), or
// on the FP64 pipe where slices_pay says so, in passes over batches and columns whose digits stay below
// slice_pass_bytes per operand (one batch and 1024 columns at least).  gemm_f64_bytes: the scratch it
// needs (0 without).
inline size_t slice_pass_bytes(const sox_context *h) {   // the handle's limit, 1 GiB at most
  const size_t most = size_t(1) << 30, b = chunk_budget(h, most);
  return b < most ? b : most;
}
size_t gemm_f64_bytes(sox_handle h, const GemmF64 &g);
Status gemm_f64(sox_handle h, const GemmF64 &g, Arena scratch, cudaStream_t s);

}  // namespace sox
