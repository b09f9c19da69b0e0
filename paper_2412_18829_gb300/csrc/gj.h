// Batched solve of K W = B by block Gauss-Jordan with partial pivoting, FP64 (gj.cu).
#pragma once
#include "internal.h"

namespace sox {

// Aug [batch][N][2N] = [K | B], real or complex (interleaved) doubles; the right half becomes
// K^-1 B.  info[1] is set when some K is singular (the results are then not valid).
// gj_pays: whether the blocked form is the faster one; scratch: gj_bytes, of this or of any larger
// batch.
bool gj_pays(int N);
size_t gj_bytes(int N, int batch, bool cplx);
Status gj_solve(sox_handle h, double *Aug, int N, int batch, bool cplx, int *info, Arena scratch, cudaStream_t s);

}  // namespace sox
