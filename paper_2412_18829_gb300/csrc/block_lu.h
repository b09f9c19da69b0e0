// Batched solve of K W = B by block LU with partial pivoting, FP64 (block_lu.cu).
#pragma once
#include "internal.h"

namespace sox {

// Aug [batch][N][2N] = [K | B], real or complex (interleaved) doubles; the right half becomes
// K^-1 B, the left half is used up.  info[1] is set when some K is singular (the results are then not valid).
// lu_pays: whether the blocked form is the faster one; scratch: lu_bytes, of this or of any larger
// batch.
bool lu_pays(int N);
size_t lu_bytes(sox_handle h, int N, int batch, bool cplx);
Status lu_solve(sox_handle h, double *Aug, int N, int batch, bool cplx, int *info, Arena scratch, cudaStream_t s);

}  // namespace sox
