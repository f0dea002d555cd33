// cf_solve64.cuh -- S-1 with FP64 factors (cf_solve64.cu).
#pragma once

#include "cf_common.cuh"

namespace cf {

// X <- M^{-1} X, n x nrhs FP64, in place.  mode 0: M unit lower (strictly
// lower part of T), 1: upper, 2: lower, 3: transposed lower.
int launch_tri_solve64(int mode, int n, int nrhs, const double *T, int ldt, double *X, int ldx, cudaStream_t st);
// perm (device int[n]) = the row order of ipiv's interchanges, T (n x nrhs,
// ld n) = the rows of B in that order.  T's first 6 n bytes serve as scratch
// before.
int launch_permute_rhs(int n, int nrhs, const int *ipiv, int *perm, const double *B, int ldb, double *T, cudaStream_t st);
int solve64_take_status(cudaStream_t st, int *status);

}  // namespace cf
