// CG run with K, or the rows that fit, resident in shared memory
// (pcg_resident.cu).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

// Workspace of a run; 0 for an N and R that it does not take.
size_t nk_cg_resident_bytes(int64_t N, int R, int sm);
// CG on (K + lam I) X = B from X = 0 until every column's recursive residual
// is at most tol ||B|| (tol_long ||B|| in iterations past NK_LONG_RUN) or maxit
// iterations; iters[R] (device) receives the columns' counts, the second
// unsigned of ws is nonzero if a barrier's wait ran out of `polls`.
#define NK_LONG_RUN 256
cudaError_t nk_cg_resident(const float* K, int64_t ldk, int64_t N, int R, const double* B, const double* minv,
                           double* X, double lam, double tol, double tol_long, int maxit, double* iters, void* ws,
                           int sm, long long polls, cudaStream_t st);
