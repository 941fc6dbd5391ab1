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
#define NK_LONG_RUN 128
cudaError_t nk_cg_resident(const float* K, int64_t ldk, int64_t N, int R, const double* B, const double* minv,
                           double* X, double lam, double tol, double tol_long, int maxit, double* iters, void* ws,
                           int sm, long long polls, cudaStream_t st);

// Whether a launch was refused before anything ran because its CTAs cannot all
// be resident: a process or a stream limited to part of the SMs.
inline bool nk_launch_refused(cudaError_t e) {
  return e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorLaunchOutOfResources || e == cudaErrorNotSupported;
}

// A CG run on the resident form while *resident holds, else on the other one;
// a refused launch clears *resident and the other form takes over, with the
// tolerance of its refinement sweeps, tol_replay.
template <class Resident, class Replay>
inline cudaError_t nk_cg_either(bool* resident, double tol, double tol_replay, Resident run_resident, Replay replay) {
  if (*resident) {
    const cudaError_t e = run_resident(tol);
    if (!nk_launch_refused(e)) return e;
    *resident = false;
    tol = tol_replay;
  }
  return replay(tol);
}
