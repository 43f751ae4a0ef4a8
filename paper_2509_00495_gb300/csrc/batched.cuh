// batched.cuh -- the two forms of the batched solve: round by round
// (batched_rounds.cu), and one thread group per matrix (batched.cu).
#pragma once
#include <stddef.h>
#include <cuda_runtime.h>

// mpj_syev_batched (see mpjacobi.h) with validated arguments; picks the form.
int mpj_batched_rounds(int batch, const int* n_host, const double* const* A_dev, double* const* W_dev,
                       double* const* Q_dev, double tol, int* sweeps_host, cudaStream_t s);
// Frees its cached workspaces.
void mpj_batched_rounds_release();

// One thread group of G (256, 512 or 1024) threads per matrix, `grid` CTAs of 1024
// threads that pull matrices from a queue.  order, n: matrix and size by place in
// it (sizes at most nmax); counter and flags zeroed by the caller;
// MPJ_FLAG_TIMEOUT in *flags means that a sweep cap was reached; `work` of
// mpj_batched_groups_bytes.
size_t mpj_batched_groups_bytes(int G, int grid, int nmax);
cudaError_t mpj_batched_groups(int G, int grid, int nmax, const int* order, const int* n, const double* const* A,
                               double* const* W, double* const* Q, int batch, double tol, void* work, int* counter,
                               int* sweeps, unsigned* flags, cudaStream_t s);
