// batched.cuh -- the round-by-round batched solve (batched_rounds.cu).
#pragma once
#include <cuda_runtime.h>

// mpj_syev_batched (see mpjacobi.h) with validated arguments.
int mpj_batched_rounds(int batch, const int* n_host, const double* const* A_dev, double* const* W_dev,
                       double* const* Q_dev, double tol, int* sweeps_host, cudaStream_t s);
// Frees its cached workspaces.
void mpj_batched_rounds_release();
