// batch.cuh -- how the kernels of the single-matrix stages address a batch of
// matrices with n <= 256 that go through their rounds together (batched_rounds.cu).
//
// The matrices are ordered by decreasing padded size N (n rounded up to a
// multiple of 32, so there are eight classes); every buffer holds them one
// after the other in that order with leading dimension N.  A launch covers
// the tasks of all matrices of the classes lo .. 7; a block finds its matrix
// by walking the classes, largest first.
#pragma once
#include <cuda_bf16.h>

#include "common.cuh"

constexpr int BATCH_CLASSES = 8;
constexpr int BATCH_NMAX = 32 * BATCH_CLASSES;

struct BatchShape {
  int cnt[BATCH_CLASSES];         // matrices of class c (N = 32 (c + 1))
  int first[BATCH_CLASSES];       // place of the first one
  long long el[BATCH_CLASSES];    // elements (sum of N^2) before it
  int pairs[BATCH_CLASSES];       // block pairs (sum of N / 32) before it
  long long oz[BATCH_CLASSES];    // sliced-operand elements (8 Rp N each) before it
  const int* n;                   // true size by place
  const int* active;              // by place: 0 when the matrix takes no part (null: all do)
};

struct BatchTask {
  int place, n, N, local, pair0;
  long long el, oz;
};

// Rows of a sliced operand of class N: whole 128-row tiles.
__host__ __device__ inline int batch_rp(int N) { return (N + 127) / 128 * 128; }

// The matrix and the task within it of block `bid`, when matrix class c has
// tiles(c + 1) tasks; false when there is none or its matrix is not active.
template <class F>
MPJ_DEV bool batch_find(const BatchShape& b, int lo, int bid, F tiles, BatchTask& t) {
#pragma unroll
  for (int c = BATCH_CLASSES - 1; c >= 0; --c) {
    if (c < lo) break;
    const int per = tiles(c + 1), tot = b.cnt[c] * per;
    if (bid < tot) {
      const int j = bid / per, N = 32 * (c + 1);
      t.local = bid - j * per;
      t.place = b.first[c] + j;
      t.N = N;
      t.el = b.el[c] + (long long)j * N * N;
      t.oz = b.oz[c] + (long long)j * 8 * batch_rp(N) * N;
      t.pair0 = b.pairs[c] + j * (c + 1);
      t.n = b.n[t.place];
      return !b.active || b.active[t.place] != 0;
    }
    bid -= tot;
  }
  return false;
}

// Blocks of a launch over classes lo .. 7 with tiles(c + 1) tasks each.
template <class F>
inline long long batch_blocks(const BatchShape& b, int lo, F tiles) {
  long long t = 0;
  for (int c = lo; c < BATCH_CLASSES; ++c) t += (long long)b.cnt[c] * tiles(c + 1);
  return t;
}

// The smallest class that still has a round R (class c has rounds 0 .. 2 c).
inline int batch_lowest_class(int R) { return (R + 1) / 2; }

// Round R of the FP32 stage (stage1.cu): subproblems, then V <- V U~ and
// A <- U~^T A U~ in one launch.  A32, V32: by elements; S, U: 1024 floats per
// block pair.
cudaError_t mpj_batch_stage1_round(const BatchShape& b, int R, float* A32, float* V32, float* S, float* U,
                                   cudaStream_t s);

// Round R of the FP64 sweeps (blocked64.cu): subproblems, then V <- V U~ and
// B = A U~ in one launch, then A = B^T U~.  skip_abs by place; sl, ex, rot as
// in the single-matrix sweeps, per block pair.
size_t mpj_batch_digit_bytes(int pairs);
cudaError_t mpj_batch_sweep64_round(const BatchShape& b, int R, double* A, double* V, double* B, const double* skip_abs,
                                    void* digits, int pairs, unsigned* flags, cudaStream_t s);

// Products of the batch on the exact-slice engine (ozaki.cu).  An operand is
// sliced from `X` (by elements, ld N) or from the user's matrices `ptr` (by
// order, ld n); byrow: its rows are rows of X, else columns.
struct BatchOperand {
  __nv_bfloat16* sl;
  int* ex;  // 256 exponents per place
};
cudaError_t mpj_batch_oz_prepare(const BatchShape& b, const double* X, const double* const* ptr, const int* order,
                                 bool byrow, const BatchOperand& op, cudaStream_t s);
// C = alpha op(A) op(B) + beta Cin + dg I (ld N); sym: only the lower triangle
// is formed and mirrored.
cudaError_t mpj_batch_oz_gemm(const BatchShape& b, const BatchOperand& oa, const BatchOperand& ob, double alpha,
                              double beta, const double* Cin, double dg, double* C, bool sym, unsigned* flags,
                              cudaStream_t s);
