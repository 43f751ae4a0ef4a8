// backward.cu -- eigen-adjoint of the symmetric eigensolver (not in the paper;
// the standard first-order perturbation result, e.g. Giles 2008, "Collected
// matrix derivative results"):
//   M = Q^T dQ,  G_ii = dW_i,  G_ij = M_ij / (w_j - w_i) (i != j),
//   dA = sym(Q G Q^T) = Q sym(G) Q^T,  sym(X) = (X + X^T)/2.
// Symmetrizing G first makes the last product symmetric in exact arithmetic,
// so dA is written exactly symmetric (its lower triangle mirrored).  The three
// products run as FP64-accurate products on the tensor cores (exact bf16
// slices, ozaki.cu), each step one launch over a group of matrices: one n = 512
// product has 32 output tiles for 152 SMs, and 18 launches per matrix over side
// streams were bound by the host (64 matrices: 6.4 ms, 5.3 ms with the faster
// products; grouped 4.9 ms, 3.4 ms with kept scratch and whole-line slicing).  With MPJ_GEMM_TC=0 they run on the FP64 DMMA
// kernel, batched over blockIdx.z (the last one as a lower-tile product).
#include "common.cuh"
#include "gemm64.cuh"
#include "ozaki.cuh"

namespace {

constexpr int TB = 32;  // tile side of the transposing kernels

// Gs = sym(G) from M (may be null: M = 0), w, dW (may be null: dW = 0): off the
// diagonal (M_ij - M_ji) / (2 (w_j - w_i)), one division per entry pair.  A
// block forms tile (ti, tj), ti >= tj, and its mirror through shared memory, so
// both triangles are read and written along columns.
__global__ void __launch_bounds__(256) adjoint_core(const double* __restrict__ M, const double* __restrict__ W,
                                                    const double* __restrict__ dW, int n, double* __restrict__ Gs,
                                                    unsigned* __restrict__ flags) {
  const int ti = blockIdx.x, tj = blockIdx.y;
  if (ti < tj) return;
  __shared__ double lo[TB][TB + 1], up[TB][TB + 1];  // [column][row] of tiles (ti, tj) and (tj, ti)
  const size_t b = blockIdx.z;
  const double* w = W + b * n;
  const double* Mb = M ? M + b * n * n : nullptr;
  double* G = Gs + b * n * n;
  const int lane = threadIdx.x & 31, i0 = ti * TB, j0 = tj * TB;
  for (int c = threadIdx.x >> 5; c < TB; c += 8) {
    lo[c][lane] = (Mb && i0 + lane < n && j0 + c < n) ? Mb[(size_t)(j0 + c) * n + i0 + lane] : 0.0;
    up[c][lane] = (Mb && j0 + lane < n && i0 + c < n) ? Mb[(size_t)(i0 + c) * n + j0 + lane] : 0.0;
  }
  __syncthreads();
  for (int c = threadIdx.x >> 5; c < TB; c += 8) {
    const int i = i0 + lane, j = j0 + c;
    double g = 0.0;
    if (i < n && j < n) {
      if (i == j) {
        g = dW ? dW[b * n + i] : 0.0;
      } else {
        const double mij = lo[c][lane], mji = up[lane][c], gap = w[j] - w[i];
        if (gap == 0.0) {
          if (mij != 0.0 || mji != 0.0) atomicOr(flags, MPJ_FLAG_DEGENERATE);
        } else {
          g = 0.5 * ((mij - mji) / gap);  // F_ij M_ij and F_ji M_ji, F_ij = 1 / (w_j - w_i)
        }
      }
      G[(size_t)j * n + i] = g;
    }
    lo[c][lane] = g;  // read above by this thread only
  }
  if (ti == tj) return;  // a diagonal tile is written in full above
  __syncthreads();
  for (int c = threadIdx.x >> 5; c < TB; c += 8)
    if (i0 + c < n && j0 + lane < n) G[(size_t)(i0 + c) * n + j0 + lane] = lo[lane][c];
}

// B(j, i) = B(i, j) for i > j (the lower triangle mirrored), by tiles, batched
// over blockIdx.z
__global__ void __launch_bounds__(256) bwd_mirror(double* __restrict__ B, int ldb, long long sb, int n) {
  const int ti = blockIdx.x, tj = blockIdx.y;
  if (ti < tj) return;
  __shared__ double t[TB][TB + 1];
  double* Bb = B + (size_t)blockIdx.z * sb;
  const int lane = threadIdx.x & 31, i0 = ti * TB, j0 = tj * TB;
  for (int c = threadIdx.x >> 5; c < TB; c += 8)
    if (i0 + lane < n && j0 + c < n) t[c][lane] = Bb[(size_t)(j0 + c) * ldb + i0 + lane];
  __syncthreads();
  for (int c = threadIdx.x >> 5; c < TB; c += 8)
    if (i0 + c < n && j0 + lane < n && i0 + c > j0 + lane) Bb[(size_t)(i0 + c) * ldb + j0 + lane] = t[lane][c];
}

}  // namespace

extern "C" int mpj_syev_backward(int batch, int n, const double* W, const double* Q, int ldq, const double* dW,
                                 const double* dQ, int lddq, double* dA, int ldda, void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
  if (batch < 0 || n < 0 || ldq < n || lddq < n || ldda < n || ldq < 1 || lddq < 1 || ldda < 1) return MPJ_EINVAL;
  if (batch == 0 || n == 0) return MPJ_OK;
  if (!W || !Q || !dA) return MPJ_EINVAL;
  size_t sq = (size_t)n * n;
  const bool tc = mpj_gemm_tc_enabled();
  // tensor-core products: groups of equal size whose two sliced operands take
  // at most half a GB (or one matrix)
  const size_t ob = tc ? mpj_oz_operand_bytes(n, n) : 0;
  int group = batch;
  if (tc) {
    const size_t fit = ((size_t)512 << 20) / (2 * ob);
    const int most = fit < 1 ? 1 : fit > 32768 ? 32768 : (int)fit;
    const int groups = (batch + most - 1) / most;
    group = (batch + groups - 1) / groups;
  }
  void* w = nullptr;
  size_t bytes = ((2 * (size_t)batch * sq * sizeof(double) + 255) & ~(size_t)255) + 512 + 2 * ob * (size_t)(tc ? group : 0);
  if (mpj_alloc_async(&w, bytes, s) != cudaSuccess) return MPJ_ENOMEM;
  mpj_count_alloc();
  double* M = (double*)w;
  double* T = M + (size_t)batch * sq;
  char* o0 = (char*)(T + (size_t)batch * sq);  // sliced operands (256-byte aligned when batch * sq is a multiple of 16)
  o0 = (char*)(((size_t)o0 + 255) & ~(size_t)255);
  char* o1 = o0 + ob * (size_t)group;
  unsigned* flags = (unsigned*)((char*)w + bytes - 256);
  int st = MPJ_OK;
  unsigned hflags = 0;
  cudaError_t e = cudaMemsetAsync(flags, 0, sizeof(unsigned), s);
  long long sQ = (long long)ldq * n, sdQ = (long long)lddq * n, sA = (long long)ldda * n, sN = (long long)sq;
  const int nt = (n + TB - 1) / TB;
  auto core = [&](int b0, int nb) -> cudaError_t {  // T = sym(G)
    for (int b = b0; b < b0 + nb; b += 32768) {
      const int k = b0 + nb - b < 32768 ? b0 + nb - b : 32768;
      adjoint_core<<<dim3(nt, nt, k), 256, 0, s>>>(dQ ? M + b * sN : nullptr, W + (size_t)b * n,
                                                   dW ? dW + (size_t)b * n : nullptr, n, T + b * sN, flags);
      mpj_count_launch();
    }
    return cudaGetLastError();
  };
  if (tc) {
    for (int b0 = 0; b0 < batch && e == cudaSuccess; b0 += group) {
      const int nb = batch - b0 < group ? batch - b0 : group;
      const double* Qb = Q + b0 * sQ;
      double *Mb = M + b0 * sN, *Tb = T + b0 * sN, *Ab = dA + b0 * sA;
      OzOperand p, q;
      if (dQ) {  // M = Q^T dQ: columns of Q and of dQ over the row index
        e = mpj_oz_prepare(Qb, ldq, 1, n, n, o0, &p, s, nb, sQ);
        if (e == cudaSuccess) e = mpj_oz_prepare(dQ + b0 * sdQ, lddq, 1, n, n, o1, &q, s, nb, sdQ);
        if (e == cudaSuccess) e = mpj_oz_gemm(p, q, n, n, 1.0, 0.0, nullptr, n, Mb, n, flags, s, false, nb, sN);
      }
      if (e == cudaSuccess) e = core(b0, nb);
      // M = Q T, then dA = M Q^T (rows of Q left of T, right of M; the lower triangle, mirrored)
      if (e == cudaSuccess) e = mpj_oz_prepare(Qb, 1, ldq, n, n, o0, &p, s, nb, sQ);
      if (e == cudaSuccess) e = mpj_oz_prepare(Tb, n, 1, n, n, o1, &q, s, nb, sN);
      if (e == cudaSuccess) e = mpj_oz_gemm(p, q, n, n, 1.0, 0.0, nullptr, n, Mb, n, flags, s, false, nb, sN);
      if (e == cudaSuccess) e = mpj_oz_prepare(Mb, 1, n, n, n, o1, &q, s, nb, sN);
      if (e == cudaSuccess) e = mpj_oz_gemm(q, p, n, n, 1.0, 0.0, nullptr, n, Ab, ldda, flags, s, true, nb, sA);
      if (e == cudaSuccess) {
        bwd_mirror<<<dim3(nt, nt, nb), 256, 0, s>>>(Ab, ldda, sA, n);
        mpj_count_launch();
        e = cudaGetLastError();
      }
    }
  } else {
    if (e == cudaSuccess && dQ) {
      GemmArgs g{n, n, n, 1.0, 0.0, Q, ldq, sQ, dQ, lddq, sdQ, nullptr, n, 0, M, n, sN, 0};
      e = mpj_gemm64_launch(g, true, false, batch, s);
    }
    if (e == cudaSuccess) e = core(0, batch);
    if (e == cudaSuccess) {
      GemmArgs g{n, n, n, 1.0, 0.0, Q, ldq, sQ, T, n, sN, nullptr, n, 0, M, n, sN, 0};
      e = mpj_gemm64_launch(g, false, false, batch, s);
    }
    if (e == cudaSuccess) {
      GemmArgs g2{n, n, n, 1.0, 0.0, M, n, sN, Q, ldq, sQ, nullptr, n, 0, dA, ldda, sA, 1};
      e = mpj_gemm64_launch(g2, false, true, batch, s);
    }
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(&hflags, flags, sizeof(unsigned), cudaMemcpyDeviceToHost, s);
  if (e != cudaSuccess) {
    mpj_set_cuda_error(e, "mpj_syev_backward", __LINE__);
    st = MPJ_ECUDA;
  }
  cudaFreeAsync(w, s);
  e = cudaStreamSynchronize(s);
  if (e != cudaSuccess && st >= 0) {
    mpj_set_cuda_error(e, "mpj_syev_backward sync", __LINE__);
    st = MPJ_ECUDA;
  }
  if (st == MPJ_OK && (hflags & MPJ_FLAG_DEGENERATE)) st = MPJ_EDEGENERATE;
  if (st == MPJ_OK && (hflags & MPJ_FLAG_TIMEOUT)) st = MPJ_ETIMEOUT;
  return st;
}
