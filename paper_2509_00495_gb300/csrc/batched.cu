// batched.cu -- many independent symmetric eigenproblems (sizes 1..256): the C
// entry point, and the solve with one thread group per matrix in one persistent
// launch, taken for batches of small matrices (the others go round by round, see
// batched_rounds.cu) and for all when MPJ_BATCHED_GROUP is set.  Not in the paper:
// each matrix runs the mixed method of Algorithm 9 (Sec. 5.1) on its own.
//
// A CTA of 1024 threads holds 1024/G groups of G threads (G = 256, 512 or
// 1024, picked by the autotuner below); each group pulls matrix indices from
// an atomic work queue ordered by decreasing n (longest job first) and, for
// its matrix,
//   1. FP32 round-robin Jacobi on fl32(A) from V32 = I until
//      off(A32) <= n 2^-24 ||A||_F (cap max32), Q_l = double(V32);
//   2. Newton-Schulz X <- 1.5 X - 0.5 X (X^T X), ns_steps times (FP64 DMMA);
//   3. A_cond = X^T (A X) (FP64 DMMA, lower tiles mirrored);
//   4. FP64 round-robin Jacobi on A_cond until off <= tol (cap max64), also
//      skipping pairs with |a_pq| <= tol/n (threshold Jacobi), its rotations
//      applied to the columns of X = Q_d directly (Q = Q_d V by associativity);
//   5. W = sorted diag, Q = the rotated X with its columns permuted.
// Groups synchronize with named barriers (bar.sync id, G), so small matrices
// share an SM.  The round-robin ordering, the rotation records and the
// 2x2-block update are those of common.cuh; one round is one barrier-separated
// phase of the group.  The group's matrices live in a per-group slice of
// global workspace, except the stage-1 matrices: A32 lives in shared memory
// for n <= about 233 / 160 / 106 (G = 1024 / 512 / 256), V32 too for
// n <= about 165 / 113 / 75.  FP64 work sets the floor: GB300 issues about
// 2 FP64 FMA per clock per SM, so the batch costs at least its total FP64
// work over 152 SMs; barrier-separated rounds add latency on top.
//
// Planning and replay (with MPJ_BATCHED_GROUP): the first call for a given batch (sizes, pointer
// arrays, tolerance) allocates the workspace, sorts the queue, picks G (timed
// on the batch itself unless a cached choice exists for its size histogram)
// and captures [queue reset, kernel, result copies] in a CUDA graph; later
// identical calls only launch that graph.
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <mutex>
#include <string>
#include <vector>

#include "batched.cuh"
#include "common.cuh"

namespace {

constexpr int NTH = 1024;
constexpr int NMAX = 256;
constexpr int MAXG = 4;  // groups per CTA at the smallest group size

struct Grp {
  int t;    // thread index in the group
  int n;    // threads in the group
  int bar;  // named barrier id (1 + group index)
  int id;   // group index in the CTA
};

MPJ_DEV void gsync(const Grp& g) { asm volatile("bar.sync %0, %1;\n" ::"r"(g.bar), "r"(g.n) : "memory"); }

struct Bufs {
  float* A32;
  float* V32;
  double* X;
  double* M;
  double* Y;
};

MPJ_DEV double group_sum(const Grp& g, double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  gsync(g);
  if ((g.t & 31) == 0) red[g.t >> 5] = v;
  gsync(g);
  double t = 0.0;
  if (g.t < 32) {
    t = g.t < (g.n >> 5) ? red[g.t] : 0.0;
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (g.t == 0) red[32] = t;
  }
  gsync(g);
  return red[32];
}

MPJ_DEV void dmma(double& c0, double& c1, double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};\n"
               : "+d"(c0), "+d"(c1)
               : "d"(a), "d"(b));
}

// Group-level D = alpha op(A) op(B) + beta Cin (n x n, column-major, ld n),
// warp tasks of 16 x 16 outputs on m8n8k4 DMMA.
template <bool TA, bool TB>
MPJ_DEV void grp_gemm(const Grp& g, int n, double alpha, const double* A, const double* B, double beta,
                      const double* Cin, double* C, bool sym) {
  const int lane = g.t & 31, warp = g.t >> 5, nw = g.n >> 5;
  const int gid = lane >> 2, tig = lane & 3;
  const int nt = (n + 15) / 16;
  for (int t = warp; t < nt * nt; t += nw) {
    int ti = t % nt, tj = t / nt;
    if (sym && ti < tj) continue;
    int m0 = ti * 16, n0 = tj * 16;
    double acc[2][2][2] = {{{0, 0}, {0, 0}}, {{0, 0}, {0, 0}}};
#pragma unroll 8
    for (int k = 0; k < n; k += 4) {
      int kk = k + tig;
      double af[2], bf[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        int r = m0 + i * 8 + gid;
        af[i] = (r < n && kk < n) ? (TA ? A[(size_t)r * n + kk] : A[(size_t)kk * n + r]) : 0.0;
      }
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        int c = n0 + j * 8 + gid;
        bf[j] = (c < n && kk < n) ? (TB ? B[(size_t)kk * n + c] : B[(size_t)c * n + kk]) : 0.0;
      }
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) dmma(acc[i][j][0], acc[i][j][1], af[i], bf[j]);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          int r = m0 + i * 8 + gid, c = n0 + j * 8 + tig * 2 + e;
          if (r >= n || c >= n || (sym && r < c)) continue;
          double v = alpha * acc[i][j][e];
          if (beta != 0.0) v = fma(beta, Cin[(size_t)c * n + r], v);
          C[(size_t)c * n + r] = v;
          if (sym && r != c) C[(size_t)r * n + c] = v;
        }
  }
  gsync(g);
}

// One round-robin Jacobi sweep at group level on a symmetric n x n matrix A
// (ld n) with vectors V (ld n).  rec: m/2 records in shared memory.  Pairs
// with |a_pq| <= skip sqrt|a_pp a_qq| or |a_pq| <= skip_abs are skipped.
template <typename T>
MPJ_DEV void grp_rr_sweep(const Grp& g, int n, T* A, T* V, RotRec<T>* rec, T skip, T skip_abs) {
  const int m = n + (n & 1), h = m / 2;
  for (int r = 0; r < m - 1; ++r) {
    for (int i = g.t; i < h; i += g.n) {
      int x, y;
      rr_slot(m, r, i, x, y);
      T dx = x < n ? A[(size_t)x * n + x] : T(0);
      T dy = y < n ? A[(size_t)y * n + y] : T(0);
      T axy = (x < n && y < n) ? A[(size_t)y * n + x] : T(0);
      RotRec<T> rr;
      rr_make_rec<T>(m, n, r, x, y, dx, dy, axy, skip, rr, skip_abs);
      rec[i] = rr;
    }
    gsync(g);
#pragma unroll 4
    for (int e = g.t; e < h * h; e += g.n) {
      int a = e % h, b = e / h;
      if (a < b) continue;
      RotRec<T> ra = rec[a];
      bool rota = rec_rotated(ra.cm1, ra.sig);
      int xa, ya, xb, yb;
      rr_slot(m, r, a, xa, ya);
      if (a == b) {
        if (rota) {
          A[(size_t)xa * n + xa] = ra.dx;
          A[(size_t)ya * n + ya] = ra.dy;
          A[(size_t)ya * n + xa] = T(0);
          A[(size_t)xa * n + ya] = T(0);
        }
        continue;
      }
      RotRec<T> rb = rec[b];
      bool rotb = rec_rotated(rb.cm1, rb.sig);
      if (!rota && !rotb) continue;
      rr_slot(m, r, b, xb, yb);
      bool vxa = xa < n, vya = ya < n, vxb = xb < n, vyb = yb < n;
      T vxx = (vxa && vxb) ? A[(size_t)xb * n + xa] : T(0);
      T vxy = (vxa && vyb) ? A[(size_t)yb * n + xa] : T(0);
      T vyx = (vya && vxb) ? A[(size_t)xb * n + ya] : T(0);
      T vyy = (vya && vyb) ? A[(size_t)yb * n + ya] : T(0);
      if (rota) {
        rot_apply(ra.cm1, ra.sig, vxx, vyx);
        rot_apply(ra.cm1, ra.sig, vxy, vyy);
      }
      if (rotb) {
        rot_apply(rb.cm1, rb.sig, vxx, vxy);
        rot_apply(rb.cm1, rb.sig, vyx, vyy);
      }
      if (vxa && vxb) A[(size_t)xb * n + xa] = A[(size_t)xa * n + xb] = vxx;
      if (vxa && vyb) A[(size_t)yb * n + xa] = A[(size_t)xa * n + yb] = vxy;
      if (vya && vxb) A[(size_t)xb * n + ya] = A[(size_t)ya * n + xb] = vyx;
      if (vya && vyb) A[(size_t)yb * n + ya] = A[(size_t)ya * n + yb] = vyy;
    }
#pragma unroll 8
    for (int e = g.t; e < n * h; e += g.n) {
      int row = e % n, b = e / n;
      RotRec<T> rb = rec[b];
      if (!rec_rotated(rb.cm1, rb.sig)) continue;
      int xb, yb;
      rr_slot(m, r, b, xb, yb);
      T vx = V[(size_t)xb * n + row], vy = V[(size_t)yb * n + row];
      rot_apply(rb.cm1, rb.sig, vx, vy);
      V[(size_t)xb * n + row] = vx;
      V[(size_t)yb * n + row] = vy;
    }
    gsync(g);
  }
}

// Record of one slot for the scaled FP64 sweep: multipliers mx, my (zero:
// not rotated), c - 1 of the rotation, true diagonals after it.
struct SRec {
  double mx, my, cm1, dx, dy;
};

MPJ_DEV bool srec_rotated(const SRec& r) {
  return (__double_as_longlong(r.mx) | __double_as_longlong(r.my)) != 0;  // bit test, not an FP64 compare
}

// One round-robin sweep of the FP64 stage with scaled rotations (the scheme
// of the single-matrix sweeps): off the diagonal A = D Ã D and V = Ṽ D with
// one scale vector d (double-double, in shared memory), so a rotation costs
// one FMA per entry and side, Ã_x -= mx Ã_y, Ã_y += my Ã_x with
// mx = τ d_y / d_x, my = τ d_x / d_y, and d_x, d_y take the factor c; the true
// diagonal stays in A's diagonal entries.  The scales are folded back at the
// end of the sweep (at most n - 1 <= 255 factors c >= 2^-1/2 per index, so d
// stays far above the FP64 range limit).  Pairs with |a_pq| <= skip sqrt|a_pp
// a_qq| or |a_pq| <= skip_abs are skipped (a_pq the true coupling).
MPJ_DEV void grp_rr_sweep_fast(const Grp& g, int n, double* A, double* V, SRec* rec, double2* d, double skip,
                               double skip_abs) {
  const int m = n + (n & 1), h = m / 2;
  for (int i = g.t; i < n; i += g.n) d[i] = make_double2(1.0, 0.0);
  gsync(g);
  for (int r = 0; r < m - 1; ++r) {
    for (int i = g.t; i < h; i += g.n) {
      int x, y;
      rr_slot(m, r, i, x, y);
      const bool vx = x < n, vy = y < n;
      SRec rr;
      rr.mx = 0.0;
      rr.my = 0.0;
      rr.cm1 = 0.0;
      rr.dx = vx ? A[(size_t)x * n + x] : 0.0;
      rr.dy = vy ? A[(size_t)y * n + y] : 0.0;
      if (vx && vy) {
        const double sx = d[x].x, sy = d[y].x;
        const double axy = A[(size_t)y * n + x] * sx * sy;  // true coupling
        const bool xp = x < y;
        const double app = xp ? rr.dx : rr.dy, aqq = xp ? rr.dy : rr.dx;
        double t, cm1, s;
        if (jacobi_pair<double>(app, aqq, axy, skip, t, cm1, s, skip_abs)) {
          const double np = app - t * axy, nq = aqq + t * axy;
          const double tau = xp ? t : -t;
          rr.mx = tau * (sy / sx);
          rr.my = tau * (sx / sy);
          rr.cm1 = cm1;
          rr.dx = xp ? np : nq;
          rr.dy = xp ? nq : np;
        }
      }
      rec[i] = rr;
    }
    gsync(g);
#pragma unroll 4
    for (int e = g.t; e < h * h; e += g.n) {
      int a = e % h, b = e / h;
      if (a < b) continue;
      const SRec ra = rec[a];
      const bool rota = srec_rotated(ra);
      int xa, ya, xb, yb;
      rr_slot(m, r, a, xa, ya);
      if (a == b) {
        if (rota) {
          A[(size_t)xa * n + xa] = ra.dx;
          A[(size_t)ya * n + ya] = ra.dy;
          A[(size_t)ya * n + xa] = 0.0;
          A[(size_t)xa * n + ya] = 0.0;
        }
        continue;
      }
      const SRec rb = rec[b];
      const bool rotb = srec_rotated(rb);
      if (!rota && !rotb) continue;
      rr_slot(m, r, b, xb, yb);
      const bool vxa = xa < n, vya = ya < n, vxb = xb < n, vyb = yb < n;
      double vxx = (vxa && vxb) ? A[(size_t)xb * n + xa] : 0.0;
      double vxy = (vxa && vyb) ? A[(size_t)yb * n + xa] : 0.0;
      double vyx = (vya && vxb) ? A[(size_t)xb * n + ya] : 0.0;
      double vyy = (vya && vyb) ? A[(size_t)yb * n + ya] : 0.0;
      if (rota) {  // rows x_a, y_a
        double t0 = fma(-ra.mx, vyx, vxx), t1 = fma(ra.my, vxx, vyx);
        double t2 = fma(-ra.mx, vyy, vxy), t3 = fma(ra.my, vxy, vyy);
        vxx = t0;
        vyx = t1;
        vxy = t2;
        vyy = t3;
      }
      if (rotb) {  // columns x_b, y_b
        double t0 = fma(-rb.mx, vxy, vxx), t1 = fma(rb.my, vxx, vxy);
        double t2 = fma(-rb.mx, vyy, vyx), t3 = fma(rb.my, vyx, vyy);
        vxx = t0;
        vxy = t1;
        vyx = t2;
        vyy = t3;
      }
      if (vxa && vxb) A[(size_t)xb * n + xa] = A[(size_t)xa * n + xb] = vxx;
      if (vxa && vyb) A[(size_t)yb * n + xa] = A[(size_t)xa * n + yb] = vxy;
      if (vya && vxb) A[(size_t)xb * n + ya] = A[(size_t)ya * n + xb] = vyx;
      if (vya && vyb) A[(size_t)yb * n + ya] = A[(size_t)ya * n + yb] = vyy;
    }
#pragma unroll 4
    for (int e = g.t; e < n * h; e += g.n) {
      int row = e % n, b = e / n;
      const SRec rb = rec[b];
      if (!srec_rotated(rb)) continue;
      int xb, yb;
      rr_slot(m, r, b, xb, yb);
      double vx = V[(size_t)xb * n + row], vy = V[(size_t)yb * n + row];
      V[(size_t)xb * n + row] = fma(-rb.mx, vy, vx);
      V[(size_t)yb * n + row] = fma(rb.my, vx, vy);
    }
    // scales of the rotated indices (read again only in the next record phase)
    for (int i = g.t; i < h; i += g.n) {
      const SRec rr = rec[i];
      if (!srec_rotated(rr)) continue;
      int x, y;
      rr_slot(m, r, i, x, y);
      d[x] = dd_scale(d[x], rr.cm1);
      d[y] = dd_scale(d[y], rr.cm1);
    }
    gsync(g);
  }
  // fold the scales back: A_ij = Ã_ij d_i d_j off the diagonal, V_ij = Ṽ_ij d_j
  for (int e = g.t; e < n * n; e += g.n) {
    int i = e % n, j = e / n;
    const double sj = d[j].x + d[j].y;
    if (i != j) {
      const double si = d[i].x + d[i].y;
      A[e] = (A[e] * si) * sj;
    }
    V[e] *= sj;
  }
  gsync(g);
}

template <typename T>
MPJ_DEV double grp_off2(const Grp& g, int n, const T* A, double* red) {
  double s = 0.0;
  for (int e = g.t; e < n * n; e += g.n) {
    int i = e % n, j = e / n;
    if (i != j) {
      double x = (double)A[e];
      s += x * x;
    }
  }
  return group_sum(g, s, red);
}

// Elements of a group's buffer for one matrix (order at most nmax), and the bytes
// of a group's five buffers.
size_t group_cap(int nmax) { return ((size_t)nmax * nmax + 31) & ~(size_t)31; }
size_t group_bytes(int nmax) { return group_cap(nmax) * (2 * sizeof(float) + 3 * sizeof(double)); }

// order, nvec: matrix and size by place in the queue; cap: elements per buffer.
template <int G>
__global__ void __launch_bounds__(NTH, 1)
    batched_syev(const int* __restrict__ order, const int* __restrict__ nvec, const double* const* __restrict__ Aptr,
                 double* const* __restrict__ Wptr, double* const* __restrict__ Qptr, int batch, double tol_in,
                 int max32, int max64, int ns_steps, char* __restrict__ work, size_t cap,
                 int* __restrict__ counter, int* __restrict__ sweeps_out, unsigned* __restrict__ flags,
                 int region) {
  constexpr int NG = NTH / G;
  // stage 1 keeps A32 (and V32 when both fit) in this group's `region` floats
  // of shared memory
  extern __shared__ __align__(16) float dsm1[];
  __shared__ double red[NG][33];
  __shared__ SRec rec64[NG][NMAX / 2 + 1];
  __shared__ double2 dsc[NG][NMAX];
  __shared__ RotRec<float> rec32[NG][NMAX / 2 + 1];
  __shared__ int job[NG];
  __shared__ int rank_sh[NG][NMAX];
  Grp g;
  g.id = threadIdx.x / G;
  g.t = threadIdx.x % G;
  g.n = G;
  g.bar = 1 + g.id;
  char* base = work + ((size_t)blockIdx.x * NG + g.id) * cap * (2 * sizeof(float) + 3 * sizeof(double));
  Bufs B;
  B.A32 = (float*)base;
  B.V32 = B.A32 + cap;
  B.X = (double*)(base + 2 * cap * sizeof(float));
  B.M = B.X + cap;
  B.Y = B.M + cap;
  const int tid = g.t;
  for (;;) {
    if (tid == 0) job[g.id] = atomicAdd(counter, 1);
    gsync(g);
    const int jb = job[g.id];
    gsync(g);
    if (jb >= batch) break;
    const int idx = order[jb];
    const int n = nvec[jb];
    const double* A = Aptr[idx];
    double* W = Wptr[idx];
    double* Q = Qptr[idx];
    // a0: norms and finiteness
    double s = 0.0;
    bool bad = false;
    for (int e = tid; e < n * n; e += G) {
      double x = A[e];
      if (!isfinite(x)) bad = true;
      s += x * x;
    }
    if (bad) atomicOr(flags, MPJ_FLAG_NONFINITE);
    double normA = sqrt(group_sum(g, s, red[g.id]));
    double tol = tol_in > 0 ? tol_in : (double)n * 0x1p-53 * normA;
    double tol32 = (double)n * 0x1p-24 * normA;
    // 1. stage 1 (FP32 round-robin), in shared memory where it fits
    float* reg = dsm1 + (size_t)g.id * region;
    const int nn = n * n;
    float* A32 = nn <= region ? reg : B.A32;
    float* V32 = 2 * nn <= region ? reg + nn : B.V32;
    for (int e = tid; e < n * n; e += G) {
      A32[e] = (float)A[e];
      V32[e] = (e % n == e / n) ? 1.0f : 0.0f;
    }
    gsync(g);
    for (int sw = 0; sw < max32; ++sw) {
      double off2 = grp_off2<float>(g, n, A32, red[g.id]);
      if (!(off2 > tol32 * tol32)) break;
      grp_rr_sweep<float>(g, n, A32, V32, rec32[g.id], 0x1p-24f, 0.0f);
    }
    for (int e = tid; e < n * n; e += G) B.X[e] = (double)V32[e];
    gsync(g);
    // 2. Newton-Schulz
    double* X = B.X;
    double* Y = B.Y;
    for (int k = 0; k < ns_steps; ++k) {
      grp_gemm<true, false>(g, n, 1.0, X, X, 0.0, nullptr, B.M, true);
      grp_gemm<false, false>(g, n, -0.5, X, B.M, 1.5, X, Y, false);
      double* t = X;
      X = Y;
      Y = t;
    }
    // 3. A_cond = X^T (A X) -> M
    grp_gemm<false, false>(g, n, 1.0, A, X, 0.0, nullptr, Y, false);
    grp_gemm<true, false>(g, n, 1.0, X, Y, 0.0, nullptr, B.M, true);
    // 4. FP64 sweeps; their rotations are applied to Q_d's columns directly
    // (Q = Q_d V by associativity, no final product)
    double* V = X;
    int sweeps = 0;
    for (;;) {
      double off2 = grp_off2<double>(g, n, B.M, red[g.id]);
      if (!(off2 > tol * tol) || n < 2) break;
      if (sweeps >= max64) {
        if (tid == 0) atomicOr(flags, MPJ_FLAG_TIMEOUT);  // cap reached: reported as not converged
        break;
      }
      grp_rr_sweep_fast(g, n, B.M, V, rec64[g.id], dsc[g.id], 0x1p-53, tol / n);  // threshold variant
      ++sweeps;
    }
    // 5. sort; Q's columns are the rotated Q_d's, permuted
    for (int i = tid; i < n; i += G) {
      double wi = B.M[(size_t)i * n + i];
      int r = 0;
      for (int j = 0; j < n; ++j) {
        double wj = B.M[(size_t)j * n + j];
        r += (wj < wi) || (wj == wi && j < i);
      }
      rank_sh[g.id][i] = r;
      W[r] = wi;
    }
    gsync(g);
    for (int e = tid; e < n * n; e += G) {
      int i = e % n, j = e / n;
      Q[(size_t)rank_sh[g.id][j] * n + i] = V[e];
    }
    if (tid == 0) sweeps_out[idx] = sweeps;
    gsync(g);
  }
}

// ---------------------------------------------------------------- host side
typedef void (*KernelFn)(const int*, const int*, const double* const*, double* const*, double* const*, int, double,
                         int, int, int, char*, size_t, int*, int*, unsigned*, int);

// Shared memory for the stage-1 matrices: all the opt-in shared memory next to
// the kernel's static part, split evenly among the groups of a CTA.
cudaError_t stage1_smem(KernelFn k, int G, int* region, size_t* dyn) {
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaFuncAttributes fa;
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k);
  if (e != cudaSuccess) return e;
  const int ng = NTH / G;
  long budget = (long)optin - (long)fa.sharedSizeBytes - 1024;
  long per = budget > 0 ? budget / (ng * (long)sizeof(float)) : 0;
  per &= ~3L;  // keep each region 16-byte aligned
  if (per > 2L * NMAX * NMAX) per = 2L * NMAX * NMAX;
  *region = (int)per;
  *dyn = (size_t)ng * per * sizeof(float);
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)*dyn);
}

KernelFn kernel_for(int G) {
  if (G == 256) return batched_syev<256>;
  if (G == 512) return batched_syev<512>;
  return batched_syev<1024>;
}

const int kGroupSizes[3] = {256, 512, 1024};

struct Plan {
  int device = -1;
  int batch = 0;
  unsigned long long size_hash = 0, ptr_hash = 0;
  double tol = 0;
  int G = 0, grid = 0;
  void* work = nullptr;      // device workspace (groups) + queue + results
  int* h_sweeps = nullptr;   // pinned
  unsigned* h_flags = nullptr;
  cudaGraphExec_t exec = nullptr;
  cudaStream_t cap = nullptr;
};

std::mutex g_mu;
std::vector<Plan*> g_plans;  // most recent last
constexpr size_t kMaxPlans = 4;

// Autotune cache: size-histogram signature -> group size.
struct TuneEntry {
  std::string key;
  int G;
};
std::vector<TuneEntry> g_tune;
bool g_tune_loaded = false;

std::string signature(int batch, const int* n) {
  // counts in 8 size buckets of 32, each rounded to a power of two
  int c[8] = {0};
  for (int i = 0; i < batch; ++i) c[(n[i] - 1) / 32]++;
  char buf[128];
  int len = 0;
  for (int k = 0; k < 8; ++k) {
    int p = 0;
    while ((1 << p) < c[k]) ++p;
    len += snprintf(buf + len, sizeof buf - len, "%s%d", k ? "-" : "", c[k] ? p + 1 : 0);
  }
  return std::string(buf, len);
}

void tune_load() {
  if (g_tune_loaded) return;
  g_tune_loaded = true;
  const char* path = getenv("MPJ_AUTOTUNE_CACHE");
  if (!path) return;
  FILE* f = fopen(path, "r");
  if (!f) return;
  char key[128];
  int G;
  while (fscanf(f, "%127s %d", key, &G) == 2) g_tune.push_back({key, G});
  fclose(f);
}

void tune_store(const std::string& key, int G) {
  g_tune.push_back({key, G});
  const char* path = getenv("MPJ_AUTOTUNE_CACHE");
  if (!path) return;
  FILE* f = fopen(path, "a");
  if (!f) return;
  fprintf(f, "%s %d\n", key.c_str(), G);
  fclose(f);
}

int tune_lookup(const std::string& key) {
  for (auto& e : g_tune)
    if (e.key == key) return e.G;
  return 0;
}

unsigned long long fnv(const void* p, size_t bytes, unsigned long long h = 1469598103934665603ull) {
  const unsigned char* c = (const unsigned char*)p;
  for (size_t i = 0; i < bytes; ++i) h = (h ^ c[i]) * 1099511628211ull;
  return h;
}

void free_plan(Plan* p) {
  if (p->exec) cudaGraphExecDestroy(p->exec);
  if (p->cap) cudaStreamDestroy(p->cap);
  if (p->work) cudaFree(p->work);
  if (p->h_sweeps) cudaFreeHost(p->h_sweeps);
  if (p->h_flags) cudaFreeHost(p->h_flags);
  delete p;
}

struct Layout {
  size_t groups_bytes, order, nvec, sweeps, counter, total;
};

Layout layout_for(int batch, int grid) {
  Layout L;
  L.groups_bytes = group_bytes(NMAX) * (size_t)grid * MAXG;  // enough for the smallest group size
  L.order = L.groups_bytes;
  L.nvec = L.order + (((size_t)batch * sizeof(int) + 255) & ~(size_t)255);
  L.sweeps = L.nvec + (((size_t)batch * sizeof(int) + 255) & ~(size_t)255);
  L.counter = L.sweeps + (((size_t)batch * sizeof(int) + 255) & ~(size_t)255);
  L.total = L.counter + 256;
  return L;
}

cudaError_t launch_groups(int G, int grid, int nmax, const int* order, const int* n, const double* const* A,
                          double* const* W, double* const* Q, int batch, double tol, void* work, int* counter,
                          int* sweeps, unsigned* flags, cudaStream_t s) {
  int region = 0;
  size_t dyn = 0;
  const cudaError_t e = stage1_smem(kernel_for(G), G, &region, &dyn);
  if (e != cudaSuccess) return e;
  kernel_for(G)<<<grid, NTH, dyn, s>>>(order, n, A, W, Q, batch, tol, 15, 30, 2, (char*)work, group_cap(nmax), counter,
                                       sweeps, flags, region);
  return cudaGetLastError();
}

cudaError_t enqueue(const Plan* p, const Layout& L, const double* const* A, double* const* W, double* const* Q,
                    int G, cudaStream_t s, bool count) {
  char* base = (char*)p->work;
  int* d_counter = (int*)(base + L.counter);
  unsigned* d_flags = (unsigned*)(d_counter + 1);
  cudaError_t e = cudaMemsetAsync(d_counter, 0, 2 * sizeof(int), s);
  if (e != cudaSuccess) return e;
  e = launch_groups(G, p->grid, NMAX, (const int*)(base + L.order), (const int*)(base + L.nvec), A, W, Q, p->batch,
                    p->tol, base, d_counter, (int*)(base + L.sweeps), d_flags, s);
  if (count) mpj_count_launch();
  if (e != cudaSuccess) return e;
  e = cudaMemcpyAsync(p->h_sweeps, base + L.sweeps, sizeof(int) * p->batch, cudaMemcpyDeviceToHost, s);
  if (e != cudaSuccess) return e;
  return cudaMemcpyAsync(p->h_flags, d_flags, sizeof(unsigned), cudaMemcpyDeviceToHost, s);
}

}  // namespace

size_t mpj_batched_groups_bytes(int G, int grid, int nmax) { return group_bytes(nmax) * (size_t)grid * (NTH / G); }

cudaError_t mpj_batched_groups(int G, int grid, int nmax, const int* order, const int* n, const double* const* A,
                               double* const* W, double* const* Q, int batch, double tol, void* work, int* counter,
                               int* sweeps, unsigned* flags, cudaStream_t s) {
  mpj_count_launch();
  return launch_groups(G, grid, nmax, order, n, A, W, Q, batch, tol, work, counter, sweeps, flags, s);
}

extern "C" void mpj_release_plans(void) {
  mpj_release_pools();
  mpj_batched_rounds_release();
  std::lock_guard<std::mutex> lock(g_mu);
  for (Plan* p : g_plans) free_plan(p);
  g_plans.clear();
}

extern "C" int mpj_syev_batched(int batch, const int* n_host, const double* const* A_dev, double* const* W_dev,
                                double* const* Q_dev, double tol, int* sweeps_host, void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
  if (batch < 0 || (batch > 0 && (!n_host || !A_dev || !W_dev || !Q_dev))) return MPJ_EINVAL;
  if (batch == 0) return MPJ_OK;
  for (int i = 0; i < batch; ++i)
    if (n_host[i] < 1 || n_host[i] > NMAX) return MPJ_EINVAL;
  // Which form: by the sizes (choose_group in batched_rounds.cu) unless the
  // environment asks for the thread groups with their tuning and their graph.
  if (!getenv("MPJ_BATCHED_GROUP")) return mpj_batched_rounds(batch, n_host, A_dev, W_dev, Q_dev, tol, sweeps_host, s);
  int dev = 0, sms = 0;
  MPJ_CUDA_TRY(cudaGetDevice(&dev));
  MPJ_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  unsigned long long size_hash = fnv(n_host, sizeof(int) * (size_t)batch);
  unsigned long long ptr_hash = fnv(&A_dev, sizeof A_dev, fnv(&W_dev, sizeof W_dev, fnv(&Q_dev, sizeof Q_dev)));

  std::lock_guard<std::mutex> lock(g_mu);
  Plan* plan = nullptr;
  for (Plan* p : g_plans)
    if (p->device == dev && p->batch == batch && p->size_hash == size_hash && p->ptr_hash == ptr_hash &&
        p->tol == tol)
      plan = p;
  const int grid = sms;  // one CTA of 1024 threads per SM
  const Layout L = layout_for(batch, grid);
  if (!plan) {
    plan = new Plan;
    plan->device = dev;
    plan->batch = batch;
    plan->size_hash = size_hash;
    plan->ptr_hash = ptr_hash;
    plan->tol = tol;
    plan->grid = grid;
    cudaError_t e = cudaMalloc(&plan->work, L.total);
    mpj_count_alloc();
    if (e == cudaSuccess) e = cudaMallocHost((void**)&plan->h_sweeps, sizeof(int) * (size_t)batch);
    if (e == cudaSuccess) e = cudaMallocHost((void**)&plan->h_flags, sizeof(unsigned));
    mpj_count_alloc();
    mpj_count_alloc();
    if (e != cudaSuccess) {
      mpj_set_cuda_error(e, "batched plan allocation", __LINE__);
      free_plan(plan);
      return MPJ_ENOMEM;
    }
    // longest job first: order by decreasing n (counting sort), ties by index
    std::vector<int> order(batch), n_place(batch);
    {
      int cnt[NMAX + 2] = {0}, start[NMAX + 2];
      for (int i = 0; i < batch; ++i) cnt[n_host[i]]++;
      int acc = 0;
      for (int v = NMAX; v >= 1; --v) {
        start[v] = acc;
        acc += cnt[v];
      }
      for (int i = 0; i < batch; ++i) order[start[n_host[i]]++] = i;
      for (int i = 0; i < batch; ++i) n_place[i] = n_host[order[i]];
    }
    char* base = (char*)plan->work;
    e = cudaMemcpy(base + L.order, order.data(), sizeof(int) * (size_t)batch, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(base + L.nvec, n_place.data(), sizeof(int) * (size_t)batch, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
      mpj_set_cuda_error(e, "batched plan upload", __LINE__);
      free_plan(plan);
      return MPJ_ECUDA;
    }
    // autotune the group size on this batch unless its size histogram is known
    tune_load();
    const std::string key = signature(batch, n_host);
    int G = tune_lookup(key);
    if (const char* force = getenv("MPJ_BATCHED_GROUP")) {  // fixed group size (testing)
      int f = atoi(force);
      if (f == 256 || f == 512 || f == 1024) G = f;
    }
    if (!G) {
      float best = 1e30f;
      cudaEvent_t e0, e1;
      cudaEventCreate(&e0);
      cudaEventCreate(&e1);
      for (int c = 0; c < 3; ++c) {
        cudaEventRecord(e0, s);
        cudaError_t ee = enqueue(plan, L, A_dev, W_dev, Q_dev, kGroupSizes[c], s, true);
        cudaEventRecord(e1, s);
        if (ee == cudaSuccess) ee = cudaStreamSynchronize(s);
        if (ee != cudaSuccess) {
          mpj_set_cuda_error(ee, "batched autotune", __LINE__);
          cudaEventDestroy(e0);
          cudaEventDestroy(e1);
          free_plan(plan);
          return MPJ_ECUDA;
        }
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (ms < best) {
          best = ms;
          G = kGroupSizes[c];
        }
      }
      cudaEventDestroy(e0);
      cudaEventDestroy(e1);
      tune_store(key, G);
    }
    plan->G = G;
    // capture the replayable launch
    e = cudaStreamCreateWithFlags(&plan->cap, cudaStreamNonBlocking);
    cudaGraph_t graph = nullptr;
    if (e == cudaSuccess) e = cudaStreamBeginCapture(plan->cap, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
      cudaError_t eq = enqueue(plan, L, A_dev, W_dev, Q_dev, G, plan->cap, false);
      e = cudaStreamEndCapture(plan->cap, &graph);
      if (eq != cudaSuccess) e = eq;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&plan->exec, graph, 0);
    if (graph) cudaGraphDestroy(graph);
    if (e != cudaSuccess) {
      mpj_set_cuda_error(e, "batched graph capture", __LINE__);
      free_plan(plan);
      return MPJ_ECUDA;
    }
    if (g_plans.size() >= kMaxPlans) {
      free_plan(g_plans.front());
      g_plans.erase(g_plans.begin());
    }
    g_plans.push_back(plan);
  }
  cudaError_t e = cudaGraphLaunch(plan->exec, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    mpj_set_cuda_error(e, "mpj_syev_batched", __LINE__);
    return MPJ_ECUDA;
  }
  mpj_count_launch();  // the graph's kernel
  if (sweeps_host) memcpy(sweeps_host, plan->h_sweeps, sizeof(int) * (size_t)batch);
  unsigned hflags = *plan->h_flags;
  if (hflags & MPJ_FLAG_NONFINITE) return MPJ_ENONFINITE;
  if (hflags & MPJ_FLAG_TIMEOUT) return MPJ_NOT_CONVERGED;
  return MPJ_OK;
}

extern "C" int mpj_batched_group_size(int batch, const int* n_host) {
  std::lock_guard<std::mutex> lock(g_mu);
  tune_load();
  if (batch <= 0 || !n_host) return 0;
  return tune_lookup(signature(batch, n_host));
}
