// stage1.cu -- stage 1 of the mixed algorithm: approximate eigenvectors Q_l
// from an FP32 Jacobi (the paper's stage 1 is eig(single(A)), Sec. 4.1 and
// Algorithm 9; only an approximate Q_l with ||A Q_l - Q_l D_l|| <~ n u_l ||A||
// is needed, so the FP32 stage may use any convergent Jacobi ordering).
//
// Ordering: block round-robin.  The padded index range [0, N) (N a multiple
// of 32, pads inert: zero rows/columns never rotate) is cut into nb = N/16
// blocks of 16.  A sweep is nb-1 outer rounds of the circle method on blocks;
// in each round the nb/2 disjoint block pairs (I, J) each run one inner
// round-robin sweep over the 32 indices of I u J (31 inner rounds of 16
// disjoint pairs, Algorithm 2 with the skip test of Algorithm 4 at u_l = 2^-24)
// on their 32 x 32 diagonal subproblem, held in shared memory, accumulating the
// 32 x 32 orthogonal U_IJ.  The rotations of one round touch disjoint index
// sets, so applying them to the rest of the matrix afterwards as products
//   A[P,Q] <- U_P^T A[P,Q] U_Q,   V[:,Q] <- V[:,Q] U_Q
// (P, Q = index sets of block pairs) gives the same iterates as applying them
// one by one.  Each round is the subproblem solves and two block products
// (FP32 FMA, rmul32 or rmul32_pipe): V <- V U~ and A <- U~^T A U~ (the lower
// tiles, each formed once and mirrored), so that A32 and V32 are touched once
// per round instead of once per pair step.  off(A32) is reduced after each sweep; stop
// at off(A32) <= tol32 or the sweep cap.
#include <memory>
#include <mutex>
#include <vector>
#include <cuda_fp16.h>
#include <stdlib.h>

#include "batch.cuh"
#include "common.cuh"
#include "stage1.cuh"
#include "tc32.cuh"

namespace {

constexpr int BS = 16;  // block size
constexpr int W2 = 32;  // indices per block pair
constexpr int LD = 33;  // padded shared-memory leading dimension

// global index of local index l in block pair (I, J)
MPJ_DEV int gidx(int I, int J, int l) { return l < BS ? I * BS + l : J * BS + (l - BS); }

MPJ_DEV void block_pair(int nb, int R, int slot, int& I, int& J) {
  int x, y;
  rr_slot(nb, R, slot, x, y);
  I = x < y ? x : y;
  J = x < y ? y : x;
}

// Where the two blocks of pair `slot` of round R >= 1 were in round R - 1: slots
// a (of the lower block) and q, and the blocks' offsets in those pairs.
MPJ_DEV void prev_slots(int nb, int R, int slot, int& a, int& oa, int& q, int& oq) {
  int I, J, y, lo, hi;
  block_pair(nb, R, slot, I, J);
  rr_slot_of(nb, R - 1, I, a, y);
  block_pair(nb, R - 1, a, lo, hi);
  oa = I == hi ? BS : 0;
  rr_slot_of(nb, R - 1, J, q, y);
  block_pair(nb, R - 1, q, lo, hi);
  oq = J == hi ? BS : 0;
}

// hq: the half-precision stage (binary16 values; Ch. 6 further work item 3):
// every stored value and rotation parameter is rounded to binary16.
MPJ_DEV float qh(float v, bool hq) { return hq ? __half2float(__float2half_rn(v)) : v; }

__global__ void init32(const double* __restrict__ A, int lda, int n, int N, float* __restrict__ A32,
                       float* __restrict__ V32, bool hq) {
  size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  size_t total = (size_t)N * N;
  for (; idx < total; idx += (size_t)gridDim.x * blockDim.x) {
    int i = (int)(idx % N), j = (int)(idx / N);
    A32[idx] = (i < n && j < n) ? qh((float)A[(size_t)j * lda + i], hq) : 0.0f;
    V32[idx] = (i == j) ? 1.0f : 0.0f;
  }
}

__global__ void widen(const float* __restrict__ V32, int N, int n, double* __restrict__ Q, int ldq) {
  size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  size_t total = (size_t)n * n;
  for (; idx < total; idx += (size_t)gridDim.x * blockDim.x) {
    int i = (int)(idx % n), j = (int)(idx / n);
    Q[(size_t)j * ldq + i] = (double)V32[(size_t)j * N + i];
  }
}

// The rotation of pair (p, q), p < q, for the FP32 inner sweep: Algorithm 2
// with the skip test of Algorithm 4 (compared in squares) in half-angle form,
// which has the shortest chain of special functions: z = |sin 2 theta| =
// 1 / sqrt(1 + tau^2), c^2 = (1 + |tau| z) / 2, s = z / (2 c) with tau's sign
// ('+' for 0), c - 1 = -s^2 / (1 + c), and t a_pq = s a_pq / c for the diagonal
// a_pp - t a_pq, a_qq + t a_pq.  c - 1 comes from s, so an error of c enters
// (1 + cm1)^2 + s^2 - 1 by less than a quarter.  |tau| is capped at 1e18: s
// is then below FP32 resolution.  The flush-to-zero forms take half the latency
// (19 against 41 cycles); their operands are normal numbers whenever apq^2 > 0
// passes the skip test.  No branch: lanes that skip select zeros.
struct Rot32 {
  float cm1, sig;
};
MPJ_DEV bool rot32(float& app, float& aqq, float apq, float skip, Rot32& rr) {
  const bool rot = apq * apq > (skip * skip) * fabsf(app * aqq);
  const float tau = (aqq - app) * rcp_ftz(2.0f * apq), at = fminf(fabsf(tau), 1e18f);
  const float z = rsqrt_ftz(fmaf(at, at, 1.0f));
  const float c2 = fmaf(0.5f * at, z, 0.5f);
  const float ic = rsqrt_ftz(c2);
  const float sa = 0.5f * z * ic, s = tau >= 0.0f ? sa : -sa;
  const float c1 = fmaf(c2, ic, 1.0f);  // 1 + c
  const float ta = rot ? s * ic * apq : 0.0f;
  rr.cm1 = rot ? -(s * s) * rcp_ftz(c1) : 0.0f;
  rr.sig = rot ? s : 0.0f;
  app -= ta;
  aqq += ta;
  return rot;
}

// One entry of a rotated pair: `own` with the other index's entry `oth`
// (sg = -sig for the pair's first index, +sig for its second).
MPJ_DEV float rot_one(float cm1, float sg, float own, float oth) { return fmaf(cm1, own, fmaf(sg, oth, own)); }

// v with a zero bit inserted at position h, and with bit h taken out
MPJ_DEV int ins0(int v, int h) { return ((v >> h) << (h + 1)) | (v & ((1 << h) - 1)); }
MPJ_DEV int del0(int v, int h) { return ((v >> (h + 1)) << h) | (v & ((1 << h) - 1)); }

// One CTA per block pair of outer round R: inner sweep on the 32 x 32
// subproblem; writes the rotated subproblem S (column-major), the accumulated
// U (row-major for the FP32 products, column-major, urow false, for the
// tensor-core panel) and the set T of its indices that rotated (Mbuf, bit l
// for local index l, if not null): U is the identity outside T x T.
//
// The inner sweep runs the exclusive-or ordering: round r = 1 .. 31 rotates
// the 16 disjoint pairs (i, i ^ r), every pair once per sweep.  Pair k of
// round r is p = k with a zero bit inserted at r's highest bit h, q = p ^ r, so
// p < q always, and the 2 x 2 blocks between two pairs are enumerated by bit
// operations alone.  S is held once per unordered index pair, entry {i, j} at
// (i ^ j) * SLD + min(i, j), so a block is read and written once without a
// mirror.  What bounds the kernel is the chain coupling -> angle -> records ->
// next round's coupling: the 16 couplings of the next round all lie in eight
// blocks of this one, so warp 0 recomputes just those 16 entries and forms the
// next round's rotations, with every address of the round computed before the
// barrier that opens it; the blocks are left to warps 1-8 (half a block, one
// row, per thread) and U to warps 9-16 (lane = row, two column pairs each).
// S alternates between two buffers, so one barrier per round is enough.
// Measured at n = 4096 (128 CTAs): circle ordering, two barriers, IEEE
// divisions 23.8 us per launch; two index sets per thread and four-task warps
// 18.4 us; this form 12.3 us.  The sweeps to reach
// the stopping test are the same or one fewer (n = 96 .. 512, three spectra).
// One subproblem: pair `slot` of round R of a matrix with nb blocks, and where
// its S, U and T go.
struct Sub32 {
  const float* A;
  int N, nb, slot;
  float *S, *U;
  unsigned* M;
  const float *Sp, *Up, *T;  // looking ahead: S and U of the previous round's pairs, this pair's saved tile
};
struct OneSub32 {  // the block pairs of one matrix
  const float* A;
  int N, nb;
  float *S, *U;
  unsigned* M;
  const float *Sp, *Up, *T;
  MPJ_DEV bool get(int bid, Sub32& v) const {
    v = Sub32{A, N, nb, bid, S + (size_t)bid * W2 * W2, U + (size_t)bid * W2 * W2, M ? M + bid : nullptr,
              Sp, Up, T + (size_t)bid * W2 * W2};
    return true;
  }
};
struct BatchSub32 {  // the block pairs of a batch
  BatchShape b;
  int lo;
  const float* A;
  float *S, *U;
  MPJ_DEV bool get(int bid, Sub32& v) const {
    BatchTask t;
    if (!batch_find(b, lo, bid, [](int np) { return np; }, t)) return false;
    const size_t o = (size_t)(t.pair0 + t.local) * W2 * W2;
    v = Sub32{A + t.el, t.N, t.N / BS, t.local, S + o, U + o, nullptr, nullptr, nullptr, nullptr};
    return true;
  }
};
constexpr int S32_THREADS = 544;
constexpr int SLD = 40;  // row stride of the packed S (8 more than 32: rows of d, d + 1, .. start 8 banks apart)
// The CTA's barrier from the three roles' own code paths.
MPJ_DEV void s32_barrier() { asm volatile("bar.sync 0, %0;\n" ::"n"(S32_THREADS) : "memory"); }

template <bool HQ, class Src>
__global__ void __launch_bounds__(S32_THREADS, 1) solve32(Src src, int R, bool urow) {
  __shared__ float S[2][W2 * SLD];
  __shared__ float U[W2][LD];  // U[column][row]
  __shared__ float dg[W2];     // the diagonal (warp 0 only)
  __shared__ float Uh[2][W2][BS];  // looking ahead: the halves of U_a and U_q
  __shared__ Rot32 rec[2][W2 / 2];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  pdl_wait();
  Sub32 sub;
  if (!src.get(blockIdx.x, sub)) return;
  int I, J;
  block_pair(sub.nb, R, sub.slot, I, J);
  unsigned* const Mbuf = sub.M;
  if (sub.Sp) {
    // the subproblem before A has received the previous round's update: its two
    // diagonal blocks are blocks of that round's solved subproblems, its
    // coupling block is U_a^T T U_q on the tile T between their pairs
    int a, oa, q, oq;
    prev_slots(sub.nb, R, sub.slot, a, oa, q, oq);
    const float *Sa = sub.Sp + (size_t)a * W2 * W2, *Sq = sub.Sp + (size_t)q * W2 * W2;
    const float *Ua = sub.Up + (size_t)a * W2 * W2, *Uq = sub.Up + (size_t)q * W2 * W2;
    float(*Ts)[LD] = reinterpret_cast<float(*)[LD]>(S[1]);  // T(r, k) at [k][r]
    for (int e = tid; e < W2 * W2; e += S32_THREADS) {
      const int li = e % W2, lj = e / W2;
      Ts[lj][li] = sub.T[e];
      if (li <= lj && (lj < BS || li >= BS)) {
        const float v = lj < BS ? Sa[(oa + lj) * W2 + oa + li] : Sq[(oq + lj - BS) * W2 + oq + li - BS];
        if (li == lj)
          dg[li] = v;
        else
          S[0][(li ^ lj) * SLD + li] = v;
      }
      if (e < W2 * BS) {
        const int k = e / BS, c = e % BS;
        Uh[0][k][c] = Ua[k * W2 + oa + c];
        Uh[1][k][c] = Uq[k * W2 + oq + c];
      }
    }
    __syncthreads();
    if (tid < W2 * BS) {  // T U_q, into U's place as [column][row]
      float acc = 0.0f;
#pragma unroll 8
      for (int k = 0; k < W2; ++k) acc = fmaf(Ts[k][lane], Uh[1][k][warp], acc);
      U[warp][lane] = acc;
    }
    __syncthreads();
    if (tid < BS * BS) {
      const int i = tid % BS, j = tid / BS;
      float acc = 0.0f;
#pragma unroll 8
      for (int r = 0; r < W2; ++r) acc = fmaf(Uh[0][r][i], U[j][r], acc);
      S[0][(i ^ (BS + j)) * SLD + i] = qh(acc, HQ);
    }
    __syncthreads();
    for (int e = tid; e < W2 * W2; e += S32_THREADS) U[e / W2][e % W2] = (e % W2 == e / W2) ? 1.0f : 0.0f;
  } else {
    for (int e = tid; e < W2 * W2; e += S32_THREADS) {
      const int li = e % W2, lj = e / W2;
      const float v = sub.A[(size_t)gidx(I, J, lj) * sub.N + gidx(I, J, li)];
      if (li == lj)
        dg[li] = v;
      else if (li < lj)
        S[0][(li ^ lj) * SLD + li] = v;
      U[lj][li] = (li == lj) ? 1.0f : 0.0f;
    }
  }
  __syncthreads();
  const float skip = HQ ? 0x1p-11f : 0x1p-24f;
  if (warp == 0) {
    unsigned tmask = 0u;  // the indices that rotated so far
    float held = 0.0f;    // the pair's own coupling after its rotation
    const int k = lane & 15;
    // rotation of pair (p, q), record k, from its coupling, into rec[buf]
    auto rotate = [&](int p, int q, float app, float aqq, float apq, int buf) {
      Rot32 rr;
      const bool rot = rot32(app, aqq, apq, skip, rr);
      if (HQ) {  // c and s as binary16, new diagonal rounded
        rr.cm1 = qh(1.0f + rr.cm1, true) - 1.0f;
        rr.sig = qh(rr.sig, true);
        app = rot ? qh(app, true) : app;
        aqq = rot ? qh(aqq, true) : aqq;
      }
      __syncwarp();  // every lane has read the diagonal
      if (lane < W2 / 2) {
        rec[buf][k] = rr;
        dg[p] = app;
        dg[q] = aqq;
      }
      held = rot ? 0.0f : apq;
      if (Mbuf) {
        const unsigned bits = rec_rotated(rr.cm1, rr.sig) ? ((1u << p) | (1u << q)) : 0u;
        tmask |= __reduce_or_sync(0xFFFFFFFFu, bits);
      }
    };
    rotate(2 * k, 2 * k + 1, dg[2 * k], dg[2 * k + 1], S[0][SLD + 2 * k], 0);
    int p_cur = 2 * k;
#pragma unroll 1
    for (int r = 1; r < W2; ++r) {
      const int cur = (r - 1) & 1;
      const int h = 31 - __clz(r), rn = r + 1, hn = 31 - __clz(rn);
      const int p = ins0(k, hn), q = p ^ rn, po = p ^ r, qo = q ^ r;
      // this round's pairs of p and of q: records and the side of each
      const bool p2 = (p >> h) & 1, q2 = (q >> h) & 1;
      const Rot32* pa = &rec[cur][del0(p2 ? po : p, h)];
      const Rot32* pb = &rec[cur][del0(q2 ? qo : q, h)];
      const int dA = (rn & 31) * SLD, dB = ((rn ^ r) & 31) * SLD;
      const int i00 = dA + min(p, q), i11 = dA + min(po, qo);
      const int i01 = dB + min(p, qo), i10 = dB + min(po, q);
      float* Sh = &S[cur ^ 1][r * SLD + p_cur];
      const float* Sc = S[cur];
      s32_barrier();
      if (lane < W2 / 2) *Sh = held;
      if (rn < W2) {
        const Rot32 ra = *pa, rb = *pb;
        const float app = dg[p], aqq = dg[q];
        const float e00 = Sc[i00], e01 = Sc[i01], e10 = Sc[i10], e11 = Sc[i11];
        const float sa = p2 ? ra.sig : -ra.sig, sb = q2 ? rb.sig : -rb.sig;
        const float t0 = rot_one(ra.cm1, sa, e00, e10), t1 = rot_one(ra.cm1, sa, e01, e11);
        rotate(p, q, app, aqq, qh(rot_one(rb.cm1, sb, t0, t1), HQ), cur ^ 1);
        p_cur = p;
      }
    }
    if (lane == 0 && Mbuf) *Mbuf = tmask;
  } else if (warp < 9) {
    // half a block: pairs with 4-bit labels xl and yl = xl ^ dl, xl's bit at
    // dl's highest bit zero (15 x 8 unordered label pairs), and the row of
    // xl's first (side 0) or second index
    const int bt = (tid - 32) >> 1, side = tid & 1, dl = 1 + (bt >> 3);
    const int xl = ins0(bt & 7, 31 - __clz(dl)), yl = xl ^ dl;
    const bool on = bt < 120;
#pragma unroll 1
    for (int h = 0; h < 5; ++h) {
      const int x = ins0(xl, h), y = ins0(yl, h), d0 = x ^ y;
#pragma unroll 1
      for (int r = 1 << h; r < (2 << h); ++r) {
        const int cur = (r - 1) & 1, rn = r + 1;
        const int i = side ? x ^ r : x, io = i ^ r, y2 = y ^ r, d1 = d0 ^ r;
        const int ds = side ? d1 : d0, dt = side ? d0 : d1;  // i ^ y and i ^ y2
        const int i0 = ds * SLD + min(i, y), i1 = dt * SLD + min(i, y2);
        const int o0 = dt * SLD + min(io, y), o1 = ds * SLD + min(io, y2);
        const float* Sc = S[cur];
        float* Sn = S[cur ^ 1];
        s32_barrier();
        if (on) {
          const Rot32 ra = rec[cur][xl], rb = rec[cur][yl];
          const float v0 = Sc[i0], v1 = Sc[i1], w0 = Sc[o0], w1 = Sc[o1];
          const float sg = side ? ra.sig : -ra.sig;
          const float t0 = rot_one(ra.cm1, sg, v0, w0), t1 = rot_one(ra.cm1, sg, v1, w1);
          // warp 0 holds the next round's couplings
          if (ds != rn) Sn[i0] = qh(rot_one(rb.cm1, -rb.sig, t0, t1), HQ);
          if (dt != rn) Sn[i1] = qh(rot_one(rb.cm1, rb.sig, t1, t0), HQ);
        }
      }
    }
  } else {
    const int k0 = 2 * (warp - 9);
#pragma unroll 1
    for (int h = 0; h < 5; ++h) {
      const int pa = ins0(k0, h), pb = ins0(k0 + 1, h);
#pragma unroll 1
      for (int r = 1 << h; r < (2 << h); ++r) {
        const int cur = (r - 1) & 1;
        float *u0 = &U[pa][lane], *u1 = &U[pa ^ r][lane], *w0 = &U[pb][lane], *w1 = &U[pb ^ r][lane];
        s32_barrier();
        const Rot32 ra = rec[cur][k0], rb = rec[cur][k0 + 1];
        const float a0 = *u0, a1 = *u1, b0 = *w0, b1 = *w1;
        *u0 = qh(rot_one(ra.cm1, -ra.sig, a0, a1), HQ);
        *u1 = qh(rot_one(ra.cm1, ra.sig, a1, a0), HQ);
        *w0 = qh(rot_one(rb.cm1, -rb.sig, b0, b1), HQ);
        *w1 = qh(rot_one(rb.cm1, rb.sig, b1, b0), HQ);
      }
    }
  }
  s32_barrier();
  float *So = sub.S, *Uo = sub.U;
  for (int e = tid; e < W2 * W2; e += S32_THREADS) {
    const int li = e % W2, lj = e / W2;
    So[e] = li == lj ? dg[li] : S[1][(li ^ lj) * SLD + min(li, lj)];
    Uo[e] = urow ? U[li][lj] : U[lj][li];
  }
}


// Saves, for every pair of round R >= 1, the 32 x 32 tile of A between the pairs
// of round R - 1 that held its two blocks (rows of the lower block's pair).
__global__ void __launch_bounds__(256) snap32(const float* __restrict__ A32, int N, int nb, int R,
                                              float* __restrict__ T) {
  pdl_wait();
  int a, oa, q, oq, Ia, Ja, Iq, Jq;
  prev_slots(nb, R, blockIdx.x, a, oa, q, oq);
  block_pair(nb, R - 1, a, Ia, Ja);
  block_pair(nb, R - 1, q, Iq, Jq);
  float* t = T + (size_t)blockIdx.x * W2 * W2;
  for (int e = threadIdx.x; e < W2 * W2; e += 256)
    t[e] = A32[(size_t)gidx(Iq, Jq, e / W2) * N + gidx(Ia, Ja, e % W2)];
}

// Packed pairs of FP32 values (low word first) and the paired FMA
// d = a * b + d, each half rounded to nearest like fmaf.
MPJ_DEV unsigned long long pk2(float lo, float hi) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
MPJ_DEV void unpk2(unsigned long long v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
MPJ_DEV void fma2(unsigned long long& d, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

// ---------------------------------------------------------------- block update
enum { R32_ALL = 0, R32_BOTH = 1 };
constexpr int RT = 128;
constexpr int XLD = 132;  // padded row length of the X tile (k-major), 16-byte aligned rows
constexpr int ULD = 40;   // padded row length of U_Q, 16-byte aligned rows

// The 32 x 32 product of one warp: acc(4 g + i, 8 h + j) = sum_k L(k, 4 g + i) R(k, 8 h + j)
// for lane (g, h) = (lane mod 8, lane / 8), L and R k-major in shared memory
// (row stride LDL, LDR floats); packed FP32 pairs, each half rounded as fmaf.
template <int LDL, int LDR>
MPJ_DEV void warp_mm32(const float* L, const float* R, int g, int h, float acc[4][8]) {
  unsigned long long acc2[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int jp = 0; jp < 4; ++jp) acc2[i][jp] = 0ULL;
#pragma unroll 4
  for (int k = 0; k < W2; ++k) {
    const float4 x = *reinterpret_cast<const float4*>(L + k * LDL + 4 * g);
    const float4 u0 = *reinterpret_cast<const float4*>(R + k * LDR + 8 * h);
    const float4 u1 = *reinterpret_cast<const float4*>(R + k * LDR + 8 * h + 4);
    const float xa[4] = {x.x, x.y, x.z, x.w};
    const unsigned long long up[4] = {pk2(u0.x, u0.y), pk2(u0.z, u0.w), pk2(u1.x, u1.y), pk2(u1.z, u1.w)};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const unsigned long long xx = pk2(xa[i], xa[i]);
#pragma unroll
      for (int jp = 0; jp < 4; ++jp) fma2(acc2[i][jp], xx, up[jp]);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int jp = 0; jp < 4; ++jp) unpk2(acc2[i][jp], acc[i][2 * jp], acc[i][2 * jp + 1]);
}

// warp_mm32 with the contraction restricted to the indices k in `mask` (in
// increasing order: the terms it leaves out are exact zeros, so the sums
// are those of the full contraction).
template <int LDL, int LDR>
MPJ_DEV void warp_mm32_masked(const float* L, const float* R, int g, int h, unsigned mask, float acc[4][8]) {
  unsigned long long acc2[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int jp = 0; jp < 4; ++jp) acc2[i][jp] = 0ULL;
  for (unsigned m = mask; m; m &= m - 1) {
    const int k = __ffs(m) - 1;
    const float4 x = *reinterpret_cast<const float4*>(L + k * LDL + 4 * g);
    const float4 u0 = *reinterpret_cast<const float4*>(R + k * LDR + 8 * h);
    const float4 u1 = *reinterpret_cast<const float4*>(R + k * LDR + 8 * h + 4);
    const float xa[4] = {x.x, x.y, x.z, x.w};
    const unsigned long long up[4] = {pk2(u0.x, u0.y), pk2(u0.z, u0.w), pk2(u1.x, u1.y), pk2(u1.z, u1.w)};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const unsigned long long xx = pk2(xa[i], xa[i]);
#pragma unroll
      for (int jp = 0; jp < 4; ++jp) fma2(acc2[i][jp], xx, up[jp]);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int jp = 0; jp < 4; ++jp) unpk2(acc2[i][jp], acc[i][2 * jp], acc[i][2 * jp + 1]);
}

// U(k, c) of block pair P (32 x 32 in Ubuf, row-major, or column-major when
// ucol) into Us[k][c]
MPJ_DEV void load_u(const float* __restrict__ Ubuf, int P, float (*Us)[ULD], int t, int nt, bool ucol) {
  const float* Uq = Ubuf + (size_t)P * W2 * W2;
  for (int e = 4 * t; e < W2 * W2; e += 4 * nt) {
    const float4 v = *reinterpret_cast<const float4*>(Uq + e);
    if (!ucol) {
      *reinterpret_cast<float4*>(&Us[e / W2][e % W2]) = v;
    } else {
      const int k = e % W2, c = e / W2;
      Us[k][c] = v.x;
      Us[k + 1][c] = v.y;
      Us[k + 2][c] = v.z;
      Us[k + 3][c] = v.w;
    }
  }
}

// The round's rotations applied to the rest of A32 and to V32 as block-diagonal
// right multiplications Y[:, g_Q(c)] = X_Q U_Q (FP32 FMA, K = 32) over tiles
// (a, Q): block pair Q and the 128 rows that are the 32 indices of each of
// the block pairs a = 4 gx .. 4 gx + 3.  Modes:
//   R32_ALL    V <- V U~ (every tile, in place);
//   R32_BOTH   A <- U~^T A U~ in one pass, in place: tile (a, Q), a > Q, gets
//              U_a^T (A[P_a, Q] U_Q) (the second product on the first one's
//              result in shared memory), written to both triangles; the
//              diagonal tiles a = Q are the solved subproblems S.  The tiles
//              read (a > Q) are only those their own CTA writes, the mirrors
//              (Q, a) are read by no CTA.
// 128 threads: the tile's 128 x 32 values of X_Q and U_Q in shared memory,
// then warp w forms the 32 x 32 block of tile rows 32 w .. +31 (block pair
// a0 + w) and lane (g, h) = (t mod 8, t / 8 mod 4) the 4 x 8 block of rows
// 32 w + 4 g .. +3 and columns 8 h .. +7: per k one float4 of X (8 distinct
// in a warp: one shared-memory wavefront) and two float4 of U_Q (4 distinct:
// one wavefront each) feed 32 FMAs.
template <int NUA>
struct __align__(16) Rmul32Smem {
  float Xs[W2][XLD];       // Xs[k][r] = X_Q(r, k); R32_BOTH: then T = X_Q U_Q per warp
  float Us[W2][ULD];       // Us[k][c] = U_Q(k, c)
  float Ua[NUA][W2][ULD];  // R32_BOTH: U_a of each warp's pair
};
template <int TRI, bool MASKED, int NUA>
MPJ_DEV void rmul32_tile(Rmul32Smem<NUA>& sm, const float* X, float* Y, int N, int nb, int R,
                         const float* __restrict__ Sbuf, const float* __restrict__ Ubuf, bool hq, bool ucol,
                         const unsigned* __restrict__ Mbuf, int gx, int Q) {
  auto& Xs = sm.Xs;
  auto& Us = sm.Us;
  auto& Ua = sm.Ua;
  const int tid = threadIdx.x;
  const int npairs = nb / 2;
  const int a0 = 4 * gx, a1 = min(4 * gx + 3, npairs - 1);
  if (TRI == R32_BOTH && a1 < Q) return;
  const int warp = tid >> 5, lane = tid & 31;
  const int a = a0 + warp;  // this warp's block pair
  // the indices of block pairs Q and a that rotated (U is the identity
  // outside them); loaded together with the U blocks, used after them
  const unsigned mQ = MASKED ? Mbuf[Q] : 0xFFFFFFFFu;
  const unsigned ma = !MASKED ? 0xFFFFFFFFu : (TRI == R32_BOTH && a < npairs) ? Mbuf[a] : 0u;
  int IQ, JQ;
  block_pair(nb, R, Q, IQ, JQ);
  load_u(Ubuf, Q, Us, tid, RT, ucol);
  if (TRI == R32_BOTH && a < npairs && a > Q) load_u(Ubuf, a, Ua[warp], lane, 32, ucol);
  if (TRI == R32_ALL && mQ == 0u) return;  // V U~ leaves these columns as they are
  {
    // X_Q(r, k) = X[g_Q(k) N + row(r)]; thread t: tile rows 4 (t mod 32) .. +3
    // (consecutive rows of one block), contraction indices k = t / 32 + 4 i
    const int rq = tid & 31, ar = a0 + (rq >> 3);
    int row = -1;
    if (ar < npairs && (TRI != R32_BOTH || ar > Q)) {
      int I, J;
      block_pair(nb, R, ar, I, J);
      row = gidx(I, J, (4 * rq) & 31);
    }
#pragma unroll
    for (int i = 0; i < W2 / 4; ++i) {
      const int k = (tid >> 5) + 4 * i;
      if (TRI == R32_ALL && !((mQ >> k) & 1u)) continue;  // column not read (V U~ contracts over T_Q only)
      const float4 v = row >= 0 ? *reinterpret_cast<const float4*>(X + (size_t)gidx(IQ, JQ, k) * N + row)
                                : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      *reinterpret_cast<float4*>(&Xs[k][4 * rq]) = v;
    }
  }
  __syncthreads();
  const int g = lane & 7, h = lane >> 3;
  const int c0 = 8 * h;
  if (a >= npairs) return;
  if (TRI == R32_BOTH && a < Q) return;
  int I, J;
  block_pair(nb, R, a, I, J);
  const int row0 = gidx(I, J, 4 * g);  // rows row0 .. row0 + 3 (one block)
  const int col0 = gidx(IQ, JQ, c0);   // columns col0 .. col0 + 7 (one block)
  if (TRI == R32_BOTH && a == Q) {
    // the diagonal tile: the solved subproblem
    const float* Sq = Sbuf + (size_t)Q * W2 * W2;
#pragma unroll
    for (int cc = 0; cc < 8; ++cc) {
      const float4 o = *reinterpret_cast<const float4*>(Sq + 4 * g + W2 * (c0 + cc));
      *reinterpret_cast<float4*>(Y + (size_t)(col0 + cc) * N + row0) = o;
    }
    return;
  }
  if (TRI == R32_BOTH && mQ == 0u && ma == 0u) return;  // U_a^T A U_Q = A on this tile
  // a column c outside T_Q: (X U_Q)(:, c) = X(:, c); else the contraction over T_Q
  float acc[4][8];
  if (mQ == 0xFFFFFFFFu) {
    warp_mm32<XLD, ULD>(&Xs[0][32 * warp], &Us[0][0], g, h, acc);
  } else {
    warp_mm32_masked<XLD, ULD>(&Xs[0][32 * warp], &Us[0][0], g, h, mQ, acc);
    if (TRI == R32_BOTH) {
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (!((mQ >> (c0 + j)) & 1u)) {
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[i][j] = Xs[c0 + j][32 * warp + 4 * g + i];
        }
    }
  }
  if (TRI == R32_BOTH) {
    // T = X_Q U_Q over this warp's 32 x 32 block of Xs (T(i, c) at Xs[i][32 w + c]),
    // then U_a^T T (a row r outside T_a: (U_a^T T)(r, :) = T(r, :))
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      *reinterpret_cast<float4*>(&Xs[4 * g + i][32 * warp + c0]) =
          make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
      *reinterpret_cast<float4*>(&Xs[4 * g + i][32 * warp + c0 + 4]) =
          make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]);
    }
    __syncwarp();
    if (ma == 0xFFFFFFFFu) {
      warp_mm32<ULD, XLD>(&Ua[warp][0][0], &Xs[0][32 * warp], g, h, acc);
    } else {
      warp_mm32_masked<ULD, XLD>(&Ua[warp][0][0], &Xs[0][32 * warp], g, h, ma, acc);
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (!((ma >> (4 * g + i)) & 1u)) {
#pragma unroll
          for (int j = 0; j < 8; ++j) acc[i][j] = Xs[4 * g + i][32 * warp + c0 + j];
        }
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = qh(acc[i][j], hq);
#pragma unroll
  for (int j = 0; j < 8; ++j)
    if (TRI == R32_BOTH || ((mQ >> (c0 + j)) & 1u))  // V: only the columns in T_Q change
      *reinterpret_cast<float4*>(Y + (size_t)(col0 + j) * N + row0) =
          make_float4(acc[0][j], acc[1][j], acc[2][j], acc[3][j]);
  if (TRI == R32_BOTH) {  // the mirror: rows col0 .. +7 of columns row0 .. +3
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      *reinterpret_cast<float4*>(Y + (size_t)(row0 + i) * N + col0) =
          make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
      *reinterpret_cast<float4*>(Y + (size_t)(row0 + i) * N + col0 + 4) =
          make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]);
    }
  }
}

template <int TRI, bool MASKED>
__global__ void __launch_bounds__(RT) rmul32(const float* X, float* Y, int N, int nb, int R,
                                             const float* __restrict__ Sbuf, const float* __restrict__ Ubuf, bool hq,
                                             bool ucol, const unsigned* __restrict__ Mbuf) {
  __shared__ Rmul32Smem<TRI == R32_BOTH ? 4 : 1> sm;
  pdl_wait();
  rmul32_tile<TRI, MASKED>(sm, X, Y, N, nb, R, Sbuf, Ubuf, hq, ucol, Mbuf, blockIdx.x, blockIdx.y);
}

// ---------------------------------------------------------------- both updates in one launch
// The tiles of A <- U~^T A U~ and V <- V U~ formed by persistent CTAs of two
// warps, each from a queue: while a tile is multiplied, the next one's values
// and rotations are on their way (cp.async, two stages).  Half-warp w forms the
// 32 x 32 block of block pair 4 gx + w, each lane 8 x 8 of it: 16 shared-memory
// floats per 64 FMAs, where rmul32's 4 x 8 take 12 per 32.  What rmul32 spends
// its time on at n = 4096 (A 46 us, V 33 us, DRAM traffic 46 and 79 MB): its
// loads keep the shared-memory pipe 70-75 % busy, and every tile waits for its
// values with 17 to 25 warps resident.  More outputs per lane alone, without the
// pipeline, lost (A's and V's rounds 88 us instead of 82: half the warps to hide
// the wait with).  Measured per round, subproblems included (they overlap):
// see update_form.
constexpr int PT = 64;
template <bool VONLY>
struct __align__(16) PipeStage {
  float X[W2][XLD];     // X[k][r] = X_Q(r, k); A: then T = X_Q U_Q per half-warp
  float U[W2][W2];      // U[k][c] = U_Q(k, c)
  float Ua[4][W2][W2];  // A: U_a of each half-warp's pair
};
template <>
struct __align__(16) PipeStage<true> {
  float X[W2][XLD];
  float U[W2][W2];
};

MPJ_DEV void cp16(float* dst, const float* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(valid ? 16 : 0)
               : "memory");
}

// The 32 x 32 product of a half-warp: acc(i, j) = sum_k L(k, r_i) R(k, c_j) for
// the lane's rows r = {0 .. 3, 16 .. 19} and columns c alike, relative to L and R
// (k-major, row strides LDL, LDR); the sums are warp_mm32's.
template <int LDL, int LDR>
MPJ_DEV void half_mm32(const float* L, const float* R, float acc[8][8]) {
  unsigned long long acc2[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int jp = 0; jp < 4; ++jp) acc2[i][jp] = 0ULL;
#pragma unroll 4
  for (int k = 0; k < W2; ++k) {
    const float4 x0 = *reinterpret_cast<const float4*>(L + k * LDL);
    const float4 x1 = *reinterpret_cast<const float4*>(L + k * LDL + 16);
    const float4 u0 = *reinterpret_cast<const float4*>(R + k * LDR);
    const float4 u1 = *reinterpret_cast<const float4*>(R + k * LDR + 16);
    const float xa[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
    const unsigned long long up[4] = {pk2(u0.x, u0.y), pk2(u0.z, u0.w), pk2(u1.x, u1.y), pk2(u1.z, u1.w)};
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const unsigned long long xx = pk2(xa[i], xa[i]);
#pragma unroll
      for (int jp = 0; jp < 4; ++jp) fma2(acc2[i][jp], xx, up[jp]);
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int jp = 0; jp < 4; ++jp) unpk2(acc2[i][jp], acc[i][2 * jp], acc[i][2 * jp + 1]);
}

// Tile t of the queue: A's first (row groups gx >= Q / 4 of column Q; the
// larger ones, so that the end is of small ones), then V's.
struct PipeTile {
  int gx, Q;
  bool both;  // A <- U~^T A U~
};
__host__ __device__ inline int pipe_before(int gxn, int grp) { return 4 * grp * gxn - 2 * grp * (grp - 1); }
__host__ __device__ inline int pipe_tiles_a(int npairs) {  // column groups of 4: gxn - group tiles per column
  const int gxn = (npairs + 3) / 4;
  return pipe_before(gxn, gxn) - (4 * gxn - npairs);
}
__host__ __device__ inline int pipe_tiles_v(int npairs) { return npairs * ((npairs + 3) / 4); }
__host__ __device__ inline PipeTile pipe_tile(int npairs, int t) {
  const int gxn = (npairs + 3) / 4, ta = pipe_tiles_a(npairs);
  if (t >= ta) return {(t - ta) % gxn, (t - ta) / gxn, false};
  // the group: largest grp with pipe_before(grp) <= t
  const float b = 2.0f * gxn + 1.0f;
  int grp = (int)(0.5f * (b - sqrtf(fmaxf(b * b - 2.0f * t, 0.0f))));
  grp = grp < 0 ? 0 : grp >= gxn ? gxn - 1 : grp;
  while (grp > 0 && pipe_before(gxn, grp) > t) --grp;
  while (grp + 1 < gxn && pipe_before(gxn, grp + 1) <= t) ++grp;
  const int rest = t - pipe_before(gxn, grp);
  return {grp + rest % (gxn - grp), 4 * grp + rest / (gxn - grp), true};
}

// Tiles first .. end - 1 of the queue (VONLY: all of them V's; half the shared
// memory).  queue[0]: tiles handed out beyond the first gridDim.x, queue[1]:
// CTAs done; both 0 before and after.
template <bool VONLY>
__global__ void __launch_bounds__(PT, VONLY ? 5 : 3) rmul32_pipe(float* A32, float* V32, int N, int nb, int R,
                                                     const float* __restrict__ Sbuf, const float* __restrict__ Ubuf,
                                                     bool hq, int first, int end, unsigned* queue) {
  extern __shared__ __align__(16) unsigned char pipe_raw[];
  PipeStage<VONLY>* st = reinterpret_cast<PipeStage<VONLY>*>(pipe_raw);
  __shared__ int slot[2];
  const int tid = threadIdx.x, npairs = nb / 2;
  const int w = tid >> 4, g = tid & 3, h = (tid >> 2) & 3;
  pdl_wait();
  auto fetch = [&](PipeStage<VONLY>& p, int t) {
    if (t < end) {
      PipeTile q = pipe_tile(npairs, t);
      if (VONLY) q.both = false;
      int I, J, IQ, JQ;
      block_pair(nb, R, q.Q, IQ, JQ);
      // X_Q(r, k) = X[g_Q(k) N + row(r)]: rows 4 (t mod 32) .. +3, k = t / 32 + 2 i
      const int rq = tid & 31, ar = 4 * q.gx + (rq >> 3);
      const bool valid = ar < npairs && (!q.both || ar > q.Q);
      block_pair(nb, R, valid ? ar : q.Q, I, J);
      const float* x = (q.both ? A32 : V32) + gidx(I, J, (4 * rq) & 31);
#pragma unroll
      for (int i = 0; i < W2 / 2; ++i) {
        const int k = (tid >> 5) + 2 * i;
        cp16(&p.X[k][4 * rq], x + (size_t)gidx(IQ, JQ, k) * N, valid);
      }
      const float* u = Ubuf + (size_t)q.Q * W2 * W2 + 4 * tid;
#pragma unroll
      for (int i = 0; i < 4; ++i) cp16(&p.U[0][0] + 4 * tid + 256 * i, u + 256 * i, true);
      if constexpr (!VONLY) {
        if (q.both)
          for (int j = 0; j < 4; ++j) {
            const int a = 4 * q.gx + j;
            if (a <= q.Q || a >= npairs) continue;
            const float* ua = Ubuf + (size_t)a * W2 * W2 + 4 * tid;
#pragma unroll
            for (int i = 0; i < 4; ++i) cp16(&p.Ua[j][0][0] + 4 * tid + 256 * i, ua + 256 * i, true);
          }
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  int t = first + blockIdx.x;
  fetch(st[0], t);
  if (tid == 0) slot[1] = first + gridDim.x + atomicAdd(queue, 1u);
  __syncthreads();
  for (int it = 0; t < end; ++it) {
    const int next = slot[(it + 1) & 1];
    unsigned after = 0;
    if (tid == 0 && next < end) after = atomicAdd(queue, 1u);
    fetch(st[(it + 1) & 1], next);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    PipeStage<VONLY>& p = st[it & 1];
    PipeTile q = pipe_tile(npairs, t);
    if (VONLY) q.both = false;
    const int a = 4 * q.gx + w, aw = 4 * q.gx + 2 * (tid >> 5);  // this half-warp's block pair, the warp's first
    if (aw < npairs && (!q.both || aw + 1 >= q.Q)) {
      float acc[8][8];
      half_mm32<XLD, W2>(&p.X[0][32 * w + 4 * g], &p.U[0][4 * h], acc);
      if constexpr (!VONLY) {
        if (q.both) {
          // T = X_Q U_Q in place of X_Q (T(i, c) at X[i][32 w + c]), then U_a^T T
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            float* d = &p.X[4 * g + (i & 3) + 4 * (i & 4)][32 * w + 4 * h];
            *reinterpret_cast<float4*>(d) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
            *reinterpret_cast<float4*>(d + 16) = make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]);
          }
          __syncwarp();
          half_mm32<W2, XLD>(&p.Ua[w][0][4 * g], &p.X[0][32 * w + 4 * h], acc);
        }
      }
      if (a < npairs && (!q.both || a >= q.Q)) {
        int I, J, IQ, JQ;
        block_pair(nb, R, a, I, J);
        block_pair(nb, R, q.Q, IQ, JQ);
        const int r0 = I * BS + 4 * g, r1 = J * BS + 4 * g, c0 = IQ * BS + 4 * h, c1 = JQ * BS + 4 * h;
        float* Y = q.both ? A32 : V32;
        if (q.both && a == q.Q) {
          // the diagonal tile: the solved subproblem
          const float* Sq = Sbuf + (size_t)q.Q * W2 * W2 + 4 * g;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float* c = Sq + W2 * (4 * h + (j & 3) + 4 * (j & 4));
            float* y = Y + (size_t)(j < 4 ? c0 + j : c1 + j - 4) * N;
            *reinterpret_cast<float4*>(y + r0) = *reinterpret_cast<const float4*>(c);
            *reinterpret_cast<float4*>(y + r1) = *reinterpret_cast<const float4*>(c + 16);
          }
        } else {
#pragma unroll
          for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] = qh(acc[i][j], hq);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            float* y = Y + (size_t)(j < 4 ? c0 + j : c1 + j - 4) * N;
            *reinterpret_cast<float4*>(y + r0) = make_float4(acc[0][j], acc[1][j], acc[2][j], acc[3][j]);
            *reinterpret_cast<float4*>(y + r1) = make_float4(acc[4][j], acc[5][j], acc[6][j], acc[7][j]);
          }
          if (q.both) {  // the mirror
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              float* y = Y + (size_t)(i < 4 ? r0 + i : r1 + i - 4) * N;
              *reinterpret_cast<float4*>(y + c0) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
              *reinterpret_cast<float4*>(y + c1) = make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]);
            }
          }
        }
      }
    }
    if (tid == 0) slot[it & 1] = next < end ? (int)(first + gridDim.x + after) : end;
    t = next;
    __syncthreads();
  }
  if (tid == 0 && atomicAdd(queue + 1, 1u) == gridDim.x - 1) {  // the last CTA: no one asks any more
    queue[0] = 0;
    queue[1] = 0;
  }
}

// A batch: the tiles of A <- U~^T A U~, then those of V <- V U~, per matrix.
MPJ_DEV int batch_tiles32(int np) { return 2 * ((np + 3) / 4) * np; }
__global__ void __launch_bounds__(RT) rmul32_batch(BatchShape b, int lo, int R, float* A32, float* V32,
                                                   const float* __restrict__ S, const float* __restrict__ U) {
  __shared__ Rmul32Smem<4> sm;
  pdl_wait();
  BatchTask t;
  if (!batch_find(b, lo, blockIdx.x, batch_tiles32, t)) return;
  const int np = t.N / W2, per = ((np + 3) / 4) * np, nb = t.N / BS;
  const float *Sm = S + (size_t)t.pair0 * W2 * W2, *Um = U + (size_t)t.pair0 * W2 * W2;
  if (t.local < per)
    rmul32_tile<R32_BOTH, false>(sm, A32 + t.el, A32 + t.el, t.N, nb, R, Sm, Um, false, false, nullptr, t.local / np,
                                 t.local % np);
  else
    rmul32_tile<R32_ALL, false>(sm, V32 + t.el, V32 + t.el, t.N, nb, R, Sm, Um, false, false, nullptr,
                                (t.local - per) / np, (t.local - per) % np);
}

}  // namespace

cudaError_t mpj_batch_stage1_round(const BatchShape& b, int R, float* A32, float* V32, float* S, float* U,
                                   cudaStream_t s) {
  const int lo = batch_lowest_class(R);
  const long long subs = batch_blocks(b, lo, [](int np) { return np; });
  if (subs == 0) return cudaSuccess;
  cudaError_t e = mpj_launch_pdl(solve32<false, BatchSub32>, dim3((unsigned)subs), dim3(S32_THREADS), 0, s,
                                 BatchSub32{b, lo, A32, S, U}, R, true);
  if (e != cudaSuccess) return e;
  const long long tiles = batch_blocks(b, lo, [](int np) { return 2 * ((np + 3) / 4) * np; });
  return mpj_launch_pdl(rmul32_batch, dim3((unsigned)tiles), dim3(RT), 0, s, b, lo, R, A32, V32, (const float*)S,
                        (const float*)U);
}

int mpj_stage1_padded(int n) { return ((n + W2 - 1) / W2) * W2; }

// A32, V32, two sets of the per-pair S and U (alternate rounds), the
// tensor-core update's transposed intermediate B^T, flag and queue words, two sets of
// the per-pair rotated-index masks, two of the saved tiles.
static int stage1_tensor_cores();

size_t mpj_stage1_bytes(int n) {
  size_t N = (size_t)mpj_stage1_padded(n);
  size_t nb = N / BS;
  return 3 * N * N * sizeof(float) + 6 * (nb / 2) * W2 * W2 * sizeof(float) + 4096 + 2 * (nb / 2) * sizeof(unsigned);
}

// MPJ_STAGE1_TC=1 runs the A update of each block round on the tcgen05
// tensor cores (3xTF32, two panel products, see tc32.cu) and the V update on
// the FP32 pipe.  Off by default: on GB300 at n = 4096 it is slower (600 vs
// 178 ms for the stage), and V must stay on the FP32 pipe because the tensor
// cores' FP32 accumulation drifts the column norms over thousands of products
// (||V^T V - I||_F 0.08 instead of 0.007).
static int stage1_tensor_cores() {
  static int env = -1;
  if (env < 0) {
    const char* e = getenv("MPJ_STAGE1_TC");
    env = (e && e[0] == '1') ? 1 : 0;
  }
  return env;
}


cudaError_t mpj_sumsq32(const float* A, int lda, int n, double* partial, double* out, cudaStream_t s);


namespace {
// One stage-1 sweep (nb - 1 block rounds) enqueued on stream s.
//
// The subproblems of round R + 1 do not wait for round R's update of A: their
// diagonal blocks come from round R's solved subproblems and their coupling
// blocks from tiles of A saved before that update (snap32).  So the chain of a
// sweep is the subproblems alone; A's updates (with the saving of tiles) and
// V's run on side streams (when given; in one launch, update_form), two rounds
// behind at most: round R's subproblems wait for the tiles saved after round
// R - 2's update, which also frees the S, U and T sets that alternate between
// rounds, and for V's update of round R - 2.  The streams are joined into s at
// the end.  Before, a round was the subproblems, then A's update: n = 96 25 us a
// round, now 20; n = 300 20.6, now 16.5; n = 1024 20.0, now 15.7 (the
// subproblems alone 12.5).
struct Stage1Bufs {
  int N, nb;
  float *A32, *V32, *Sb[2], *Ub[2], *Tb[2], *Bt;
  unsigned* tflag;  // word 0: flags of the tensor-core update; from 8, 16: rmul32_pipe's queues
  unsigned* Mb[2];  // per-pair rotated-index masks, by round parity
  bool half;
  bool sparse;  // products over the rotated indices only (masked kernels)
  int tc;
};

// The side streams and events of a sweep; joined into the owner stream on every
// exit (owner = null: the caller has joined them, e.g. inside a captured graph).
struct SweepStreams {
  cudaStream_t owner = nullptr, sa = nullptr, sv = nullptr;
  cudaEvent_t solved[2] = {nullptr, nullptr}, a[2] = {nullptr, nullptr}, v[2] = {nullptr, nullptr};
  bool ok = true;
  explicit SweepStreams(cudaStream_t s) : owner(s) {
    ok = cudaStreamCreateWithFlags(&sa, cudaStreamNonBlocking) == cudaSuccess &&
         cudaStreamCreateWithFlags(&sv, cudaStreamNonBlocking) == cudaSuccess;
    for (cudaEvent_t* e : {&solved[0], &solved[1], &a[0], &a[1], &v[0], &v[1]})
      ok = ok && cudaEventCreateWithFlags(e, cudaEventDisableTiming) == cudaSuccess;
    if (!ok) (void)cudaGetLastError();
  }
  ~SweepStreams() {
    if (ok && owner) {
      if (cudaEventRecord(a[0], sa) == cudaSuccess) (void)cudaStreamWaitEvent(owner, a[0], 0);
      if (cudaEventRecord(v[0], sv) == cudaSuccess) (void)cudaStreamWaitEvent(owner, v[0], 0);
    }
    for (cudaEvent_t e : {solved[0], solved[1], a[0], a[1], v[0], v[1]})
      if (e) cudaEventDestroy(e);
    if (sv) cudaStreamDestroy(sv);
    if (sa) cudaStreamDestroy(sa);
  }
};

// How a round's updates run.  Microseconds per round (subproblems included)
// with rmul32 per matrix / both matrices in one rmul32_pipe / one rmul32_pipe
// each:
//   n    257   512   768   1024  1280  1536  2048  2560  2944  3072  4096  6144
//        17.2  16.2  15.6  19.8  18.9  22.3  27.0  37.1  44.9  47.7  82.2  171
//        16.5  15.4  15.6  15.7  19.4  22.4  31.5  44.1        58.2  97.0
//                          15.7  21.4  25.5  32.7  39.2  45.7  46.6  69.8  147
// One launch wins while all its tiles run at once, three CTAs per SM (a launch
// and a stream's events fewer per round); one launch each, V's tiles five CTAs
// per SM, once A's fill the SMs several times over (two per SM leave room for V's
// and for the next subproblems: three took 80 us at n = 4096).  In between the
// waves of rmul32's CTAs fit better around the subproblems.
enum { UPD_RMUL, UPD_ONE, UPD_EACH };
int update_form(const Stage1Bufs& b) {
  if (b.tc == 1 || b.sparse) return UPD_RMUL;
  const int np = b.nb / 2, ta = pipe_tiles_a(np), tv = pipe_tiles_v(np), sms = sm_count();
  return ta + tv <= 3 * sms ? UPD_ONE : 2 * ta >= 15 * sms ? UPD_EACH : UPD_RMUL;
}

template <bool VONLY>
cudaError_t pipe_attr() {
  return cudaFuncSetAttribute(rmul32_pipe<VONLY>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              2 * (int)sizeof(PipeStage<VONLY>));
}
template <bool VONLY>
cudaError_t pipe_launch(const Stage1Bufs& b, int R, const float* S, const float* U, int first, int end, int per_sm,
                        cudaStream_t s) {
  const int most = per_sm * sm_count();
  return mpj_launch_pdl(rmul32_pipe<VONLY>, dim3(end - first < most ? end - first : most), dim3(PT),
                        2 * sizeof(PipeStage<VONLY>), s, b.A32, b.V32, b.N, b.nb, R, S, U, b.half, first, end,
                        b.tflag + (VONLY ? 16 : 8));
}

// Kernels of one sweep.
long long stage1_sweep_launches(const Stage1Bufs& b) {
  const long long rounds = b.nb - 1;
  return b.tc == 1 ? 4 * rounds : (update_form(b) == UPD_ONE ? 2 : 3) * rounds + (rounds - 1);
}

cudaError_t stage1_sweep(const Stage1Bufs& b, cudaStream_t s, SweepStreams* side) {
  const int N = b.N, nb = b.nb, npairs = nb / 2, rounds = nb - 1;
  const dim3 g32((npairs + 3) / 4, npairs);
  const int form = update_form(b), ta = pipe_tiles_a(npairs), tv = pipe_tiles_v(npairs);
  const bool look = b.tc != 1;  // the tensor-core update transposes through Bt, in order
  cudaStream_t sa = side ? side->sa : s, sv = side ? side->sv : s;
  cudaError_t e = cudaSuccess;
#define S1_TRY(x)                    \
  do {                               \
    e = (x);                         \
    if (e != cudaSuccess) return e;  \
  } while (0)
  auto snap = [&](int R, cudaStream_t st) {
    return mpj_launch_pdl(snap32, dim3(npairs), dim3(256), 0, st, (const float*)b.A32, N, nb, R, b.Tb[R & 1]);
  };
  if (form != UPD_RMUL) {
    S1_TRY(pipe_attr<false>());
    S1_TRY(pipe_attr<true>());
  }
  if (look && rounds > 1) S1_TRY(snap(1, s));
  for (int R = 0; R < rounds; ++R) {
    const int par = R & 1;
    float *Sbuf = b.Sb[par], *Ubuf = b.Ub[par];
    if (side && R >= 2) {
      S1_TRY(cudaStreamWaitEvent(s, side->a[par], 0));
      if (form != UPD_ONE) S1_TRY(cudaStreamWaitEvent(s, side->v[par], 0));
    }
    unsigned* Mbuf = b.sparse ? b.Mb[par] : nullptr;
    const bool ahead = look && R > 0;
    S1_TRY(mpj_launch_pdl(b.half ? solve32<true, OneSub32> : solve32<false, OneSub32>, dim3(npairs), dim3(S32_THREADS),
                          0, s,
                          OneSub32{b.A32, N, nb, Sbuf, Ubuf, Mbuf, ahead ? b.Sb[par ^ 1] : nullptr, b.Ub[par ^ 1],
                                   b.Tb[par]},
                          R, b.tc != 1));
    if (side) {
      S1_TRY(cudaEventRecord(side->solved[par], s));
      S1_TRY(cudaStreamWaitEvent(sa, side->solved[par], 0));
      if (form != UPD_ONE) S1_TRY(cudaStreamWaitEvent(sv, side->solved[par], 0));
    }
    if (b.tc == 1) {
      // A' = U^T A U = (A U)^T U (A symmetric): B^T = (A U)^T, then
      // A' = (B^T)(:, I_q) U_q on the tensor cores; V U on the FP32 pipe
      S1_TRY(mpj_tc_panel(N, nb, R, Ubuf, b.A32, b.Bt, 1, nullptr, nullptr, b.tflag, s));
      S1_TRY(mpj_tc_panel(N, nb, R, Ubuf, b.Bt, b.A32, 0, nullptr, nullptr, b.tflag, s));
    } else {
      // A <- U~^T A U~ in one pass (tiles a > Q, mirrored; S on the diagonal)
      if (form == UPD_RMUL) {
        auto amul = b.sparse ? rmul32<R32_BOTH, true> : rmul32<R32_BOTH, false>;
        S1_TRY(mpj_launch_pdl(amul, g32, dim3(RT), 0, sa, (const float*)b.A32, b.A32, N, nb, R, (const float*)Sbuf,
                              (const float*)Ubuf, b.half, false, (const unsigned*)Mbuf));
      } else {
        S1_TRY(pipe_launch<false>(b, R, Sbuf, Ubuf, 0, form == UPD_ONE ? ta + tv : ta, form == UPD_ONE ? 3 : 2, sa));
      }
      if (R + 2 < rounds) S1_TRY(snap(R + 2, sa));
    }
    if (side) S1_TRY(cudaEventRecord(side->a[par], sa));
    if (form == UPD_ONE) continue;
    // V <- V U~
    if (form == UPD_EACH) {
      S1_TRY(pipe_launch<true>(b, R, Sbuf, Ubuf, ta, ta + tv, 5, sv));
    } else {
      auto vmul = b.sparse ? rmul32<R32_ALL, true> : rmul32<R32_ALL, false>;
      S1_TRY(mpj_launch_pdl(vmul, g32, dim3(RT), 0, sv, (const float*)b.V32, b.V32, N, nb, R, (const float*)Sbuf,
                            (const float*)Ubuf, b.half, b.tc == 1, (const unsigned*)Mbuf));
    }
    if (side) S1_TRY(cudaEventRecord(side->v[par], sv));
  }
  if (side)
    for (int par = 0; par < 2 && par < rounds; ++par) {
      S1_TRY(cudaStreamWaitEvent(s, side->a[par], 0));
      if (form != UPD_ONE) S1_TRY(cudaStreamWaitEvent(s, side->v[par], 0));
    }
#undef S1_TRY
  return cudaGetLastError();
}

// A sweep captured once as a CUDA graph (the fork to the side stream and the
// dependent launches become graph edges) and replayed for every sweep.  The
// kernels' arguments are the workspace addresses, so an executable graph is
// kept per (device, workspace, N, precision, update engine) and reused by
// later calls with the same workspace.
struct SweepGraph {
  int dev, N, tc;
  bool half, side, sparse;
  void* work;
  cudaGraphExec_t exec;
  long long launches;  // kernels in one sweep
  ~SweepGraph() {
    if (exec) cudaGraphExecDestroy(exec);
  }
};
// Shared ownership: an entry evicted by one thread stays valid for a solve
// that is replaying it on another.  The registry itself is never destroyed
// (no CUDA calls during static destruction at process exit).
std::mutex g_sweep_mu;
std::vector<std::shared_ptr<SweepGraph>>& sweep_registry() {
  static auto* r = new std::vector<std::shared_ptr<SweepGraph>>();
  return *r;
}
constexpr size_t kMaxSweepGraphs = 4;

bool sweep_graphs_enabled() {
  static int env = -1;
  if (env < 0) {
    const char* e = getenv("MPJ_STAGE1_GRAPH");
    env = (e && e[0] == '0') ? 0 : 1;
  }
  return env == 1;
}

// The executable graph of one sweep for these buffers (captured on first use),
// or null if capture is not possible (the sweep is then enqueued directly).
std::shared_ptr<SweepGraph> sweep_graph(const Stage1Bufs& b, void* work, bool use_side) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    (void)cudaGetLastError();
    return nullptr;
  }
  std::lock_guard<std::mutex> lock(g_sweep_mu);
  auto& reg = sweep_registry();
  for (const auto& g : reg)
    if (g->dev == dev && g->work == work && g->N == b.N && g->half == b.half && g->tc == b.tc && g->side == use_side &&
        g->sparse == b.sparse)
      return g;
  cudaStream_t cap = nullptr;
  if (cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking) != cudaSuccess) {
    (void)cudaGetLastError();
    return nullptr;
  }
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  cudaError_t e = cudaSuccess;
  const long long per = stage1_sweep_launches(b);
  {
    std::unique_ptr<SweepStreams> side;
    if (use_side) {
      side.reset(new SweepStreams(cap));
      if (!side->ok) e = cudaErrorUnknown;
      side->owner = nullptr;  // joined inside the captured sweep
    }
    if (e == cudaSuccess) e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
      const cudaError_t eq = stage1_sweep(b, cap, side.get());
      e = cudaStreamEndCapture(cap, &graph);
      if (eq != cudaSuccess) e = eq;
    }
  }
  if (e == cudaSuccess) mpj_count_launches(-per);  // captured, not launched
  if (e == cudaSuccess) e = cudaGraphInstantiate(&exec, graph, 0);
  if (graph) cudaGraphDestroy(graph);
  cudaStreamDestroy(cap);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    if (exec) cudaGraphExecDestroy(exec);
    return nullptr;
  }
  if (reg.size() >= kMaxSweepGraphs) reg.erase(reg.begin());
  auto g = std::make_shared<SweepGraph>();
  g->dev = dev;
  g->N = b.N;
  g->tc = b.tc;
  g->half = b.half;
  g->side = use_side;
  g->sparse = b.sparse;
  g->work = work;
  g->exec = exec;
  g->launches = per;
  reg.push_back(g);
  return g;
}
}  // namespace

int mpj_stage1_run(int n, const double* A, int lda, double* Ql, int ldq, double tol32, int max_sweeps, int* sweeps_out,
                   double* off_out, void* work, double* partial, double* dscal, cudaStream_t s, bool half,
                   bool sparse) {
  Stage1Bufs b;
  b.N = mpj_stage1_padded(n);
  b.nb = b.N / BS;
  const int N = b.N, nb = b.nb;
  b.A32 = (float*)work;
  b.V32 = b.A32 + (size_t)N * N;
  const size_t pset = (size_t)(nb / 2) * W2 * W2;
  b.Sb[0] = b.V32 + (size_t)N * N;
  b.Sb[1] = b.Sb[0] + pset;
  b.Ub[0] = b.Sb[1] + pset;
  b.Ub[1] = b.Ub[0] + pset;
  b.Bt = b.Ub[1] + pset;
  b.tflag = (unsigned*)(b.Bt + (size_t)N * N);
  b.Mb[0] = b.tflag + 64;
  b.Mb[1] = b.Mb[0] + nb / 2;
  b.Tb[0] = (float*)(((size_t)(b.Mb[1] + nb / 2) + 255) & ~(size_t)255);
  b.Tb[1] = b.Tb[0] + pset;
  b.half = half;
  b.sparse = sparse;
  b.tc = stage1_tensor_cores() && !half;
  float* A32 = b.A32;
  float* V32 = b.V32;
  MPJ_CUDA_TRY(cudaMemsetAsync(b.tflag, 0, 64 * sizeof(unsigned), s));
  init32<<<1024, 256, 0, s>>>(A, lda, n, N, A32, V32, half);
  mpj_count_launch();
  MPJ_CUDA_TRY(cudaGetLastError());
  double off2 = 0.0;
  MPJ_CUDA_TRY(mpj_sumsq32(A32, N, N, partial, dscal, s));
  MPJ_CUDA_TRY(cudaMemcpyAsync(&off2, dscal, sizeof(double), cudaMemcpyDeviceToHost, s));
  MPJ_CUDA_TRY(cudaStreamSynchronize(s));
  double off = sqrt(off2);
  int sweeps = 0, status = MPJ_OK;
  const bool use_side = mpj_v_overlap_enabled() && nb / 2 >= 2;
  std::shared_ptr<SweepGraph> graph;
  std::unique_ptr<SweepStreams> side;
  while (off > tol32) {
    if (sweeps >= max_sweeps) {
      status = MPJ_NOT_CONVERGED;
      break;
    }
    if (sweeps == 0 && sweep_graphs_enabled()) graph = sweep_graph(b, work, use_side);
    if (graph) {
      MPJ_CUDA_TRY(cudaGraphLaunch(graph->exec, s));
      mpj_count_launches(graph->launches);
    } else {
      if (use_side && !side) {
        side.reset(new SweepStreams(s));
        if (!side->ok) side.reset();
      }
      MPJ_CUDA_TRY(stage1_sweep(b, s, side.get()));
    }
    ++sweeps;
    MPJ_CUDA_TRY(mpj_sumsq32(A32, N, N, partial, dscal, s));
    unsigned tf = 0;
    MPJ_CUDA_TRY(cudaMemcpyAsync(&off2, dscal, sizeof(double), cudaMemcpyDeviceToHost, s));
    MPJ_CUDA_TRY(cudaMemcpyAsync(&tf, b.tflag, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
    MPJ_CUDA_TRY(cudaStreamSynchronize(s));
    if (tf & MPJ_FLAG_TIMEOUT) return MPJ_ETIMEOUT;
    off = sqrt(off2);
  }
  widen<<<1024, 256, 0, s>>>(V32, N, n, Ql, ldq);
  mpj_count_launch();
  MPJ_CUDA_TRY(cudaGetLastError());
  if (sweeps_out) *sweeps_out = sweeps;
  if (off_out) *off_out = off;
  return status;
}
