// batched_rounds.cu -- a batch of symmetric eigenproblems (sizes 1 .. 256)
// solved round by round: every launch does one round of one stage for all
// matrices at once, with the kernels of the single-matrix solve (Algorithm 9,
// Sec. 5.1, per matrix; the batch is not in the paper).
//
//   1. FP32 block round-robin sweeps until off(A32) <= n 2^-24 ||A||_F (cap 15);
//   2. two Newton-Schulz steps, 3. A_cond = Q_d^T (A Q_d), both as FP64-exact
//      products on the tensor cores;
//   4. FP64 block round-robin sweeps until off <= tol (cap 30, threshold
//      Jacobi), applied to the columns of Q_d directly;
//   5. W = sorted diagonal, Q = the rotated columns permuted.
// Matrices that have converged take no part in further sweeps (their blocks
// return at once); the host reads the number still active after each sweep.
//
// Why rounds and not one thread group per matrix: a group's scalar round-robin
// sweeps are n - 1 barrier-separated rounds on the FP64 pipe (2 FMA per clock
// and SM), bound by that pipe and by the latency of the rounds; here a sweep
// is at most 15 rounds whose subproblems of all matrices run side by side, and
// the FP64 work is on the tensor cores.  2048 matrices, n uniform in [8, 256]:
// 453 ms with one group per matrix, 125 ms here.  Small matrices do better in
// groups: see choose_group.
#include <string.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "batch.cuh"
#include "batched.cuh"

namespace {

constexpr int kMaxSweeps32 = 15, kMaxSweeps64 = 30, kNsSteps = 2;
constexpr size_t kChunkBytes = (size_t)6 << 30;  // workspace of the matrices solved together
constexpr int BT = 256;

// CTA sum in a fixed order
MPJ_DEV double cta_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  for (int w = 0; w < BT / 32; ++w) t += red[w];
  return t;
}

struct State {  // by place
  double* tol;       // FP64 stop
  double* tol32;     // stage-1 stop
  double* skip_abs;  // tol / n
  int* active;
  int* sweeps;
};

// ||A||_F, tolerances, A32 = fl32(A 2^-e) and V32 = I padded to N.  e = 0 unless
// ||A||_F is below 2^-24 or above 2^24: the FP32 sweeps compare squares of entries,
// which leave FP32's range for matrices of 1e-23 and 1e19 (entries themselves
// beyond 1e-38 and 1e38); e = log2 ||A||_F there.  The FP32 rotations do not depend
// on a power of two.
__global__ void __launch_bounds__(BT) batch_init(BatchShape b, const double* const* __restrict__ Aptr,
                                                 const int* __restrict__ order, double tol_in, float* __restrict__ A32,
                                                 float* __restrict__ V32, State st, unsigned* __restrict__ flags) {
  __shared__ double red[BT / 32];
  BatchTask t;
  if (!batch_find(b, 0, blockIdx.x, [](int) { return 1; }, t)) return;
  const int n = t.n, N = t.N;
  const double* A = Aptr[order[t.place]];
  double s = 0.0;
  bool bad = false;
  for (int e = threadIdx.x; e < N * N; e += BT) {
    const int i = e % N, j = e / N;
    const double x = (i < n && j < n) ? A[(size_t)j * n + i] : 0.0;
    if (!isfinite(x)) bad = true;
    s = fma(x, x, s);
    A32[t.el + e] = (float)x;
    V32[t.el + e] = i == j ? 1.0f : 0.0f;
  }
  if (bad) atomicOr(flags, MPJ_FLAG_NONFINITE);
  s = cta_sum(s, red);
  const double norm = sqrt(s);
  double scale = 1.0;
  if (norm > 0.0 && isfinite(norm) && (norm < 0x1p-24 || norm > 0x1p24)) {
    scale = __hiloint2double((2046 - ((__double2hiint(norm) >> 20) & 0x7FF)) << 20, 0);
    for (int e = threadIdx.x; e < N * N; e += BT) {
      const int i = e % N, j = e / N;
      if (i < n && j < n) A32[t.el + e] = (float)(A[(size_t)j * n + i] * scale);
    }
  }
  if (threadIdx.x == 0) {
    const double tol = tol_in > 0 ? tol_in : (double)n * 0x1p-53 * norm;
    st.tol[t.place] = tol;
    st.tol32[t.place] = (double)n * 0x1p-24 * (norm * scale);
    st.skip_abs[t.place] = tol / n;
    st.sweeps[t.place] = 0;
  }
}

// Which matrices still need a sweep: off(A) > tol (false for NaN); *count is
// their number.  `sweeps` (may be null) counts the sweep that follows.
template <typename T>
__global__ void __launch_bounds__(BT) batch_check(BatchShape b, const T* __restrict__ A, const double* __restrict__ tol,
                                                  int* __restrict__ active, int* __restrict__ sweeps, int last,
                                                  int* __restrict__ count) {
  __shared__ double red[BT / 32];
  BatchTask t;
  if (!batch_find(b, 0, blockIdx.x, [](int) { return 1; }, t)) return;
  const int N = t.N;
  const T* a = A + t.el;
  double s = 0.0;
  for (int e = threadIdx.x; e < N * N; e += BT) {
    const double x = (double)a[e];
    if (e % (N + 1) != 0) s = fma(x, x, s);
  }
  s = cta_sum(s, red);
  if (threadIdx.x == 0) {
    const double lim = tol[t.place];
    const int on = t.n > 1 && s > lim * lim;
    active[t.place] = on;
    if (on) {
      atomicAdd(count, 1);
      if (sweeps && !last) sweeps[t.place] += 1;
    }
  }
}

__global__ void batch_widen(const float* __restrict__ V32, double* __restrict__ X, long long count) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x)
    X[i] = (double)V32[i];
}

// W ascending, Q's columns permuted to match (ties by index)
__global__ void __launch_bounds__(BT) batch_final(BatchShape b, const double* __restrict__ A, const double* __restrict__ V,
                                                  const int* __restrict__ order, double* const* __restrict__ Wptr,
                                                  double* const* __restrict__ Qptr, const int* __restrict__ sweeps,
                                                  int* __restrict__ sweeps_out) {
  __shared__ double w[BATCH_NMAX];
  __shared__ int rank[BATCH_NMAX];
  BatchTask t;
  if (!batch_find(b, 0, blockIdx.x, [](int) { return 1; }, t)) return;
  const int n = t.n, N = t.N, idx = order[t.place];
  double* W = Wptr[idx];
  double* Q = Qptr[idx];
  for (int i = threadIdx.x; i < n; i += BT) w[i] = A[t.el + (long long)i * (N + 1)];
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += BT) {
    const double wi = w[i];
    int r = 0;
    for (int j = 0; j < n; ++j) r += (w[j] < wi) || (w[j] == wi && j < i);
    rank[i] = r;
    W[r] = wi;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < n * n; e += BT) {
    const int i = e % n, j = e / n;
    Q[(size_t)rank[j] * n + i] = V[t.el + (long long)j * N + i];
  }
  if (threadIdx.x == 0) sweeps_out[idx] = sweeps[t.place];
}

inline size_t al(size_t x) { return (x + 255) & ~(size_t)255; }

struct Chunk {
  int p0, count;  // places
  BatchShape shape;
  long long el, oz;
  int pairs, cmax;
};

// The workspace of a chunk: three FP64 matrices each, and one area used in turn
// by stage 1 (A32, V32, S, U), the products (two sliced operands) and the
// sweeps (B and the digit tiles).
struct Layout {
  size_t X, M, Y, area, total;
  size_t A32, V32, S, U, oz[2], ozx[2], B, digits;
};
Layout layout(const Chunk& c) {
  Layout L;
  const size_t sq = al((size_t)c.el * sizeof(double)), sf = al((size_t)c.el * sizeof(float));
  const size_t su = al((size_t)c.pairs * 1024 * sizeof(float));
  const size_t ozs = al((size_t)c.oz * 2), ozx = al((size_t)c.count * BATCH_NMAX * sizeof(int));
  L.X = 0;
  L.M = sq;
  L.Y = 2 * sq;
  L.area = 3 * sq;
  L.A32 = L.area;
  L.V32 = L.A32 + sf;
  L.S = L.V32 + sf;
  L.U = L.S + su;
  L.oz[0] = L.area;
  L.ozx[0] = L.oz[0] + ozs;
  L.oz[1] = L.ozx[0] + ozx;
  L.ozx[1] = L.oz[1] + ozs;
  L.B = L.area;
  L.digits = L.B + sq;
  size_t end = L.U + su;
  if (L.ozx[1] + ozx > end) end = L.ozx[1] + ozx;
  if (L.digits + al(mpj_batch_digit_bytes(c.pairs)) > end) end = L.digits + al(mpj_batch_digit_bytes(c.pairs));
  L.total = end;
  return L;
}

// How a list of sizes is solved: places by decreasing size, cut into chunks.
struct Plan {
  std::vector<int> sizes, order, n_place;
  std::vector<Chunk> chunks;
  size_t work = 0;         // bytes of the largest chunk
  int group = 0, grid = 0; // one thread group of that size per matrix instead, in so many CTAs
};
// What a device keeps between calls, which run one after the other: the last
// plan, and memory grown to the largest one so far (a workspace of at most
// kChunkBytes or one matrix, and some words per matrix).  Calls with changing
// lists of sizes plan again on the host but allocate nothing once it is grown.
struct Device {
  int id = -1;
  Plan plan;
  bool uploaded = false;  // plan.order and plan.n_place are in `small`
  void *work = nullptr, *small = nullptr;
  int* pinned = nullptr;  // count, flags, then the sweeps by matrix
  size_t work_bytes = 0, small_bytes = 0, pinned_bytes = 0;
};
std::mutex g_mu;
std::vector<Device*>& devices() {  // never destroyed (no CUDA calls at process exit)
  static auto* d = new std::vector<Device*>();
  return *d;
}

void give_back(Device* d) {
  if (d->work) cudaFree(d->work);
  if (d->small) cudaFree(d->small);
  if (d->pinned) cudaFreeHost(d->pinned);
  delete d;
}

// *p of at least `need` bytes; what it held is lost when it has to grow.
template <class Alloc, class Free>
cudaError_t grow(void** p, size_t* have, size_t need, Alloc alloc, Free release) {
  if (*have >= need) return cudaSuccess;
  if (*p) release(*p);
  *p = nullptr;
  *have = 0;
  const cudaError_t e = alloc(p, need);
  mpj_count_alloc();
  if (e == cudaSuccess)
    *have = need;
  else
    (void)cudaGetLastError();
  return e;
}
cudaError_t grow_device(void** p, size_t* have, size_t need) {
  return grow(p, have, need, [](void** q, size_t b) { return cudaMalloc(q, b); }, [](void* q) { cudaFree(q); });
}

// The small area: order, n by place, then the state by place, then count, flags
// and the sweeps by matrix (copied to the pinned words in one piece).
struct Small {
  int *order, *n, *sweeps_out, *count;
  unsigned* flags;
  State st;
  size_t total;
};
Small small_ptrs(char* b, int batch) {
  Small s;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    char* p = b + o;
    o += al(bytes);
    return p;
  };
  s.order = (int*)take(sizeof(int) * (size_t)batch);
  s.n = (int*)take(sizeof(int) * (size_t)batch);
  s.st.active = (int*)take(sizeof(int) * (size_t)batch);
  s.st.sweeps = (int*)take(sizeof(int) * (size_t)batch);
  s.st.tol = (double*)take(sizeof(double) * (size_t)batch);
  s.st.tol32 = (double*)take(sizeof(double) * (size_t)batch);
  s.st.skip_abs = (double*)take(sizeof(double) * (size_t)batch);
  s.count = (int*)take(sizeof(int) * ((size_t)batch + 2));
  s.flags = (unsigned*)(s.count + 1);
  s.sweeps_out = s.count + 2;
  s.total = o;
  return s;
}

int class_of(int n) { return (n + 31) / 32 - 1; }

// Round by round (0) or one thread group per matrix (its threads), by an estimate
// of the milliseconds of each, for 152 SMs:
//   a group of G threads   a n + c n^3 per matrix, a = 0.018 .. 0.0195 (the rounds' latency, their
//                          work), as long as the slowest matrix and all of them
//                          over the resident groups take;
//   round by round         0.67 ms for one block pair per matrix and 0.36 for each
//                          class more, or 0.42 and 0.23 and for each matrix 2.2 us
//                          (n <= 32), 5.2 (n <= 64): a matrix is padded to whole
//                          classes.
// Batches with a matrix above n = 64 go by rounds: a group alone takes longer than
// they do.  Measured (ms; 256, 512, 1024 threads, rounds), the coefficients fitted
// to 110 such rows, the choice within 10 % of the best:
//   1 x 8         0.15  0.16  0.17   0.61     152 x 24      0.86  0.63  0.54   0.76
//   608 x 8       0.20  0.35  0.66   1.58     2048 x 24     3.19  4.08  7.00   5.08
//   2048 x 8      0.68  1.09  2.15   4.80     200 x [8,48]  2.73  2.21  1.49   1.36
//   1 x 32        0.72  0.70  0.72   0.68     608 x [8,48]  3.31  2.22  2.92   2.78
//   2048 x 32     4.76  5.99  9.69   5.12     2048 x [8,48] 4.46  6.07  9.43   7.67
//   1 x 48        1.87  1.64  1.54   0.96     2048 x [8,64] 8.33  10.4  14.7   8.80
//   2048 x 48     13.0  15.1  20.5   11.9     2048 x [8,96] 23.2  25.3  32.6   16.4
constexpr int kGroupMax = 64;
int choose_group(const std::vector<int>& n_place, int sms) {
  const int nmax = n_place.front(), cmax = class_of(nmax);
  if (nmax > kGroupMax) return 0;
  double work = 0.0;
  for (int n : n_place) work += n <= 32 ? 0.0022 : 0.0052;
  work *= 152.0 / sms;
  double best = std::max(0.67 + 0.36 * cmax, 0.42 + 0.23 * cmax + work);
  int form = 0;
  const struct {
    int threads;
    double a, c;
  } groups[3] = {{256, 0.018, 2.3e-5}, {512, 0.019, 1.1e-5}, {1024, 0.0195, 6e-6}};
  for (const auto& g : groups) {
    auto ms = [&](int n) { return g.a * n + g.c * n * n * n; };
    double sum = 0.0;
    for (int n : n_place) sum += ms(n);
    const double t = std::max(ms(nmax), sum / ((double)sms * (1024 / g.threads)));
    if (t < best) {
      best = t;
      form = g.threads;
    }
  }
  return form;
}

// The plan of a list of sizes with chunks of at most `limit` bytes (at least one
// matrix each).
void make_plan(int batch, const int* n_host, size_t limit, Plan* p) {
  p->sizes.assign(n_host, n_host + batch);
  p->order.resize(batch);
  p->n_place.resize(batch);
  p->chunks.clear();
  p->work = 0;
  // decreasing size class, then decreasing n (counting sort), ties by index
  int start[BATCH_NMAX + 1], cnt[BATCH_NMAX + 1] = {0};
  for (int i = 0; i < batch; ++i) cnt[n_host[i]]++;
  for (int v = BATCH_NMAX, acc = 0; v >= 1; --v) {
    start[v] = acc;
    acc += cnt[v];
  }
  for (int i = 0; i < batch; ++i) p->order[start[n_host[i]]++] = i;
  for (int i = 0; i < batch; ++i) p->n_place[i] = n_host[p->order[i]];
  const int sms = sm_count();
  p->group = choose_group(p->n_place, sms);
  if (p->group) {
    p->grid = sms;  // also for fewer matrices: they then spread over the SMs
    p->work = mpj_batched_groups_bytes(p->group, p->grid, p->n_place.front());
    return;
  }
  for (int p0 = 0; p0 < batch;) {
    Chunk c;
    memset(&c, 0, sizeof c);
    c.p0 = p0;
    c.cmax = class_of(p->n_place[p0]);
    int cls = -1;
    for (int i = p0; i < batch; ++i) {
      const int k = class_of(p->n_place[i]), N = 32 * (k + 1);
      Chunk d = c;
      d.count += 1;
      d.el += (long long)N * N;
      d.oz += 8LL * batch_rp(N) * N;
      d.pairs += k + 1;
      if (c.count > 0 && layout(d).total > limit) break;
      if (k != cls) {
        cls = k;
        d.shape.first[k] = i - p0;
        d.shape.el[k] = c.el;
        d.shape.pairs[k] = c.pairs;
        d.shape.oz[k] = c.oz;
      }
      d.shape.cnt[k] += 1;
      c = d;
    }
    const size_t t = layout(c).total;
    if (t > p->work) p->work = t;
    p->chunks.push_back(c);
    p0 += c.count;
  }
}

// The plan and its memory on the device.  Where the memory for chunks of
// kChunkBytes cannot be had, the batch is cut into smaller ones (until other
// sizes are planned or the memory is given back), down to the largest matrix alone.
int prepare(Device* d, int batch, const int* n_host, cudaStream_t s) {
  const bool same = (int)d->plan.sizes.size() == batch &&
                    memcmp(d->plan.sizes.data(), n_host, sizeof(int) * (size_t)batch) == 0;
  if (!same || !d->uploaded) {
    d->uploaded = false;
    cudaError_t e = cudaSuccess;
    for (size_t limit = kChunkBytes, last = ~(size_t)0;; limit = last / 2) {
      make_plan(batch, n_host, limit, &d->plan);
      if (d->plan.work >= last) break;  // one matrix needs that much
      last = d->plan.work;
      e = grow_device(&d->work, &d->work_bytes, last);
      if (e != cudaErrorMemoryAllocation) break;
    }
    const size_t small = small_ptrs(nullptr, batch).total, pinned = sizeof(int) * ((size_t)batch + 2);
    if (e == cudaSuccess) e = grow_device(&d->small, &d->small_bytes, small);
    if (e == cudaSuccess)
      e = grow((void**)&d->pinned, &d->pinned_bytes, pinned, [](void** q, size_t b) { return cudaMallocHost(q, b); },
               [](void* q) { cudaFreeHost(q); });
    if (e != cudaSuccess) {
      mpj_set_cuda_error(e, "batched plan allocation", __LINE__);
      return MPJ_ENOMEM;
    }
    const Small sm = small_ptrs((char*)d->small, batch);
    e = cudaMemcpyAsync(sm.order, d->plan.order.data(), sizeof(int) * (size_t)batch, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(sm.n, d->plan.n_place.data(), sizeof(int) * (size_t)batch, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
      mpj_set_cuda_error(e, "batched plan upload", __LINE__);
      return MPJ_ECUDA;
    }
    for (Chunk& c : d->plan.chunks) c.shape.n = sm.n + c.p0;
    d->uploaded = true;
  }
  return MPJ_OK;
}

// One chunk on stream s; *not_converged is set when a sweep cap was reached
// with a matrix above its tolerance.
int run_chunk(const Device& d, const Chunk& c, const double* const* A, double* const* W, double* const* Q, double tol,
              bool* not_converged, cudaStream_t s) {
  const Small sm0 = small_ptrs((char*)d.small, (int)d.plan.sizes.size());
  State st = sm0.st;
  st.active += c.p0;
  st.sweeps += c.p0;
  st.tol += c.p0;
  st.tol32 += c.p0;
  st.skip_abs += c.p0;
  const int* order = sm0.order + c.p0;
  const Layout L = layout(c);
  char* w = (char*)d.work;
  double *X = (double*)(w + L.X), *M = (double*)(w + L.M), *Y = (double*)(w + L.Y);
  float *A32 = (float*)(w + L.A32), *V32 = (float*)(w + L.V32), *S = (float*)(w + L.S), *U = (float*)(w + L.U);
  const BatchOperand o0{(__nv_bfloat16*)(w + L.oz[0]), (int*)(w + L.ozx[0])};
  const BatchOperand o1{(__nv_bfloat16*)(w + L.oz[1]), (int*)(w + L.ozx[1])};
  BatchShape all = c.shape, act = c.shape;
  all.active = nullptr;
  act.active = st.active;
  const int rounds = 2 * c.cmax + 1;
  int* h_count = d.pinned;
  // the number of matrices that need another sweep
  auto count = [&](auto check) -> cudaError_t {
    cudaError_t e = cudaMemsetAsync(sm0.count, 0, sizeof(int), s);
    if (e != cudaSuccess) return e;
    check();
    mpj_count_launch();
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(h_count, sm0.count, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    return e;
  };
  batch_init<<<c.count, BT, 0, s>>>(all, A, order, tol, A32, V32, st, sm0.flags);
  mpj_count_launch();
  MPJ_CUDA_TRY(cudaGetLastError());
  // 1. FP32 stage
  for (int sweep = 0;; ++sweep) {
    MPJ_CUDA_TRY(count([&] { batch_check<float><<<c.count, BT, 0, s>>>(all, A32, st.tol32, st.active, nullptr, 0, sm0.count); }));
    if (*h_count == 0 || sweep >= kMaxSweeps32) break;
    for (int R = 0; R < rounds; ++R) MPJ_CUDA_TRY(mpj_batch_stage1_round(act, R, A32, V32, S, U, s));
  }
  batch_widen<<<2048, BT, 0, s>>>(V32, X, c.el);
  mpj_count_launch();
  MPJ_CUDA_TRY(cudaGetLastError());
  // 2. Newton-Schulz: E = I - X^T X, X <- X + X E / 2
  for (int k = 0; k < kNsSteps; ++k) {
    MPJ_CUDA_TRY(mpj_batch_oz_prepare(all, X, nullptr, order, false, o0, s));
    MPJ_CUDA_TRY(mpj_batch_oz_gemm(all, o0, o0, -1.0, 0.0, nullptr, 1.0, M, true, sm0.flags, s));
    MPJ_CUDA_TRY(mpj_batch_oz_prepare(all, X, nullptr, order, true, o0, s));
    MPJ_CUDA_TRY(mpj_batch_oz_prepare(all, M, nullptr, order, false, o1, s));
    MPJ_CUDA_TRY(mpj_batch_oz_gemm(all, o0, o1, 0.5, 1.0, X, 0.0, Y, false, sm0.flags, s));
    double* t = X;
    X = Y;
    Y = t;
  }
  // 3. A_cond = Q_d^T (A Q_d)
  MPJ_CUDA_TRY(mpj_batch_oz_prepare(all, nullptr, A, order, true, o0, s));
  MPJ_CUDA_TRY(mpj_batch_oz_prepare(all, X, nullptr, order, false, o1, s));
  MPJ_CUDA_TRY(mpj_batch_oz_gemm(all, o0, o1, 1.0, 0.0, nullptr, 0.0, Y, false, sm0.flags, s));
  MPJ_CUDA_TRY(mpj_batch_oz_prepare(all, Y, nullptr, order, false, o0, s));
  MPJ_CUDA_TRY(mpj_batch_oz_gemm(all, o1, o0, 1.0, 0.0, nullptr, 0.0, M, true, sm0.flags, s));
  // 4. FP64 sweeps
  double* B = (double*)(w + L.B);
  for (int sweep = 0;; ++sweep) {
    const int last = sweep >= kMaxSweeps64;
    MPJ_CUDA_TRY(count([&] { batch_check<double><<<c.count, BT, 0, s>>>(all, M, st.tol, st.active, st.sweeps, last, sm0.count); }));
    if (*h_count == 0) break;
    if (last) {
      *not_converged = true;
      break;
    }
    for (int R = 0; R < rounds; ++R)
      MPJ_CUDA_TRY(mpj_batch_sweep64_round(act, R, M, X, B, st.skip_abs, w + L.digits, c.pairs, sm0.flags, s));
  }
  // 5. sorted eigenvalues, permuted vectors
  batch_final<<<c.count, BT, 0, s>>>(all, M, X, order, W, Q, st.sweeps, sm0.sweeps_out);
  mpj_count_launch();
  MPJ_CUDA_TRY(cudaGetLastError());
  return MPJ_OK;
}

}  // namespace

void mpj_batched_rounds_release() {
  std::lock_guard<std::mutex> lock(g_mu);
  for (Device* d : devices()) give_back(d);
  devices().clear();
}

int mpj_batched_rounds(int batch, const int* n_host, const double* const* A_dev, double* const* W_dev,
                       double* const* Q_dev, double tol, int* sweeps_host, cudaStream_t s) {
  int dev = 0;
  MPJ_CUDA_TRY(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lock(g_mu);  // a device's memory serves one call at a time
  Device* d = nullptr;
  for (Device* x : devices())
    if (x->id == dev) d = x;
  if (!d) {
    d = new Device;
    d->id = dev;
    devices().push_back(d);
  }
  int st = prepare(d, batch, n_host, s);
  if (st != MPJ_OK) return st;
  const Small sm = small_ptrs((char*)d->small, batch);
  MPJ_CUDA_TRY(cudaMemsetAsync(sm.count, 0, 2 * sizeof(int), s));  // and the flags
  bool not_converged = false;
  if (d->plan.group)
    MPJ_CUDA_TRY(mpj_batched_groups(d->plan.group, d->plan.grid, d->plan.n_place.front(), sm.order, sm.n, A_dev, W_dev,
                                    Q_dev, batch, tol, d->work, sm.count, sm.sweeps_out, sm.flags, s));
  for (const Chunk& c : d->plan.chunks) {
    st = run_chunk(*d, c, A_dev, W_dev, Q_dev, tol, &not_converged, s);
    if (st != MPJ_OK) break;
  }
  if (st != MPJ_OK) {
    (void)cudaStreamSynchronize(s);  // nothing of this call may still use the workspace
    return st;
  }
  MPJ_CUDA_TRY(cudaMemcpyAsync(d->pinned, sm.count, sizeof(int) * ((size_t)batch + 2), cudaMemcpyDeviceToHost, s));
  MPJ_CUDA_TRY(cudaStreamSynchronize(s));
  if (sweeps_host) memcpy(sweeps_host, d->pinned + 2, sizeof(int) * (size_t)batch);
  const unsigned flags = (unsigned)d->pinned[1];
  if (flags & MPJ_FLAG_NONFINITE) return MPJ_ENONFINITE;
  if (flags & MPJ_FLAG_TIMEOUT) return d->plan.group ? MPJ_NOT_CONVERGED : MPJ_ETIMEOUT;
  return not_converged ? MPJ_NOT_CONVERGED : MPJ_OK;
}
