// blocked64.cu -- FP64 Jacobi sweeps in block round-robin order with the
// block updates on the tcgen05 tensor cores (the block Jacobi procedure the
// paper names as further work, Ch. 6; the rotations themselves are the
// paper's Algorithm 2 with the skip test of Algorithm 4).
//
// Ordering: the padded index range [0, N) (N = n rounded up to a multiple of
// 32; indices >= n are inert) is cut into nb = N/16 blocks of 16.  A sweep is
// nb - 1 outer rounds of the circle method on blocks; in round R the nb/2
// disjoint block pairs P = (I, J) each run one inner round-robin sweep (31
// inner rounds of 16 disjoint pairs) over the 32 indices of I u J on their
// 32 x 32 diagonal subproblem A[P, P] in shared memory, accumulating U_P,
// which is then made orthogonal to FP64 precision (blk_solve).  This is the
// rotation sequence of the block round-robin ordering one rotation at a time:
// the subproblem's rotations depend only on its own entries, and the pairs of
// one round are disjoint.
// The rest of the matrix then receives the round's rotations as products
//   A <- U~^T A U~,  V <- V U~,   U~ = blockdiag(U_P) (in index-set order),
// run as three block-diagonal right multiplications, each panel
// Y[:, P] = X_P U_P with X_P one of
//   A[:, P]          (B = A U~),
//   B[P, :]^T        (C = B^T U~ = U~^T A U~ for symmetric A, written to A:
//                     only its lower triangle is formed, each entry also
//                     written to its mirror, so A stays exactly symmetric),
//   V[:, P]          (V <- V U~, in place).
//
// The right multiplication is FP64-accurate on the 16-bit tensor cores: each
// CTA takes 128 rows of X_P (K = 32 values each), finds each row's largest
// exponent e_r (max |x_rk| < 2^e_r), and cuts x_rk * 2^(56 - e_r), rounded to
// an integer (magnitude below 2^56; the rounding is below 2^(e_r - 57)), into
// seven signed digits of 8 bits (|d_0| <= 256, |d_i| <= 128, each exactly a
// binary16).  U_P's columns are cut the same way when the subproblem is solved.
// The digit products of levels L = i + j <= 6 (28 pairs) go to seven FP32
// accumulators in tensor memory; over K = 32 a level sum is an integer of
// magnitude at most (2 * 256 * 128 + 5 * 128^2) * 32 = 2^22.2.  Measured on
// this GPU: the tensor cores' FP32 accumulation of such integer sums is exact
// below 2^23 but not in [2^23, 2^24) (unsigned byte digits, whose level sums
// reach 2^23.8, lost accuracy), so every bound here is kept below 2^23.  The
// epilogue reads the level sums, forms Z = sum_L s_L 2^(8 (6 - L)) exactly in
// two 64-bit integers, rounds Z to FP64 once and scales by 2^(e_r + f_c - 64).
// Dropped levels (L >= 7) are below 2^-55 of max|x_r.| max|u_.c| per term.
#include <cuda_fp16.h>
#include <stdint.h>
#include <stdio.h>

#include "batch.cuh"
#include "common.cuh"
#include "jacobi64.cuh"

namespace {

constexpr int BS = 16;                 // block size
constexpr int W2 = 32;                 // indices per block pair (K and N of the products)
constexpr int LDS = 33;                // padded shared-memory leading dimension
constexpr int NSL = 7;                 // 8-bit digits per value
constexpr int NLEV = 7;                // levels 0..6 kept
constexpr int TM = 128;                // rows per CTA of the right multiplication
constexpr uint32_t TMEM_COLS = 256;    // >= NLEV * 32
constexpr int USL_BYTES = W2 * W2 * 2;          // one 32 x 32 binary16 digit tile
constexpr int XSL_BYTES = TM * W2 * 2;          // one 128 x 32 binary16 digit tile
constexpr long long WAIT_CYCLES = 4000000000LL;

MPJ_DEV uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

MPJ_DEV int gidx(int I, int J, int l) { return l < BS ? I * BS + l : J * BS + (l - BS); }

MPJ_DEV void block_pair(int nb, int R, int slot, int& I, int& J) {
  int x, y;
  rr_slot(nb, R, slot, x, y);
  I = x < y ? x : y;
  J = x < y ? y : x;
}

// byte offset of (row, k), k in [0, 32), in a K-major tile of 8-row x 16-byte
// core matrices (k-adjacent cores 128 bytes apart, 8-row groups 512 apart)
MPJ_DEV int kmaj16(int row, int k) { return (((row >> 3) * 4 + (k >> 3)) << 7) + ((row & 7) << 4) + ((k & 7) << 1); }

// Seven signed digits of 8 bits of x on the grid 2^e (|x| < 2^e): x = sum_i d_i
// 2^(e - 8 (i + 1)) + r, |r| <= 2^(e - 57), |d_0| <= 256, |d_i| <= 128 (i >= 1).
// Y = |x| 2^(56 - e) rounded to an integer (half up; Y < 2^56); adding 128 to
// each of its six low bytes (one 64-bit add, carries included) makes byte j of
// the sum T d_(6-j) + 128 for centred digits d in [-128, 127], and the part
// above bit 48 d_0 in [0, 256].  Centred digits keep every level sum of the
// products below 2^23 (see the file comment).
constexpr unsigned long long DIGIT_BIAS = 0x0000808080808080ULL;
MPJ_DEV unsigned long long biased_digits(double x, int e) {
  const uint32_t xh = (uint32_t)__double2hiint(x), xl = (uint32_t)__double2loint(x);
  const int ex = (int)((xh >> 20) & 0x7FF);
  const uint32_t mh = (xh & 0xFFFFFu) | (ex ? 0x100000u : 0u);
  const int r = min(e + 1022 - max(ex, 1), 63);  // 2 Y = (mantissa 2^4) 2^-r, r >= 0
  const unsigned long long w = (((unsigned long long)mh << 32) | xl) << 4;
  return ((w >> r) + (1ULL + 2 * DIGIT_BIAS)) >> 1;  // rounding and bias in one add
}

// The digits of two values (T from biased_digits, the signs in bit 31 of s0,
// s1) as pairs of binary16 integers, first value in the low half.  A byte b
// becomes 1024 + b by its bit pattern, and one packed FMA gives sign (b - 128):
// three instructions for two digits, where FP32 patterns packed to bf16 took
// five.
MPJ_DEV void digit_pairs(unsigned long long T0, uint32_t s0, unsigned long long T1, uint32_t s1, uint32_t d[NSL]) {
  const uint32_t lo0 = (uint32_t)T0, hi0 = (uint32_t)(T0 >> 32), lo1 = (uint32_t)T1, hi1 = (uint32_t)(T1 >> 32);
  const uint32_t sg = ((s0 >> 16) & 0x8000u) | (s1 & 0x80000000u);
  const uint32_t one = 0x3C003C00u | sg, c128 = 0xE480E480u ^ sg, c0 = 0xE400E400u ^ sg;  // sign, -1152 sign, -1024 sign
  auto digit = [&](uint32_t v, uint32_t c) {
    uint32_t r;
    asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(v | 0x64006400u), "r"(one), "r"(c));
    return r;
  };
  d[6] = digit(__byte_perm(lo0, lo1, 0x0400) & 0x00FF00FFu, c128);
  d[5] = digit(__byte_perm(lo0, lo1, 0x0501) & 0x00FF00FFu, c128);
  d[4] = digit(__byte_perm(lo0, lo1, 0x0602) & 0x00FF00FFu, c128);
  d[3] = digit(__byte_perm(lo0, lo1, 0x0703) & 0x00FF00FFu, c128);
  d[2] = digit(__byte_perm(hi0, hi1, 0x0400) & 0x00FF00FFu, c128);
  d[1] = digit(__byte_perm(hi0, hi1, 0x0501) & 0x00FF00FFu, c128);
  d[0] = digit(__byte_perm(hi0, hi1, 0x7632), c0);
}

// Z 2^E rounded to the nearest double (ties to even), Z = hi 2^32 + lo with
// |Z| < 2^72, using integer instructions only.  Results outside the normal
// range go through ldexp (never for the operands of the sweeps).
MPJ_DEV double z_to_double(long long hi, long long lo, int E) {
  unsigned long long zl = ((unsigned long long)hi << 32) + (unsigned long long)lo;
  long long zh = (hi >> 32) + (lo >> 63) + (zl < (unsigned long long)lo ? 1 : 0);
  const unsigned long long sign = zh < 0 ? (1ULL << 63) : 0ULL;
  if (zh < 0) {  // |Z|
    zl = ~zl + 1ULL;
    zh = ~zh + (zl == 0 ? 1 : 0);
  }
  const unsigned long long h = (unsigned long long)zh;
  if (h == 0 && zl == 0) return __longlong_as_double((long long)sign);
  const int pos = h ? 127 - __clzll((long long)h) : 63 - __clzll((long long)zl);  // leading bit
  unsigned long long mant;
  if (pos <= 52) {
    mant = zl << (52 - pos);
  } else {
    const int sh = pos - 52;  // 1 .. 72
    unsigned long long lo_part, rnd, sticky;
    if (sh < 64) {
      mant = (zl >> sh) | (sh ? (h << (64 - sh)) : 0ULL);
      rnd = (zl >> (sh - 1)) & 1ULL;
      sticky = (sh >= 2) ? (zl & ((1ULL << (sh - 1)) - 1ULL)) : 0ULL;
    } else {
      mant = h >> (sh - 64);
      rnd = (sh == 64) ? (zl >> 63) : ((h >> (sh - 65)) & 1ULL);
      lo_part = (sh == 64) ? (zl & ((1ULL << 63) - 1ULL)) : (zl | (sh > 65 ? (h & ((1ULL << (sh - 65)) - 1ULL)) : 0ULL));
      sticky = lo_part;
    }
    mant &= (1ULL << 53) - 1ULL;
    if (rnd && (sticky || (mant & 1ULL))) ++mant;
  }
  int p2 = pos;
  if (mant >> 53) {
    mant >>= 1;
    ++p2;
  }
  const int biased = p2 + E + 1023;
  if (biased <= 0 || biased >= 2047) return ldexp(__longlong_as_double((long long)(sign | (1023ULL << 52) |
                                                                                   (mant & ((1ULL << 52) - 1ULL)))),
                                                 p2 + E);
  return __longlong_as_double((long long)(sign | ((unsigned long long)biased << 52) | (mant & ((1ULL << 52) - 1ULL))));
}

// ---------------------------------------------------------------- subproblems
// Pairs of FP32 values v = hi + lo (about 48 bits).  The subproblem's entries
// and U_P are held this way: an FP64 instruction takes 64 FP32 issue slots on
// this GPU, and only U_P leaves the subproblem, which is made orthogonal to
// FP64 precision (and 2^-60 in fixed point) before it is applied.
MPJ_DEV float2 df_norm(float hi, float lo) {  // |hi| >= |lo|
  const float s = __fadd_rn(hi, lo);
  return make_float2(s, __fsub_rn(lo, __fsub_rn(s, hi)));
}
// a * b as an unnormalised pair (relative error about 2^-47)
MPJ_DEV float2 df_mul(float2 a, float2 b) {
  const float p = __fmul_rn(a.x, b.x);
  float e = __fmaf_rn(a.x, b.x, -p);
  e = __fmaf_rn(a.x, b.y, e);
  e = __fmaf_rn(a.y, b.x, e);
  return make_float2(p, e);
}
MPJ_DEV float2 df_add(float2 a, float2 b) {
  const float s = __fadd_rn(a.x, b.x);
  const float bb = __fsub_rn(s, a.x);
  const float err = __fadd_rn(__fsub_rn(a.x, __fsub_rn(s, bb)), __fsub_rn(b.x, bb));
  return df_norm(s, __fadd_rn(err, __fadd_rn(a.y, b.y)));
}
MPJ_DEV float2 df_neg(float2 a) { return make_float2(-a.x, -a.y); }
// c x + s y
MPJ_DEV float2 df_rot(float2 c, float2 x, float2 s, float2 y) { return df_add(df_mul(c, x), df_mul(s, y)); }

// x 2^-eo as a pair (integer instructions): truncated to 24 bits, then the
// remaining 29 rounded; parts below the normal FP32 range become zero.
MPJ_DEV float2 df_split(double x, int eo) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7FF);
  if (ex == 0) return make_float2(0.0f, 0.0f);
  const unsigned long long m = (b & 0xFFFFFFFFFFFFFULL) | (1ULL << 52);
  const int k = ex - 1075 - eo;  // x 2^-eo = +- m 2^k
  const float sg = (b >> 63) ? -1.0f : 1.0f;
  const int kh = k + 29;
  const float h = kh >= -126 ? __int_as_float((min(kh, 127) + 127) << 23) : 0.0f;
  const float l = k >= -126 ? __int_as_float((min(k, 127) + 127) << 23) : 0.0f;
  return make_float2(sg * (float)(unsigned)(m >> 29) * h, sg * (float)(unsigned)(m & 0x1FFFFFFFULL) * l);
}

// Two values held as pairs (hi and lo parts packed two and two): the packed
// FP32 instructions do both with one issue slot.
struct Df2 {
  unsigned long long h, l;
};
MPJ_DEV unsigned long long pk(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
MPJ_DEV void unpk(unsigned long long v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
MPJ_DEV unsigned long long mul2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
MPJ_DEV unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
MPJ_DEV unsigned long long add2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
MPJ_DEV unsigned long long sub2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// Two rotations' coefficients for df2_rot: c, s and their negatives.
struct RotC {
  unsigned long long ch, cl, nch, sh, sl, nsh, nsl;
};
// c x + s y for two (x, y) (NEG: c x - s y); the products' errors are exact and
// enter the low parts, the leading parts are added with their error.
template <bool NEG>
MPJ_DEV Df2 df2_rot(const RotC& r, const Df2& x, const Df2& y) {
  const unsigned long long sh = NEG ? r.nsh : r.sh, nsh = NEG ? r.sh : r.nsh, sl = NEG ? r.nsl : r.sl;
  const unsigned long long np = mul2(r.nch, x.h), nq = mul2(nsh, y.h);  // minus the products
  const unsigned long long e = fma2(r.cl, x.h, fma2(r.ch, x.l, fma2(r.ch, x.h, np)));
  const unsigned long long f = fma2(sl, y.h, fma2(sh, y.l, fma2(sh, y.h, nq)));
  const unsigned long long n = add2(np, nq), bb = sub2(n, np);
  const unsigned long long er = add2(sub2(np, sub2(n, bb)), sub2(nq, bb));
  const unsigned long long lo = sub2(add2(e, f), er);
  Df2 o;
  o.h = sub2(lo, n);
  o.l = sub2(lo, add2(o.h, n));
  return o;
}

// Algorithm 2 on FP32 pairs for the slot's indices (x, y): coupling a, d =
// a_yy - a_xx, giving t (the root of a t^2 + d t - a with |t| <= 1, the sign of
// `tie` for d = 0), c = 1 / sqrt(1 + t^2) and s = t c.  From an FP32 seed t0,
// one Newton step with the residual formed in pairs gives t = t0 - dt to about
// 2^-44; c and s are formed at t0 in pairs beside it (c by one step from its
// own FP32 seed) and moved to t by their derivatives -t c^3 and c^3, which
// leaves dt^2.  (|a| < 2^-110 gives values that the caller does not use.)
MPJ_DEV void df_angle(float2 a, float2 d, float tie, float2& t, float2& c, float2& s) {
  const float tau = d.x * rcp_ftz(2.0f * a.x), at = fabsf(tau);
  const float den = at > 1e9f ? 2.0f * at : at + sqrt_ftz(fmaf(at, at, 1.0f));
  const float t0 = copysignf(rcp_ftz(den), tau == 0.0f ? tie : tau);
  // f = (a t0 + d) t0 - a, dt = f / (2 a t0 + d); the leading parts of f
  // cancel exactly (they agree to the seed's 2^-21)
  const float inv = rcp_ftz(fmaf(2.0f * a.x, t0, d.x));
  const float p = __fmul_rn(a.x, t0);
  const float pe = __fmaf_rn(a.y, t0, __fmaf_rn(a.x, t0, -p));
  const float g = __fadd_rn(p, d.x), bb = __fsub_rn(g, p);
  const float q = __fmul_rn(g, t0);
  const float ge = __fadd_rn(__fadd_rn(__fsub_rn(p, __fsub_rn(g, bb)), __fsub_rn(d.x, bb)), __fadd_rn(pe, d.y));
  const float qe = __fmaf_rn(ge, t0, __fmaf_rn(g, t0, -q));
  const float dt = __fadd_rn(__fsub_rn(q, a.x), __fsub_rn(qe, a.y)) * inv;
  // c at t0: e = 1 - (1 + t0^2) c0^2, c0 (1 + e / 2 + 3 e^2 / 8)
  const float c0 = rsqrt_ftz(fmaf(t0, t0, 1.0f));
  const float u = __fmul_rn(c0, c0), ue = __fmaf_rn(c0, c0, -u);
  const float t2 = __fmul_rn(t0, t0), wh = __fadd_rn(1.0f, t2);
  const float wl = __fadd_rn(__fsub_rn(t2, __fsub_rn(wh, 1.0f)), __fmaf_rn(t0, t0, -t2));
  const float2 m = df_mul(make_float2(wh, wl), make_float2(u, ue));
  const float e = __fsub_rn(__fsub_rn(1.0f, m.x), m.y);
  const float cc = c0 * fmaf(0.375f * e, e, 0.5f * e), c3 = c0 * u;
  // s at t0: t0 (c0 + cc)
  const float sp = __fmul_rn(t0, c0);
  const float se = __fmaf_rn(t0, cc, __fmaf_rn(t0, c0, -sp));
  const float co = __fmaf_rn(t0 * c3, dt, cc), so = __fmaf_rn(-c3, dt, se);
  c.x = __fadd_rn(c0, co);
  c.y = __fadd_rn(__fsub_rn(c0, c.x), co);
  s = df_norm(sp, so);
  t.x = __fsub_rn(t0, dt);
  t.y = __fsub_rn(__fsub_rn(t0, t.x), dt);
}

// One CTA per block pair of round R: one inner round-robin sweep (circle
// method, 31 rounds of 16 disjoint pairs, Algorithm 2 with the skip test of
// Algorithm 4) on the 32 x 32 subproblem, then one Newton-Schulz correction of
// U_P and U_P's columns cut into digits for the tensor products.  Writes per
// block pair: NSL digit tiles (32 x 32 binary16, K-major over the rows of U_P, one
// "row" per column of U_P), 32 column exponents, and whether any rotation
// happened (when none did, U_P = I and only that flag is written).
//
// Arithmetic.  The couplings and U_P are FP32 pairs, the couplings scaled by
// the power of two of the largest; the diagonal is the FP64 diagonal at the
// start plus a pair with its change, and a_qq - a_pp is formed from the FP64
// difference, so nearly equal diagonal entries keep their gap.  U_P comes out
// orthogonal to about 2^-43; in 60-bit fixed point E = U_P^T U_P - I is then
// formed exactly enough (2^-59) with integer products, and U_P - U_P E / 2 is
// orthogonal to 2^-59.  (The digits the products use have 2^-57.)  Entries
// whose range does not fit pairs (more than 2^70 between the couplings, or
// 2^100 between a coupling and the diagonal: graded matrices) run the same
// sweep in FP64 instructions instead (solve_wide).
//
// What bounds it: the chain coupling -> angle -> record -> next coupling, and
// beside it the number of instructions a warp has to get through per round.
// Positions instead of indices: slot k's x is at position k, its y at 31 - k,
// so a round rotates (k, 31 - k) and every address is a constant of the thread;
// moving on to the next round takes position p to p - 1 (0 to 30, 31 stays),
// done by writing the new values where they belong next.  The 16 couplings of
// the next round lie in blocks known in advance: warp 0 recomputes just those
// entries and the next round's rotations, eight warps update the 2 x 2 blocks
// (one row of a block per thread) and eight U_P (in registers, eight lanes per
// row).  The couplings alternate between two buffers, so one barrier per round
// is enough.  Three warps rest: they share warp 0's scheduler, and its
// instructions should not queue behind theirs.  In FP64 instructions the chain
// alone was about 60 dependent instructions of 65 cycles per round.  Measured
// at n = 4096 (128 CTAs): 101 us per launch in FP64, 34.8 us in pairs with two
// 288-thread roles and index arithmetic per round, 24.6 us in this form.
constexpr int SOLVE_THREADS = 640;
constexpr int SWEEP_THREADS = 17 * 32;  // warps 0 - 7, 9 - 11, 13 - 15, 17 - 19
constexpr int SSTR = 136;  // stride of the four entries' arrays (120 blocks; 64 bytes off a multiple of 128)
constexpr int UFL = 36;  // row stride of the fixed-point U (16-byte rows, conflict-free 16-byte reads)
struct SolveSmem {
  union {
    struct {
      float2 S[2][4 * SSTR];       // couplings by block, see pos_at
      float2 U[W2][LDS];           // U[column][row]
      float2 gap[W2 - 1][W2 / 2];  // starting a_yy - a_xx of each round's slots
    } p;
    struct {                      // FP64 form (solve_wide)
      double U[W2][LDS];          // U~[column][row]
      double cs[2][W2 / 2][2];    // mx, my
      double dg[2][W2 / 2][2];    // the pair's new true diagonal
      double d[W2], e[W2];        // scales and their reciprocals
      int p[2][W2 / 2], q[2][W2 / 2], rot[2][W2 / 2];
      int slot_of[2][W2];         // pair slot of each index in the round
    } w;
    struct {
      int u1[W2][UFL], u0[W2][UFL];  // U = (u1 + u0 2^-30) 2^-30, [column][row]
      float Ef[W2][UFL];             // E = U^T U - I
    } f;
  };
  double A[W2][LDS];      // the subproblem as loaded; FP64 form: in place
  float4 rec[2][W2 / 2];  // c, s oriented to the slot's (x, y)
  unsigned emax_off, emin_off, emax_dg, any;
};

// The packed coefficients of two rotations from their records (c, s as pairs).
MPJ_DEV RotC rot_coef(const float4& a, const float4& b) {
  return RotC{pk(a.x, b.x), pk(a.y, b.y), pk(-a.x, -b.x), pk(a.z, b.z), pk(a.w, b.w), pk(-a.z, -b.z), pk(-a.w, -b.w)};
}

// The barrier of the sweep's 17 warps.
MPJ_DEV void solve_barrier() { asm volatile("bar.sync 1, %0;\n" ::"n"(SWEEP_THREADS) : "memory"); }

// Position p of this round in the next one, and the position it came from.
MPJ_DEV int pos_next(int p) { return p == 31 ? 31 : p == 0 ? 30 : p - 1; }
MPJ_DEV int pos_prev(int p) { return p == 31 ? 31 : p == 30 ? 0 : p + 1; }
// Where the coupling of positions i and j (of different slots) is kept: one
// array per place in the 2 x 2 block (row x or y, column x or y), one element
// per block of slots a < b, so a warp reads its blocks without bank conflicts.
MPJ_DEV int pos_at(int i, int j) {
  const int si = i < 16 ? i : 31 - i, sj = j < 16 ? j : 31 - j;
  const int a = min(si, sj), b = max(si, sj), ea = si < sj ? i > 15 : j > 15, eb = si < sj ? j > 15 : i > 15;
  return (2 * ea + eb) * SSTR + (a * (31 - a)) / 2 + (b - a - 1);
}

// The same sweep in FP64 instructions on sm.A (both triangles), for entries whose
// range does not fit pairs; U_P into sm.w.U, sm.any set when a pair rotates.
// Scaled rotations: off the diagonal S = D S~ D and U = U~ D with one scale vector
// d (and e = 1 / d), the diagonal holds the true values, so a rotation (t, c) of
// pair p < q costs one FMA per entry and side:
//   x_p <- x_p - mx x_q,  x_q <- x_q + my x_p  (old values),
//   mx = t d_q / d_p,  my = t d_p / d_q,  d_p, d_q <- c d_p, c d_q.
// Warp 0 updates the blocks that hold a pair of the next round and forms that
// round's rotations while the other warps update the remaining blocks and U~: one
// barrier per inner round.  An FP64 instruction is 65 cycles here, so the length
// of warp 0's chain is the time.  Microseconds per round (with the products), n =
// 1024, D B D with D = 2^-60 .. 1: 125; with c - 1 carried, two FMAs an entry and
// side, divisions and roots and no looking ahead 145; this form with divisions and
// roots 138.  (Rounds of pairs: 50.)
MPJ_DEV void solve_wide(SolveSmem& sm, double skip, double skip_abs) {
  auto& w = sm.w;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int e = tid; e < W2 * W2; e += SOLVE_THREADS) w.U[e / W2][e % W2] = (e / W2 == e % W2) ? 1.0 : 0.0;
  if (tid < W2) w.d[tid] = w.e[tid] = 1.0;
  __syncthreads();
  // the rotation of the pair in slot k of inner round rho; the pair's scales are
  // updated here (no one else touches them this round)
  auto rotation = [&](int rho, int k, int buf) {
    int x, y;
    rr_slot(W2, rho, k, x, y);
    const int p = min(x, y), q = max(x, y);
    const double app = sm.A[p][p], aqq = sm.A[q][q], dp = w.d[p], dq = w.d[q], apq = sm.A[p][q] * dp * dq;
    double mx = 0.0, my = 0.0;
    const bool rot = above_skip(app, aqq, apq, skip) && fabs(apq) > skip_abs;
    if (rot) {
      double t, c;
      jacobi_angle(aqq - app, apq, t, c);
      const double h = fma(t, t, 1.0) * c, ep = w.e[p], eq = w.e[q];  // h = 1 / c
      mx = t * dq * ep;
      my = t * dp * eq;
      w.d[p] = dp * c;
      w.d[q] = dq * c;
      w.e[p] = ep * h;
      w.e[q] = eq * h;
      w.dg[buf][k][0] = app - t * apq;
      w.dg[buf][k][1] = aqq + t * apq;
      sm.any = 1u;
    }
    w.cs[buf][k][0] = mx;
    w.cs[buf][k][1] = my;
    w.rot[buf][k] = rot;
    w.p[buf][k] = p;
    w.q[buf][k] = q;
    w.slot_of[buf][p] = k;
    w.slot_of[buf][q] = k;
  };
  // the 2 x 2 block between slots a and b: rows by a's rotation, columns by b's,
  // the mirror block the same values
  auto block = [&](int a, int b, int buf) {
    if (!w.rot[buf][a] && !w.rot[buf][b]) return;
    const int pa = w.p[buf][a], qa = w.q[buf][a], pb = w.p[buf][b], qb = w.q[buf][b];
    const double mxa = w.cs[buf][a][0], mya = w.cs[buf][a][1], mxb = w.cs[buf][b][0], myb = w.cs[buf][b][1];
    const double b00 = sm.A[pa][pb], b01 = sm.A[pa][qb], b10 = sm.A[qa][pb], b11 = sm.A[qa][qb];
    const double t00 = fma(-mxa, b10, b00), t10 = fma(mya, b00, b10);
    const double t01 = fma(-mxa, b11, b01), t11 = fma(mya, b01, b11);
    sm.A[pa][pb] = sm.A[pb][pa] = fma(-mxb, t01, t00);
    sm.A[pa][qb] = sm.A[qb][pa] = fma(myb, t00, t01);
    sm.A[qa][pb] = sm.A[pb][qa] = fma(-mxb, t11, t10);
    sm.A[qa][qb] = sm.A[qb][qa] = fma(myb, t10, t11);
  };
  if (warp == 0 && lane < W2 / 2) rotation(0, lane, 0);
  __syncthreads();
#pragma unroll 1
  for (int rho = 0; rho < W2 - 1; ++rho) {
    const int cur = rho & 1;
    const bool more = rho + 1 < W2 - 1;
    if (warp == 0) {
      if (lane < W2 / 2) {  // the pairs' own blocks: new diagonal, no coupling
        if (w.rot[cur][lane]) {
          const int p = w.p[cur][lane], q = w.q[cur][lane];
          sm.A[p][p] = w.dg[cur][lane][0];
          sm.A[q][q] = w.dg[cur][lane][1];
          sm.A[p][q] = sm.A[q][p] = 0.0;
        }
      } else if (more) {  // the block that holds the next round's pair lane - 16
        int x, y;
        rr_slot(W2, rho + 1, lane - W2 / 2, x, y);
        if (w.slot_of[cur][x] > w.slot_of[cur][y]) {
          const int t = x;
          x = y;
          y = t;
        }
        const int a = w.slot_of[cur][x], b = w.slot_of[cur][y];
        // two next pairs may share a block: the smaller index of a takes it
        const int o = w.p[cur][a] == x ? w.q[cur][a] : w.p[cur][a];
        const bool twice = w.slot_of[cur][rr_partner(W2, rho + 1, o)] == b;
        if (a != b && (!twice || x < o)) block(a, b, cur);
      }
      __syncwarp();
      if (more && lane < W2 / 2) rotation(rho + 1, lane, cur ^ 1);
    } else {
      for (int task = tid - 32; task < 120 + (W2 / 2) * W2; task += SOLVE_THREADS - 32) {
        if (task < 120) {
          int a = 0, rem = task;
          while (rem >= 15 - a) {
            rem -= 15 - a;
            ++a;
          }
          const int b = a + 1 + rem;
          // a block that holds a pair of the next round is warp 0's
          if (more && (w.slot_of[cur][rr_partner(W2, rho + 1, w.p[cur][a])] == b ||
                       w.slot_of[cur][rr_partner(W2, rho + 1, w.q[cur][a])] == b))
            continue;
          block(a, b, cur);
        } else {
          const int k = (task - 120) / W2, j = (task - 120) % W2;
          if (!w.rot[cur][k]) continue;
          double &up = w.U[w.p[cur][k]][j], &uq = w.U[w.q[cur][k]][j];
          const double u0 = up, u1 = uq;
          up = fma(-w.cs[cur][k][0], u1, u0);
          uq = fma(w.cs[cur][k][1], u0, u1);
        }
      }
    }
    __syncthreads();
  }
  for (int e = tid; e < W2 * W2; e += SOLVE_THREADS) w.U[e / W2][e % W2] *= w.d[e / W2];
}

// One subproblem: pair P of round R of a matrix, and where its digits,
// exponents and flag go.
struct Sub64 {
  const double* A;
  int lda, n, nb, P;
  double skip_abs;
  __half* sl;
  int *ex, *rot;
  unsigned* nrot;
};
struct OneSub64 {  // the block pairs of one matrix
  const double* A;
  int lda, n, nb;
  double skip_abs;
  __half* sl;
  int *ex, *rot;
  unsigned* nrot;
  MPJ_DEV bool get(int bid, Sub64& v) const {
    v = Sub64{A, lda, n, nb, bid, skip_abs, sl + (size_t)bid * NSL * (USL_BYTES / 2), ex + bid * W2, rot + bid, nrot};
    return true;
  }
};
struct BatchSub64 {  // the block pairs of a batch
  BatchShape b;
  int lo;
  const double* A;
  const double* skip_abs;
  __half* sl;
  int *ex, *rot;
  MPJ_DEV bool get(int bid, Sub64& v) const {
    BatchTask t;
    if (!batch_find(b, lo, bid, [](int np) { return np; }, t)) return false;
    const int o = t.pair0 + t.local;
    v = Sub64{A + t.el, t.N, t.n, t.N / BS, t.local, skip_abs[t.place], sl + (size_t)o * NSL * (USL_BYTES / 2),
              ex + o * W2, rot + o, nullptr};
    return true;
  }
};
// CTAS: resident CTAs per SM the registers are limited for.  One (80 registers, 82
// in a batch) has the shorter latency and is taken when every subproblem of a round
// finds its own SM; beyond that two (48 registers, two of them spilled for a single
// matrix) have the higher rate: 16 against 21 us per subproblem and SM.
template <int CTAS, class Src>
__global__ void __launch_bounds__(SOLVE_THREADS, CTAS) blk_solve(Src src, int R, double skip) {
  __shared__ __align__(16) SolveSmem sm;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    sm.emax_off = 0u;
    sm.emin_off = 0xFFFFu;
    sm.emax_dg = 0u;
    sm.any = 0u;
  }
  __syncthreads();
  pdl_wait();
  Sub64 sub;
  if (!src.get(blockIdx.x, sub)) return;
  const double* __restrict__ A = sub.A;
  const int lda = sub.lda, n = sub.n;
  const double skip_abs = sub.skip_abs;
  int I, J;
  block_pair(sub.nb, R, sub.P, I, J);
  constexpr int NE = (W2 * W2 + SOLVE_THREADS - 1) / SOLVE_THREADS;
  double v0[NE];
  {
    unsigned mo = 0u, mn = 0xFFFFu, md = 0u, big = 0u;
#pragma unroll
    for (int it = 0; it < NE; ++it) {
      const int e = tid + it * SOLVE_THREADS, li = e % W2, lj = e / W2;
      v0[it] = 0.0;
      if (e >= W2 * W2) continue;
      const int gi = gidx(I, J, li), gj = gidx(I, J, lj);
      const double v = (gi < n && gj < n) ? A[(size_t)gj * lda + gi] : 0.0;
      v0[it] = v;
      sm.A[li][lj] = v;
      const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFULL;
      const unsigned ex = (unsigned)(b >> 52);
      if (li == lj) {
        md = max(md, ex);
      } else if (b != 0) {
        mo = max(mo, ex);
        mn = min(mn, ex);
        // |v| > skip_abs, as bit patterns
        if (b > (unsigned long long)__double_as_longlong(skip_abs)) big = 1u;
      }
    }
    mo = __reduce_max_sync(0xFFFFFFFFu, mo);
    mn = __reduce_min_sync(0xFFFFFFFFu, mn);
    md = __reduce_max_sync(0xFFFFFFFFu, md);
    big = __reduce_or_sync(0xFFFFFFFFu, big);
    if (lane == 0) {
      atomicMax(&sm.emax_off, mo);
      atomicMin(&sm.emin_off, mn);
      atomicMax(&sm.emax_dg, md);
      if (big) atomicOr(&sm.any, 1u);
    }
  }
  __syncthreads();
  if (!sm.any) {  // every coupling is zero or at most skip_abs: nothing rotates
    if (tid == 0) *sub.rot = 0;
    return;
  }
  const int emax_off = (int)sm.emax_off, emin_off = (int)sm.emin_off;
  const int etop = max(emax_off, (int)sm.emax_dg);
  const bool pairs = emin_off > 0 && emax_off - emin_off <= 70 && etop - emin_off <= 100 && etop < 2000;
  const int eo = emax_off - 1022;  // couplings scaled by 2^-eo: at most 1
  if (pairs) {
#pragma unroll
    for (int it = 0; it < NE; ++it) {
      const int e = tid + it * SOLVE_THREADS, li = e % W2, lj = e / W2;
      if (e >= W2 * W2) continue;
      if (li > lj && li + lj != 31) sm.p.S[0][pos_at(li, lj)] = df_split(v0[it], eo);
    }
    for (int e = tid; e < (W2 - 1) * (W2 / 2); e += SOLVE_THREADS) {
      int x, y;
      rr_slot(W2, e / (W2 / 2), e % (W2 / 2), x, y);
      sm.p.gap[e / (W2 / 2)][e % (W2 / 2)] = df_split(sm.A[y][y] - sm.A[x][x], eo);
    }
    __syncthreads();
    if (tid == 0) sm.any = 0u;  // read by all above; set again by warp 0
    if (warp == 0) {
      // skip_abs 2^-eo rounded to FP32 (infinite when it is beyond every
      // coupling), at least 2^-110: smaller couplings wait for a later sweep
      float sabs;
      {
        const int k = (int)(((unsigned long long)__double_as_longlong(skip_abs) >> 52) & 0x7FF) - 1023 - eo;
        sabs = skip_abs <= 0.0 ? 0.0f : k > 100 ? __int_as_float(0x7F800000) : k < -110 ? 0.0f : df_split(skip_abs, eo).x;
        sabs = fmaxf(sabs, 0x1p-110f);
      }
      const float skf = (float)skip;
      const int k = lane & 15;                // slot; lanes 16-31 repeat lanes 0-15
      float2 held = make_float2(0.0f, 0.0f);  // the slot's own coupling after its rotation
      float2 cx = held, cy = held;            // change of the slot's diagonal entries (scaled pairs)
      float dx = df_split(sm.A[k][k], eo).x, dy = df_split(sm.A[31 - k][31 - k], eo).x;  // the entries themselves
      bool mine = false;
      // rotation of the slot in round rho from its coupling a, d = a_yy - a_xx and the skip test's bound
      auto rotate = [&](int rho, float2 a, float2 d, float lim, int buf) {
        const bool rot = fabsf(a.x) > lim;
        const float tie = k == 0 || rho < k || rho > 30 - k ? 1.0f : -1.0f;  // x < y: '+'
        float2 t, c, s;
        df_angle(a, d, tie, t, c, s);
        mine |= rot;
        const float2 z = make_float2(0.0f, 0.0f);
        held = rot ? z : a;
        if (lane < W2 / 2) sm.rec[buf][k] = rot ? make_float4(c.x, c.y, s.x, s.y) : make_float4(1.0f, 0.0f, 0.0f, 0.0f);
        const float2 ta = rot ? df_mul(t, a) : z;
        cx = df_add(cx, df_neg(ta));
        cy = df_add(cy, ta);
        dx -= ta.x;
        dy += ta.x;
      };
      // the skip test's bound max(skip sqrt(|a_xx a_yy|), skip_abs)
      auto bound = [&]() { return fmaxf(skf * sqrt_ftz(fabsf(dx)) * sqrt_ftz(fabsf(dy)), sabs); };
      // the next round's slot k lies at positions (i, j) now
      const int i = pos_prev(k), j = pos_prev(31 - k), io = 31 - i, jo = 31 - j;
      const int a00 = pos_at(i, j), a01 = pos_at(i, jo), a10 = pos_at(io, j), a11 = pos_at(io, jo);
      const int own = pos_at(pos_next(k), pos_next(31 - k));
      const bool iy = i > 15, jy = j > 15;
      const int sa = iy ? io : i, sb = jy ? jo : j;
      rotate(0, df_split(sm.A[k][31 - k], eo), sm.p.gap[0][k], bound(), 0);
#pragma unroll 1
      for (int rho = 0; rho < W2 - 1; ++rho) {
        const int cur = rho & 1;
        const float2* Sc = sm.p.S[cur];
        // the diagonal entries of the next round's slot (two lanes on either side)
        {
          const float2 nx = make_float2(__shfl_down_sync(~0u, cx.x, 1, 16), __shfl_down_sync(~0u, cx.y, 1, 16));
          const float2 py = make_float2(__shfl_up_sync(~0u, cy.x, 1, 16), __shfl_up_sync(~0u, cy.y, 1, 16));
          const float2 x0 = make_float2(__shfl_sync(~0u, cx.x, 0, 16), __shfl_sync(~0u, cx.y, 0, 16));
          const float ndx = __shfl_down_sync(~0u, dx, 1, 16), pdy = __shfl_up_sync(~0u, dy, 1, 16);
          const float d0 = __shfl_sync(~0u, dx, 0, 16);
          cx = k == 15 ? cy : nx;
          dx = k == 15 ? dy : ndx;
          cy = k == 0 ? cy : k == 1 ? x0 : py;
          dy = k == 0 ? dy : k == 1 ? d0 : pdy;
        }
        const float2 d = df_add(sm.p.gap[min(rho + 1, W2 - 2)][k], df_add(cy, df_neg(cx)));
        const float lim = bound();
        const float2 h = held;
        __syncwarp();
        const float4 ra = sm.rec[cur][sa], rb = sm.rec[cur][sb];  // this warp's own writes
        const float2 ca = make_float2(ra.x, ra.y), cb = make_float2(rb.x, rb.y);
        const float2 ga = iy ? make_float2(ra.z, ra.w) : make_float2(-ra.z, -ra.w);
        const float2 gb = jy ? make_float2(rb.z, rb.w) : make_float2(-rb.z, -rb.w);
        solve_barrier();
        if (rho + 1 < W2 - 1) {
          const float2 t0 = df_rot(ca, Sc[a00], ga, Sc[a10]), t1 = df_rot(ca, Sc[a01], ga, Sc[a11]);
          rotate(rho + 1, df_rot(cb, t0, gb, t1), d, lim, cur ^ 1);
        }
        if (lane < W2 / 2) sm.p.S[cur ^ 1][own] = h;
      }
      if (mine) sm.any = 1u;
    } else if (warp < 4 || (warp > 4 && warp < 8) || warp == 9 || warp == 10) {
      // one row of the 2 x 2 block of slots ba < bb: position i (its other one io)
      const int w = warp < 4 ? warp - 1 : warp < 8 ? warp - 2 : warp - 3, side = lane & 1;
      int ba = 0, rem = w * 16 + (lane >> 1);
      const bool on = rem < 120;
      while (on && rem >= 15 - ba) {
        rem -= 15 - ba;
        ++ba;
      }
      const int bb = on ? ba + 1 + rem : 1;
      const int i = side ? 31 - ba : ba, io = 31 - i, jx = bb, jy = 31 - bb;
      const int i0 = pos_at(i, jx), i1 = pos_at(i, jy), o0 = pos_at(io, jx), o1 = pos_at(io, jy);
      const int w0 = pos_at(pos_next(i), pos_next(jx)), w1 = pos_at(pos_next(i), pos_next(jy));
      // couplings of the next round are left to warp 0
      const bool keep0 = on && pos_next(i) + pos_next(jx) != 31, keep1 = on && pos_next(i) + pos_next(jy) != 31;
#pragma unroll 2
      for (int rho = 0; rho < W2 - 1; ++rho) {
        const int cur = rho & 1;
        const float2* Sc = sm.p.S[cur];
        float2* Sn = sm.p.S[cur ^ 1];
        solve_barrier();
        const float4 ra = sm.rec[cur][ba], rb = sm.rec[cur][bb];
        const float2 v0 = Sc[i0], u0 = Sc[o0], v1 = Sc[i1], u1 = Sc[o1];
        const float2 ca = make_float2(ra.x, ra.y), cb = make_float2(rb.x, rb.y), gb = make_float2(rb.z, rb.w);
        const float2 ga = side ? make_float2(ra.z, ra.w) : make_float2(-ra.z, -ra.w);
        const float2 t0 = df_rot(ca, v0, ga, u0), t1 = df_rot(ca, v1, ga, u1);
        if (keep0) Sn[w0] = df_rot(cb, t0, df_neg(gb), t1);
        if (keep1) Sn[w1] = df_rot(cb, t1, gb, t0);
      }
    } else if (warp != 8 && warp != 12 && warp != 16) {
      // U_P in registers: eight lanes per row, lane e the columns at slots 2 e
      // and 2 e + 1.  The columns move with the positions: x_k <- x_(k+1), y_k
      // <- y_(k-1), x_15 <- y_15, y_1 <- x_0, and y_0 (index 31) stays.
      const int e = lane & 7, w = warp == 4 ? 0 : warp == 11 ? 1 : warp < 16 ? warp - 11 : warp - 12;
      const int row = w * 4 + (lane >> 3);
      float xh[2], xl[2], yh[2], yl[2];
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        xh[t] = 2 * e + t == row ? 1.0f : 0.0f;
        yh[t] = 31 - 2 * e - t == row ? 1.0f : 0.0f;
        xl[t] = yl[t] = 0.0f;
      }
      // one round behind: its records are loaded while the others work, not
      // in the burst of loads after the barrier
      solve_barrier();
      float4 r0 = sm.rec[0][2 * e], r1 = sm.rec[0][2 * e + 1];
#pragma unroll 2
      for (int rho = 0; rho < W2 - 1; ++rho) {
        if (rho + 1 < W2 - 1) solve_barrier();
        const RotC r = rot_coef(r0, r1);
        const Df2 ux{pk(xh[0], xh[1]), pk(xl[0], xl[1])}, uy{pk(yh[0], yh[1]), pk(yl[0], yl[1])};
        const Df2 nx = df2_rot<true>(r, ux, uy), ny = df2_rot<false>(r, uy, ux);
        float x0h, x0l, y0h, y0l, y1h, y1l;
        unpk(nx.h, x0h, xh[0]);  // the new x_0 is this round's x_1
        unpk(nx.l, x0l, xl[0]);
        unpk(ny.h, y0h, y1h);
        unpk(ny.l, y0l, y1l);
        const float nh = __shfl_down_sync(0xFFFFFFFFu, x0h, 1), nl = __shfl_down_sync(0xFFFFFFFFu, x0l, 1);
        const float ph = __shfl_up_sync(0xFFFFFFFFu, y1h, 1), pl = __shfl_up_sync(0xFFFFFFFFu, y1l, 1);
        xh[1] = e == 7 ? y1h : nh;
        xl[1] = e == 7 ? y1l : nl;
        yh[0] = e == 0 ? y0h : ph;
        yl[0] = e == 0 ? y0l : pl;
        yh[1] = e == 0 ? x0h : y0h;
        yl[1] = e == 0 ? x0l : y0l;
        if (rho + 1 < W2 - 1) {
          r0 = sm.rec[(rho + 1) & 1][2 * e];
          r1 = sm.rec[(rho + 1) & 1][2 * e + 1];
        }
      }
      // after 31 rounds the positions are the indices again
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        sm.p.U[2 * e + t][row] = make_float2(xh[t], xl[t]);
        sm.p.U[31 - 2 * e - t][row] = make_float2(yh[t], yl[t]);
      }
    }
  } else {
    __syncthreads();
    if (tid == 0) sm.any = 0u;  // read by all above
    solve_wide(sm, skip, skip_abs);
  }
  __syncthreads();
  if (!sm.any) {
    if (tid == 0) *sub.rot = 0;
    return;
  }
  // U_P in fixed point, U = (u1 + u0 2^-30) 2^-30 with u0 in [-2^29, 2^29]
  int u1[NE], u0[NE];
#pragma unroll
  for (int it = 0; it < NE; ++it) {
    const int e = tid + it * SOLVE_THREADS, row = e % W2, col = e / W2;
    u1[it] = u0[it] = 0;
    if (e >= W2 * W2) continue;
    if (pairs) {  // each part on the grid 2^-30, its exact remainder on 2^-60
      const float2 v = sm.p.U[col][row];
      const float xh = v.x * 0x1p30f, xl = v.y * 0x1p30f;
      const int ah = __float2int_rn(xh), al = __float2int_rn(xl);
      const int b = __float2int_rn((xh - (float)ah) * 0x1p30f) + __float2int_rn((xl - (float)al) * 0x1p30f);
      const int carry = (b + (1 << 29)) >> 30;  // |b| <= 2^30
      u1[it] = ah + al + carry;
      u0[it] = b - (carry << 30);
    } else {
      const long long F = __double2ll_rn(sm.w.U[col][row] * 0x1p60);
      const long long t = (F + (1LL << 29)) >> 30;
      u1[it] = (int)t;
      u0[it] = (int)(F - (t << 30));
    }
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < NE; ++it) {
    const int e = tid + it * SOLVE_THREADS;
    if (e < W2 * W2) {
      sm.f.u1[e / W2][e % W2] = u1[it];
      sm.f.u0[e / W2][e % W2] = u0[it];
    }
  }
  __syncthreads();
  // One Newton-Schulz step on U_P (Sec. 4.3.4): U <- U - U E / 2, E = U^T U - I.
  // U_P carries the rounding of its 496 rotations; applied to all of A and V
  // every round, that departure from orthogonality would accumulate over the
  // sweeps, so each U_P is made orthogonal first.  E (symmetric: the 528
  // entries i <= j, mirrored) from sums of integer products on the grid 2^-60:
  // sum u1 v1 modulo 2^32, which is enough because |E| < 2^-29 (the identity's
  // 2^60 vanishes), and the cross terms at weight 2^-30 (below 2^62.5); u0 v0
  // (below 2^-59 in all) is left out.
  for (int idx = tid; idx < 528; idx += SOLVE_THREADS) {
    int i = 0, rem = idx;
    while (rem >= W2 - i) {
      rem -= W2 - i;
      ++i;
    }
    const int j = i + rem;
    unsigned g = 0u;
    long long x = 0;
#pragma unroll
    for (int k = 0; k < W2; k += 4) {
      const int4 a1 = *reinterpret_cast<const int4*>(&sm.f.u1[i][k]), b1 = *reinterpret_cast<const int4*>(&sm.f.u1[j][k]);
      const int4 a0 = *reinterpret_cast<const int4*>(&sm.f.u0[i][k]), b0 = *reinterpret_cast<const int4*>(&sm.f.u0[j][k]);
      g += (unsigned)a1.x * (unsigned)b1.x + (unsigned)a1.y * (unsigned)b1.y + (unsigned)a1.z * (unsigned)b1.z +
           (unsigned)a1.w * (unsigned)b1.w;
      x += (long long)a1.x * b0.x + (long long)a1.y * b0.y + (long long)a1.z * b0.z + (long long)a1.w * b0.w;
      x += (long long)a0.x * b1.x + (long long)a0.y * b1.y + (long long)a0.z * b1.z + (long long)a0.w * b1.w;
    }
    // x 2^-30 taken out of g's grid first, so the small difference is exact
    const int gx = (int)(g + (unsigned)(x >> 30));
    const float ev = fmaf((float)(int)(x & 0x3FFFFFFF), 0x1p-90f, (float)gx * 0x1p-60f);
    sm.f.Ef[i][j] = ev;
    sm.f.Ef[j][i] = ev;
  }
  __syncthreads();
  // U E / 2 in FP32: |E| is about 2^-43, so its error is below 2^-65.  Warp w
  // takes columns w and w + 20; lane = row.
  {
    float ur[W2];
#pragma unroll
    for (int k = 0; k < W2; ++k) ur[k] = (float)sm.f.u1[k][lane];  // U(lane, k) 2^30
    long long Fn[2];
#pragma unroll
    for (int jj = 0; jj < 2; ++jj) {
      const int j = warp + 20 * jj;
      Fn[jj] = 0;
      if (j < W2) {
        float acc = 0.0f;
#pragma unroll
        for (int k = 0; k < W2; k += 4) {
          const float4 ev = *reinterpret_cast<const float4*>(&sm.f.Ef[j][k]);
          acc = fmaf(ur[k], ev.x, acc);
          acc = fmaf(ur[k + 1], ev.y, acc);
          acc = fmaf(ur[k + 2], ev.z, acc);
          acc = fmaf(ur[k + 3], ev.w, acc);
        }
        Fn[jj] = ((long long)sm.f.u1[j][lane] << 30) + sm.f.u0[j][lane] - __float2int_rn(acc * 0x1p29f);
      }
    }
    __syncthreads();
    long long* Fs = reinterpret_cast<long long*>(&sm.f);  // [column][row], row stride LDS
#pragma unroll
    for (int jj = 0; jj < 2; ++jj)
      if (warp + 20 * jj < W2) Fs[(warp + 20 * jj) * LDS + lane] = Fn[jj];
    __syncthreads();
  }
  // digits of U_P's columns: column c is "row" c of the right operand, over
  // k = row of U_P; eight threads per column, four values each
  __half* dst = sub.sl;
  if (tid < 8 * W2) {
    const long long* Fs = reinterpret_cast<const long long*>(&sm.f);
    const int c = tid >> 3, k0 = (tid & 7) * 4;
    long long v[4];
    unsigned long long top = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      v[j] = Fs[c * LDS + k0 + j];
      top |= (unsigned long long)(v[j] < 0 ? -v[j] : v[j]);  // same leading bit as the largest
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) top |= __shfl_xor_sync(0xffffffffu, top, o);
    const int bits = 64 - __clzll((long long)top);  // max|F| < 2^bits
    if ((tid & 7) == 0) sub.ex[c] = bits - 60;
    const int sh = bits - 56;  // Y = |F| 2^-sh rounded
    unsigned long long T[4];
    uint32_t neg[4], d[2][NSL];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const unsigned long long m = (unsigned long long)(v[j] < 0 ? -v[j] : v[j]);
      T[j] = (sh > 0 ? (m + (1ULL << (sh - 1))) >> sh : m << -sh) + DIGIT_BIAS;
      neg[j] = (uint32_t)((unsigned long long)v[j] >> 32);
    }
    digit_pairs(T[0], neg[0], T[1], neg[1], d[0]);
    digit_pairs(T[2], neg[2], T[3], neg[3], d[1]);
#pragma unroll
    for (int sl = 0; sl < NSL; ++sl)
      *reinterpret_cast<uint2*>(reinterpret_cast<char*>(dst + (size_t)sl * (USL_BYTES / 2)) + kmaj16(c, k0)) =
          make_uint2(d[0][sl], d[1][sl]);
  }
  if (tid == 0) {
    *sub.rot = 1;
    if (sub.nrot) atomicAdd(sub.nrot, 1u);
  }
}

// ---------------------------------------------------------------- right multiplication
MPJ_DEV uint64_t sdesc(uint32_t saddr) {
  // K-major, no swizzle: LBO = 128 bytes (k-adjacent cores), SBO = 512 bytes (8-row groups)
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)(512 >> 4) << 32) |
         ((uint64_t)1 << 46);
}

// kind::f16 instruction descriptor: D F32, A and B binary16, both K-major
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// One MMA.  A's use of the collector buffer: successive products with the same
// A tile read it from shared memory once (fill, use .., last) -- with N = 32 the
// 4 KB of A per product are what the tensor core waits for.
enum { A_ONCE = 0, A_FILL = 1, A_USE = 2, A_LAST = 3 };
template <int COLLECT>
MPJ_DEV void mma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
#define BLK_MMA(usage)                                                          \
  asm volatile(                                                                 \
      "{\n\t.reg .pred p;\n\t"                                                 \
      "setp.ne.b32 p, %4, 0;\n\t"                                              \
      "tcgen05.mma.cta_group::1.kind::f16" usage " [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d), \
      "l"(a), "l"(b), "r"(idesc), "r"(acc)                                      \
      : "memory")
  if (COLLECT == A_FILL)
    BLK_MMA(".collector::a::fill");
  else if (COLLECT == A_USE)
    BLK_MMA(".collector::a::use");
  else if (COLLECT == A_LAST)
    BLK_MMA(".collector::a::lastuse");
  else
    BLK_MMA("");
#undef BLK_MMA
}

// Waits up to about a microsecond in hardware for the phase of that parity.
MPJ_DEV bool mbar_try(uint32_t mbar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(mbar), "r"(parity), "r"(1000u)
      : "memory");
  return ok != 0;
}

struct __align__(1024) RmulSmem {
  unsigned char xs[NSL][XSL_BYTES];  // digits of the 128 x 32 tile of X_P
  unsigned char us[NSL][USL_BYTES];  // digits of U_P
  int uexp[W2];  // column exponent of U_P, shifted to a double's exponent field
  int rexp[TM];
  uint64_t mbar;
  uint32_t tmem;
};

enum { XMODE_COLS = 0, XMODE_ROWS = 1 };

// Y[r, g_Q(c)] = sum_k X_Q(r, k) U_Q(k, c) for block pair Q = blockIdx.y and
// the CTA's 128 rows r: the 32 indices of each of the block pairs
// a = 4 blockIdx.x .. +3 (rows 32 j .. +31 of the tile are pair 4 blockIdx.x + j,
// so epilogue warp w handles exactly pair 4 blockIdx.x + (w mod 4)).
// X_Q(r, k) = X[r + g_Q(k) ldx] (XMODE_COLS) or X[g_Q(k) + r ldx] (XMODE_ROWS).
// Y may alias X in XMODE_COLS (each CTA reads and writes only its own rows of
// its own panel).  Which tiles (a, Q) are formed:
//   TRI_ALL   every tile (V <- V U~);
//   TRI_FIRST tiles a <= Q (B = A U~: only the tiles the second step reads);
//   TRI_SECOND tiles a >= Q of C = B^T U~, written to Y and to the mirror
//             tile (Q, a); in the diagonal tile a = Q the entries on and below
//             the diagonal, mirrored.  So Y = U~^T A U~ stays exactly
//             symmetric, and the second step reads B only in tiles (Q, a),
//             Q <= a, the ones TRI_FIRST formed.
// 512 threads: thread t digitizes eight values, tile row t / 4 and quarter t mod
// 4 of the contraction index (two quarters per block I, J of Q); warp w reads
// the TMEM lanes of rows 32 (w mod 4) .. +31 and the 8 output columns
// 8 (w / 4) .. +7 of each level.
//
// What bounds it: instructions and their latency (DRAM 10 - 14 %, tensor pipe 5
// - 7 %), so both ends are counted.  Per value the digits take one shift, one
// add and 1.5 instructions per digit (digit_pairs); per output the level sums
// become integers by one FP32 add each (the conversion instruction issues at
// an eighth of that rate), two shift-adds and two 64-bit multiply-adds place
// them in the mantissas of two doubles with a fixed leading bit, and two FP64
// adds remove it and round (the integer normalisation they replace took some
// 30 instructions).  32 warps per SM hide what latency remains.
// Measured at n = 4096, all block pairs rotating: V U~ 187 -> 139 us, A U~
// 111 -> 81 us, B^T U~ 147 -> 96 us (its mirror also written in 64-byte runs);
// of that 3 % from reading each A tile into the tensor core once and from
// waiting for the products in hardware instead of polling.
constexpr int RM_THREADS = 512;
constexpr int QK = 8;  // values per thread
enum { TRI_ALL = 0, TRI_FIRST = 1, TRI_SECOND = 2 };

// The 8 values X_Q(row, k), k = g0 .. g0 + 7 (half of block I or J of Q); zeros
// for row < 0 (no such block pair or a tile that is not formed), row >= n, or
// indices >= n.
MPJ_DEV void load_xrow(const double* X, int ldx, int xmode, int n, int row, int g0, double x[QK]) {
  if (row < 0) {
#pragma unroll
    for (int k = 0; k < QK; ++k) x[k] = 0.0;
  } else if (xmode == XMODE_COLS) {
#pragma unroll
    for (int k = 0; k < QK; ++k) x[k] = (row < n && g0 + k < n) ? X[(size_t)(g0 + k) * ldx + row] : 0.0;
  } else if (row < n && g0 + QK <= n && ((((size_t)row * ldx + g0) & 1) == 0)) {
    const double2* src = reinterpret_cast<const double2*>(X + (size_t)row * ldx + g0);
#pragma unroll
    for (int k = 0; k < QK / 2; ++k) {
      const double2 v = src[k];
      x[2 * k] = v.x;
      x[2 * k + 1] = v.y;
    }
  } else {
#pragma unroll
    for (int k = 0; k < QK; ++k) x[k] = (row < n && g0 + k < n) ? X[(size_t)row * ldx + g0 + k] : 0.0;
  }
}

// the global index of tile row rl (pair 4 gx + rl / 32, index rl mod 32), or
// -1 when that pair does not exist
MPJ_DEV int tile_row(int nb, int R, int gx, int rl) {
  const int a = 4 * gx + (rl >> 5);
  if (a >= nb / 2) return -1;
  int I, J;
  block_pair(nb, R, a, I, J);
  return gidx(I, J, rl & 31);
}

MPJ_DEV bool tile_needed(int tri, int a, int Q) {
  return tri == TRI_ALL || (tri == TRI_FIRST ? a <= Q : a >= Q);
}

MPJ_DEV void blk_rmul_tile(const double* X, int ldx, int xmode, double* Y, int ldy, int n, int nb, int R,
                           const __half* __restrict__ Usl, const int* __restrict__ Uexp,
                           const int* __restrict__ rotated, unsigned* __restrict__ flags, int tri, int gx, int Q) {
  extern __shared__ __align__(1024) unsigned char dsm_raw[];
  RmulSmem& sm = *reinterpret_cast<RmulSmem*>(dsm_raw + ((1024 - (smem_u32(dsm_raw) & 1023)) & 1023));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int a0 = 4 * gx, a1 = min(4 * gx + 3, nb / 2 - 1);
  if (tri == TRI_FIRST && a0 > Q) return;
  if (tri == TRI_SECOND && a1 < Q) return;
  int I, J;
  block_pair(nb, R, Q, I, J);
  if (!rotated[Q]) {
    // no rotation in this block pair: U_Q = I exactly, Y_Q = X_Q (nothing to
    // do in place).  For A, a tile between two block pairs without rotations
    // keeps its values: the second step leaves it alone, so the first need not
    // copy it to B.
    if (X == Y && xmode == XMODE_COLS) return;
    const int rl = tid >> 2, qk = tid & 3;
    const int a = a0 + (rl >> 5);
    const int row = tile_row(nb, R, gx, rl);
    const int g0 = (qk & 2 ? J : I) * BS + QK * (qk & 1);
    if (row >= 0 && row < n && tile_needed(tri, a, Q) && (tri == TRI_ALL || rotated[a])) {
      double x[QK];
      load_xrow(X, ldx, xmode, n, row, g0, x);
#pragma unroll
      for (int c = 0; c < QK; ++c) {
        const int g = g0 + c;
        if (g < n && (tri != TRI_SECOND || a > Q || row >= g)) {
          Y[(size_t)g * ldy + row] = x[c];
          if (tri == TRI_SECOND && (a > Q || row > g)) Y[(size_t)row * ldy + g] = x[c];
        }
      }
    }
    return;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sm.tmem)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&sm.mbar)) : "memory");
  // U_Q digits (contiguous, NSL x 2 KB) and column exponents
  {
    const uint4* src = reinterpret_cast<const uint4*>(Usl + (size_t)Q * NSL * (USL_BYTES / 2));
    uint4* dst = reinterpret_cast<uint4*>(sm.us[0]);
    for (int i = tid; i < NSL * USL_BYTES / 16; i += RM_THREADS) dst[i] = src[i];
    if (tid < W2) sm.uexp[tid] = Uexp[Q * W2 + tid] << 20;
  }
  // digits of X_Q: this thread's tile row, 8 values of one block (zeros for
  // rows of tiles that are not formed)
  {
    const int rl = tid >> 2, qk = tid & 3;
    const int row = tile_row(nb, R, gx, rl);
    const int g0 = (qk & 2 ? J : I) * BS + QK * (qk & 1);
    double x[QK];
    load_xrow(X, ldx, xmode, n, tile_needed(tri, a0 + (rl >> 5), Q) ? row : -1, g0, x);
    uint32_t mh = 0, ml = 0;  // largest high word of the magnitudes, all low words
#pragma unroll
    for (int k = 0; k < QK; ++k) {
      mh = max(mh, (uint32_t)__double2hiint(x[k]) & 0x7FFFFFFFu);
      ml |= (uint32_t)__double2loint(x[k]);
    }
    mh = max(mh, __shfl_xor_sync(0xffffffffu, mh, 1));
    mh = max(mh, __shfl_xor_sync(0xffffffffu, mh, 2));
    ml |= __shfl_xor_sync(0xffffffffu, ml, 1);
    ml |= __shfl_xor_sync(0xffffffffu, ml, 2);
    // max|x| < 2^er; subnormal rows take the bound 2^-1021 (their grid is finer than any double's)
    const int er = (mh | ml) == 0 ? 0 : max((int)(mh >> 20), 1) - 1022;
    if (qk == 0) sm.rexp[rl] = er;
    uint32_t d[QK / 2][NSL];
#pragma unroll
    for (int j = 0; j < QK / 2; ++j)
      digit_pairs(biased_digits(x[2 * j], er), (uint32_t)__double2hiint(x[2 * j]), biased_digits(x[2 * j + 1], er),
                  (uint32_t)__double2hiint(x[2 * j + 1]), d[j]);
#pragma unroll
    for (int s = 0; s < NSL; ++s)
      *reinterpret_cast<uint4*>(sm.xs[s] + kmaj16(rl, QK * qk)) = make_uint4(d[0][s], d[1][s], d[2][s], d[3][s]);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = sm.tmem;
  const uint32_t mb = smem_u32(&sm.mbar);
  if (tid == 0) {
    constexpr uint32_t idesc = idesc_f16(TM, W2);
    const uint64_t xd = sdesc(smem_u32(sm.xs[0])), ud = sdesc(smem_u32(sm.us[0]));
    // digit pair (i, j), i + j <= 6: level i + j; the products of one A tile in a row
#pragma unroll
    for (int i = 0; i < NSL; ++i) {
#pragma unroll
      for (int kk = 0; kk < W2 / 16; ++kk) {
        const uint64_t ad = xd + (uint64_t)((i * XSL_BYTES + kk * 256) >> 4);
#pragma unroll
        for (int j = 0; i + j < NLEV; ++j) {
          const uint64_t bd = ud + (uint64_t)((j * USL_BYTES + kk * 256) >> 4);
          const uint32_t d = tmem + (uint32_t)((i + j) * W2), acc = i > 0 || kk > 0;
          if (i == NSL - 1)
            mma_f16<A_ONCE>(d, ad, bd, idesc, acc);
          else if (j == 0)
            mma_f16<A_FILL>(d, ad, bd, idesc, acc);
          else if (i + j == NLEV - 1)
            mma_f16<A_LAST>(d, ad, bd, idesc, acc);
          else
            mma_f16<A_USE>(d, ad, bd, idesc, acc);
        }
      }
    }
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mb) : "memory");
  }
  // bounded wait for the products
  bool ok = true;
  {
    const long long t0 = clock64();
    while (!mbar_try(mb, 0)) {
      if (clock64() - t0 > WAIT_CYCLES) {
        ok = false;
        break;
      }
    }
    if (!ok) {
      if (lane == 0 && flags) atomicOr(flags, MPJ_FLAG_TIMEOUT);
      const long long t1 = clock64();  // the products may still be in flight
      while (!mbar_try(mb, 0) && clock64() - t1 <= WAIT_CYCLES) {
      }
    }
  }
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const int quad = warp & 3, ch = warp >> 2;
  const int a = a0 + quad;  // this warp's block pair (warp-uniform)
  if (ok && a < nb / 2 && tile_needed(tri, a, Q)) {
    const int rl = quad * 32 + lane;
    const int row = tile_row(nb, R, gx, rl);
    const int er = sm.rexp[rl];
    const int g0 = (ch & 2 ? J : I) * BS + QK * (ch & 1);
    const bool diag = tri == TRI_SECOND && a == Q;
    double out[QK];
#pragma unroll
    for (int c0 = 0; c0 < QK; c0 += 4) {
      uint32_t v[NLEV][4];
#pragma unroll
      for (int l = 0; l < NLEV; ++l)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                     : "=r"(v[l][0]), "=r"(v[l][1]), "=r"(v[l][2]), "=r"(v[l][3])
                     : "r"(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(l * W2 + ch * QK + c0)));
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      const int4 ue = *reinterpret_cast<const int4*>(&sm.uexp[ch * QK + c0]);
      const int uec[4] = {ue.x, ue.y, ue.z, ue.w};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        // Z = sum_L s_L 2^(8 (6 - L)) = hi 2^32 + lo, hi = s0 2^16 + (s1 2^8 + s2),
        // lo = (s3 2^8 + s4) 2^16 + (s5 2^8 + s6); the bracketed pairs fit 32 bits
        // (|s_L| < 2^22.2).  s + 1.5 2^23 has the bit pattern 0x4B400000 + s.
        uint32_t q[NLEV];
#pragma unroll
        for (int l = 0; l < NLEV; ++l) q[l] = __float_as_uint(__fadd_rn(__uint_as_float(v[l][c]), 12582912.0f));
        constexpr uint32_t B0 = 0x4B400000u, B1 = (B0 << 8) + B0;
        const int t0 = (int)(q[0] - B0), t1 = (int)((q[1] << 8) + q[2] - B1);
        const int t2 = (int)((q[3] << 8) + q[4] - B1), t3 = (int)((q[5] << 8) + q[6] - B1);
        if ((unsigned)(er + 900) < 1800u) {
          // |hi| < 2^39, |lo| < 2^47: with 1.5 2^52 added they are mantissas of the doubles
          // (1.5 2^52 + hi) 2^(32 + E) and (1.5 2^52 + lo) 2^E, E = er + ue - 64.  Taking
          // 1.5 2^(52 + E) (2^32 + 1) from the first is exact and leaves hi 2^(32 + E) minus the
          // second's bias, so the last add is the one rounding of Z 2^E.
          const int kh = ((er + 32 - 64 + 1075) << 20) + uec[c] + 0x80000, kl = kh - (32 << 20);
          const long long hi = (long long)t0 * 65536 + (((long long)kh << 32) + (long long)t1);
          const long long lo = (long long)t2 * 65536 + (((long long)kl << 32) + (long long)t3);
          const double x = __dsub_rn(__longlong_as_double(hi), __hiloint2double(kh, 0x00180000));
          out[c0 + c] = __dadd_rn(x, __longlong_as_double(lo));
        } else {
          out[c0 + c] = z_to_double(((long long)t0 << 16) + t1, ((long long)t2 << 16) + t3, er + (uec[c] >> 20) - 64);
        }
      }
    }
    if (row >= 0 && row < n) {
#pragma unroll
      for (int c = 0; c < QK; ++c) {
        const int g = g0 + c;
        if (g < n && (!diag || row >= g)) Y[(size_t)g * ldy + row] = out[c];
      }
    }
    if (tri == TRI_SECOND) {
      // the mirror entries, through shared memory so that eight lanes write
      // 64 contiguous bytes (the digit tiles are free: the products are done)
      double* buf = reinterpret_cast<double*>(sm.xs[0]) + warp * 32 * (QK + 1);
#pragma unroll
      for (int c = 0; c < QK; ++c) buf[lane * (QK + 1) + c] = out[c];
      __syncwarp();
      int Ia, Ja;
      block_pair(nb, R, a, Ia, Ja);
      const int g = g0 + (lane & 7);
#pragma unroll
      for (int i = 0; i < QK; ++i) {
        const int l = 4 * i + (lane >> 3), r = gidx(Ia, Ja, l);
        if (r < n && g < n && (!diag || r > g)) Y[(size_t)r * ldy + g] = buf[l * (QK + 1) + (lane & 7)];
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
}

__global__ void __launch_bounds__(RM_THREADS, 2)
    blk_rmul(const double* X, int ldx, int xmode, double* Y, int ldy, int n, int nb, int R,
             const __half* __restrict__ Usl, const int* __restrict__ Uexp, const int* __restrict__ rotated,
             unsigned* __restrict__ flags, int tri) {
  pdl_wait();
  blk_rmul_tile(X, ldx, xmode, Y, ldy, n, nb, R, Usl, Uexp, rotated, flags, tri, blockIdx.x, blockIdx.y);
}

// A batch: step 0, the tiles of B = A U~ and then of V <- V U~ per matrix;
// step 1, those of A = B^T U~.
__global__ void __launch_bounds__(RM_THREADS, 2)
    blk_rmul_batch(BatchShape b, int lo, int R, int step, double* A, double* V, double* B,
                   const __half* __restrict__ sl, const int* __restrict__ ex, const int* __restrict__ rot,
                   unsigned* __restrict__ flags) {
  pdl_wait();
  BatchTask t;
  const int kinds = step == 0 ? 2 : 1;
  if (!batch_find(b, lo, blockIdx.x, [kinds](int np) { return kinds * ((np + 3) / 4) * np; }, t)) return;
  const int np = t.N / W2, per = ((np + 3) / 4) * np;
  const bool v = t.local >= per;
  const int l = v ? t.local - per : t.local;
  const double* X = step == 1 ? B : v ? V : A;
  double* Y = step == 1 ? A : v ? V : B;
  blk_rmul_tile(X + t.el, t.N, step == 1 ? XMODE_ROWS : XMODE_COLS, Y + t.el, t.N, t.n, t.N / BS, R,
                sl + (size_t)t.pair0 * NSL * (USL_BYTES / 2), ex + t.pair0 * W2, rot + t.pair0, flags,
                step == 1 ? TRI_SECOND : v ? TRI_ALL : TRI_FIRST, l / np, l % np);
}

inline size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

// One set of U_P digit tiles, exponents and rotation flags for a round.
static size_t uset_bytes(int npairs) {
  return al256((size_t)npairs * NSL * USL_BYTES) + al256((size_t)npairs * W2 * sizeof(int)) +
         al256((size_t)npairs * sizeof(int));
}

// Two sets (rounds alternate between them, so the V update of a round may
// still read its set while the next round's subproblems write the other).
size_t mpj_blocked_scratch_bytes(int n) {
  const int N = (n + 2 * BS - 1) / (2 * BS) * (2 * BS);
  return 2 * uset_bytes(N / (2 * BS)) + 256;
}

namespace {
struct USet {
  __half* sl;
  int* ex;
  int* rot;
};
USet uset(void* scratch, int n, int parity) {
  const int N = (n + 2 * BS - 1) / (2 * BS) * (2 * BS);
  const int npairs = N / (2 * BS);
  char* base = (char*)scratch + (size_t)parity * uset_bytes(npairs);
  USet u;
  u.sl = (__half*)base;
  u.ex = (int*)(base + al256((size_t)npairs * NSL * USL_BYTES));
  u.rot = (int*)((char*)u.ex + al256((size_t)npairs * W2 * sizeof(int)));
  return u;
}
size_t rmul_smem() {
  // at least 80 KB of shared memory per CTA: at most two CTAs per SM, the two
  // that the 512 TMEM columns hold (256 each), so no CTA waits in tcgen05.alloc
  return sizeof(RmulSmem) + 1024 > 80 * 1024 ? sizeof(RmulSmem) + 1024 : 80 * 1024;
}
cudaError_t rmul_attr(const void* kernel) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rmul_smem());
}
}  // namespace

// Before the sweeps of a call: the kernels' shared-memory limit, which belongs to
// the current device (a limit set on one device says nothing about another).
cudaError_t mpj_blocked_prepare() { return rmul_attr((const void*)blk_rmul); }

// Round R, step 1: the subproblems of the block pairs, U_P into set R mod 2;
// *nrot (if not null) counts the block pairs that rotated.
cudaError_t mpj_blocked_solve(const double* A, int lda, int n, int R, double skip, double skip_abs, void* scratch,
                              unsigned* nrot, cudaStream_t s) {
  const int N = (n + 2 * BS - 1) / (2 * BS) * (2 * BS);
  const int nb = N / BS;
  const USet u = uset(scratch, n, R & 1);
  return mpj_launch_pdl(nb / 2 <= sm_count() ? blk_solve<1, OneSub64> : blk_solve<2, OneSub64>, dim3(nb / 2),
                        dim3(SOLVE_THREADS), 0, s, OneSub64{A, lda, n, nb, skip_abs, u.sl, u.ex, u.rot, nrot}, R, skip);
}

// The products for A run ahead of those for V (a side stream's), which nothing
// waits for before the next round but one: A's CTAs take every slot that falls
// free.  FP64 sweeps at n = 1500 (twelve) 74.0 -> 71.3 ms, n = 2048 24.1 -> 23.2,
// n = 4096 258 -> 256.  The subproblems gained nothing by it (and 75 ms with both).
// A stream that is above the side stream already keeps its own priority.
static int rm_a_priority(cudaStream_t s) {
  int p = 0;
  if (cudaStreamGetPriority(s, &p) != cudaSuccess) (void)cudaGetLastError();
  return p < 0 ? 0 : -1;
}

// Round R, step 2: A <- U~^T A U~ through B (two right multiplications).
cudaError_t mpj_blocked_update_A(double* A, int lda, double* B, int n, int R, void* scratch, unsigned* flags,
                                 cudaStream_t s) {
  const int N = (n + 2 * BS - 1) / (2 * BS) * (2 * BS);
  const int nb = N / BS;
  const USet u = uset(scratch, n, R & 1);
  const dim3 grid((nb / 2 + 3) / 4, nb / 2);
  const int prio = rm_a_priority(s);
  const cudaError_t e = mpj_launch_pdl_at(prio, blk_rmul, grid, dim3(RM_THREADS), rmul_smem(), s, (const double*)A,
                                          lda, (int)XMODE_COLS, B, n, n, nb, R, (const __half*)u.sl,
                                          (const int*)u.ex, (const int*)u.rot, flags, (int)TRI_FIRST);
  if (e != cudaSuccess) return e;
  return mpj_launch_pdl_at(prio, blk_rmul, grid, dim3(RM_THREADS), rmul_smem(), s, (const double*)B, n,
                           (int)XMODE_ROWS, A, lda, n, nb, R, (const __half*)u.sl, (const int*)u.ex,
                           (const int*)u.rot, flags, (int)TRI_SECOND);
}

// Round R, step 3: V <- V U~ (in place); independent of step 2.
cudaError_t mpj_blocked_update_V(double* V, int ldv, int n, int R, void* scratch, unsigned* flags, cudaStream_t s) {
  const int N = (n + 2 * BS - 1) / (2 * BS) * (2 * BS);
  const int nb = N / BS;
  const USet u = uset(scratch, n, R & 1);
  const dim3 grid((nb / 2 + 3) / 4, nb / 2);
  return mpj_launch_pdl(blk_rmul, grid, dim3(RM_THREADS), rmul_smem(), s, (const double*)V, ldv, (int)XMODE_COLS, V,
                        ldv, n, nb, R, (const __half*)u.sl, (const int*)u.ex, (const int*)u.rot, flags,
                        (int)TRI_ALL);
}

size_t mpj_batch_digit_bytes(int pairs) { return uset_bytes(pairs); }

cudaError_t mpj_batch_sweep64_round(const BatchShape& b, int R, double* A, double* V, double* B, const double* skip_abs,
                                    void* digits, int pairs, unsigned* flags, cudaStream_t s) {
  const int lo = batch_lowest_class(R);
  const long long subs = batch_blocks(b, lo, [](int np) { return np; });
  if (subs == 0) return cudaSuccess;
  cudaError_t e = rmul_attr((const void*)blk_rmul_batch);
  if (e != cudaSuccess) return e;
  __half* sl = (__half*)digits;
  int* ex = (int*)((char*)digits + al256((size_t)pairs * NSL * USL_BYTES));
  int* rot = (int*)((char*)ex + al256((size_t)pairs * W2 * sizeof(int)));
  const BatchSub64 src{b, lo, A, skip_abs, sl, ex, rot};
  e = mpj_launch_pdl(subs <= sm_count() ? blk_solve<1, BatchSub64> : blk_solve<2, BatchSub64>, dim3((unsigned)subs),
                     dim3(SOLVE_THREADS), 0, s, src, R, 0x1p-53);
  const long long tiles = batch_blocks(b, lo, [](int np) { return ((np + 3) / 4) * np; });
  for (int step = 0; step < 2 && e == cudaSuccess; ++step)
    e = mpj_launch_pdl(blk_rmul_batch, dim3((unsigned)(step == 0 ? 2 * tiles : tiles)), dim3(RM_THREADS), rmul_smem(),
                       s, b, lo, R, step, A, V, B, (const __half*)sl, (const int*)ex, (const int*)rot, flags);
  return e;
}

int mpj_blocked_rounds_per_sweep(int n) {
  const int N = (n + 2 * BS - 1) / (2 * BS) * (2 * BS);
  return N / BS - 1;
}

// A = (A + A^T) / 2 (the paper's end-of-sweep symmetrization; the blocked
// update computes both triangles, which agree only to rounding).
__global__ void blk_symmetrize(double* __restrict__ A, int lda, int n) {
  const size_t total = (size_t)n * n;
  for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(idx % n), j = (int)(idx / n);
    if (i > j) {
      const double v = 0.5 * (A[(size_t)j * lda + i] + A[(size_t)i * lda + j]);
      A[(size_t)j * lda + i] = v;
      A[(size_t)i * lda + j] = v;
    }
  }
}

cudaError_t mpj_blocked_symmetrize(double* A, int lda, int n, cudaStream_t s) {
  size_t b = ((size_t)n * n + 255) / 256;
  blk_symmetrize<<<(int)(b > 4096 ? 4096 : (b < 1 ? 1 : b)), 256, 0, s>>>(A, lda, n);
  mpj_count_launch();
  return cudaGetLastError();
}
