// Truncated SVD of one charge block by an FP32 eigendecomposition and a
// refinement of the kept singular vectors alone.
//
// A gate keeps about a quarter of its singular triplets (chi of up to 4 chi),
// and only the kept ones are needed to full precision.  So, for a block B
// (m x n, n <= m):
//   1. eig_start:  G = B^T B to FP32, Householder tridiagonalisation, all
//      eigenvalues by multisection (Sturm counts), eigenvectors of the
//      tridiagonal matrix by inverse iteration (LU with partial pivoting,
//      two steps), back-transformation, Newton-Schulz steps until the vectors
//      X are orthonormal to FP32.  About 3 n^3 multiply-adds with one team
//      barrier per Householder step, against 7 sweeps of 6 n^3 for one-sided
//      Jacobi in FP32.
//   2. (the caller decides from the eigenvalues, with error bounds, which
//      columns can be kept at all)
//   3. eig_refine: for the kept columns x_k alone
//        w = B x, lambda = |w|^2, r = B^T w - lambda x,
//      and the first-order correction with all FP32 vectors X as the basis,
//        x <- x + X t,  t_i = X_i . r / (lambda - lambda_i),  t_k = (1 - |x|^2) / 2
//      (Ogita and Aishima, Japan J. Indust. Appl. Math. 35 (2018) 1007, with the
//      residual formed before the projection, so that the products with X and
//      the update only need FP32).  It converges quadratically in the kept vectors and
//      by 1e-6 over the relative distance of the eigenvalues along the dropped ones,
//      whose eigenvalues stay FP32: on the gates of N = 14, chi = 128 states |t| is at
//      most 1e-4, then 1e-8, so two corrections, sometimes three.  x, w and lambda are
//      FP64 (with double-floats of 48 bits the vectors and the truncated tensor were off
//      by up to 1e-14, 9 to 24 columns by 1.5 times an FP64 Jacobi SVD; now by 1e-15 and
//      a quarter of it, for 1.5 to 4 % of the time of a call).  Last, the kept
//      vectors are orthonormalised by their inner products (I + (I - X^T X) / 2): the
//      corrections alone leave 1e-13, and the matrix elements ten times the rounding
//      error of an FP64 SVD.
// Whatever this cannot do (a kept singular value below 5e-3 of the block's
// largest one, a cluster that leaves X dependent, a correction that does not
// shrink) is reported, and the caller takes the one-sided Jacobi SVD.
//
// The products with B run on the tensor cores with operands cut into 8-bit signed
// digits (Ozaki, Ogita, Oishi, Rump, Numer. Algorithms 59 (2012) 95): every digit is
// an exact BF16 number and a digit product is at most 2^14, so the sum of one order over K
// entries is an integer of at most (order - 1) K 2^14, exact in FP32 below 2^24: in every
// order for K <= 146, and for the 256 rows that a bond allows in the orders up to 5 and in
// all three of the Gram matrix.  Beyond, only digits that are nearly all of one sign and at
// their limit reach it; then the last unit of such an order is rounded, 2^-44 of the
// operands' scales in order 6 (whose leading digits would have to be at their limit in both
// operands, which a unit vector's are not), 2^-52 and 2^-60 in the orders 7 and 8, below the
// rounding of the result.  Seven digits (resolution
// 2^-54 of the block's largest entry) with the 28 products of order up to 8 carry the
// accuracy of FP64 sums.  A multiply-add costs 28/2048
// of a warp-wide mma against 12 FP32 instructions in double-float and 64 issue cycles
// in FP64 (GB300's FP64 rate is 1/64 of its FP32 rate).  mma.sync and not tcgen05: the
// blocks are 10 to 80 wide and eight to thirty columns are kept, far below a tcgen05
// tile, and the operands of a warp come straight from L2 in fragment order.
#pragma once
#include <cuda_runtime.h>

namespace tnqe {
namespace {

constexpr int EIG_NE = 5;                          // lanes' share of a row: n <= 32 EIG_NE
constexpr int EIG_MAXN = 32 * EIG_NE;
// A correction below this is the last.  (1e-8 leaves errors of 5e-16 in overlaps of N = 12, chi = 64 states with
// decaying spectra where an FP64 SVD and 1e-9 leave 1e-16; rotation of N = 14, chi = 128 83 against 87 ms.)
constexpr float EIG_ACCEPT = 1e-9f;
constexpr float EIG_MIN_LAMBDA = 3e-5f;            // kept lambda over the block's largest: sigma ratio 5.5e-3
constexpr int EIG_TC = 8;                          // kept columns per task (an mma's n)
constexpr int EIG_DIG = 7;                         // digits of an operand

__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
// The larger of two values, a NaN if either is one.
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
// Row stride of the n x n FP32 arrays: a multiple of 4 (16-byte rows) and 4 mod 8, so
// that 16-byte accesses of eight consecutive rows fall into distinct banks.
__host__ __device__ constexpr __forceinline__ int eig_ld(int n) {
  const int l = (n + 3) & ~3;
  return (l & 7) == 4 ? l : l + 4;
}
__host__ __device__ constexpr __forceinline__ int eig_kp(int k) { return (k + EIG_TC - 1) & ~(EIG_TC - 1); }
__host__ __device__ __forceinline__ int pad16(int n) { return (n + 15) & ~15; }
// floats of the small vectors of eig_start (V: 2 ld, W: ld, P: 2 ld, d, e, tau, lam, scale, a dummy row)
__host__ __device__ __forceinline__ int eig_vec_floats(int n) { return 11 * eig_ld(n) + 32; }
// floats that eig_refine needs at least: lk (kp doubles), lh, ek and exs (kp), lam (ld), R (kp x ld), T (n x kp)
__host__ __device__ constexpr __forceinline__ int eig_refine_words(int n, int kc) {
  const int kp = eig_kp(kc), ld = eig_ld(n);
  return 5 * kp + ld + kp * ld + n * kp;
}
// Tells the compiler that a generic pointer points to shared memory.
#define EIG_SHARED(p) __builtin_assume(__isShared(p))

// Two FP32 multiply-adds in one instruction.
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
  unsigned long long x, y, z, r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(a.x), "f"(a.y));
  asm("mov.b64 %0, {%1, %2};" : "=l"(y) : "f"(b.x), "f"(b.y));
  asm("mov.b64 %0, {%1, %2};" : "=l"(z) : "f"(c.x), "f"(c.y));
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(x), "l"(y), "l"(z));
  float2 o;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(o.x), "=f"(o.y) : "l"(r));
  return o;
}

// Uniform in [-1, 1] from a pair of indices (a start vector only has to be generic): an integer hash, the pair
// combined by the golden-ratio constant 0x9E3779B1 and 0x85EBCA77 (two primes of Collet's xxHash32), finished with the
// shifts and multipliers 15, 0x2C1B3C6D, 12, 0x297A2D39, 15 that Wellons found by search (hash-prospector).
__device__ __forceinline__ float eig_noise(unsigned i, unsigned u) {
  unsigned h = i * 0x9E3779B1u ^ (u + 0x7F4A7C15u) * 0x85EBCA77u;
  h ^= h >> 15;
  h *= 0x2C1B3C6Du;
  h ^= h >> 12;
  h *= 0x297A2D39u;
  h ^= h >> 15;
  return (float)(int)h * 4.656612873e-10f;
}

// ----------------------------------------------------------------------------- digits and mma fragments
// A value v, |v| < 2, is the integer I = v 2^54 and I = sum_{s=1..7} d_s 2^(8 (7 - s)), d_s in
// [-128, 128]: v = sum d_s 2^(2 - 8 s).
// x / 2^ex 2^54 of a double, |x| < 2^(1 + ex), to the nearest integer
__device__ __forceinline__ long long fix_double(double x, int ex) {
  const long long b = __double_as_longlong(x);
  const int e = (int)((b >> 52) & 2047);
  const long long m = e ? ((b & 0xfffffffffffffll) | 0x10000000000000ll) : 0;
  const int sh = e - 1023 - ex + 2;
  const long long v = sh >= 0 ? m << min(sh, 10) : (sh > -54 ? (m + (1ll << (-sh - 1))) >> -sh : 0);
  return b < 0 ? -v : v;
}
// the digits of a pair of integers as BF16 pairs (first in the low half)
__device__ __forceinline__ void digits_pair(long long a, long long b, unsigned (&w)[EIG_DIG]) {
  const long long bias = 0x808080808080ll;
  a += bias;
  b += bias;
  const float ta = __int_as_float(0x4B400000 + (int)(a >> 48)) - 12582912.f;
  const float tb = __int_as_float(0x4B400000 + (int)(b >> 48)) - 12582912.f;
  w[0] = __byte_perm((unsigned)__float_as_int(ta), (unsigned)__float_as_int(tb), 0x7632);
  const unsigned al = (unsigned)a, ah = (unsigned)((unsigned long long)a >> 32);
  const unsigned bl = (unsigned)b, bh = (unsigned)((unsigned long long)b >> 32);
#pragma unroll
  for (int s = 1; s < EIG_DIG; ++s) {
    const int by = EIG_DIG - 1 - s;                // byte 5 .. 0
    const unsigned sel = 0x7440u | (by & 3);       // byte, 0, 0, 0x4B
    const float fa = __int_as_float((int)__byte_perm(by > 3 ? ah : al, 0x4B000000u, sel)) - 8388736.f;
    const float fb = __int_as_float((int)__byte_perm(by > 3 ? bh : bl, 0x4B000000u, sel)) - 8388736.f;
    w[s] = __byte_perm((unsigned)__float_as_int(fa), (unsigned)__float_as_int(fb), 0x7632);
  }
}
__device__ __forceinline__ unsigned transpose8x8(unsigned x) {
  unsigned r;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(x));
  return r;
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint4& a, const uint2& b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y));
}

// A-operand fragments of B (rows of B) in A and of B^T in At, tile by tile: the 16 x 16 tile
// (it, kt) of a matrix with KT column tiles has its EIG_DIG digits at ((it KT + kt) EIG_DIG + s) 32
// + lane.  raw: B column-major (m x n), |entries| < 2^(1 + ex).  A warp takes a tile of
// B; its transpose comes from the registers (movmatrix) unless At is null.
template <class Team>
__device__ __noinline__ void eig_digits(const Team tm, const double* raw, int m, int n, int ex, uint4* A, uint4* At) {
  const int lane = threadIdx.x & 31, warp = tm.rank() >> 5, nw = tm.size() >> 5;
  const int mt = pad16(m) >> 4, nt = pad16(n) >> 4, g = lane >> 2, t2 = 2 * (lane & 3);
  for (int t = warp; t < mt * nt; t += nw) {
    const int it = t % mt, kt = t / mt;
    double v[4][2];                                // registers (rows g, g + 8) x (columns t2, t2 + 8), pairs along the row
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = 16 * it + g + 8 * (q & 1), c = 16 * kt + t2 + 8 * (q >> 1) + h;
        const double x = raw[(size_t)min(c, n - 1) * m + min(r, m - 1)];
        v[q][h] = (r < m && c < n) ? x : 0.0;
      }
    unsigned w[4][EIG_DIG];
#pragma unroll
    for (int q = 0; q < 4; ++q) digits_pair(fix_double(v[q][0], ex), fix_double(v[q][1], ex), w[q]);
    uint4* a = A + (size_t)(it * nt + kt) * EIG_DIG * 32 + lane;
    uint4* b = At + (size_t)(kt * mt + it) * EIG_DIG * 32 + lane;
#pragma unroll
    for (int s = 0; s < EIG_DIG; ++s) {
      a[s * 32] = make_uint4(w[0][s], w[1][s], w[2][s], w[3][s]);
      if (At) b[s * 32] = make_uint4(transpose8x8(w[0][s]), transpose8x8(w[2][s]), transpose8x8(w[1][s]), transpose8x8(w[3][s]));
    }
  }
  tm.sync();
}

// B-operand fragments of the columns k = 0..kp-1 of V (column k at k ldv, |entries| <
// 2^(1 + exs[k]), exs null: 2; length K padded with zeros to a multiple of 16): the 16 x 8 tile (kt, jt)
// has its digits at ((kt JT + jt) ND + s) 32 + lane.
template <int ND, class Team>
__device__ __noinline__ void eig_digits_cols(const Team tm, const double* V, int ldv, int K, int kp, const int* exs,
                                             uint2* D) {
  const int lane = threadIdx.x & 31, warp = tm.rank() >> 5, nw = tm.size() >> 5;
  const int kt = pad16(K) >> 4, jt = kp >> 3, g = lane >> 2, t2 = 2 * (lane & 3);
  for (int t = warp; t < kt * jt; t += nw) {
    const int k = t / jt, j = t % jt;
    const int ex = exs ? exs[8 * j + g] : 0;
    const double2* p = reinterpret_cast<const double2*>(V + (size_t)(8 * j + g) * ldv + 16 * k + t2);
    const double2 lo = p[0], hi = p[4];
    unsigned a[EIG_DIG], b[EIG_DIG];
    digits_pair(fix_double(lo.x, ex), fix_double(lo.y, ex), a);
    digits_pair(fix_double(hi.x, ex), fix_double(hi.y, ex), b);
    uint2* d = D + (size_t)t * ND * 32 + lane;
#pragma unroll
    for (int s = 0; s < ND; ++s) d[s * 32] = make_uint2(a[s], b[s]);
  }
  tm.sync();
}

// One 16 x 8 tile of the product: NA digits of the first operand (tile row `it`, KT tiles), NB of the
// second (tile column j of JT), products of order up to NS.  acc[o] holds the sums of order
// o + 2 in units of 2^(4 - 8 (o + 2)).  The first operand comes from L2, one tile ahead of
// its use.  (Two tiles sharing its loads, without that: 96.0 against 91.6 ms of rotation on
// N = 14, chi = 128.)
template <int NA, int NB, int NS>
__device__ __forceinline__ void mma_tile(const uint4* A, const uint2* D, int it, int j, int KT, int JT, int lane,
                                         float (&acc)[NS - 1][4]) {
#pragma unroll
  for (int o = 0; o < NS - 1; ++o)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[o][q] = 0.f;
  const uint4* ap = A + (size_t)it * KT * EIG_DIG * 32 + lane;
  uint4 an[NA];
#pragma unroll
  for (int s = 0; s < NA; ++s) an[s] = ap[s * 32];
  for (int k = 0; k < KT; ++k) {
    uint4 a[NA];
    uint2 b[NB];
#pragma unroll
    for (int s = 0; s < NA; ++s) a[s] = an[s];
    const uint2* bp = D + (size_t)(k * JT + j) * NB * 32 + lane;
#pragma unroll
    for (int s = 0; s < NB; ++s) b[s] = bp[s * 32];
    if (k + 1 < KT) {
      ap += EIG_DIG * 32;
#pragma unroll
      for (int s = 0; s < NA; ++s) an[s] = ap[s * 32];
    }
#pragma unroll
    for (int i = 0; i < NA; ++i)
#pragma unroll
      for (int s = 0; s < NB; ++s)
        if (i + s + 2 <= NS) mma_bf16(acc[i + s], a[i], b[s]);
  }
}
// i 2^e, |i| < 2^51, |e| < 900 (one FP64 addition; the conversion instruction and the scaling would be three)
__device__ __forceinline__ double small_double(long long i, int e) {
  const long long one = 0x4338000000000000ll + ((long long)e << 52);          // 1.5 2^(52 + e)
  return __longlong_as_double(one + i) - __longlong_as_double(one);
}
// The sums of all orders times 2^e, rounded once to FP64: the orders up to 4 and those above as two integers (at
// most 2^48).
template <int NS>
__device__ __forceinline__ double mma_value(const float (&acc)[NS - 1][4], int q, int e) {
  long long hi = 0, lo = 0;
#pragma unroll
  for (int o = 0; o < NS - 1; ++o) {
    const long long x = __float2int_rn(acc[o][q]);
    if (o < 3) hi = (hi << 8) + x;
    else lo = (lo << 8) + x;
  }
  return small_double(hi, e - 28) + small_double(lo, e + 4 - 8 * NS);
}

// ----------------------------------------------------------------------------- Gram matrix
// S (n x n, row stride ld, both triangles, pad columns zero) = B^T B to FP32: three digits, the six
// products of order up to 4.  The fragments of B^T serve as both operands.
template <class Team>
__device__ __noinline__ void eig_gram(const Team tm, const uint4* At, int m, int n, float* S, int ld) {
  EIG_SHARED(S);
  const int tr = tm.rank(), ts = tm.size(), lane = threadIdx.x & 31, warp = tr >> 5, nw = ts >> 5;
  const int mt = pad16(m) >> 4, nt = pad16(n) >> 4, g = lane >> 2, t2 = 2 * (lane & 3);
  for (int x = tr; x < n * (ld - n); x += ts) S[(x / (ld - n)) * ld + n + x % (ld - n)] = 0.f;
  for (int t = warp; t < nt * 2 * nt; t += nw) {
    const int it = t / (2 * nt), j8 = t % (2 * nt), jt = j8 >> 1;
    if (jt < it || 8 * j8 >= n) continue;
    float acc[3][4];
#pragma unroll
    for (int o = 0; o < 3; ++o)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[o][q] = 0.f;
    const uint4* ap = At + (size_t)it * mt * EIG_DIG * 32 + lane;
    const uint4* bp = At + (size_t)jt * mt * EIG_DIG * 32 + lane;
#pragma unroll 2
    for (int k = 0; k < mt; ++k) {
      uint4 a[3];
      uint2 b[3];
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        a[s] = ap[(k * EIG_DIG + s) * 32];
        const uint4 v = bp[(k * EIG_DIG + s) * 32];
        b[s] = (j8 & 1) ? make_uint2(v.y, v.w) : make_uint2(v.x, v.z);
      }
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int s = 0; s + i < 3; ++s) mma_bf16(acc[i + s], a[i], b[s]);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = 16 * it + g + 8 * (q >> 1), j = 8 * j8 + t2 + (q & 1);
      if (i < n && j < n) {
        const float v = fmaf(acc[0][q], 0x1p-12f, fmaf(acc[1][q], 0x1p-20f, acc[2][q] * 0x1p-28f));
        S[i * ld + j] = v;
        if (jt > it) S[j * ld + i] = v;
      }
    }
  }
  tm.sync();
}

// ----------------------------------------------------------------------------- tridiagonalisation
// Householder reduction of the symmetric A (row stride ld): diagonal d, off-diagonal
// e, reflectors I - tau v v^T; reflector t is left in row t - 1 of A, the first in V
// (zero up to component t).
//
// n - 2 dependent steps with one team barrier and one reduction each; bound by the
// instructions of a step where four teams share an SM, by their latency otherwise.  The
// rows of the trailing matrix belong to 8-lane groups; a group applies the last rank-2
// update to its rows and multiplies them with the new reflector in one pass, two rows
// at a time, in packed FP32 pairs.  Every warp forms the reflector of row t by itself,
// from the row in memory, the products p = tau A v of the last step and the last
// reflector v (v_t = 1):
//   w = p - K v, K = tau p.v / 2,   row t of A - v w^T - w v^T  =  u + kappa v,
//   u = a - p, kappa = 2 K - p_t,
// so that K and the norm of the row come from sums over p, u and v that do not wait
// for one another (where they cancel, the norm is summed again).  W and P (two, by
// parity) hold w and p; all warps write the same values into the reflectors and W.
template <int NE, class Team>
__device__ __noinline__ void eig_tridiag_ne(const Team tm, float* A, int n, int ld, float* V, float* W, float* P, float* d,
                                            float* e, float* tau, float* dummy) {
  // 32-bit offsets into the pool: a pointer select per row would cost 64-bit arithmetic
  extern __shared__ float4 rot_pool[];
  float* const S = reinterpret_cast<float*>(rot_pool);
  const int Vo = (int)(V - S), Wo = (int)(W - S), Ao = (int)(A - S), Po = (int)(P - S), Do = (int)(dummy - S);
  const int so = (int)(d - S), eo = (int)(e - S), to = (int)(tau - S);
  const int tr = tm.rank(), ts = tm.size();
  const int lane = threadIdx.x & 31, grp = tr >> 3, ngrp = ts >> 3, gl = tr & 7;
  const unsigned gmask = 0xffu << ((lane >> 3) * 8);
  const bool one = tr == 0;
  for (int c = tr; c < ld; c += ts) {
    S[Vo + c] = 0.f;
    S[Vo + ld + c] = 0.f;                          // the reflector before the first
    S[Wo + c] = 0.f;
    S[Po + c] = 0.f;
    S[Po + ld + c] = 0.f;
    S[Do + c] = 0.f;                               // stays finite: its products meet zeros
  }
  tm.sync();
  float v[NE];
  float tl = 0.f;                                  // tau of the last reflector
  int rfirst = grp;                                // the group's first row of the trailing matrix
#pragma unroll
  for (int q = 0; q < NE; ++q) v[q] = 0.f;
  int vp = Vo + ld, vc = Vo;                       // the last and the new reflector
#pragma unroll 1
  for (int t = 0; t + 1 < n; ++t) {
    const int pc = Po + (t & 1) * ld, pp = Po + ((t & 1) ^ 1) * ld, ar = Ao + t * ld;
    const float pt = S[pp + t], at = S[ar + t];
    const float an = S[ar + t + 1], pn = S[pp + t + 1], vn = S[vp + t + 1];
    float p[NE], u[NE];
    float s1 = 0.f, s2 = 0.f, s3 = 0.f, s4 = 0.f;
#pragma unroll
    for (int q = 0; q < NE; ++q) {
      const int c = lane + 32 * q, cc = NE == 1 || c < ld ? c : 0;
      p[q] = c < ld ? S[pp + cc] : 0.f;            // v is zero before t and from n on
      u[q] = c < ld ? S[ar + cc] - p[q] : 0.f;
      s1 = fmaf(p[q], v[q], s1);
      const float um = c > t + 1 ? u[q] : 0.f, vm = c > t + 1 ? v[q] : 0.f;
      s2 = fmaf(um, um, s2);
      s3 = fmaf(um, vm, s3);
      s4 = fmaf(vm, vm, s4);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s1 += __shfl_xor_sync(0xffffffffu, s1, o);
      s2 += __shfl_xor_sync(0xffffffffu, s2, o);
      s3 += __shfl_xor_sync(0xffffffffu, s3, o);
      s4 += __shfl_xor_sync(0xffffffffu, s4, o);
    }
    const float K = 0.5f * tl * s1, kap = 2.f * K - pt;
    const float x0 = fmaf(kap, vn, an - pn);
    if (t + 2 == n) {                              // the last 2 x 2 block needs no reflector
      if (one) {
        const int c = n - 1;
        const float vl = S[vp + c], wl = fmaf(-K, vl, S[pp + c]);
        S[so + t] = at - pt + kap;
        S[eo + t] = x0;
        S[so + c] = S[Ao + c * ld + c] - 2.f * vl * wl;
      }
      break;
    }
    const float big = fmaf(kap * kap, s4, s2);
    s2 = fmaf(kap, fmaf(kap, s4, 2.f * s3), s2);
    if (s2 < 0.02f * big) {                        // the sums cancelled
      s2 = 0.f;
#pragma unroll
      for (int q = 0; q < NE; ++q) {
        const float x = fmaf(kap, v[q], u[q]);
        if (lane + 32 * q > t + 1) s2 = fmaf(x, x, s2);
      }
      s2 = warp_sum_f(s2);
    }
    float tj = 0.f, beta = x0, inv = 0.f;
    if (s2 > 1e-30f) {
      const float h2 = fmaf(x0, x0, s2), ri = rsqrtf(h2), h = h2 * ri;
      beta = -copysignf(h, x0);
      tj = fmaf(fabsf(x0), ri, 1.f);
      inv = copysignf(__fdividef(1.f, fabsf(x0) + h), x0);
    }
#pragma unroll
    for (int q = 0; q < NE; ++q) {
      const int c = lane + 32 * q;
      const float w = fmaf(-K, v[q], p[q]), x = fmaf(kap, v[q], u[q]) * inv;
      v[q] = (c == t + 1) ? 1.f : ((c > t + 1) ? x : 0.f);
      if (c < ld) {
        S[Wo + c] = w;
        S[vc + c] = v[q];
      }
    }
    if (one) {
      S[so + t] = at - pt + kap;
      S[eo + t] = beta;
      S[to + t] = tj;
    }
    __syncwarp();
    // rows t + 1.. of the trailing matrix: the last update, and the product with the new
    // reflector (what lies outside goes to a dummy row)
    const int c0 = ((t + 1) & ~3) + 4 * gl;
    if (rfirst < t + 1) rfirst += ngrp;
#pragma unroll 1
    for (int r = rfirst; r < n; r += 2 * ngrp) {
      const int r2 = r + ngrp, rb = r2 < n ? r2 : r;
      const float va = -S[vp + r], wa = -S[Wo + r], vb = -S[vp + rb], wb = -S[Wo + rb];
      const int Ra = Ao + r * ld, Rb = r2 < n ? Ao + r2 * ld : Do;
      const float2 va2 = make_float2(va, va), wa2 = make_float2(wa, wa), vb2 = make_float2(vb, vb), wb2 = make_float2(wb, wb);
      float2 sa = make_float2(0.f, 0.f), sb = sa;
#pragma unroll 1
      for (int c = c0; c < ld; c += 32) {
        const float4 vq = *reinterpret_cast<const float4*>(S + vp + c), wq = *reinterpret_cast<const float4*>(S + Wo + c);
        const float4 nq = *reinterpret_cast<const float4*>(S + vc + c);
        float4 xa = *reinterpret_cast<const float4*>(S + Ra + c), xb = *reinterpret_cast<const float4*>(S + Rb + c);
        const float2 v0 = make_float2(vq.x, vq.y), v1 = make_float2(vq.z, vq.w), w0 = make_float2(wq.x, wq.y),
                     w1 = make_float2(wq.z, wq.w), n0 = make_float2(nq.x, nq.y), n1 = make_float2(nq.z, nq.w);
        const float2 a0 = ffma2(va2, w0, ffma2(wa2, v0, make_float2(xa.x, xa.y)));
        const float2 a1 = ffma2(va2, w1, ffma2(wa2, v1, make_float2(xa.z, xa.w)));
        const float2 b0 = ffma2(vb2, w0, ffma2(wb2, v0, make_float2(xb.x, xb.y)));
        const float2 b1 = ffma2(vb2, w1, ffma2(wb2, v1, make_float2(xb.z, xb.w)));
        *reinterpret_cast<float4*>(S + Ra + c) = make_float4(a0.x, a0.y, a1.x, a1.y);
        *reinterpret_cast<float4*>(S + Rb + c) = make_float4(b0.x, b0.y, b1.x, b1.y);
        sa = ffma2(a0, n0, ffma2(a1, n1, sa));
        sb = ffma2(b0, n0, ffma2(b1, n1, sb));
      }
      float ya = sa.x + sa.y, yb = sb.x + sb.y;
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        ya += __shfl_xor_sync(gmask, ya, o);
        yb += __shfl_xor_sync(gmask, yb, o);
      }
      if (gl == 0) S[pc + r] = tj * ya;
      if (gl == 1 && r2 < n) S[pc + r2] = tj * yb;
    }
    tm.sync();
    tl = tj;
    vp = vc;
    vc = Ao + t * ld;                              // row t is dead now
  }
  if (n == 1 && one) S[so] = S[Ao];
  tm.sync();
}
// More than four warps (two up to n = 48, eight from n = 97 on) only add redundant work to the steps.
template <class Team>
__device__ void eig_tridiag(const Team& tm, float* A, int n, int ld, float* V, float* W, float* P, float* d, float* e,
                            float* tau, float* dummy) {
  const auto sub = tm.part(n <= 48 ? 64 : (n <= 96 ? 128 : 256));
  if (sub.rank() < sub.size()) {
    if (n <= 28) eig_tridiag_ne<1>(sub, A, n, ld, V, W, P, d, e, tau, dummy);
    else if (n <= 60) eig_tridiag_ne<2>(sub, A, n, ld, V, W, P, d, e, tau, dummy);
    else if (n <= 92) eig_tridiag_ne<3>(sub, A, n, ld, V, W, P, d, e, tau, dummy);
    else eig_tridiag_ne<EIG_NE + 1>(sub, A, n, ld, V, W, P, d, e, tau, dummy);
  }
  tm.sync();
}

// ----------------------------------------------------------------------------- eigenvalues
// All eigenvalues of the tridiagonal (d, e), descending in lam, by multisection: two
// lanes per eigenvalue split its interval in three, fourteen times.  d and e are scaled
// in place by the returned 1 / norm (the eigenvalues too).  The Sturm sequence is the
// division-free recurrence p_i = (d_i - x) p_{i-1} - e_{i-1}^2 p_{i-2} (two FMAs per
// step; a reciprocal per step would be bound by 16 lanes per clock and SM), rescaled
// every four steps by the exponent of the values four steps before, which keeps the
// rescaling off the dependent chain; the signs are shifted into a word and counted 32
// at a time.  de holds the pairs (d_i, e_{i-1}^2).
template <class Team>
__device__ __noinline__ float eig_values(const Team tm, float* d, float* e, int n, int ld, float2* de, float* lam) {
  EIG_SHARED(d);
  EIG_SHARED(e);
  EIG_SHARED(de);
  EIG_SHARED(lam);
  const int tr = tm.rank(), ts = tm.size(), lane = threadIdx.x & 31;
  float nm = 0.f;                                  // Gershgorin bound, the same in every warp
  for (int c = lane; c < n; c += 32)
    nm = fmaxf(nm, fabsf(d[c]) + (c > 0 ? fabsf(e[c - 1]) : 0.f) + (c + 1 < n ? fabsf(e[c]) : 0.f));
  nm = warp_max_f(nm);
  const float sc = nm > 1e-30f ? __fdividef(1.f, nm) : 1.f;
  tm.sync();
  for (int c = tr; c < ld; c += ts) {
    const float ep = (c > 0 && c < n ? e[c - 1] : 0.f) * sc;
    // pad rows never change a sign: p_i = (2 - x) p_{i-1}
    de[c] = make_float2(c < n ? d[c] * sc : 2.f, c < n ? fmaxf(ep * ep, 1e-18f) : 0.f);
  }
  tm.sync();
  for (int c = tr; c < ld; c += ts) {
    d[c] = c < n ? d[c] * sc : 0.f;
    e[c] = c + 1 < n ? e[c] * sc : 0.f;
  }
  const int sub = tr >> 1, nsub = ts >> 1, sl = tr & 1;
  const unsigned smask = 3u << (lane & 30);
  const float4* de4 = reinterpret_cast<const float4*>(de);
  for (int t0 = sub; t0 < n; t0 += nsub) {
    float lo = -1e-5f, wd = 1.0002f;               // the interval: lo, width
    for (int pass = 0; pass < 14; ++pass) {
      const float st = wd * 0.333333343f, x = fmaf((float)(sl + 1), st, lo);
      float p = 0.f, q = 1.f;                      // p_{i-2}, p_{i-1}
      unsigned bits = 0, last = 0, cnt = 0;
      float4 ga = de4[0], gb = de4[1];
      for (int i = 0; i < n; i += 4) {
        const float4 ha = ga, hb = gb;
        if (i + 4 < ld) {
          ga = de4[(i >> 1) + 2];
          gb = de4[(i >> 1) + 3];
        }
        const int ex = (__float_as_int(fmaxf(fabsf(p), fabsf(q))) >> 23) & 255;
        const float f = __int_as_float((ex > 40 ? 294 - ex : 254) << 23);     // towards 2^40
        const float dd[4] = {ha.x, ha.z, hb.x, hb.z}, ee[4] = {ha.y, ha.w, hb.y, hb.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float r = fmaf(dd[u] - x, q, -(ee[u] * p));
          bits = __funnelshift_l((unsigned)__float_as_int(r), bits, 1);
          p = q;
          q = r;
        }
        p *= f;
        q *= f;
        if ((i & 31) == 28 || i + 4 >= n) {        // up to 32 signs: their changes, the first against the last word's
          const int have = (i & 31) + 4;
          const unsigned al = bits << (32 - have);
          cnt += __popc((al ^ ((al >> 1) | (last << 31))) & (0xffffffffu << (32 - have)));
          last = bits & 1u;
        }
      }
      // cnt = eigenvalues below x: the points with at most t0 of them lie below eigenvalue t0 (ascending)
      const int below = cnt <= (unsigned)t0 ? 1 : 0;
      const int np = below + __shfl_xor_sync(smask, below, 1);
      lo = fmaf((float)np, st, lo);
      wd = st;
    }
    if (sl == 0) lam[n - 1 - t0] = fmaf(0.5f, wd, lo);
  }
  tm.sync();
  return sc;
}

// ----------------------------------------------------------------------------- eigenvectors of the tridiagonal
// One thread per vector: LU with partial pivoting of T - lam, then two steps of inverse
// iteration; the first starts from a generic right-hand side after the forward
// elimination, so it is a back substitution alone.  X[u * ld + i] is component i of
// vector u; SM (n x n pairs, row stride n, global memory) keeps the pivots and the
// multipliers, loaded eight rows ahead of the eight in use (L2 latency).  A row swap at
// step i shows as |pivot_i| < |e_i|.  inorm[u] gets 1 / |vector u|.
template <bool XS, class Team>
__device__ __noinline__ void eig_vectors(const Team tm, const float* d, const float* e, const float* lam, int n,
                                         float* X, int ld, float2* SM, float* inorm) {
  EIG_SHARED(d);
  EIG_SHARED(e);
  EIG_SHARED(lam);
  EIG_SHARED(inorm);
  if (XS) EIG_SHARED(X);
  const int tr = tm.rank(), ts = tm.size();
  constexpr float TINY = 3e-8f;                    // of |T| = 1
  constexpr int AH = 8;
  for (int u = tr; u < n; u += ts) {
    const float x = lam[u];
    float* Xu = X + u * ld;
    float2* sm = SM + u;
    float a = d[0] - x, b = e[0];
    for (int i = 0; i + 1 < n; i += 4) {
      // rows i .. i + 3: d_{i+1..i+4}, e_{i..i+4} (zero beyond the end)
      const float4 e4 = *reinterpret_cast<const float4*>(e + i), d4 = *reinterpret_cast<const float4*>(d + i);
      const float el = i + 4 < ld ? e[i + 4] : 0.f, dl = i + 4 < ld ? d[i + 4] : 0.f;
      const float ev[5] = {e4.x, e4.y, e4.z, e4.w, el}, dv[4] = {d4.y, d4.z, d4.w, dl};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (i + k + 1 < n) {
          const float ei = ev[k], en = ev[k + 1], dn = dv[k] - x;
          const bool swp = fabsf(a) < fabsf(ei);
          if (!swp && fabsf(a) < TINY) a = copysignf(TINY, a);
          const float mlt = __fdividef(swp ? a : ei, swp ? ei : a);
          sm[(i + k) * n] = make_float2(a, mlt);
          a = fmaf(-mlt, swp ? dn : b, swp ? b : dn);
          b = swp ? -mlt * en : en;
        }
      }
    }
    if (fabsf(a) < TINY) a = copysignf(TINY, a);
    const float ial = __fdividef(1.f, a);
    float f = 1.f;
    for (int it = 0; it < 2; ++it) {
      float r = it ? Xu[0] * f : eig_noise(n - 1, u);
      if (it) {                                    // forward elimination of the first vector
        float2 nx[AH];
#pragma unroll
        for (int k = 0; k < AH; ++k) nx[k] = sm[min(k, n - 1) * n];
        for (int i0 = 0; i0 + 1 < n; i0 += AH) {
          float2 cu[AH];
          float xv[AH], ev[AH];
#pragma unroll
          for (int k = 0; k < AH; ++k) {
            cu[k] = nx[k];
            xv[k] = Xu[min(i0 + k + 1, n - 1)] * f;
            ev[k] = fabsf(e[min(i0 + k, n - 1)]);
          }
#pragma unroll
          for (int k = 0; k < AH; ++k) nx[k] = sm[min(i0 + AH + k, n - 1) * n];
#pragma unroll
          for (int k = 0; k < AH; ++k) {
            if (i0 + k + 1 < n) {
              const bool swp = fabsf(cu[k].x) < ev[k];
              Xu[i0 + k] = swp ? xv[k] : r;
              r = fmaf(-cu[k].y, swp ? xv[k] : r, swp ? r : xv[k]);
            }
          }
        }
      }
      float x1 = r * ial, x2 = 0.f, nn = x1 * x1;
      Xu[n - 1] = x1;
      // rows n - 2 .. 0; row i also needs the pivot and the multiplier of row i - 1
      float2 nx[AH + 1];
#pragma unroll
      for (int k = 0; k <= AH; ++k) nx[k] = sm[max(n - 2 - k, 0) * n];
      for (int i0 = n - 2; i0 >= 0; i0 -= AH) {
        float2 cu[AH + 1];
        float y[AH], iu0[AH], u1[AH], u2[AH];
#pragma unroll
        for (int k = 0; k <= AH; ++k) cu[k] = nx[k];
#pragma unroll
        for (int k = 0; k <= AH; ++k) nx[k] = sm[max(i0 - AH - k, 0) * n];
#pragma unroll
        for (int k = 0; k < AH; ++k) {             // all that does not wait for the row before
          const int i = max(i0 - k, 0);
          const float ei = e[i], en = e[i + 1], ep = e[max(i - 1, 0)], dn = d[i + 1] - x;
          const bool swp = fabsf(cu[k].x) < fabsf(ei), swq = i > 0 && fabsf(cu[k + 1].x) < fabsf(ep);
          y[k] = it ? Xu[i] : eig_noise(i, u);
          iu0[k] = __fdividef(1.f, swp ? ei : cu[k].x);
          u1[k] = swp ? dn : (swq ? -cu[k + 1].y * ei : ei);
          u2[k] = swp ? en : 0.f;
        }
#pragma unroll
        for (int k = 0; k < AH; ++k) {
          if (i0 - k >= 0) {
            const float xi = fmaf(-u1[k], x1, fmaf(-u2[k], x2, y[k])) * iu0[k];
            Xu[i0 - k] = xi;
            nn = fmaf(xi, xi, nn);
            x2 = x1;
            x1 = xi;
          }
        }
      }
      f = rsqrtf(nn);
    }
    inorm[u] = f;
  }
  tm.sync();
}

// X <- H_0 ... H_{n-3} X diag(inorm): a 4-lane group holds NV vectors in registers, each
// lane NC chunks of four consecutive components (16 c + 4 lane ..).
template <int NC, int NV, bool XS, class Team>
__device__ __noinline__ void eig_back(const Team tm, const float* A, const float* V0, const float* tau, int n, float* X,
                                      int ld, const float* inorm) {
  EIG_SHARED(A);
  EIG_SHARED(V0);
  EIG_SHARED(tau);
  EIG_SHARED(inorm);
  if (XS) EIG_SHARED(X);
  const int tr = tm.rank(), ts = tm.size(), lane = threadIdx.x & 31;
  const int grp = tr >> 2, ngrp = ts >> 2, gl = tr & 3;
  const unsigned gmask = 0xfu << (lane & 28);
  for (int u0 = grp; u0 < n; u0 += NV * ngrp) {
    float4 z[NV][NC];
#pragma unroll
    for (int q = 0; q < NV; ++q) {
      const int u = u0 + q * ngrp;
      const float f = u < n ? inorm[u] : 0.f;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (u < n && 16 * c + 4 * gl < ld) v = *reinterpret_cast<const float4*>(X + u * ld + 16 * c + 4 * gl);
        z[q][c] = make_float4(v.x * f, v.y * f, v.z * f, v.w * f);
      }
    }
    for (int j = n - 3; j >= 0; --j) {
      const float t = tau[j];
      const float* Aj = (j > 0 ? A + (j - 1) * ld : V0) + 4 * gl;   // reflector j
      float4 rv[NC];
      float2 ds[NV];
      float dt[NV];
#pragma unroll
      for (int q = 0; q < NV; ++q) ds[q] = make_float2(0.f, 0.f);
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        rv[c] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (16 * c + 4 * gl < ld) rv[c] = *reinterpret_cast<const float4*>(Aj + 16 * c);
      }
#pragma unroll
      for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int q = 0; q < NV; ++q)
          ds[q] = ffma2(make_float2(rv[c].x, rv[c].y), make_float2(z[q][c].x, z[q][c].y),
                        ffma2(make_float2(rv[c].z, rv[c].w), make_float2(z[q][c].z, z[q][c].w), ds[q]));
#pragma unroll
      for (int q = 0; q < NV; ++q) dt[q] = ds[q].x + ds[q].y;
#pragma unroll
      for (int o = 2; o > 0; o >>= 1)
#pragma unroll
        for (int q = 0; q < NV; ++q) dt[q] += __shfl_xor_sync(gmask, dt[q], o);
#pragma unroll
      for (int q = 0; q < NV; ++q) {
        const float g = -t * dt[q];
        const float2 g2 = make_float2(g, g);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const float2 lo = ffma2(g2, make_float2(rv[c].x, rv[c].y), make_float2(z[q][c].x, z[q][c].y));
          const float2 hi = ffma2(g2, make_float2(rv[c].z, rv[c].w), make_float2(z[q][c].z, z[q][c].w));
          z[q][c] = make_float4(lo.x, lo.y, hi.x, hi.y);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < NV; ++q) {
      const int u = u0 + q * ngrp;
#pragma unroll
      for (int c = 0; c < NC; ++c)
        if (u < n && 16 * c + 4 * gl < ld) *reinterpret_cast<float4*>(X + u * ld + 16 * c + 4 * gl) = z[q][c];
    }
  }
  tm.sync();
}

// Vectors of eigenvalues closer than EIG_CLUSTER (ten times their resolution) to the one before come out of
// inverse iteration nearly parallel: Gram-Schmidt, twice, within such a run.  Runs are rare
// and short (the eigenvalues at the rounding level of G); the first warp does it alone.
constexpr float EIG_CLUSTER = 2e-6f;
template <bool XS, class Team>
__device__ __noinline__ void eig_clusters(const Team tm, const float* lam, int n, float* X, int ld) {
  EIG_SHARED(lam);
  if (XS) EIG_SHARED(X);
  const int tr = tm.rank(), lane = threadIdx.x & 31;
  if (tr < 32) {
    int start = 0;
    for (int u = 1; u < n; ++u) {
      if (lam[u - 1] - lam[u] >= EIG_CLUSTER) {
        start = u;
        continue;
      }
      float* y = X + u * ld;
      for (int rep = 0; rep < 2; ++rep) {
        for (int w = start; w < u; ++w) {
          const float* x = X + w * ld;
          float dt = 0.f;
          for (int i = lane; i < n; i += 32) dt = fmaf(x[i], y[i], dt);
          dt = warp_sum_f(dt);
          for (int i = lane; i < n; i += 32) y[i] = fmaf(-dt, x[i], y[i]);
          __syncwarp();
        }
        float nn = 0.f;
        for (int i = lane; i < n; i += 32) nn = fmaf(y[i], y[i], nn);
        nn = rsqrtf(fmaxf(warp_sum_f(nn), 1e-20f));
        for (int i = lane; i < n; i += 32) y[i] *= nn;
        __syncwarp();
      }
    }
  }
  tm.sync();
}

// ----------------------------------------------------------------------------- orthonormalisation
// E = I - X X^T over the vectors (rows of X; n x n, pad entries zero); returns the largest |entry|.
template <bool XS, class Team>
__device__ __noinline__ float eig_defect(const Team tm, const float* X, int n, int ld, float* E) {
  EIG_SHARED(E);
  if (XS) EIG_SHARED(X);
  const int tr = tm.rank(), ts = tm.size();
  const int nq = (n + 3) >> 2, ntile = nq * (nq + 1) / 2;
  float worst = 0.f;
  for (int x = tr; x < n * (ld - n); x += ts) E[(x / (ld - n)) * ld + n + x % (ld - n)] = 0.f;
  for (int t = tr; t < ntile; t += ts) {
    int jq = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
    while (jq * (jq + 1) / 2 > t) --jq;
    while ((jq + 1) * (jq + 2) / 2 <= t) ++jq;
    const int iq = t - jq * (jq + 1) / 2;
    float2 acc[4][4];
    const float4* xi[4];
    const float4* xj[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      xi[a] = reinterpret_cast<const float4*>(X + min(4 * iq + a, n - 1) * ld);
      xj[a] = reinterpret_cast<const float4*>(X + min(4 * jq + a, n - 1) * ld);
#pragma unroll
      for (int b = 0; b < 4; ++b) acc[a][b] = make_float2(0.f, 0.f);
    }
    for (int r = 0; r < nq; ++r) {
      float4 va[4], vb[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        va[a] = xi[a][r];
        vb[a] = xj[a][r];
      }
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b)
          acc[a][b] = ffma2(make_float2(va[a].x, va[a].y), make_float2(vb[b].x, vb[b].y),
                            ffma2(make_float2(va[a].z, va[a].w), make_float2(vb[b].z, vb[b].w), acc[a][b]));
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int i = 4 * iq + a, j = 4 * jq + b;
        if (i < n && j < n && i <= j) {
          const float v = (i == j ? 1.f : 0.f) - (acc[a][b].x + acc[a][b].y);
          worst = max_nan(worst, fabsf(v));
          E[i * ld + j] = v;
          E[j * ld + i] = v;
        }
      }
  }
  if (!(worst <= 1e30f)) worst = 1e30f;            // a NaN too
  return tm.max(worst);                            // ends with a team barrier
}
// out (row stride lo = ld) = X + E X / 2 over the vectors
template <bool XS, class Team>
__device__ __noinline__ void eig_correct(const Team tm, const float* X, const float* E, int n, int ld, float* out, int lo) {
  EIG_SHARED(E);
  if (XS) EIG_SHARED(X);
  const int tr = tm.rank(), ts = tm.size();
  const int nq = (n + 3) >> 2, nc = lo >> 2;
  for (int t = tr; t < nq * nc; t += ts) {
    const int iq = t / nc, jq = t % nc;            // vectors 4 iq.., components 4 jq.. (pad components zero)
    float2 acc[4][2];
#pragma unroll
    for (int a = 0; a < 4; ++a) acc[a][0] = acc[a][1] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int k = 0; k < n; ++k) {
      const float4 x = *reinterpret_cast<const float4*>(X + k * ld + 4 * jq);
      const float4 y = *reinterpret_cast<const float4*>(E + k * ld + 4 * iq);
      const float2 x0 = make_float2(x.x, x.y), x1 = make_float2(x.z, x.w);
      const float ya[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const float2 y2 = make_float2(ya[a], ya[a]);
        acc[a][0] = ffma2(y2, x0, acc[a][0]);
        acc[a][1] = ffma2(y2, x1, acc[a][1]);
      }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int i = 4 * iq + a;
      if (i < n) {
        const float4 x = *reinterpret_cast<const float4*>(X + i * ld + 4 * jq);   // pad components are zero
        *reinterpret_cast<float4*>(out + i * lo + 4 * jq) =
            make_float4(fmaf(0.5f, acc[a][0].x, x.x), fmaf(0.5f, acc[a][0].y, x.y), fmaf(0.5f, acc[a][1].x, x.z),
                        fmaf(0.5f, acc[a][1].y, x.w));
      }
    }
  }
  tm.sync();
}
// 16-byte copies, `words` a multiple of 4 and both sides aligned
template <class Team>
__device__ __forceinline__ void eig_copy(const Team& tm, const float* from, int words, float* to) {
  const float4* f = reinterpret_cast<const float4*>(from);
  float4* t = reinterpret_cast<float4*>(to);
#pragma unroll 4
  for (int x = tm.rank(); x < words / 4; x += tm.size()) t[x] = f[x];
  tm.sync();
}

template <bool XS, class Team>
__device__ int eig_start_at(const Team tm, const uint4* At, int m, int n, float* A, float* X, float* V, float* Xg,
                            float* lamg, float2* Sg, float* trace) {
  const int tr = tm.rank(), ts = tm.size();
  const int ld = eig_ld(n);
  float* W = V + 2 * ld;
  float* P = W + ld;
  float* d = P + 2 * ld;
  float* e = d + ld;
  float* tau = e + ld;
  float* lam = tau + ld;
  float* inorm = lam + ld;
  eig_gram(tm, At, m, n, A, ld);
  if (tr < 32) {                                   // (this warp takes part in the first barrier of the reduction)
    float t = 0.f;
    for (int i = tr; i < n; i += 32) t += A[i * ld + i];
    t = warp_sum_f(t);
    if (tr == 0) *trace = t;
  }
  int coupled = 0;
  for (int x = tr; x < n * n; x += ts) {
    const int i = x / n, j = x - i * n;
    const float g = A[i * ld + j];
    coupled |= i < j && !(g * g <= 1e-12f * A[i * ld + i] * A[j * ld + j]);
  }
  if (!tm.any(coupled)) return 5;
  eig_tridiag(tm, A, n, ld, V, W, P, d, e, tau, inorm + ld);
  const float sc = eig_values(tm, d, e, n, ld, reinterpret_cast<float2*>(P), lam);
  for (int x = tr; x < n * (ld - n); x += ts) X[(x / (ld - n)) * ld + n + x % (ld - n)] = 0.f;
  eig_vectors<XS>(tm, d, e, lam, n, X, ld, Sg, inorm);
  if (n <= 16) eig_back<1, 2, XS>(tm, A, V, tau, n, X, ld, inorm);
  else if (n <= 48) eig_back<3, 2, XS>(tm, A, V, tau, n, X, ld, inorm);
  else if (n <= 80) eig_back<5, 2, XS>(tm, A, V, tau, n, X, ld, inorm);
  else eig_back<EIG_MAXN / 16, 1, XS>(tm, A, V, tau, n, X, ld, inorm);
  eig_clusters<XS>(tm, lam, n, X, ld);
  const float isc = __fdividef(1.f, sc);
  for (int u = tr; u < n; u += ts) lamg[u] = fmaxf(lam[u] * isc, 0.f);
  // Newton-Schulz X <- (3 I - X X^T) X / 2: the defect of inverse iteration is 1e-2 at most for
  // well separated eigenvalues, up to 1 in clusters
  for (int it = 0; it < 10; ++it) {
    const float worst = eig_defect<XS>(tm, X, n, ld, A);
    if (!(worst < 1.5f)) return 3;
    eig_correct<XS>(tm, X, A, n, ld, Xg, ld);
    if (worst < 5e-4f) return 0;                   // the defect after the correction is its square
    eig_copy(tm, Xg, n * ld, X);
  }
  return 3;
}
// Approximate eigenvectors and eigenvalues of B^T B.  At: the digits of B^T (eig_digits); arena:
// `words` floats of shared memory (16-byte aligned); Xg (n x ld floats, one vector per
// row, pad components zero, eigenvalues descending) and lamg (n floats) receive the result, Sg (n x
// n pairs) and Xalt (n x ld floats, for X where the arena only holds A) are scratch, all
// in global memory; *trace gets the sum of all eigenvalues.  Returns 0, 1 if the block does not fit (no result), 3 if X is not
// orthonormal in the end (the eigenvalues hold), or 5 if the columns of B are orthogonal to FP32 already (no result).
template <class Team>
__device__ int eig_start(const Team& tm, const uint4* At, int m, int n, float* arena, int words, float* Xg, float* lamg,
                         float2* Sg, float* Xalt, float* trace) {
  const int ld = eig_ld(n);
  if (n > EIG_MAXN || n * ld + eig_vec_floats(n) > words) return 1;
  if (2 * n * ld + eig_vec_floats(n) <= words)
    return eig_start_at<true>(tm, At, m, n, arena, arena + n * ld, arena + 2 * n * ld, Xg, lamg, Sg, trace);
  return eig_start_at<false>(tm, At, m, n, arena, Xalt, arena + n * ld, Xg, lamg, Sg, trace);
}

// ----------------------------------------------------------------------------- refinement
// W (column k at k ldw, rows padded to 16) = B X from the digits of B (A) and of X (D): NA, NB, NS
// as for mma_tile.
template <int NA, int NB, int NS, class Team>
__device__ __noinline__ void eig_bx(const Team tm, const uint4* A, const uint2* D, int m, int n, int kp, double* W,
                                    int ldw) {
  const int lane = threadIdx.x & 31, warp = tm.rank() >> 5, nw = tm.size() >> 5;
  const int mt = pad16(m) >> 4, KT = pad16(n) >> 4, JT = kp >> 3, g = lane >> 2, t2 = 2 * (lane & 3);
  for (int t = warp; t < mt * JT; t += nw) {
    const int it = t % mt, j = t / mt;
    float acc[NS - 1][4];
    mma_tile<NA, NB, NS>(A, D, it, j, KT, JT, lane, acc);
#pragma unroll
    for (int q = 0; q < 4; ++q) W[(8 * j + t2 + (q & 1)) * ldw + 16 * it + g + 8 * (q >> 1)] = mma_value<NS>(acc, q, 0);
  }
  tm.sync();
}
// R (column k at k ld) = B^T W - X lambda from the digits of B^T (At) and of W (D, scaled by 2^-exs[k]).
template <int NA, int NB, int NS, class Team>
__device__ __noinline__ void eig_residual(const Team tm, const uint4* At, const uint2* D, int m, int n, int kp,
                                          const double* Xd, int ldx, const double* lk, const int* exs, float* R,
                                          int ld) {
  EIG_SHARED(lk);
  EIG_SHARED(R);
  const int lane = threadIdx.x & 31, warp = tm.rank() >> 5, nw = tm.size() >> 5;
  const int nt = pad16(n) >> 4, KT = pad16(m) >> 4, JT = kp >> 3, g = lane >> 2, t2 = 2 * (lane & 3);
  for (int t = warp; t < nt * JT; t += nw) {
    const int it = t % nt, j = t / nt;
    double xv[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) xv[q] = Xd[(8 * j + t2 + (q & 1)) * ldx + 16 * it + g + 8 * (q >> 1)];
    float acc[NS - 1][4];
    mma_tile<NA, NB, NS>(At, D, it, j, KT, JT, lane, acc);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int k = 8 * j + t2 + (q & 1), c = 16 * it + g + 8 * (q >> 1);
      const float r = (float)fma(-lk[k], xv[q], mma_value<NS>(acc, q, exs[k]));
      if (c < ld) R[k * ld + c] = c < n ? r : 0.f;
    }
  }
  tm.sync();
}
// |column k|^2 of V (column k at k ldv, length K): eight lanes per column; f(k, value) runs on one lane.
template <class Team, class F>
__device__ __forceinline__ void eig_norms(const Team& tm, const double* V, int ldv, int K, int kp, F f) {
  const int lane = threadIdx.x & 31, warp = tm.rank() >> 5, nw = tm.size() >> 5;
  for (int t = warp; t < kp / 4; t += nw) {
    const int k = 4 * t + (lane >> 3);
    const double* src = V + (size_t)k * ldv;
    double l = 0.0;
#pragma unroll 4
    for (int r = lane & 7; r < K; r += 8) l = fma(src[r], src[r], l);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if ((lane & 7) == 0) f(k, l);
  }
}
// T (row i at i kp) = X R / (lambda_k - lambda_i), half the norm's defect ek on the diagonal: lanes are
// vectors i.  lk: the eigenvalues of the kept vectors, lh the same in FP32; lam: those of the discarded vectors, FP32
// (1e-6 lam[0] or better): a correction leaves 1e-6 lam[0] / |lambda_k - lambda_i| of itself along those.  Returns the largest |entry|, along
// discarded vectors closer than 1e-3 lam[0] times 1e-3 lam[0] / |lambda_k - lambda_i|.
template <class Team>
__device__ __noinline__ float eig_angles(const Team tm, const float* X, const float* R, int n, int ld, int kc, int kp,
                                         const double* lk, const float* lh, const float* ek, const float* lam,
                                         float* T) {
  EIG_SHARED(R);
  EIG_SHARED(lk);
  EIG_SHARED(lh);
  EIG_SHARED(ek);
  EIG_SHARED(lam);
  EIG_SHARED(T);
  const int lane = threadIdx.x & 31, warp = tm.rank() >> 5, nw = tm.size() >> 5;
  const int rc = (n + 31) >> 5, kcn = kp / EIG_TC, nq = (n + 3) >> 2;
  float worst = 0.f;
  for (int t = warp; t < rc * kcn; t += nw) {
    const int i = (t % rc) * 32 + lane, k0 = (t / rc) * EIG_TC;
    float s[EIG_TC];
    float2 s2[EIG_TC];
#pragma unroll
    for (int q = 0; q < EIG_TC; ++q) s2[q] = make_float2(0.f, 0.f);
    const float4* xp = reinterpret_cast<const float4*>(X + min(i, n - 1) * ld);
    const float4* rp = reinterpret_cast<const float4*>(R + k0 * ld);
    const int l4 = ld >> 2;
#pragma unroll 2
    for (int c = 0; c < nq; ++c) {
      const float4 x = xp[c];
#pragma unroll
      for (int q = 0; q < EIG_TC; ++q) {
        const float4 r = rp[q * l4 + c];
        s2[q] = ffma2(make_float2(x.x, x.y), make_float2(r.x, r.y), ffma2(make_float2(x.z, x.w), make_float2(r.z, r.w), s2[q]));
      }
    }
#pragma unroll
    for (int q = 0; q < EIG_TC; ++q) s[q] = s2[q].x + s2[q].y;
    if (i < n) {
      const double li = i < kc ? lk[i] : 0.0;
      const float near = i < kc ? 0.f : 1e-3f * lam[0];
      float o[EIG_TC];
#pragma unroll
      for (int q = 0; q < EIG_TC; ++q) {
        const int k = k0 + q;
        float v = 0.f, w = 1.f;
        if (k < kc) {
          if (i == k) {
            v = 0.5f * ek[k];
          } else {
            const float den = i < kc ? (float)(lk[k] - li) : lh[k] - lam[i];
            v = den != 0.f ? __fdividef(s[q], den) : (s[q] == 0.f ? 0.f : 1e30f);
            if (fabsf(den) < near) w = __fdividef(near, fabsf(den));
          }
          worst = max_nan(worst, w * fabsf(v));
        }
        o[q] = v;
      }
      *reinterpret_cast<float4*>(T + i * kp + k0) = make_float4(o[0], o[1], o[2], o[3]);
      *reinterpret_cast<float4*>(T + i * kp + k0 + 4) = make_float4(o[4], o[5], o[6], o[7]);
    }
  }
  if (!(worst <= 1e30f)) worst = 1e30f;            // a NaN too
  return tm.max(worst);
}
// T (row i at i kp, kc rows) = half the defect of the kept vectors' inner products, (I - X^T X) / 2: eight
// lanes per pair.
template <class Team>
__device__ __noinline__ void eig_orth(const Team tm, const double* Xd, int ldx, int n, int kc, int kp, float* T) {
  EIG_SHARED(T);
  const int gl = tm.rank() & 7, ng = tm.size() >> 3, np = kc * (kc + 1) / 2;
  for (int x = tm.rank(); x < kc * kp; x += tm.size()) T[x] = 0.f;   // (columns beyond kc)
  tm.sync();
  for (int p0 = 0; p0 < np; p0 += ng) {
    const int p = min(p0 + (tm.rank() >> 3), np - 1);
    const float f = 8.f * (float)p + 1.f;
    int k = (int)((f * rsqrtf(f) - 1.f) * 0.5f);
    while (k * (k + 1) / 2 > p) --k;
    while ((k + 2) * (k + 1) / 2 <= p) ++k;
    const int i = p - k * (k + 1) / 2;
    const double* a = Xd + (size_t)i * ldx;
    const double* b = Xd + (size_t)k * ldx;
    double l = 0.0;
#pragma unroll 2
    for (int r = gl; r < n; r += 8) l = fma(a[r], b[r], l);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (gl == 0) {
      const float e = 0.5f * (float)((i == k ? 1.0 : 0.0) - l);
      T[i * kp + k] = e;
      T[k * kp + i] = e;
    }
  }
  tm.sync();
}
// Xd (column k at k ldx) += X^T T (nv rows), and the FP32 vectors Xg (row k at k ld) follow: lanes are components.
template <class Team>
__device__ __noinline__ void eig_update(const Team tm, const float* X, const float* T, int nv, int n, int ld, int kc,
                                        int kp, double* Xd, int ldx, float* Xg) {
  EIG_SHARED(T);
  const int lane = threadIdx.x & 31, warp = tm.rank() >> 5, nw = tm.size() >> 5;
  const int rc = (n + 31) >> 5, kcn = kp / EIG_TC;
  for (int t = warp; t < rc * kcn; t += nw) {
    const int i = (t % rc) * 32 + lane, k0 = (t / rc) * EIG_TC, ic = min(i, n - 1);
    float2 s2[EIG_TC / 2];
    double xv[EIG_TC];
#pragma unroll
    for (int q = 0; q < EIG_TC; ++q) xv[q] = Xd[(size_t)(k0 + q) * ldx + ic];
#pragma unroll
    for (int q = 0; q < EIG_TC / 2; ++q) s2[q] = make_float2(0.f, 0.f);
    const float* xp = X + ic;
#pragma unroll 4
    for (int v = 0; v < nv; ++v) {
      const float x = xp[v * ld];
      const float2 x2 = make_float2(x, x);
      const float4 ra = *reinterpret_cast<const float4*>(T + v * kp + k0);
      const float4 rb = *reinterpret_cast<const float4*>(T + v * kp + k0 + 4);
      s2[0] = ffma2(x2, make_float2(ra.x, ra.y), s2[0]);
      s2[1] = ffma2(x2, make_float2(ra.z, ra.w), s2[1]);
      s2[2] = ffma2(x2, make_float2(rb.x, rb.y), s2[2]);
      s2[3] = ffma2(x2, make_float2(rb.z, rb.w), s2[3]);
    }
    const float s[EIG_TC] = {s2[0].x, s2[0].y, s2[1].x, s2[1].y, s2[2].x, s2[2].y, s2[3].x, s2[3].y};
    if (i < n) {
#pragma unroll
      for (int q = 0; q < EIG_TC; ++q) {
        const double v = xv[q] + (double)s[q];
        Xd[(size_t)(k0 + q) * ldx + i] = v;
        if (k0 + q < kc) Xg[(k0 + q) * ld + i] = X[(k0 + q) * ld + i] + s[q];
      }
    }
  }
  tm.sync();
}

// |B - W X^T|^2 for the kc columns of W = B X, of which Wf has the digits over 2^ex as fragments of W and Xf those of X
// (eig_digits): what the other singular values weigh, without the cancellation of a difference of norms (down to
// 1e-4 of the block's: 2e-11 of the weight with double-float vectors, 1e-12 in FP64).  B = raw / 2^e with
// inv = 2^-e, column-major.  tsum: 2 pad16(m) pad16(n) / 256 doubles of the team's memory.  The same on every
// thread, and the same sum whatever the team's size.
template <class Team>
__device__ __noinline__ double eig_rest(const Team tm, const uint4* Wf, const uint4* Xf, int ex, const double* raw,
                                        double inv, int m, int n, int kc, double* tsum) {
  const int lane = threadIdx.x & 31, warp = tm.rank() >> 5, nw = tm.size() >> 5;
  const int mt = pad16(m) >> 4, jt = (n + 7) >> 3, KT = pad16(kc) >> 4, g = lane >> 2, t2 = 2 * (lane & 3);
  for (int t = warp; t < mt * jt; t += nw) {
    const int it = t % mt, j8 = t / mt;
    float acc[EIG_DIG][4];
#pragma unroll
    for (int o = 0; o < EIG_DIG; ++o)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[o][q] = 0.f;
    for (int k = 0; k < KT; ++k) {
      const uint4* ap = Wf + (size_t)(it * KT + k) * EIG_DIG * 32 + lane;
      const uint4* bp = Xf + (size_t)((j8 >> 1) * KT + k) * EIG_DIG * 32 + lane;
      uint4 a[EIG_DIG];
      uint2 b[EIG_DIG];
#pragma unroll
      for (int s = 0; s < EIG_DIG; ++s) {
        a[s] = ap[s * 32];
        const uint4 v = bp[s * 32];
        b[s] = (j8 & 1) ? make_uint2(v.y, v.w) : make_uint2(v.x, v.z);
      }
#pragma unroll
      for (int i = 0; i < EIG_DIG; ++i)
#pragma unroll
        for (int s = 0; s < EIG_DIG; ++s)
          if (i + s < EIG_DIG) mma_bf16(acc[i + s], a[i], b[s]);
    }
    double sum = 0.0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = 16 * it + g + 8 * (q >> 1), c = 8 * j8 + t2 + (q & 1);
      const double d = r < m && c < n ? fma(raw[(size_t)c * m + r], inv, -mma_value<EIG_DIG + 1>(acc, q, ex)) : 0.0;
      sum = fma(d, d, sum);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) tsum[t] = sum;
  }
  tm.sync();
  double sum = 0.0;
  for (int t = lane; t < mt * jt; t += 32) sum += tsum[t];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  return sum;
}

// Refines the first kc vectors of Xg (n x ld, one per row; updated) as described at the top.  A, At: the
// digits of B and B^T; lam0 the approximate eigenvalues.  Outputs: Wout (column j at j m), Qout
// (column j at j n) in FP64, the singular values in sig[0..kc).  Wd, Xd (kp columns of length m
// and n padded to 16), Dg (digits of either) and Xalt (n x ld floats) are global
// scratch, used where the arena is too small.  *rest (if wanted) gets eig_rest of the block raw / scale (A and At are
// overwritten for it).  Returns 0, or 1 if the corrections do not converge or the block does not fit.
template <class Team>
__device__ int eig_refine(const Team& tm, uint4* A, uint4* At, int m, int n, int kc, float* Xg,
                          const float* lam0, float* arena, int words, double* Wd, double* Xd, uint2* Dg, float* Xalt,
                          double* Wout, double* Qout, double* sig, double scale, const double* raw, double* rest) {
  const int tr = tm.rank(), ts = tm.size();
  const int ld = eig_ld(n), kp = eig_kp(kc), m16 = pad16(m), n16 = pad16(n);
  // arena: lk (kp doubles), lh, ek and exs (kp), lam (ld), R (kp x ld), then the digits or, after them, T
  // (n x kp) and X (n x ld)
  const int fix = 5 * kp + ld + kp * ld, dig = m16 * kp * EIG_DIG / 2, tx = n * kp;
  if (eig_refine_words(n, kc) > words) return 1;
  double* lk = reinterpret_cast<double*>(arena);
  float* lh = arena + 2 * kp;
  float* ek = lh + kp;
  int* exs = reinterpret_cast<int*>(ek + kp);
  float* lam = ek + 2 * kp;
  float* R = lam + ld;
  float* T = R + kp * ld;
  uint2* D = fix + dig <= words ? reinterpret_cast<uint2*>(T) : Dg;
  const bool xin = fix + tx + n * ld <= words;
  float* X = xin ? T + tx : Xalt;
  // what is left behind the larger of the two takes the columns themselves
  int at = fix + max(fix + dig <= words ? dig : 0, tx + (xin ? n * ld : 0));
  if (at + 2 * n16 * kp <= words) {
    Xd = reinterpret_cast<double*>(arena + at);
    at += 2 * n16 * kp;
  }
  if (at + 2 * m16 * kp <= words) Wd = reinterpret_cast<double*>(arena + at);
  for (int x = tr; x < n16 * kp; x += ts) {
    const int k = x / n16, c = x % n16;
    float v = (k < kc && c < n) ? Xg[k * ld + c] : 0.f;
    // four digits carry the start vectors: entries below 2^-7 are rounded to 2^-30
    if (fabsf(v) < 0.0078125f) v = __fsub_rn(__fadd_rn(v, 0.01171875f), 0.01171875f);
    Xd[x] = (double)v;
  }
  for (int x = tr; x < n; x += ts) lam[x] = lam0[x];
  tm.sync();
  for (int it = 0; it < 6; ++it) {
    // the first correction starts from 1e-6 and needs 1e-10: six digits of B, four of X
    if (it == 0) {
      eig_digits_cols<4>(tm, Xd, n16, n, kp, nullptr, D);
      eig_bx<6, 4, 7>(tm, A, D, m, n, kp, Wd, m16);
    } else {
      eig_digits_cols<EIG_DIG>(tm, Xd, n16, n, kp, nullptr, D);
      eig_bx<EIG_DIG, EIG_DIG, EIG_DIG + 1>(tm, A, D, m, n, kp, Wd, m16);
    }
    eig_norms(tm, Wd, m16, m, kp, [&](int k, double l) {
      lk[k] = l;
      lh[k] = (float)l;
      exs[k] = (((__double2hiint(l) >> 20) & 2047) - 1023) >> 1;     // |w| < 2^(1 + exs); a padding column -512
    });
    eig_norms(tm, Xd, n16, n, kp, [&](int k, double l) { ek[k] = (float)(1.0 - l); });
    tm.sync();
    if (it == 0) {
      eig_digits_cols<6>(tm, Wd, m16, m, kp, exs, D);
      eig_residual<6, 6, 7>(tm, At, D, m, n, kp, Xd, n16, lk, exs, R, ld);
    } else {
      eig_digits_cols<EIG_DIG>(tm, Wd, m16, m, kp, exs, D);
      eig_residual<EIG_DIG, EIG_DIG, EIG_DIG + 1>(tm, At, D, m, n, kp, Xd, n16, lk, exs, R, ld);
    }
    eig_copy(tm, Xg, n * ld, X);
    const float worst = eig_angles(tm, X, R, n, ld, kc, kp, lk, lh, ek, lam, T);
    if (!(worst < 0.25f)) return 1;
    eig_update(tm, X, T, n, n, ld, kc, kp, Xd, n16, Xg);
    if (worst <= EIG_ACCEPT) break;
    if (it == 5) return 1;
  }
  // The kept vectors orthonormal to the working precision: what is left of the corrections' products, and the
  // rounding of R over the differences of the eigenvalues, which differs in T_ik and T_ki.
  eig_orth(tm, Xd, n16, n, kc, kp, T);
  eig_copy(tm, Xg, kc * ld, X);
  eig_update(tm, X, T, kc, n, ld, kc, kp, Xd, n16, Xg);
  eig_digits_cols<EIG_DIG>(tm, Xd, n16, n, kp, nullptr, D);
  eig_bx<EIG_DIG, EIG_DIG, EIG_DIG + 1>(tm, A, D, m, n, kp, Wd, m16);
  eig_norms(tm, Wd, m16, m, kp, [&](int k, double l) {
    if (k < kc) sig[k] = sqrt(l) * scale;
  });
  for (int x = tr; x < m * kc; x += ts) Wout[x] = Wd[(size_t)(x / m) * m16 + x % m];
  for (int x = tr; x < n * kc; x += ts) Qout[x] = Xd[(size_t)(x / n) * n16 + x % n];
  if (!rest || kc == n) {
    tm.sync();
    return 0;
  }
  int ex = exs[0];
  for (int k = 1; k < kc; ++k) ex = max(ex, exs[k]);
  tm.sync();
  eig_digits(tm, Wout, m, kc, ex, A, nullptr);
  eig_digits(tm, Qout, n, kc, 0, At, nullptr);
  *rest = eig_rest(tm, A, At, ex, raw, 1.0 / scale, m, n, kc, reinterpret_cast<double*>(arena));
  tm.sync();
  return 0;
}

}  // namespace
}  // namespace tnqe
