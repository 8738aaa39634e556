// FP64 combinations of n = 64 elements on split products (lqt_split.cuh), one
// CTA of 512 threads per combination.
//
// What bounds it: in FP64 a full combination is 2.0 M multiply-adds, 500 us on
// one SM's FP64 pipe (820 us as measured, with the barriers of the LU).  Here
// its fourteen 64^3 products are FP16 tensor-core products of seven digits.  A
// full combination takes 0.24 ms, alone or 66 at once (ncu, 512 threads on an SM): the
// ALU pipe is 31% busy (splitting 8 k entries and assembling 4 k results a
// product), the FP64 pipe 24% (vectors), the
// tensor pipe 18%, and the warps wait on one another's digits and on shared
// memory.  Each entry is split once, by the warp that owns eight rows of the left
// or columns of the right operand, and the digits are kept in shared memory in
// fragment order; each of the sixteen warps then forms 16 x 16 outputs.  (Eight
// warps with the left digits in registers, split twice, took 27 k cycles a
// product against 23.7 k.)  W = I + C1 J2 is inverted in FP32 (Gauss-Jordan in
// registers, 64 k cycles) and refined by Newton steps, as for n = 16
// (lqt_warp16.cuh), with the FP64 elimination behind it where that does not
// converge, and in FP64 altogether in mixed units (lqt_split.cuh).
#pragma once

#include <cuda_runtime.h>

#include "lqt_split.cuh"
#include "lqt_team.cuh"
#include "lqt_warp16.cuh"

namespace lqt {
namespace s64 {

using split::C64;
constexpr int ND = C64::ND;
using team::Rec;
constexpr int N = 64;
constexpr int kThreads = 512;
constexpr int kLd = 66;  // row stride of the shared buffers (16-byte rows that start in different banks)
constexpr int kBuf = N * kLd;

// Shared memory of a CTA.
struct Shared {
  double W[kBuf], M[kBuf];
  double vec[8][N];
  uint4 dA[4 * 4 * ND * 32];  // (16 rows, 16-deep slab, digit, lane): an A fragment
  uint2 dB[8 * 4 * ND * 32];  // (8 columns, slab, digit, lane): a B fragment
  unsigned eB[8 * 8 * 32];    // exponents of the right operand's entries, two a word: (8 columns, word, lane)
  alignas(16) float col[2][N];
  float rowp[N], scale[N];
  unsigned cand[8];
  int pivot[N], step[N], rowE[N], colE[N];
  double red[kThreads / 32];
};

// Two 64 x 64 buffers (row stride kLd) of the CTA in global memory (L2).
struct Slot {
  double *T1, *K1;
};
constexpr int kSlotDoubles = 2 * kBuf;

// Entry k of vector v at p[v sv + k sk] (rows of a left operand, columns of a
// right one).
struct Mat {
  const double* p;
  int sv, sk;
};
__device__ __forceinline__ Mat rows_of(const double* p, int ld) { return {p, ld, 1}; }
__device__ __forceinline__ Mat cols_of(const double* p, int ld) { return {p, 1, ld}; }

// o(i, j) = sum_k a(i, k) b(k, j) + diag (i == j), or o -= the product
// (kSubtract), o at o[i ld + j].  o may be one of the operands.  Above the limit
// the product is formed in FP64, or given up (kTry: see product16).  Returns the
// largest biased exponent of the entries this warp set.
static __device__ __noinline__ int product64(Shared& sm, Mat a, Mat b, double* o, int ld, int diag, int store,
                                             int limit = split::kGradeLimit) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, c = 2 * (lane & 3);
  // warps 0 .. 7: rows 8 w + g of a; warps 8 .. 15: columns of b.  Entries k
  // = 16 s + c, c + 1, c + 8, c + 9 of the vector and its largest exponent.
  const bool left = warp < 8;
  const int blk = warp & 7;
  const int rb = warp >> 2, cb = warp & 3;
  int top = 0;
  bool graded = limit < 0;
  if (!graded) {
    unsigned xe[8];  // the entries' exponents, two a word
    int e = 0;
    const Mat m = left ? a : b;
    const int v = 8 * blk + g;
    const double* p = m.p + (int64_t)v * m.sv + c * m.sk;
    double x[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) x[q] = p[(16 * (q >> 2) + (q & 1) + 8 * ((q >> 1) & 1)) * m.sk];
    unsigned bits = 0;
#pragma unroll
    for (int q = 0; q < 16; q += 2) {
      const int e0 = split::biased_exp(x[q]), e1 = split::biased_exp(x[q + 1]);
      e = max(e, max(e0, e1));
      bits |= split::magnitude_bits(x[q]) | split::magnitude_bits(x[q + 1]);
      xe[q >> 1] = (unsigned)e0 | (unsigned)e1 << 16;
    }
    e = max(e, __shfl_xor_sync(0xffffffffu, e, 1));
    e = max(e, __shfl_xor_sync(0xffffffffu, e, 2));
    const bool odd = split::odd_vector(e, bits);
    if ((lane & 3) == 0) (left ? sm.rowE : sm.colE)[v] = e;
    if (!left) {
#pragma unroll
      for (int w = 0; w < 8; ++w) sm.eB[(blk * 8 + w) * 32 + lane] = xe[w];
    }
    // an A fragment's registers: rows g (k c .., k c + 8 ..), then rows g + 8
    uint2* d = left ? reinterpret_cast<uint2*>(sm.dA) + (((blk >> 1) * 4 * ND) * 32 + lane) * 2 + (blk & 1)
                    : sm.dB + (blk * 4 * ND) * 32 + lane;
    const int step = left ? 64 : 32;
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      const unsigned long long u0 = split::digits<C64>(x[4 * s], e), u1 = split::digits<C64>(x[4 * s + 1], e);
      const unsigned long long u2 = split::digits<C64>(x[4 * s + 2], e), u3 = split::digits<C64>(x[4 * s + 3], e);
#pragma unroll
      for (int i = 0; i < ND; ++i)
        d[(s * ND + i) * step] = make_uint2(split::digit_pair<C64>(u0, u1, i), split::digit_pair<C64>(u2, u3, i));
    }
    __syncthreads();
    // diagonal entry i = 8 blk + g: this lane of warp blk holds the k of row i that
    // the same lane of warp 8 + blk holds of column i
    int worst = 0;
    if (left) {
      unsigned term = 0;
#pragma unroll
      for (int w = 0; w < 8; ++w) term = __vmaxu2(term, xe[w] + sm.eB[(blk * 8 + w) * 32 + lane]);
      int t = max((int)(term & 0xffffu), (int)(term >> 16));
      t = max(t, __shfl_xor_sync(0xffffffffu, t, 1));
      t = max(t, __shfl_xor_sync(0xffffffffu, t, 2));
      worst = split::grade(e, sm.colE[8 * blk + g], t);
    }
    graded = __syncthreads_or(odd || worst > limit) != 0;
  }
  if (graded) {
    if (store == split::kTry) return split::kGraded;
    double s[2][4] = {};
#pragma unroll 1
    for (int k = 0; k < N; ++k)
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int i = 16 * rb + g + 8 * (q >> 1), j = 16 * cb + 8 * t + c + (q & 1);
          s[t][q] = fma(a.p[i * a.sv + k * a.sk], b.p[j * b.sv + k * b.sk], s[t][q]);
        }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int i = 16 * rb + g + 8 * (q >> 1), j = 16 * cb + 8 * t + c + (q & 1);
        const double v = s[t][q] + (i == j ? (double)diag : 0.0);
        top = max(top, split::biased_exp(v));
        double* w = o + (int64_t)i * ld + j;
        *w = store == split::kSubtract ? *w - v : v;
      }
    __syncthreads();
    return __reduce_max_sync(0xffffffffu, top);
  }
  const uint4* fa = sm.dA + rb * 4 * ND * 32 + lane;
#pragma unroll 1
  for (int t = 0; t < 2; ++t) {
    float acc[ND][4];
#pragma unroll
    for (int w = 0; w < ND; ++w)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[w][q] = 0.0f;
    const uint2* fb = sm.dB + (2 * cb + t) * 4 * ND * 32 + lane;
#pragma unroll 1
    for (int s = 0; s < 4; ++s) {
      uint2 bf[ND];
#pragma unroll
      for (int j = 0; j < ND; ++j) bf[j] = fb[(s * ND + j) * 32];
#pragma unroll
      for (int i = 0; i < ND; ++i) {
        const uint4 f = fa[(s * ND + i) * 32];
        const unsigned af[4] = {f.x, f.z, f.y, f.w};
#pragma unroll
        for (int j = 0; j < ND - i; ++j) split::mma16816(acc[i + j], af, bf[j].x, bf[j].y);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = 16 * rb + g + 8 * (q >> 1), j = 16 * cb + 8 * t + c + (q & 1);
      const double v =
          split::finish<C64>(split::to_int<C64>(acc, q), sm.rowE[i], sm.colE[j], i == j ? diag : 0);
      top = max(top, split::biased_exp(v));
      double* w = o + (int64_t)i * ld + j;
      *w = store == split::kSubtract ? *w - v : v;
    }
  }
  __syncthreads();
  return __reduce_max_sync(0xffffffffu, top);
}

// base + sum_l m(i, l) x(l) for row i = thread / 8 (x in shared memory), eight
// threads per row; every thread of the eight returns it.
__device__ __forceinline__ double matvec(Mat m, const double* x, double base) {
  const int i = threadIdx.x >> 3, q = threadIdx.x & 7;
  const double* p = m.p + (int64_t)i * m.sv + q * m.sk;
  double s = q == 0 ? base : 0.0, u = 0.0;
#pragma unroll
  for (int l = 0; l < 8; l += 2) {
    s = fma(p[8 * l * m.sk], x[8 * l + q], s);
    u = fma(p[8 * (l + 1) * m.sk], x[8 * (l + 1) + q], u);
  }
  s += u;
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  return s + __shfl_xor_sync(0xffffffffu, s, 4);
}

__device__ __forceinline__ float pick8(const float (&x)[8], int k) {
  const float a = (k & 1) ? x[1] : x[0], b = (k & 1) ? x[3] : x[2], c = (k & 1) ? x[5] : x[4],
              d = (k & 1) ? x[7] : x[6];
  const float e = (k & 2) ? b : a, f = (k & 2) ? d : c;
  return (k & 4) ? f : e;
}

// sm.M <- the FP32 inverse of sm.W: in-place Gauss-Jordan with partial
// pivoting; thread (j, q) owns rows 8 q .. 8 q + 7 of column j.  Rows are not
// exchanged: step k takes the largest entry of column k in the rows not taken
// yet, p_k, and in the end entry (p_k, j) is entry (k, p_j) of the inverse.
// Two barriers a step (column and candidates, then the pivot row).  False (in
// every thread) when a pivot is not above 2^-10 of its row's largest magnitude
// (at least 1) or not finite.
static __device__ __noinline__ bool inverse_f32(Shared& sm) {
  const int tid = threadIdx.x, j = tid & 63, q = tid >> 6;
  float m[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) m[r] = (float)sm.W[(8 * q + r) * kLd + j];
  {
    float s = 1.0f;
    const double* w = sm.W + (tid >> 3) * kLd + (tid & 7);
#pragma unroll
    for (int l = 0; l < 8; ++l) s = fmaxf(s, fabsf((float)w[8 * l]));
    s = fmaxf(s, __shfl_xor_sync(0xffffffffu, s, 1));
    s = fmaxf(s, __shfl_xor_sync(0xffffffffu, s, 2));
    s = fmaxf(s, __shfl_xor_sync(0xffffffffu, s, 4));
    if ((tid & 7) == 0) sm.scale[tid >> 3] = s;
  }
  bool ok = true;
  unsigned taken = 0;  // this thread's rows that were pivots
#pragma unroll 1
  for (int k = 0; k < N; ++k) {
    float* col = sm.col[k & 1];
    if (j == k) {
      unsigned best = 0;
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const unsigned key = (__float_as_uint(m[r]) & 0x7fffffc0u) | (unsigned)(63 - 8 * q - r);
        best = (taken >> r & 1u) ? best : max(best, key);
      }
      sm.cand[q] = best;
      reinterpret_cast<float4*>(col + 8 * q)[0] = make_float4(m[0], m[1], m[2], m[3]);
      reinterpret_cast<float4*>(col + 8 * q)[1] = make_float4(m[4], m[5], m[6], m[7]);
#pragma unroll
      for (int r = 0; r < 8; ++r) m[r] = 0.0f;  // column k of the inverse grows here
    }
    __syncthreads();
    unsigned best = sm.cand[tid & 7];
    best = max(best, __shfl_xor_sync(0xffffffffu, best, 1));
    best = max(best, __shfl_xor_sync(0xffffffffu, best, 2));
    best = max(best, __shfl_xor_sync(0xffffffffu, best, 4));
    const int p = 63 - (int)(best & 63u);
    if (q == (p >> 3)) sm.rowp[j] = j == k ? 1.0f : pick8(m, p & 7);
    const float d = col[p], sp = sm.scale[p];
    if (tid == 0) {
      sm.pivot[k] = p;
      sm.step[p] = k;
    }
    const float4 f0 = reinterpret_cast<const float4*>(col + 8 * q)[0];
    const float4 f1 = reinterpret_cast<const float4*>(col + 8 * q)[1];
    const float inv = __frcp_rn(d);
    ok = ok && fabsf(d) > 0x1p-10f * sp && fabsf(d) < 0x1p100f;
    __syncthreads();
    const float pr = sm.rowp[j] * inv;
    m[0] = fmaf(-f0.x, pr, m[0]);
    m[1] = fmaf(-f0.y, pr, m[1]);
    m[2] = fmaf(-f0.z, pr, m[2]);
    m[3] = fmaf(-f0.w, pr, m[3]);
    m[4] = fmaf(-f1.x, pr, m[4]);
    m[5] = fmaf(-f1.y, pr, m[5]);
    m[6] = fmaf(-f1.z, pr, m[6]);
    m[7] = fmaf(-f1.w, pr, m[7]);
    if (q == (p >> 3)) {
#pragma unroll
      for (int r = 0; r < 8; ++r) m[r] = r == (p & 7) ? pr : m[r];
      taken |= 1u << (p & 7);
    }
  }
  __syncthreads();
  const int pj = sm.pivot[j];
#pragma unroll
  for (int r = 0; r < 8; ++r) sm.M[sm.step[8 * q + r] * kLd + pj] = (double)m[r];
  __syncthreads();
  return ok;
}

// sm.M <- the inverse of sm.W by the FP64 elimination (the pivots and the
// SINGULAR test of team::lu_solve); the digit buffers are scratch.
static __device__ __noinline__ void inverse_f64(Shared& sm) {
  const int tid = threadIdx.x;
  double* Wc = reinterpret_cast<double*>(sm.dA);
  double* R = reinterpret_cast<double*>(sm.dB);
  double* fs = R + N * N;
  int* is = reinterpret_cast<int*>(fs + 2 * kThreads);
  static_assert(sizeof(sm.dB) >= (N * N + 2 * kThreads) * sizeof(double) + kThreads * sizeof(int), "scratch");
  for (int e = tid; e < N * N; e += kThreads) {
    Wc[e] = sm.W[(e >> 6) * kLd + (e & 63)];
    R[e] = (e >> 6) == (e & 63) ? 1.0 : 0.0;
  }
  __syncthreads();
  team::lu_solve<N, kThreads, N>(tid, Wc, R, fs, is);
  __syncthreads();
  for (int e = tid; e < N * N; e += kThreads) sm.M[(e >> 6) * kLd + (e & 63)] = R[e];
  __syncthreads();
}

// sm.M <- sm.W^-1: the FP32 inverse and Newton steps M <- M - M (W M - I) until
// the residual is below 2^-28 before the last step; where the residual does
// not shrink, the FP64 inverse and one step.  E (row stride kLd) is scratch;
// limit: split::kAllFp64 or the products' own.
__device__ __forceinline__ void inverse(Shared& sm, double* E, int limit) {
  constexpr int kExp1 = 1023;  // biased exponent of 1
  bool fast = limit >= 0 && inverse_f32(sm);
  int last = kExp1 - 1;
  for (int it = 0; it < 4; ++it) {
    if (!fast) inverse_f64(sm);
    const int top = product64(sm, rows_of(sm.W, kLd), cols_of(sm.M, kLd), E, kLd, -1, split::kSet, limit);
    // row sums: 64 entries below 2^(top - 1022)
    const bool done = __syncthreads_and(top <= kExp1 - 35) != 0 || !fast;
    const bool lost = __syncthreads_or(top > last - 3 || top > kExp1 - 7) != 0;
    if (!done && (lost || it == 3)) {
      fast = false;
      it = 2;
      continue;
    }
    last = top;
    product64(sm, rows_of(sm.M, kLd), cols_of(E, kLd), sm.M, kLd, 0, split::kSubtract,
              limit < 0 ? limit : split::kNoLimit);
    if (done) break;
  }
}

// x <- W^-1 r with one step of refinement (see w16::solve_refined); r, x in
// shared memory, r is overwritten.
__device__ __forceinline__ void solve_refined(Shared& sm, double* r, double* x) {
  const int i = threadIdx.x >> 3;
  const bool own = (threadIdx.x & 7) == 0;
  const double x0 = matvec(rows_of(sm.M, kLd), r, 0.0);
  if (own) x[i] = x0;
  __syncthreads();
  const double wx = matvec(rows_of(sm.W, kLd), x, 0.0);
  const double d = r[i] - wx;
  __syncthreads();
  if (own) r[i] = d;
  __syncthreads();
  const double x1 = matvec(rows_of(sm.M, kLd), r, x0);
  __syncthreads();
  if (own) x[i] = x1;
  __syncthreads();
}

// Sum of one value per thread over the CTA, in every thread.
__device__ __forceinline__ double cta_sum(Shared& sm, double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sm.red[threadIdx.x >> 5] = x;
  __syncthreads();
  double s = 0.0;
#pragma unroll
  for (int w = 0; w < kThreads / 32; ++w) s += sm.red[w];
  return s;
}

// W = I + C J into sm.W, and the limit of the combination's other products: in
// mixed units all of them are formed in FP64 (see split::kFoldLimit).
__device__ __forceinline__ int product_w(Shared& sm, Mat c, Mat j) {
  if (product64(sm, c, j, sm.W, kLd, 1, split::kTry, split::kFoldLimit) != split::kGraded) return split::kGradeLimit;
  product64(sm, c, j, sm.W, kLd, 1, split::kSet, split::kAllFp64);
  return split::kAllFp64;
}

// out = e1 (x) e2 (full elements in global memory; out aliases neither).
__device__ inline void combine(Shared& sm, Slot sl, Rec<N> e1, Rec<N> e2, Rec<N> out) {
  using split::kSet;
  const int tid = threadIdx.x, i = tid >> 3;
  const bool own = (tid & 7) == 0;
  double *b1 = sm.vec[0], *eta2 = sm.vec[1], *rr = sm.vec[2], *wv = sm.vec[3], *z0 = sm.vec[4], *l0 = sm.vec[5];
  if (tid < N) b1[tid] = e1.b()[tid];
  else if (tid < 2 * N) eta2[tid - N] = e2.eta()[tid - N];
  // W = I + C1 J2, T1 = J2 A1 (C1, J2 symmetric)
  const int limit = product_w(sm, rows_of(e1.C(), N), rows_of(e2.J(), N));
  product64(sm, rows_of(e2.J(), N), cols_of(e1.A(), N), sl.T1, kLd, 0, kSet, limit);
  {
    const double r = matvec(rows_of(e1.C(), N), eta2, b1[i]);
    const double w = matvec(rows_of(e2.J(), N), b1, 0.0);
    if (own) {
      rr[i] = r;
      wv[i] = eta2[i] - w;
    }
  }
  __syncthreads();
  inverse(sm, sl.K1, limit);
  solve_refined(sm, rr, z0);
  product64(sm, rows_of(sm.M, kLd), cols_of(e1.A(), N), sl.K1, kLd, 0, kSet, limit);
  product64(sm, rows_of(sm.M, kLd), rows_of(e1.C(), N), sm.W, kLd, 0, kSet, limit);  // M C1
  // l0 = J2 z0 - eta2 ; zeta ; b = A2 z0 + b2 ; eta = K1^T wv + eta1
  {
    const double jz = matvec(rows_of(e2.J(), N), z0, 0.0);
    if (own) l0[i] = jz - eta2[i];
    const double bo = matvec(rows_of(e2.A(), N), z0, e2.b()[i]);
    const double et = matvec(cols_of(sl.K1, kLd), wv, e1.eta()[i]);
    if (own) {
      out.b()[i] = bo;
      out.eta()[i] = et;
    }
    __syncthreads();
    const double cl = matvec(rows_of(e1.C(), N), l0, 0.0);
    const double z = cta_sum(sm, own ? w16::saddle_term(z0[i], jz, eta2[i], l0[i], b1[i], cl) : 0.0);
    if (tid == 0) *out.zeta() = *e1.zeta() + *e2.zeta() + z;
  }
  // K1^T T1 ; A = A2 K1 ; A2 M C1 ; A2 M C1 A2^T
  product64(sm, cols_of(sl.K1, kLd), cols_of(sl.T1, kLd), sm.M, kLd, 0, kSet, limit);
  product64(sm, rows_of(e2.A(), N), cols_of(sl.K1, kLd), out.A(), N, 0, kSet, limit);
  product64(sm, rows_of(e2.A(), N), cols_of(sm.W, kLd), sl.K1, kLd, 0, kSet, limit);
  product64(sm, rows_of(sl.K1, kLd), rows_of(e2.A(), N), sm.W, kLd, 0, kSet, limit);
  // symmetric by taking the upper triangle
  double *oJ = out.J(), *oC = out.C();
  const double *J1 = e1.J(), *C2 = e2.C();
  for (int e = tid; e < N * N; e += kThreads) {
    const int r = e >> 6, c = e & 63;
    const int o = r < c ? r * kLd + c : c * kLd + r;
    oJ[e] = J1[e] + sm.M[o];
    oC[e] = C2[e] + sm.W[o];
  }
  __syncthreads();
}

// Value form (see team::combine_value): out = e (x) V; V and out value records
// (S, v, zeta) in global memory; the map Psi in sl.K1 (row stride kLd), alpha
// in sm.vec[4].
__device__ inline void combine_value(Shared& sm, Slot sl, Rec<N> e, const double* V, double* out, double* zeta_inc) {
  using split::kSet;
  const int tid = threadIdx.x, i = tid >> 3;
  const bool own = (tid & 7) == 0;
  const double *S2 = V, *v2g = V + N * N;
  double *b = sm.vec[0], *v2 = sm.vec[1], *rr = sm.vec[2], *wv = sm.vec[3], *alpha = sm.vec[4], *l0 = sm.vec[5];
  if (tid < N) b[tid] = e.b()[tid];
  else if (tid < 2 * N) v2[tid - N] = v2g[tid - N];
  const int limit = product_w(sm, rows_of(e.C(), N), rows_of(S2, N));
  product64(sm, rows_of(S2, N), cols_of(e.A(), N), sl.T1, kLd, 0, kSet, limit);
  {
    const double r = matvec(rows_of(e.C(), N), v2, b[i]);
    const double w = matvec(rows_of(S2, N), b, 0.0);
    if (own) {
      rr[i] = r;
      wv[i] = v2[i] - w;
    }
  }
  __syncthreads();
  inverse(sm, sl.K1, limit);
  solve_refined(sm, rr, alpha);
  product64(sm, rows_of(sm.M, kLd), cols_of(e.A(), N), sl.K1, kLd, 0, kSet, limit);  // Psi
  product64(sm, cols_of(sl.K1, kLd), cols_of(sl.T1, kLd), sm.W, kLd, 0, kSet, limit);
  {
    const double sz = matvec(rows_of(S2, N), alpha, 0.0);
    if (own) l0[i] = sz - v2[i];
    const double vo = matvec(cols_of(sl.K1, kLd), wv, e.eta()[i]);
    if (own) out[N * N + i] = vo;
    __syncthreads();
    const double cl = matvec(rows_of(e.C(), N), l0, 0.0);
    const double z = cta_sum(sm, own ? w16::saddle_term(alpha[i], sz, v2[i], l0[i], b[i], cl) : 0.0);
    if (tid == 0) {
      const double inc = *e.zeta() + z;  // the element's own share; the carry's zeta added after
      out[N * N + N] = inc + V[N * N + N];
      *zeta_inc = inc;
    }
  }
  const double* J = e.J();
  for (int q = tid; q < N * N; q += kThreads) {
    const int r = q >> 6, c = q & 63;
    out[q] = J[q] + sm.W[r < c ? r * kLd + c : c * kLd + r];
  }
  __syncthreads();
}

// (P, p) <- (P Psi, P alpha + p), Psi and alpha as combine_value leaves them;
// P (row stride N) and p in global memory.
__device__ inline void compose_right(Shared& sm, Slot sl, double* P, double* p) {
  const int i = threadIdx.x >> 3;
  const double pa = matvec(rows_of(P, N), sm.vec[4], p[i]);
  __syncthreads();
  product64(sm, rows_of(P, N), cols_of(sl.K1, kLd), P, N, 0, split::kSet);
  if ((threadIdx.x & 7) == 0) p[i] = pa;
  __syncthreads();
}

}  // namespace s64
}  // namespace lqt
