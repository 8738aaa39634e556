// FP64 combinations of n = 64 elements on split products (lqt_split.cuh), one
// CTA of 256 threads per combination.
//
// What bounds it: in FP64 a full combination is 2.0 M multiply-adds, 500 us on
// one SM's FP64 pipe (820 us as measured, with the barriers of the LU).  Here
// its fourteen 64^3 products are FP16 tensor-core products of seven digits;
// per product the splitting of 12 k entries and the assembly of 4 k results
// (integer work) take longer than the 28 digit products.  The right operand's
// digits are made once, by the warp that owns eight of its columns, and kept
// in shared memory in fragment order; the left operand's are made by the two
// warps that share sixteen of its rows and stay in registers.  W = I + C1 J2
// is inverted in FP32 (Gauss-Jordan in registers) and refined by Newton steps,
// as for n = 16 (lqt_warp16.cuh), with the FP64 elimination behind it where
// that does not converge.
#pragma once

#include <cuda_runtime.h>

#include "lqt_split.cuh"
#include "lqt_team.cuh"

namespace lqt {
namespace s64 {

using split::C64;
using team::Rec;
constexpr int N = 64;
constexpr int kThreads = 256;
constexpr int kLd = 66;  // row stride of the shared buffers (16-byte rows that start in different banks)
constexpr int kBuf = N * kLd;
constexpr int kDigitWords = 8 * 4 * C64::ND * 32;  // 8-byte words: (8-column tile, 16-deep slab, digit, lane)

// Shared memory of a CTA.
struct Shared {
  double W[kBuf], M[kBuf], T1[kBuf], K1[kBuf];
  double vec[8][N];
  uint2 digit[kDigitWords];
  float col[2][N], rowk[N], rowp[N], scale[N];
  unsigned cand[4];
  int perm[N], colE[N];
  double red[kThreads / 32];
};

// Entry k of vector v at p[v sv + k sk] (rows of a left operand, columns of a
// right one).
struct Mat {
  const double* p;
  int sv, sk;
};
__device__ __forceinline__ Mat rows_of(const double* p, int ld) { return {p, ld, 1}; }
__device__ __forceinline__ Mat cols_of(const double* p, int ld) { return {p, 1, ld}; }

// Sixteen entries of vector v (k = 16 s + c, c + 1, c + 8, c + 9, c = 2 (lane %
// 4)) and its largest exponent.
__device__ __forceinline__ int load_vector(int lane, Mat m, int v, double (&x)[16]) {
  const double* p = m.p + (int64_t)v * m.sv + 2 * (lane & 3) * m.sk;
  int e = 0;
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int h = 0; h < 4; ++h) x[4 * s + h] = p[(16 * s + (h & 1) + 8 * (h >> 1)) * m.sk];
#pragma unroll
  for (int q = 0; q < 16; ++q) e = max(e, split::biased_exp(x[q]));
  e = max(e, __shfl_xor_sync(0xffffffffu, e, 1));
  return max(e, __shfl_xor_sync(0xffffffffu, e, 2));
}

// o(i, j) = sum_k a(i, k) b(k, j) + diag (i == j), or o -= the product
// (kSubtract), o at o[i ld + j].  o may be one of the operands.  Returns the
// largest biased exponent of the entries this warp set.
static __device__ __noinline__ int product64(Shared& sm, Mat a, Mat b, double* o, int ld, int diag, int store) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, c = 2 * (lane & 3);
  {
    double x[16];
    const int e = load_vector(lane, b, 8 * warp + g, x);
    if ((lane & 3) == 0) sm.colE[8 * warp + g] = e;
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      const unsigned long long u0 = split::digits<C64>(x[4 * s], e), u1 = split::digits<C64>(x[4 * s + 1], e);
      const unsigned long long u2 = split::digits<C64>(x[4 * s + 2], e), u3 = split::digits<C64>(x[4 * s + 3], e);
#pragma unroll
      for (int i = 0; i < C64::ND; ++i)
        sm.digit[((warp * 4 + s) * C64::ND + i) * 32 + lane] =
            make_uint2(split::digit_pair<C64>(u0, u1, i), split::digit_pair<C64>(u2, u3, i));
    }
  }
  unsigned af[4][C64::ND][4];
  int ea[2];
  const int r0 = 16 * (warp >> 1);
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    double x[16];
    ea[r] = load_vector(lane, a, r0 + g + 8 * r, x);
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const unsigned long long u = split::digits<C64>(x[4 * s + 2 * h], ea[r]);
        const unsigned long long v = split::digits<C64>(x[4 * s + 2 * h + 1], ea[r]);
#pragma unroll
        for (int i = 0; i < C64::ND; ++i) af[s][i][r + 2 * h] = split::digit_pair<C64>(u, v, i);
      }
  }
  __syncthreads();
  int top = 0;
#pragma unroll 1
  for (int t = 0; t < 4; ++t) {
    const int tile = 4 * (warp & 1) + t;
    float acc[C64::ND][4];
#pragma unroll
    for (int w = 0; w < C64::ND; ++w)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[w][q] = 0.0f;
    const uint2* d = sm.digit + tile * 4 * C64::ND * 32 + lane;
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int j = 0; j < C64::ND; ++j) {
        const uint2 bf = d[(s * C64::ND + j) * 32];
#pragma unroll
        for (int i = 0; i < C64::ND - j; ++i) split::mma16816(acc[i + j], af[s][i], bf.x, bf.y);
      }
    const int e0 = sm.colE[8 * tile + c], e1 = sm.colE[8 * tile + c + 1];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = r0 + g + 8 * (q >> 1), j = 8 * tile + c + (q & 1);
      const double v =
          split::finish<C64>(split::to_int<C64>(acc, q), ea[q >> 1], (q & 1) ? e1 : e0, i == j ? diag : 0);
      top = max(top, split::biased_exp(v));
      double* w = o + (int64_t)i * ld + j;
      *w = store == split::kSubtract ? *w - v : v;
    }
  }
  __syncthreads();
  return __reduce_max_sync(0xffffffffu, top);
}

// base + sum_l m(i, l) x(l) for row i = thread / 4 (x in shared memory), four
// threads per row; every thread of the four returns it.
__device__ __forceinline__ double matvec(Mat m, const double* x, double base) {
  const int i = threadIdx.x >> 2, q = threadIdx.x & 3;
  const double* p = m.p + (int64_t)i * m.sv + q * m.sk;
  double s = q == 0 ? base : 0.0, u = 0.0;
#pragma unroll
  for (int l = 0; l < 16; l += 2) {
    s = fma(p[4 * l * m.sk], x[4 * l + q], s);
    u = fma(p[4 * (l + 1) * m.sk], x[4 * (l + 1) + q], u);
  }
  s += u;
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  return s + __shfl_xor_sync(0xffffffffu, s, 2);
}

__device__ __forceinline__ float pick16(const float (&x)[16], int k) {
  float a[8], b[4];
#pragma unroll
  for (int i = 0; i < 8; ++i) a[i] = (k & 1) ? x[2 * i + 1] : x[2 * i];
#pragma unroll
  for (int i = 0; i < 4; ++i) b[i] = (k & 2) ? a[2 * i + 1] : a[2 * i];
  const float c = (k & 4) ? b[1] : b[0], d = (k & 4) ? b[3] : b[2];
  return (k & 8) ? d : c;
}

// sm.M <- the FP32 inverse of sm.W (partial pivoting; thread (j, q) owns rows
// 16 q .. 16 q + 15 of column j).  False (in every thread) when a pivot is not
// above 2^-10 of its row's largest magnitude (at least 1) or not finite.
static __device__ __noinline__ bool inverse_f32(Shared& sm) {
  const int tid = threadIdx.x, j = tid & 63, q = tid >> 6;
  float m[16];
#pragma unroll
  for (int r = 0; r < 16; ++r) m[r] = (float)sm.W[(16 * q + r) * kLd + j];
  {
    float s = 1.0f;
    const double* w = sm.W + (tid >> 2) * kLd + (tid & 3);
#pragma unroll
    for (int l = 0; l < 16; ++l) s = fmaxf(s, fabsf((float)w[4 * l]));
    s = fmaxf(s, __shfl_xor_sync(0xffffffffu, s, 1));
    s = fmaxf(s, __shfl_xor_sync(0xffffffffu, s, 2));
    if ((tid & 3) == 0) sm.scale[tid >> 2] = s;
    if (tid < N) sm.perm[tid] = tid;
  }
  bool ok = true;
#pragma unroll 1
  for (int k = 0; k < N; ++k) {
    float* col = sm.col[k & 1];
    if (j == k) {
      unsigned best = 0;
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        col[16 * q + r] = m[r];
        const unsigned key = (__float_as_uint(m[r]) & 0x7fffffc0u) | (unsigned)(63 - 16 * q - r);
        best = (16 * q + r >= k) ? max(best, key) : best;
      }
      sm.cand[q] = best;
    }
    __syncthreads();
    const unsigned best = max(max(sm.cand[0], sm.cand[1]), max(sm.cand[2], sm.cand[3]));
    const int p = 63 - (int)(best & 63u);
    const float d = col[p], sp = sm.scale[p], fk = col[k];
    if (q == (k >> 4)) sm.rowk[j] = pick16(m, k & 15);
    if (q == (p >> 4)) sm.rowp[j] = pick16(m, p & 15);
    __syncthreads();
    if (tid == 0) {
      sm.scale[p] = sm.scale[k];
      sm.scale[k] = sp;
      const int t = sm.perm[p];
      sm.perm[p] = sm.perm[k];
      sm.perm[k] = t;
    }
    ok = ok && fabsf(d) > 0x1p-10f * sp && fabsf(d) < 0x1p100f;
    const float vk = sm.rowk[j], pr = (j == k ? 1.0f : sm.rowp[j]) * __frcp_rn(d);
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      const int i = 16 * q + r;
      const float x = i == p ? vk : m[r], f = i == p ? fk : col[i];
      const float v = fmaf(-f, pr, j == k ? 0.0f : x);
      m[r] = i == k ? pr : v;
    }
  }
  __syncthreads();
  const int pj = sm.perm[j];
#pragma unroll
  for (int r = 0; r < 16; ++r) sm.M[(16 * q + r) * kLd + pj] = (double)m[r];
  __syncthreads();
  return ok;
}

// sm.M <- the inverse of sm.W by the FP64 elimination (the pivots and the
// SINGULAR test of team::lu_solve); sm.K1 and the digit buffer are scratch.
static __device__ __noinline__ void inverse_f64(Shared& sm) {
  const int tid = threadIdx.x;
  double* R = reinterpret_cast<double*>(sm.digit);
  double* fs = R + N * N;
  int* is = reinterpret_cast<int*>(fs + 2 * kThreads);
  static_assert(sizeof(sm.digit) >= (N * N + 2 * kThreads) * sizeof(double) + kThreads * sizeof(int), "scratch");
  for (int e = tid; e < N * N; e += kThreads) {
    sm.K1[e] = sm.W[(e >> 6) * kLd + (e & 63)];
    R[e] = (e >> 6) == (e & 63) ? 1.0 : 0.0;
  }
  __syncthreads();
  team::lu_solve<N, kThreads, N>(tid, sm.K1, R, fs, is);
  __syncthreads();
  for (int e = tid; e < N * N; e += kThreads) sm.M[(e >> 6) * kLd + (e & 63)] = R[e];
  __syncthreads();
}

// sm.M <- sm.W^-1: the FP32 inverse and Newton steps M <- M - M (W M - I) until
// the residual is below 2^-28 before the last step; where the residual does
// not shrink, the FP64 inverse and one step.  sm.K1 is scratch.
__device__ __forceinline__ void inverse(Shared& sm) {
  constexpr int kExp1 = 1023;  // biased exponent of 1
  bool fast = inverse_f32(sm);
  int last = kExp1 - 1;
  for (int it = 0; it < 4; ++it) {
    if (!fast) inverse_f64(sm);
    const int top = product64(sm, rows_of(sm.W, kLd), cols_of(sm.M, kLd), sm.K1, kLd, -1, split::kSet);
    // row sums: 64 entries below 2^(top - 1022)
    const bool done = __syncthreads_and(top <= kExp1 - 35) != 0 || !fast;
    const bool lost = __syncthreads_or(top > last - 3 || top > kExp1 - 7) != 0;
    if (!done && (lost || it == 3)) {
      fast = false;
      it = 2;
      continue;
    }
    last = top;
    product64(sm, rows_of(sm.M, kLd), cols_of(sm.K1, kLd), sm.M, kLd, 0, split::kSubtract);
    if (done) break;
  }
}

// x <- W^-1 r with one step of refinement (see w16::solve_refined); r, x in
// shared memory, r is overwritten.
__device__ __forceinline__ void solve_refined(Shared& sm, double* r, double* x) {
  const int i = threadIdx.x >> 2;
  const bool own = (threadIdx.x & 3) == 0;
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

// out = e1 (x) e2 (full elements in global memory; out aliases neither).
__device__ inline void combine(Shared& sm, Rec<N> e1, Rec<N> e2, Rec<N> out) {
  using split::kSet;
  const int tid = threadIdx.x, i = tid >> 2;
  const bool own = (tid & 3) == 0;
  double *b1 = sm.vec[0], *eta2 = sm.vec[1], *rr = sm.vec[2], *wv = sm.vec[3], *z0 = sm.vec[4], *l0 = sm.vec[5];
  if (tid < N) b1[tid] = e1.b()[tid];
  else if (tid < 2 * N) eta2[tid - N] = e2.eta()[tid - N];
  // W = I + C1 J2, T1 = J2 A1 (C1, J2 symmetric)
  product64(sm, rows_of(e1.C(), N), rows_of(e2.J(), N), sm.W, kLd, 1, kSet);
  product64(sm, rows_of(e2.J(), N), cols_of(e1.A(), N), sm.T1, kLd, 0, kSet);
  {
    const double r = matvec(rows_of(e1.C(), N), eta2, b1[i]);
    const double w = matvec(rows_of(e2.J(), N), b1, 0.0);
    if (own) {
      rr[i] = r;
      wv[i] = eta2[i] - w;
    }
  }
  __syncthreads();
  inverse(sm);
  solve_refined(sm, rr, z0);
  product64(sm, rows_of(sm.M, kLd), cols_of(e1.A(), N), sm.K1, kLd, 0, kSet);
  product64(sm, rows_of(sm.M, kLd), rows_of(e1.C(), N), sm.W, kLd, 0, kSet);  // M C1
  // l0 = J2 z0 - eta2 ; zeta ; b = A2 z0 + b2 ; eta = K1^T wv + eta1
  {
    const double jz = matvec(rows_of(e2.J(), N), z0, 0.0);
    if (own) l0[i] = jz - eta2[i];
    const double bo = matvec(rows_of(e2.A(), N), z0, e2.b()[i]);
    const double et = matvec(cols_of(sm.K1, kLd), wv, e1.eta()[i]);
    if (own) {
      out.b()[i] = bo;
      out.eta()[i] = et;
    }
    __syncthreads();
    const double cl = matvec(rows_of(e1.C(), N), l0, 0.0);
    const double z = cta_sum(sm, own ? fma(0.5 * l0[i], cl, z0[i] * fma(0.5, jz, -eta2[i])) : 0.0);
    if (tid == 0) *out.zeta() = *e1.zeta() + *e2.zeta() + z;
  }
  // K1^T T1 ; A = A2 K1 ; A2 M C1 ; A2 M C1 A2^T
  product64(sm, cols_of(sm.K1, kLd), cols_of(sm.T1, kLd), sm.T1, kLd, 0, kSet);
  product64(sm, rows_of(e2.A(), N), cols_of(sm.K1, kLd), out.A(), N, 0, kSet);
  product64(sm, rows_of(e2.A(), N), cols_of(sm.W, kLd), sm.K1, kLd, 0, kSet);
  product64(sm, rows_of(sm.K1, kLd), rows_of(e2.A(), N), sm.W, kLd, 0, kSet);
  // symmetric by taking the upper triangle
  double *oJ = out.J(), *oC = out.C();
  const double *J1 = e1.J(), *C2 = e2.C();
  for (int e = tid; e < N * N; e += kThreads) {
    const int r = e >> 6, c = e & 63;
    const int o = r < c ? r * kLd + c : c * kLd + r;
    oJ[e] = J1[e] + sm.T1[o];
    oC[e] = C2[e] + sm.W[o];
  }
  __syncthreads();
}

// Value form (see team::combine_value): out = e (x) V; V and out value records
// (S, v, zeta) in global memory; the map Psi in sm.K1 (row stride kLd), alpha
// in sm.vec[4].
__device__ inline void combine_value(Shared& sm, Rec<N> e, const double* V, double* out, double* zeta_inc) {
  using split::kSet;
  const int tid = threadIdx.x, i = tid >> 2;
  const bool own = (tid & 3) == 0;
  const double *S2 = V, *v2g = V + N * N;
  double *b = sm.vec[0], *v2 = sm.vec[1], *rr = sm.vec[2], *wv = sm.vec[3], *alpha = sm.vec[4], *l0 = sm.vec[5];
  if (tid < N) b[tid] = e.b()[tid];
  else if (tid < 2 * N) v2[tid - N] = v2g[tid - N];
  product64(sm, rows_of(e.C(), N), rows_of(S2, N), sm.W, kLd, 1, kSet);
  product64(sm, rows_of(S2, N), cols_of(e.A(), N), sm.T1, kLd, 0, kSet);
  {
    const double r = matvec(rows_of(e.C(), N), v2, b[i]);
    const double w = matvec(rows_of(S2, N), b, 0.0);
    if (own) {
      rr[i] = r;
      wv[i] = v2[i] - w;
    }
  }
  __syncthreads();
  inverse(sm);
  solve_refined(sm, rr, alpha);
  product64(sm, rows_of(sm.M, kLd), cols_of(e.A(), N), sm.K1, kLd, 0, kSet);  // Psi
  product64(sm, cols_of(sm.K1, kLd), cols_of(sm.T1, kLd), sm.T1, kLd, 0, kSet);
  {
    const double sz = matvec(rows_of(S2, N), alpha, 0.0);
    if (own) l0[i] = sz - v2[i];
    const double vo = matvec(cols_of(sm.K1, kLd), wv, e.eta()[i]);
    if (own) out[N * N + i] = vo;
    __syncthreads();
    const double cl = matvec(rows_of(e.C(), N), l0, 0.0);
    const double z = cta_sum(sm, own ? fma(0.5 * l0[i], cl, alpha[i] * fma(0.5, sz, -v2[i])) : 0.0);
    if (tid == 0) {
      const double inc = *e.zeta() + z;  // the element's own share; the carry's zeta added after
      out[N * N + N] = inc + V[N * N + N];
      *zeta_inc = inc;
    }
  }
  const double* J = e.J();
  for (int q = tid; q < N * N; q += kThreads) {
    const int r = q >> 6, c = q & 63;
    out[q] = J[q] + sm.T1[r < c ? r * kLd + c : c * kLd + r];
  }
  __syncthreads();
}

// (P, p) <- (P Psi, P alpha + p), Psi and alpha as combine_value leaves them;
// P (row stride N) and p in global memory.
__device__ inline void compose_right(Shared& sm, double* P, double* p) {
  const int i = threadIdx.x >> 2;
  const double pa = matvec(rows_of(P, N), sm.vec[4], p[i]);
  __syncthreads();
  product64(sm, rows_of(P, N), cols_of(sm.K1, kLd), P, N, 0, split::kSet);
  if ((threadIdx.x & 3) == 0) p[i] = pa;
  __syncthreads();
}

}  // namespace s64
}  // namespace lqt
