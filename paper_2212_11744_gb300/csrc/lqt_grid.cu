// The general method on a state grid: the nonlinear scalar example of
// Sec. VI-B (dx/dt = d0 + d1 x + d2 x^2 + u, running cost q x^2/2 + rho u^2/2,
// terminal cost qf x^2/2), each conditional value function held as the G x G
// array V(x_i, s; x_j, s') on the grid x_i = x_min + i dx, combined by the
// minimisation of Theorem HJB-comb over the grid and refined by the
// quadratic interpolation of App. E.
//
//   block    the one-step function (an explicit Euler step with any control)
//            combined with itself `substeps` times, left to right;
//   combine  out(i, j) = min_k A(i, k) + B(k, j), refined;
//   values   V(., t_k) for k = 0..T.  The model is time-invariant, so every
//            block has the same conditional value function (Sec. VI-B) and
//            the scan's partial products are its powers.  The powers
//            P_{l+1} = P_l (x) P_l are formed once (log2 T products); then for
//            each bit l, lowest first, every k whose T - k has bit l set
//            updates w_k <- P_l (x) w_k, all such k and all grid points in one
//            launch.  After the last bit w_k = V(., t_k).
//
// Both products are one kernel: a tile of outputs per CTA, several per thread, the
// reduction index staged in shared memory.  The minimum is defined on FP64 sums, ascending k, strict improvement only (the
// lowest index wins a tie).  GB300 retires FP64 adds at 1/64 of its FP32
// rate, so every candidate is first screened in FP32 (a bracket around its
// sum) and only the few whose bracket reaches the smallest upper bound are
// summed in FP64; the screen provably keeps every k that could be the FP64
// minimum, so the result is the one of the plain FP64 scan (which remains the
// path for operands outside the screen's float range).  FP64 comparisons run
// on integer keys that order doubles like the FP64 comparison does (the two
// zeros equal).  This is tropical (min, +) algebra: no multiply-accumulate, so
// no tensor-core form applies.
//
// Every floating-point expression uses explicit round-to-nearest intrinsics,
// in the order the definitions state them, so no multiply-add contraction
// changes a rounding: on the same inputs the grid minimisers are the same as
// those of any evaluation that follows the same formulas in IEEE double.
#include <climits>

#include <cuda_runtime.h>

#include "lqt_device.cuh"
#include "lqt_internal.h"

namespace lqt {

namespace {

struct GridArgs {
  int32_t G;
  double x_min, dx, d0, d1, d2, q, rho, qf, tau;
  int32_t substeps;
  int64_t T;
  int32_t interp;
};

GridArgs grid_args(const lqt_grid_problem& p) {
  return GridArgs{p.G, p.x_min, p.dx, p.d0, p.d1, p.d2, p.q, p.rho, p.qf, p.tau, p.substeps, p.T, p.interp};
}

// A CTA of 256 threads forms a tile of 16 P x 16 Q outputs, P x Q per thread; the
// reduction index is staged in shared memory in float, at most kKC at a time (a
// grid of <= 224 points: once).
constexpr int kThreads = 256;
constexpr int kKC = 224;

__device__ __forceinline__ double grid_x(const GridArgs& a, int i) { return __dadd_rn(a.x_min, __dmul_rn((double)i, a.dx)); }

// Integer key with key(u) < key(v) exactly when u < v for non-NaN doubles
// (and key(-0) == key(+0)): the bit pattern for u >= +0, its negated
// magnitude for u <= -0.
__device__ __forceinline__ long long order_key(double v) {
  const long long b = __double_as_longlong(v);
  return b < 0 ? LLONG_MIN - b : b;
}

// App. E: the curvature a = (p + m - 2 c) / (2 dx^2) and slope
// b = (p - m) / (2 dx) of the quadratic through (m, c, p) at (k-1, k, k+1).
__device__ __forceinline__ double2 curvature(const GridArgs& a, double m, double c, double p) {
  const double den2 = __dmul_rn(2.0, __dmul_rn(a.dx, a.dx));
  const double den1 = __dmul_rn(2.0, a.dx);
  return make_double2(__ddiv_rn(__dsub_rn(__dadd_rn(p, m), __dmul_rn(2.0, c)), den2), __ddiv_rn(__dsub_rn(p, m), den1));
}

// App. E: the grid minimum `best` = g_k + f_k lowered by b^2 / (4a), with
// a = a_g + a_f and b = b_g + b_f; unchanged when a <= 0.
__device__ __forceinline__ double refine_with(double best, double2 g, double2 f) {
  const double cv = __dadd_rn(g.x, f.x), sl = __dadd_rn(g.y, f.y);
  if (!(cv > 0.0)) return best;
  return __dsub_rn(best, __ddiv_rn(__dmul_rn(sl, sl), __dmul_rn(4.0, cv)));
}

// Curvature and slope of every power's rows at every interior k, as pairs
// tab[l][i][k] (zero at k = 0 and G-1): they depend on (l, i, k) alone, so the
// values levels read them instead of dividing again for every row of w.
__global__ void grid_curv_kernel(GridArgs a, const double* __restrict__ pw, int L, double2* __restrict__ tab) {
  const int64_t GG = (int64_t)a.G * a.G;
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= L * GG) return;
  const int k = (int)(e % a.G);
  tab[e] = (k > 0 && k < a.G - 1) ? curvature(a, pw[e - 1], pw[e], pw[e + 1]) : make_double2(0.0, 0.0);
}

// C(i, j): from x_i to x_j in one step dt = tau / substeps of
// x' = x + dt (drift(x) + u), so u = (x_j - x_i)/dt - drift(x_i) and the cost
// is dt (q x_i^2 + rho u^2) / 2.
__global__ void grid_one_step_kernel(GridArgs a, double* __restrict__ C) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)a.G * a.G) return;
  const int i = (int)(e / a.G), j = (int)(e % a.G);
  const double dt = __ddiv_rn(a.tau, (double)a.substeps);
  const double xi = grid_x(a, i), xj = grid_x(a, j);
  const double drift = __dadd_rn(__dadd_rn(a.d0, __dmul_rn(a.d1, xi)), __dmul_rn(__dmul_rn(a.d2, xi), xi));
  const double u = __dsub_rn(__ddiv_rn(__dsub_rn(xj, xi), dt), drift);
  C[e] = __dmul_rn(__dmul_rn(dt, 0.5), __dadd_rn(__dmul_rn(__dmul_rn(a.q, xi), xi), __dmul_rn(__dmul_rn(a.rho, u), u)));
}

// Values mode: column c of the product is the c-th k (ascending e = T - k)
// whose e has bit l set.  Such e run in blocks of 2^l: e = (2m+1) 2^l + r.
// Row k starts in buffer popc(e) & 1 and moves to the other buffer at every
// set bit of e, so before level l it is in buffer popc(e >> l) & 1 and after
// its last set bit in buffer 0.
struct ValCol {
  const double* in;
  double* out;
};

__device__ __forceinline__ ValCol value_column(const GridArgs& a, int l, int64_t c, double* X0, double* X1) {
  const int64_t low = ((int64_t)1 << l) - 1;
  const int64_t e = ((2 * (c >> l) + 1) << l) + (c & low);
  const int64_t k = a.T - e;
  const bool odd = __popcll((unsigned long long)(e >> l)) & 1;
  const int64_t off = k * a.G;
  return odd ? ValCol{X1 + off, X0 + off} : ValCol{X0 + off, X1 + off};
}

// Operands of one product.  kValues = false: A(i, k), B(k, j), out(i, j), all
// G x G row-major.  kValues = true: A = P_l, column c of B is w_in of the c-th
// updated row (see value_column), out column c is its w_out.
template <bool kValues>
struct Operands {
  const GridArgs& a;
  const double* __restrict__ A;
  const double* Bm;
  double* Om;
  double* X0;
  double* X1;
  int l;
  __device__ __forceinline__ double av(int i, int k) const { return A[(int64_t)i * a.G + k]; }
  // Column c of B: combine mode strides by G, values mode is contiguous.
  __device__ __forceinline__ const double* bcol(int64_t c) const {
    return kValues ? value_column(a, l, c, X0, X1).in : Bm + c;
  }
  __device__ __forceinline__ double bv(const double* col, int k) const {
    return kValues ? col[k] : col[(int64_t)k * a.G];
  }
};

// FP32 screen of a grid minimum (exactness argument below).  The operands are
// truncated to float by bit operations (relative error < 2^-23; magnitudes
// below 2^-126 become 0), summed in float, and bracketed:
//   lo_k = s_k - c t_k - d  <=  g_k + f_k  <=  hi_k = s_k + c t_k,
// t_k = |a_k| + |b_k|, c = 2^-20, d = 2^-100, with margins of more than four
// times the truncation and rounding errors and of the gap between two doubles
// that round to the same FP64 sum.  With U = min_k hi_k (+ d), every k whose
// FP64 sum g_k + f_k equals the FP64 minimum has lo_k <= U; every k with
// lo_k > U has a larger FP64 sum.  So the exact minimum, with the lowest-index
// rule, is taken over the survivors lo_k <= U alone, in ascending k, in FP64.
// Where no operand of a stage is negative, t_k is s_k itself, so that the smallest
// hi_k of the stage is s_min + c s_min, and with none negative in the whole tile
// lo_k <= U is a bound on s_k: a candidate then costs one addition and one
// minimum, and one addition and one comparison in the second pass (a bound
// rounded up keeps a few candidates more, never fewer).
// Operands of magnitude >= 2^100 (or not finite) fall outside the screen's
// float range: a CTA that meets one evaluates every candidate in FP64.
constexpr float kScreenC = 9.5367431640625e-07f;  // 2^-20
constexpr float kScreenD = 7.888609052210118e-31f;  // 2^-100
constexpr float kScreenPad = 1.329227995784916e+36f;  // 2^120: k beyond the grid
constexpr int kMaxSurvivors = 4;

__device__ __forceinline__ bool screen_range(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  return ((b >> 52) & 0x7ff) < 1023 + 100;
}

// Truncation toward zero of a double in the screen's range to float.
__device__ __forceinline__ float screen_float(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int eb = (int)((b >> 52) & 0x7ff);
  if (eb < 1023 - 126) return 0.0f;
  const unsigned fb = ((unsigned)(b >> 63) << 31) | ((unsigned)(eb - 1023 + 127) << 23) |
                      (unsigned)((b >> 29) & 0x7fffff);
  return __uint_as_float(fb);
}

__device__ __forceinline__ float screen_hi(float a, float b) {
  return __fmaf_rn(kScreenC, __fadd_rn(fabsf(a), fabsf(b)), __fadd_rn(a, b));
}
__device__ __forceinline__ float screen_lo(float a, float b) {
  return __fmaf_rn(-kScreenC, __fadd_rn(fabsf(a), fabsf(b)), __fadd_rn(a, b));
}

// Row stride (floats) of the staged tiles for kc values of k: a multiple of 4
// that is 4 modulo 32, so that 16-byte reads of eight consecutive rows fall on
// different banks.
__host__ __device__ __forceinline__ int screen_stride(int kc) { return ((kc + 27) / 32) * 32 + 4; }

// Float tiles of the A rows i0 .. and the B columns c0 .., k0 <= k < k0 + kc; k
// beyond the grid holds kScreenPad.  Returns bit 0: an operand outside the
// screen's range, bit 1: a negative operand.
template <int TR, int TC, bool kValues>
__device__ __forceinline__ int stage_float(const Operands<kValues>& op, float* As, float* Bs, int S, int t, int i0,
                                           int64_t c0, int64_t ncols, int k0, int kc) {
  const int G = op.a.G, warp = t >> 5, lane = t & 31;
  int bad = 0;
  // U loads in flight at a time: one by one, their latency was a fifth of a
  // small product's time (G = 201: 27 us a product, 22 so)
  constexpr int U = 7;
  auto put = [&](float* dst, bool live, int gk, double x) {
    float v = kScreenPad;
    if (gk < G) {
      v = 0.0f;
      if (live) {
        v = screen_float(x);  // (signs compared in float: an FP64 comparison takes 64 cycles)
        bad |= (screen_range(x) ? 0 : 1) | (v < 0.0f ? 2 : 0);
      }
    }
    *dst = v;
  };
  auto put_row = [&](float* dst, const double* src, bool live) {  // src: k0 onwards
    for (int kb = lane; kb < kc; kb += 32 * U) {
      double x[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int kk = kb + 32 * u;
        x[u] = live && kk < kc && k0 + kk < G ? src[kk] : 0.0;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int kk = kb + 32 * u;
        if (kk < kc) put(dst + kk, live, k0 + kk, x[u]);
      }
    }
  };
  for (int r = warp; r < TR; r += kThreads / 32)
    put_row(As + r * S, op.A + (int64_t)(i0 + r) * G + k0, i0 + r < G);
  if (kValues) {
    for (int r = warp; r < TC; r += kThreads / 32) {
      const bool col = c0 + r < ncols;
      put_row(Bs + r * S, col ? op.bcol(c0 + r) + k0 : nullptr, col);
    }
  } else {
    const int r = t % TC;
    const bool col = c0 + r < ncols;
    constexpr int step = kThreads / TC;
    for (int kb = t / TC; kb < kc; kb += step * U) {
      double x[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int kk = kb + step * u;
        x[u] = col && kk < kc && k0 + kk < G ? op.Bm[(int64_t)(k0 + kk) * G + c0 + r] : 0.0;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int kk = kb + step * u;
        if (kk < kc) put(Bs + r * S + kk, col, k0 + kk, x[u]);
      }
    }
  }
  return bad;
}

// A tile of 16 P x 16 Q outputs (i, c) per CTA, P x Q per thread (rows t % 16 +
// 16 p, columns t / 16 + 16 q: a warp's 16-byte reads of the staged rows are free
// of conflicts, and in the values mode 16 consecutive lanes store 16
// consecutive i): the FP32 screen over all k (two passes: the bound U, then the
// survivors), the FP64 minimum over the survivors, App. E's refinement, the
// store.  Bound by the FP32 and ALU instructions of the two passes and, per
// output, by some 30 FP64 instructions of the refinement (its three divisions)
// at 64 cycles each.  One output per thread, with staging again in the second
// pass, took 4.43 ms for the block and the values at G = 201, T = 10^4, 2 x 4 outputs
// and two CTAs on an SM 3.09, 2 x 2 and three CTAs 2.59, and with the operands'
// signs compared in float instead of FP64 2.29 (G = 60, T = 10^4, the values alone:
// 670 us with one output per thread, 710 with the FP64 comparisons, 668).  The
// small tiles take four CTAs on an SM: the values at T = 10^4 in one graph 408 -> 369 us
// at G = 20, 489 -> 477 at 40, 609 -> 558 at 60.
template <int P, int Q, bool kValues>
__global__ void __launch_bounds__(kThreads, P * Q == 1 ? 4 : 3)
    grid_minplus_kernel(GridArgs a, const double* __restrict__ A, const double* Bm, double* Om, double* X0,
                        double* X1, int l, int64_t ncols, const double2* __restrict__ tab) {
  constexpr int TR = 16 * P, TC = 16 * Q;
  extern __shared__ __align__(16) float grid_smem[];
  const Operands<kValues> op{a, A, Bm, Om, X0, X1, l};
  const int G = a.G, t = threadIdx.x, ti = t & 15, tc = t >> 4;
  const int i0 = blockIdx.y * TR;
  const int64_t c0 = (int64_t)blockIdx.x * TC;
  const int kc = G < kKC ? ((G + 3) & ~3) : kKC;  // staged values of k (padded)
  const int S = screen_stride(kc);
  float* As = grid_smem;
  float* Bs = As + TR * S;

  int bad = 0;
  float U[P][Q];
#pragma unroll
  for (int p = 0; p < P; ++p)
#pragma unroll
    for (int q = 0; q < Q; ++q) U[p][q] = __int_as_float(0x7f800000);  // +inf
  // pass 1: the smallest upper bracket, where a stage holds nothing negative by
  // way of its smallest sum (the bracket grows with it)
  bool neg = false;
  for (int k0 = 0; k0 < G; k0 += kc) {
    if (k0) __syncthreads();
    const int here = stage_float<TR, TC>(op, As, Bs, S, t, i0, c0, ncols, k0, kc);
    bad |= here;
    const bool signs = __syncthreads_or(here & 2) != 0;
    neg = neg || signs;
    float m[P][Q];
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
      for (int q = 0; q < Q; ++q) m[p][q] = __int_as_float(0x7f800000);
    auto pass1 = [&](auto sum) {
      for (int kk = 0; kk < kc; kk += 4) {
        float4 x[P], y[Q];
#pragma unroll
        for (int p = 0; p < P; ++p) x[p] = *reinterpret_cast<const float4*>(As + (ti + 16 * p) * S + kk);
#pragma unroll
        for (int q = 0; q < Q; ++q) y[q] = *reinterpret_cast<const float4*>(Bs + (tc + 16 * q) * S + kk);
#pragma unroll
        for (int p = 0; p < P; ++p)
#pragma unroll
          for (int q = 0; q < Q; ++q) {
            const float m0 = fminf(sum(x[p].x, y[q].x), sum(x[p].y, y[q].y));
            const float m1 = fminf(sum(x[p].z, y[q].z), sum(x[p].w, y[q].w));
            m[p][q] = fminf(m[p][q], fminf(m0, m1));
          }
      }
    };
    if (signs)
      pass1([](float x, float y) { return screen_hi(x, y); });
    else
      pass1([](float x, float y) { return __fadd_rn(x, y); });
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
      for (int q = 0; q < Q; ++q)
        U[p][q] = fminf(U[p][q], signs ? m[p][q] : __fmaf_rn(kScreenC, m[p][q], m[p][q]));
  }
  const bool range = __syncthreads_or(bad & 1) != 0;
  unsigned long long pk[P][Q];  // survivors' indices, 16 bits each (G <= 16384)
  int ns[P][Q];
#pragma unroll
  for (int p = 0; p < P; ++p)
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      pk[p][q] = 0;
      ns[p][q] = range ? kMaxSurvivors + 1 : 0;
    }
  auto push = [&](int p, int q, int k) {
    if (ns[p][q] < kMaxSurvivors) pk[p][q] |= (unsigned long long)k << (16 * ns[p][q]);
    ++ns[p][q];
  };
  if (!range && !neg) {
    // s_k - c s_k <= s_min + c s_min + d holds for no s_k above this bound
    float thr[P][Q];
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const float ub = __fadd_ru(U[p][q], kScreenD);
        thr[p][q] = __fmaf_ru(2.0f * kScreenC, ub, ub);
      }
    for (int k0 = 0; k0 < G; k0 += kc) {
      if (G > kc) {  // one stage: pass 1's is still in place
        __syncthreads();
        stage_float<TR, TC>(op, As, Bs, S, t, i0, c0, ncols, k0, kc);
        __syncthreads();
      }
      for (int kk = 0; kk < kc; kk += 4) {
        float4 x[P], y[Q];
#pragma unroll
        for (int p = 0; p < P; ++p) x[p] = *reinterpret_cast<const float4*>(As + (ti + 16 * p) * S + kk);
#pragma unroll
        for (int q = 0; q < Q; ++q) y[q] = *reinterpret_cast<const float4*>(Bs + (tc + 16 * q) * S + kk);
#pragma unroll
        for (int p = 0; p < P; ++p)
#pragma unroll
          for (int q = 0; q < Q; ++q) {
            const float s0 = __fadd_rn(x[p].x, y[q].x), s1 = __fadd_rn(x[p].y, y[q].y);
            const float s2 = __fadd_rn(x[p].z, y[q].z), s3 = __fadd_rn(x[p].w, y[q].w);
            if (fminf(fminf(s0, s1), fminf(s2, s3)) <= thr[p][q]) {
              if (s0 <= thr[p][q]) push(p, q, k0 + kk);
              if (s1 <= thr[p][q]) push(p, q, k0 + kk + 1);
              if (s2 <= thr[p][q]) push(p, q, k0 + kk + 2);
              if (s3 <= thr[p][q]) push(p, q, k0 + kk + 3);
            }
          }
      }
    }
  } else if (!range) {
    // negative operands: the brackets with their own t_k (a padded k's is far
    // above every bound)
    for (int k0 = 0; k0 < G; k0 += kc) {
      if (G > kc) {
        __syncthreads();
        stage_float<TR, TC>(op, As, Bs, S, t, i0, c0, ncols, k0, kc);
        __syncthreads();
      }
      for (int kk = 0; kk < kc; kk += 4) {
        float4 x[P], y[Q];
#pragma unroll
        for (int p = 0; p < P; ++p) x[p] = *reinterpret_cast<const float4*>(As + (ti + 16 * p) * S + kk);
#pragma unroll
        for (int q = 0; q < Q; ++q) y[q] = *reinterpret_cast<const float4*>(Bs + (tc + 16 * q) * S + kk);
#pragma unroll
        for (int p = 0; p < P; ++p)
#pragma unroll
          for (int q = 0; q < Q; ++q) {
            const float ub = __fadd_ru(U[p][q], kScreenD);
            if (screen_lo(x[p].x, y[q].x) <= ub) push(p, q, k0 + kk);
            if (screen_lo(x[p].y, y[q].y) <= ub) push(p, q, k0 + kk + 1);
            if (screen_lo(x[p].z, y[q].z) <= ub) push(p, q, k0 + kk + 2);
            if (screen_lo(x[p].w, y[q].w) <= ub) push(p, q, k0 + kk + 3);
          }
      }
    }
  }
#pragma unroll
  for (int p = 0; p < P; ++p)
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int i = i0 + ti + 16 * p;
      const int64_t c = c0 + tc + 16 * q;
      if (i >= G || c >= ncols) continue;
      const double* col = op.bcol(c);
      double best = 0.0;
      int bk = 0;
      long long bestk = LLONG_MAX;
      const bool listed = ns[p][q] <= kMaxSurvivors;
      const int cnt = listed ? ns[p][q] : G;  // too many survivors: every k
      for (int r = 0; r < cnt; ++r) {
        const int k = listed ? (int)((pk[p][q] >> (16 * r)) & 0xffff) : r;
        const double v = __dadd_rn(op.av(i, k), op.bv(col, k));
        const long long key = order_key(v);
        if (key < bestk) {
          bestk = key;
          best = v;
          bk = k;
        }
      }
      double res = best;
      if (a.interp && bk > 0 && bk < G - 1) {
        const double2 gc =
            tab ? tab[(int64_t)i * G + bk] : curvature(a, op.av(i, bk - 1), op.av(i, bk), op.av(i, bk + 1));
        res = refine_with(best, gc, curvature(a, op.bv(col, bk - 1), op.bv(col, bk), op.bv(col, bk + 1)));
      }
      if (kValues) value_column(a, l, c, X0, X1).out[i] = res;
      else Om[(int64_t)i * G + c] = res;
      if (!isfinite(res)) flag(kStatusNonFinite);
    }
}

// Row k of the values starts as phi(x_i) = qf x_i^2 / 2 in the buffer it
// occupies before level 0: X0 when popc(T - k) is even, so that after its
// last update it lands in X0.
__global__ void grid_terminal_kernel(GridArgs a, double* __restrict__ X0, double* __restrict__ X1) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (a.T + 1) * a.G) return;
  const int64_t k = e / a.G;
  const double x = grid_x(a, (int)(e % a.G));
  const double phi = __dmul_rn(__dmul_rn(__dmul_rn(0.5, a.qf), x), x);
  const bool odd = __popcll((unsigned long long)(a.T - k)) & 1;
  (odd ? X1 : X0)[e] = phi;
}

unsigned cdiv_u(int64_t x, int64_t y) { return (unsigned)((x + y - 1) / y); }

int grid_levels(int64_t T) {
  int L = 0;
  while (((int64_t)1 << L) <= T) ++L;
  return L;
}

// Number of e in [1, T] with bit l set.
int64_t set_count(int64_t T, int l) {
  const int64_t blk = (int64_t)1 << (l + 1), half = (int64_t)1 << l;
  const int64_t full = (T + 1) / blk, rem = (T + 1) % blk;
  return full * half + (rem > half ? rem - half : 0);
}

template <int P, int Q, bool kValues>
cudaError_t launch_tiles(const GridArgs& a, const double* A, const double* B, double* out, double* X0, double* X1,
                         int l, int64_t ncols, const double2* tab, cudaStream_t st) {
  const int kc = a.G < kKC ? ((a.G + 3) & ~3) : kKC;
  constexpr size_t per_stride = (size_t)(16 * P + 16 * Q) * sizeof(float);
  const size_t smem = per_stride * screen_stride(kc);  // at most 58 KB
  const auto kernel = grid_minplus_kernel<P, Q, kValues>;
  // the limit of the largest G, whatever this G: the attribute belongs to all of
  // the process's threads, and one with a small G must not lower it between
  // another's call here and its launch
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)(per_stride * screen_stride(kKC)));
  if (e != cudaSuccess) return e;
  const dim3 grid(cdiv_u(ncols, 16 * Q), cdiv_u(a.G, 16 * P));
  kernel<<<grid, kThreads, smem, st>>>(a, A, B, out, X0, X1, l, ncols, tab);
  count_launch();
  return cudaGetLastError();
}

// 32 x 32 tiles where they fill the SMs (three CTAs on each of 152, so that one
// CTA's FP64 refinement runs beside another's screen), 16 x 16 otherwise: a
// product of two 201 x 201 matrices has 49 of the large tiles and 169 of the
// small ones.
template <bool kValues>
cudaError_t launch_minplus(const GridArgs& a, const double* A, const double* B, double* out, double* X0, double* X1,
                           int l, int64_t ncols, const double2* tab, cudaStream_t st) {
  const int64_t large = (int64_t)cdiv_u(ncols, 32) * cdiv_u(a.G, 32);
  return large >= 3 * 152 ? launch_tiles<2, 2, kValues>(a, A, B, out, X0, X1, l, ncols, tab, st)
                          : launch_tiles<1, 1, kValues>(a, A, B, out, X0, X1, l, ncols, tab, st);
}

cudaError_t launch_combine(const GridArgs& a, const double* A, const double* B, double* out, cudaStream_t st) {
  return launch_minplus<false>(a, A, B, out, nullptr, nullptr, 0, a.G, nullptr, st);
}

}  // namespace

size_t grid_workspace_bytes(const lqt_grid_problem& p, int which) {
  const size_t GG = (size_t)p.G * p.G;
  if (which == 0) return 2 * GG * sizeof(double);
  // powers, one double of alignment slack, their (curvature, slope) pairs, the
  // second buffer of the values
  return ((size_t)grid_levels(p.T) * GG * 3 + 1 + ((size_t)p.T + 1) * p.G) * sizeof(double);
}

cudaError_t run_grid_block(const lqt_grid_problem& p, double* Vblock, char* ws, cudaStream_t st) {
  const GridArgs a = grid_args(p);
  const size_t GG = (size_t)p.G * p.G;
  double* C = (double*)ws;
  double* tmp = C + GG;
  grid_one_step_kernel<<<cdiv_u((int64_t)GG, 256), 256, 0, st>>>(a, C);
  count_launch();
  cudaError_t e = cudaGetLastError();
  // M_1 = C, M_{m+1} = M_m (x) C, ping-ponging between Vblock and tmp so that
  // M_substeps ends in Vblock.
  double* cur = (p.substeps & 1) ? Vblock : tmp;
  if (e == cudaSuccess) e = cudaMemcpyAsync(cur, C, GG * sizeof(double), cudaMemcpyDeviceToDevice, st);
  for (int m = 1; m < p.substeps && e == cudaSuccess; ++m) {
    double* nxt = cur == Vblock ? tmp : Vblock;
    e = launch_combine(a, cur, C, nxt, st);
    cur = nxt;
  }
  return e;
}

cudaError_t run_grid_combine(const lqt_grid_problem& p, const double* A, const double* B, double* out,
                             cudaStream_t st) {
  return launch_combine(grid_args(p), A, B, out, st);
}

cudaError_t run_grid_values(const lqt_grid_problem& p, const double* Vblock, double* V, char* ws, cudaStream_t st) {
  const GridArgs a = grid_args(p);
  const size_t GG = (size_t)p.G * p.G;
  const int L = grid_levels(p.T);
  double* pw = (double*)ws;  // P_0 .. P_{L-1}
  // their (curvature, slope) pairs, on a 16-byte boundary
  double2* tab = (double2*)(((uintptr_t)(pw + (size_t)L * GG) + 15) & ~(uintptr_t)15);
  double* X1 = (double*)(tab + (size_t)L * GG);  // second buffer of the values (V is the first)
  cudaError_t e = cudaMemcpyAsync(pw, Vblock, GG * sizeof(double), cudaMemcpyDeviceToDevice, st);
  for (int l = 1; l < L && e == cudaSuccess; ++l)
    e = launch_combine(a, pw + (l - 1) * GG, pw + (l - 1) * GG, pw + l * GG, st);
  if (e != cudaSuccess) return e;
  if (p.interp) {
    grid_curv_kernel<<<cdiv_u((int64_t)L * GG, 256), 256, 0, st>>>(a, pw, L, tab);
    count_launch();
  }
  grid_terminal_kernel<<<cdiv_u((p.T + 1) * p.G, 256), 256, 0, st>>>(a, V, X1);
  count_launch();
  for (int l = 0; l < L; ++l) {
    const int64_t nc = set_count(p.T, l);
    e = launch_minplus<true>(a, pw + l * GG, nullptr, nullptr, V, X1, l, nc, p.interp ? tab + l * GG : nullptr, st);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

}  // namespace lqt
