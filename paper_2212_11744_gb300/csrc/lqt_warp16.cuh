// The combinations for n = 16 (the rule of Sec. IV-A, eq. lqt_comb, full and value
// form; the linear solve of I + C1 J2, App. B).  On this GPU a warp's FP64
// instruction occupies its sub-partition for 64 cycles whatever the number of
// active lanes, which decides both forms here:
//
// FP64 (combine_split, combine_value_split): the 16^3 products on the FP16 tensor
// cores as split products (lqt_split.cuh) and an inverse made in FP32 and refined
// by Newton steps; two warps per combination in the scans, one in Method 2's
// fold.  See the section's own comment below.
//
// Mixed precision (combine, combine_value): FP32 products by one warp, and the
// solve as a register resident FP64 Gauss-Jordan elimination.  The elimination is
// a chain of 16 dependent pivot steps.  Written as an LU in shared memory with a
// barrier after every step (and a second pass for the back substitution), the
// chain left the FP64 pipe idle most of the time.  Here each lane owns one column
// of [W | X1] in registers (lanes 0..15: W, lanes 16..31: X1) and one row slice of
// X2 and of the vector x, so one pass of 16 steps solves W [X1 | X2 | x] = [X1 | X2
// | x]_in with 16-26 independent FMAs per lane per step, no shared-memory traffic
// and no barriers inside the elimination.
//
// The element operand of every combination is staged in shared memory by the
// TMA unit (cp.async.bulk, completion on an mbarrier with a bounded wait),
// from the public element arrays when they are 16-byte aligned; otherwise by
// coalesced plain loads.
#pragma once

#include <cuda_runtime.h>

#include "lqt_device.cuh"
#include "lqt_internal.h"
#include "lqt_split.cuh"

namespace lqt {
namespace w16 {

constexpr int N = 16;
constexpr unsigned kFull = 0xffffffffu;
// element record in shared memory: A (256), b (16), C (256), eta (16), J
// (256), zeta (1): the packed record order; every matrix and vector starts on
// a 16-byte boundary
constexpr int kOffA = 0, kOffB = 256, kOffC = 272, kOffEta = 528, kOffJ = 544, kOffZeta = 800;
constexpr int kRec = 801;
constexpr int kRecPad = 802;  // keeps the next buffer 16-byte aligned
constexpr int kWld = 17;      // row stride of W (odd: row and column accesses are both conflict-free)
constexpr int kRld = 33;      // row stride of the solved block [K1 | MC1 | z0]
// bounded waits: iterations of mbarrier try_wait before the wait gives up
constexpr unsigned kWaitLimit = 1u << 24;

// ---------------------------------------------------------------------------
// TMA bulk copies into shared memory, completion on an mbarrier
// ---------------------------------------------------------------------------

__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// global -> shared bulk copy of `bytes` (a multiple of 16; both addresses
// 16-byte aligned), counted on `bar`
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned bytes, unsigned long long* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
// orders this thread's earlier generic-proxy shared-memory accesses before
// later async-proxy (TMA) accesses
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Waits for phase `parity` of `bar`, at most kWaitLimit polls.  On time-out
// the status word gets kStatusTimeout, and the wait is retried once more
// (bounded again) so that no copy is left landing in shared memory after the
// caller moves on.
__device__ __forceinline__ void mbar_wait_bounded(unsigned long long* bar, unsigned parity) {
  unsigned it = 0;
  while (!mbar_try_wait(bar, parity)) {
    if (++it >= kWaitLimit) {
      flag(kStatusTimeout);
      for (unsigned j = 0; j < kWaitLimit && !mbar_try_wait(bar, parity); ++j) {
      }
      return;
    }
  }
}

// Where element k of a scan level lives: the public arrays (level 0) or a
// packed record (levels above).
struct ElemSrc {
  ElemPtrs el;         // public layout (level 0)
  const double* rec;   // packed records (levels >= 1), or null
  bool bulk;           // public arrays 16-byte aligned: stage by TMA
};

// Stages element k into the shared record `dst` (kRec doubles).  The warp, or
// the CTA of NW warps, calls it with its thread index; on return the record is
// complete.  `bar` is its mbarrier and `phase` its parity, flipped per use.
template <int NW = 1>
__device__ __forceinline__ void stage(int tid, const ElemSrc& s, int64_t k, double* dst, unsigned long long* bar,
                                      unsigned& phase, const double* zero_zeta) {
  constexpr int NT = 32 * NW;
  if (s.rec == nullptr && s.bulk) {
    fence_proxy_async();  // this thread's earlier reads of dst before the copy's writes
    split::sync16<NW>();
    if (tid == 0) {
      mbar_expect_tx(bar, (3 * 256 + 2 * 16) * 8);
      bulk_g2s(dst + kOffA, s.el.A + k * 256, 256 * 8, bar);
      bulk_g2s(dst + kOffB, s.el.b + k * 16, 16 * 8, bar);
      bulk_g2s(dst + kOffC, s.el.C + k * 256, 256 * 8, bar);
      bulk_g2s(dst + kOffEta, s.el.eta + k * 16, 16 * 8, bar);
      bulk_g2s(dst + kOffJ, s.el.J + k * 256, 256 * 8, bar);
      dst[kOffZeta] = s.el.zeta ? s.el.zeta[k] : *zero_zeta;
    }
    mbar_wait_bounded(bar, phase);
    phase ^= 1u;
  } else if (s.rec == nullptr) {
    for (int e = tid; e < 256; e += NT) {
      dst[kOffA + e] = s.el.A[k * 256 + e];
      dst[kOffC + e] = s.el.C[k * 256 + e];
      dst[kOffJ + e] = s.el.J[k * 256 + e];
    }
    if (tid < 16) {
      dst[kOffB + tid] = s.el.b[k * 16 + tid];
      dst[kOffEta + tid] = s.el.eta[k * 16 + tid];
    }
    if (tid == 0) dst[kOffZeta] = s.el.zeta ? s.el.zeta[k] : *zero_zeta;
  } else {
    const double* r = s.rec + k * kRec;
    for (int e = tid; e < kRec; e += NT) dst[e] = r[e];
  }
  split::sync16<NW>();
}

// ---------------------------------------------------------------------------
// products and vectors
// ---------------------------------------------------------------------------

// out(i, j) <- sum_l a(i, l) b(l, j), 16 x 16 x 16: lane (j = lane & 15,
// h = lane >> 4) owns rows 8h..8h+7 of column j (8 independent accumulators);
// a(i, l) is read by the 16 lanes of a half at one address, b(l, j) by
// consecutive lanes at consecutive addresses.
template <typename G, class FA, class FB, class FO>
__device__ __forceinline__ void gemm(int lane, FA a, FB b, FO out) {
  const int j = lane & 15, i0 = (lane >> 4) * 8;
  G acc[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) acc[r] = (G)0;
#pragma unroll 4
  for (int l = 0; l < 16; ++l) {
    const G bv = (G)b(l, j);
#pragma unroll
    for (int r = 0; r < 8; ++r) acc[r] = fma((G)a(i0 + r, l), bv, acc[r]);
  }
#pragma unroll
  for (int r = 0; r < 8; ++r) out(i0 + r, j, acc[r]);
}

// y(i) = base(i) + sum_l m(i, l) x(l): lane (i = lane & 15, h) sums l in
// 8h..8h+7, the halves are added with one shuffle; every lane returns y(its i).
template <typename G, class FM, class FX>
__device__ __forceinline__ G matvec(int lane, FM m, FX x, G base) {
  const int i = lane & 15, l0 = (lane >> 4) * 8;
  G s = (lane >> 4) ? (G)0 : base;
#pragma unroll
  for (int l = 0; l < 8; ++l) s = fma((G)m(i, l0 + l), (G)x(l0 + l), s);
  return s + __shfl_xor_sync(kFull, s, 16);
}

__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
  return x;
}

// ---------------------------------------------------------------------------
// Gauss-Jordan elimination with partial pivoting on [W | X1 | X2 | x]
// ---------------------------------------------------------------------------

// On entry lane c < 16 holds column c of W in col[], lane 16 + c column c of
// X1; lane l holds x(l & 15) in xv and, when HAS_X2, row (l & 15) of X2,
// columns 8 (l >> 4) .. +7, in row[]; rk is the magnitude key of row (l & 15)'s
// scale max(1, max_j |W_lj|).  On return X1, X2, x are replaced by
// W^-1 X1, W^-1 X2, W^-1 x in the same places.  A pivot no larger than 2^-40
// of its row's scale sets the SINGULAR status bit (pivot_too_small).
template <bool HAS_X2>
__device__ __forceinline__ void gauss_jordan(int lane, double (&col)[16], double (&row)[8], double& xv,
                                             unsigned long long rk) {
  const int myrow = lane & 15, half = lane >> 4;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    // pivot: the largest |W(i, k)|, i >= k, lowest i on ties (lane k's column)
    unsigned long long best = mag_key(col[k]);
    int p = k;
#pragma unroll
    for (int i = k + 1; i < 16; ++i) {
      const unsigned long long key = mag_key(col[i]);
      if (key > best) {
        best = key;
        p = i;
      }
    }
    p = __shfl_sync(kFull, p, k);
    best = __shfl_sync(kFull, best, k);
    const unsigned long long rk_k = __shfl_sync(kFull, rk, k), rk_p = __shfl_sync(kFull, rk, p);
    if (myrow == k) rk = rk_p;
    else if (myrow == p) rk = rk_k;
    if (lane == 0 && pivot_too_small(__longlong_as_double((long long)best), rk_p)) flag(kStatusSingular);
    // exchange rows k and p: the column registers by predicated selects, the
    // row-distributed values between the lanes that hold rows k and p
    {
      double nk = col[k];
#pragma unroll
      for (int i = k + 1; i < 16; ++i) {
        const bool s = (p == i);
        const double ci = col[i];
        col[i] = s ? col[k] : ci;
        nk = s ? ci : nk;
      }
      col[k] = nk;
      const int src = myrow == k ? p + 16 * half : (myrow == p ? k + 16 * half : lane);
      if constexpr (HAS_X2) {
#pragma unroll
        for (int j = 0; j < 8; ++j) row[j] = __shfl_sync(kFull, row[j], src);
      }
      xv = __shfl_sync(kFull, xv, src);
    }
    const double d = __shfl_sync(kFull, col[k], k);
    const double inv = 1.0 / d;
    double rkrow[8];
    if constexpr (HAS_X2) {
#pragma unroll
      for (int j = 0; j < 8; ++j) rkrow[j] = __shfl_sync(kFull, row[j], k + 16 * half);
    }
    const double xk = __shfl_sync(kFull, xv, k);
    // new row k = row k / d; row i -= W(i, k) (new row k) for i != k
    const double pr = col[k] * inv;
    double myf = 0.0;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const double f = __shfl_sync(kFull, col[i], k);
      myf = (i == myrow) ? f : myf;
      if (i != k) col[i] = fma(-f, pr, col[i]);
    }
    col[k] = pr;
    // the row-distributed values: one fma each, a = inv - 1 on row k itself
    const double a = (myrow == k) ? inv - 1.0 : -myf * inv;
    if constexpr (HAS_X2) {
#pragma unroll
      for (int j = 0; j < 8; ++j) row[j] = fma(a, rkrow[j], row[j]);
    }
    xv = fma(a, xk, xv);
  }
}

// Row scale key of row (lane & 15) of W (row stride kWld): max(1, max_j |W_ij|).
__device__ __forceinline__ unsigned long long row_scale(int lane, const double* W) {
  const int i = lane & 15, j0 = (lane >> 4) * 8;
  unsigned long long rk = mag_key(1.0);
#pragma unroll
  for (int j = 0; j < 8; ++j) rk = umax64(rk, mag_key(W[i * kWld + j0 + j]));
  return umax64(rk, __shfl_xor_sync(kFull, rk, 16));
}

// ---------------------------------------------------------------------------
// the combinations
// ---------------------------------------------------------------------------

// Scratch of combine(): W (16 x 17), R (16 x 33), T1 (16 x 17), vectors.
constexpr int kScrW = 0, kScrR = 16 * kWld, kScrT = kScrR + 16 * kRld, kScrV = kScrT + 16 * kWld;
constexpr int kScratch = kScrV + 6 * 16;

// e1 <- e1 (x) e2 in place (both full records in shared memory, kRec layout).
// G: the type the products are formed in (double, or float for the mixed
// path); the solve is FP64 in both.
template <typename G>
__device__ void combine(int lane, double* e1, const double* e2, double* scr) {
  double* W = scr + kScrW;
  double* R = scr + kScrR;
  double* T1 = scr + kScrT;
  double* z0 = scr + kScrV;
  double* J2z = z0 + 16;
  double* l0 = J2z + 16;
  double* wv = l0 + 16;
  const double* A1 = e1 + kOffA;
  const double* C1 = e1 + kOffC;
  const double* b1 = e1 + kOffB;
  const double* A2 = e2 + kOffA;
  const double* C2 = e2 + kOffC;
  const double* J2 = e2 + kOffJ;
  const double* b2 = e2 + kOffB;
  const double* eta2 = e2 + kOffEta;
  const int i = lane & 15, h = lane >> 4;
  // W = I + C1 J2 ; T1 = J2 A1 ; r = b1 + C1 eta2 ; wv = eta2 - J2 b1 (C1, J2
  // symmetric: their rows are read as columns)
  gemm<G>(lane, [&](int r, int l) { return C1[r * 16 + l]; }, [&](int l, int c) { return J2[l * 16 + c]; },
          [&](int r, int c, G v) { W[r * kWld + c] = (double)v + (r == c ? 1.0 : 0.0); });
  gemm<G>(lane, [&](int r, int l) { return J2[r * 16 + l]; }, [&](int l, int c) { return A1[l * 16 + c]; },
          [&](int r, int c, G v) { T1[r * kWld + c] = (double)v; });
  const double rv = (double)matvec<G>(lane, [&](int r, int l) { return C1[l * 16 + r]; },
                                      [&](int l) { return eta2[l]; }, (G)b1[i]);
  const double w = (double)matvec<G>(lane, [&](int r, int l) { return -J2[l * 16 + r]; },
                                     [&](int l) { return b1[l]; }, (G)eta2[i]);
  if (h == 0) wv[i] = w;
  __syncwarp();
  // [K1 | MC1 | z0] = W^-1 [A1 | C1 | r] (FP64)
  {
    double col[16], row[8];
    const double* src = lane < 16 ? W + lane : A1 + (lane - 16);
    const int ld = lane < 16 ? kWld : 16;
#pragma unroll
    for (int r = 0; r < 16; ++r) col[r] = src[r * ld];
#pragma unroll
    for (int j = 0; j < 8; ++j) row[j] = C1[(8 * h + j) * 16 + i];
    double xv = rv;
    const unsigned long long rk = row_scale(lane, W);
    gauss_jordan<true>(lane, col, row, xv, rk);
    if (lane >= 16) {
#pragma unroll
      for (int r = 0; r < 16; ++r) R[r * kRld + (lane - 16)] = col[r];
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) R[i * kRld + 16 + 8 * h + j] = row[j];
    if (h == 0) {
      R[i * kRld + 32] = xv;
      z0[i] = xv;
    }
  }
  __syncwarp();
  // J2 z0, l0 = J2 z0 - eta2 ; zeta ; eta = K1^T wv + eta1 ; b = A2 z0 + b2
  {
    const G jz = matvec<G>(lane, [&](int r, int l) { return J2[l * 16 + r]; }, [&](int l) { return z0[l]; }, (G)0);
    if (h == 0) {
      J2z[i] = (double)jz;
      l0[i] = (double)jz - eta2[i];
    }
    const G et = matvec<G>(lane, [&](int r, int l) { return R[l * kRld + r]; }, [&](int l) { return wv[l]; },
                           (G)e1[kOffEta + i]);
    const G bo = matvec<G>(lane, [&](int r, int l) { return A2[r * 16 + l]; }, [&](int l) { return z0[l]; },
                           (G)b2[i]);
    __syncwarp();
    const G cl = matvec<G>(lane, [&](int r, int l) { return C1[l * 16 + r]; }, [&](int l) { return l0[l]; }, (G)0);
    double zt = (h == 0) ? fma(0.5 * l0[i], (double)cl, z0[i] * fma(0.5, J2z[i], -eta2[i])) : 0.0;
    const double z = warp_sum(zt);
    __syncwarp();
    if (h == 0) {
      e1[kOffEta + i] = (double)et;
      e1[kOffB + i] = (double)bo;
    }
    if (lane == 0) e1[kOffZeta] = e1[kOffZeta] + e2[kOffZeta] + z;
  }
  // W <- K1^T T1 ; A1 <- A2 K1 (A1 was consumed by the solve and T1)
  gemm<G>(lane, [&](int r, int l) { return R[l * kRld + r]; }, [&](int l, int c) { return T1[l * kWld + c]; },
          [&](int r, int c, G v) { W[r * kWld + c] = (double)v; });
  gemm<G>(lane, [&](int r, int l) { return A2[r * 16 + l]; }, [&](int l, int c) { return R[l * kRld + c]; },
          [&](int r, int c, G v) { e1[kOffA + r * 16 + c] = (double)v; });
  __syncwarp();
  // J = J1 + sym(K1^T T1) ; T1 <- (A2 MC1)^T
  for (int e = lane; e < 256; e += 32) {
    const int r = e >> 4, c = e & 15;
    e1[kOffJ + e] += 0.5 * (W[r * kWld + c] + W[c * kWld + r]);
  }
  gemm<G>(lane, [&](int r, int l) { return A2[r * 16 + l]; }, [&](int l, int c) { return R[l * kRld + 16 + c]; },
          [&](int r, int c, G v) { T1[c * kWld + r] = (double)v; });
  __syncwarp();
  // C = C2 + sym(A2 (A2 MC1)^T)
  gemm<G>(lane, [&](int r, int l) { return A2[r * 16 + l]; }, [&](int l, int c) { return T1[l * kWld + c]; },
          [&](int r, int c, G v) { W[r * kWld + c] = (double)v; });
  __syncwarp();
  for (int e = lane; e < 256; e += 32) {
    const int r = e >> 4, c = e & 15;
    e1[kOffC + e] = C2[e] + 0.5 * (W[r * kWld + c] + W[c * kWld + r]);
  }
  __syncwarp();
}

// Value record: S (256), v (16), zeta.
constexpr int kVal = 273;
// Scratch of combine_value(): W (16 x 17), T1 (16 x 17), vectors.
constexpr int kVScrW = 0, kVScrT = 16 * kWld, kVScrV = kVScrT + 16 * kWld;
constexpr int kVScratch = kVScrV + 4 * 16;

// out = e (x) V (value form, out may not alias V), and the one-sub-interval
// map Psi (16 x 16 row-major), alpha (16).  e: full record in shared memory.
// W = I + C S2 and b + C v2 are formed in FP64 whatever G is: they define the
// map the state scan composes T times.
template <typename G>
__device__ void combine_value(int lane, const double* e, const double* V, double* out, double* Psi, double* alpha,
                              double* scr, double* zeta_inc = nullptr) {
  double* W = scr + kVScrW;
  double* T1 = scr + kVScrT;
  double* wv = scr + kVScrV;
  double* Sz = wv + 16;
  double* l0 = Sz + 16;
  const double* A = e + kOffA;
  const double* C = e + kOffC;
  const double* b = e + kOffB;
  const double* S2 = V;
  const double* v2 = V + 256;
  const int i = lane & 15, h = lane >> 4;
  gemm<double>(lane, [&](int r, int l) { return C[r * 16 + l]; }, [&](int l, int c) { return S2[l * 16 + c]; },
               [&](int r, int c, double v) { W[r * kWld + c] = v + (r == c ? 1.0 : 0.0); });
  gemm<G>(lane, [&](int r, int l) { return S2[r * 16 + l]; }, [&](int l, int c) { return A[l * 16 + c]; },
          [&](int r, int c, G v) { T1[r * kWld + c] = (double)v; });
  const double rv = matvec<double>(lane, [&](int r, int l) { return C[l * 16 + r]; }, [&](int l) { return v2[l]; },
                                   b[i]);
  const double w = (double)matvec<G>(lane, [&](int r, int l) { return -S2[l * 16 + r]; },
                                     [&](int l) { return b[l]; }, (G)v2[i]);
  if (h == 0) wv[i] = w;
  __syncwarp();
  {
    double col[16], row[8];
    const double* src = lane < 16 ? W + lane : A + (lane - 16);
    const int ld = lane < 16 ? kWld : 16;
#pragma unroll
    for (int r = 0; r < 16; ++r) col[r] = src[r * ld];
    double xv = rv;
    const unsigned long long rk = row_scale(lane, W);
    gauss_jordan<false>(lane, col, row, xv, rk);
    if (lane >= 16) {
#pragma unroll
      for (int r = 0; r < 16; ++r) Psi[r * 16 + (lane - 16)] = col[r];
    }
    if (h == 0) alpha[i] = xv;
  }
  __syncwarp();
  // Sz = S2 alpha, l0 = Sz - v2 ; v = eta + Psi^T wv ; W <- Psi^T T1 ; zeta
  {
    const G sz = matvec<G>(lane, [&](int r, int l) { return S2[l * 16 + r]; }, [&](int l) { return alpha[l]; },
                           (G)0);
    if (h == 0) {
      Sz[i] = (double)sz;
      l0[i] = (double)sz - v2[i];
    }
    const G vo = matvec<G>(lane, [&](int r, int l) { return Psi[l * 16 + r]; }, [&](int l) { return wv[l]; },
                           (G)e[kOffEta + i]);
    gemm<G>(lane, [&](int r, int l) { return Psi[l * 16 + r]; }, [&](int l, int c) { return T1[l * kWld + c]; },
            [&](int r, int c, G v) { W[r * kWld + c] = (double)v; });
    __syncwarp();
    const G cl = matvec<G>(lane, [&](int r, int l) { return C[l * 16 + r]; }, [&](int l) { return l0[l]; }, (G)0);
    const double zt = (h == 0) ? fma(0.5 * l0[i], (double)cl, alpha[i] * fma(0.5, Sz[i], -v2[i])) : 0.0;
    const double z = warp_sum(zt);
    if (h == 0) out[256 + i] = (double)vo;
    if (lane == 0) {
      const double inc = e[kOffZeta] + z;  // the element's own share; the carry's zeta added after
      out[272] = inc + V[272];
      if (zeta_inc) *zeta_inc = inc;
    }
  }
  for (int q = lane; q < 256; q += 32) {
    const int r = q >> 4, c = q & 15;
    out[q] = e[kOffJ + q] + 0.5 * (W[r * kWld + c] + W[c * kWld + r]);
  }
  __syncwarp();
}

// (P, p) <- (P Psi, P alpha + p); Tm: 16 x 17 scratch.
__device__ __forceinline__ void compose_right(int lane, double* P, double* p, const double* Psi, const double* alpha,
                                              double* Tm) {
  gemm<double>(lane, [&](int r, int l) { return P[r * 16 + l]; }, [&](int l, int c) { return Psi[l * 16 + c]; },
               [&](int r, int c, double v) { Tm[r * kWld + c] = v; });
  const double pa = matvec<double>(lane, [&](int r, int l) { return P[r * 16 + l]; },
                                   [&](int l) { return alpha[l]; }, p[lane & 15]);
  __syncwarp();
  for (int q = lane; q < 256; q += 32) P[q] = Tm[(q >> 4) * kWld + (q & 15)];
  if (lane < 16) p[lane] = pa;
  __syncwarp();
}

// ---------------------------------------------------------------------------
// the FP64 combinations: split products (lqt_split.cuh) and an inverse
// ---------------------------------------------------------------------------
//
// Done in FP64, a combination is bound by that pipe, at 64 cycles a warp
// instruction: five to six 16^3 products took 128 instructions each and the
// elimination of 2 n + 1 right-hand sides 530.  The products now run on the
// tensor core (about 800 cycles of a sub-partition each, integer work, against
// 8192), and W is inverted instead of eliminated: a Gauss-Jordan inverse in
// FP32 and Newton steps M <- M - M (W M - I), whose residual the split product
// forms to 2^-57 of |W| |M|.  A residual below 2^-28 makes the step that
// follows exact to FP64 rounding, so M is as accurate as its own rounding.
// Where an FP32 pivot falls below 2^-10 of its row or the residual does not
// shrink (cond(W) beyond some 1e5), the inverse is made in FP64 with the
// pivots and the SINGULAR test of gauss_jordan, and the Newton step polishes
// that one.  In states of mixed units (split::kFoldLimit) the inverse and all
// products are FP64, the Newton step too: it takes out what the elimination's
// pivots, which feel the units, leave.
// Level 0 of a scan, T = 4104 (ncu, 6.8 CTAs on an SM): the ALU pipe, which splits
// and assembles, is 50% busy, the FP64 pipe (vectors, inverse) 40%, the tensor pipe
// 6%; the warps wait on their own results and on instruction fetches.

// x[k], k = 0..7, without indexing a local array.
template <typename X>
__device__ __forceinline__ X pick8(const X (&x)[8], int k) {
  const X a = (k & 1) ? x[1] : x[0], b = (k & 1) ? x[3] : x[2], c = (k & 1) ? x[5] : x[4], d = (k & 1) ? x[7] : x[6];
  const X e = (k & 2) ? b : a, f = (k & 2) ? d : c;
  return (k & 4) ? f : e;
}

// The FP32 inverse: layout as invert16 below; scale: the largest magnitude of
// row (lane & 15), at least 1.  False when a pivot is not safely away from 0.
__device__ __forceinline__ bool invert16_f32(int lane, float (&m)[8], float scale, int& perm) {
  const int j = lane & 15, h = lane >> 4;
  perm = j;
  bool ok = true;
#pragma unroll 1
  for (int k = 0; k < 16; ++k) {
    // largest magnitude of column k below the diagonal, to 2^-19, with its row
    unsigned best = 0;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const unsigned key = (__float_as_uint(m[r]) & 0x7ffffff0u) | (unsigned)(15 - 8 * h - r);
      best = (8 * h + r >= k) ? max(best, key) : best;
    }
    best = max(__shfl_sync(kFull, best, k), __shfl_sync(kFull, best, k + 16));
    const int p = 15 - (int)(best & 15u);
    const float sk = __shfl_sync(kFull, scale, k), sp = __shfl_sync(kFull, scale, p);
    const int pk = __shfl_sync(kFull, perm, k), pp = __shfl_sync(kFull, perm, p);
    scale = j == k ? sp : (j == p ? sk : scale);
    perm = j == k ? pp : (j == p ? pk : perm);
    const float vk = __shfl_sync(kFull, pick8(m, k & 7), j + 16 * (k >> 3));
    const float vp = __shfl_sync(kFull, pick8(m, p & 7), j + 16 * (p >> 3));
    const float d = __shfl_sync(kFull, vp, k);
    ok = ok && fabsf(d) > 0x1p-10f * sp && fabsf(d) < 0x1p100f;
    const float pr = (j == k ? 1.0f : vp) * __frcp_rn(d);
#pragma unroll
    for (int r = 0; r < 8; ++r) m[r] = (8 * h + r == p) ? vk : m[r];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const float f = __shfl_sync(kFull, m[r], k + 16 * h);
      const float v = fmaf(-f, pr, j == k ? 0.0f : m[r]);
      m[r] = (8 * h + r == k) ? pr : v;
    }
  }
  return ok;
}

// Inverse of W in place with partial pivoting: lane (j = lane & 15, h = lane
// >> 4) holds rows 8h .. 8h + 7 of column j in m; rk as in gauss_jordan.  On
// return m holds column j of (P W)^-1, which is column perm of W^-1.  Pivots
// as in gauss_jordan (the same rows, the same SINGULAR test).
__device__ __forceinline__ int invert16(int lane, double (&m)[8], unsigned long long rk) {
  const int j = lane & 15, h = lane >> 4;
  int perm = j;
#pragma unroll 1
  for (int k = 0; k < 16; ++k) {
    unsigned long long best = 0;
    int p = k;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const unsigned long long key = (8 * h + r >= k) ? mag_key(m[r]) : 0ull;
      if (key > best) {
        best = key;
        p = 8 * h + r;
      }
    }
    {
      const unsigned long long ob = __shfl_xor_sync(kFull, best, 16);
      const int op = __shfl_xor_sync(kFull, p, 16);
      if (ob > best || (ob == best && op < p)) {
        best = ob;
        p = op;
      }
    }
    p = __shfl_sync(kFull, p, k);
    best = __shfl_sync(kFull, best, k);
    const unsigned long long rk_k = __shfl_sync(kFull, rk, k), rk_p = __shfl_sync(kFull, rk, p);
    const int pm_k = __shfl_sync(kFull, perm, k), pm_p = __shfl_sync(kFull, perm, p);
    if (j == k) {
      rk = rk_p;
      perm = pm_p;
    } else if (j == p) {
      rk = rk_k;
      perm = pm_k;
    }
    if (lane == 0 && pivot_too_small(__longlong_as_double((long long)best), rk_p)) flag(kStatusSingular);
    // exchange rows k and p
    const double mk = pick8(m, k & 7), mp = pick8(m, p & 7);
    const double vk = __shfl_sync(kFull, mk, j + 16 * (k >> 3));
    const double vp = __shfl_sync(kFull, mp, j + 16 * (p >> 3));
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const double x = (8 * h + r == p) ? vk : m[r];
      m[r] = (8 * h + r == k) ? vp : x;
    }
    const double inv = 1.0 / __shfl_sync(kFull, vp, k);
    const double pr = (j == k ? 1.0 : vp) * inv;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const double f = __shfl_sync(kFull, m[r], k + 16 * h);
      const double v = fma(-f, pr, j == k ? 0.0 : m[r]);
      m[r] = (8 * h + r == k) ? pr : v;
    }
  }
  return perm;
}

// Offset of a shared-memory buffer from the CTA's dynamic shared memory.
__device__ __forceinline__ int sm_off(const double* p) {
  extern __shared__ __align__(16) double split_smem[];
  return (int)(p - split_smem);
}
// Rows (kWld or 16 doubles apart) of a buffer as vectors, and its columns.
__device__ __forceinline__ split::Mat16 rows_of(const double* p, int ld) { return {sm_off(p), ld, 1}; }
__device__ __forceinline__ split::Mat16 cols_of(const double* p, int ld) { return {sm_off(p), 1, ld}; }

// Minv (row stride kWld) <- W^-1 by the elimination in FP64.
static __device__ __noinline__ void inverse_f64(const double* W, double* Minv) {
  const int lane = threadIdx.x & 31, j = lane & 15, i0 = 8 * (lane >> 4);
  double m[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) m[r] = W[(i0 + r) * kWld + j];
  const int perm = invert16(lane, m, row_scale(lane, W));
#pragma unroll
  for (int r = 0; r < 8; ++r) Minv[(i0 + r) * kWld + perm] = m[r];
  __syncwarp();
}

// Minv <- the FP32 inverse of W, by one warp; false: see invert16_f32.
__device__ __forceinline__ bool inverse_f32(int lane, const double* W, double* Minv) {
  const int j = lane & 15, i0 = 8 * (lane >> 4);
  float m[8];
  float s = 1.0f;
#pragma unroll
  for (int r = 0; r < 8; ++r) s = fmaxf(s, fabsf((float)W[j * kWld + i0 + r]));
  s = fmaxf(s, __shfl_xor_sync(kFull, s, 16));
#pragma unroll
  for (int r = 0; r < 8; ++r) m[r] = (float)W[(i0 + r) * kWld + j];
  int perm;
  const bool ok = invert16_f32(lane, m, s, perm);
#pragma unroll
  for (int r = 0; r < 8; ++r) Minv[(i0 + r) * kWld + perm] = (double)m[r];
  __syncwarp();
  return ok;
}

// Newton steps on Minv (row stride kWld), which holds the FP32 inverse of W
// (row stride kWld) when `fast` (the same in every thread); E (row stride ld)
// is scratch.  limit: split::kAllFp64 or the products' own.
template <int NW>
__device__ __forceinline__ void refine_inverse(const double* W, double* Minv, double* E, int ld, bool fast,
                                               int limit) {
  constexpr int kExp1 = 1023;  // biased exponent of 1
  // at most four steps: |W M - I| < 2^-28 (row sum: sixteen entries below 2^-32)
  // before the last one
  int last = kExp1 - 1;
  for (int it = 0; it < 4; ++it) {
    if (!fast) {
      if (NW == 1 || threadIdx.x < 32) inverse_f64(W, Minv);
      split::sync16<NW>();
    }
    const int top = split::product16<NW>(rows_of(W, kWld), cols_of(Minv, kWld), rows_of(E, ld), -1, split::kSet,
                                           limit);
    // the residual must fall at least eightfold per step, from below 1/16
    bool done = top <= kExp1 - 33, lost = top > last - 3 || top > kExp1 - 5;
    if constexpr (NW > 1) {
      done = __syncthreads_and(done) != 0;
      lost = __syncthreads_or(lost) != 0;
    }
    done = done || !fast;
    if (!done && (lost || it == 3)) {
      fast = false;  // not converging: the FP64 inverse, then its one step
      it = 2;
      continue;
    }
    last = top;
    split::product16<NW>(rows_of(Minv, kWld), cols_of(E, ld), rows_of(Minv, kWld), 0, split::kSubtract,
                         limit < 0 ? limit : split::kNoLimit);  // E is small: its products' errors are, too
    if (done) break;
  }
}

// x = W^-1 r from M = W^-1, r and x in shared memory (r is overwritten), one
// warp: x = M r and one step of refinement, so that W x - r is of the size an
// elimination leaves (x = M r alone leaves up to cond(W) times that, which the
// zeta and eta terms, made from J2 x - eta2 with its cancellation, would feel).
__device__ __forceinline__ void solve_refined(int lane, const double* W, const double* Minv, double* r, double* x) {
  const int i = lane & 15, h = lane >> 4;
  const double x0 = matvec<double>(lane, [&](int a, int l) { return Minv[a * kWld + l]; }, [&](int l) { return r[l]; },
                                   0.0);
  if (h == 0) x[i] = x0;
  __syncwarp();
  const double d = matvec<double>(lane, [&](int a, int l) { return -W[a * kWld + l]; }, [&](int l) { return x[l]; },
                                  r[i]);
  __syncwarp();
  if (h == 0) r[i] = d;
  __syncwarp();
  const double x1 = matvec<double>(lane, [&](int a, int l) { return Minv[a * kWld + l]; }, [&](int l) { return r[l]; },
                                   x0);
  __syncwarp();
  if (h == 0) x[i] = x1;
  __syncwarp();
}

// Entry of zeta's saddle value z'Jz/2 - z'eta + l'(b - z) - l'Cl/2 at z0 = (I +
// C J)^-1 (b + C eta), l0 = J z0 - eta (Sec. IV-A, the minimiser and multiplier
// at x = 0).  At the exact saddle b - z0 = C l0 and this is l0'Cl0/2 + z0'Jz0/2 -
// z0'eta; in this form an error of z0 or l0 enters to second order only, so
// that zeta does not feel the conditioning of I + C J (at cond 1e8, n = 64, the
// other form was 2e-6 off after 130 combinations).
__device__ __forceinline__ double saddle_term(double z, double Jz, double eta, double l, double b, double Cl) {
  return fma(z, fma(0.5, Jz, -eta), l * ((b - z) - 0.5 * Cl));
}

// W = I + C J, and the limit of the combination's other products: in mixed units
// all of them are formed in FP64 (see kFoldLimit).
template <int NW>
__device__ __forceinline__ int product_w(split::Mat16 c, split::Mat16 j, split::Mat16 w) {
  if (split::product16<NW>(c, j, w, 1, split::kTry, split::kFoldLimit) != split::kGraded) return split::kGradeLimit;
  split::product16<NW>(c, j, w, 1, split::kSet, split::kAllFp64);
  return split::kAllFp64;
}

// Scratch of combine_split(): four 16 x 17 buffers and vectors.
constexpr int kSplitBuf = 16 * kWld;
constexpr int kSplitScratch = 4 * kSplitBuf + 6 * 16;

// e1 <- e1 (x) e2 in place, FP64 (both full records in shared memory), by one
// warp or a CTA of two: the second warp takes products that do not wait for
// the inverse or for the vectors, and eight columns of the others.
template <int NW>
__device__ inline void combine_split(double* e1, const double* e2, double* scr) {
  using split::kSet;
  using split::product16;
  using split::sync16;
  double* W = scr;               // W, then M C1, then A2 M C1 A2^T
  double* Mi = W + kSplitBuf;    // M = W^-1
  double* T1 = Mi + kSplitBuf;   // J2 A1, then K1^T J2 A1
  double* K1 = T1 + kSplitBuf;   // the Newton residual, K1 = M A1, A2 M C1
  double* z0 = K1 + kSplitBuf;
  double* J2z = z0 + 16;
  double* l0 = J2z + 16;
  double* wv = l0 + 16;
  double* rr = wv + 16;
  int* fast = reinterpret_cast<int*>(rr + 16);
  const double* A1 = e1 + kOffA;
  const double* C1 = e1 + kOffC;
  const double* b1 = e1 + kOffB;
  const double* A2 = e2 + kOffA;
  const double* C2 = e2 + kOffC;
  const double* J2 = e2 + kOffJ;
  const double* b2 = e2 + kOffB;
  const double* eta2 = e2 + kOffEta;
  const int tid = NW == 1 ? (int)(threadIdx.x & 31) : (int)threadIdx.x;
  const int lane = tid & 31, i = lane & 15, h = lane >> 4;
  const bool first = NW == 1 || tid < 32, second = NW == 1 || tid >= 32;
  // W = I + C1 J2, T1 = J2 A1 (C1, J2 symmetric: their rows are their columns)
  const int limit = product_w<NW>(rows_of(C1, 16), rows_of(J2, 16), rows_of(W, kWld));
  if (first) {
    const bool ok = limit >= 0 && inverse_f32(lane, W, Mi);
    if (lane == 0) *fast = ok ? 1 : 0;
  }
  if (second) {
    product16<1>(rows_of(J2, 16), cols_of(A1, 16), rows_of(T1, kWld), 0, kSet, limit);
    const double rv = matvec<double>(lane, [&](int r, int l) { return C1[l * 16 + r]; },
                                     [&](int l) { return eta2[l]; }, b1[i]);
    const double w = matvec<double>(lane, [&](int r, int l) { return -J2[l * 16 + r]; }, [&](int l) { return b1[l]; },
                                    eta2[i]);
    if (h == 0) {
      wv[i] = w;
      rr[i] = rv;
    }
  }
  sync16<NW>();
  refine_inverse<NW>(W, Mi, K1, kWld, *fast != 0, limit);
  product16<NW>(rows_of(Mi, kWld), cols_of(A1, 16), rows_of(K1, kWld), 0, kSet, limit);
  double bo = 0.0, zs = 0.0, et = 0.0;
  if (first) {
    // z0 = M (b1 + C1 eta2), l0 = J2 z0 - eta2 ; zeta ; b = A2 z0 + b2
    solve_refined(lane, W, Mi, rr, z0);
    const double jz = matvec<double>(lane, [&](int r, int l) { return J2[l * 16 + r]; }, [&](int l) { return z0[l]; },
                                     0.0);
    if (h == 0) {
      J2z[i] = jz;
      l0[i] = jz - eta2[i];
    }
    bo = matvec<double>(lane, [&](int r, int l) { return A2[r * 16 + l]; }, [&](int l) { return z0[l]; }, b2[i]);
    __syncwarp();
    const double cl = matvec<double>(lane, [&](int r, int l) { return C1[l * 16 + r]; }, [&](int l) { return l0[l]; },
                                     0.0);
    const double zt = (h == 0) ? saddle_term(z0[i], J2z[i], eta2[i], l0[i], b1[i], cl) : 0.0;
    zs = warp_sum(zt);
  }
  if (second) {
    // eta = K1^T wv + eta1 ; K1^T T1 ; A = A2 K1 (A1 was consumed by T1, K1)
    et = matvec<double>(lane, [&](int r, int l) { return K1[l * kWld + r]; }, [&](int l) { return wv[l]; },
                        e1[kOffEta + i]);
    product16<1>(cols_of(K1, kWld), cols_of(T1, kWld), rows_of(T1, kWld), 0, kSet, limit);
    product16<1>(rows_of(A2, 16), cols_of(K1, kWld), rows_of(e1 + kOffA, 16), 0, kSet, limit);
  }
  sync16<NW>();
  if (first) {
    if (h == 0) e1[kOffB + i] = bo;
    if (lane == 0) e1[kOffZeta] = e1[kOffZeta] + e2[kOffZeta] + zs;
  }
  if (second && h == 0) e1[kOffEta + i] = et;
  // C = A2 (M C1) A2^T + C2
  product16<NW>(rows_of(Mi, kWld), rows_of(C1, 16), rows_of(W, kWld), 0, kSet, limit);
  product16<NW>(rows_of(A2, 16), cols_of(W, kWld), rows_of(K1, kWld), 0, kSet, limit);
  product16<NW>(rows_of(K1, kWld), rows_of(A2, 16), rows_of(W, kWld), 0, kSet, limit);
  // symmetric by taking the upper triangle
  for (int e = tid; e < 256; e += 32 * NW) {
    const int r = e >> 4, c = e & 15;
    const int o = r < c ? r * kWld + c : c * kWld + r;
    e1[kOffJ + e] += T1[o];
    e1[kOffC + e] = C2[e] + W[o];
  }
  sync16<NW>();
}

// Scratch of combine_value_split(): three 16 x 17 buffers and vectors.
constexpr int kVSplitScratch = 3 * kSplitBuf + 5 * 16;

// combine_value() in FP64 with split products, by a CTA of two warps.
__device__ inline void combine_value_split(const double* e, const double* V, double* out, double* Psi, double* alpha,
                                           double* scr, double* zeta_inc) {
  constexpr int NW = 2;
  using split::kSet;
  using split::product16;
  double* W = scr;
  double* T1 = W + kSplitBuf;  // S2 A, then Psi^T S2 A
  double* Mi = T1 + kSplitBuf;
  double* wv = Mi + kSplitBuf;
  double* Sz = wv + 16;
  double* l0 = Sz + 16;
  double* rr = l0 + 16;
  int* fast = reinterpret_cast<int*>(rr + 16);
  const double* A = e + kOffA;
  const double* C = e + kOffC;
  const double* b = e + kOffB;
  const double* S2 = V;
  const double* v2 = V + 256;
  const int tid = threadIdx.x, lane = tid & 31, i = lane & 15, h = lane >> 4;
  const int limit = product_w<NW>(rows_of(C, 16), rows_of(S2, 16), rows_of(W, kWld));
  if (tid < 32) {
    const bool ok = limit >= 0 && inverse_f32(lane, W, Mi);
    if (lane == 0) *fast = ok ? 1 : 0;
  } else {
    product16<1>(rows_of(S2, 16), cols_of(A, 16), rows_of(T1, kWld), 0, kSet, limit);
    const double rv = matvec<double>(lane, [&](int r, int l) { return C[l * 16 + r]; }, [&](int l) { return v2[l]; },
                                     b[i]);
    const double w = matvec<double>(lane, [&](int r, int l) { return -S2[l * 16 + r]; }, [&](int l) { return b[l]; },
                                    v2[i]);
    if (h == 0) {
      wv[i] = w;
      rr[i] = rv;
    }
  }
  __syncthreads();
  refine_inverse<NW>(W, Mi, Psi, 16, *fast != 0, limit);
  product16<NW>(rows_of(Mi, kWld), cols_of(A, 16), rows_of(Psi, 16), 0, kSet, limit);
  if (tid < 32) {
    // alpha ; Sz = S2 alpha, l0 = Sz - v2 ; zeta
    solve_refined(lane, W, Mi, rr, alpha);
    const double sz = matvec<double>(lane, [&](int r, int l) { return S2[l * 16 + r]; },
                                     [&](int l) { return alpha[l]; }, 0.0);
    if (h == 0) {
      Sz[i] = sz;
      l0[i] = sz - v2[i];
    }
    __syncwarp();
    const double cl = matvec<double>(lane, [&](int r, int l) { return C[l * 16 + r]; }, [&](int l) { return l0[l]; },
                                     0.0);
    const double zt = (h == 0) ? saddle_term(alpha[i], Sz[i], v2[i], l0[i], b[i], cl) : 0.0;
    const double z = warp_sum(zt);
    if (lane == 0) {
      const double inc = e[kOffZeta] + z;  // the element's own share; the carry's zeta added after
      out[272] = inc + V[272];
      *zeta_inc = inc;
    }
  } else {
    // v = eta + Psi^T wv ; Psi^T T1
    const double vo = matvec<double>(lane, [&](int r, int l) { return Psi[l * 16 + r]; },
                                     [&](int l) { return wv[l]; }, e[kOffEta + i]);
    if (h == 0) out[256 + i] = vo;
    product16<1>(cols_of(Psi, 16), cols_of(T1, kWld), rows_of(T1, kWld), 0, kSet, limit);
  }
  __syncthreads();
  for (int q = tid; q < 256; q += 32 * NW) {
    const int r = q >> 4, c = q & 15;
    out[q] = e[kOffJ + q] + T1[r < c ? r * kWld + c : c * kWld + r];
  }
  __syncthreads();
}

// (P, p) <- (P Psi, P alpha + p), by a CTA of two warps.
__device__ inline void compose_right_split(double* P, double* p, const double* Psi, const double* alpha) {
  const int lane = threadIdx.x & 31;
  double pa = 0.0;
  if (threadIdx.x < 32)
    pa = matvec<double>(lane, [&](int r, int l) { return P[r * 16 + l]; }, [&](int l) { return alpha[l]; },
                        p[lane & 15]);
  __syncthreads();
  split::product16<2>(rows_of(P, 16), cols_of(Psi, 16), rows_of(P, 16), 0, split::kSet);
  if (threadIdx.x < 16) p[lane] = pa;
  __syncthreads();
}

}  // namespace w16
}  // namespace lqt
