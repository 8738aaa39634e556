// Stage (a): conditional value function elements of every sub-interval, one
// CUDA thread per sub-interval, state in registers (Sec. IV-B, Theorem
// Backward_HJB_LQT; boundary eq. abcej_boundary; terminal element Sec. IV-D,
// eq. LQT_final_initialisation).
//
// Also the coefficient preparation kernel: B = L U^-1 L^T is used only through
// a factor Lt = L R^-T (U = R R^T), so that A B J = (A Lt)(J Lt)^T,
// A B A^T = (A Lt)(A Lt)^T, J B J = (J Lt)(J Lt)^T and B eta = Lt (Lt^T eta);
// with m < n this cuts the FP64 work of every right-hand side.
#include <cuda_runtime.h>

#include "lqt_device.cuh"
#include "lqt_internal.h"
#include "lqt_uniform.cuh"

namespace lqt {

// ---------------------------------------------------------------------------
// coefficient preparation
// ---------------------------------------------------------------------------

struct PrepArgs {
  int32_t n, m, nr, K, M;
  int64_t T;
  Coef L, U, H, X, r;
  int32_t mode_Lt, mode_Q, mode_qr;
  int64_t cnt_Lt, cnt_Q, cnt_qr, cnt_Ku;
  double *Lt, *Q, *qr, *Ku;
};

// Index of the input sample that a derived sample s (of mode `dmode`) uses.
__device__ __forceinline__ int64_t input_index(int32_t imode, int32_t dmode, int64_t s, int32_t K, int64_t T) {
  if (imode == kConst) return 0;
  if (dmode == imode) return s;
  // dmode == kStageBlock: s = (2K+1) j + p
  const int64_t j = s / (2 * K + 1);
  const int32_t p = (int32_t)(s - j * (2 * K + 1));
  return sample_index(imode, j, p, K);
}

// Cholesky U = R R^T of the m x m sample (lower R, row-major), in place.
__device__ void cholesky_lower(double* R, int m) {
  for (int j = 0; j < m; ++j) {
    double d = R[j * m + j];
    for (int k = 0; k < j; ++k) d -= R[j * m + k] * R[j * m + k];
    if (!(d > 0.0)) flag(kStatusSingular);
    d = sqrt(d);
    R[j * m + j] = d;
    const double inv = 1.0 / d;
    for (int i = j + 1; i < m; ++i) {
      double s = R[i * m + j];
      for (int k = 0; k < j; ++k) s -= R[i * m + k] * R[j * m + k];
      R[i * m + j] = s * inv;
    }
    for (int i = 0; i < j; ++i) R[i * m + j] = 0.0;
  }
}

constexpr int kMaxM = 16;
constexpr int kMaxN = 64;

// One thread per derived sample; blockIdx.y selects the quantity (with two
// rows in the grid only Lt and Ku are made).
__global__ void prepare_kernel(PrepArgs a) {
  const int which = gridDim.y == 2 ? (blockIdx.y == 0 ? 0 : 3) : blockIdx.y;
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int n = a.n, m = a.m, nr = a.nr;
  if (which == 0) {  // Lt = L R^-T, zero-padded to M columns
    if (s >= a.cnt_Lt) return;
    const double* L = a.L.ptr + input_index(a.L.mode, a.mode_Lt, s, a.K, a.T) * n * m;
    const double* U = a.U.ptr + input_index(a.U.mode, a.mode_Lt, s, a.K, a.T) * m * m;
    double R[kMaxM * kMaxM];
    for (int i = 0; i < m * m; ++i) R[i] = U[i];
    cholesky_lower(R, m);
    double* out = a.Lt + s * n * a.M;
    for (int i = 0; i < n; ++i) {
      // solve Lt_i R^T = L_i  (forward substitution over columns)
      double row[kMaxM];
      for (int c = 0; c < m; ++c) {
        double v = L[i * m + c];
        for (int k = 0; k < c; ++k) v -= row[k] * R[c * m + k];
        row[c] = v / R[c * m + c];
      }
      for (int c = 0; c < a.M; ++c) out[i * a.M + c] = c < m ? row[c] : 0.0;
    }
  } else if (which == 1) {  // Q = H^T X H (full n x n, symmetrised); only when H is given
    if (s >= a.cnt_Q) return;
    const double* X = a.X.ptr + input_index(a.X.mode, a.mode_Q, s, a.K, a.T) * nr * nr;
    const double* H = a.H.ptr + input_index(a.H.mode, a.mode_Q, s, a.K, a.T) * nr * n;
    double* out = a.Q + s * (n * n);
    for (int i = 0; i < n; ++i)
      for (int j = i; j < n; ++j) {
        double vij = 0.0, vji = 0.0;
        for (int k = 0; k < nr; ++k)
          for (int l = 0; l < nr; ++l) {
            vij += H[k * n + i] * X[k * nr + l] * H[l * n + j];
            vji += H[k * n + j] * X[k * nr + l] * H[l * n + i];
          }
        out[i * n + j] = out[j * n + i] = 0.5 * (vij + vji);
      }
  } else if (which == 2) {  // qr = [H^T X r, r^T X r]
    if (s >= a.cnt_qr) return;
    const double* X = a.X.ptr + input_index(a.X.mode, a.mode_qr, s, a.K, a.T) * nr * nr;
    const double* H = a.H.ptr ? a.H.ptr + input_index(a.H.mode, a.mode_qr, s, a.K, a.T) * nr * n : nullptr;
    const double* r = a.r.ptr ? a.r.ptr + input_index(a.r.mode, a.mode_qr, s, a.K, a.T) * nr : nullptr;
    double* out = a.qr + s * (n + 1);
    double Xr[kMaxN];
    double rho = 0.0;
    for (int k = 0; k < nr; ++k) {
      double v = 0.0;
      if (r)
        for (int l = 0; l < nr; ++l) v += X[k * nr + l] * r[l];
      Xr[k] = v;
      if (r) rho += r[k] * v;
    }
    for (int i = 0; i < n; ++i) {
      double v;
      if (!H) {
        v = Xr[i];
      } else {
        v = 0.0;
        for (int k = 0; k < nr; ++k) v += H[k * n + i] * Xr[k];
      }
      out[i] = v;
    }
    out[n] = rho;
  } else {  // Ku = U^-1 L^T at the boundaries (solve U Ku = L^T)
    if (s >= a.cnt_Ku) return;
    // boundary k = s uses sample (j, p) = (k, 0), or (T-1, 2K) at k = T
    int64_t j = s < a.T ? s : a.T - 1;
    int32_t p = s < a.T ? 0 : 2 * a.K;
    if (a.cnt_Ku == 1) { j = 0; p = 0; }
    const double* L = a.L.ptr + sample_index(a.L.mode, j, p, a.K) * n * m;
    const double* U = a.U.ptr + sample_index(a.U.mode, j, p, a.K) * m * m;
    double R[kMaxM * kMaxM];
    for (int i = 0; i < m * m; ++i) R[i] = U[i];
    cholesky_lower(R, m);
    double* out = a.Ku + s * m * n;
    for (int col = 0; col < n; ++col) {
      double y[kMaxM];
      for (int i = 0; i < m; ++i) {  // R y = L^T[:, col]
        double v = L[col * m + i];
        for (int k = 0; k < i; ++k) v -= R[i * m + k] * y[k];
        y[i] = v / R[i * m + i];
      }
      for (int i = m - 1; i >= 0; --i) {  // R^T z = y
        double v = y[i];
        for (int k = i + 1; k < m; ++k) v -= R[k * m + i] * y[k];
        y[i] = v / R[i * m + i];
      }
      for (int i = 0; i < m; ++i) out[i * n + col] = y[i];
    }
  }
}

// Lt and Ku of one (L, U) sample by a CTA of 128 threads (n <= 64): the
// Cholesky factor in shared memory (R, kMaxM^2), its columns and updates over
// the threads, then one thread per row of Lt (threads 0 .. 63) and per column
// of Ku (64 .. 127).  The sums run in the order of prepare_kernel's.
__device__ void prepare_sample_cta(int n, int m, int M, const double* __restrict__ L, const double* __restrict__ U,
                                   double* __restrict__ Lt, double* __restrict__ Ku, double* R) {
  const int tid = threadIdx.x;
  for (int e = tid; e < m * m; e += blockDim.x) R[e] = U[e];
  __syncthreads();
  for (int j = 0; j < m; ++j) {
    if (tid == 0) {
      const double d = R[j * m + j];
      if (!(d > 0.0)) flag(kStatusSingular);
      R[j * m + j] = sqrt(d);
    }
    __syncthreads();
    const double inv = 1.0 / R[j * m + j];
    if (tid < j) R[tid * m + j] = 0.0;
    if (tid > j && tid < m) R[tid * m + j] *= inv;
    __syncthreads();
    const int w = m - 1 - j;
    for (int e = tid; e < w * w; e += blockDim.x) {
      const int i = j + 1 + e / w, k = j + 1 + e % w;
      if (k <= i) R[i * m + k] = fma(-R[i * m + j], R[k * m + j], R[i * m + k]);
    }
    __syncthreads();
  }
  if (tid < n) {  // Lt_i R^T = L_i
    double row[kMaxM];
#pragma unroll
    for (int c = 0; c < kMaxM; ++c) {
      row[c] = 0.0;
      if (c < m) {
        double v = L[tid * m + c];
#pragma unroll
        for (int k = 0; k < c; ++k) v = fma(-row[k], R[c * m + k], v);
        row[c] = v / R[c * m + c];
      }
      if (c < M) Lt[tid * M + c] = row[c];
    }
  } else if (tid >= 64 && tid - 64 < n) {  // R y = L^T[:, col], R^T z = y
    const int col = tid - 64;
    double y[kMaxM];
#pragma unroll
    for (int i = 0; i < kMaxM; ++i) {
      y[i] = 0.0;
      if (i < m) {
        double v = L[col * m + i];
#pragma unroll
        for (int k = 0; k < i; ++k) v = fma(-R[i * m + k], y[k], v);
        y[i] = v / R[i * m + i];
      }
    }
#pragma unroll
    for (int i = kMaxM - 1; i >= 0; --i)
      if (i < m) {
        double v = y[i];
#pragma unroll
        for (int k = i + 1; k < kMaxM; ++k)
          if (k < m) v = fma(-R[k * m + i], y[k], v);
        y[i] = v / R[i * m + i];
        Ku[i * n + col] = y[i];
      }
  }
}

// Constant L and U: their one sample by one CTA.  A thread alone took 21 us at
// n = 4, m = 2, 163 us at n = 16, m = 8 and 1.49 ms at n = 64, m = 16, with the
// rest of the GPU waiting.
__global__ void __launch_bounds__(128) prepare_const_kernel(int n, int m, int M, const double* L, const double* U,
                                                            double* Lt, double* Ku) {
  __shared__ double R[kMaxM * kMaxM];
  prepare_sample_cta(n, m, M, L, U, Lt, Ku, R);
}

// q = X r, rho = r^T X r per sample when H is the identity (one thread per
// sample, loops unrolled for the compiled n).
template <int N>
__global__ void __launch_bounds__(256) qr_identity_kernel(const double* __restrict__ X, int32_t X_mode,
                                                          const double* __restrict__ r, int32_t r_mode, int32_t dmode,
                                                          int64_t cnt, int32_t K, int64_t T, double* __restrict__ qr) {
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= cnt) return;
  const double* Xs = X + input_index(X_mode, dmode, s, K, T) * N * N;
  double rr[N], q[N];
  if (r) {
    const double* rs = r + input_index(r_mode, dmode, s, K, T) * N;
#pragma unroll
    for (int i = 0; i < N; ++i) rr[i] = rs[i];
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) rr[i] = 0.0;
  }
  double rho = 0.0;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    double v = 0.0;
#pragma unroll
    for (int l = 0; l < N; ++l) v = fma(Xs[i * N + l], rr[l], v);
    q[i] = v;
    rho = fma(rr[i], v, rho);
  }
  double* out = qr + s * (N + 1);
#pragma unroll
  for (int i = 0; i < N; ++i) out[i] = q[i];
  out[N] = rho;
}

// The same with N consecutive threads per sample (N a power of two <= 32),
// thread i forming row i of X r: a warp reads 32 consecutive rows, so the
// stream of X samples (the largest input when X is sampled per half-step) is
// read in full 128-byte lines; rho is reduced over the N lanes.
template <int N, bool VEC>
__global__ void __launch_bounds__(256) qr_rows_kernel(const double* __restrict__ X, int32_t X_mode,
                                                      const double* __restrict__ r, int32_t r_mode, int32_t dmode,
                                                      int64_t cnt, int32_t K, int64_t T, double* __restrict__ qr) {
  static_assert(N >= 2 && N <= 32 && (N & (N - 1)) == 0, "rows kernel needs a power-of-two N <= 32");
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t s = tid / N;
  const int i = (int)(tid % N);
  const bool live = s < cnt;
  double q = 0.0, ri = 0.0;
  if (live) {
    const double* row = X + input_index(X_mode, dmode, s, K, T) * N * N + i * N;
    if (r) {
      const double* rs = r + input_index(r_mode, dmode, s, K, T) * N;
      if constexpr (VEC) {
        // X and r start on 16-byte boundaries (checked by the launcher) and N is
        // even, so every row and sample does: read them in pairs
        const double2* row2 = reinterpret_cast<const double2*>(row);
        const double2* rs2 = reinterpret_cast<const double2*>(rs);
#pragma unroll
        for (int l = 0; l < N / 2; ++l) {
          const double2 a = __ldg(row2 + l), b = __ldg(rs2 + l);
          q = fma(a.x, b.x, q);
          q = fma(a.y, b.y, q);
        }
      } else {
#pragma unroll
        for (int l = 0; l < N; ++l) q = fma(row[l], rs[l], q);
      }
      ri = rs[i];
    }
  }
  double rho = ri * q;
#pragma unroll
  for (int o = N / 2; o > 0; o >>= 1) rho += __shfl_xor_sync(0xffffffffu, rho, o);
  if (live) {
    qr[s * (N + 1) + i] = q;
    if (i == 0) qr[s * (N + 1) + N] = rho;
  }
}

// The same with 64 threads per sample (N = 64), thread i forming row i of X r;
// its row's lines stay in L1 over the row's 64 entries (one thread per sample:
// 286 us at T = 4096).
__global__ void __launch_bounds__(256) qr_rows64_kernel(const double* __restrict__ X, int32_t X_mode,
                                                        const double* __restrict__ r, int32_t r_mode, int32_t dmode,
                                                        int64_t cnt, int32_t K, int64_t T, double* __restrict__ qr) {
  __shared__ double rs[4][64], part[8];
  const int g = threadIdx.x >> 6, i = threadIdx.x & 63;
  const int64_t s = (int64_t)blockIdx.x * 4 + g;
  const bool live = s < cnt;
  rs[g][i] = (live && r) ? r[input_index(r_mode, dmode, s, K, T) * 64 + i] : 0.0;
  __syncthreads();
  double q = 0.0;
  if (live && r) {
    const double* row = X + input_index(X_mode, dmode, s, K, T) * 4096 + i * 64;
#pragma unroll 8
    for (int l = 0; l < 64; ++l) q = fma(row[l], rs[g][l], q);
  }
  double rho = rs[g][i] * q;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) rho += __shfl_xor_sync(0xffffffffu, rho, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = rho;
  __syncthreads();
  if (live) {
    qr[s * 65 + i] = q;
    if (i == 0) qr[s * 65 + 64] = part[2 * g] + part[2 * g + 1];
  }
}

template <int N>
static void launch_qr_identity(const PrepArgs& a, cudaStream_t st) {
  const int threads = 256;
  if constexpr (N >= 2 && N <= 32 && (N & (N - 1)) == 0) {
    const int64_t total = a.cnt_qr * N;
    const unsigned grid = (unsigned)((total + threads - 1) / threads);
    const bool vec = ((reinterpret_cast<uintptr_t>(a.X.ptr) | reinterpret_cast<uintptr_t>(a.r.ptr)) & 15u) == 0;
    if (vec)
      qr_rows_kernel<N, true><<<grid, threads, 0, st>>>(a.X.ptr, a.X.mode, a.r.ptr, a.r.mode, a.mode_qr, a.cnt_qr,
                                                         a.K, a.T, a.qr);
    else
      qr_rows_kernel<N, false><<<grid, threads, 0, st>>>(a.X.ptr, a.X.mode, a.r.ptr, a.r.mode, a.mode_qr, a.cnt_qr,
                                                          a.K, a.T, a.qr);
  } else if constexpr (N == 64) {
    qr_rows64_kernel<<<(unsigned)((a.cnt_qr + 3) / 4), threads, 0, st>>>(a.X.ptr, a.X.mode, a.r.ptr, a.r.mode,
                                                                          a.mode_qr, a.cnt_qr, a.K, a.T, a.qr);
  } else {
    qr_identity_kernel<N><<<(unsigned)((a.cnt_qr + threads - 1) / threads), threads, 0, st>>>(
        a.X.ptr, a.X.mode, a.r.ptr, a.r.mode, a.mode_qr, a.cnt_qr, a.K, a.T, a.qr);
  }
  count_launch();
}

// The derived coefficients of problem p into the given arrays (Lt, Q, qr, Ku
// laid out as the Layout's modes say); cf describes p's coefficients with
// those arrays.  Q is written only when H is given.
cudaError_t launch_prepare_into(const lqt_problem& p, const Layout& lay, double* Lt, double* Q, double* qr,
                                double* Ku, Coefs& cf, cudaStream_t st) {
  PrepArgs a;
  a.n = p.n; a.m = p.m; a.nr = p.nr; a.K = p.K; a.M = lay.M; a.T = p.T;
  a.L = {p.L.ptr, p.L.mode};
  a.U = {p.U.ptr, p.U.mode};
  a.H = {p.H.ptr, p.H.mode};
  a.X = {p.X.ptr, p.X.mode};
  a.r = {p.r.ptr, p.r.mode};
  a.mode_Lt = lay.mode_Lt; a.mode_Q = lay.mode_Q; a.mode_qr = lay.mode_qr;
  a.cnt_Lt = sample_count(lay.mode_Lt, p.T, p.K);
  a.cnt_Q = sample_count(lay.mode_Q, p.T, p.K);
  a.cnt_qr = sample_count(lay.mode_qr, p.T, p.K);
  const bool ku_const = p.L.mode == LQT_CONST && p.U.mode == LQT_CONST;
  a.cnt_Ku = ku_const ? 1 : p.T + 1;
  a.Lt = Lt;
  a.Q = Q;
  a.qr = qr;
  a.Ku = Ku;
  // Lt and Ku always; H^T X H only when H is given; H^T X r by the dedicated
  // kernel when H is the identity.
  const bool h_identity = p.H.ptr == nullptr;
  int64_t most = a.cnt_Lt > a.cnt_Ku ? a.cnt_Lt : a.cnt_Ku;
  if (!h_identity) {
    if (a.cnt_Q > most) most = a.cnt_Q;
    if (a.cnt_qr > most) most = a.cnt_qr;
  }
  const int threads = 128;
  const int64_t blocks = (most + threads - 1) / threads;
  if (h_identity) {
    if (a.cnt_Lt == 1 && a.cnt_Ku == 1)
      prepare_const_kernel<<<1, 128, 0, st>>>(a.n, a.m, a.M, a.L.ptr, a.U.ptr, a.Lt, a.Ku);
    else  // which = 0 (Lt) and 3 (Ku): map blockIdx.y 0 -> 0, 1 -> 3
      prepare_kernel<<<dim3((unsigned)blocks, 2), threads, 0, st>>>(a);
    count_launch();
    switch (p.n) {
      case 1: launch_qr_identity<1>(a, st); break;
      case 2: launch_qr_identity<2>(a, st); break;
      case 3: launch_qr_identity<3>(a, st); break;
      case 4: launch_qr_identity<4>(a, st); break;
      case 8: launch_qr_identity<8>(a, st); break;
      case 16: launch_qr_identity<16>(a, st); break;
      case 64: launch_qr_identity<64>(a, st); break;
      default: return cudaErrorInvalidValue;
    }
  } else {
    prepare_kernel<<<dim3((unsigned)blocks, 4), threads, 0, st>>>(a);
    count_launch();
  }
  cf = coefs_view(p, lay, Lt, Q, qr, Ku);
  return cudaGetLastError();
}

Coefs coefs_view(const lqt_problem& p, const Layout& lay, double* Lt, double* Q, double* qr, double* Ku) {
  const bool h_identity = p.H.ptr == nullptr;
  const bool ku_const = p.L.mode == LQT_CONST && p.U.mode == LQT_CONST;
  Coefs cf;
  cf.F = {p.F.ptr, p.F.mode};
  cf.c = {p.c.ptr, p.c.ptr ? p.c.mode : kConst};
  cf.Lt = {Lt, lay.mode_Lt};
  cf.Q = h_identity ? Coef{p.X.ptr, p.X.mode} : Coef{Q, lay.mode_Q};
  cf.qr = {qr, lay.mode_qr};
  cf.Ku = Ku;
  cf.Ku_per_boundary = ku_const ? 0 : 1;
  cf.M = lay.M;
  cf.uni = nullptr;
  cf.repeat = nullptr;
  return cf;
}

cudaError_t launch_prepare_coefs(const lqt_problem& p, const Layout& lay, char* ws, Coefs& cf, cudaStream_t st) {
  const cudaError_t e = launch_prepare_into(p, lay, (double*)(ws + lay.off_Lt), (double*)(ws + lay.off_Q),
                                            (double*)(ws + lay.off_qr), (double*)(ws + lay.off_Ku), cf, st);
  if (lay.uniform) cf.uni = (const double*)(ws + lay.off_uni);
  return e;
}

// ---------------------------------------------------------------------------
// element build
// ---------------------------------------------------------------------------

// Right-hand side of the backward conditional HJB ODEs in s:
//   dA/ds    =  A B J - A F                = AL P^T - A F
//   db/ds    = -A B eta - A c               = -AL w - A c
//   dC/ds    = -A B A^T                     = -AL AL^T
//   deta/ds  = -q - F^T eta + J c + J B eta = -q - F^T eta + J c + P w
//   dJ/ds    = -Q - J F - F^T J + J B J     = -Q - JF - (JF)^T + P P^T
//   dzeta/ds = -rho/2 + eta^T B eta / 2 + eta^T c = -rho/2 + |w|^2/2 + eta^T c
// with AL = A Lt, P = J Lt, w = Lt^T eta, q = H^T X r, rho = r^T X r.
//
// nzF, nzL: bit l N + j (l M + a) is set where F_lj (Lt_la) may be nonzero.
// With constant F and L the bits are the same in every thread of a warp, and a
// product by an exact zero is skipped by a branch instead of taking its 64
// cycles of the FP64 pipe: models made of integrator chains have few nonzeros
// (the point mass: 2 of 16 in F, 2 of 8 in L; its right-hand side then takes
// 146 FP64 instructions of 300).  Dense or sampled F, L: every bit set.
//
// ROLE: the fields this thread integrates, kCostSide (eta, J, zeta), kFlowSide
// (A, b, C) or both.  The cost side is closed in itself and hands P and w on
// with `give`; the flow side alone takes them with `take`.
constexpr int kCostSide = 1, kFlowSide = 2, kBothSides = 3;

struct NoExchange {
  template <int N, int M>
  __device__ __forceinline__ void give(const double*, const double*) {}
  template <int N, int M>
  __device__ __forceinline__ void take(double*, double*) {}
};

template <int N, int M, int ROLE, class X>
__device__ __forceinline__ void element_rhs_by_entry(const Elem<N>& y, const double* __restrict__ F,
                                                     const double* __restrict__ c, const double* __restrict__ Lt,
                                                     const double* __restrict__ Q, const double* __restrict__ qr,
                                                     Elem<N>& k, unsigned long long nzF, unsigned long long nzL,
                                                     X xch) {
  constexpr bool kFlow = (ROLE & kFlowSide) != 0, kCost = (ROLE & kCostSide) != 0;
  double AL[N * M], P[N * M], w[M];
#pragma unroll
  for (int e = 0; e < N * M; ++e) AL[e] = P[e] = 0.0;
#pragma unroll
  for (int a = 0; a < M; ++a) w[a] = 0.0;
#pragma unroll
  for (int l = 0; l < N; ++l)
#pragma unroll
    for (int a = 0; a < M; ++a)
      for (unsigned on = taken_if(nzL >> (l * M + a) & 1ull); on != 0u; on >>= 1) {
        const double lt = Lt[l * M + a];
#pragma unroll
        for (int i = 0; i < N; ++i) {
          if constexpr (kFlow) AL[i * M + a] = fma(y.A[i * N + l], lt, AL[i * M + a]);
          if constexpr (kCost) P[i * M + a] = fma(y.J[sidx<N>(i, l)], lt, P[i * M + a]);
        }
        if constexpr (kCost) w[a] = fma(lt, y.eta[l], w[a]);
      }
  if constexpr (ROLE == kCostSide) xch.template give<N, M>(P, w);
  if constexpr (ROLE == kFlowSide) xch.template take<N, M>(P, w);
  // dA = AL P^T - A F, JF = J F, deta = -q - F^T eta ...
  double JF[N * N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    if constexpr (kCost) k.eta[i] = -qr[i];
#pragma unroll
    for (int j = 0; j < N; ++j) {
      if constexpr (kFlow) {
        double s = 0.0;
#pragma unroll
        for (int a = 0; a < M; ++a) s = fma(AL[i * M + a], P[j * M + a], s);
        k.A[i * N + j] = s;
      }
      JF[i * N + j] = 0.0;
    }
  }
#pragma unroll
  for (int l = 0; l < N; ++l)
#pragma unroll
    for (int j = 0; j < N; ++j)
      for (unsigned on = taken_if(nzF >> (l * N + j) & 1ull); on != 0u; on >>= 1) {
        const double f = F[l * N + j];
#pragma unroll
        for (int i = 0; i < N; ++i) {
          if constexpr (kFlow) k.A[i * N + j] = fma(-y.A[i * N + l], f, k.A[i * N + j]);
          if constexpr (kCost) JF[i * N + j] = fma(y.J[sidx<N>(i, l)], f, JF[i * N + j]);
        }
        if constexpr (kCost) k.eta[j] = fma(-f, y.eta[l], k.eta[j]);
      }
  if constexpr (kFlow) {
    // db = -AL w - A c
#pragma unroll
    for (int i = 0; i < N; ++i) {
      double s = 0.0;
#pragma unroll
      for (int a = 0; a < M; ++a) s = fma(-AL[i * M + a], w[a], s);
      if (c) {
#pragma unroll
        for (int l = 0; l < N; ++l) s = fma(-y.A[i * N + l], c[l], s);
      }
      k.b[i] = s;
    }
    // dC = -AL AL^T
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
      for (int j = i; j < N; ++j) {
        double s = 0.0;
#pragma unroll
        for (int a = 0; a < M; ++a) s = fma(-AL[i * M + a], AL[j * M + a], s);
        k.C[sidx<N>(i, j)] = s;
      }
  }
  if constexpr (kCost) {
    // deta ... + J c + P w
#pragma unroll
    for (int i = 0; i < N; ++i) {
      double s = k.eta[i];
      if (c) {
#pragma unroll
        for (int l = 0; l < N; ++l) s = fma(y.J[sidx<N>(i, l)], c[l], s);
      }
#pragma unroll
      for (int a = 0; a < M; ++a) s = fma(P[i * M + a], w[a], s);
      k.eta[i] = s;
    }
    // dJ = -Q - JF - (JF)^T + P P^T
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
      for (int j = i; j < N; ++j) {
        double s = -Q[i * N + j] - JF[i * N + j] - JF[j * N + i];
#pragma unroll
        for (int a = 0; a < M; ++a) s = fma(P[i * M + a], P[j * M + a], s);
        k.J[sidx<N>(i, j)] = s;
      }
    // dzeta
    double z = -0.5 * qr[N];
#pragma unroll
    for (int a = 0; a < M; ++a) z = fma(0.5 * w[a], w[a], z);
    if (c) {
#pragma unroll
      for (int l = 0; l < N; ++l) z = fma(y.eta[l], c[l], z);
    }
    k.zeta = z;
  }
}

// The same without the branches around each entry, output by output: at n = 8 a
// thread's fields are mostly spilled, and with every bit set the order above,
// which keeps whole products in flight, was slower (n = 8, uneven grid, T = 40000:
// 8.29 ms against 6.94 so; the same sums in the same order, so the same bits).
template <int N, int M>
__device__ __forceinline__ void element_rhs_dense(const Elem<N>& y, const double* __restrict__ F,
                                                  const double* __restrict__ c, const double* __restrict__ Lt,
                                                  const double* __restrict__ Q, const double* __restrict__ qr,
                                                  Elem<N>& k) {
  double AL[N * M], P[N * M], w[M];
#pragma unroll
  for (int i = 0; i < N; ++i)
#pragma unroll
    for (int a = 0; a < M; ++a) {
      double s1 = 0.0, s2 = 0.0;
#pragma unroll
      for (int l = 0; l < N; ++l) {
        const double lt = Lt[l * M + a];
        s1 = fma(y.A[i * N + l], lt, s1);
        s2 = fma(y.J[sidx<N>(i, l)], lt, s2);
      }
      AL[i * M + a] = s1;
      P[i * M + a] = s2;
    }
#pragma unroll
  for (int a = 0; a < M; ++a) {
    double s = 0.0;
#pragma unroll
    for (int l = 0; l < N; ++l) s = fma(Lt[l * M + a], y.eta[l], s);
    w[a] = s;
  }
  // dA = AL P^T - A F
#pragma unroll
  for (int i = 0; i < N; ++i)
#pragma unroll
    for (int j = 0; j < N; ++j) {
      double s = 0.0;
#pragma unroll
      for (int a = 0; a < M; ++a) s = fma(AL[i * M + a], P[j * M + a], s);
#pragma unroll
      for (int l = 0; l < N; ++l) s = fma(-y.A[i * N + l], F[l * N + j], s);
      k.A[i * N + j] = s;
    }
  // db = -AL w - A c
#pragma unroll
  for (int i = 0; i < N; ++i) {
    double s = 0.0;
#pragma unroll
    for (int a = 0; a < M; ++a) s = fma(-AL[i * M + a], w[a], s);
    if (c) {
#pragma unroll
      for (int l = 0; l < N; ++l) s = fma(-y.A[i * N + l], c[l], s);
    }
    k.b[i] = s;
  }
  // dC = -AL AL^T
#pragma unroll
  for (int i = 0; i < N; ++i)
#pragma unroll
    for (int j = i; j < N; ++j) {
      double s = 0.0;
#pragma unroll
      for (int a = 0; a < M; ++a) s = fma(-AL[i * M + a], AL[j * M + a], s);
      k.C[sidx<N>(i, j)] = s;
    }
  // deta = -q - F^T eta + J c + P w
#pragma unroll
  for (int i = 0; i < N; ++i) {
    double s = -qr[i];
#pragma unroll
    for (int l = 0; l < N; ++l) s = fma(-F[l * N + i], y.eta[l], s);
    if (c) {
#pragma unroll
      for (int l = 0; l < N; ++l) s = fma(y.J[sidx<N>(i, l)], c[l], s);
    }
#pragma unroll
    for (int a = 0; a < M; ++a) s = fma(P[i * M + a], w[a], s);
    k.eta[i] = s;
  }
  // dJ = -Q - JF - (JF)^T + P P^T
  double JF[N * N];
#pragma unroll
  for (int i = 0; i < N; ++i)
#pragma unroll
    for (int j = 0; j < N; ++j) {
      double s = 0.0;
#pragma unroll
      for (int l = 0; l < N; ++l) s = fma(y.J[sidx<N>(i, l)], F[l * N + j], s);
      JF[i * N + j] = s;
    }
#pragma unroll
  for (int i = 0; i < N; ++i)
#pragma unroll
    for (int j = i; j < N; ++j) {
      double s = -Q[i * N + j] - JF[i * N + j] - JF[j * N + i];
#pragma unroll
      for (int a = 0; a < M; ++a) s = fma(P[i * M + a], P[j * M + a], s);
      k.J[sidx<N>(i, j)] = s;
    }
  // dzeta
  double z = -0.5 * qr[N];
#pragma unroll
  for (int a = 0; a < M; ++a) z = fma(0.5 * w[a], w[a], z);
  if (c) {
#pragma unroll
    for (int l = 0; l < N; ++l) z = fma(y.eta[l], c[l], z);
  }
  k.zeta = z;
}

// n = 8 out of line: its fields are in local memory either way, and inlined at
// each of the four stages the two forms took minutes to compile.
template <int M, bool kDense>
static __device__ __noinline__ void element_rhs8(const Elem<8>& y, const double* F, const double* c, const double* Lt,
                                                 const double* Q, const double* qr, Elem<8>& k,
                                                 unsigned long long nzF, unsigned long long nzL) {
  if constexpr (kDense)
    element_rhs_dense<8, M>(y, F, c, Lt, Q, qr, k);
  else
    element_rhs_by_entry<8, M, kBothSides>(y, F, c, Lt, Q, qr, k, nzF, nzL, NoExchange());
}

template <int N, int M, int ROLE, class X>
__device__ __forceinline__ void element_rhs(const Elem<N>& y, const double* __restrict__ F,
                                            const double* __restrict__ c, const double* __restrict__ Lt,
                                            const double* __restrict__ Q, const double* __restrict__ qr,
                                            Elem<N>& k, unsigned long long nzF, unsigned long long nzL, X xch) {
  if constexpr (N == 8) {
    if (8 * __popcll(nzF) >= 7 * N * N)  // F (nearly) full
      element_rhs8<M, true>(y, F, c, Lt, Q, qr, k, nzF, nzL);
    else
      element_rhs8<M, false>(y, F, c, Lt, Q, qr, k, nzF, nzL);
  } else {
    element_rhs_by_entry<N, M, ROLE>(y, F, c, Lt, Q, qr, k, nzF, nzL, xch);
  }
}

// The right-hand side at the boundary A = I, J = 0, eta = 0, where every
// sub-interval starts.
template <int N, int M, int ROLE = kBothSides>
__device__ __forceinline__ void element_rhs_start(const double* __restrict__ F, const double* __restrict__ c,
                                                  const double* __restrict__ Lt, const double* __restrict__ Q,
                                                  const double* __restrict__ qr, Elem<N>& k) {
  if constexpr ((ROLE & kFlowSide) != 0) {
#pragma unroll
    for (int e = 0; e < N * N; ++e) k.A[e] = 0.0 - F[e];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      k.b[i] = c ? 0.0 - c[i] : 0.0;
#pragma unroll
      for (int j = i; j < N; ++j) {
        double s = 0.0;
#pragma unroll
        for (int a = 0; a < M; ++a) s = fma(-Lt[i * M + a], Lt[j * M + a], s);
        k.C[sidx<N>(i, j)] = s;
      }
    }
  }
  if constexpr ((ROLE & kCostSide) != 0) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      k.eta[i] = -qr[i];
#pragma unroll
      for (int j = i; j < N; ++j) k.J[sidx<N>(i, j)] = -Q[i * N + j];
    }
    k.zeta = -0.5 * qr[N];
  }
}

// y <- base + s * k over every field of ROLE.
template <int N, int ROLE = kBothSides>
__device__ __forceinline__ void axpy_to(Elem<N>& y, const Elem<N>& base, double s, const Elem<N>& k) {
  if constexpr ((ROLE & kFlowSide) != 0) {
#pragma unroll
    for (int i = 0; i < N * N; ++i) y.A[i] = fma(s, k.A[i], base.A[i]);
#pragma unroll
    for (int i = 0; i < N; ++i) y.b[i] = fma(s, k.b[i], base.b[i]);
#pragma unroll
    for (int i = 0; i < Dim<N>::NS; ++i) y.C[i] = fma(s, k.C[i], base.C[i]);
  }
  if constexpr ((ROLE & kCostSide) != 0) {
#pragma unroll
    for (int i = 0; i < N; ++i) y.eta[i] = fma(s, k.eta[i], base.eta[i]);
#pragma unroll
    for (int i = 0; i < Dim<N>::NS; ++i) y.J[i] = fma(s, k.J[i], base.J[i]);
    y.zeta = fma(s, k.zeta, base.zeta);
  }
}

// The same over A, eta and J, which drive the element flow: b, C and zeta
// appear on no right-hand side, so a stage input needs none of them.
template <int N, int ROLE = kBothSides>
__device__ __forceinline__ void axpy_flow(Elem<N>& y, const Elem<N>& base, double s, const Elem<N>& k) {
  if constexpr ((ROLE & kFlowSide) != 0) {
#pragma unroll
    for (int i = 0; i < N * N; ++i) y.A[i] = fma(s, k.A[i], base.A[i]);
  }
  if constexpr ((ROLE & kCostSide) != 0) {
#pragma unroll
    for (int i = 0; i < N; ++i) y.eta[i] = fma(s, k.eta[i], base.eta[i]);
#pragma unroll
    for (int i = 0; i < Dim<N>::NS; ++i) y.J[i] = fma(s, k.J[i], base.J[i]);
  }
}

struct BuildArgs {
  int64_t T;
  int32_t K;
  const double* t;
  Coefs cf;
  ElemPtrs out;
};

template <int N>
__device__ __forceinline__ const double* coef_at(const Coef& c, int64_t j, int32_t p, int32_t K, int stride) {
  return c.ptr + sample_index(c.mode, j, p, K) * stride;
}

// Element y in the full layout (A, b, C, eta, J with C and J written in full,
// zeta): 3 N^2 + 2 N + 1 doubles at dst.
template <int N>
__device__ __forceinline__ void store_full(const Elem<N>& y, double* dst) {
  double* o = dst;
#pragma unroll
  for (int i = 0; i < N * N; ++i) *o++ = y.A[i];
#pragma unroll
  for (int i = 0; i < N; ++i) *o++ = y.b[i];
#pragma unroll
  for (int i = 0; i < N; ++i)
#pragma unroll
    for (int c = 0; c < N; ++c) *o++ = y.C[sidx<N>(i, c)];
#pragma unroll
  for (int i = 0; i < N; ++i) *o++ = y.eta[i];
#pragma unroll
  for (int i = 0; i < N; ++i)
#pragma unroll
    for (int c = 0; c < N; ++c) *o++ = y.J[sidx<N>(i, c)];
  *o = y.zeta;
}

// K classical RK4 steps of the backward conditional HJB ODEs for sub-interval
// j, from the boundary A = I, b = C = eta = J = 0, zeta = 0 at s = t_{j+1}
// down to s = t_j (Sec. IV-B, eq. abcej_boundary).  With kStages the four
// stage inputs of every step go to stages[i][0..3] (full layout), for the
// discrete adjoint's reverse sweep.
template <int N, int M, bool kStages = false, int ROLE = kBothSides, class X = NoExchange>
__device__ __forceinline__ void build_one(const Coefs& cf, const double* t, int64_t j, int32_t K, Elem<N>& y,
                                          double* stages = nullptr, X xch = X()) {
  constexpr int FS = 3 * N * N + 2 * N + 1;
  const double h = (t[j + 1] - t[j]) / K;
  Elem<N> yn, yt, k;
#pragma unroll
  for (int i = 0; i < N * N; ++i) y.A[i] = (i % (N + 1) == 0) ? 1.0 : 0.0;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    y.b[i] = 0.0;
    y.eta[i] = 0.0;
  }
#pragma unroll
  for (int i = 0; i < Dim<N>::NS; ++i) {
    y.C[i] = 0.0;
    y.J[i] = 0.0;
  }
  y.zeta = 0.0;
  if constexpr (kStages) yt = y;  // the stored b, C, zeta of a stage input are zero
  const unsigned long long nzF = nonzero_bits<N * N>(cf.F), nzL = nonzero_bits<N * M>(cf.Lt);
  for (int32_t i = K - 1; i >= 0; --i) {
    // stage times (in half steps from t_j): 2i+2, 2i+1, 2i+1, 2i
    const int32_t ps[3] = {2 * i + 2, 2 * i + 1, 2 * i};
    const double* F[3];
    const double* c[3];
    const double* Lt[3];
    const double* Q[3];
    const double* qr[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      F[q] = coef_at<N>(cf.F, j, ps[q], K, N * N);
      c[q] = cf.c.ptr ? coef_at<N>(cf.c, j, ps[q], K, N) : nullptr;
      Lt[q] = coef_at<N>(cf.Lt, j, ps[q], K, N * M);
      Q[q] = coef_at<N>(cf.Q, j, ps[q], K, N * N);
      qr[q] = coef_at<N>(cf.qr, j, ps[q], K, N + 1);
    }
    double* st = kStages ? stages + (int64_t)i * 4 * FS : nullptr;
    if constexpr (kStages) store_full<N>(y, st);
    if (i == K - 1)
      element_rhs_start<N, M, ROLE>(F[0], c[0], Lt[0], Q[0], qr[0], k);
    else
      element_rhs<N, M, ROLE>(y, F[0], c[0], Lt[0], Q[0], qr[0], k, nzF, nzL, xch);
    axpy_to<N, ROLE>(yn, y, -h / 6.0, k);
    axpy_flow<N, ROLE>(yt, y, -0.5 * h, k);
    if constexpr (kStages) store_full<N>(yt, st + FS);
    element_rhs<N, M, ROLE>(yt, F[1], c[1], Lt[1], Q[1], qr[1], k, nzF, nzL, xch);
    axpy_to<N, ROLE>(yn, yn, -h / 3.0, k);
    axpy_flow<N, ROLE>(yt, y, -0.5 * h, k);
    if constexpr (kStages) store_full<N>(yt, st + 2 * FS);
    element_rhs<N, M, ROLE>(yt, F[1], c[1], Lt[1], Q[1], qr[1], k, nzF, nzL, xch);
    axpy_to<N, ROLE>(yn, yn, -h / 3.0, k);
    axpy_flow<N, ROLE>(yt, y, -h, k);
    if constexpr (kStages) store_full<N>(yt, st + 3 * FS);
    element_rhs<N, M, ROLE>(yt, F[2], c[2], Lt[2], Q[2], qr[2], k, nzF, nzL, xch);
    axpy_to<N, ROLE>(y, yn, -h / 6.0, k);
  }
}

template <int N, int M>
__global__ void __launch_bounds__(128) build_kernel(BuildArgs a) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= a.T || uniform_near(a.cf.uni, a.t, j, a.K)) return;
  Elem<N> y;
  build_one<N, M>(a.cf, a.t, j, a.K, y);
  store_public<N>(a.out, j, y);
}

// The cost side's P = J Lt and w = Lt^T eta of one right-hand side, from the
// first warp of a 64-thread CTA to the second through one of two buffers in
// shared memory.  One barrier per right-hand side: a buffer is written again
// two right-hand sides later, after the barrier of the one between, which the
// reader reaches only when it has read.
struct PairExchange {
  double* buf;    // two buffers of (N M + M) x 32
  unsigned* odd;  // this thread's count of exchanges, low bit
  // the two warps meet from different code, so by a named barrier
  __device__ __forceinline__ void meet() { asm volatile("barrier.sync 1, 64;" ::: "memory"); }
  template <int N, int M>
  __device__ __forceinline__ double* slot() {
    double* p = buf + (*odd & 1u) * ((N * M + M) * 32) + (threadIdx.x & 31);
    *odd ^= 1u;
    return p;
  }
  template <int N, int M>
  __device__ __forceinline__ void give(const double* P, const double* w) {
    double* p = slot<N, M>();
#pragma unroll
    for (int e = 0; e < N * M; ++e) p[e * 32] = P[e];
#pragma unroll
    for (int a = 0; a < M; ++a) p[(N * M + a) * 32] = w[a];
    meet();
  }
  template <int N, int M>
  __device__ __forceinline__ void take(double* P, double* w) {
    meet();
    const double* p = slot<N, M>();
#pragma unroll
    for (int e = 0; e < N * M; ++e) P[e] = p[e * 32];
#pragma unroll
    for (int a = 0; a < M; ++a) w[a] = p[(N * M + a) * 32];
  }
};

// Two warps per 32 sub-intervals: the first integrates eta, J, zeta, the second
// A, b, C (about half of the FP64 instructions each), exchanging P and w once
// per right-hand side.  The results are the same bits as build_kernel's.  A
// warp alone on its sub-partition waits for its own FP64 results between
// issues; two warps, and half of the chain, hide that.  Lanes without a
// sub-interval of their own integrate the last one and store nothing, so that
// every thread meets every barrier.
template <int N, int M>
__global__ void __launch_bounds__(64) build_pair_kernel(BuildArgs a) {
  __shared__ double buf[2 * (N * M + M) * 32];
  int64_t j = (int64_t)blockIdx.x * 32 + (threadIdx.x & 31);
  const bool live = j < a.T && !uniform_near(a.cf.uni, a.t, j, a.K);
  if (!__syncthreads_or(live)) return;
  if (j >= a.T) j = a.T - 1;
  unsigned odd = 0;
  const PairExchange xch{buf, &odd};
  Elem<N> y;
  if (threadIdx.x < 32) {
    build_one<N, M, false, kCostSide>(a.cf, a.t, j, a.K, y, nullptr, xch);
    if (live) store_public_cost<N>(a.out, j, y);
  } else {
    build_one<N, M, false, kFlowSide>(a.cf, a.t, j, a.K, y, nullptr, xch);
    if (live) store_public_flow<N>(a.out, j, y);
  }
}

// The same for sub-intervals j0 .. j0 + T - 1 (a.T counts the range), writing
// every RK4 stage input of sub-interval j0 + i to stages + i K 4 (3N^2 + 2N + 1)
// (full layout, step i = K-1 .. 0 at slot i); the element itself is stored
// only when a.out.A is not null.
template <int N, int M>
__global__ void __launch_bounds__(128) build_stages_kernel(BuildArgs a, int64_t j0, double* stages) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.T || uniform_near(a.cf.uni, a.t, j0 + i, a.K)) return;
  constexpr int FS = 3 * N * N + 2 * N + 1;
  Elem<N> y;
  build_one<N, M, true>(a.cf, a.t, j0 + i, a.K, y, stages + i * (int64_t)a.K * 4 * FS);
  if (a.out.A) store_public<N>(a.out, j0 + i, y);
}

// Terminal element a_T: A = b = C = 0, J = Hf^T Xf Hf, eta = Hf^T Xf rf,
// zeta = 1/2 rf^T Xf rf.
struct TermArgs {
  int32_t n, nr;
  const double *Hf, *Xf, *rf;
  double *A, *b, *C, *eta, *J, *zeta;  // the terminal record (any of A, b, C, zeta may be null)
};

// One CTA: X_H = Xf Hf and Xf rf into shared memory, then J = sym(Hf' X_H), eta
// = Hf' Xf rf, zeta (a thread per entry doing both sums was 0.97 ms at n = 64).
__global__ void __launch_bounds__(256) terminal_kernel(TermArgs a) {
  extern __shared__ double tsm[];
  const int n = a.n, nr = a.nr, tid = threadIdx.x;
  double* XH = tsm;              // nr x n
  double* xr = XH + nr * n;      // nr
  for (int e = tid; e < nr * n; e += 256) {
    const int k = e / n, j = e % n;
    double s = 0.0;
    if (a.Hf) {
      for (int l = 0; l < nr; ++l) s = fma(a.Xf[k * nr + l], a.Hf[l * n + j], s);
    } else {
      s = a.Xf[k * nr + j];
    }
    XH[e] = s;
  }
  for (int k = tid; k < nr; k += 256) {
    double s = 0.0;
    if (a.rf)
      for (int l = 0; l < nr; ++l) s = fma(a.Xf[k * nr + l], a.rf[l], s);
    xr[k] = s;
  }
  __syncthreads();
  for (int e = tid; e < n * n; e += 256) {
    const int i = e / n, j = e % n;
    double vij = 0.0, vji = 0.0;
    if (a.Hf) {
      for (int k = 0; k < nr; ++k) {
        vij = fma(a.Hf[k * n + i], XH[k * n + j], vij);
        vji = fma(a.Hf[k * n + j], XH[k * n + i], vji);
      }
    } else {
      vij = XH[i * n + j];
      vji = XH[j * n + i];
    }
    a.J[e] = 0.5 * (vij + vji);
    if (a.A) a.A[e] = 0.0;
    if (a.C) a.C[e] = 0.0;
  }
  for (int i = tid; i < n; i += 256) {
    if (a.b) a.b[i] = 0.0;
    double et = 0.0;
    if (a.Hf) {
      for (int k = 0; k < nr; ++k) et = fma(a.Hf[k * n + i], xr[k], et);
    } else {
      et = xr[i];
    }
    a.eta[i] = et;
  }
  if (tid == 0 && a.zeta) {
    double rho = 0.0;
    if (a.rf)
      for (int k = 0; k < nr; ++k) rho = fma(a.rf[k], xr[k], rho);
    *a.zeta = 0.5 * rho;
  }
}

static void launch_terminal(const TermArgs& t, cudaStream_t st) {
  // nr <= 64, n <= 64: at most 33 KB
  terminal_kernel<<<1, 256, ((size_t)t.nr * t.n + t.nr) * sizeof(double), st>>>(t);
  count_launch();
}

cudaError_t launch_terminal_values(const lqt_problem& p, double* J, double* eta, double* zeta, cudaStream_t st) {
  TermArgs t{p.n, p.nr, p.Hf, p.Xf, p.rf, nullptr, nullptr, nullptr, eta, J, zeta};
  launch_terminal(t, st);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// batches: coefficient preparation and element build over the concatenation
// ---------------------------------------------------------------------------

// Lt and Ku of every problem (constant L, U), one CTA each.
__global__ void __launch_bounds__(128) batch_prepare_kernel(BatchDev bd) {
  __shared__ double R[kMaxM * kMaxM];
  const BatchProb& P = bd.probs[blockIdx.x];
  prepare_sample_cta(bd.n, bd.m, bd.M, P.L, P.U, const_cast<double*>(P.cf.Lt.ptr), const_cast<double*>(P.cf.Ku), R);
}

// q = X r, rho = r'Xr of every qr sample (X constant, H = identity).
__global__ void batch_qr_kernel(BatchDev bd) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int n = bd.n;
  if (g >= bd.total_qr) return;
  const int32_t b = batch_find(bd.off_qr, bd.B, g);
  const BatchProb& P = bd.probs[b];
  const int64_t s = g - bd.off_qr[b];
  const double* r = P.r ? P.r + (P.r_mode == kConst ? 0 : s) * n : nullptr;
  double* out = const_cast<double*>(P.cf.qr.ptr) + s * (n + 1);
  double rho = 0.0;
  for (int i = 0; i < n; ++i) {
    double v = 0.0;
    if (r)
      for (int l = 0; l < n; ++l) v = fma(P.X[i * n + l], r[l], v);
    out[i] = v;
    if (r) rho = fma(r[i], v, rho);
  }
  out[n] = rho;
}

cudaError_t batch_prepare(const BatchDev& bd, cudaStream_t st) {
  batch_prepare_kernel<<<(unsigned)bd.B, 128, 0, st>>>(bd);
  count_launch();
  batch_qr_kernel<<<(unsigned)((bd.total_qr + 127) / 128), 128, 0, st>>>(bd);
  count_launch();
  return cudaGetLastError();
}

// One thread per boundary of the concatenation: element j of problem b, or its
// terminal element (j = T_b; Hf = identity: J = Xf, eta = Xf rf,
// zeta = rf'Xf rf / 2).
template <int N, int M>
__global__ void __launch_bounds__(128) batch_build_kernel(BatchDev bd, ElemPtrs out) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= bd.total) return;
  const int32_t b = batch_find(bd.off, bd.B, g);
  const BatchProb& P = bd.probs[b];
  const int64_t j = g - P.off;
  Elem<N> y;
  if (j < P.T) {
    if (uniform_near(P.cf.uni, P.t, j, bd.K)) return;
    build_one<N, M>(P.cf, P.t, j, bd.K, y);
  } else {
#pragma unroll
    for (int i = 0; i < N * N; ++i) y.A[i] = 0.0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      y.b[i] = 0.0;
      double e = 0.0;
      if (P.rf)
        for (int l = 0; l < N; ++l) e = fma(P.Xf[i * N + l], P.rf[l], e);
      y.eta[i] = e;
    }
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
      for (int c = i; c < N; ++c) {
        y.C[sidx<N>(i, c)] = 0.0;
        y.J[sidx<N>(i, c)] = 0.5 * (P.Xf[i * N + c] + P.Xf[c * N + i]);
      }
    double z = 0.0;
    if (P.rf)
      for (int i = 0; i < N; ++i) z = fma(P.rf[i], y.eta[i], z);
    y.zeta = 0.5 * z;
  }
  store_public<N>(out, g, y);
}

template <int N, int M>
static void launch_batch_build_nm(const BatchDev& bd, const ElemPtrs& el, cudaStream_t st) {
  batch_build_kernel<N, M><<<(unsigned)((bd.total + 127) / 128), 128, 0, st>>>(bd, el);
  count_launch();
}

cudaError_t batch_build(const BatchDev& bd, const ElemPtrs& el, char* team_scratch, cudaStream_t st) {
  switch (bd.n) {
    case 1: launch_batch_build_nm<1, 1>(bd, el, st); break;
    case 2:
      if (bd.M == 1) launch_batch_build_nm<2, 1>(bd, el, st);
      else launch_batch_build_nm<2, 2>(bd, el, st);
      break;
    case 3:
      if (bd.M == 1) launch_batch_build_nm<3, 1>(bd, el, st);
      else if (bd.M == 2) launch_batch_build_nm<3, 2>(bd, el, st);
      else launch_batch_build_nm<3, 4>(bd, el, st);
      break;
    case 4:
      if (bd.M == 1) launch_batch_build_nm<4, 1>(bd, el, st);
      else if (bd.M == 2) launch_batch_build_nm<4, 2>(bd, el, st);
      else launch_batch_build_nm<4, 4>(bd, el, st);
      break;
    case 8:
      if (bd.M == 1) launch_batch_build_nm<8, 1>(bd, el, st);
      else if (bd.M == 2) launch_batch_build_nm<8, 2>(bd, el, st);
      else if (bd.M == 4) launch_batch_build_nm<8, 4>(bd, el, st);
      else launch_batch_build_nm<8, 8>(bd, el, st);
      break;
    case 16:
    case 64: return batch_build_team(bd, el, (double*)team_scratch, st);
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// Two warps per 32 sub-intervals up to this T for n = 2..4, one thread each
// beyond, where the sub-partitions have several warps either way.  Whole element
// builds on an uneven grid, one thread -> two warps: n = 4, m = 2, K = 10: 681
// -> 521 us at T = 10007, 2385 -> 2089 at 60000, 6451 -> 6089 at 200000, 15154
// -> 15362 at 500000; n = 3, m = 2, K = 4: 187 -> 122 at 2048, 576 -> 518 at
// 60000; n = 2, m = 1, K = 10: 167 -> 125 at 2048, 519 -> 502 at 60000, 1331 ->
// 1344 at 200000.  n = 1 has too little to share (60 -> 64 at 10007).
// The windows of a host call (equal runs of a long horizon, one after the other
// behind their copies) stay with one thread: n = 4, T = 2^17, K = 4 took 2890 us
// with pairs, 2855 without.
constexpr int64_t kPairMaxT = 1 << 17;

template <int N, int M>
static void launch_build_nm(const BuildArgs& a, cudaStream_t st, double* stages, int64_t j0, bool window) {
  const int threads = 128;
  const int64_t blocks = (a.T + threads - 1) / threads;
  count_launch();
  if (stages) {
    build_stages_kernel<N, M><<<(unsigned)blocks, threads, 0, st>>>(a, j0, stages);
    return;
  }
  if constexpr (N >= 2 && N <= 4) {
    if (a.T <= kPairMaxT && !window) {
      build_pair_kernel<N, M><<<(unsigned)((a.T + 31) / 32), 64, 0, st>>>(a);
      return;
    }
  }
  build_kernel<N, M><<<(unsigned)blocks, threads, 0, st>>>(a);
}

template <int N>
static cudaError_t launch_build_n(const BuildArgs& a, int M, cudaStream_t st, double* stages = nullptr,
                                  int64_t j0 = 0, bool window = false) {
  switch (M) {
    case 1: launch_build_nm<N, 1>(a, st, stages, j0, window); break;
    case 2: if constexpr (N >= 2) { launch_build_nm<N, 2>(a, st, stages, j0, window); break; } else return cudaErrorInvalidValue;
    case 4: if constexpr (N >= 3) { launch_build_nm<N, 4>(a, st, stages, j0, window); break; } else return cudaErrorInvalidValue;
    case 8: if constexpr (N >= 8) { launch_build_nm<N, 8>(a, st, stages, j0, window); break; } else return cudaErrorInvalidValue;
    default: return cudaErrorInvalidValue;
  }
  return cudaSuccess;
}

// The RK4 stage inputs of sub-intervals j0 .. j0 + cnt - 1 of p (n <= 8), the
// stages of sub-interval j0 + i at stages + i K 4 (3n^2 + 2n + 1) (full
// layout); the elements themselves go to `out` when out.A is not null.
cudaError_t launch_build_stages_range(const lqt_problem& p, const Layout& lay, const Coefs& cf, int64_t j0,
                                      int64_t cnt, double* stages, cudaStream_t st, const ElemPtrs& out) {
  BuildArgs a{};
  a.T = cnt; a.K = p.K; a.t = p.t; a.cf = cf; a.out = out;
  if (team_build_preferred(p.n, cnt)) return team_launch_build_small(p, lay, cf, j0, cnt, stages, out, st);
  switch (p.n) {
    case 1: return launch_build_n<1>(a, lay.M, st, stages, j0);
    case 2: return launch_build_n<2>(a, lay.M, st, stages, j0);
    case 3: return launch_build_n<3>(a, lay.M, st, stages, j0);
    case 4: return launch_build_n<4>(a, lay.M, st, stages, j0);
    case 8: return launch_build_n<8>(a, lay.M, st, stages, j0);
    default: return cudaErrorInvalidValue;
  }
}

// Elements 0..T-1 of p alone (no terminal element), n <= 8; cf.uni, when set,
// holds a finished table.
cudaError_t launch_build_range(const lqt_problem& p, const Layout& lay, const Coefs& cf, const ElemPtrs& out,
                               cudaStream_t st) {
  BuildArgs a;
  a.T = p.T; a.K = p.K; a.t = p.t; a.cf = cf; a.out = out;
  if (cf.uni) {
    const cudaError_t e = launch_uniform_expand(p, cf, out, st);
    if (e != cudaSuccess) return e;
  }
  switch (p.n) {
    case 1: return launch_build_n<1>(a, lay.M, st, nullptr, 0, true);
    case 2: return launch_build_n<2>(a, lay.M, st, nullptr, 0, true);
    case 3: return launch_build_n<3>(a, lay.M, st, nullptr, 0, true);
    case 4: return launch_build_n<4>(a, lay.M, st, nullptr, 0, true);
    case 8: return launch_build_n<8>(a, lay.M, st, nullptr, 0, true);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_build(const lqt_problem& p, const Layout& lay, const Coefs& cf_in, const ElemPtrs& out,
                         cudaStream_t st, double* team_scratch) {
  Coefs cf = cf_in;
  // the mixed-precision path's FP32 products amplify a last-bit change of an
  // element to their own rounding: its elements stay as the general build
  // makes them
  if (mixed_precision()) cf.uni = nullptr;
  BuildArgs a;
  a.T = p.T; a.K = p.K; a.t = p.t; a.cf = cf; a.out = out;
  cudaError_t e;
  if (cf.uni) {
    e = launch_uniform_master(p, cf, st);
    if (e == cudaSuccess) e = launch_uniform_expand(p, cf, out, st);
    if (e != cudaSuccess) return e;
  }
  if (team_build_preferred(p.n, p.T)) {
    e = team_launch_build_small(p, lay, cf, 0, p.T, nullptr, out, st);
    if (e != cudaSuccess) return e;
    return launch_terminal_element(p, out, st);
  }
  switch (p.n) {
    case 1: e = launch_build_n<1>(a, lay.M, st); break;
    case 2: e = launch_build_n<2>(a, lay.M, st); break;
    case 3: e = launch_build_n<3>(a, lay.M, st); break;
    case 4: e = launch_build_n<4>(a, lay.M, st); break;
    case 8: e = launch_build_n<8>(a, lay.M, st); break;
    case 16:
    case 64: e = team_launch_build(p, lay, cf, out, team_scratch, st); break;
    default: return cudaErrorInvalidValue;
  }
  if (e != cudaSuccess) return e;
  return launch_terminal_element(p, out, st);
}

// Terminal element a_T into index T of the public arrays.
cudaError_t launch_terminal_element(const lqt_problem& p, const ElemPtrs& out, cudaStream_t st) {
  const int64_t T = p.T;
  const int n = p.n;
  TermArgs t{p.n, p.nr, p.Hf, p.Xf, p.rf, out.A + T * n * n, out.b + T * n, out.C + T * n * n,
             out.eta + T * n, out.J + T * n * n, out.zeta ? out.zeta + T : nullptr};
  launch_terminal(t, st);
  return cudaGetLastError();
}

}  // namespace lqt
