// Element build for constant F, L, U, X (and H) without drift, r constant or
// one sample per sub-interval, on a (nearly) uniform grid.
//
// The K RK4 steps of Theorem Backward_HJB_LQT (Sec. IV-B) then depend on the
// sub-interval only through its step h_j and its q_j = H'Xr_j: A, C, J are
// functions of h alone, eta and b are linear in q and zeta is quadratic,
//     eta_j = E(h_j) q_j,  b_j = Bq(h_j) q_j,
//     zeta_j = h_j K rho_j / 2 + q_j' Z(h_j) q_j / 2,
// and RK4 commutes with these linear maps.  So one element with the matrices
// (A, C, J, E, Bq, Z) in the place of (A, b, C, eta, J, zeta) serves every
// sub-interval: dE = -I - F'E + P W, dBq = -AL W, dZ = W'W with W = Lt'E (the
// eta, b and zeta equations with q = the unit vectors).  The steps of a grid
// built in floating point differ by rounding (|h_j - h| / h ~ 1e-12 at t_j / h
// = 1e4), which the results feel to first order, so the element is integrated
// at three steps, h and h (1 +- 1e-4), and sub-interval j takes
//     E_j = E(h) + c_j (E(h+) - E(h-)),   c_j = (h_j - h) / (h+ - h-).
// A sub-interval within 1e-9 of h is served this way: the terms dropped are
// below 1e-17 relative.  Any other sub-interval is left to the general build
// kernels, which skip the ones served here (uniform_near), so a grid may be
// partly uniform.
//
// What bounds it: the general build is bound by the FP64 pipe (K (40 n^3 +
// 60 n^2) flop per sub-interval); here a sub-interval costs 18 n^2 FP64
// operations and the store of its element.  One CTA per step value holds the
// integrated element in shared memory (n <= 16); at n = 64, where one
// element's integration is 70 Mflop, a cluster of eight CTAs shares it through
// its workspace (L2) with a cluster barrier between the phases of a stage.
// Measured, whole solves before and after: n = 16, m = 8, K = 4, T = 8192:
// 8.10 -> 3.99 ms; n = 64, m = 16, K = 2, T = 4096: 109.1 -> 59.4 ms; a batch of
// 256 problems, n in {2, 4, 8, 16}, T up to 8192: 220 -> 60.7 ms.  Errors against
// 64-bit references are the general build's (n = 64: 4.5e-14 both).
#include <cuda_runtime.h>

#include "lqt_device.cuh"
#include "lqt_internal.h"
#include "lqt_uniform.cuh"

namespace lqt {

static size_t ual(size_t x) { return (x + 255) & ~(size_t)255; }

// Doubles of integrator state per step value: y, its low part and the RK4 sum
// of the step (six n x n blocks each), two buffers of the stage input's (A, J,
// E), AL, P, W.
__host__ __device__ __forceinline__ int64_t uni_work_doubles(int n, int M) {
  return 24 * (int64_t)n * n + 3 * (int64_t)n * M;
}

int64_t uniform_table_doubles(int n, int M) {
  return kUniHeader + 24 * (int64_t)n * n + (n > 16 ? 3 * uni_work_doubles(n, M) : 0);
}

size_t uniform_table_bytes(int n, int M) { return ual((size_t)uniform_table_doubles(n, M) * sizeof(double)); }

// Shortest horizon for which the three integrations (one element's latency,
// spread over a CTA) cost less than the general build of all sub-intervals.
static int64_t uniform_min_T(int n) { return n <= 3 ? 32768 : n == 4 ? 8192 : n == 8 ? 1024 : n == 16 ? 512 : 128; }

bool uniform_eligible(const lqt_problem& p) {
  const bool cst = p.F.mode == LQT_CONST && p.L.mode == LQT_CONST && p.U.mode == LQT_CONST &&
                   p.X.mode == LQT_CONST && (!p.H.ptr || p.H.mode == LQT_CONST);
  return cst && !p.c.ptr && (!p.r.ptr || p.r.mode != LQT_PER_STAGE) && p.T >= uniform_min_T(p.n);
}

struct UniArgs {
  int32_t n, M, K, B;
  int64_t T;               // single problem
  const double* t;
  Coefs cf;                // single problem; cf.uni = its table
  const BatchProb* probs;  // batches (null: the single problem)
  int32_t cluster;         // CTAs per step value
};

__device__ __forceinline__ void uni_sync(int cluster) {
  if (cluster > 1) {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  } else {
    __syncthreads();
  }
}

// Entry (i, j), i <= j, of the e-th position of an n x n upper triangle.
__device__ __forceinline__ void tri_index(int e, int n, int& i, int& j) {
  i = 0;
  int row = n;
  while (e >= row) {
    e -= row;
    --row;
    ++i;
  }
  j = i + e;
}

// (y, lo) += p + e exactly rounded to the pair (Knuth's two-sum): the element
// serves every sub-interval, so a rounding of its RK4 sums would be the same
// error in all of them and add up over the horizon, where the general build's
// roundings differ from one sub-interval to the next.
__device__ __forceinline__ void pair_add(double& y, double& lo, double p, double e) {
  const double t = __dadd_rn(y, p), b = __dsub_rn(t, y);
  const double err = __dadd_rn(__dsub_rn(y, __dsub_rn(t, b)), __dsub_rn(p, b));
  const double l = __dadd_rn(lo, __dadd_rn(err, e));
  y = __dadd_rn(t, l);
  lo = __dsub_rn(l, __dsub_rn(y, t));
}

// One step value's integration: 256 threads of each CTA of the cluster own
// entries of the six blocks (upper triangles of C, J, Z); two barriers per RK4
// stage, before and after the entries that need AL, P, W of the stage input.
template <bool kShared>
__global__ void __launch_bounds__(256) uniform_master_kernel(UniArgs a) {
  extern __shared__ double sm[];
  __shared__ int good;
  const int n = a.n, M = a.M, K = a.K, nn = n * n, nM = n * M;
  const int cl = a.cluster;
  const int rank = (int)(blockIdx.x % cl);
  const int var = (int)((blockIdx.x / cl) % 3);
  const int64_t pb = blockIdx.x / (3 * (int64_t)cl);
  const Coefs cf = a.probs ? a.probs[pb].cf : a.cf;
  const double* t = a.probs ? a.probs[pb].t : a.t;
  const int64_t T = a.probs ? a.probs[pb].T : a.T;
  double* tab = const_cast<double*>(cf.uni);
  if (tab == nullptr) return;  // the same for every CTA of the cluster
  const int tid = rank * 256 + (int)threadIdx.x, nth = cl * 256;
  // the mean step; not worth the integration when fewer than half of (up to)
  // 4096 sampled sub-intervals have it
  const double h0 = (t[T] - t[0]) / ((double)T * K);
  if (threadIdx.x == 0) good = 0;
  __syncthreads();
  const int64_t cnt = T < 4096 ? T : 4096;
  int mine = 0;
  for (int64_t s = threadIdx.x; s < cnt; s += 256) mine += uniform_near_h(h0, t, s * T / cnt, K) ? 1 : 0;
  atomicAdd(&good, mine);
  __syncthreads();
  const bool valid = h0 > 0.0 && isfinite(h0) && 2 * (int64_t)good >= cnt;
  if (tid == 0 && var == 0) {
    tab[0] = valid ? 1.0 : 0.0;
    tab[1] = h0;
    tab[2] = 1.0 / (h0 * (1.0 + kUniStep) - h0 * (1.0 - kUniStep));
  }
  if (!valid) return;
  const double h = var == 0 ? h0 : var == 1 ? h0 * (1.0 + kUniStep) : h0 * (1.0 - kUniStep);
  // F and Lt in shared memory; the state there too, or in the table's work area
  double* Fs = sm;
  double* Ls = Fs + nn;
  double* y = kShared ? Ls + nM : tab + kUniHeader + 24 * (int64_t)nn + var * uni_work_doubles(n, M);
  double* lo = y + 6 * nn;
  double* sum = lo + 6 * nn;
  double* stg = sum + 6 * nn;  // two buffers of (A, J, E)
  double* AL = stg + 6 * nn;
  double* P = AL + nM;
  double* W = P + nM;
  for (int e = threadIdx.x; e < nn; e += 256) Fs[e] = cf.F.ptr[e];
  for (int e = threadIdx.x; e < nM; e += 256) Ls[e] = cf.Lt.ptr[e];
  for (int e = tid; e < 6 * nn; e += nth) {
    const double v = (e < nn && e % (n + 1) == 0) ? 1.0 : 0.0;
    y[e] = v;
    lo[e] = 0.0;
    if (e < 3 * nn) stg[e] = e < nn ? v : 0.0;
  }
  uni_sync(cl);
  const int tri = n * (n + 1) / 2;
  const int work = 3 * nn + 3 * tri;
  // h / 6 to twice the precision
  const double h6 = h / 6.0, h6l = fma(-6.0, h6, h) / 6.0;
  int cur = 0;
  for (int step = 0; step < 4 * K; ++step) {
    const int q = step & 3;
    const double* As = stg + cur * 3 * nn;
    const double* Js = As + nn;
    const double* Es = Js + nn;
    double* An = stg + (cur ^ 1) * 3 * nn;
    for (int e = tid; e < 3 * nM; e += nth) {
      const int which = e / nM, r = e - which * nM;
      double s = 0.0;
      if (which < 2) {  // AL, P
        const double* X = (which == 0 ? As : Js) + (r / M) * n;
        const int c = r % M;
        for (int l = 0; l < n; ++l) s = fma(X[l], Ls[l * M + c], s);
      } else {  // W
        const int c = r / n, j = r % n;
        for (int l = 0; l < n; ++l) s = fma(Ls[l * M + c], Es[l * n + j], s);
      }
      AL[e] = s;  // AL, P, W are contiguous
    }
    uni_sync(cl);
    const double ak = -h * (q < 2 ? 0.5 : 1.0);
    for (int g = tid; g < work; g += nth) {
      int kind, i, j;
      if (g < 3 * nn) {  // A, E, Bq: full
        const int f = g / nn, e = g - f * nn;
        kind = f == 0 ? 0 : f == 1 ? 3 : 4;
        i = e / n;
        j = e - i * n;
      } else {  // J, C, Z: upper triangles
        const int f = (g - 3 * nn) / tri;
        kind = f == 0 ? 2 : f == 1 ? 1 : 5;
        tri_index(g - 3 * nn - f * tri, n, i, j);
      }
      double s = 0.0;
      if (kind == 0) {
        for (int c = 0; c < M; ++c) s = fma(AL[i * M + c], P[j * M + c], s);
        for (int l = 0; l < n; ++l) s = fma(-As[i * n + l], Fs[l * n + j], s);
      } else if (kind == 1) {
        for (int c = 0; c < M; ++c) s = fma(-AL[i * M + c], AL[j * M + c], s);
      } else if (kind == 2) {
        double u = 0.0, v = 0.0;
        for (int l = 0; l < n; ++l) {
          u = fma(Js[i * n + l], Fs[l * n + j], u);
          v = fma(Js[l * n + j], Fs[l * n + i], v);
        }
        s = -cf.Q.ptr[i * n + j] - u - v;
        for (int c = 0; c < M; ++c) s = fma(P[i * M + c], P[j * M + c], s);
      } else if (kind == 3) {
        s = i == j ? -1.0 : 0.0;
        for (int l = 0; l < n; ++l) s = fma(-Fs[l * n + i], Es[l * n + j], s);
        for (int c = 0; c < M; ++c) s = fma(P[i * M + c], W[c * n + j], s);
      } else if (kind == 4) {
        for (int c = 0; c < M; ++c) s = fma(-AL[i * M + c], W[c * n + j], s);
      } else {
        for (int c = 0; c < M; ++c) s = fma(W[c * n + i], W[c * n + j], s);
      }
      const int e = kind * nn + i * n + j, et = kind * nn + j * n + i;
      const bool mirror = kind == 1 || kind == 2 || kind == 5;
      double nx;
      if (q == 3) {
        const double k = -(sum[e] + s), p = h6 * k;
        double ye = y[e], le = lo[e];
        pair_add(ye, le, p, fma(h6, k, -p) + h6l * k);
        nx = ye;
        y[e] = ye;
        lo[e] = le;
        if (mirror) {
          y[et] = ye;
          lo[et] = le;
        }
      } else {
        sum[e] = q == 0 ? s : fma(2.0, s, sum[e]);
        nx = fma(ak, s, y[e]);
      }
      // the next stage input's A, J, E
      if (kind == 0 || kind == 3) An[(kind == 0 ? 0 : 2 * nn) + i * n + j] = nx;
      if (kind == 2) {
        An[nn + i * n + j] = nx;
        An[nn + j * n + i] = nx;
      }
    }
    uni_sync(cl);
    cur ^= 1;
  }
  // A, C, J as they are, E and Bq transposed (the expansion's lanes run over
  // their rows), Z
  double* out = tab + kUniHeader + var * 6 * nn;
  for (int e = tid; e < 6 * nn; e += nth) {
    const int blk = e / nn, r = e - blk * nn, i = r / n, j = r - i * n;
    const int o = (blk == 3 || blk == 4) ? blk * nn + j * n + i : e;
    out[e] = y[o];
    if (var == 0) out[18 * nn + e] = lo[o];
  }
}

struct UniExpandArgs {
  int32_t K;
  int64_t T;
  const double* t;
  Coefs cf;
  ElemPtrs out;
  // batches: the chunks of problem b are CTAs off_chunk[b] .. off_chunk[b + 1] - 1
  const BatchProb* probs;
  const int64_t* off_chunk;
  int32_t B;
};

// Sub-intervals per CTA of the expansion.
__host__ __device__ constexpr int uni_chunk(int n) { return n <= 8 ? 64 : 16; }
int64_t uniform_chunks(int n, int64_t T) { return (T + uni_chunk(n) - 1) / uni_chunk(n); }

// The elements of one chunk of sub-intervals from the table: a thread holds
// the entries e of A, C, J (value and slope) in registers and writes them for
// every sub-interval of the chunk (consecutive lanes, consecutive addresses);
// for eta, b and the rows of Z q a thread owns row i of one or more
// sub-intervals.  Bound by its 18 n^2 FP64 operations per sub-interval (FP64 pipe
// 81% busy at n = 16, T = 4104), which at 64 cycles a warp instruction take longer
// than the store of 3 n^2 + 2 n + 1 doubles at every n.
// Batches: one CTA per chunk of a problem that has a table, found by the chunks'
// prefix sum.  (A grid of the longest problem's chunks times B was 16.8 million
// CTAs for one problem of T = 2^19 beside 2047 of T = 64, n = 4: 47.5 ms for the
// batch, now 16.0; from 2^31 CTAs on it could not be launched.)
template <int N>
__global__ void __launch_bounds__(256) uniform_expand_kernel(UniExpandArgs a) {
  constexpr int CH = uni_chunk(N), NN = N * N;
  __shared__ double cj[CH], hk[CH], qs[CH * (N + 1)], zp[CH * N];
  __shared__ int near[CH];
  const int32_t pb = a.probs ? batch_find(a.off_chunk, a.B, blockIdx.x) : 0;
  const int64_t j0 = (blockIdx.x - (a.probs ? a.off_chunk[pb] : 0)) * CH;
  const Coefs& cf = a.probs ? a.probs[pb].cf : a.cf;
  const double* t = a.probs ? a.probs[pb].t : a.t;
  const int64_t T = a.probs ? a.probs[pb].T : a.T;
  const int64_t off = a.probs ? a.probs[pb].off : 0;
  const double* tab = cf.uni;
  if (tab == nullptr || tab[0] == 0.0 || j0 >= T) return;
  const int cnt = T - j0 < CH ? (int)(T - j0) : CH;
  const int tid = threadIdx.x;
  const double h0 = tab[1];
  for (int k = tid; k < CH; k += 256) {
    const bool nr = k < cnt && uniform_near_h(h0, t, j0 + k, a.K);
    near[k] = nr;
    const double h = nr ? uniform_step(t, j0 + k, a.K) : h0;
    cj[k] = (h - h0) * tab[2];
    hk[k] = h * a.K;
  }
  for (int e = tid; e < CH * (N + 1); e += 256) {
    const int k = e / (N + 1);
    qs[e] = k < cnt ? cf.qr.ptr[sample_index(cf.qr.mode, j0 + k, 0, a.K) * (N + 1) + (e - k * (N + 1))] : 0.0;
  }
  __syncthreads();
  const double* T0 = tab + kUniHeader;
  const double* Tp = T0 + 6 * NN;
  const double* Tm = Tp + 6 * NN;
  const double* Tl = Tm + 6 * NN;  // low part of T0
  {
    constexpr int GR = NN >= 256 ? 1 : 256 / NN;  // threads that share an entry
    const int g = NN >= 256 ? 0 : tid / NN;
    double* dst[3] = {a.out.A, a.out.C, a.out.J};
#pragma unroll
    for (int blk = 0; blk < 3; ++blk)
      for (int e = NN >= 256 ? tid : tid - g * NN; e < NN && g < GR; e += NN >= 256 ? 256 : NN) {
        const double v = T0[blk * NN + e], d = Tp[blk * NN + e] - Tm[blk * NN + e], l = Tl[blk * NN + e];
        double* o = dst[blk] + (off + j0) * NN + e;
        for (int k = g; k < cnt; k += GR)
          if (near[k]) o[(int64_t)k * NN] = v + fma(cj[k], d, l);
      }
  }
  {
    constexpr int GR = 256 / N;
    constexpr int R = (CH + GR - 1) / GR;
    const int g = tid / N, i = tid - g * N;
    if (g < GR) {
      double e[R], b[R], z[R];
#pragma unroll
      for (int r = 0; r < R; ++r) e[r] = b[r] = z[r] = 0.0;
      for (int c = 0; c < N; ++c) {
        const int o = c * N + i;
        const double e0 = T0[3 * NN + o], de = Tp[3 * NN + o] - Tm[3 * NN + o], el = Tl[3 * NN + o];
        const double b0 = T0[4 * NN + o], db = Tp[4 * NN + o] - Tm[4 * NN + o], bl = Tl[4 * NN + o];
        const double z0 = T0[5 * NN + o], dz = Tp[5 * NN + o] - Tm[5 * NN + o], zl = Tl[5 * NN + o];
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int k = g + r * GR;
          if (k < CH) {
            const double qc = qs[k * (N + 1) + c], w = cj[k];
            e[r] = fma(e0 + fma(w, de, el), qc, e[r]);
            b[r] = fma(b0 + fma(w, db, bl), qc, b[r]);
            z[r] = fma(z0 + fma(w, dz, zl), qc, z[r]);
          }
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int k = g + r * GR;
        if (k < CH) {
          zp[k * N + i] = z[r] * qs[k * (N + 1) + i];
          if (k < cnt && near[k]) {
            a.out.eta[(off + j0 + k) * N + i] = e[r];
            a.out.b[(off + j0 + k) * N + i] = b[r];
          }
        }
      }
    }
  }
  __syncthreads();
  if (a.out.zeta)
    for (int k = tid; k < cnt; k += 256)
      if (near[k]) {
        double s = hk[k] * qs[k * (N + 1) + N];
        for (int i = 0; i < N; ++i) s += zp[k * N + i];
        a.out.zeta[off + j0 + k] = 0.5 * s;
      }
}

static cudaError_t launch_master(const UniArgs& a, int64_t problems, cudaStream_t st) {
  const int n = a.n;
  const size_t base = ((size_t)n * n + (size_t)n * a.M) * sizeof(double);
  if (n <= 16) {
    const size_t smem = base + (size_t)uni_work_doubles(n, a.M) * sizeof(double);
    cudaError_t e = cudaFuncSetAttribute(uniform_master_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         96 * 1024);
    if (e != cudaSuccess) return e;
    UniArgs b = a;
    b.cluster = 1;
    uniform_master_kernel<true><<<(unsigned)(3 * problems), 256, smem, st>>>(b);
  } else {
    UniArgs b = a;
    b.cluster = 8;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(3 * 8 * problems));
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = base;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 8;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, uniform_master_kernel<false>, b);
    if (e != cudaSuccess) return e;
  }
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_uniform_master(const lqt_problem& p, const Coefs& cf, cudaStream_t st) {
  UniArgs a{};
  a.n = p.n; a.M = cf.M; a.K = p.K; a.B = 1; a.T = p.T; a.t = p.t; a.cf = cf;
  return launch_master(a, 1, st);
}

static cudaError_t launch_expand(int n, const UniExpandArgs& b, int64_t chunks, cudaStream_t st) {
  const unsigned grid = (unsigned)chunks;
  switch (n) {
    case 1: uniform_expand_kernel<1><<<grid, 256, 0, st>>>(b); break;
    case 2: uniform_expand_kernel<2><<<grid, 256, 0, st>>>(b); break;
    case 3: uniform_expand_kernel<3><<<grid, 256, 0, st>>>(b); break;
    case 4: uniform_expand_kernel<4><<<grid, 256, 0, st>>>(b); break;
    case 8: uniform_expand_kernel<8><<<grid, 256, 0, st>>>(b); break;
    case 16: uniform_expand_kernel<16><<<grid, 256, 0, st>>>(b); break;
    case 64: uniform_expand_kernel<64><<<grid, 256, 0, st>>>(b); break;
    default: return cudaErrorInvalidValue;
  }
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_uniform_expand(const lqt_problem& p, const Coefs& cf, const ElemPtrs& out, cudaStream_t st) {
  UniExpandArgs a{};
  a.K = p.K; a.T = p.T; a.t = p.t; a.cf = cf; a.out = out;
  return launch_expand(p.n, a, uniform_chunks(p.n, p.T), st);
}

cudaError_t batch_uniform(const BatchDev& bd, const ElemPtrs& out, cudaStream_t st) {
  UniArgs a{};
  a.n = bd.n; a.M = bd.M; a.K = bd.K; a.B = bd.B; a.probs = bd.probs;
  const cudaError_t e = launch_master(a, bd.B, st);
  if (e != cudaSuccess) return e;
  UniExpandArgs x{};
  x.K = bd.K; x.out = out; x.probs = bd.probs; x.off_chunk = bd.off_chunk; x.B = bd.B;
  return launch_expand(bd.n, x, bd.total_chunks, st);
}

}  // namespace lqt
