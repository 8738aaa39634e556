// Reverse mode of the constant-coefficient build (lqt_uniform.cu): the element
// adjoints of the sub-intervals that one integrated element serves, n <= 8, H =
// Hf = I, no drift.
//
// With element j = (A(h_j), Bq(h_j) q_j, C(h_j), E(h_j) q_j, J(h_j), h_j K rho_j
// / 2 + q_j' Z(h_j) q_j / 2), the adjoint of the shared (A, Bq, C, E, J, Z) is
// the sum over j of
//     (Abar_j, bbar_j q_j', Cbar_j, etabar_j q_j', Jbar_j, zetabar_j q_j q_j' / 2),
// and the RK4 reverse sweep (step 5 of lqt_adjoint.cu) is linear in it, so it
// runs once on the sum instead of once per sub-interval.  h_j enters as in the
// forward build: E_j = E(h) + c_j (E(h+) - E(h-)) gives the sums weighted by c_j
// to the sweeps at h+ and h- (with opposite signs).  Per sub-interval remain
// q_j's and r_j's adjoints, three matrix-vector products.
//
// Measured at n = 8, m = 4, T = 2^14: 4.96 ms for a reverse sweep and 1.65 ms
// for the recorded RK4 stages of every sub-interval, bound by the FP64 pipe,
// against the three sweeps here (one CTA each) and one pass over the element
// adjoints.
#include <cuda_runtime.h>

#include "lqt_device.cuh"
#include "lqt_internal.h"
#include "lqt_uniform.cuh"

namespace lqt {

constexpr int kChunk = 32;

// Sums over the served sub-intervals, one partial per CTA: [6 n^2 | 6 n^2
// (weighted by c_j) | n^2 (X)] in the order A, C, J, E, Bq, Z; rbar_j into pr
// (stage sample 0, zeros in the others), zeros into the sub-interval's rows of
// pF, pB, pX.
__global__ void __launch_bounds__(256) uniform_adjoint_sums_kernel(UniAdjArgs a) {
  const double* tab = a.cf.uni;
  const int n = a.n, nn = n * n, fs = 3 * nn + 2 * n + 1, tid = threadIdx.x;
  __shared__ double cj[kChunk], hk[kChunk], qs[kChunk * 9], rs[kChunk * 8], qb[kChunk * 8], rb[kChunk];
  __shared__ int near[kChunk];
  double acc0[2] = {0.0, 0.0}, acc1[2] = {0.0, 0.0};
  const bool valid = tab[0] != 0.0;
  const double* T0 = tab + kUniHeader;
  const double* Tp = T0 + 6 * nn;
  const double* Tm = Tp + 6 * nn;
  const double* Tl = Tm + 6 * nn;
  for (int64_t j0 = (int64_t)blockIdx.x * kChunk; valid && j0 < a.T; j0 += (int64_t)gridDim.x * kChunk) {
    const int cnt = a.T - j0 < kChunk ? (int)(a.T - j0) : kChunk;
    __syncthreads();
    for (int k = tid; k < kChunk; k += 256) {
      const bool nr = k < cnt && uniform_near_h(tab[1], a.t, j0 + k, a.K);
      near[k] = nr;
      const double h = nr ? uniform_step(a.t, j0 + k, a.K) : tab[1];
      cj[k] = (h - tab[1]) * tab[2];
      hk[k] = h * a.K;
    }
    for (int e = tid; e < cnt * (n + 1); e += 256) {
      const int k = e / (n + 1), c = e - k * (n + 1);
      qs[e] = a.cf.qr.ptr[sample_index(a.cf.qr.mode, j0 + k, 0, a.K) * (n + 1) + c];
    }
    for (int e = tid; e < cnt * n; e += 256) {
      const int k = e / n, c = e - k * n;
      rs[e] = a.r ? a.r[sample_index(a.r_mode, j0 + k, 0, a.K) * n + c] : 0.0;
    }
    __syncthreads();
    // qbar_c = sum_i E_ic etabar_i + Bq_ic bbar_i + zetabar Z_ci q_i
    for (int e = tid; e < cnt * n; e += 256) {
      const int k = e / n, c = e - k * n;
      const double* eb = a.ebar + (j0 + k) * fs;
      const double zb = eb[3 * nn + 2 * n];
      double s = 0.0;
      for (int i = 0; i < n; ++i) {
        const int o = c * n + i;  // E and Bq are stored transposed, Z is symmetric
        const double E = T0[3 * nn + o] + fma(cj[k], Tp[3 * nn + o] - Tm[3 * nn + o], Tl[3 * nn + o]);
        const double B = T0[4 * nn + o] + fma(cj[k], Tp[4 * nn + o] - Tm[4 * nn + o], Tl[4 * nn + o]);
        const double Z = T0[5 * nn + o] + fma(cj[k], Tp[5 * nn + o] - Tm[5 * nn + o], Tl[5 * nn + o]);
        s = fma(E, eb[2 * nn + n + i], s);
        s = fma(B, eb[nn + i], s);
        s = fma(zb * Z, qs[k * (n + 1) + i], s);
      }
      qb[e] = s;
      if (c == 0) rb[k] = 0.5 * zb * hk[k];
    }
    __syncthreads();
    // rbar = X' qbar + rhobar (X + X') r
    for (int e = tid; e < cnt * n; e += 256) {
      const int k = e / n, i = e - k * n;
      if (!near[k]) continue;
      double s = 0.0, u = 0.0;
      for (int l = 0; l < n; ++l) {
        s = fma(a.X[l * n + i], qb[k * n + l], s);
        u = fma(a.X[i * n + l] + a.X[l * n + i], rs[k * n + l], u);
      }
      double* pr = a.pr + (j0 + k) * (2 * a.K + 1) * n + i;
      pr[0] = fma(rb[k], u, s);
      for (int p = 1; p <= 2 * a.K; ++p) pr[p * n] = 0.0;
    }
    for (int e = tid; e < cnt * nn; e += 256)
      if (near[e / nn]) {
        a.pF[j0 * nn + e] = 0.0;
        a.pB[j0 * nn + e] = 0.0;
        a.pX[j0 * nn + e] = 0.0;
      }
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const int e = tid + 256 * s;
      if (e >= 7 * nn) continue;
      const int kind = e / nn, r = e - kind * nn, i = r / n, c = r - i * n;
      const int off = kind == 0 ? r : kind == 1 ? nn + n + r : kind == 2 ? 2 * nn + 2 * n + r
                      : kind == 3 ? 2 * nn + n + i : kind == 4 ? nn + i : 3 * nn + 2 * n;
      for (int k = 0; k < cnt; ++k) {
        if (!near[k]) continue;
        double v;
        if (kind == 6) {
          v = fma(qb[k * n + i], rs[k * n + c], rb[k] * rs[k * n + i] * rs[k * n + c]);
        } else {
          v = a.ebar[(j0 + k) * fs + off];
          if (kind == 3 || kind == 4) v *= qs[k * (n + 1) + c];
          if (kind == 5) v *= 0.5 * qs[k * (n + 1) + i] * qs[k * (n + 1) + c];
          acc1[s] = fma(cj[k], v, acc1[s]);
        }
        acc0[s] += v;
      }
    }
  }
  double* out = a.part + (int64_t)blockIdx.x * 13 * nn;
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int e = tid + 256 * s;
    if (e < 6 * nn) {
      out[e] = acc0[s];
      out[6 * nn + e] = acc1[s];
    } else if (e < 7 * nn) {
      out[6 * nn + e] = acc0[s];
    }
  }
}

// The reverse sweep of one step value (block 0: h, 1: h+, 2: h-), on the sums;
// writes Fbar, Bbar and Xbar as rows T + block of pF, pB, pX.
__global__ void __launch_bounds__(256) uniform_adjoint_sweep_kernel(UniAdjArgs a) {
  extern __shared__ double sm[];
  const int n = a.n, nn = n * n, M = a.cf.M, K = a.K, tid = threadIdx.x, v = blockIdx.x;
  const double* tab = a.cf.uni;
  double* oF = a.pF + (a.T + v) * nn;
  double* oB = a.pB + (a.T + v) * nn;
  double* oX = a.pX + (a.T + v) * nn;
  if (tab[0] == 0.0) {
    for (int e = tid; e < nn; e += 256) oF[e] = oB[e] = oX[e] = 0.0;
    return;
  }
  const double h0 = tab[1];
  const double h = v == 0 ? h0 : v == 1 ? h0 * (1.0 + kUniStep) : h0 * (1.0 - kUniStep);
  double* F = sm;
  double* B = F + nn;
  double* G = B + nn;        // B J
  double* H = G + nn;        // B E
  double* AA = H + nn;       // A' kA
  double* AB = AA + nn;      // A' kB
  double* CA = AB + nn;      // kC A
  double* Gb = CA + nn;
  double* Hb = Gb + nn;
  double* Fb = Hb + nn;
  double* Bb = Fb + nn;
  double* Qb = Bb + nn;
  double* yb = Qb + nn;      // adjoint of the step's output: A, C, J, E, Bq, Z
  double* kb = yb + 6 * nn;  // adjoint of one stage's rates
  double* ac = kb + 6 * nn;  // adjoint of one stage's input: A, J, E
  double* tot = ac + 3 * nn; // their sum over the step
  double* st = tot + 3 * nn; // stage inputs: [4 K][A, J, E]
  const double* Q = a.X;
  for (int e = tid; e < nn; e += 256) {
    const int i = e / n, j = e - i * n;
    double s = 0.0;
    for (int l = 0; l < M; ++l) s = fma(a.cf.Lt.ptr[i * M + l], a.cf.Lt.ptr[j * M + l], s);
    B[e] = s;
    F[e] = a.cf.F.ptr[e];
    Fb[e] = Bb[e] = Qb[e] = 0.0;
    st[e] = i == j ? 1.0 : 0.0;
    st[nn + e] = st[2 * nn + e] = 0.0;
  }
  // seeds: the CTAs' sums
  for (int e = tid; e < 6 * nn; e += 256) {
    double s = 0.0;
    for (int b = 0; b < a.parts; ++b) s += a.part[(int64_t)b * 13 * nn + (v ? 6 * nn : 0) + e];
    yb[e] = v == 2 ? -s : s;
  }
  __syncthreads();
  for (int f = 0; f < 3; ++f) {  // C, J, Z are symmetric
    const int blk = f == 0 ? 1 : f == 1 ? 2 : 5;
    for (int e = tid; e < nn; e += 256) {
      const int i = e / n, j = e - i * n;
      if (i < j) {
        const double s = 0.5 * (yb[blk * nn + e] + yb[blk * nn + j * n + i]);
        yb[blk * nn + e] = s;
        yb[blk * nn + j * n + i] = s;
      }
    }
  }
  // forward: the stage inputs; tot holds the step's RK4 sum, ac the step's start
  for (int s = 0; s < 4 * K; ++s) {
    const int q = s & 3;
    const double* A = st + s * 3 * nn;
    const double* J = A + nn;
    const double* E = J + nn;
    __syncthreads();
    if (q == 0)
      for (int e = tid; e < 3 * nn; e += 256) ac[e] = tot[e] = A[e];
    for (int u = tid; u < 2 * nn; u += 256) {
      const int e = u % nn, i = e / n, j = e - i * n;
      const double* X = u < nn ? J : E;
      double x = 0.0;
      for (int l = 0; l < n; ++l) x = fma(B[i * n + l], X[l * n + j], x);
      (u < nn ? G : H)[e] = x;
    }
    __syncthreads();
    const double wk = -h * ((q == 0 || q == 3) ? 1.0 / 6.0 : 1.0 / 3.0), ak = -h * (q < 2 ? 0.5 : 1.0);
    for (int u = tid; u < 3 * nn; u += 256) {
      const int f = u / nn, e = u - f * nn, i = e / n, j = e - i * n;
      double k = 0.0;
      if (f == 0) {
        for (int l = 0; l < n; ++l) k = fma(A[i * n + l], G[l * n + j] - F[l * n + j], k);
      } else if (f == 1) {
        k = -0.5 * (Q[i * n + j] + Q[j * n + i]);
        for (int l = 0; l < n; ++l) {
          k = fma(J[i * n + l], G[l * n + j] - F[l * n + j], k);
          k = fma(-F[l * n + i], J[l * n + j], k);
        }
      } else {
        k = i == j ? -1.0 : 0.0;
        for (int l = 0; l < n; ++l) {
          k = fma(J[i * n + l], H[l * n + j], k);
          k = fma(-F[l * n + i], E[l * n + j], k);
        }
      }
      tot[u] = fma(wk, k, tot[u]);
      if (s + 1 < 4 * K) st[(s + 1) * 3 * nn + u] = q == 3 ? tot[u] : fma(ak, k, ac[u]);
    }
  }
  __syncthreads();
  // reverse
  for (int s = 4 * K - 1; s >= 0; --s) {
    const int q = s & 3;
    const double* A = st + s * 3 * nn;
    const double* J = A + nn;
    const double* E = J + nn;
    // rates' adjoint: the step output's share and, through the next stage's
    // input, that stage's (its J part symmetrised, as the rate is)
    const double wk = -h * ((q == 0 || q == 3) ? 1.0 / 6.0 : 1.0 / 3.0), ak = -h * (q < 2 ? 0.5 : 1.0);
    for (int u = tid; u < 6 * nn; u += 256) {
      const int f = u / nn, e = u - f * nn, i = e / n, j = e - i * n, et = j * n + i;
      double k = wk * (f == 2 ? 0.5 * (yb[u] + yb[2 * nn + et]) : yb[u]);
      if (q < 3) {
        if (f == 0) k = fma(ak, ac[e], k);
        if (f == 2) k = fma(0.5 * ak, ac[nn + e] + ac[nn + et], k);
        if (f == 3) k = fma(ak, ac[2 * nn + e], k);
      }
      kb[u] = k;
    }
    __syncthreads();
    const double *kA = kb, *kC = kb + nn, *kJ = kb + 2 * nn, *kE = kb + 3 * nn, *kB = kb + 4 * nn, *kZ = kb + 5 * nn;
    for (int u = tid; u < 5 * nn; u += 256) {
      const int f = u / nn, e = u - f * nn, i = e / n, j = e - i * n;
      double x = 0.0;
      if (f < 2) {
        const double* X = f == 0 ? J : E;
        for (int l = 0; l < n; ++l) x = fma(B[i * n + l], X[l * n + j], x);
      } else if (f < 4) {
        const double* X = f == 2 ? kA : kB;
        for (int l = 0; l < n; ++l) x = fma(A[l * n + i], X[l * n + j], x);
      } else {
        for (int l = 0; l < n; ++l) x = fma(kC[i * n + l], A[l * n + j], x);
      }
      G[u] = x;  // G, H, AA, AB, CA are contiguous
    }
    __syncthreads();
    for (int u = tid; u < 7 * nn; u += 256) {
      const int f = u / nn, e = u - f * nn, i = e / n, j = e - i * n;
      double x = 0.0;
      if (f == 0) {  // Abar = kA (G - F)' - kB H' - 2 kC A B
        for (int l = 0; l < n; ++l) {
          x = fma(kA[i * n + l], G[j * n + l] - F[j * n + l], x);
          x = fma(-kB[i * n + l], H[j * n + l], x);
          x = fma(-2.0 * CA[i * n + l], B[l * n + j], x);
        }
        ac[e] = x;
      } else if (f == 1) {  // Jbar = kE H' - kJ F' - F kJ + kJ G' (+ B Gbar)
        for (int l = 0; l < n; ++l) {
          x = fma(kE[i * n + l], H[j * n + l], x);
          x = fma(kJ[i * n + l], G[j * n + l] - F[j * n + l], x);
          x = fma(-F[i * n + l], kJ[l * n + j], x);
        }
        ac[nn + e] = x;
      } else if (f == 2) {  // Ebar = -F kE + H kZ (+ B Hbar)
        for (int l = 0; l < n; ++l) {
          x = fma(-F[i * n + l], kE[l * n + j], x);
          x = fma(H[i * n + l], kZ[l * n + j], x);
        }
        ac[2 * nn + e] = x;
      } else if (f == 3) {  // Gbar = A' kA + J kJ
        x = AA[e];
        for (int l = 0; l < n; ++l) x = fma(J[i * n + l], kJ[l * n + j], x);
        Gb[e] = x;
      } else if (f == 4) {  // Hbar = -A' kB + J kE + E kZ
        x = -AB[e];
        for (int l = 0; l < n; ++l) {
          x = fma(J[i * n + l], kE[l * n + j], x);
          x = fma(E[i * n + l], kZ[l * n + j], x);
        }
        Hb[e] = x;
      } else if (f == 5) {  // Fbar -= A' kA + E kE' + 2 J kJ
        x = AA[e];
        for (int l = 0; l < n; ++l) {
          x = fma(E[i * n + l], kE[j * n + l], x);
          x = fma(2.0 * J[i * n + l], kJ[l * n + j], x);
        }
        Fb[e] -= x;
      } else {  // Bbar -= A' kC A ; Qbar -= kJ
        for (int l = 0; l < n; ++l) x = fma(A[l * n + i], CA[l * n + j], x);
        Bb[e] -= x;
        Qb[e] -= kJ[e];
      }
    }
    __syncthreads();
    for (int u = tid; u < 3 * nn; u += 256) {
      const int f = u / nn, e = u - f * nn, i = e / n, j = e - i * n;
      double x = 0.0;
      if (f == 0) {
        for (int l = 0; l < n; ++l) x = fma(B[i * n + l], Gb[l * n + j], x);
        ac[nn + e] += x;
      } else if (f == 1) {
        for (int l = 0; l < n; ++l) x = fma(B[i * n + l], Hb[l * n + j], x);
        ac[2 * nn + e] += x;
      } else {
        for (int l = 0; l < n; ++l) {
          x = fma(Gb[i * n + l], J[j * n + l], x);
          x = fma(Hb[i * n + l], E[j * n + l], x);
        }
        Bb[e] += x;
      }
    }
    __syncthreads();
    // the step input's adjoint: the output's plus the four stage inputs'
    for (int u = tid; u < 3 * nn; u += 256) {
      const int f = u / nn, e = u - f * nn;
      const double x = (q == 3 ? 0.0 : tot[u]) + ac[u];
      if (q == 0)
        yb[(f == 0 ? 0 : f == 1 ? 2 : 3) * nn + e] += x;
      else
        tot[u] = x;
    }
    __syncthreads();
  }
  for (int e = tid; e < nn; e += 256) {
    const int i = e / n, j = e - i * n;
    oF[e] = Fb[e];
    oB[e] = Bb[e];
    double x = 0.5 * (Qb[e] + Qb[j * n + i]);
    if (v == 0)
      for (int b = 0; b < a.parts; ++b) x += a.part[(int64_t)b * 13 * nn + 12 * nn + e];
    oX[e] = x;
  }
}

int uniform_adjoint_parts(int64_t T) {
  const int64_t c = (T + kChunk - 1) / kChunk;
  return (int)(c < 304 ? c : 304);
}

cudaError_t launch_uniform_adjoint(const UniAdjArgs& a, cudaStream_t st) {
  const int nn = a.n * a.n;
  uniform_adjoint_sums_kernel<<<(unsigned)a.parts, 256, 0, st>>>(a);
  count_launch();
  // the limit of the largest n and K (8, 8: 65 KB), whatever these: the attribute
  // belongs to all of the process's threads (lqt_grid.cu, launch_tiles)
  auto bytes = [](int K, int n) { return (size_t)(12 + 6 + 6 + 3 + 3 + 12 * K) * n * n * sizeof(double); };
  const size_t smem = bytes(a.K, a.n);
  const cudaError_t e = cudaFuncSetAttribute(uniform_adjoint_sweep_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)bytes(8, 8));
  if (e != cudaSuccess) return e;
  uniform_adjoint_sweep_kernel<<<3, 256, smem, st>>>(a);
  count_launch();
  return cudaGetLastError();
}

}  // namespace lqt
