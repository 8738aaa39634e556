// Device declarations of the constant-coefficient element build
// (lqt_uniform.cu) that the general build kernels need to leave its
// sub-intervals alone.
#pragma once

#include <cuda_runtime.h>

namespace lqt {

// Table of one problem, in doubles: header (valid flag, step h, 1 / (h+ -
// h-)), then A, C, J, E^T, Bq^T, Z (n x n each) at the steps h, h+, h-, then the
// low parts of those at h.
constexpr int kUniHeader = 16;
constexpr double kUniStep = 1e-4;      // (h+- - h) / h
constexpr double kUniNear = 1e-9;      // largest |h_j - h| / h served by the table

// The RK4 step of sub-interval j and whether the table serves it.  Written
// with explicit roundings so that every kernel takes the same decision.
__device__ __forceinline__ double uniform_step(const double* t, int64_t j, int32_t K) {
  return __ddiv_rn(__dsub_rn(t[j + 1], t[j]), (double)K);
}
__device__ __forceinline__ bool uniform_near_h(double h0, const double* t, int64_t j, int32_t K) {
  return fabs(__dsub_rn(uniform_step(t, j, K), h0)) <= __dmul_rn(kUniNear, h0);
}
// True when sub-interval j's element is written by the table's expansion.
__device__ __forceinline__ bool uniform_near(const double* tab, const double* t, int64_t j, int32_t K) {
  return tab != nullptr && tab[0] != 0.0 && uniform_near_h(tab[1], t, j, K);
}

}  // namespace lqt
