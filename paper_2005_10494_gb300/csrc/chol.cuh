// Cholesky factorisation of one correlation matrix by a warp or by a thread: the
// same operations on every entry, so the same factors bit for bit.
#pragma once

#include <cmath>

#include "mcd_internal.cuh"

namespace mcd {

// Sigma = L L^T (FP64, lower triangle read) for d <= 20: lane i holds row i in
// registers.  Column by column the pivot comes from its lane by a shuffle, the
// lanes below divide by its root, and each entry takes its updates in the order
// k = 0, 1, .. as one fused multiply-add each: entry for entry the arithmetic of
// the textbook triple loop.  One thread doing that loop waited on every FP64
// operation in turn (164 us at d = 20, 39 us at d = 10, per launch).  Returns
// false when a pivot is not positive and finite.
__device__ __forceinline__ bool warp_cholesky(double (&a)[kMaxD], int d) {
    const int i = threadIdx.x & 31;
#pragma unroll
    for (int c = 0; c < kMaxD; ++c) {
        if (c < d) {                                      // d is warp-uniform
            const double p = __shfl_sync(0xffffffffu, a[c], c);
            if (!(p > 0.0) || !isfinite(p)) return false;
            const double r = sqrt(p);
            if (i == c) a[c] = r;
            else if (i > c) a[c] = a[c] / r;
#pragma unroll
            for (int j = c + 1; j < kMaxD; ++j) {
                if (j < d) {
                    const double ljc = __shfl_sync(0xffffffffu, a[c], j);
                    if (i >= j) a[j] = fma(-a[c], ljc, a[j]);
                }
            }
        }
    }
    return true;
}

// Factor Sigma (row-major d x d) into the packed lower triangles L64 and L32
// (zeros when it fails).
__device__ __forceinline__ bool warp_factor(const double* __restrict__ Sigma, int d, double* __restrict__ L64,
                                            float* __restrict__ L32) {
    const int i = threadIdx.x & 31;
    double a[kMaxD];
#pragma unroll
    for (int j = 0; j < kMaxD; ++j) a[j] = (i < d && j <= i) ? Sigma[i * d + j] : 0.0;
    const bool good = warp_cholesky(a, d);
    if (i < d) {
#pragma unroll
        for (int j = 0; j < kMaxD; ++j) {
            if (j <= i) {
                const double v = good ? a[j] : 0.0;
                L64[i * (i + 1) / 2 + j] = v;
                L32[i * (i + 1) / 2 + j] = static_cast<float>(v);
            }
        }
    }
    return good;
}

// The same by one thread, entry after entry.  It takes a 1/32 of the FP64 lanes,
// so it is the faster one where the scenarios fill the GPU by themselves, and up
// to d = 5 its chain is no longer than the warp's exchanges (us for one scenario,
// thread and warp: d = 1 4.1, 6.2; 3 6.2, 10.3; 5 12.3, 12.4; 6 16.4, 14.4; 10 37, 20;
// 20 160, 35).
constexpr int kCholThreadD = 5;
__device__ __forceinline__ bool thread_factor(const double* __restrict__ Sigma, int d, double* L64, float* L32) {
    bool good = true;
    for (int i = 0; i < d && good; ++i) {
        for (int j = 0; j <= i; ++j) {
            double sum = Sigma[i * d + j];
            for (int k = 0; k < j; ++k) sum -= L64[i * (i + 1) / 2 + k] * L64[j * (j + 1) / 2 + k];
            if (i == j) {
                if (!(sum > 0.0) || !isfinite(sum)) { good = false; break; }
                L64[i * (i + 1) / 2 + i] = sqrt(sum);
            } else {
                L64[i * (i + 1) / 2 + j] = sum / L64[j * (j + 1) / 2 + j];
            }
        }
    }
    for (int q = 0; q < d * (d + 1) / 2; ++q) {
        if (!good) L64[q] = 0.0;
        L32[q] = static_cast<float>(L64[q]);
    }
    return good;
}

}  // namespace mcd
