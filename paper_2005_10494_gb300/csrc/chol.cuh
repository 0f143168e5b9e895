// Cholesky factorisation of one correlation matrix by a warp.
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

}  // namespace mcd
