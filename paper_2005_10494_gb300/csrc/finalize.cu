// Count -> probability and gradient finalisation (FP64).
#include <cmath>
#include <cstdint>
#include <utility>

#include "finalize.cuh"

namespace mcd {

namespace {

__device__ __forceinline__ int tri(int i, int j) { return i * (i + 1) / 2 + j; }

// Counts to probabilities, one thread per design.
__device__ __forceinline__ double finalize_counts(const FinalizeParams& P, int j, bool write) {
    const uint64_t N = P.n_draws[j];
    const uint64_t h_any = P.hits[j];
    const bool any = (P.region == MCD_ANY_EXCEEDS);
    const double Nd = static_cast<double>(N);
    const double p_any = N ? static_cast<double>(h_any) / Nd : 0.0;
    if (write) {
        const double p = any ? p_any : (N ? 1.0 - p_any : 0.0);
        if (P.out_hits) P.out_hits[j] = any ? h_any : N - h_any;
        if (P.out_p) P.out_p[j] = p;
        if (P.out_se) P.out_se[j] = N ? sqrt(p * (1.0 - p) / Nd) : 0.0;
    }
    return p_any;
}

__global__ void finalize_kernel(const FinalizeParams P) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < P.n_design) finalize_counts(P, j, true);
}

// Solve L^T g = v in place (L packed lower, FP64), with the reciprocals
// rdiag[i] = 1 / L_ii.
template <int D>
__device__ __forceinline__ void solve_lt(const double* L, const double (&rdiag)[D], double (&v)[D]) {
#pragma unroll
    for (int i = D - 1; i >= 0; --i) {
        double s = v[i];
#pragma unroll
        for (int k = i + 1; k < D; ++k) s -= L[tri(k, i)] * v[k];
        v[i] = s * rdiag[i];
    }
}

__device__ __forceinline__ double group_sum(double v, int Q) {
    for (int o = Q >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Gradients of the designs of dimension D: Q lanes per design, which share its
// batch slots (slot q, q + Q, ..).  A thread per design read its 3 D x 32
// accumulators and solved 32 triangular systems in one chain, with a few
// thousand threads on the GPU: 1.07 ms for 4096 designs of d = 20, 0.46 ms for
// 1024 of d = 10, 0.37 ms for 65,536 of d = 3.  The FP64 operations (two lanes
// a clock and SM) bound it now, so the lanes are kept few where the designs
// are many: the final estimate is formed by all Q lanes alike.
// W <= Q lanes of a design share its reciprocals (W = 2 for Q = 2, else 8).
template <int D, int W>
__global__ void __launch_bounds__(128) finalize_grad_kernel(const FinalizeParams P, int Q) {
    const int j = (blockIdx.x * 128 + threadIdx.x) / Q, q = threadIdx.x % Q;
    const bool there = j < P.n_design && P.designs[j < P.n_design ? j : 0].d == D;
    if (!__any_sync(0xffffffffu, there)) return;
    const int jj = there ? j : 0;
    const DesignRec dr = P.designs[jj];
    const double p_any = finalize_counts(P, jj, there && q == 0);
    const int B = there ? P.batches : 0;
    const uint64_t N = P.n_draws[jj];
    const double Nd = static_cast<double>(N);
    const double rN = N ? 1.0 / Nd : 0.0;
    const double sign = P.region == MCD_ANY_EXCEEDS ? 1.0 : -1.0;
    const double* L = P.L64 + P.L_off[dr.scen];
    const int k = P.k;
    const int nout = k > 0 ? k : D;
    const int64_t out_off = k > 0 ? static_cast<int64_t>(jj) * k : dr.vec_off;
    const double* J = P.jac ? P.jac + dr.vec_off * k : nullptr;
    if (k > 0 && !J) return;   // the host rejects this; never dereference a missing Jacobian
    const unsigned long long* acc = P.gacc + dr.acc_off;
    const uint64_t* bd = P.batch_draws + static_cast<int64_t>(jj) * P.batches;

    double G[D], rdiag[D];
    // reciprocal pivots, each formed by one of W lanes of the design
    double own[(D + W - 1) / W];
    const int sub = threadIdx.x & (W - 1);
#pragma unroll
    for (int e = 0; e < (D + W - 1) / W; ++e) {
        const int i = sub + W * e;
        own[e] = there && i < D ? 1.0 / L[tri(i, i)] : 0.0;
    }
#pragma unroll
    for (int i = 0; i < D; ++i) rdiag[i] = __shfl_sync(0xffffffffu, own[i / W], i % W, W);
    // sums over the slots in whole numbers (high and low halves apart, so that
    // no total can overflow), converted once
    long long sh[3 * D];
    unsigned long long sl[3 * D];
#pragma unroll
    for (int e = 0; e < 3 * D; ++e) { sh[e] = 0; sl[e] = 0ull; }
    int nonempty = 0;
    for (int bt = q; bt < B; bt += Q) {
        const unsigned long long* a = acc + static_cast<int64_t>(bt) * 3 * D;
#pragma unroll
        for (int e = 0; e < 3 * D; ++e) {
            const unsigned long long v = a[e];
            sh[e] += static_cast<long long>(v) >> 32;
            sl[e] += v & 0xffffffffull;
        }
        if (bd[bt] > 0) ++nonempty;
    }
    const double unit = 1.0 / static_cast<double>(1ull << kGradFixBits);
    auto total = [&](int e) {
        long long h = sh[e];
        unsigned long long l = sl[e];
        for (int o = Q >> 1; o > 0; o >>= 1) {
            h += __shfl_xor_sync(0xffffffffu, h, o);
            l += __shfl_xor_sync(0xffffffffu, l, o);
        }
        return (static_cast<double>(h) * 4294967296.0 + static_cast<double>(l)) * unit;
    };
    // likelihood ratio with the zero-mean control variate: L^-T (A - p B) / N
    double g[D];
#pragma unroll
    for (int i = 0; i < D; ++i) {
        g[i] = (total(i) - p_any * total(D + i)) * rN;
        G[i] = P.hinv > 0.0 ? total(2 * D + i) * P.hinv * rN : 0.0;
    }
    for (int o = Q >> 1; o > 0; o >>= 1) nonempty += __shfl_xor_sync(0xffffffffu, nonempty, o);
    if (there) solve_lt<D>(L, rdiag, g);
    // component m of the chained gradient -(dt/dtheta)^T v (or v itself)
    auto chain = [&](const double (&v)[D], int m) {
        double c = 0.0;
        if (k > 0) {
#pragma unroll
            for (int i = 0; i < D; ++i) c -= J[i * k + m] * v[i];
        } else {
#pragma unroll
            for (int i = 0; i < D; ++i)
                if (i == m) c = v[i];
        }
        return sign * c;
    };
    if (there && q == 0) {
        for (int m = 0; m < nout; ++m) {
            if (P.g_lr) P.g_lr[out_off + m] = chain(g, m);
            if (P.g_sig && P.hinv > 0.0) P.g_sig[out_off + m] = chain(G, m);
        }
    }
    if (!P.g_se) return;
    // batch means: per batch the same estimator on its own draws
    constexpr int M = D > 8 ? D : 8;                     // outputs: D, or k <= 8
    double ss[M], est[M];
#pragma unroll
    for (int m = 0; m < M; ++m) {
        ss[m] = 0.0;
        est[m] = m < nout && there ? chain(g, m) : 0.0;
    }
    for (int bt = q; bt < B; bt += Q) {
        const uint64_t nb = bd[bt];
        if (!nb) continue;
        const double nbd = static_cast<double>(nb), rnb = unit / nbd;
        const unsigned long long* a = acc + static_cast<int64_t>(bt) * 3 * D;
        double v[D];
#pragma unroll
        for (int i = 0; i < D; ++i) v[i] = (static_cast<double>(static_cast<long long>(a[i])) - p_any * static_cast<double>(static_cast<long long>(a[D + i]))) * rnb;
        solve_lt<D>(L, rdiag, v);
#pragma unroll
        for (int m = 0; m < M; ++m) {
            if (m < nout) {
                const double dev = chain(v, m) - est[m];
                ss[m] += nbd * dev * dev;
            }
        }
    }
#pragma unroll
    for (int m = 0; m < M; ++m) {
        if (m < nout) {                                   // the same for all lanes
            const double s = group_sum(ss[m], Q);
            if (there && q == 0 && m < nout)
                P.g_se[out_off + m] = nonempty >= 2 ? sqrt(s / (Nd * (nonempty - 1))) : NAN;
        }
    }
}

}  // namespace

cudaError_t launch_finalize(const FinalizeParams& p, bool grad, cudaStream_t stream) {
    if (p.n_design == 0) return cudaSuccess;
    if (grad) return cudaErrorInvalidValue;               // launch_finalize_grad
    const int threads = 128;
    finalize_kernel<<<(p.n_design + threads - 1) / threads, threads, 0, stream>>>(p);
    return cudaGetLastError();
}

namespace {

using FinalizeFn = void (*)(FinalizeParams, int);
template <int W, int... I>
FinalizeFn finalize_fn(int d, std::integer_sequence<int, I...>) {
    constexpr FinalizeFn table[] = {&finalize_grad_kernel<I + 1, W>...};
    return table[d - 1];
}

}  // namespace

cudaError_t launch_finalize_grad(const FinalizeParams& p, uint32_t dims, cudaStream_t stream) {
    if (p.n_design == 0) return cudaSuccess;
    const int Q = p.n_design >= 8 * kFinalizeMany ? 2 : p.n_design >= kFinalizeMany ? 8 : 32, threads = 128;
    for (int d = 1; d <= kMaxD; ++d) {
        if (!(dims >> d & 1u)) continue;
        const unsigned grid = static_cast<unsigned>((static_cast<int64_t>(p.n_design) * Q + threads - 1) / threads);
        const auto all = std::make_integer_sequence<int, kMaxD>();
        (Q < 8 ? finalize_fn<2>(d, all) : finalize_fn<8>(d, all))<<<grid, threads, 0, stream>>>(p, Q);
    }
    return cudaGetLastError();
}

}  // namespace mcd
