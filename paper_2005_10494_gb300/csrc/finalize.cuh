// Gradient finalisation (finalize.cu, finalize_mixed.cu).
#pragma once

#include <cmath>

#include "mcd_internal.cuh"

namespace mcd {

// Threads per block: small blocks, so that 65,536 designs spread evenly (128
// threads leave 3 or 4 blocks an SM; d = 3, 4 slots, Jacobian: 74 us, 64 threads 66).
constexpr int kFinThreads = 64;

// The designs by dimension: those of dimension d are order[first[d - 1] .. first[d]);
// `order` is NULL when all have the same.
struct FinalizeDims {
    const uint32_t* order;
    int32_t first[kMaxD + 1];
    int32_t block0[kMaxD + 1];         // first block of dimension d + 1 (set by the launch)
};

// Counts, estimates and gradients of every design, in one launch.
cudaError_t launch_finalize_grad(const FinalizeParams& p, const FinalizeDims& t, cudaStream_t stream);
cudaError_t launch_finalize_mixed(const FinalizeParams& p, const FinalizeDims& t, int lanes, cudaStream_t stream);

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

// Solve L^T g = v in place (L packed lower, FP64), with the reciprocals
// rdiag[i * stride] = 1 / L_ii.
template <int D>
__device__ __forceinline__ void solve_lt(const double* L, const double* rdiag, int stride, double (&v)[D]) {
#pragma unroll
    for (int i = D - 1; i >= 0; --i) {
        double s = v[i];
#pragma unroll
        for (int k = i + 1; k < D; ++k) s -= L[tri(k, i)] * v[k];
        v[i] = s * rdiag[i * stride];
    }
}

template <typename T>
__device__ __forceinline__ T group_sum(T v, int Q) {
    for (int o = Q >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Gradients of design j (dimension D; `there`: this lane has one).  Q lanes of a
// warp per design share its batch slots (slot q, q + Q, ..) and form its
// reciprocal pivots in shared memory (rdiag[i * stride] of this design).
// Few designs wait on the chain of their slots and solves, many on the FP64 rate
// (two lanes a clock and SM): lanes help while they have slots of their own and
// cost every further operation of the design where they have not.  Us, a thread
// per design before, a launch per dimension and at least two lanes whatever the
// slots, and this form: 5000 designs of d = 10 with one slot 29, 53, 16; with 32
// slots 408, 121, 110; 5000 of d = 3..10 with one slot 31, 205, 18; with 32 slots
// 411, 448, 79; 65,536 of d = 3 with 32 slots 298, 250, 243.
template <int D>
__device__ __forceinline__ void finalize_grad(const FinalizeParams& P, int Q, int j, int q, bool there, double* rdiag,
                                              int stride) {
    const DesignRec dr = P.designs[j];
    const double p_any = finalize_counts(P, j, there && q == 0);
    const int B = there ? P.batches : 0;
    const uint64_t N = P.n_draws[j];
    const double Nd = static_cast<double>(N);
    const double rN = N ? 1.0 / Nd : 0.0;
    const double sign = P.region == MCD_ANY_EXCEEDS ? 1.0 : -1.0;
    const double* L = P.L64 + P.L_off[dr.scen];
    const int k = P.k;
    const int nout = k > 0 ? k : D;
    const int64_t out_off = k > 0 ? static_cast<int64_t>(j) * k : dr.vec_off;
    const double* J = P.jac ? P.jac + dr.vec_off * k : nullptr;
    if (k > 0 && !J) return;   // the host rejects this; never dereference a missing Jacobian
    const long long* acc = reinterpret_cast<const long long*>(P.gacc) + dr.acc_off;
    const uint64_t* bd = P.batch_draws + static_cast<int64_t>(j) * P.batches;

    if (there)
        for (int i = q; i < D; i += Q) rdiag[i * stride] = 1.0 / L[tri(i, i)];
    __syncwarp();
    // Likelihood ratio with the zero-mean control variate: L^-T (A - p B) / N.
    // The slots are summed in whole numbers and converted once.  Up to 2^32 draws
    // (of at most 5.8 x 2^28 each) fit 63 bits; beyond, the high and the low
    // halves of the slots are summed one after the other.
    double g[D], G[D];
#pragma unroll
    for (int i = 0; i < D; ++i) g[i] = G[i] = 0.0;
    const double unit = 1.0 / static_cast<double>(1ull << kGradFixBits);
    const bool wide = __any_sync(0xffffffffu, there && N > (1ull << 32));
    int nonempty = 0;
#pragma unroll 1
    for (int half = wide ? 1 : 0; half >= 0; --half) {
        long long sum[3 * D];
#pragma unroll
        for (int e = 0; e < 3 * D; ++e) sum[e] = 0;
        const int sh = half ? 32 : 0;
        const long long keep = wide && !half ? 0xffffffffll : -1ll;
        for (int bt = q; bt < B; bt += Q) {
            const long long* a = acc + static_cast<int64_t>(bt) * 3 * D;
#pragma unroll
            for (int e = 0; e < 3 * D; ++e) sum[e] += (a[e] >> sh) & keep;
            if (!half && bd[bt] > 0) ++nonempty;
        }
        const double scale = half ? unit * 4294967296.0 : unit;
        auto total = [&](int e) { return static_cast<double>(group_sum(sum[e], Q)) * scale; };
#pragma unroll
        for (int i = 0; i < D; ++i) {
            g[i] += (total(i) - p_any * total(D + i)) * rN;
            if (P.hinv > 0.0) G[i] += total(2 * D + i) * P.hinv * rN;
        }
    }
    nonempty = group_sum(nonempty, Q);
    if (there) solve_lt<D>(L, rdiag, stride, g);
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
    constexpr int M = D > 8 ? D : 8;                     // outputs: D, or k <= 8
    double est[M];
#pragma unroll
    for (int m = 0; m < M; ++m) {
        est[m] = 0.0;
        if (m < nout && there) {
            est[m] = chain(g, m);
            if (q == 0) {
                if (P.g_lr) P.g_lr[out_off + m] = est[m];
                if (P.g_sig && P.hinv > 0.0) P.g_sig[out_off + m] = chain(G, m);
            }
        }
    }
    if (!P.g_se) return;
    const bool spread = there && nonempty >= 2;           // else no standard error: NaN
    if (there && !spread && q == 0)
        for (int m = 0; m < nout; ++m) P.g_se[out_off + m] = NAN;
    if (!__any_sync(0xffffffffu, spread)) return;
    // batch means: per batch the same estimator on its own draws
    double ss[M];
#pragma unroll
    for (int m = 0; m < M; ++m) ss[m] = 0.0;
    uint64_t nb_last = 0;
    double rnb = 0.0;                                     // unit / nb, formed only when nb changes
    for (int bt = q; bt < (spread ? B : 0); bt += Q) {
        const uint64_t nb = bd[bt];
        if (!nb) continue;
        const double nbd = static_cast<double>(nb);
        if (nb != nb_last) { rnb = unit / nbd; nb_last = nb; }
        const long long* a = acc + static_cast<int64_t>(bt) * 3 * D;
        double v[D];
#pragma unroll
        for (int i = 0; i < D; ++i) v[i] = (static_cast<double>(a[i]) - p_any * static_cast<double>(a[D + i])) * rnb;
        solve_lt<D>(L, rdiag, stride, v);
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
            if (spread && q == 0) P.g_se[out_off + m] = sqrt(s / (Nd * (nonempty - 1)));
        }
    }
}

}  // namespace mcd
