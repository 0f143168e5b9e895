// Small kernels around the sampling pass: the FP64 Cholesky factorisation of
// each scenario's Sigma and the unit-check normals.
#include <cmath>
#include <cstdint>

#include "chol.cuh"
#include "mcd_internal.cuh"
#include "rng.cuh"

namespace mcd {

namespace {

// Sigma_s = L L^T, a warp or a thread per scenario.
constexpr int kCholWarps = 2, kCholThreads = 64;

template <bool WARP>
__global__ void __launch_bounds__(64) cholesky_kernel(const double* __restrict__ Sigma, const int64_t* __restrict__ sig_off,
                                                      const int32_t* __restrict__ scen_d, const int64_t* __restrict__ L_off,
                                                      int n_scen, float* __restrict__ L32, double* __restrict__ L64,
                                                      int32_t* __restrict__ scen_ok, DevStatus* status) {
    const int s = WARP ? blockIdx.x * kCholWarps + (threadIdx.x >> 5) : blockIdx.x * kCholThreads + threadIdx.x;
    if (s >= n_scen) return;
    const bool good = WARP ? warp_factor(Sigma + sig_off[s], scen_d[s], L64 + L_off[s], L32 + L_off[s])
                           : thread_factor(Sigma + sig_off[s], scen_d[s], L64 + L_off[s], L32 + L_off[s]);
    if (!WARP || (threadIdx.x & 31) == 0) {
        scen_ok[s] = good ? 1 : 0;
        if (!good) set_status(status, MCD_ENOTSPD, s);
    }
}

__global__ void debug_normals_kernel(uint64_t seed, uint64_t key, uint64_t m_begin, uint64_t count,
                                     float* z32, double* z64, uint32_t* words) {
    uint32_t rk0[10], rk1[10];
    for (int r = 0; r < 10; ++r) {
        rk0[r] = static_cast<uint32_t>(seed) + static_cast<uint32_t>(r) * kPhiloxW0;
        rk1[r] = static_cast<uint32_t>(seed >> 32) + static_cast<uint32_t>(r) * kPhiloxW1;
    }
    const uint64_t first_call = m_begin >> 2;
    const uint64_t ncalls = count ? ((m_begin + count - 1) >> 2) - first_call + 1 : 0;
    const uint64_t idx = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (idx < count) {
        const uint64_t m = m_begin + idx;
        const uint4 w = philox_full(m >> 2, key, rk0, rk1);
        float f[4];
        double g[4];
        normals4<float>(w, f);
        normals4<double>(w, g);
        if (z32) z32[idx] = f[m & 3];
        if (z64) z64[idx] = g[m & 3];
    }
    if (words && idx < ncalls) {
        const uint4 w = philox_full(first_call + idx, key, rk0, rk1);
        words[4 * idx + 0] = w.x;
        words[4 * idx + 1] = w.y;
        words[4 * idx + 2] = w.z;
        words[4 * idx + 3] = w.w;
    }
}

}  // namespace

// A warp per scenario costs 32 lanes' worth of the FP64 rate: us for a thread and
// for a warp each, with 1024, 2048, 4096 and 8192 scenarios: d = 6 16.5, 18.5; 16.4,
// 29; 16.5, 55; 16.5, 103; d = 10 41, 29; 41, 45; 41, 90; 41, 172; d = 20 190, 57; 194, 96; 195,
// 191; 197, 373.  `max_d` is the largest dimension of the scenarios, whose chain a
// launch of threads waits for.
cudaError_t launch_cholesky(const double* Sigma, const int64_t* sig_off, const int32_t* scen_d,
                            const int64_t* L_off, int n_scen, int max_d, float* L32, double* L64,
                            int32_t* scen_ok, DevStatus* status, cudaStream_t stream) {
    if (max_d > kCholThreadD && n_scen <= 230 * (max_d - 4))
        cholesky_kernel<true><<<(n_scen + kCholWarps - 1) / kCholWarps, 32 * kCholWarps, 0, stream>>>(
            Sigma, sig_off, scen_d, L_off, n_scen, L32, L64, scen_ok, status);
    else
        cholesky_kernel<false><<<(n_scen + kCholThreads - 1) / kCholThreads, kCholThreads, 0, stream>>>(
            Sigma, sig_off, scen_d, L_off, n_scen, L32, L64, scen_ok, status);
    return cudaGetLastError();
}

cudaError_t launch_debug_normals(uint64_t seed, uint64_t key, uint64_t m_begin, uint64_t count,
                                 float* z32, double* z64, uint32_t* words, cudaStream_t stream) {
    if (count == 0) return cudaSuccess;
    const uint64_t ncalls = ((m_begin + count - 1) >> 2) - (m_begin >> 2) + 1;
    const uint64_t n = count > ncalls ? count : ncalls;
    const int threads = 256;
    debug_normals_kernel<<<static_cast<unsigned>((n + threads - 1) / threads), threads, 0, stream>>>(
        seed, key, m_begin, count, z32, z64, words);
    return cudaGetLastError();
}

}  // namespace mcd
