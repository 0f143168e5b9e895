// Count -> probability and gradient finalisation (FP64).
#include <utility>

#include "finalize.cuh"

namespace mcd {

namespace {

__global__ void finalize_kernel(const FinalizeParams P) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < P.n_design) finalize_counts(P, j, true);
}

// Every design has dimension D.  Seven blocks per SM (128 registers) up to d = 10
// hold 65,536 designs at once (d = 10, 4 slots, Jacobian: 237 us at 168
// registers, 141); beyond, that would spill several hundred bytes a thread.
template <int D>
__global__ void __launch_bounds__(kFinThreads, D <= 10 ? 7 : 1) finalize_grad_kernel(const FinalizeParams P, int Q) {
    __shared__ double rdiag[D * kFinThreads];
    const int j = static_cast<int>((blockIdx.x * static_cast<unsigned>(kFinThreads) + threadIdx.x) / Q);
    const bool there = j < P.n_design;
    if (!__any_sync(0xffffffffu, there)) return;
    finalize_grad<D>(P, Q, there ? j : 0, threadIdx.x % Q, there, rdiag + threadIdx.x / Q, kFinThreads / Q);
}

// Lanes per design: enough for about 24,000 threads, no more than it has slots,
// and two at least where it has 16 or more.  Us with 1, 2, 4, 8, 16 and 32 lanes
// (d = 10, 32 slots): 64 designs 216, 125, 72, 45, 35, 31; 5000 257, 127, 121, 110,
// 129, 182; 20,000 452, 328, 353, 328, 456, 669.  With 4 slots, 1, 2 and 4 lanes:
// 5000 49, 33, 43; 65,536 164, 219, 286.
int finalize_lanes(int n_design, int batches) {
    const int least = batches < 16 ? 1 : 2;
    int Q = 32;
    while (Q > least && (Q > batches || static_cast<int64_t>(Q) * n_design > 24000)) Q >>= 1;
    return Q;
}

using FinalizeFn = void (*)(FinalizeParams, int);
template <int... I>
FinalizeFn finalize_fn(int d, std::integer_sequence<int, I...>) {
    constexpr FinalizeFn table[] = {&finalize_grad_kernel<I + 1>...};
    return table[d - 1];
}

}  // namespace

cudaError_t launch_finalize(const FinalizeParams& p, cudaStream_t stream) {
    if (p.n_design == 0) return cudaSuccess;
    const int threads = 128;
    finalize_kernel<<<(p.n_design + threads - 1) / threads, threads, 0, stream>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_finalize_grad(const FinalizeParams& p, const FinalizeDims& t, cudaStream_t stream) {
    if (p.n_design == 0) return cudaSuccess;
    const int Q = finalize_lanes(p.n_design, p.batches);
    if (t.order) return launch_finalize_mixed(p, t, Q, stream);
    int d = 1;
    while (t.first[d] == 0) ++d;
    const int64_t threads = static_cast<int64_t>(p.n_design) * Q;
    finalize_fn(d, std::make_integer_sequence<int, kMaxD>())<<<static_cast<int>((threads + kFinThreads - 1) / kFinThreads),
                                                               kFinThreads, 0, stream>>>(p, Q);
    return cudaGetLastError();
}

}  // namespace mcd
