// Gradient finalisation of designs of several dimensions in one launch: a block
// has designs of one dimension, from a list by dimension.
#include "finalize.cuh"

namespace mcd {

namespace {

__global__ void __launch_bounds__(kFinThreads) finalize_mixed_kernel(const FinalizeParams P, const FinalizeDims T, int Q) {
    __shared__ double rdiag[kMaxD * kFinThreads];
    int d = 1;
    while (d < kMaxD && static_cast<int>(blockIdx.x) >= T.block0[d]) ++d;
    const int at = static_cast<int>(((blockIdx.x - T.block0[d - 1]) * static_cast<unsigned>(kFinThreads) + threadIdx.x) / Q);
    const bool there = at < T.first[d] - T.first[d - 1];
    if (!__any_sync(0xffffffffu, there)) return;
    const int j = static_cast<int>(T.order[T.first[d - 1] + (there ? at : 0)]), q = threadIdx.x % Q;
    double* rd = rdiag + threadIdx.x / Q;
    switch (d) {
#define MCD_FIN_CASE(D) case D: finalize_grad<D>(P, Q, j, q, there, rd, kFinThreads / Q); break;
        MCD_FIN_CASE(1) MCD_FIN_CASE(2) MCD_FIN_CASE(3) MCD_FIN_CASE(4) MCD_FIN_CASE(5) MCD_FIN_CASE(6) MCD_FIN_CASE(7)
        MCD_FIN_CASE(8) MCD_FIN_CASE(9) MCD_FIN_CASE(10) MCD_FIN_CASE(11) MCD_FIN_CASE(12) MCD_FIN_CASE(13)
        MCD_FIN_CASE(14) MCD_FIN_CASE(15) MCD_FIN_CASE(16) MCD_FIN_CASE(17) MCD_FIN_CASE(18) MCD_FIN_CASE(19)
        MCD_FIN_CASE(20)
#undef MCD_FIN_CASE
        default: break;
    }
}

}  // namespace

cudaError_t launch_finalize_mixed(const FinalizeParams& p, const FinalizeDims& t, int lanes, cudaStream_t stream) {
    FinalizeDims b = t;
    b.block0[0] = 0;
    for (int d = 1; d <= kMaxD; ++d)
        b.block0[d] = b.block0[d - 1] + static_cast<int>((static_cast<int64_t>(t.first[d] - t.first[d - 1]) * lanes + kFinThreads - 1) / kFinThreads);
    finalize_mixed_kernel<<<b.block0[kMaxD], kFinThreads, 0, stream>>>(p, b, lanes);
    return cudaGetLastError();
}

}  // namespace mcd
