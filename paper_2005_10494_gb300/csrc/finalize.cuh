// Gradient finalisation (finalize.cu).
#pragma once

#include "mcd_internal.cuh"

namespace mcd {

constexpr int kFinalizeMany = 2048;    // from here on eight lanes per design, from eight times as many two, a warp below

// Counts, estimates and gradients of every design; `dims` has bit d set for
// each dimension that the designs have (a launch per dimension).
cudaError_t launch_finalize_grad(const FinalizeParams& p, uint32_t dims, cudaStream_t stream);

}  // namespace mcd
