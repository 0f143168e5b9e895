// Ranked shared-draw kernels, dimensions 1..6.
#include "ranked.cuh"

namespace mcd {

const void* rank_kernels_a(int d, int words, RankKernels* k) {
    switch (d) {
        case 1: return rank_kernels<1>(words, k);
        case 2: return rank_kernels<2>(words, k);
        case 3: return rank_kernels<3>(words, k);
        case 4: return rank_kernels<4>(words, k);
        case 5: return rank_kernels<5>(words, k);
        case 6: return rank_kernels<6>(words, k);
        default: return nullptr;
    }
}

}  // namespace mcd
