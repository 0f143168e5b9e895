// Ranked shared-draw kernels, dimensions 17..20.
#include "ranked.cuh"

namespace mcd {

const void* rank_kernels_d(int d, int words, RankKernels* k) {
    switch (d) {
        case 17: return rank_kernels<17>(words, k);
        case 18: return rank_kernels<18>(words, k);
        case 19: return rank_kernels<19>(words, k);
        case 20: return rank_kernels<20>(words, k);
        default: return nullptr;
    }
}

}  // namespace mcd
