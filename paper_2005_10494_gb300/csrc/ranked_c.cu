// Ranked shared-draw kernels, dimensions 13..16.
#include "ranked.cuh"

namespace mcd {

const void* rank_kernels_c(int d, int words, RankKernels* k) {
    switch (d) {
        case 13: return rank_kernels<13>(words, k);
        case 14: return rank_kernels<14>(words, k);
        case 15: return rank_kernels<15>(words, k);
        case 16: return rank_kernels<16>(words, k);
        default: return nullptr;
    }
}

}  // namespace mcd
