// Ranked shared-draw kernels, dimensions 7..12.
#include "ranked.cuh"

namespace mcd {

const void* rank_kernels_b(int d, int words, RankKernels* k) {
    switch (d) {
        case 7: return rank_kernels<7>(words, k);
        case 8: return rank_kernels<8>(words, k);
        case 9: return rank_kernels<9>(words, k);
        case 10: return rank_kernels<10>(words, k);
        case 11: return rank_kernels<11>(words, k);
        case 12: return rank_kernels<12>(words, k);
        default: return nullptr;
    }
}

}  // namespace mcd
