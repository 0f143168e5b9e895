// Host interface of the ranked shared-draw path (ranked.cuh, ranked.cu).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "mcd_internal.cuh"

namespace mcd {

constexpr int kRankMaxFamily = 4096;   // designs that share one set of sorted thresholds
constexpr int kRankSortThreads = 512;
constexpr int kRankDrawThreads = 512;      // block size of the draws kernel (one group of draws per thread)

// Designs of one common-random-number group: list[list_off .. list_off + cnt).
struct RankFam {
    uint64_t key;
    uint32_t list_off;
    int32_t  cnt;
    int32_t  scen;
    int32_t  pad;
};

// Draws [start, start + n) of a family's stream; its ranks go to draws
// ws_off.. of the workspace, made as tiles tile0.. of the launch.
struct RankSeg {
    uint64_t start;
    uint64_t ws_off;
    int64_t  tile0;
    uint32_t n;
    int32_t  fam;
};

// A chunk of a family's designs against one segment: batches unit0.. of the launch.
struct RankItem {
    int64_t unit0;
    int32_t seg;
    int32_t chunk;
};

struct RankParams {
    const RankFam*   fams;
    const RankSeg*   segs;
    const RankItem*  items;
    const uint32_t*  list;          // design indices
    const DesignRec* designs;
    const double*    mu;
    const double*    b;
    const float*     L32;
    const int64_t*   L_off;
    const int32_t*   scen_ok;
    float*           distinct;      // [family of the batch][d][fam_cap] distinct thresholds, ascending, then +inf
    int32_t*         n_distinct;    // [family of the batch][d]
    uint16_t*        pos;           // [family of the batch][d][fam_cap] position of each design's threshold
    uint16_t*        ranks;         // [draw][d padded to 4]
    unsigned long long* hits;
    DevStatus*       status;
    int64_t          n_tiles, n_units;
    int32_t          fam_cap;       // power of two >= every family's designs
    int32_t          fam0, n_fam;   // families of this batch
    int32_t          seg0, seg1, item0, item1;
    uint32_t         rk0[10], rk1[10];
};

int rank_words(int d, int cnt);                      // words per row for families of cnt designs
int rank_family(int d);                              // largest family
int rank_batch(int d, int words, int* threads);      // draws per batch (and block size) of the count kernel
cudaError_t launch_rank_sort(int d, const RankParams& p, cudaStream_t stream);
cudaError_t launch_rank_draws(int d, const RankParams& p, int sms, cudaStream_t stream);
cudaError_t launch_rank_count(int d, int words, const RankParams& p, int sms, cudaStream_t stream);

}  // namespace mcd
