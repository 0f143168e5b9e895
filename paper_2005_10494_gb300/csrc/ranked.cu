// Threshold sort of the ranked shared-draw path, and its launches.
#include <algorithm>

#include "ranked.cuh"

namespace mcd {

const void* rank_kernels_a(int d, int words, RankKernels* k);
const void* rank_kernels_b(int d, int words, RankKernels* k);
const void* rank_kernels_c(int d, int words, RankKernels* k);
const void* rank_kernels_d(int d, int words, RankKernels* k);

namespace {

bool select_rank(int d, int words, RankKernels* k) {
    if (d < 1 || d > kMaxD) return false;
    const void* fn = d <= 6 ? rank_kernels_a(d, words, k) : d <= 12 ? rank_kernels_b(d, words, k)
                   : d <= 16 ? rank_kernels_c(d, words, k) : rank_kernels_d(d, words, k);
    return fn != nullptr;
}

// A block per family and coordinate: bitonic sort of the thresholds as ordered
// 32-bit keys, kKeys neighbouring ones per thread in registers (strides below
// kKeys inside a thread, below 32 kKeys by shuffles, above through shared
// memory), then the distinct values and each design's position among them by
// binary search.
constexpr int kKeys = kRankMaxFamily / kRankSortThreads;

// Place of sorted value q in shared memory: a gap every 32 words keeps the
// power-of-two strides of the binary search on different banks.
__device__ __forceinline__ int skew(int q) { return q + (q >> 5); }


__global__ void __launch_bounds__(kRankSortThreads) rank_sort_kernel(const __grid_constant__ RankParams R, int d) {
    __shared__ uint32_t sk[kRankMaxFamily + kRankMaxFamily / 32];
    __shared__ int swarp[kRankSortThreads / 32];
    const int i = blockIdx.y, tid = threadIdx.x, e0 = tid * kKeys;
    const RankFam fm = R.fams[R.fam0 + blockIdx.x];
    int size = 32;
    while (size < fm.cnt) size <<= 1;
    const uint32_t inf = order_float(INFINITY);
    // the thresholds of designs tid, tid + kRankSortThreads, ..: all loads in flight
    uint32_t mine[kKeys], key[kKeys];
    int64_t vo[kKeys];
    double bb[kKeys], mm[kKeys];
#pragma unroll
    for (int r = 0; r < kKeys; ++r) {
        const int q = tid + r * kRankSortThreads;
        vo[r] = q < fm.cnt ? R.designs[R.list[fm.list_off + q]].vec_off + i : -1;
    }
#pragma unroll
    for (int r = 0; r < kKeys; ++r) {
        bb[r] = vo[r] >= 0 ? R.b[vo[r]] : 0.0;
        mm[r] = vo[r] >= 0 ? R.mu[vo[r]] : 0.0;
    }
#pragma unroll
    for (int r = 0; r < kKeys; ++r) {
        const int q = tid + r * kRankSortThreads;
        mine[r] = 0xffffffffu;
        if (q < fm.cnt) {
            const double tt = bb[r] - mm[r];
            if (tt != tt) {
                set_status(R.status, MCD_ENAN, R.list[fm.list_off + q]);
                mine[r] = inf;                            // exceeded by no draw
            } else {
                mine[r] = order_float(static_cast<float>(tt) + 0.0f);   // -0 and +0 compare equal: one key
            }
        }
        if (q < size) sk[q] = mine[r];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kKeys; ++r) key[r] = e0 + r < size ? sk[e0 + r] : 0xffffffffu;
    for (int k = 2; k <= size; k <<= 1) {
        for (int s = k >> 1; s >= kKeys; s >>= 1) {
            const bool keep_min = ((e0 & s) == 0) == ((e0 & k) == 0);
            if (s >= 32 * kKeys) {
                __syncthreads();
#pragma unroll
                for (int r = 0; r < kKeys; ++r) sk[r * kRankSortThreads + tid] = key[r];
                __syncthreads();
#pragma unroll
                for (int r = 0; r < kKeys; ++r) {
                    const uint32_t o = sk[r * kRankSortThreads + (tid ^ (s / kKeys))];
                    key[r] = keep_min ? min(key[r], o) : max(key[r], o);
                }
            } else {
#pragma unroll
                for (int r = 0; r < kKeys; ++r) {
                    const uint32_t o = __shfl_xor_sync(0xffffffffu, key[r], s / kKeys);
                    key[r] = keep_min ? min(key[r], o) : max(key[r], o);
                }
            }
        }
#pragma unroll
        for (int s = kKeys / 2; s > 0; s >>= 1) {
            if (s >= k) continue;
#pragma unroll
            for (int r = 0; r < kKeys; ++r) {
                if (r & s) continue;
                const uint32_t lo = min(key[r], key[r + s]), hi = max(key[r], key[r + s]);
                const bool up = ((e0 + r) & k) == 0;
                key[r] = up ? lo : hi;
                key[r + s] = up ? hi : lo;
            }
        }
    }
    __syncthreads();
    // distinct finite keys: flags, block scan, compaction into sk
#pragma unroll
    for (int r = 0; r < kKeys; ++r) sk[e0 + r] = key[r];
    __syncthreads();
    uint32_t prev = e0 > 0 ? sk[e0 - 1] : 0u;
    bool first = e0 == 0;
    unsigned flags = 0u;
    int c = 0;
#pragma unroll
    for (int r = 0; r < kKeys; ++r) {
        const bool f = e0 + r < size && key[r] < inf && (first || key[r] != prev);
        flags |= f ? 1u << r : 0u;
        c += f ? 1 : 0;
        prev = key[r];
        first = false;
    }
    const int lane = tid & 31, warp = tid >> 5;
    int sum = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, sum, o);
        if (lane >= o) sum += v;
    }
    __syncthreads();
    if (lane == 31) swarp[warp] = sum;
    __syncthreads();
    int at = sum - c, total = 0;
    for (int w = 0; w < kRankSortThreads / 32; ++w) {
        if (w < warp) at += swarp[w];
        total += swarp[w];
    }
#pragma unroll
    for (int r = 0; r < kKeys; ++r)
        if (flags >> r & 1u) sk[skew(at++)] = key[r];     // (every key is in a register by now)
    __syncthreads();
    const int64_t base = (static_cast<int64_t>(blockIdx.x) * d + i) * R.fam_cap;
    for (int q = tid; q < R.fam_cap; q += kRankSortThreads)
        R.distinct[base + q] = q < total ? unorder_float(sk[skew(q)]) : INFINITY;
    int lo[kKeys];                                        // distinct values below each threshold
#pragma unroll
    for (int r = 0; r < kKeys; ++r) lo[r] = 0;
    for (int st = kRankMaxFamily / 2; st > 0; st >>= 1) {
#pragma unroll
        for (int r = 0; r < kKeys; ++r)
            if (lo[r] + st <= total && sk[skew(lo[r] + st - 1)] < mine[r]) lo[r] += st;
    }
#pragma unroll
    for (int r = 0; r < kKeys; ++r) {
        const int q = tid + r * kRankSortThreads;
        if (q < fm.cnt) R.pos[base + q] = mine[r] < inf ? static_cast<uint16_t>(lo[r]) : kRankNone;
    }
    if (tid == 0) R.n_distinct[blockIdx.x * d + i] = total;
}

}  // namespace

int rank_family(int d) { return d <= 6 ? 4096 : d <= 13 ? 2048 : 1024; }

int rank_words(int d, int cnt) { return cnt <= 128 ? 4 : (cnt <= 256 || d > 3) ? 8 : 16; }

int rank_batch(int d, int words, int* threads) {
    RankKernels k;
    if (!select_rank(d, words, &k)) return 0;
    if (threads) *threads = k.threads;
    return k.batch;
}

cudaError_t launch_rank_sort(int d, const RankParams& p, cudaStream_t stream) {
    rank_sort_kernel<<<dim3(p.n_fam, d), kRankSortThreads, 0, stream>>>(p, d);
    return cudaGetLastError();
}

namespace {

// Dynamic shared memory of the two kernels for families of up to `cap` designs.
size_t draws_smem(int d, int cap) { return static_cast<size_t>(d) * cap * sizeof(float); }
size_t count_smem(const RankKernels& k, int d, int cap) {
    return k.count_rows + static_cast<size_t>(d) * (cap / 32 + 1) * 8;
}

// The limit is a property of the function, common to every context and thread,
// so it is always written with the same value: what the largest family needs
// (106 KB and 218 KB at most).  A value per launch let a thread with small
// families lower it between another's call here and its launch, which then failed.
cudaError_t set_limit(const void* fn, size_t largest) {
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(largest));
}

}  // namespace

cudaError_t launch_rank_draws(int d, const RankParams& p, int sms, cudaStream_t stream) {
    RankKernels k;
    if (!select_rank(d, 4, &k)) return cudaErrorInvalidValue;
    const size_t smem = draws_smem(d, p.fam_cap);
    cudaError_t e = set_limit(k.draws, draws_smem(d, rank_family(d)));
    if (e != cudaSuccess) return e;
    int bps = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, k.draws, kRankDrawThreads, smem)) != cudaSuccess) return e;
    const int64_t grid = std::min<int64_t>(static_cast<int64_t>(std::max(bps, 1)) * sms, p.n_tiles);
    void* args[] = {const_cast<RankParams*>(&p)};
    return cudaLaunchKernel(k.draws, dim3(static_cast<unsigned>(grid)), dim3(kRankDrawThreads), args, smem, stream);
}

cudaError_t launch_rank_count(int d, int words, const RankParams& p, int sms, cudaStream_t stream) {
    RankKernels k;
    if (!select_rank(d, words, &k)) return cudaErrorInvalidValue;
    const size_t smem = count_smem(k, d, p.fam_cap);
    cudaError_t e = set_limit(k.count, count_smem(k, d, rank_family(d)));
    if (e != cudaSuccess) return e;
    int bps = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, k.count, k.threads, smem)) != cudaSuccess) return e;
    if (bps < 1) return cudaErrorLaunchOutOfResources;
    const int64_t grid = std::min<int64_t>(static_cast<int64_t>(bps) * sms, p.n_units);
    void* args[] = {const_cast<RankParams*>(&p)};
    return cudaLaunchKernel(k.count, dim3(static_cast<unsigned>(grid)), dim3(k.threads), args, smem, stream);
}

}  // namespace mcd
