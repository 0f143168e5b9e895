// Shared-draw adjoint at d = 10..12 and 17..20 (kBoxed): draws that no design of a warp can tell
// apart are added, or dropped, without testing them design by design.
#pragma once

#include "shared.cuh"

namespace mcd {

// The dimensions that have the kernel.  Time without it / with it on 32 x 32, 64 x 64
// and 9 x 15 grids of 1 to 12 ms (geometric mean, least), and on as many scattered
// designs, which fall back to the direct loop: d = 9 0.97, 0.90 and 0.99; 10 1.07, 1.00
// and 0.99; 11 1.15, 1.00 and 1.00; 12 1.16, 1.00 and 0.99; 14 1.04, 0.96 and 0.98; 16 1.07,
// 0.96 and 0.95; 17 1.09, 1.00 and 1.00; 18 1.12, 1.01 and 0.98 (before
// kAgain, below); 19 1.13, 1.02 and 1.00; 20 1.24, 1.03 and 0.97.  At d = 13 and 15 one block fits an SM and the shorter loops
// leave latencies open: 0.91, 0.89.  At d = 5..8, two designs per thread, 0.83, 0.87.
// Not where it loses on either (9, 14, 16); at 20 scattered designs are 2 to 4 % slower
// in the sampling, the price of 24 % on grids.
template <int D>
constexpr bool kBoxed = (D >= 10 && D <= 12) || D >= 17;

// Whole numbers in the order of the floats: a warp's extremes take one reduction
// instead of ten shuffles and minima (0.5 to 1 % where a tile has 256 draws).
__device__ __forceinline__ int order_key(float x) {
    const int b = __float_as_int(x);
    return b ^ (b >> 31 & 0x7fffffff);
}
__device__ __forceinline__ float order_value(int k) { return __int_as_float(k ^ (k >> 31 & 0x7fffffff)); }

// A warp holds a word of 32 designs in each of its DPT slots.  For a word and a
// draw let L = min_i (min_j t_ji - y_i) and U = min_i (max_j t_ji - y_i) over the
// box of the word's thresholds.  FP32 subtraction is monotone, so every design's
// smallest difference lies in [L, U], and with w the half-width of the
// sigmoid's window (0 without the sigmoid sums)
//   L >= w    no design is hit or in its window: the draw adds nothing;
//   U < -w    every design is hit and none in its window: z goes to all sums A;
//   else      the draw is tested design by design, as test_draws does.
// Each lane decides one of 32 draws, and the draws left are taken in order, so
// every sum has the terms and the order of test_draws, bit for bit.
// A NaN threshold counts as +inf in the maxima only (and drops out of the
// minima), which keeps the bounds valid for the other designs.
template <int D, int DPT>
__device__ __forceinline__ void word_boxes(const float (&t)[DPT][D], const int (&dsg)[DPT], float* box) {
    constexpr int DP = SharedShape<D, true>::kDP;
#pragma unroll
    for (int q = 0; q < DPT; ++q) {
#pragma unroll
        for (int i = 0; i < D; ++i) {
            const bool nan = t[q][i] != t[q][i];
            const int lo = __reduce_min_sync(0xffffffffu, dsg[q] >= 0 && !nan ? order_key(t[q][i]) : order_key(INFINITY));
            const int hi = __reduce_max_sync(0xffffffffu, dsg[q] >= 0 ? order_key(nan ? INFINITY : t[q][i]) : order_key(-INFINITY));
            if ((threadIdx.x & 31) == 0) {
                box[2 * q * DP + i] = order_value(lo);
                box[(2 * q + 1) * DP + i] = order_value(hi);
            }
        }
    }
}

// Smallest difference of a row of thresholds and a draw.
template <int D, int DP>
__device__ __forceinline__ float least(const float* __restrict__ row, const float (&y)[DP]) {
    float v[DP], m = INFINITY;
    load_row<DP>(row, v);
#pragma unroll
    for (int i = 0; i < D; i += 2) m = i + 1 < D ? fmin3(m, v[i] - y[i], v[i + 1] - y[i + 1]) : fminf(m, v[i] - y[i]);
    return m;
}

// The batch's draws against this thread's first nq designs.
template <int D, int DPT>
__device__ __forceinline__ void box_draws(const float* sy, const float* sz, int nb, int nq, const float* box,
                                          const float (&t)[DPT][D], float nhl2e, float wsk, uint32_t (&cnt)[DPT],
                                          float (&A)[DPT][SharedShape<D, true>::kDA],
                                          GSums<D, DPT, SharedShape<D, true>::kWide>& G) {
    constexpr int DP = SharedShape<D, true>::kDP;
    constexpr int DA = SharedShape<D, true>::kDA;
    static_assert(DPT == 1, "one design per thread");
    // At d = 18 the differences are formed again where the sigmoid needs them: kept,
    // they cost 172 bytes of spills more than the direct kernel has (grids 1.06 -> 1.10
    // of its speed, scattered designs 0.975 -> 0.99).  At d = 10..12, 17, 19 and 20 keeping them
    // measured 1 to 3 % faster on grids.
    constexpr bool kAgain = D == 18;
    const float w = fmaxf(wsk, 0.0f);
    for (int d0 = 0; d0 < nb; d0 += 32) {             // rows up to kBD exist: past nb they hold y = -inf
        uint32_t ev[DPT], in[DPT];
        int left = 0;
        {
            float y[DP];
            load_row<DP>(sy + (d0 + (threadIdx.x & 31)) * DP, y);
#pragma unroll
            for (int q = 0; q < DPT; ++q) {
                ev[q] = in[q] = 0u;
                if (q < nq) {
                    const float L = least<D, DP>(box + 2 * q * DP, y), U = least<D, DP>(box + (2 * q + 1) * DP, y);
                    const bool far = L >= w, all = U < -w;
                    in[q] = __ballot_sync(0xffffffffu, all && !far);
                    ev[q] = __ballot_sync(0xffffffffu, !all && !far);
                    left += __popc(ev[q]);
                }
            }
        }
        if (left > 16 * nq) {                          // scattered thresholds: the batch's rest draw by draw
            test_draws<D, true, DPT, DPT>(sy + d0 * DP, sz + d0 * DP, nb - d0, t, nhl2e, wsk, cnt, A, G);
            return;
        }
#pragma unroll
        for (int q = 0; q < DPT; ++q) {
            for (uint32_t m = ev[q] | in[q]; m; m &= m - 1u) {
                const int b = __ffs(m) - 1;
                float zz[DP];
                load_row<DP>(sz + (d0 + b) * DP, zz);
                bool hit = true;
                float dif[D], dmin = 0.0f;
                const bool test = ev[q] >> b & 1u;      // warp-uniform
                if (test) {
                    float y[DP], v[D];
                    load_row<DP>(sy + (d0 + b) * DP, y);
                    diffs<D>(t[q], y, v);
                    dmin = v[0];
#pragma unroll
                    for (int i = 1; i < D; i += 2) dmin = i + 1 < D ? fmin3(dmin, v[i], v[i + 1]) : fminf(dmin, v[i]);
                    hit = dmin < 0.0f;
                    if constexpr (!kAgain) {
#pragma unroll
                        for (int i = 0; i < D; ++i) dif[i] = v[i];
                    }
                }
                if constexpr (!SharedShape<D, true>::kCnt) cnt[q] += hit ? 1u : 0u;
                if (hit) {
#pragma unroll
                    for (int i = 0; i + 1 < DA; i += 2) {
                        const float2 a = __fadd2_rn(make_float2(A[q][i], A[q][i + 1]), make_float2(zz[i], zz[i + 1]));
                        A[q][i] = a.x;
                        A[q][i + 1] = a.y;
                    }
                    if constexpr (DA % 2 != 0) A[q][DA - 1] = __fadd_rn(A[q][DA - 1], zz[DA - 1]);
                }
                if (test && __any_sync(0xffffffffu, fabsf(dmin) < wsk)) {
                    if constexpr (kAgain) {
                        float y[DP];
                        load_row<DP>(sy + (d0 + b) * DP, y);
                        diffs<D>(t[q], y, dif);
                    }
                    float keep[D], prod = 1.0f;
                    const float2 nh2 = make_float2(nhl2e, nhl2e), one2 = make_float2(1.0f, 1.0f);
#pragma unroll
                    for (int i = 0; i + 1 < D; i += 2) {
                        const float2 x = __fmul2_rn(make_float2(dif[i], dif[i + 1]), nh2);
                        const float2 u = __fadd2_rn(one2, make_float2(ex2_approx(x.x), ex2_approx(x.y)));
                        keep[i] = rcp_approx(u.x);
                        keep[i + 1] = rcp_approx(u.y);
                    }
                    if constexpr (D % 2 != 0) keep[D - 1] = rcp_approx(1.0f + ex2_approx(dif[D - 1] * nhl2e));
#pragma unroll
                    for (int i = 0; i < D; ++i) prod *= keep[i];
                    const float2 pr2 = make_float2(prod, prod), m1 = make_float2(-1.0f, -1.0f);
#pragma unroll
                    for (int i = 0; i + 1 < D; i += 2) {
                        const float2 omk = __ffma2_rn(make_float2(keep[i], keep[i + 1]), m1, one2);
                        const float2 g = __ffma2_rn(pr2, omk, make_float2(G(q, i), G(q, i + 1)));
                        G(q, i) = g.x;
                        G(q, i + 1) = g.y;
                    }
                    if constexpr (D % 2 != 0) G(q, D - 1) = fmadd(prod, 1.0f - keep[D - 1], G(q, D - 1));
                }
            }
        }
    }
}

// The persistent loop over the tiles of shared draws.
template <int D>
__device__ __forceinline__ void box_body(const SampleParams& P, const SharedTile* __restrict__ tiles,
                                            const uint32_t* __restrict__ list) {
    using S = Shape<D>;
    using SS = SharedShape<D, true>;
    constexpr int DPT = SS::kDpt, DP = SS::kDP;
    extern __shared__ __align__(16) float sh[];
    float* sy = sh;                                   // [kBD][kDP]
    float* sz = sh + SS::kBD * DP;                    // [kBD][kDP]
    __shared__ __align__(16) float sL[LPad<float>::rowoff(D) + 4];
    __shared__ float sB[kMaxWarps][D];
    __shared__ unsigned int s_tile;
    __shared__ __align__(16) float sbox[kSharedThreads / 32][2 * DPT * DP];
    float* box = sbox[threadIdx.x >> 5];              // this warp's words: minima and maxima
    __shared__ float sGw[SS::kWide ? kSharedThreads * DPT * D : 1];   // G slots (kWide)

    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(P.ticket, 1u);
        __syncthreads();
        const unsigned int tk = s_tile;
        if (static_cast<int64_t>(tk) >= P.n_tiles) break;
        const SharedTile tl = tiles[tk];
        const int ok = P.scen_ok[tl.scen];
        const int64_t loff = P.L_off[tl.scen];
        for (int r = threadIdx.x; r < D; r += blockDim.x) {
            const int po = LPad<float>::rowoff(r), pk = r * (r + 1) / 2;
            for (int q = 0; q < LPad<float>::chunks(r) * LPad<float>::V; ++q)
                sL[po + q] = q <= r ? P.L32[loff + pk + q] : 0.0f;
        }
        // this thread's designs (list positions threadIdx.x + q * blockDim.x)
        // and their thresholds; a missing design gets t = +inf (never a hit)
        const int nq = static_cast<int>((tl.list_cnt + blockDim.x - 1) / blockDim.x);   // block-uniform
        int dsg[DPT];
        float t[DPT][D];
#pragma unroll
        for (int q = 0; q < DPT; ++q) {
            const uint32_t li = threadIdx.x + q * blockDim.x;
            dsg[q] = li < tl.list_cnt ? static_cast<int>(list[tl.list_off + li]) : -1;
            const int64_t vo = dsg[q] >= 0 ? P.designs[dsg[q]].vec_off : 0;
#pragma unroll
            for (int i = 0; i < D; ++i) {
                const double tt = dsg[q] >= 0 ? P.b[vo + i] - P.mu[vo + i] : 0.0;
                if (dsg[q] >= 0 && tt != tt) set_status(P.status, MCD_ENAN, dsg[q]);
                t[q][i] = dsg[q] >= 0 ? static_cast<float>(tt) : INFINITY;
            }
        }
        word_boxes<D, DPT>(t, dsg, box);
        __syncthreads();                              // sL and the boxes complete
        if (!ok) continue;                            // block-uniform; the next ticket read is behind a barrier

        const uint64_t g_first = tl.start / S::kG;
        const uint32_t ofs = static_cast<uint32_t>(tl.start - g_first * S::kG);
        const uint32_t ngroups = (ofs + tl.n + S::kG - 1) / S::kG;
        const uint64_t call_first = g_first * static_cast<uint64_t>(S::kNC);
        const uint64_t call_last = (g_first + ngroups) * static_cast<uint64_t>(S::kNC) - 1;
        const bool fast = (call_first >> 32) == (call_last >> 32);
        // the sigmoid's exponent scale -log2(e)/h, and the half-width
        // 25.03 h / log2(e) of the window of differences in which its work
        // is taken (box_draws; -1 when the sigmoid sums are off)
        const float nhl2e = -P.hinv_log2e;
        const float wsk = P.sig_skip_w;
        const Round1 r1 = round1_consts(static_cast<uint32_t>(call_first >> 32), tl.key, P.rk0, P.rk1);

        uint32_t cnt[DPT];
        float A[DPT][SS::kDA], bsum[D];
        GSums<D, DPT, SS::kWide> G;
        G.s = sGw + threadIdx.x;
#pragma unroll
        for (int q = 0; q < DPT; ++q) {
            cnt[q] = 0;
#pragma unroll
            for (int i = 0; i < SS::kDA; ++i) A[q][i] = 0.0f;
#pragma unroll
            for (int i = 0; i < D; ++i)
                G(q, i) = 0.0f;
        }
#pragma unroll
        for (int i = 0; i < D; ++i) bsum[i] = 0.0f;

        for (uint32_t g0 = 0; g0 < ngroups; g0 += blockDim.x) {
            const uint32_t gi = g0 + threadIdx.x;
            make_batch<D, true>(sL, call_first + static_cast<uint64_t>(gi) * S::kNC,
                                static_cast<uint32_t>(call_first) + gi * S::kNC, fast, r1, tl.key, P,
                                gi * S::kG, ofs, gi < ngroups ? tl.n : 0u, sy, sz, bsum);
            __syncthreads();
            const int nb = static_cast<int>(min(static_cast<uint32_t>(SS::kBD), (ngroups - g0) * S::kG));
            box_draws<D, DPT>(sy, sz, nb, nq, box, t, nhl2e, wsk, cnt, A, G);
            __syncthreads();                          // the next batch rewrites sy / sz
        }

        // hits: each design of the tile belongs to exactly one thread
        if constexpr (SS::kCnt) {
#pragma unroll
            for (int q = 0; q < DPT; ++q) cnt[q] = static_cast<uint32_t>(A[q][D]);
        }
#pragma unroll
        for (int q = 0; q < DPT; ++q)
            if (dsg[q] >= 0 && cnt[q]) atomicAdd(&P.hits[dsg[q]], static_cast<unsigned long long>(cnt[q]));
        {
            // the sum of z over the tile's draws is common to all its designs
            const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
            for (int i = 0; i < D; ++i) {
                const float w = warp_sum(bsum[i]);
                if (lane == 0) sB[warp][i] = w;
            }
            __syncthreads();
            const double fix = static_cast<double>(1ull << kGradFixBits);
#pragma unroll
            for (int q = 0; q < DPT; ++q) {
                if (dsg[q] < 0) continue;
                unsigned long long* slot = P.gacc + P.designs[dsg[q]].acc_off + static_cast<int64_t>(tl.batch) * 3 * D;
#pragma unroll
                for (int i = 0; i < D; ++i) {
                    double s = 0.0;
                    for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) s += static_cast<double>(sB[w][i]);
                    atomicAdd(slot + i, static_cast<unsigned long long>(__double2ll_rn(static_cast<double>(A[q][i]) * fix)));
                    atomicAdd(slot + D + i, static_cast<unsigned long long>(__double2ll_rn(s * fix)));
                    atomicAdd(slot + 2 * D + i, static_cast<unsigned long long>(__double2ll_rn(static_cast<double>(G(q, i)) * fix)));
                }
            }
        }
        // the next iteration's ticket read sits behind a barrier, so sB and
        // the per-tile shared state are not overwritten early
    }
}

// Two resident blocks per SM, one at odd d from 17 on, whose batches take more than
// half of the shared memory.
template <int D>
__global__ void __launch_bounds__(kSharedThreads, D <= 12 || D % 2 == 0 ? 2 : 1)
box_kernel(const __grid_constant__ SampleParams P, const SharedTile* __restrict__ tiles,
           const uint32_t* __restrict__ list) {
    box_body<D>(P, tiles, list);
}

template <int D>
const void* box_fn() {
    if constexpr (kBoxed<D>) return reinterpret_cast<const void*>(&box_kernel<D>);
    else return shared_fn<D, true>();
}

}  // namespace mcd
