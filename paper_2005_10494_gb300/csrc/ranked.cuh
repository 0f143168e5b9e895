// Ranked shared-draw sampling: hit counts of common-random-number groups from
// threshold ranks instead of one comparison per design, draw and coordinate.
//
// The designs of a group see the same draws, and design j is hit by draw n
// exactly when y_i > t_ji for some coordinate i.  For one coordinate the
// designs that a draw exceeds are the designs of the rank(y_i) smallest
// thresholds: a prefix of the designs sorted by t_.i.  So a draw is reduced to
// d ranks, made once per family (up to rank_family(d) designs of a group),
// and a block that owns a chunk of 32 W designs holds, per coordinate, the
// designs of every prefix as a row of W bit words in shared memory.  The hits
// of one draw on 32 designs are then the or of d words: 1/32 of an operation
// per design and coordinate.  Ranks come from FP32 comparisons of the same y
// and t as the other kernels', so the counts are bit-identical to them.
//
// Three kernels, queued per batch of families and draws:
//   rank_sort_kernel   a block per family and coordinate sorts the thresholds
//                      t = b - mu (read at every launch), and writes the
//                      distinct values and each design's position among them;
//   rank_draws_kernel  makes the draws (the Philox, Box-Muller and transform
//                      arithmetic of sample.cuh) and finds each coordinate's
//                      rank by a branch-free binary search in shared memory;
//   rank_count_kernel  a block builds its chunk's rows and adds the or-ed
//                      words of its draws into bit-sliced counters.
//
// Measured on a d=3 grid (4 scenarios x 4096 designs x 1e6 draws): sort 30 us,
// draws 51 us, count 328 us; the kernel that tests every design against every
// draw takes 2.53 ms.  The count kernel is bound by shared memory (19 wavefronts
// a warp step of 8 draws x 512 designs, 65 % of the pipe busy) and the latency
// of its loads at 16 warps per SM; 24 or 20 warps (768, 640 threads) need the
// counters in fewer planes and spill, and measured the same or 6 % slower.
#pragma once

#include <cstdint>

#include "ranked_api.cuh"
#include "rng.cuh"
#include "sample.cuh"

namespace mcd {


// Ranks of one draw are stored as u16, padded to whole 8-byte vectors.
__host__ __device__ constexpr int rank_pad(int d) { return (d + 3) / 4 * 4; }

// ---- threshold ranks --------------------------------------------------------

// Per family and coordinate: distinct finite thresholds ascending (the rest
// +inf), their number, and per design the position of its threshold
// (kRankNone: +inf or NaN, exceeded by no draw).
constexpr uint16_t kRankNone = 0xffffu;

__device__ __forceinline__ uint32_t order_float(float f) {
    const uint32_t u = __float_as_uint(f);
    return (u >> 31) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float unorder_float(uint32_t k) {
    return __uint_as_float((k >> 31) ? (k & 0x7fffffffu) : ~k);
}

// ---- rows of a chunk ----------------------------------------------------------

// Layout of a chunk's rows for dimension D and W words per row.  A shared
// memory line of 128 bytes holds the rows of S = 32 / W coordinates; eight
// lanes (one phase of a 16-byte load) cover S draws, and draw slot s takes the
// coordinates of a line group rotated by s, so that the S draws read
// different columns of their lines and the phase has no bank conflict.  A
// group of m < S coordinates repeats them over the columns (conflict-free
// when m divides S).
template <int D, int W>
struct RankRows {
    static constexpr int S = 32 / W;                       // coordinates per line, draws per load phase
    static constexpr int kGroups = (D + S - 1) / S;        // line groups
    static constexpr int C = 32 * W;                       // designs of a chunk
    static constexpr int kLines = C + 1;                   // prefixes 0..C
    static constexpr int kDR = rank_pad(D);
    static constexpr int LPR = W / 4;                      // lanes per draw (16 bytes each)
    static constexpr int kThreads = 512;
    static constexpr int kWarps = kThreads / 32;
    static constexpr int kStep = kWarps * 32 / LPR;        // draws of one step of the block
    static constexpr int kSteps = (D <= 3 && W == 16) ? 16 : D <= 4 ? 8 : D <= 10 ? 4 : 2;
    static constexpr int kBatch = kStep * kSteps;          // draws of one batch
    static constexpr int kPer = kBatch / kThreads;     // draws a thread maps per batch
    static constexpr int kPlanes = W == 4 ? 11 : 12;       // bits of a lane's counters
    static constexpr int kSegRows = 32;                    // rows per segment of the prefix pass
    static constexpr int kSegs = (kLines + kSegRows - 1) / kSegRows;
    __host__ __device__ static constexpr int members(int g) { return D - g * S < S ? D - g * S : S; }
    // shared memory (bytes): rows | presence | offsets | counters | segment totals
    __host__ __device__ static constexpr size_t rows_bytes() { return static_cast<size_t>(kGroups) * kLines * 128; }
    static constexpr size_t smem() {        // without the presence words, D (fam_cap / 32 + 1) of 8 bytes
        return rows_bytes() + static_cast<size_t>(kBatch) * kDR * 4 + static_cast<size_t>(C) * 4 +
               static_cast<size_t>(kGroups) * kSegs * 128;
    }
};

// One draw's word of hits on a lane's 4 x 32 designs.
struct Word4 {
    uint32_t w[4];
};

template <int D, int W>
__device__ __forceinline__ void build_rows(const RankParams& R, int fam, int chunk, uint32_t* rows, uint2* pres,
                                           uint32_t* tot) {
    using RR = RankRows<D, W>;
    const int fw = R.fam_cap / 32 + 1;
    const int cnt = R.fams[fam].cnt;
    const int j0 = chunk * RR::C;
    const int nj = min(RR::C, cnt - j0);
    const int tid = threadIdx.x;
    for (int q = tid; q < RR::kGroups * RR::kLines * 8; q += RR::kThreads)
        reinterpret_cast<uint4*>(rows)[q] = make_uint4(0u, 0u, 0u, 0u);
    for (int q = tid; q < D * fw; q += RR::kThreads) pres[q] = make_uint2(0u, 0u);
    __syncthreads();
    const uint16_t* pos = R.pos + static_cast<int64_t>(fam - R.fam0) * D * R.fam_cap + j0;
    for (int q = tid; q < D * RR::C; q += RR::kThreads) {
        const int i = q / RR::C, j = q % RR::C;
        if (j < nj) {
            const uint32_t r = pos[static_cast<int64_t>(i) * R.fam_cap + j];
            if (r != kRankNone) atomicOr(&pres[i * fw + (r >> 5)].x, 1u << (r & 31));
        }
    }
    __syncthreads();
    // running number of present thresholds before each word: a warp per coordinate
    for (int i = tid >> 5; i < D; i += RR::kThreads / 32) {
        const int lane = tid & 31;
        uint32_t base = 0;
        for (int w0 = 0; w0 < fw; w0 += 32) {
            const int w = w0 + lane;
            const uint32_t c = w < fw ? __popc(pres[i * fw + w].x) : 0u;
            uint32_t s = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t v = __shfl_up_sync(0xffffffffu, s, o);
                if (lane >= o) s += v;
            }
            if (w < fw) pres[i * fw + w].y = base + s - c;
            base += __shfl_sync(0xffffffffu, s, 31);
        }
    }
    __syncthreads();
    // design j enters every prefix longer than its local rank: its bit goes
    // into row (local rank + 1), and the prefix pass carries it upwards
    for (int q = tid; q < D * RR::C; q += RR::kThreads) {
        const int i = q / RR::C, j = q % RR::C;
        if (j < nj) {
            const uint32_t r = pos[static_cast<int64_t>(i) * R.fam_cap + j];
            if (r != kRankNone) {
                const uint2 pw = pres[i * fw + (r >> 5)];
                const uint32_t l = pw.y + __popc(pw.x & ((1u << (r & 31)) - 1u)) + 1u;
                const int g = i / RR::S, m = D - g * RR::S < RR::S ? D - g * RR::S : RR::S;
                for (int col = i - g * RR::S; col < RR::S; col += m)
                    atomicOr(&rows[(static_cast<uint32_t>(g) * RR::kLines + l) * 32 + col * W + (j >> 5)], 1u << (j & 31));
            }
        }
    }
    __syncthreads();
    constexpr int kJobs = RR::kGroups * RR::kSegs * 32;
    for (int q = tid; q < kJobs; q += RR::kThreads) {
        const int w = q & 31, sg = (q >> 5) % RR::kSegs, g = (q >> 5) / RR::kSegs;
        uint32_t* p = rows + (static_cast<uint32_t>(g) * RR::kLines + sg * RR::kSegRows) * 32 + w;
        const int n = min(RR::kSegRows, RR::kLines - sg * RR::kSegRows);
        uint32_t acc = 0u;
        for (int l = 0; l < n; ++l) {
            acc |= p[l * 32];
            p[l * 32] = acc;
        }
        tot[q] = acc;
    }
    __syncthreads();
    for (int q = tid; q < kJobs; q += RR::kThreads) {
        const int w = q & 31, sg = (q >> 5) % RR::kSegs, g = (q >> 5) / RR::kSegs;
        uint32_t before = 0u;
        for (int s = 0; s < sg; ++s) before |= tot[(g * RR::kSegs + s) * 32 + w];
        if (before) {
            uint32_t* p = rows + (static_cast<uint32_t>(g) * RR::kLines + sg * RR::kSegRows) * 32 + w;
            const int n = min(RR::kSegRows, RR::kLines - sg * RR::kSegRows);
            for (int l = 0; l < n; ++l) p[l * 32] |= before;
        }
    }
    __syncthreads();
}

// Row offsets (units of 16 bytes) of one draw's D ranks, in the order in
// which draw slot s reads them.
template <int D, int W>
__device__ __forceinline__ void map_draw(const uint16_t (&rk)[RankRows<D, W>::kDR], const uint2* pres, int fw, int s,
                                         uint16_t* off) {
    using RR = RankRows<D, W>;
#pragma unroll
    for (int i = 0; i < D; ++i) {
        const uint32_t r = rk[i];
        const uint2 pw = pres[i * fw + (r >> 5)];
        const uint32_t l = pw.y + __popc(pw.x & ((1u << (r & 31)) - 1u));
        constexpr int S = RR::S;
        const int g = i / S, a = i - g * S;
        const int m = RR::members(g);
        // position c with (c + s) mod m = a, in the repeat of the group that slot s owns
        const int sm = s % m, rep = s / m * m;
        const int c = a >= sm ? a - sm : a - sm + m;
        const int col = (rep + m <= S ? rep : 0) + a;
        off[g * S + c] = static_cast<uint16_t>((g * RR::kLines + l) * 8 + col * (W / 4));
    }
}

// The or of a draw's D rows: this lane's 16 bytes (`part` of the row) of each.
template <int D, int W>
__device__ __forceinline__ Word4 or_rows(const uint4* rows, uint32_t part2, const uint16_t* off) {
    using RR = RankRows<D, W>;
    Word4 h;
#pragma unroll
    for (int q = 0; q < RR::kDR / 4; ++q) {
        uint2 o = *reinterpret_cast<const uint2*>(off + 4 * q);
        o.x += part2;                                     // both 16-bit offsets (no carry: offsets stay below 2^16)
        o.y += part2;
        const uint32_t ob[4] = {o.x & 0xffffu, o.x >> 16, o.y & 0xffffu, o.y >> 16};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (4 * q + e < D) {
                const uint4 v = rows[ob[e]];
                if (q == 0 && e == 0) {
                    h.w[0] = v.x; h.w[1] = v.y; h.w[2] = v.z; h.w[3] = v.w;
                } else {
                    h.w[0] |= v.x; h.w[1] |= v.y; h.w[2] |= v.z; h.w[3] |= v.w;
                }
            }
        }
    }
    return h;
}

// (s, c) = a + b + c_in bitwise: sum and carry of three one-bit planes.
__device__ __forceinline__ void csa(uint32_t& s, uint32_t a, uint32_t b, uint32_t& carry) {
    const uint32_t u = s;
    s = u ^ a ^ b;
    carry = (u & a) | (u & b) | (a & b);
}

// Add one plane of weight 2^K0 into the bit-sliced counters.
template <int K0, int P>
__device__ __forceinline__ void ripple(uint32_t (&pl)[P], uint32_t c) {
#pragma unroll
    for (int k = K0; k < P; ++k) {
        const uint32_t n = pl[k] & c;
        pl[k] ^= c;
        c = n;
    }
}

// Add the lanes' bit-sliced counters to the chunk's u32 counters in shared
// memory: planes to 16-bit counts two designs per register, summed over the
// lanes that hold the same words, then one atomic per design and warp.
template <int W, int P>
__device__ __forceinline__ void flush_planes(uint32_t (&pl)[4][P], uint32_t* cnt) {
    constexpr int LPR = W / 4, LANES = 32 / LPR;
    const int lane = threadIdx.x & 31, part = lane % LPR, slot = lane / LPR;
    int item = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
#pragma unroll
        for (int b = 0; b < 16; ++b) {
            // designs b and b + 16 of word q
            uint32_t v = 0u;
#pragma unroll
            for (int k = 0; k < P; ++k) v |= ((pl[q][k] >> b) & 0x00010001u) << k;
#pragma unroll
            for (int o = LPR; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (slot == item % LANES) {
                const int j = (part * 4 + q) * 32 + b;
                if (v & 0xffffu) atomicAdd(&cnt[j], v & 0xffffu);
                if (v >> 16) atomicAdd(&cnt[j + 16], v >> 16);
            }
            ++item;
        }
#pragma unroll
        for (int k = 0; k < P; ++k) pl[q][k] = 0u;
    }
}

template <int D, int W>
__global__ void __launch_bounds__(RankRows<D, W>::kThreads, 1) rank_count_kernel(const __grid_constant__ RankParams R) {
    using RR = RankRows<D, W>;
    constexpr int P = RR::kPlanes, DR = RR::kDR;
    extern __shared__ __align__(128) unsigned char sh_rank[];
    const int fw = R.fam_cap / 32 + 1;
    uint32_t* rows = reinterpret_cast<uint32_t*>(sh_rank);
    uint2* pres = reinterpret_cast<uint2*>(sh_rank + RR::rows_bytes());
    uint16_t* off = reinterpret_cast<uint16_t*>(pres + D * fw);
    uint32_t* cnt = reinterpret_cast<uint32_t*>(off + 2 * RR::kBatch * DR);
    uint32_t* tot = cnt + RR::C;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int part = lane % RR::LPR, slot = lane / RR::LPR;
    const uint4* rows4 = reinterpret_cast<const uint4*>(sh_rank);
    const uint32_t part2 = static_cast<uint32_t>(part) * 0x00010001u;

    // this block's share of the launch's (chunk, draws) batches, in order
    const int64_t u0 = R.n_units * blockIdx.x / gridDim.x, u1 = R.n_units * (blockIdx.x + 1) / gridDim.x;
    if (u0 >= u1) return;
    int it = R.item0;
    {
        int lo = R.item0, hi = R.item1 - 1;               // last item with unit0 <= u0
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (R.items[mid].unit0 <= u0) lo = mid;
            else hi = mid - 1;
        }
        it = lo;
    }
    uint32_t pl[4][P];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int k = 0; k < P; ++k) pl[q][k] = 0u;

    int64_t u = u0;
    int cur_fam = -1, cur_chunk = -1;
    int filled = 0;                                       // draws added to each lane's counters
    while (u < u1) {
        const RankItem im = R.items[it];
        const RankSeg sg = R.segs[im.seg];
        const int64_t item_end = it + 1 < R.item1 ? R.items[it + 1].unit0 : R.n_units;
        const int64_t ue = item_end < u1 ? item_end : u1;
        if (!R.scen_ok[R.fams[sg.fam].scen]) {            // factorisation failed: no hits
            u = ue;
            ++it;
            continue;
        }
        if (sg.fam != cur_fam || im.chunk != cur_chunk) {
            __syncthreads();
            build_rows<D, W>(R, sg.fam, im.chunk, rows, pres, tot);
            for (int q = tid; q < RR::C; q += RR::kThreads) cnt[q] = 0u;
            cur_fam = sg.fam;
            cur_chunk = im.chunk;
        }
        const uint16_t* rk = R.ranks + static_cast<int64_t>(sg.ws_off) * DR;
        uint2 nx[RR::kPer][DR / 4];
        auto fetch = [&](int64_t uu) {
            const uint32_t n0 = static_cast<uint32_t>((uu - im.unit0) * RR::kBatch);
#pragma unroll
            for (int q = 0; q < RR::kPer; ++q) {
                const uint32_t n = n0 + q * RR::kThreads + tid;
#pragma unroll
                for (int v = 0; v < DR / 4; ++v)
                    nx[q][v] = n < sg.n ? __ldg(reinterpret_cast<const uint2*>(rk + static_cast<int64_t>(n) * DR) + v)
                                        : make_uint2(0u, 0u);
            }
        };
        auto map = [&](uint16_t* dst) {
#pragma unroll
            for (int q = 0; q < RR::kPer; ++q) {
                uint16_t r[DR];
#pragma unroll
                for (int v = 0; v < DR / 4; ++v) {
                    r[4 * v] = static_cast<uint16_t>(nx[q][v].x); r[4 * v + 1] = static_cast<uint16_t>(nx[q][v].x >> 16);
                    r[4 * v + 2] = static_cast<uint16_t>(nx[q][v].y); r[4 * v + 3] = static_cast<uint16_t>(nx[q][v].y >> 16);
                }
                const int n = q * RR::kThreads + tid;
                map_draw<D, W>(r, pres, fw, n % RR::S, dst + n * DR);
            }
        };
        // offsets are double-buffered: a batch's words are read while the
        // next batch's offsets are written and the one after is loaded
        int buf = 0;
        __syncthreads();                                  // the previous item's offsets are read
        fetch(u);
        map(off);
        if (u + 1 < ue) fetch(u + 1);
        __syncthreads();
        for (; u < ue; ++u) {
            const uint16_t* po = off + buf * RR::kBatch * DR + (warp * (32 / RR::LPR) + slot) * DR;
            buf ^= 1;
            if (u + 1 < ue) map(off + buf * RR::kBatch * DR);
            if (u + 2 < ue) fetch(u + 2);
            // carries of 2, 4, .. kSteps draws, then the rest of the planes
            uint32_t c1[4], c2[4], c3[4];
#pragma unroll
            for (int st = 0; st < RR::kSteps; st += 2) {
                const Word4 a = or_rows<D, W>(rows4, part2, po + st * RR::kStep * DR);
                const Word4 b = or_rows<D, W>(rows4, part2, po + (st + 1) * RR::kStep * DR);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    uint32_t t1;
                    csa(pl[q][0], a.w[q], b.w[q], t1);
                    if (RR::kSteps == 2) { ripple<1, P>(pl[q], t1); continue; }
                    if (!(st & 2)) { c1[q] = t1; continue; }
                    uint32_t t2;
                    csa(pl[q][1], c1[q], t1, t2);
                    if (RR::kSteps == 4) { ripple<2, P>(pl[q], t2); continue; }
                    if (!(st & 4)) { c2[q] = t2; continue; }
                    uint32_t t3;
                    csa(pl[q][2], c2[q], t2, t3);
                    if (RR::kSteps == 8) { ripple<3, P>(pl[q], t3); continue; }
                    if (!(st & 8)) { c3[q] = t3; continue; }
                    uint32_t t4;
                    csa(pl[q][3], c3[q], t3, t4);
                    ripple<4, P>(pl[q], t4);
                }
            }
            __syncthreads();
            filled += RR::kSteps;
            if (filled + RR::kSteps >= (1 << P)) {
                flush_planes<W, P>(pl, cnt);
                filled = 0;
            }
        }
        // leaving the chunk (or done): counters to the designs' hit counts
        const bool same = u < u1 && it + 1 < R.item1 && R.items[it + 1].chunk == im.chunk &&
                          R.segs[R.items[it + 1].seg].fam == sg.fam;
        ++it;
        if (!same) {
            flush_planes<W, P>(pl, cnt);
            filled = 0;
            __syncthreads();
            const RankFam fm = R.fams[sg.fam];
            for (int q = tid; q < RR::C; q += RR::kThreads) {
                const int j = im.chunk * RR::C + q;
                if (j < fm.cnt && cnt[q]) atomicAdd(&R.hits[R.list[fm.list_off + j]], static_cast<unsigned long long>(cnt[q]));
            }
            cur_fam = -1;
        }
    }
}

// ---- draws ---------------------------------------------------------------------

// A block takes tiles of kRankDrawThreads groups of draws of the launch's
// segments; a thread makes one group, the ranks of its draws one level of the
// D searches after the other (independent chains hide the load latency).
// A family's distinct thresholds lie in shared memory as the levels of a
// search tree, node v's children at 2 v and 2 v + 1, so that the upper levels,
// which all lanes visit, take neighbouring banks (sorted order put them a
// power of two apart: 80 % of the kernel's shared wavefronts were conflicts).
// Node 0 holds the one value that a tree of 2^levels - 1 nodes leaves out.
template <int D>
__global__ void __launch_bounds__(kRankDrawThreads, D <= 6 ? 2 : 1) rank_draws_kernel(const __grid_constant__ RankParams R) {
    using S = Shape<D>;
    constexpr int DR = rank_pad(D);
    extern __shared__ __align__(16) float sh_u[];         // [D][2^levels] search trees
    __shared__ __align__(16) float sL[LPad<float>::rowoff(D) + 4];
    const int64_t t0 = R.n_tiles * blockIdx.x / gridDim.x, t1 = R.n_tiles * (blockIdx.x + 1) / gridDim.x;
    if (t0 >= t1) return;
    int sgi = R.seg0;
    {
        int lo = R.seg0, hi = R.seg1 - 1;                 // last segment with tile0 <= t0
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (R.segs[mid].tile0 <= t0) lo = mid;
            else hi = mid - 1;
        }
        sgi = lo;
    }
    int cur_fam = -1, levels = 0;
    for (int64_t t = t0; t < t1; ++sgi) {
        const RankSeg sg = R.segs[sgi];
        const RankFam fm = R.fams[sg.fam];
        const int64_t seg_end = sgi + 1 < R.seg1 ? R.segs[sgi + 1].tile0 : R.n_tiles;
        const int64_t te = seg_end < t1 ? seg_end : t1;
        if (!R.scen_ok[fm.scen]) {                        // the count kernel skips the family too
            t = te;
            continue;
        }
        if (sg.fam != cur_fam) {
            __syncthreads();
            int umax = 1;
            for (int i = 0; i < D; ++i) umax = max(umax, R.n_distinct[(sg.fam - R.fam0) * D + i]);
            levels = 0;
            while ((1 << levels) < umax) ++levels;
            const int top = 1 << levels;                  // <= fam_cap
            const float* u = R.distinct + static_cast<int64_t>(sg.fam - R.fam0) * D * R.fam_cap;
            for (int q = threadIdx.x; q < D * top; q += kRankDrawThreads) {
                const int i = q >> levels, v = q & (top - 1);
                const int k = 31 - __clz(v | 1);          // level of node v
                const int at = v == 0 ? top - 1 : (2 * (v - (1 << k)) + 1) * (top >> (k + 1)) - 1;
                sh_u[q] = u[static_cast<int64_t>(i) * R.fam_cap + at];
            }
            const int64_t loff = R.L_off[fm.scen];
            for (int r = threadIdx.x; r < D; r += kRankDrawThreads) {
                const int po = LPad<float>::rowoff(r), pk = r * (r + 1) / 2;
                for (int q = 0; q < LPad<float>::chunks(r) * LPad<float>::V; ++q)
                    sL[po + q] = q <= r ? R.L32[loff + pk + q] : 0.0f;
            }
            cur_fam = sg.fam;
            __syncthreads();
        }
        const uint64_t g_first = sg.start / S::kG;
        const uint32_t ofs = static_cast<uint32_t>(sg.start - g_first * S::kG);
        const uint32_t ngroups = (ofs + sg.n + S::kG - 1) / S::kG;
        for (; t < te; ++t) {
            const uint32_t gi = static_cast<uint32_t>(t - sg.tile0) * kRankDrawThreads + threadIdx.x;
            if (gi >= ngroups) continue;
            const uint64_t call = (g_first + gi) * static_cast<uint64_t>(S::kNC);
            float z[S::kNZ];
#pragma unroll
            for (int g = 0; g < S::kG; ++g) {
                // the Philox calls whose normals draw g is the first to use
#pragma unroll
                for (int c = (g * D + 3) / 4; c < ((g + 1) * D + 3) / 4; ++c) {
                    const uint4 w = philox_full(call + c, fm.key, R.rk0, R.rk1);
                    normals4<float>(w, &z[4 * c]);
                }
                float y[D];
                uint32_t node[D];
#pragma unroll
                for (int i = 0; i < D; ++i) {
                    const int row = LPad<float>::rowoff(i);
                    float s = sL[row] * z[g * D];
#pragma unroll
                    for (int j = 1; j <= i; ++j) s = fmadd(sL[row + j], z[g * D + j], s);
                    y[i] = s;
                    node[i] = 1u;
                }
                for (int k = 0; k < levels; ++k) {
#pragma unroll
                    for (int i = 0; i < D; ++i)
                        node[i] = 2u * node[i] + (sh_u[(i << levels) + node[i]] < y[i] ? 1u : 0u);
                }
#pragma unroll
                for (int i = 0; i < D; ++i)
                    node[i] = node[i] - (1u << levels) + (sh_u[i << levels] < y[i] ? 1u : 0u);
                const uint32_t n = gi * S::kG + g - ofs;  // wraps for draws before the segment
                if (n < sg.n) {
                    uint2* out = reinterpret_cast<uint2*>(R.ranks + static_cast<int64_t>(sg.ws_off + n) * DR);
#pragma unroll
                    for (int v = 0; v < DR / 4; ++v) {
                        uint32_t p4[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) p4[e] = 4 * v + e < D ? node[4 * v + e < D ? 4 * v + e : 0] : 0u;
                        out[v] = make_uint2(p4[0] | (p4[1] << 16), p4[2] | (p4[3] << 16));
                    }
                }
            }
        }
    }
}

// The kernels of dimension D with `words` words per row.
struct RankKernels {
    const void* draws;
    const void* count;
    size_t count_rows;       // shared memory of the count kernel besides the presence words
    int batch;
    int threads;
};

template <int D, int W>
void rank_fill(RankKernels* k) {
    using RR = RankRows<D, W>;
    k->count = reinterpret_cast<const void*>(&rank_count_kernel<D, W>);
    k->count_rows = RR::smem();
    k->batch = RR::kBatch;
    k->threads = RR::kThreads;
}

template <int D>
const void* rank_kernels(int words, RankKernels* k) {
    k->draws = reinterpret_cast<const void*>(&rank_draws_kernel<D>);
    if (words == 4) rank_fill<D, 4>(k);
    else if (words == 8) rank_fill<D, 8>(k);
    else if constexpr (D <= 3) rank_fill<D, 16>(k);
    else return nullptr;
    return k->count;
}

}  // namespace mcd
