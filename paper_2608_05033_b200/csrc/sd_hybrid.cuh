// The hybrid family: light rows row-wise, heavy rows as chunks, all in one launch (the schedule of the paper's
// appendix listing, without its atomics).  A CTA takes one of three roles by its index:
//
//   items    chunks of the heavy rows (window-major) and rows of at least kHybridWide nonzeros, a group of 16 or 32
//            lanes each (launch_hybrid_one); LPR lanes of a group stand across the columns, its 16 / LPR or 32 / LPR
//            lane sets share the nonzeros, and their sums meet by xor shuffles.
//   medium   rows of kHybridMedium .. kHybridWide - 1 nonzeros, groups of at least eight lanes.
//   short    rows of fewer nonzeros, several per lane group (light_rows_body).
//
// What bounds it: on large matrices the rate at which L2 and L1 deliver gathered rows of B (64 bf16 columns, R-MAT scale
// 19, 16 M nonzeros: 181 us = 11.3 TB/s of rows of B; with pairs handed round by shuffle 207), on small ones the chain
// of dependent gathers of the longest item, which the lane sets cut (8 columns, 128 nonzeros: 64 steps of a pair of lanes
// before, 2 steps of a warp now; R-MAT scale 14: 51 -> 9 us).
#pragma once

#include <type_traits>

#include "sd_common.cuh"
#include "sd_group.cuh"

namespace sd {

constexpr int kHybridThreads = 256;

struct HybridArgs {
    const int32_t *colind;
    const void *vals;
    const void *B;
    float *C;
    float *scratch;          // [chunks][N]
    const int4 *items;       // chunks in the order they are taken, up to four at once: {scratch row, or row | bit 31; first nonzero; chunk; length}
    const int4 *desc;        // light rows, longest first: {row, first nonzero, its column, length}
    int64_t ldc;
    uint32_t ldb_bytes;
    int32_t N;
    int32_t chunks;          // work items of the first role: chunks, then the first `wide` entries of desc
    int32_t wide;
    int32_t medium;          // entries wide .. wide + medium - 1 of desc
    int32_t light;           // entries wide + medium .. wide + medium + light - 1
    uint32_t gc, gm;         // CTAs of the first and the second role
    float alpha, beta;
};

template <typename T, int VW, int LPR, int NV, int LANES, bool EXACT>
__device__ __forceinline__ void items_body(const HybridArgs &a, unsigned bx, GroupStage<kHybridThreads, LPR> &stage) {
    const int lane = threadIdx.x & 31, lg = threadIdx.x % LANES;
    const unsigned mask = LANES == 32 ? 0xffffffffu : ((1u << LANES % 32) - 1u) << (lane & ~(LANES - 1));
    const LaneCols<T, VW, LPR, NV, EXACT> lc(a.B, a.N, lg % LPR);
    const int32_t stride = static_cast<int32_t>(a.gc) * (kHybridThreads / LANES), n = a.chunks + a.wide;
    for (int32_t s = (static_cast<int32_t>(bx) * kHybridThreads + static_cast<int32_t>(threadIdx.x)) / LANES; s < n; s += stride) {
        const bool chunk = s < a.chunks;
        const int4 d = __ldg(chunk ? a.items + s : a.desc + (s - a.chunks));
        float acc[NV][VW];
        clear_acc(acc);
        group_sum<T, VW, LPR, NV, LANES, EXACT, false>(a, lc, stage, d.y, d.y + d.w, mask, acc);
        if (lg < LPR) {
            if (chunk && d.x >= 0) lc.store(a.scratch + static_cast<int64_t>(d.x) * a.N, acc, 1.f, 0.f);
            else lc.store(a.C + (d.x & 0x7FFFFFFF) * a.ldc, acc, a.alpha, a.beta);   // a light row, or a heavy row of one item
        }
    }
}

template <typename T, int VW, int LPR, int NV, bool EXACT>
__device__ __forceinline__ void medium_body(const HybridArgs &a, unsigned bx, GroupStage<kHybridThreads, LPR> &stage) {
    constexpr int LANES = LPR < 8 ? 8 : LPR;
    const int lane = threadIdx.x & 31, lg = threadIdx.x % LANES;
    const unsigned mask = LANES == 32 ? 0xffffffffu : ((1u << LANES % 32) - 1u) << (lane & ~(LANES - 1));
    const LaneCols<T, VW, LPR, NV, EXACT> lc(a.B, a.N, lg % LPR);
    const int4 *__restrict__ desc = a.desc + a.wide;
    const int32_t stride = static_cast<int32_t>(a.gm) * (kHybridThreads / LANES);
    for (int32_t s = (static_cast<int32_t>(bx) * kHybridThreads + static_cast<int32_t>(threadIdx.x)) / LANES; s < a.medium; s += stride) {
        const int4 cur = __ldg(desc + s);
        float acc[NV][VW];
        clear_acc(acc);
        group_sum<T, VW, LPR, NV, LANES, EXACT, false>(a, lc, stage, cur.y, cur.y + cur.w, mask, acc);
        if (lg < LPR) lc.store(a.C + cur.x * a.ldc, acc, a.alpha, a.beta);
    }
}

// Rows of fewer than kHybridMedium nonzeros, most of them one or two.  A group of LPR lanes owns R consecutive list
// entries at once, so that R gathers (one per row) are in flight per lane at every step; rows of similar length share
// a warp.  A list entry is a plan-time descriptor that names the row's first column: the first gather depends on
// nothing else (two dependent memory round trips per one-nonzero row: descriptor, row of B), and the (column, value)
// pair of step j + 1 is requested before the gathers of step j.  The lanes of a group read the same pair with one
// broadcast load.  Rows without nonzeros are written too (C = beta * C).
template <typename T, int VW, int LPR, int NV, int R, bool EXACT>
__device__ __forceinline__ void light_rows_body(const HybridArgs &a, unsigned bx) {
    const LaneCols<T, VW, LPR, NV, EXACT> lc(a.B, a.N, threadIdx.x % LPR);
    const int64_t r0 = (static_cast<int64_t>(bx) * kHybridThreads + threadIdx.x) / LPR * R;
    if (r0 >= a.light) return;
    const T *vals = static_cast<const T *>(a.vals);
    const int4 *__restrict__ desc = a.desc + a.wide + a.medium;
    int p[R], len[R], cn[R], row[R], maxlen = 0;
    float vn[R];
#pragma unroll
    for (int u = 0; u < R; ++u) {
        const int4 d = r0 + u < a.light ? __ldg(desc + r0 + u) : make_int4(-1, 0, 0, 0);
        row[u] = d.x;
        p[u] = d.y;
        cn[u] = d.z;
        len[u] = d.w;
        maxlen = max(maxlen, len[u]);
    }
#pragma unroll
    for (int u = 0; u < R; ++u) vn[u] = len[u] > 0 ? to_float(vals[p[u]]) : 0.f;
    float acc[R][NV][VW];
#pragma unroll
    for (int u = 0; u < R; ++u) clear_acc(acc[u]);
    for (int j = 0; j < maxlen; ++j) {
        Piece<T, VW> b[R][NV];
        float av[R];
#pragma unroll
        for (int u = 0; u < R; ++u) {
            lc.gather(cn[u], a.ldb_bytes, j < len[u], b[u]);
            av[u] = vn[u];
            const bool more = j + 1 < len[u];
            cn[u] = more ? __ldg(a.colind + p[u] + j + 1) : 0;
            vn[u] = more ? to_float(vals[p[u] + j + 1]) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < R; ++u)
            lc.fma(av[u], b[u], acc[u]);
    }
#pragma unroll
    for (int u = 0; u < R; ++u)
        if (row[u] >= 0) lc.store(a.C + row[u] * a.ldc, acc[u], a.alpha, a.beta);
}

// The first `gc` CTAs walk the items (persistent, grid-stride), the next `gm` the medium rows (likewise), the rest the
// short rows.  CTAs are placed in index order, so the item CTAs take the SMs first and the others fill in as they
// retire: what side streams and a high stream priority would give, without depending on how streams map to the GPU's
// hardware queues.
template <typename T, int VW, int LPR, int NV, int IL, int R, bool EXACT>
__global__ void __launch_bounds__(kHybridThreads, 4)
hybrid_kernel(const HybridArgs a) {
    __shared__ GroupStage<kHybridThreads, LPR> stage;
    overlap_wait();
    if (blockIdx.x < a.gc) items_body<T, VW, LPR, NV, IL, EXACT>(a, blockIdx.x, stage);
    else if (blockIdx.x < a.gc + a.gm) medium_body<T, VW, LPR, NV, EXACT>(a, blockIdx.x - a.gc, stage);
    else light_rows_body<T, VW, LPR, NV, R, EXACT>(a, blockIdx.x - a.gc - a.gm);
    overlap_next();
}

template <typename T, int VW, int LPR, int NV, int IL, bool EXACT>
cudaError_t launch_hybrid_exact(HybridArgs a, cudaStream_t st) {
    constexpr int R = NV * VW >= 8 ? 2 : 4;
    auto kernel = hybrid_kernel<T, VW, LPR, NV, IL, R, EXACT>;
    static std::atomic<int> occ_cache[kMaxDevices];
    const int64_t cap = static_cast<int64_t>(sm_count_cached()) * occupancy_cached(occ_cache, kernel, kHybridThreads);
    constexpr int items_per_cta = kHybridThreads / IL, medium_per_cta = kHybridThreads / (LPR < 8 ? 8 : LPR);
    const int64_t need_c = (static_cast<int64_t>(a.chunks) + a.wide + items_per_cta - 1) / items_per_cta;
    const int64_t need_m = (a.medium + medium_per_cta - 1) / medium_per_cta;
    const int64_t need_l = ((static_cast<int64_t>(a.light) + R - 1) / R * LPR + kHybridThreads - 1) / kHybridThreads;
    a.gc = static_cast<uint32_t>(need_c < cap ? need_c : cap);
    a.gm = static_cast<uint32_t>(need_m < cap ? need_m : cap);
    const int64_t total = static_cast<int64_t>(a.gc) + a.gm + need_l;
    if (total == 0) return cudaSuccess;
    if (total > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    constexpr int slab = LPR * NV * VW;
    return launch_overlapped(kernel, dim3(static_cast<unsigned>(total), static_cast<unsigned>((a.N + slab - 1) / slab)),
                             kHybridThreads, 0, st, a);
}

// Whole loads and every lane a column in every slab (8, 16, 32, ... columns): the lanes need no test.
template <typename T, int VW, int LPR, int NV, int IL>
cudaError_t launch_hybrid_il(const HybridArgs &a, cudaStream_t st) {
    if constexpr (VW * sizeof(T) == 16)
        if (a.N % (LPR * NV * VW) == 0) return launch_hybrid_exact<T, VW, LPR, NV, IL, true>(a, st);
    return launch_hybrid_exact<T, VW, LPR, NV, IL, false>(a, st);
}

// Lanes per item.  A whole warp as long as half warps would not all get an item (the chain of dependent gathers is what
// a small matrix waits for: R-MAT scale 14 at 32 columns 10.7 us, 18.3 with half warps); half a warp beyond that (fewer
// sums across lanes per nonzero: R-MAT scale 20 at 16 columns 235 us, 278 with whole warps); and with eight lanes across
// the columns and items enough to fill the GPU twice over, no lane sets at all (64 bf16 columns 430 -> 402 us).
template <typename T, int VW, int LPR, int NV>
cudaError_t launch_hybrid_one(const HybridArgs &a, cudaStream_t st) {
    if constexpr (LPR > 16) {
        return launch_hybrid_il<T, VW, LPR, NV, 32>(a, st);
    } else {
        const int64_t lanes = static_cast<int64_t>(sm_count_cached()) * 4 * kHybridThreads, items = static_cast<int64_t>(a.chunks) + a.wide;
        if (items < lanes / 16) return launch_hybrid_il<T, VW, LPR, NV, 32>(a, st);
        if constexpr (LPR == 8 && VW * sizeof(T) == 16)
            if (items >= 2 * (lanes / 8)) return launch_hybrid_il<T, VW, LPR, NV, 8>(a, st);
        return launch_hybrid_il<T, VW, LPR, NV, 16>(a, st);
    }
}

// Lanes across the columns for rows of `units` loads per row of B.  Full 16-byte loads: the next power of two up to 16, two
// loads per lane beyond (128 fp32 columns on R-MAT scale 20 as 16 x 2: 1,212 us, as 32 x 1: 1,268).  Narrower loads (odd
// widths, unaligned operands): two to four per lane, so that the work per nonzero on A is spread over more columns and few
// lane slots are idle (compared on an earlier state of this kernel, R-MAT scale 17: 41 columns as 16 lanes x 3 61 us, as one warp
// x 4 101; 25 columns as 16 x 2 46 us, as 32 x 1 56; 41 columns of 3.9 M nonzeros take 88 us now); wider rows run as slabs of
// about equal width.
template <typename T, int VW>
cudaError_t launch_hybrid(const HybridArgs &a, cudaStream_t st) {
    constexpr bool FULL = VW * sizeof(T) == 16;
    const int all = (a.N + VW - 1) / VW, widest = FULL ? 64 : 128;
    const int slabs = (all + widest - 1) / widest, units = (all + slabs - 1) / slabs;
    if constexpr (FULL) {
        if (units <= 1) return launch_hybrid_one<T, VW, 1, 1>(a, st);
        if (units <= 2) return launch_hybrid_one<T, VW, 2, 1>(a, st);
    }
    if (units <= 4) return launch_hybrid_one<T, VW, 4, 1>(a, st);
    if (units <= 8) return launch_hybrid_one<T, VW, 8, 1>(a, st);
    if constexpr (FULL) {
        if (units <= 16) return launch_hybrid_one<T, VW, 16, 1>(a, st);
        if (units <= 32) return launch_hybrid_one<T, VW, 16, 2>(a, st);
        return launch_hybrid_one<T, VW, 32, 2>(a, st);
    } else {
        if (units <= 16) return launch_hybrid_one<T, VW, 8, 2>(a, st);
        if (units <= 24) return launch_hybrid_one<T, VW, 8, 3>(a, st);
        if (units <= 32) return launch_hybrid_one<T, VW, 16, 2>(a, st);
        if (units <= 48) return launch_hybrid_one<T, VW, 16, 3>(a, st);
        if (units <= 64) return launch_hybrid_one<T, VW, 32, 2>(a, st);
        if (units <= 96) return launch_hybrid_one<T, VW, 32, 3>(a, st);
        return launch_hybrid_one<T, VW, 32, 4>(a, st);
    }
}

}  // namespace sd
