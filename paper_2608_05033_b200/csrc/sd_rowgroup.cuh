// Family (a), one group of LANES lanes per row in natural order: LPR lanes stand across the columns, LANES / LPR lane sets share
// the row's nonzeros (group_sum).  It serves every width that is not a whole number of 16-byte loads (odd widths, unaligned
// operands: two to four loads of 8, 4 or 2 bytes per lane) and rows long enough to share at the others.  Rows of more than
// kRowGroupTerms nonzeros per lane set that the rule asks for stay with the other kernels (a line from before long rows were folded).
#pragma once

#include "sd_group.cuh"

namespace sd {

constexpr int kRowGroupThreads = 256;
constexpr int kRowGroupTerms = 512;

template <typename T, int VW, int LPR, int NV, int LANES, bool EXACT, bool FOLD>
__global__ void __launch_bounds__(kRowGroupThreads, FOLD ? 4 : 5)
rowgroup_kernel(const SpmmArgs a) {
    const int lane = threadIdx.x & 31, lg = threadIdx.x % LANES;
    const unsigned mask = LANES == 32 ? 0xffffffffu : ((1u << LANES % 32) - 1u) << (lane & ~(LANES - 1));
    const int64_t row = (static_cast<int64_t>(blockIdx.x) * kRowGroupThreads + threadIdx.x) / LANES;
    int p0 = 0, p1 = 0;
    if (row < a.S) {
        p0 = __ldg(a.ptr + row);
        p1 = __ldg(a.ptr + row + 1);
    }
    overlap_wait();
    __shared__ GroupStage<kRowGroupThreads, LPR> stage;
    const LaneCols<T, VW, LPR, NV, EXACT> lc(a.B, a.N, lg % LPR);
    float acc[NV][VW];
    clear_acc(acc);
    group_sum<T, VW, LPR, NV, LANES, EXACT, FOLD>(a, lc, stage, p0, p1, mask, acc);
    overlap_next();
    if (row < a.S && lg < LPR) lc.store(a.C + row * a.ldc, acc, a.alpha, a.beta);
}

// `terms`: products that a lane set may add in one accumulator; with longer rows all are folded.  The sets are those that run, not those
// that the rule asks for: a warp has no room for four of 16 lanes.
template <typename T, int VW, int LPR, int NV, int LANES>
cudaError_t launch_rowgroup_lanes(const SpmmArgs &a, int terms, cudaStream_t st) {
    constexpr int rows = kRowGroupThreads / LANES, slab = LPR * NV * VW;
    const bool fold = a.max_len > static_cast<int64_t>(terms) * (LANES / LPR);
    auto kernel = fold ? rowgroup_kernel<T, VW, LPR, NV, LANES, false, true> : rowgroup_kernel<T, VW, LPR, NV, LANES, false, false>;
    if constexpr (VW * sizeof(T) == 16)
        if (a.N % slab == 0) kernel = fold ? rowgroup_kernel<T, VW, LPR, NV, LANES, true, true> : rowgroup_kernel<T, VW, LPR, NV, LANES, true, false>;
    return launch_overlapped(kernel, dim3(static_cast<unsigned>((a.S + rows - 1) / rows), static_cast<unsigned>((a.N + slab - 1) / slab)),
                             kRowGroupThreads, 0, st, a);
}

// Lane sets per row: 1, 4 (as many as fit a warp) or, with 8 or 16 lanes across the columns, 2.
template <typename T, int VW, int LPR, int NV>
cudaError_t launch_rowgroup_one(const SpmmArgs &a, int sets, int terms, cudaStream_t st) {
    constexpr int MANY = LPR * 4 > 32 ? 32 : LPR * 4;
    if constexpr ((LPR == 8 || LPR == 16) && NV == 1 && VW * sizeof(T) == 16)
        if (sets == 2) return launch_rowgroup_lanes<T, VW, LPR, NV, 2 * LPR>(a, terms, st);
    if (sets > 1) return launch_rowgroup_lanes<T, VW, LPR, NV, MANY>(a, terms, st);
    return launch_rowgroup_lanes<T, VW, LPR, NV, LPR>(a, terms, st);
}

template <typename T, int VW>
cudaError_t launch_rowgroup(const SpmmArgs &a, int sets, int terms, cudaStream_t st) {
    constexpr bool FULL = VW * sizeof(T) == 16;
    const int all = (a.N + VW - 1) / VW, widest = FULL ? 64 : 128;
    const int slabs = (all + widest - 1) / widest, units = (all + slabs - 1) / slabs;
    if constexpr (FULL) {
        if (units <= 1) return launch_rowgroup_one<T, VW, 1, 1>(a, sets, terms, st);
        if (units <= 2) return launch_rowgroup_one<T, VW, 2, 1>(a, sets, terms, st);
    }
    if (units <= 4) return launch_rowgroup_one<T, VW, 4, 1>(a, sets, terms, st);
    if (units <= 8) return launch_rowgroup_one<T, VW, 8, 1>(a, sets, terms, st);
    if constexpr (FULL) {
        if (units <= 16) return launch_rowgroup_one<T, VW, 16, 1>(a, sets, terms, st);
        if (units <= 32) return launch_rowgroup_one<T, VW, 16, 2>(a, sets, terms, st);
        return launch_rowgroup_one<T, VW, 32, 2>(a, sets, terms, st);
    } else {
        if (units <= 16) return launch_rowgroup_one<T, VW, 8, 2>(a, sets, terms, st);
        if (units <= 24) return launch_rowgroup_one<T, VW, 8, 3>(a, sets, terms, st);
        if (units <= 32) return launch_rowgroup_one<T, VW, 16, 2>(a, sets, terms, st);
        if (units <= 48) return launch_rowgroup_one<T, VW, 16, 3>(a, sets, terms, st);
        if (units <= 64) return launch_rowgroup_one<T, VW, 32, 2>(a, sets, terms, st);
        if (units <= 96) return launch_rowgroup_one<T, VW, 32, 3>(a, sets, terms, st);
        return launch_rowgroup_one<T, VW, 32, 4>(a, sets, terms, st);
    }
}

}  // namespace sd
