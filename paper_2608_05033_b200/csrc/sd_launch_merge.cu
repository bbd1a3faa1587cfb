#include <algorithm>

#include "sd_launch.cuh"
#include "sd_merge.cuh"
#include "sd_coo.cuh"
#include "sd_rowsplit.cuh"

namespace sd {

// The tile kernel alone, fp32 (the entry point without allocations adds the carries itself).
cudaError_t run_merge(const MergeArgs &m, bool vec, cudaStream_t st) {
    const LaneGeom g = lane_geometry(m.s.N, vec, 4, 0);
    return launch_merge<float>(m, vec, g.lpr, g.nv, st);
}

// ---- narrow dense operands: COO segmented reduction --------------------------------------------
// One instance: the grid is as many CTAs as are resident together, or as give every warp a step.  Returns the ranges.
template <typename T, int N, bool VEC, bool HOT, bool BITS, bool TURN = false>
static cudaError_t launch_coo_kernel(CooArgs a, int sm_count, int kept, cudaStream_t st, int64_t &ranges) {
    auto kernel = coo_kernel<T, N, VEC, HOT, BITS, TURN>;
    constexpr int threads = HOT ? kCooHotThreads : coo_threads(N);
    int64_t ctas = sm_count;
    if constexpr (HOT) {
        static std::atomic<bool> opted[kMaxDevices];
        const int dev = current_device();
        if (dev >= kMaxDevices || !opted[dev].load(std::memory_order_acquire)) {
            const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kCooHotBytes);
            if (e != cudaSuccess) return e;
            if (dev < kMaxDevices) opted[dev].store(true, std::memory_order_release);
        }
    } else {
        static std::atomic<int> occ[kMaxDevices];
        ctas *= std::min(occupancy_cached(occ, kernel, threads), kCooMaxWarps * 32 / threads);
    }
    const int64_t steps = coo_steps(a.count, N);
    ctas = std::min(ctas, (steps + threads / 32 - 1) / (threads / 32));
    const int64_t all = ctas * (threads / 32);
    a.warps = static_cast<int>(std::min(all, steps));
    a.per_warp = static_cast<int>((steps + static_cast<int64_t>(a.warps) * kCooRange - 1) / (static_cast<int64_t>(a.warps) * kCooRange));
    ranges = static_cast<int64_t>(a.warps) * a.per_warp;
    // Rounded up, so that the last range ends with the last step.  Longer and shorter ranges alternate: with the longer ones first, all of
    // them equally far apart, warps in rows of one length walk the same columns in step (100 rows of 300,000 nonzeros at two fp32
    // columns 107 -> 125 us).
    a.range = ((static_cast<uint64_t>(steps) << 32) + ranges - 1) / ranges;
    // Many steps per warp: neighbouring ranges go to different CTAs, since what a range costs depends on its rows and columns (60 M
    // nonzeros in rank-size rows 279 -> 271 us).  Few: to the same one, whose L1 they share (R-MAT scale 14 8.2 -> 7.7 us).
    a.spread = HOT || steps >= 8 * all;
    return launch_overlapped(kernel, static_cast<unsigned>(ctas), threads, kept, st, a);
}

template <typename T, int N, bool VEC>
static cudaError_t launch_coo_n(const CooPlan &cp, const SpmmArgs &s, int sm_count, cudaStream_t st) {
    CooArgs a{};
    a.row = cp.row;
    a.starts = cp.starts;
    a.colind = s.colind - cp.shift;
    a.vals = static_cast<const T *>(s.vals) - cp.shift;
    a.shift = cp.shift;
    a.B = s.B;
    a.ldb_bytes = s.ldb_bytes;
    a.count = cp.nnz + cp.shift;
    a.C = s.C;
    a.ldc = s.ldc;
    a.alpha = s.alpha;
    a.beta = s.beta;
    a.rowptr = cp.rowptr;
    a.M = cp.M;
    a.carry_row = cp.c1_row;
    a.carry_val = cp.c1_val;
    cudaError_t e;
    int64_t ranges = 0;
    const int kept = cp.hot * N * static_cast<int>(sizeof(T));
    const bool hot = cp.hot > 0 && kept <= kCooHotBytes;
    if (hot) {
        a.colind = cp.hot_colind;
        a.hot_cols = cp.hot_cols;
        a.hot = cp.hot;
    }
    if constexpr (N == 1) {
        const bool turn = !hot && coo_steps(a.count, N) >= int64_t{8} * 32 * sm_count;   // eight steps and more for each of 32 warps per SM
        if (cp.starts)
            e = hot    ? launch_coo_kernel<T, N, VEC, true, true>(a, sm_count, kept, st, ranges)
                : turn ? launch_coo_kernel<T, N, VEC, false, true, true>(a, sm_count, 0, st, ranges)
                       : launch_coo_kernel<T, N, VEC, false, true>(a, sm_count, 0, st, ranges);
        else
            e = hot    ? launch_coo_kernel<T, N, VEC, true, false>(a, sm_count, kept, st, ranges)
                : turn ? launch_coo_kernel<T, N, VEC, false, false, true>(a, sm_count, 0, st, ranges)
                       : launch_coo_kernel<T, N, VEC, false, false>(a, sm_count, 0, st, ranges);
    } else {
        e = hot ? launch_coo_kernel<T, N, VEC, true, false>(a, sm_count, kept, st, ranges) : launch_coo_kernel<T, N, VEC, false, false>(a, sm_count, 0, st, ranges);
    }
    if (e != cudaSuccess) return e;
    const int32_t *frow = cp.c1_row;
    const float *fval = cp.c1_val;
    int64_t fcount = 2 * ranges;
    if (fcount > kCooDirectFinal) {   // level 2
        const int64_t chunks = (fcount + kCooCarryChunk - 1) / kCooCarryChunk;
        CooArgs b = a;
        b.row = cp.c1_row;
        b.vals = cp.c1_val;
        b.count = fcount;
        b.carry_row = cp.c2_row;
        b.carry_val = cp.c2_val;
        if ((e = launch_overlapped(coo_carry_kernel<N>, static_cast<unsigned>((chunks + 7) / 8), 256, 0, st, b)) != cudaSuccess) return e;
        frow = cp.c2_row;
        fval = cp.c2_val;
        fcount = 2 * chunks;
    }
    return launch_overlapped(coo_final_kernel<N>, static_cast<unsigned>((fcount + 255) / 256), 256, 0, st, frow, fval, fcount, s.C, s.ldc, s.alpha,
                             s.beta);
}

template <typename T, int N>
static cudaError_t launch_coo_vec(const CooPlan &cp, const SpmmArgs &s, int sm_count, cudaStream_t st) {
    constexpr uintptr_t bytes = N * sizeof(T);   // of a row of B: one load if all of them start at a multiple
    if ((reinterpret_cast<uintptr_t>(s.B) | s.ldb_bytes) % bytes == 0) return launch_coo_n<T, N, true>(cp, s, sm_count, st);
    return launch_coo_n<T, N, false>(cp, s, sm_count, st);
}

template <typename T>
static cudaError_t launch_coo(const CooPlan &cp, const SpmmArgs &s, int sm_count, cudaStream_t st) {
    switch (s.N) {
    case 1: return launch_coo_n<T, 1, false>(cp, s, sm_count, st);
    case 2: return launch_coo_vec<T, 2>(cp, s, sm_count, st);
    case 3: return launch_coo_n<T, 3, false>(cp, s, sm_count, st);
    case 4: return launch_coo_vec<T, 4>(cp, s, sm_count, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t run_coo(const CooPlan &cp, const SpmmArgs &s, int dtype, int sm_count, cudaStream_t st) {
    return dtype == SD_F32 ? launch_coo<float>(cp, s, sm_count, st) : launch_coo<__nv_bfloat16>(cp, s, sm_count, st);
}

cudaError_t build_coo_rows(const int32_t *rowptr, int64_t M, int64_t nnz, int shift, int64_t steps, int32_t *row, uint8_t *starts, cudaStream_t st) {
    if (nnz == 0) return cudaSuccess;
    const int64_t count = starts ? 32 * steps : nnz + shift;
    coo_rows_kernel<<<static_cast<unsigned>((count + 255) / 256), 256, 0, st>>>(rowptr, M, nnz, shift, starts ? 8 : 1, count, row);
    if (starts) {
        const cudaError_t e = cudaMemsetAsync(starts, 0, 32 * steps, st);
        if (e != cudaSuccess) return e;
        coo_starts_kernel<<<static_cast<unsigned>((M + 255) / 256), 256, 0, st>>>(rowptr, M, nnz, shift, reinterpret_cast<unsigned *>(starts));
    }
    return cudaGetLastError();
}

}  // namespace sd
