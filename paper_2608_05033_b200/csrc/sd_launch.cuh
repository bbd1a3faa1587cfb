// Host entry points of the kernel families, one translation unit each.
#pragma once

#include "sd_common.cuh"

namespace sd {

// Every tile holds the same number of merged items whatever the lane geometry, so one tile
// table serves every dense width and both the vector and the scalar kernels.
constexpr int kMergeTile = 1024;

struct MergeArgs {
    SpmmArgs s;
    const int32_t *tile_seg;  // [ntiles + 1] row coordinate of each tile start
    float *tile_head;         // [ntiles][N]  partial of the row open at tile start, if it ends here
    float *tile_tail;         // [ntiles][N]  partial of the row still open at tile end
    int32_t ntiles;
};


// Family (a).  `vw`: elements per load of B (piece_width).
cudaError_t run_rowsplit(const SpmmArgs &a, int dtype, int vw, cudaStream_t st);
cudaError_t run_rowgroup_f32(const SpmmArgs &a, int vw, int sets, int terms, cudaStream_t st);
cudaError_t run_rowgroup_bf16(const SpmmArgs &a, int vw, int sets, int terms, cudaStream_t st);

// Hybrid family in one launch: items (chunks of the heavy rows, long light rows), medium rows, short rows.
struct HybridArgs;
cudaError_t run_hybrid_f32(const HybridArgs &a, int vw, cudaStream_t st);
cudaError_t run_hybrid_bf16(const HybridArgs &a, int vw, cudaStream_t st);

// Heavy rows: row rows[i] owns the scratch rows chunk_ptr[i] .. chunk_ptr[i+1]-1 of chunk_out ([chunks][N]); their sum, taken in
// order, is its product (a row of one chunk has been written already).  skip_above > 0: rows of more chunks are left to run_chunk_reduce_wide (list: their positions).
cudaError_t run_chunk_reduce(const float *chunk_out, const int32_t *chunk_ptr, const int32_t *rows, int64_t nl, float *C,
                             int64_t ldc, int32_t N, float alpha, float beta, cudaStream_t st, int32_t skip_above);
constexpr int kGiantChunks = 64;   // rows of more scratch rows than this are summed by a whole CTA
cudaError_t run_chunk_reduce_wide(const float *chunk_out, const int32_t *chunk_ptr, const int32_t *rows, const int32_t *list,
                                  int64_t count, float *C, int64_t ldc, int32_t N, float alpha, float beta, cudaStream_t st);

// C = beta * C.
cudaError_t run_scale_c(float *C, int64_t ldc, int64_t M, int32_t N, float beta, cudaStream_t st);

// Merge-path tile kernel, fp32; the caller adds the carries.
cudaError_t run_merge(const MergeArgs &m, bool vec, cudaStream_t st);

// Family (b) for dense widths up to kCooMaxN (beyond it the shuffles per nonzero outweigh the
// gain; measured cross-over between 4 and 8 columns): segmented reduction over the nonzeros, carries reduced in two more levels.
constexpr int kCooMaxN = 4;
constexpr int coo_items(int N) { return N <= 2 ? 8 : 4; }   // nonzeros of a lane and step
// items before the first nonzero: what a lane takes of `array` is then one load, wherever it begins
inline int coo_shift(const void *array, int element, int N) { return static_cast<int>(reinterpret_cast<uintptr_t>(array) / element % coo_items(N)); }
constexpr int64_t coo_steps(int64_t items, int N) { return (items + 32 * coo_items(N) - 1) / (32 * coo_items(N)); }
constexpr int kCooCarryChunk = 128;
constexpr int64_t kCooDirectFinal = 4096;  // carry lists up to this length skip the second level
constexpr int kCooMaxWarps = 64;           // resident on one SM; each leaves two carry entries per range
constexpr int kCooRange = 64;              // steps: longer shares of a warp are cut into several ranges
constexpr int64_t coo_most_ranges(int64_t steps, int64_t warps) { return steps < warps ? steps : warps + steps / kCooRange; }
struct CooPlan {
    const int32_t *row;    // [shift + nnz] row of every item, or with `starts` [32 steps] of every eighth
    const uint8_t *starts; // [32 steps] a bit per item that begins a row
    const int32_t *rowptr; // [M + 1]
    int64_t M;             // rows to search for empty ones (0: the matrix has none)
    int64_t nnz;
    int shift;             // items before the first nonzero
    int32_t *c1_row;      // [2 * coo_most_ranges(steps, kCooMaxWarps * SMs)] first-level carries
    float *c1_val;        // ... x N
    int32_t *c2_row;      // [2 * ceil(len(c1) / kCooCarryChunk)] second-level carries
    float *c2_val;
    const int32_t *hot_colind;   // [shift + nnz] columns, those of hot_cols renamed (hot == 0: none)
    const int32_t *hot_cols;
    int32_t hot;
};
constexpr int kCooHotBytes = 128 * 1024;   // the rest is L1 for the gathers outside: with 200 KB two fp32 columns took 281 us instead of 173
cudaError_t run_coo(const CooPlan &cp, const SpmmArgs &s, int dtype, int sm_count, cudaStream_t st);
// starts != nullptr: a bit per item and the row of every eighth; no row is empty.
cudaError_t build_coo_rows(const int32_t *rowptr, int64_t M, int64_t nnz, int shift, int64_t steps, int32_t *row, uint8_t *starts, cudaStream_t st);

struct BsrArgs {
    const int32_t *browptr;  // [Mb + 1]
    const int32_t *bcol;     // [nnzb]
    const void *bval;        // [nnzb][16][16] row-major, plan dtype
    const void *B;
    float *C;
    int64_t ldb, ldc;
    int64_t M, K;
    int32_t Mb;
    int32_t N;
    float alpha, beta;
};
cudaError_t run_bsr(const BsrArgs &a, int dtype, cudaStream_t st);
cudaError_t run_wait_expiry(int32_t *error, cudaStream_t st);   // see sd_plan_desc_t.test_wait_expiry
// Counts behind sd_plan_get_features (row-length / column-degree quartiles, column-degree moments,
// SELL slots for slice heights 16 / 32 / 512, occupied 4x4 and 8x8 blocks).  Synchronous.
struct FeatureCounts {
    int64_t row_q[3], col_q[3], col_max, col_empty;
    uint64_t sum_d2;
    int64_t sell_slots[3];
    int64_t nnzb4, nnzb8;
};
sd_status_t compute_feature_counts(const int32_t *rowptr, const int32_t *colind, int64_t M, int64_t K, int64_t nnz,
                                   cudaStream_t st, FeatureCounts *out);

}  // namespace sd
