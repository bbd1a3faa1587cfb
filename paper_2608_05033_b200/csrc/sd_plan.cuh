// The plan object and the device memory it owns.
#pragma once

#include <mutex>
#include <vector>

#include "sd_launch.cuh"

namespace sd {

// Streams and events of one product with host operands in flight.  Creating three streams costs as much as a small product takes,
// so sets are shared by the plans of a device: a plan takes one for a call and gives it back when it has waited for the
// result.  At most kHostStreamSets are kept for later calls.
struct HostStreams {
    int device = 0;
    cudaStream_t st = nullptr;                    // products
    cudaStream_t in = nullptr, out = nullptr;     // column slices: copies in and out, beside the products
    cudaEvent_t in_ev = nullptr, out_ev = nullptr, done_ev = nullptr;
};
constexpr size_t kHostStreamSets = 8;

}  // namespace sd

struct sd_plan {
    const int32_t *rowptr = nullptr;
    const int32_t *colind = nullptr;
    const void *vals = nullptr;
    int64_t M = 0, K = 0, N = 0, nnz = 0;
    int dtype = SD_F32;
    int device = 0;
    sd_plan_info_t info{};

    // MERGE and HYBRID: rows of at least h_T nonzeros ("heavy") run as chunks of the caller's CSR arrays, column window by
    // column window, the rest row-wise from a list sorted by falling length
    int32_t *h_rows = nullptr;       // [M] the heavy rows, ascending, then the light rows, longest first, ascending inside a length
    int32_t *h_chunk_ptr = nullptr;  // [h_nl + 1] first chunk of every heavy row (chunks are numbered row by row)
    int32_t *h_item_ptr = nullptr;   // [h_nl + 1] first scratch row of every heavy row
    int4 *h_items = nullptr;         // [h_ni] the chunks in the order they are taken, h_F consecutive ones of a row and window
                                     // together: {scratch row, or row | bit 31 for a row of one item; first nonzero; first chunk; length}
    int32_t *h_giant = nullptr;      // [h_ng] positions in h_rows of the rows of more than kGiantChunks chunks (a CTA sums each)
    int4 *h_desc = nullptr;          // [M - h_nl] per light row, in list order: {row, first nonzero, its column, length}
    float *chunk_out = nullptr;      // [h_ni][N] partial sums of the items
    int64_t h_nl = 0, h_nc = 0, h_ni = 0, h_ng = 0;
    int32_t h_F = 1;                 // chunks per item
    int64_t h_nm = 0;                // the first h_nm light rows have at least kHybridMedium nonzeros
    int64_t h_nw = 0;                // the first h_nw of those at least kHybridWide
    struct { unsigned long long chunks_long = 0, chunks_long2 = 0, chunks_long4 = 0, giants = 0, len_hist[256] = {}; } h_counts;   // of the scan, for sd_plan_save
    int32_t h_T = 0;                 // 0: no schedule (nothing to multiply, or another executor)

    // narrow dense operands (N <= kCooMaxN) of the merge family
    int coo_shift = 0;               // items before the first nonzero
    int32_t *coo_row = nullptr;      // row of every item, or with coo_starts of every eighth
    uint8_t *coo_starts = nullptr;   // a bit per item that begins a row (one column, no empty rows)
    int32_t *coo_c1_row = nullptr, *coo_c2_row = nullptr;
    float *coo_c1_val = nullptr, *coo_c2_val = nullptr;
    int32_t *coo_hot_colind = nullptr, *coo_hot_cols = nullptr;   // columns kept in shared memory
    int32_t coo_hot = 0;

    // BSR
    int32_t *browptr = nullptr;
    int32_t *bcol = nullptr;
    void *bval = nullptr;
    int32_t *brow_first = nullptr;    // [16 nnzb] first nonzero of every row of a block
    uint16_t *brow_mask = nullptr;    // [16 nnzb] its columns
    int32_t *dev_error = nullptr;
    int64_t nnzb = 0;
    int32_t test_wait_expiry = 0;

    // host-buffer entry point
    void *stage_B = nullptr;
    float *stage_C = nullptr;
    sd::HostStreams *host = nullptr;    // held from a host product until it has been waited for
    cudaEvent_t values_ev = nullptr;    // orders new values before the host product that follows
    bool values_recorded = false;       // values_ev is to be waited for

    std::vector<void *> allocs;   // every device allocation of the plan
    int64_t owned = 0;            // their bytes

    sd_features_t feat{};       // extended analysis, computed at the first sd_plan_get_features
    bool have_feat = false;
};

namespace sd {

// Device memory comes from one stream-ordered pool per device that the library owns.  Creating a plan took 46 cudaMalloc and
// 66 cudaFree calls (11 ms of a 15 ms plan creation for 1.9 M nonzeros), each of them a device-wide synchronisation or close
// to one; an allocation from the pool is about a microsecond.  The pool keeps at most kPoolKeep bytes between plans (more is
// given back to the device at the next synchronisation, the rest by sd_release_unused) and may be used from any thread and stream.
constexpr size_t kPoolKeep = size_t{256} << 20;
cudaError_t pool_alloc(void **out, size_t bytes, cudaStream_t st);
sd_status_t pool_release();
void host_blocks_release();

// Memory the plan owns.  Usable on `st` at once, elsewhere after the synchronisation that ends plan creation.
sd_status_t dev_alloc_bytes(sd_plan *p, void **out, size_t bytes, const char *what, cudaStream_t st);
template <typename T>
sd_status_t dev_alloc(sd_plan *p, T **out, size_t count, const char *what, cudaStream_t st) {
    return dev_alloc_bytes(p, reinterpret_cast<void **>(out), count * sizeof(T), what, st);
}

struct TempBuf {   // temporary device memory, given back in stream order on every exit path
    void *p = nullptr;
    cudaStream_t st;
    explicit TempBuf(cudaStream_t s) : st(s) {}
    ~TempBuf() { if (p) cudaFreeAsync(p, st); }
    TempBuf(const TempBuf &) = delete;
    TempBuf &operator=(const TempBuf &) = delete;
    sd_status_t get(size_t bytes, const char *what) { return dev_alloc_bytes(nullptr, &p, bytes, what, st); }
    template <typename T> T *as() const { return static_cast<T *>(p); }
};

// A page-locked host block for reading results back (a copy to pageable memory goes through a driver buffer and costs
// several times the launch of a kernel).  Blocks are recycled; at most kHostBlocks are kept.
struct HostBlock {
    static constexpr size_t kBytes = 16384;
    void *p = nullptr;
    HostBlock();
    ~HostBlock();
    HostBlock(const HostBlock &) = delete;
    HostBlock &operator=(const HostBlock &) = delete;
};

// What the structure scan of plan creation counts (all exact integers).
struct ScanAccum {
    unsigned long long row_hist[32];
    unsigned long long sum_r2, empty_rows, sum_span, sum_gap, diag, unsorted_rows, long_rows, nnz_long_rows;
    unsigned long long max_r, max_span;
    unsigned long long blk_hist[9];
    unsigned long long nnz_dense_blocks, nnzb;
    unsigned long long bad_csr;           // validation: number of offending rows / entries
    unsigned long long chunks_long;       // chunks of the rows of at least 256 nonzeros ...
    unsigned long long chunks_long2, chunks_long4;   // ... and items of two and of four chunks each (the last of a row may be shorter)
    unsigned long long giants;            // rows of more than kGiantChunks chunks
    unsigned long long len_hist[256];     // rows of exactly 0 .. 255 nonzeros
    long long nnz;                        // rowptr[M]
    unsigned int huge;                    // block-rows left to the last scan kernel
};

constexpr int kChunkNnz = 128;      // heavy rows are cut into pieces of at most this many nonzeros
constexpr int kHybridHeavy = 256;   // HYBRID: rows of at least this many nonzeros run as chunks: the long-row threshold
                                    // of the paper's appendix listing
constexpr int kHybridHeavyMax = 256;   // upper limit: a light row is one running sum per lane set
constexpr int kHybridMedium = 4;    // light rows of at least this many nonzeros take a lane group each, a step of nonzeros at a
                                    // time; shorter ones run several rows per lane group, a nonzero at a time (2 / 3 / 4 / 8 /
                                    // 16 / 32 measured on six workloads: 4 is best or level on five)
constexpr int kHybridWide = 32;     // light rows of at least this many nonzeros take 16 or 32 lanes each, like a chunk

// Counts the structure of the pattern into `out` (device, cleared here).
cudaError_t scan_structure(const int32_t *rowptr, const int32_t *colind, int64_t M, int64_t K, ScanAccum *out, cudaStream_t st);
cudaError_t validate_csr(const int32_t *rowptr, const int32_t *colind, int64_t M, int64_t K, int64_t nnz, ScanAccum *out, cudaStream_t st);

// Heavy rows as chunks inside W column windows, light rows by length (`h`: the scan's counts on the host).
sd_status_t build_schedule(sd_plan *p, int W, int32_t T, const ScanAccum &h, cudaStream_t st);
// Row index per nonzero and carry lists of the narrow-operand reduction.
sd_status_t build_coo(sd_plan *p, cudaStream_t st);
// 16x16 blocks: pointers, columns, values, tensor-core images, partition.
sd_status_t build_bsr(sd_plan *p, int64_t nnzb, cudaStream_t st);
// Values and images from the caller's current array.
cudaError_t fill_bsr(const sd_plan *p, bool overlap, cudaStream_t st);

// Introspection: built on request from the caller's CSR arrays.
sd_status_t inspect_tiles(const sd_plan *p, int32_t *host_out);
sd_status_t inspect_segments(const sd_plan *p, int W, int32_t *seg_ptr, int32_t *seg_row, int32_t *colind, void *vals, int64_t *win_seg);
sd_status_t count_segments(const sd_plan *p, int W, int64_t *count, cudaStream_t st);

}  // namespace sd
