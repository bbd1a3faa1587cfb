// Introspection of the merge family: the merge-path tile table and the window-major segment list (the paper's "packed column
// windows" for SpMM, Sec. 3.4) are built when they are asked for, from the caller's CSR arrays; sd_spmm reads neither.
#include <cub/cub.cuh>

#include "sd_plan.cuh"

namespace sd {

constexpr int kShortSegment = 32;   // segments of more nonzeros than this are listed before the others of their window

__global__ void iota_kernel(int32_t *out, int64_t n) {
    const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i < n) out[i] = static_cast<int32_t>(i);
}

// Merge-path tile table: tile_seg[t] = #{ r : ptr[r+1] + r < t*tile }.
__global__ void merge_table_kernel(const int32_t *__restrict__ ptr, int64_t S, int32_t tile, int32_t ntiles,
                                   int32_t *__restrict__ tile_seg) {
    const int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (t > ntiles) return;
    const int64_t d = min(t * tile, S + ptr[S]);
    int64_t lo = 0, hi = S;   // number of row ends placed before position d
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (ptr[mid + 1] + mid < d) lo = mid + 1;
        else hi = mid;
    }
    tile_seg[t] = static_cast<int32_t>(lo);
}

// The column range is cut into W windows of wcols columns.  Nonzeros are re-bucketed by window
// (stable, so rows stay ascending inside a window); a segment is the run of one row inside one
// window.  Windows are executed one after the other, so the slab of B a window touches can stay
// in L2 while every nonzero of that window is processed.
__global__ void __launch_bounds__(256)
window_keys_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colind, int64_t M, int32_t wcols,
                   uint32_t *__restrict__ wkey, int32_t *__restrict__ rowid) {
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
    for (int64_t row = warp0; row < M; row += nwarps)
        for (int p = rowptr[row] + lane; p < rowptr[row + 1]; p += 32) {
            wkey[p] = static_cast<uint32_t>(colind[p] / wcols);
            rowid[p] = static_cast<int32_t>(row);
        }
}

__global__ void window_rows_kernel(const int32_t *__restrict__ perm, const int32_t *__restrict__ rowid, int64_t nnz,
                                   int32_t *__restrict__ w_row) {
    const int64_t q = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (q < nnz) w_row[q] = rowid[perm[q]];
}

__global__ void window_headflag_kernel(const uint32_t *__restrict__ wkey_sorted, const int32_t *__restrict__ w_row,
                                       int64_t nnz, uint8_t *__restrict__ flag) {
    const int64_t q = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (q >= nnz) return;
    flag[q] = (q == 0) || (w_row[q] != w_row[q - 1]) || (wkey_sorted[q] != wkey_sorted[q - 1]);
}

__global__ void window_emptyflag_kernel(const int32_t *__restrict__ rowptr, int64_t M, uint8_t *__restrict__ flag) {
    const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i < M) flag[i] = rowptr[i + 1] == rowptr[i];
}

// First ordering of the segments: the E empty rows (their ids are already in seg_row[0..E)),
// then the runs of (window, row) in window-major order.  Each gets its start and length in
// the window-sorted nonzero order, its output row with the "already written" bit, and the
// sort key 3 * window + class (class 0: more than `short_len` nonzeros, class 1: 0 or
// 2..short_len nonzeros, class 2: exactly one).
__global__ void window_segments_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colind,
                                       const uint32_t *__restrict__ wkey_sorted, const int32_t *__restrict__ w_row,
                                       const int32_t *__restrict__ heads, int32_t wcols, int32_t short_len, int64_t E,
                                       int64_t S, int64_t nnz, int32_t *__restrict__ seg_start,
                                       int32_t *__restrict__ seg_len, int32_t *__restrict__ seg_row,
                                       uint32_t *__restrict__ seg_key) {
    const int64_t s = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (s >= S) return;
    if (s < E) {
        seg_start[s] = 0;
        seg_len[s] = 0;
        seg_key[s] = 1;   // window 0, short class
        return;
    }
    const int64_t h = s - E;
    const int32_t q = heads[h];
    const int32_t len = static_cast<int32_t>((h + 1 < S - E ? heads[h + 1] : nnz) - q);
    const int32_t row = w_row[q];
    const uint32_t win = wkey_sorted[q];
    const uint32_t first_win = static_cast<uint32_t>(colind[rowptr[row]] / wcols);
    seg_start[s] = q;
    seg_len[s] = len;
    seg_row[s] = row | (win != first_win ? static_cast<int32_t>(0x80000000u) : 0);
    seg_key[s] = 3 * win + (len > short_len ? 0u : (len == 1 ? 2u : 1u));
}

__global__ void window_reorder_kernel(const int32_t *__restrict__ order, const int32_t *__restrict__ seg_len,
                                      const int32_t *__restrict__ seg_row, int64_t S, int32_t *__restrict__ len2,
                                      int32_t *__restrict__ row2) {
    const int64_t s = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (s >= S) return;
    len2[s] = seg_len[order[s]];
    row2[s] = seg_row[order[s]];
}

// Final gather of the nonzeros: output position q belongs to the segment found by binary
// search in the new segment pointers; its source is that segment's run in window-sorted order.
template <typename T>
__global__ void window_gather_kernel(const int32_t *__restrict__ seg_ptr2, const int32_t *__restrict__ order,
                                     const int32_t *__restrict__ seg_start, const int32_t *__restrict__ perm,
                                     const int32_t *__restrict__ colind, const T *__restrict__ vals, int64_t S, int64_t nnz,
                                     int32_t *__restrict__ w_col, T *__restrict__ w_val) {
    const int64_t q = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (q >= nnz) return;
    int64_t lo = 0, hi = S;   // last segment with seg_ptr2[s] <= q and a non-zero length covers q
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (seg_ptr2[mid + 1] <= q) lo = mid + 1;
        else hi = mid;
    }
    const int32_t p = perm[seg_start[order[lo]] + (q - seg_ptr2[lo])];
    w_col[q] = colind[p];
    w_val[q] = vals[p];
}

// bounds[k] = first segment (in the final order) whose key is >= k, for k = 0..2W.
__global__ void window_bounds_kernel(const uint32_t *__restrict__ key_sorted, int64_t S, int32_t nkeys,
                                     int64_t *__restrict__ bounds) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k > nkeys) return;
    int64_t lo = 0, hi = S;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (key_sorted[mid] < static_cast<uint32_t>(k)) lo = mid + 1;
        else hi = mid;
    }
    bounds[k] = lo;
}

struct SegmentLists {
    TempBuf w_col, w_vals, w_ptr, w_seg_row;
    std::vector<int64_t> bounds;   // per window: first segment of each of the three classes; then the number of segments
    int64_t S = 0;
    explicit SegmentLists(cudaStream_t st) : w_col(st), w_vals(st), w_ptr(st), w_seg_row(st) {}
};

// Re-buckets the nonzeros by column window and builds the (row, window) segment list, ordered by (window, class, row): inside
// a window the long segments come first, then those of none or 2 .. kShortSegment nonzeros, then those of exactly one.
static sd_status_t segment_lists(const sd_plan *p, int W, SegmentLists &l, cudaStream_t st) {
    const int64_t nnz = p->nnz, M = p->M;
    const int32_t wcols = static_cast<int32_t>((p->K + W - 1) / W);
    const size_t es = p->dtype == SD_F32 ? 4 : 2;
    const int64_t E = p->info.empty_rows;
    sd_status_t s;
    TempBuf wkey(st), wkey_sorted(st), rowid(st), w_row(st), ids(st), perm(st), tmp(st), flag(st), nsel(st), heads(st);
    if ((s = wkey.get(4 * nnz, "window keys"))) return s;
    if ((s = wkey_sorted.get(4 * nnz, "window keys"))) return s;
    if ((s = rowid.get(4 * nnz, "row ids"))) return s;
    if ((s = w_row.get(4 * nnz, "row ids"))) return s;
    if ((s = ids.get(4 * nnz, "positions"))) return s;
    if ((s = perm.get(4 * nnz, "permutation"))) return s;
    if ((s = l.w_col.get(4 * nnz, "window-major colind"))) return s;
    if ((s = l.w_vals.get(es * nnz, "window-major values"))) return s;

    window_keys_kernel<<<148 * 8, 256, 0, st>>>(p->rowptr, p->colind, M, wcols, static_cast<uint32_t *>(wkey.p),
                                               static_cast<int32_t *>(rowid.p));
    SD_CUDA_TRY(cudaGetLastError());
    iota_kernel<<<ceil_div(nnz, 256), 256, 0, st>>>(static_cast<int32_t *>(ids.p), nnz);
    SD_CUDA_TRY(cudaGetLastError());
    int bits = 1;
    while ((1 << bits) < W) ++bits;
    size_t tb = 0;
    SD_CUDA_TRY(cub::DeviceRadixSort::SortPairs(nullptr, tb, static_cast<uint32_t *>(wkey.p),
                                                static_cast<uint32_t *>(wkey_sorted.p), static_cast<int32_t *>(ids.p),
                                                static_cast<int32_t *>(perm.p), nnz, 0, bits, st));
    if ((s = tmp.get(tb, "sort scratch"))) return s;
    SD_CUDA_TRY(cub::DeviceRadixSort::SortPairs(tmp.p, tb, static_cast<uint32_t *>(wkey.p),
                                                static_cast<uint32_t *>(wkey_sorted.p), static_cast<int32_t *>(ids.p),
                                                static_cast<int32_t *>(perm.p), nnz, 0, bits, st));
    window_rows_kernel<<<ceil_div(nnz, 256), 256, 0, st>>>(static_cast<int32_t *>(perm.p), static_cast<int32_t *>(rowid.p),
                                                          nnz, static_cast<int32_t *>(w_row.p));
    SD_CUDA_TRY(cudaGetLastError());
    // runs of (window, row): head flags -> head positions
    const int64_t nflag = nnz > M ? nnz : M;
    if ((s = flag.get(nflag, "segment flags"))) return s;
    if ((s = nsel.get(sizeof(int32_t), "segment count"))) return s;
    if ((s = heads.get(4 * nnz, "segment heads"))) return s;
    window_headflag_kernel<<<ceil_div(nnz, 256), 256, 0, st>>>(static_cast<uint32_t *>(wkey_sorted.p),
                                                              static_cast<int32_t *>(w_row.p), nnz,
                                                              static_cast<uint8_t *>(flag.p));
    SD_CUDA_TRY(cudaGetLastError());
    cub::CountingInputIterator<int32_t> cnt(0);
    size_t tb2 = 0;
    SD_CUDA_TRY(cub::DeviceSelect::Flagged(nullptr, tb2, cnt, static_cast<uint8_t *>(flag.p), static_cast<int32_t *>(heads.p),
                                           static_cast<int32_t *>(nsel.p), static_cast<int>(nflag), st));
    TempBuf tmp2(st);
    if ((s = tmp2.get(tb2, "select scratch"))) return s;
    SD_CUDA_TRY(cub::DeviceSelect::Flagged(tmp2.p, tb2, cnt, static_cast<uint8_t *>(flag.p), static_cast<int32_t *>(heads.p),
                                           static_cast<int32_t *>(nsel.p), static_cast<int>(nnz), st));
    int32_t nheads = 0;
    SD_CUDA_TRY(cudaMemcpyAsync(&nheads, nsel.p, sizeof nheads, cudaMemcpyDeviceToHost, st));
    SD_CUDA_TRY(cudaStreamSynchronize(st));
    const int64_t S = E + nheads;
    l.S = S;

    TempBuf seg_start(st), seg_len(st), seg_row1(st), seg_key(st), seg_key_sorted(st), seg_ids(st), order(st), len2(st), dbounds(st);
    if ((s = seg_start.get(4 * S, "segment starts"))) return s;
    if ((s = seg_len.get(4 * S, "segment lengths"))) return s;
    if ((s = seg_row1.get(4 * S, "segment rows"))) return s;
    if ((s = seg_key.get(4 * S, "segment keys"))) return s;
    if ((s = seg_key_sorted.get(4 * S, "segment keys"))) return s;
    if ((s = seg_ids.get(4 * S, "segment ids"))) return s;
    if ((s = order.get(4 * S, "segment order"))) return s;
    if ((s = len2.get(4 * (S + 1), "segment lengths"))) return s;
    if ((s = l.w_ptr.get(4 * (S + 1), "segment pointers"))) return s;
    if ((s = l.w_seg_row.get(4 * (S + 1), "segment rows"))) return s;
    if (E > 0) {   // ids of the empty rows, ascending, at the front of the first ordering
        window_emptyflag_kernel<<<ceil_div(M, 256), 256, 0, st>>>(p->rowptr, M, static_cast<uint8_t *>(flag.p));
        SD_CUDA_TRY(cudaGetLastError());
        SD_CUDA_TRY(cub::DeviceSelect::Flagged(tmp2.p, tb2, cnt, static_cast<uint8_t *>(flag.p),
                                               static_cast<int32_t *>(seg_row1.p), static_cast<int32_t *>(nsel.p),
                                               static_cast<int>(M), st));
    }
    window_segments_kernel<<<ceil_div(S, 256), 256, 0, st>>>(
        p->rowptr, p->colind, static_cast<uint32_t *>(wkey_sorted.p), static_cast<int32_t *>(w_row.p),
        static_cast<int32_t *>(heads.p), wcols, kShortSegment, E, S, nnz, static_cast<int32_t *>(seg_start.p),
        static_cast<int32_t *>(seg_len.p), static_cast<int32_t *>(seg_row1.p), static_cast<uint32_t *>(seg_key.p));
    SD_CUDA_TRY(cudaGetLastError());
    // stable sort of the segments by (window, class)
    iota_kernel<<<ceil_div(S, 256), 256, 0, st>>>(static_cast<int32_t *>(seg_ids.p), S);
    SD_CUDA_TRY(cudaGetLastError());
    int kbits = 1;
    while ((1 << kbits) < 3 * W) ++kbits;
    size_t tb3 = 0;
    SD_CUDA_TRY(cub::DeviceRadixSort::SortPairs(nullptr, tb3, static_cast<uint32_t *>(seg_key.p),
                                                static_cast<uint32_t *>(seg_key_sorted.p),
                                                static_cast<int32_t *>(seg_ids.p), static_cast<int32_t *>(order.p), S, 0,
                                                kbits, st));
    TempBuf tmp3(st);
    if ((s = tmp3.get(tb3, "sort scratch"))) return s;
    SD_CUDA_TRY(cub::DeviceRadixSort::SortPairs(tmp3.p, tb3, static_cast<uint32_t *>(seg_key.p),
                                                static_cast<uint32_t *>(seg_key_sorted.p),
                                                static_cast<int32_t *>(seg_ids.p), static_cast<int32_t *>(order.p), S, 0,
                                                kbits, st));
    window_reorder_kernel<<<ceil_div(S, 256), 256, 0, st>>>(static_cast<int32_t *>(order.p),
                                                           static_cast<int32_t *>(seg_len.p),
                                                           static_cast<int32_t *>(seg_row1.p), S,
                                                           static_cast<int32_t *>(len2.p), l.w_seg_row.as<int32_t>());
    SD_CUDA_TRY(cudaGetLastError());
    SD_CUDA_TRY(cudaMemsetAsync(static_cast<int32_t *>(len2.p) + S, 0, 4, st));
    size_t tb4 = 0;
    SD_CUDA_TRY(cub::DeviceScan::ExclusiveSum(nullptr, tb4, static_cast<int32_t *>(len2.p), l.w_ptr.as<int32_t>(),
                                              static_cast<int>(S + 1), st));
    TempBuf tmp4(st);
    if ((s = tmp4.get(tb4, "scan scratch"))) return s;
    SD_CUDA_TRY(cub::DeviceScan::ExclusiveSum(tmp4.p, tb4, static_cast<int32_t *>(len2.p), l.w_ptr.as<int32_t>(),
                                              static_cast<int>(S + 1), st));
    if (p->dtype == SD_F32)
        window_gather_kernel<float><<<ceil_div(nnz, 256), 256, 0, st>>>(
            l.w_ptr.as<int32_t>(), static_cast<int32_t *>(order.p), static_cast<int32_t *>(seg_start.p), static_cast<int32_t *>(perm.p),
            p->colind, static_cast<const float *>(p->vals), S, nnz, l.w_col.as<int32_t>(), static_cast<float *>(l.w_vals.p));
    else
        window_gather_kernel<uint16_t><<<ceil_div(nnz, 256), 256, 0, st>>>(
            l.w_ptr.as<int32_t>(), static_cast<int32_t *>(order.p), static_cast<int32_t *>(seg_start.p), static_cast<int32_t *>(perm.p),
            p->colind, static_cast<const uint16_t *>(p->vals), S, nnz, l.w_col.as<int32_t>(), static_cast<uint16_t *>(l.w_vals.p));
    SD_CUDA_TRY(cudaGetLastError());
    if ((s = dbounds.get(sizeof(int64_t) * (3 * W + 1), "window bounds"))) return s;
    window_bounds_kernel<<<1, 256, 0, st>>>(static_cast<uint32_t *>(seg_key_sorted.p), S, 3 * W,
                                           static_cast<int64_t *>(dbounds.p));
    SD_CUDA_TRY(cudaGetLastError());
    l.bounds.assign(3 * W + 1, 0);
    SD_CUDA_TRY(cudaMemcpyAsync(l.bounds.data(), dbounds.p, sizeof(int64_t) * (3 * W + 1), cudaMemcpyDeviceToHost, st));
    SD_CUDA_TRY(cudaStreamSynchronize(st));
    return SD_OK;
}

sd_status_t inspect_tiles(const sd_plan *p, int32_t *host_out) {
    cudaStream_t st = nullptr;
    if (p->info.class_split) {   // no tiles: one entry per window, its first segment
        SegmentLists l(st);
        if (sd_status_t s = segment_lists(p, p->info.windows, l, st)) return s;
        for (int w = 0; w < p->info.windows; ++w) host_out[w] = static_cast<int32_t>(l.bounds[3 * w]);
        return SD_OK;
    }
    const int32_t ntiles = static_cast<int32_t>(p->info.num_tiles);
    TempBuf table(st);
    if (sd_status_t s = table.get(sizeof(int32_t) * (static_cast<size_t>(ntiles) + 1), "tile table")) return s;
    merge_table_kernel<<<ceil_div(ntiles + 1, 256), 256, 0, st>>>(p->rowptr, p->M, kMergeTile, ntiles, table.as<int32_t>());
    SD_CUDA_TRY(cudaGetLastError());
    SD_CUDA_TRY(cudaMemcpyAsync(host_out, table.p, sizeof(int32_t) * (static_cast<size_t>(ntiles) + 1), cudaMemcpyDeviceToHost, st));
    SD_CUDA_TRY(cudaStreamSynchronize(st));
    return SD_OK;
}

sd_status_t inspect_segments(const sd_plan *p, int W, int32_t *seg_ptr, int32_t *seg_row, int32_t *colind, void *vals, int64_t *win_seg) {
    cudaStream_t st = nullptr;
    SegmentLists l(st);
    if (sd_status_t s = segment_lists(p, W, l, st)) return s;
    const size_t es = p->dtype == SD_F32 ? 4 : 2;
    if (seg_ptr) SD_CUDA_TRY(cudaMemcpyAsync(seg_ptr, l.w_ptr.p, 4 * (l.S + 1), cudaMemcpyDeviceToHost, st));
    if (seg_row) SD_CUDA_TRY(cudaMemcpyAsync(seg_row, l.w_seg_row.p, 4 * l.S, cudaMemcpyDeviceToHost, st));
    if (colind) SD_CUDA_TRY(cudaMemcpyAsync(colind, l.w_col.p, 4 * p->nnz, cudaMemcpyDeviceToHost, st));
    if (vals) SD_CUDA_TRY(cudaMemcpyAsync(vals, l.w_vals.p, es * p->nnz, cudaMemcpyDeviceToHost, st));
    if (win_seg) {
        for (int k = 0; k < 3 * W; ++k) win_seg[k] = l.bounds[k];
        win_seg[3 * W] = l.S;
    }
    SD_CUDA_TRY(cudaStreamSynchronize(st));
    return SD_OK;
}

// (row, window) pairs of the nonzeros; every row without nonzeros is a segment too.
__global__ void __launch_bounds__(256)
segment_count_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colind, int64_t M, int32_t wcols,
                     unsigned long long *__restrict__ out) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
    unsigned long long n = 0;
    for (int64_t row = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; row < M; row += warps) {
        const int p0 = rowptr[row], p1 = rowptr[row + 1];
        if (p0 == p1) n += lane == 0;
        for (int p = p0 + lane; p < p1; p += 32) n += p == p0 || colind[p] / wcols != colind[p - 1] / wcols;
    }
    for (int d = 16; d >= 1; d >>= 1) n += __shfl_xor_sync(0xffffffffu, n, d);
    if (lane == 0 && n) atomicAdd(out, n);
}

sd_status_t count_segments(const sd_plan *p, int W, int64_t *count, cudaStream_t st) {
    TempBuf acc(st);
    unsigned long long n = 0;
    if (sd_status_t s = acc.get(sizeof n, "segment count")) return s;
    SD_CUDA_TRY(cudaMemsetAsync(acc.p, 0, sizeof n, st));
    segment_count_kernel<<<148 * 8, 256, 0, st>>>(p->rowptr, p->colind, p->M, static_cast<int32_t>((p->K + W - 1) / W), acc.as<unsigned long long>());
    SD_CUDA_TRY(cudaGetLastError());
    SD_CUDA_TRY(cudaMemcpyAsync(&n, acc.p, sizeof n, cudaMemcpyDeviceToHost, st));
    SD_CUDA_TRY(cudaStreamSynchronize(st));
    *count = static_cast<int64_t>(n);
    return SD_OK;
}

}  // namespace sd
