// Structure scan of plan creation (paper Sec. 3.1, intrinsic pattern features; integers only): row-length histogram and
// moments, span, gap, diagonal, order, and the occupied 16x16 blocks with their fill.
//
// One pass over the column indices.  A block-row (16 rows) is contiguous in colind, so its occupied blocks are counted in
// a table in shared memory keyed by block column, instead of by sorting a 64-bit block key per nonzero (1.9 M nonzeros:
// key pass, radix sort, run-length encoding and fill count took 290 us and 39 MB of scratch).  A warp takes a block-row of
// up to kSmallNnz nonzeros; longer ones go to a list that a second kernel works off with a CTA each, and those whose
// blocks fit neither table to a third, cut by column range.
#include <algorithm>

#include "sd_plan.cuh"

namespace sd {

namespace {

constexpr int kSmallNnz = 512, kSmallSlots = 1024;     // warp table: at most half full
constexpr int kLargeNnz = 8192, kLargeSlots = 32768;   // CTA table: hashed up to kLargeNnz nonzeros, else one counter per block column
constexpr int kScanWarps = 8, kLargeThreads = 512;

__device__ __forceinline__ int hist_bin(long long v) { return v <= 0 ? 0 : 64 - __clzll(v); }

// Counters of one CTA in shared memory, added to the global ones when it ends.
struct ScanShared {
    unsigned long long sum[16];
    unsigned long long mx[2];     // longest row, largest span
    unsigned int row_hist[32], blk_hist[16], len_hist[256];
};
enum { S_R2, S_EMPTY, S_SPAN, S_GAP, S_DIAG, S_UNSORTED, S_LONG, S_NNZ_LONG, S_CHUNKS, S_GIANTS, S_DENSE, S_BLOCKS, S_CHUNKS2, S_CHUNKS4, S_COUNT };

__device__ void scan_clear(ScanShared &s) {
    for (int i = threadIdx.x; i < static_cast<int>(sizeof(ScanShared) / 4); i += blockDim.x) reinterpret_cast<unsigned int *>(&s)[i] = 0;
    __syncthreads();
}

__device__ void scan_flush(ScanShared &s, ScanAccum *out) {
    __syncthreads();
    unsigned long long *const sums[S_COUNT] = {&out->sum_r2, &out->empty_rows, &out->sum_span, &out->sum_gap, &out->diag,
                                          &out->unsorted_rows, &out->long_rows, &out->nnz_long_rows, &out->chunks_long,
                                          &out->giants, &out->nnz_dense_blocks, &out->nnzb, &out->chunks_long2, &out->chunks_long4};
    const int t = threadIdx.x;
    if (t < S_COUNT && s.sum[t]) atomicAdd(sums[t], s.sum[t]);
    if (t == 16 && s.mx[0]) atomicMax(&out->max_r, s.mx[0]);
    if (t == 17 && s.mx[1]) atomicMax(&out->max_span, s.mx[1]);
    if (t >= 32 && t < 64 && s.row_hist[t - 32]) atomicAdd(&out->row_hist[t - 32], static_cast<unsigned long long>(s.row_hist[t - 32]));
    if (t >= 64 && t < 73 && s.blk_hist[t - 64]) atomicAdd(&out->blk_hist[t - 64], static_cast<unsigned long long>(s.blk_hist[t - 64]));
    for (int i = t; i < 256; i += blockDim.x)
        if (s.len_hist[i]) atomicAdd(&out->len_hist[i], static_cast<unsigned long long>(s.len_hist[i]));
}

__device__ __forceinline__ void count_long_row(ScanShared &s, long long r) {
    const unsigned long long chunks = static_cast<unsigned long long>((r + kChunkNnz - 1) / kChunkNnz);
    atomicAdd(&s.sum[S_LONG], 1ull);
    atomicAdd(&s.sum[S_NNZ_LONG], static_cast<unsigned long long>(r));
    atomicAdd(&s.sum[S_CHUNKS], chunks);
    atomicAdd(&s.sum[S_CHUNKS2], (chunks + 1) / 2);
    atomicAdd(&s.sum[S_CHUNKS4], (chunks + 3) / 4);
    if (chunks > kGiantChunks) atomicAdd(&s.sum[S_GIANTS], 1ull);
}

// The rows of a block-row, one per lane (`mine`: the lane has a row), summed over the warp before they reach shared memory.
__device__ void count_rows(ScanShared &s, bool mine, int r, unsigned span, bool unsorted) {
    constexpr unsigned FULL = 0xffffffffu;
    const bool some = mine && r > 0;
    if (mine) {
        atomicAdd(&s.row_hist[hist_bin(r)], 1u);
        if (r < 256) atomicAdd(&s.len_hist[r], 1u);
        else count_long_row(s, r);
    }
    unsigned long long r2 = some ? static_cast<unsigned long long>(r) * static_cast<unsigned long long>(r) : 0, sp = some ? span : 0;
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
        r2 += __shfl_xor_sync(FULL, r2, d);
        sp += __shfl_xor_sync(FULL, sp, d);
    }
    const unsigned mr = __reduce_max_sync(FULL, some ? static_cast<unsigned>(r) : 0u), ms = __reduce_max_sync(FULL, some ? span : 0u);
    const int empty = __popc(__ballot_sync(FULL, mine && r == 0)), full = __popc(__ballot_sync(FULL, some)),
              uns = __popc(__ballot_sync(FULL, some && unsorted));
    if ((threadIdx.x & 31) == 0) {
        if (empty) atomicAdd(&s.sum[S_EMPTY], static_cast<unsigned long long>(empty));
        if (full) {
            atomicAdd(&s.sum[S_R2], r2);
            atomicAdd(&s.sum[S_SPAN], sp);
            atomicAdd(&s.sum[S_GAP], sp - full);
            atomicMax(&s.mx[0], static_cast<unsigned long long>(mr));
            atomicMax(&s.mx[1], static_cast<unsigned long long>(ms));
            if (uns) atomicAdd(&s.sum[S_UNSORTED], static_cast<unsigned long long>(uns));
        }
    }
}

// A block of c entries.
__device__ __forceinline__ void count_block(ScanShared &s, int c) {
    atomicAdd(&s.blk_hist[min(hist_bin(c) - 1, 8)], 1u);
    if (c >= 128) atomicAdd(&s.sum[S_DENSE], static_cast<unsigned long long>(c));
}

// Adds n entries to block column j of a hash table with `mask` + 1 slots (never full).
__device__ __forceinline__ void table_add(int *key, int *cnt, unsigned mask, int j, int n) {
    unsigned h = (static_cast<unsigned>(j) * 2654435761u) >> 7 & mask;
    for (;;) {
        const int was = atomicCAS(key + h, -1, j);
        if (was == -1 || was == j) break;
        h = (h + 1) & mask;
    }
    atomicAdd(cnt + h, n);
}

// What the scan needs to know of one nonzero and its neighbours in the row [b, e).
struct Entry {
    int c;
    bool starts, ends, out_of_order;   // begins / ends an ascending run of its row; not below its successor in the row
};
__device__ __forceinline__ Entry look(const int32_t *__restrict__ colind, int64_t p, int64_t b, int64_t e) {
    Entry x;
    x.c = __ldg(colind + p);
    const bool first = p == b, last = p + 1 == e;
    const int prev = first ? 0 : __ldg(colind + p - 1), next = last ? 0 : __ldg(colind + p + 1);
    x.starts = first || prev > x.c;
    x.ends = last || next < x.c;
    x.out_of_order = !last && next <= x.c;
    return x;
}
// Runs of equal block columns among the active lanes' consecutive entries (the active lanes are the low ones): the
// leader's run length, 0 for the others.
__device__ __forceinline__ int run_of(int j, bool in) {
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int pj = __shfl_up_sync(FULL, j, 1);
    const unsigned active = __ballot_sync(FULL, in);
    const unsigned heads = __ballot_sync(FULL, in && (lane == 0 || pj != j));
    if (!((heads >> lane) & 1u)) return 0;
    const unsigned above = lane == 31 ? 0u : heads & (FULL << (lane + 1));
    return (above ? __ffs(above) - 1 : 32 - __clz(active)) - lane;
}

// ---- first kernel: a warp per block-row ---------------------------------------------------------------
struct WarpTable {
    int key[kSmallSlots], cnt[kSmallSlots];
    int bound[17], lo[16], hi[16];
    unsigned uns;
};

__global__ void __launch_bounds__(32 * kScanWarps)
scan_small_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colind, int64_t M, int32_t *__restrict__ large,
                  ScanAccum *__restrict__ out) {
    extern __shared__ __align__(16) unsigned char smem[];
    ScanShared &s = *reinterpret_cast<ScanShared *>(smem);
    WarpTable &w = reinterpret_cast<WarpTable *>(smem + sizeof(ScanShared))[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    scan_clear(s);
    const long long last = __ldg(rowptr + M);
    if (blockIdx.x == 0 && threadIdx.x == 0) out->nnz = last;
    if (last < 0) return;   // the host refuses such a pattern
    const int64_t Mb = (M + 15) / 16, warps = static_cast<int64_t>(gridDim.x) * kScanWarps;
    unsigned long long diag = 0;
    for (int64_t I = static_cast<int64_t>(blockIdx.x) * kScanWarps + (threadIdx.x >> 5); I < Mb; I += warps) {
        const int64_t r0 = I * 16;
        if (lane < 17) w.bound[lane] = __ldg(rowptr + min(r0 + lane, M));
        __syncwarp();
        const int64_t b = w.bound[0], e = w.bound[16];
        if (e - b > kSmallNnz) {
            if (lane == 0) large[atomicAdd(&out->large, 1u)] = static_cast<int32_t>(I);
            __syncwarp();
            continue;
        }
        const int n = static_cast<int>(e - b);
        unsigned slots = 32;
        while (slots < 2u * static_cast<unsigned>(n)) slots <<= 1;
        for (unsigned i = lane; i < slots; i += 32) {
            w.key[i] = -1;
            w.cnt[i] = 0;
        }
        if (lane < 16) {
            w.lo[lane] = INT_MAX;
            w.hi[lane] = INT_MIN;
        }
        if (lane == 0) w.uns = 0;
        __syncwarp();
        int r = 0;   // row of this lane's entry: it only moves forward
        for (int i0 = 0; i0 < n; i0 += 32) {
            const int64_t p = b + i0 + lane;
            const bool in = p < e;
            int j = -1;
            if (in) {
                while (p >= w.bound[r + 1]) ++r;
                const Entry x = look(colind, p, w.bound[r], w.bound[r + 1]);
                j = x.c >> 4;
                diag += (x.c == r0 + r);
                if (x.starts) atomicMin(&w.lo[r], x.c);
                if (x.ends) atomicMax(&w.hi[r], x.c);
                if (x.out_of_order) atomicOr(&w.uns, 1u << r);
            }
            const int run = run_of(j, in);
            if (run) table_add(w.key, w.cnt, slots - 1, j, run);
        }
        __syncwarp();
        const bool mine = lane < 16 && r0 + lane < M;
        const int len = mine ? w.bound[lane + 1] - w.bound[lane] : 0;
        count_rows(s, mine, len, len > 0 ? static_cast<unsigned>(w.hi[lane]) - static_cast<unsigned>(w.lo[lane]) + 1u : 0u,
                   (w.uns >> (lane & 15)) & 1u);
        int blocks = 0;
        for (unsigned i = lane; i < slots; i += 32)
            if (const int c = w.cnt[i]) {
                ++blocks;
                count_block(s, c);
            }
        blocks = __reduce_add_sync(0xffffffffu, blocks);
        if (lane == 0 && blocks) atomicAdd(&s.sum[S_BLOCKS], static_cast<unsigned long long>(blocks));
        __syncwarp();
    }
    if (diag) atomicAdd(&s.sum[S_DIAG], diag);
    scan_flush(s, out);
}

// ---- second kernel: a CTA per listed block-row ------------------------------------------------------------
struct CtaTable {
    int bound[17], lo[16], hi[16];
    unsigned uns;
    int cnt[kLargeSlots];   // hashed: the first half are keys
};

__global__ void __launch_bounds__(kLargeThreads)
scan_large_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colind, int64_t M, int64_t Kb,
                  const int32_t *__restrict__ large, int32_t *__restrict__ huge, ScanAccum *__restrict__ out) {
    extern __shared__ __align__(16) unsigned char smem[];
    ScanShared &s = *reinterpret_cast<ScanShared *>(smem);
    CtaTable &w = *reinterpret_cast<CtaTable *>(smem + sizeof(ScanShared));
    const unsigned count = out->large;
    if (blockIdx.x >= count) return;
    scan_clear(s);
    unsigned long long diag = 0, blocks = 0;
    for (unsigned k = blockIdx.x; k < count; k += gridDim.x) {
        const int64_t I = large[k], r0 = I * 16;
        if (threadIdx.x < 17) w.bound[threadIdx.x] = __ldg(rowptr + min(r0 + threadIdx.x, M));
        if (threadIdx.x < 16) {
            w.lo[threadIdx.x] = INT_MAX;
            w.hi[threadIdx.x] = INT_MIN;
        }
        if (threadIdx.x == 0) w.uns = 0;
        __syncthreads();
        const int64_t b = w.bound[0], e = w.bound[16], n = e - b;
        const bool dense = Kb <= kLargeSlots, hashed = !dense && n <= kLargeNnz;
        unsigned slots = 64;
        if (hashed) while (slots < 2u * static_cast<unsigned>(n)) slots <<= 1;
        int *const key = w.cnt, *const cnt = dense ? w.cnt : w.cnt + kLargeSlots / 2;
        const unsigned used = dense ? static_cast<unsigned>(Kb) : (hashed ? slots : 0u);
        for (unsigned i = threadIdx.x; i < used; i += kLargeThreads) {
            cnt[i] = 0;
            if (hashed) key[i] = -1;
        }
        __syncthreads();
        int r = 0;
        for (int64_t i0 = 0; i0 < n; i0 += kLargeThreads) {
            const int64_t p = b + i0 + threadIdx.x;
            const bool in = p < e;
            int j = -1;
            if (in) {
                while (p >= w.bound[r + 1]) ++r;
                const Entry x = look(colind, p, w.bound[r], w.bound[r + 1]);
                j = x.c >> 4;
                diag += (x.c == r0 + r);
                if (x.starts) atomicMin(&w.lo[r], x.c);
                if (x.ends) atomicMax(&w.hi[r], x.c);
                if (x.out_of_order) atomicOr(&w.uns, 1u << r);
            }
            const int run = run_of(j, in);
            if (run && dense && j >= 0 && j < Kb) atomicAdd(cnt + j, run);
            if (run && hashed) table_add(key, cnt, slots - 1, j, run);
        }
        __syncthreads();
        if (threadIdx.x < 32) {
            const int t = threadIdx.x;
            const bool mine = t < 16 && r0 + t < M;
            const int len = mine ? w.bound[t + 1] - w.bound[t] : 0;
            count_rows(s, mine, len, len > 0 ? static_cast<unsigned>(w.hi[t]) - static_cast<unsigned>(w.lo[t]) + 1u : 0u, (w.uns >> (t & 15)) & 1u);
        }
        if (!dense && !hashed && threadIdx.x == 0)   // bit 31: rows out of order, every column range has to look at all of them
            huge[atomicAdd(&out->huge, 1u)] = static_cast<int32_t>(static_cast<uint32_t>(I) | (w.uns ? 0x80000000u : 0u));
        for (unsigned i = threadIdx.x; i < used; i += kLargeThreads)
            if (const int c = cnt[i]) {
                ++blocks;
                count_block(s, c);
            }
        __syncthreads();
    }
    if (diag) atomicAdd(&s.sum[S_DIAG], diag);
    if (blocks) atomicAdd(&s.sum[S_BLOCKS], blocks);
    scan_flush(s, out);
}

// ---- third kernel: blocks of the remaining block-rows, a CTA per (block-row, range of kLargeSlots block columns) -----------
__global__ void __launch_bounds__(kLargeThreads)
scan_huge_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colind, int64_t M, int64_t Kb,
                 const int32_t *__restrict__ huge, ScanAccum *__restrict__ out) {
    extern __shared__ __align__(16) unsigned char smem[];
    ScanShared &s = *reinterpret_cast<ScanShared *>(smem);
    CtaTable &w = *reinterpret_cast<CtaTable *>(smem + sizeof(ScanShared));
    const int64_t ranges = (Kb + kLargeSlots - 1) / kLargeSlots, items = static_cast<int64_t>(out->huge) * ranges;
    if (blockIdx.x >= items) return;
    scan_clear(s);
    unsigned long long blocks = 0;
    for (int64_t k = blockIdx.x; k < items; k += gridDim.x) {
        const uint32_t entry = static_cast<uint32_t>(huge[k / ranges]);
        const int64_t r0 = static_cast<int64_t>(entry & 0x7FFFFFFFu) * 16, j0 = k % ranges * kLargeSlots;
        const bool sorted = (entry >> 31) == 0;
        const int used = static_cast<int>(min(static_cast<int64_t>(kLargeSlots), Kb - j0));
        for (int i = threadIdx.x; i < used; i += kLargeThreads) w.cnt[i] = 0;
        if (threadIdx.x < 16) {   // the part of each row whose columns can fall in this range
            int b = __ldg(rowptr + min(r0 + threadIdx.x, M)), e = __ldg(rowptr + min(r0 + threadIdx.x + 1, M));
            if (sorted) {
                const int64_t want[2] = {j0 * 16, (j0 + used) * 16};
                int at[2];
                for (int q = 0; q < 2; ++q) {
                    int lo = b, hi = e;
                    while (lo < hi) {
                        const int mid = lo + ((hi - lo) >> 1);
                        if (__ldg(colind + mid) < want[q]) lo = mid + 1;
                        else hi = mid;
                    }
                    at[q] = lo;
                }
                b = at[0];
                e = at[1];
            }
            w.lo[threadIdx.x] = b;
            w.hi[threadIdx.x] = e;
        }
        __syncthreads();
        for (int r = 0; r < 16; ++r) {
            const int64_t b = w.lo[r], e = w.hi[r];
            for (int64_t i0 = b; i0 < e; i0 += kLargeThreads) {
                const int64_t p = i0 + threadIdx.x;
                const bool in = p < e;
                const int j = in ? (__ldg(colind + p) >> 4) : -1;
                const int run = run_of(j, in);
                if (run && j >= j0 && j < j0 + used) atomicAdd(w.cnt + (j - j0), run);
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < used; i += kLargeThreads)
            if (const int c = w.cnt[i]) {
                ++blocks;
                count_block(s, c);
            }
        __syncthreads();
    }
    if (blocks) atomicAdd(&s.sum[S_BLOCKS], blocks);
    scan_flush(s, out);
}

// CSR validation: rowptr[0] == 0, rowptr non-decreasing, 0 <= col < K.
__global__ void validate_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colind, int64_t M, int64_t K,
                                int64_t nnz, ScanAccum *__restrict__ out) {
    unsigned long long bad = 0;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    const int64_t i0 = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    for (int64_t i = i0; i < M; i += stride) bad += (rowptr[i + 1] < rowptr[i]);
    for (int64_t p = i0; p < nnz; p += stride) bad += (colind[p] < 0 || colind[p] >= K);
    if (i0 == 0) bad += (rowptr[0] != 0);
    if (bad) atomicAdd(&out->bad_csr, bad);
}

}  // namespace

cudaError_t validate_csr(const int32_t *rowptr, const int32_t *colind, int64_t M, int64_t K, int64_t nnz, ScanAccum *out, cudaStream_t st) {
    validate_kernel<<<148 * 8, 256, 0, st>>>(rowptr, colind, M, K, nnz, out);
    return cudaGetLastError();
}

cudaError_t scan_structure(const int32_t *rowptr, const int32_t *colind, int64_t M, int64_t K, ScanAccum *out, cudaStream_t st) {
    const int64_t Mb = (M + 15) / 16, Kb = (K + 15) / 16;
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(ScanAccum), st);
    if (e != cudaSuccess || M == 0) return e;
    void *lists = nullptr;   // [Mb] block-rows for the second kernel, [Mb] for the third
    if ((e = pool_alloc(&lists, sizeof(int32_t) * 2 * Mb, st)) != cudaSuccess) return e;
    int32_t *large = static_cast<int32_t *>(lists), *huge = large + Mb;
    const int small_smem = static_cast<int>(sizeof(ScanShared) + kScanWarps * sizeof(WarpTable));
    const int large_smem = static_cast<int>(sizeof(ScanShared) + sizeof(CtaTable));
    static std::atomic<int> attr_set[kMaxDevices];
    const int dev = current_device();
    if (dev >= kMaxDevices || !attr_set[dev].load(std::memory_order_acquire)) {
        if ((e = cudaFuncSetAttribute(scan_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, small_smem)) != cudaSuccess ||
            (e = cudaFuncSetAttribute(scan_large_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, large_smem)) != cudaSuccess ||
            (e = cudaFuncSetAttribute(scan_huge_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, large_smem)) != cudaSuccess) {
            cudaFreeAsync(lists, st);
            return e;
        }
        if (dev < kMaxDevices) attr_set[dev].store(1, std::memory_order_release);
    }
    const int sms = sm_count_cached();
    const int64_t want = (Mb + kScanWarps - 1) / kScanWarps;
    scan_small_kernel<<<static_cast<unsigned>(std::min<int64_t>(want, 3 * sms)), 32 * kScanWarps, small_smem, st>>>(rowptr, colind, M, large, out);
    e = cudaGetLastError();
    if (e == cudaSuccess) {
        scan_large_kernel<<<static_cast<unsigned>(std::min<int64_t>(Mb, sms)), kLargeThreads, large_smem, st>>>(rowptr, colind, M, Kb, large, huge, out);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && Kb > kLargeSlots) {
        scan_huge_kernel<<<static_cast<unsigned>(sms), kLargeThreads, large_smem, st>>>(rowptr, colind, M, Kb, huge, out);
        e = cudaGetLastError();
    }
    cudaFreeAsync(lists, st);
    return e;
}

}  // namespace sd
