// Representation builders of plan creation.
#include <algorithm>

#include <cub/cub.cuh>

#include "sd_plan.cuh"

namespace sd {

// =====================================================================================
// memory
// =====================================================================================
static std::mutex g_pool_mutex;
static std::atomic<cudaMemPool_t> g_pools[kMaxDevices];

cudaError_t pool_alloc(void **out, size_t bytes, cudaStream_t st) {
    *out = nullptr;
    if (bytes == 0) bytes = 16;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= kMaxDevices) return cudaMallocAsync(out, bytes, st);
    cudaMemPool_t pool = g_pools[dev].load(std::memory_order_acquire);
    if (!pool) {
        std::lock_guard<std::mutex> lock(g_pool_mutex);
        pool = g_pools[dev].load(std::memory_order_acquire);
        if (!pool) {
            cudaMemPoolProps props{};
            props.allocType = cudaMemAllocationTypePinned;
            props.location.type = cudaMemLocationTypeDevice;
            props.location.id = dev;
            uint64_t keep = kPoolKeep;
            if ((e = cudaMemPoolCreate(&pool, &props)) != cudaSuccess) return e;
            if ((e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep)) != cudaSuccess) return e;
            g_pools[dev].store(pool, std::memory_order_release);
        }
    }
    return cudaMallocFromPoolAsync(out, bytes, pool, st);
}

// Gives back what the pools hold beyond the memory in use.
sd_status_t pool_release() {
    int prev = 0;
    SD_CUDA_TRY(cudaGetDevice(&prev));
    sd_status_t s = SD_OK;
    for (int dev = 0; dev < kMaxDevices && s == SD_OK; ++dev) {
        cudaMemPool_t pool = g_pools[dev].load(std::memory_order_acquire);
        if (!pool) continue;
        cudaError_t e = cudaSetDevice(dev);
        if (e == cudaSuccess) e = cudaDeviceSynchronize();   // a block that was freed in stream order leaves the pool once the stream got there
        if (e == cudaSuccess) e = cudaMemPoolTrimTo(pool, 0);
        if (e != cudaSuccess) s = cuda_fail(e, "releasing unused memory");
    }
    cudaSetDevice(prev);
    return s;
}

sd_status_t dev_alloc_bytes(sd_plan *p, void **out, size_t bytes, const char *what, cudaStream_t st) {
    if (bytes == 0) bytes = 16;
    const cudaError_t e = pool_alloc(out, bytes, st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        *out = nullptr;
        set_error(SD_ERR_ALLOC, "allocating %zu bytes for %s failed: %s", bytes, what, cudaGetErrorString(e));
        return SD_ERR_ALLOC;
    }
    if (p) {
        p->owned += static_cast<int64_t>(bytes);
        p->allocs.push_back(*out);
    }
    return SD_OK;
}

static std::mutex g_block_mutex;
static std::vector<void *> g_blocks;
constexpr size_t kHostBlocks = 8;

HostBlock::HostBlock() {
    {
        std::lock_guard<std::mutex> lock(g_block_mutex);
        if (!g_blocks.empty()) {
            p = g_blocks.back();
            g_blocks.pop_back();
        }
    }
    if (!p && cudaHostAlloc(&p, kBytes, cudaHostAllocPortable) != cudaSuccess) {
        cudaGetLastError();
        p = nullptr;
    }
}

HostBlock::~HostBlock() {
    if (!p) return;
    {
        std::lock_guard<std::mutex> lock(g_block_mutex);
        if (g_blocks.size() < kHostBlocks) {
            g_blocks.push_back(p);
            return;
        }
    }
    cudaFreeHost(p);
}

void host_blocks_release() {
    std::lock_guard<std::mutex> lock(g_block_mutex);
    for (void *p : g_blocks) cudaFreeHost(p);
    g_blocks.clear();
}

// =====================================================================================
// schedule of the merge and hybrid families
// =====================================================================================
// Rows by length: a stable counting sort on the key 0 (heavy) or T - length, one pass over the row pointers to count and one
// to place.  The row-length histogram of the scan gives every key's first position, so the only scan left is over the
// tiles of one key.  A tile is PER x 256 rows: large ones mean fewer counters, small ones more CTAs and shorter chains (65,536 rows: placing 13 us
// with PER = 8, 6 with 2).  The kernels' launches overlap.
constexpr int kSortWarps = 8, kSortBins = kHybridHeavyMax + 1;

__device__ __forceinline__ int sort_key(int len, int T) { return len >= T ? 0 : T - len; }

// Keys of a warp's rows (PER per lane), counted into its bins.
template <int PER>
__device__ __forceinline__ void count_keys(const int32_t *__restrict__ rowptr, int64_t M, int64_t base, int T, int (&key)[PER], int *bins) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int64_t r = base + i * 32 + lane;
        key[i] = r < M ? sort_key(__ldg(rowptr + r + 1) - __ldg(rowptr + r), T) : -1;
    }
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const unsigned same = __match_any_sync(0xffffffffu, key[i]);
        if (key[i] >= 0 && lane == __ffs(same) - 1) bins[key[i]] += __popc(same);
        __syncwarp();
    }
}

template <int PER>
__global__ void __launch_bounds__(32 * kSortWarps)
sort_count_kernel(const int32_t *__restrict__ rowptr, int64_t M, int T, int32_t ntiles, int32_t *__restrict__ hist) {
    __shared__ int bins[kSortWarps][kSortBins];
    overlap_next();
    for (int i = threadIdx.x; i < kSortWarps * kSortBins; i += blockDim.x) (&bins[0][0])[i] = 0;
    __syncthreads();
    int key[PER];
    count_keys<PER>(rowptr, M, static_cast<int64_t>(blockIdx.x) * PER * 256 + (threadIdx.x >> 5) * (PER * 32), T, key, bins[threadIdx.x >> 5]);
    __syncthreads();
    for (int k = threadIdx.x; k <= T; k += blockDim.x) {
        int n = 0;
#pragma unroll
        for (int w = 0; w < kSortWarps; ++w) n += bins[w][k];
        hist[static_cast<int64_t>(k) * ntiles + blockIdx.x] = n;
    }
}

struct SortBases {
    int32_t first[kSortBins];
};

// One warp per key: counts become first positions.
__global__ void __launch_bounds__(256)
sort_prefix_kernel(const SortBases b, int T, int32_t ntiles, int32_t *__restrict__ hist) {
    const int k = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    overlap_next();
    overlap_wait();
    if (k > T) return;
    int run = b.first[k];
    for (int t0 = 0; t0 < ntiles; t0 += 32) {
        int32_t *h = hist + static_cast<int64_t>(k) * ntiles + t0 + lane;
        const int n = t0 + lane < ntiles ? *h : 0;
        int x = n;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, d);
            if (lane >= d) x += y;
        }
        if (t0 + lane < ntiles) *h = run + x - n;
        run += __shfl_sync(0xffffffffu, x, 31);
    }
}

// Places the rows; a light row's descriptor holds everything its first gather needs, in one 16-byte load.
template <int PER>
__global__ void __launch_bounds__(32 * kSortWarps)
sort_place_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colind, int64_t M, int T, int32_t ntiles,
                  const int32_t *__restrict__ hist, int32_t nl, int32_t *__restrict__ rows, int4 *__restrict__ desc) {
    __shared__ int bins[kSortWarps][kSortBins];
    overlap_next();
    for (int i = threadIdx.x; i < kSortWarps * kSortBins; i += blockDim.x) (&bins[0][0])[i] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t base = static_cast<int64_t>(blockIdx.x) * PER * 256 + warp * (PER * 32);
    int key[PER];
    count_keys<PER>(rowptr, M, base, T, key, bins[warp]);
    overlap_wait();
    __syncthreads();
    for (int k = threadIdx.x; k <= T; k += blockDim.x) {   // counts of the warps become their first positions
        int at = hist[static_cast<int64_t>(k) * ntiles + blockIdx.x];
#pragma unroll
        for (int w = 0; w < kSortWarps; ++w) {
            const int n = bins[w][k];
            bins[w][k] = at;
            at += n;
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const unsigned same = __match_any_sync(0xffffffffu, key[i]);
        int at = 0;
        if (key[i] >= 0) at = bins[warp][key[i]] + __popc(same & ((1u << lane) - 1u));
        __syncwarp();
        if (key[i] >= 0 && lane == __ffs(same) - 1) bins[warp][key[i]] += __popc(same);
        __syncwarp();
        if (key[i] < 0) continue;
        const int64_t r = base + i * 32 + lane;
        rows[at] = static_cast<int32_t>(r);
        if (at >= nl) {
            const int32_t p0 = __ldg(rowptr + r), len = __ldg(rowptr + r + 1) - p0;
            desc[at - nl] = make_int4(static_cast<int32_t>(r), p0, len > 0 ? __ldg(colind + p0) : 0, len);
        }
    }
}

// Chunk and item pointers of the heavy rows and the list of the rows of very many items: one CTA walks the rows (a few
// thousand).  chunk_off / item_off: counts before every (row, window) pair; null with one window, where a row's length says
// how many it has.
__global__ void __launch_bounds__(1024)
chunk_ptr_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ rows, const int32_t *__restrict__ chunk_off,
                 const int32_t *__restrict__ item_off, int32_t W, int32_t F, int64_t nl, int32_t *__restrict__ chunk_ptr,
                 int32_t *__restrict__ item_ptr, int32_t *__restrict__ giant, int32_t *__restrict__ ngiant) {
    using Scan = cub::BlockScan<int, 1024>;
    __shared__ typename Scan::TempStorage tmp;
    overlap_next();
    overlap_wait();
    int c = 0, m = 0, g = 0;   // chunks, items and listed rows before this step, the same in all threads
    for (int64_t i0 = 0; i0 < nl; i0 += 1024) {
        const int64_t i = i0 + threadIdx.x;
        int n = 0, k = 0;
        if (i < nl) {
            if (chunk_off) {
                n = chunk_off[(i + 1) * W] - chunk_off[i * W];
                k = item_off[(i + 1) * W] - item_off[i * W];
            } else {
                const int32_t r = rows[i];
                n = (__ldg(rowptr + r + 1) - __ldg(rowptr + r) + kChunkNnz - 1) / kChunkNnz;
                k = (n + F - 1) / F;
            }
        }
        int before, total, ibefore, itotal, listed, all;
        Scan(tmp).ExclusiveSum(n, before, total);
        __syncthreads();
        Scan(tmp).ExclusiveSum(k, ibefore, itotal);
        __syncthreads();
        Scan(tmp).ExclusiveSum(k > kGiantChunks ? 1 : 0, listed, all);
        __syncthreads();
        if (i < nl) {
            chunk_ptr[i] = c + before;
            item_ptr[i] = m + ibefore;
            if (k > kGiantChunks) giant[g + listed] = static_cast<int32_t>(i);
        }
        c += total;
        m += itotal;
        g += all;
    }
    if (threadIdx.x == 0) {
        chunk_ptr[nl] = c;
        item_ptr[nl] = m;
        *ngiant = g;
    }
}

// One window: the items in row order.  A warp per heavy row.
__global__ void __launch_bounds__(256)
items_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ rows, const int32_t *__restrict__ chunk_ptr,
             const int32_t *__restrict__ item_ptr, int32_t F, int64_t nl, int4 *__restrict__ items) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
    overlap_wait();
    for (int64_t i = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; i < nl; i += warps) {
        const int32_t r = rows[i], p0 = __ldg(rowptr + r), p1 = __ldg(rowptr + r + 1), c0 = chunk_ptr[i], m0 = item_ptr[i], m1 = item_ptr[i + 1];
        for (int32_t m = m0 + lane; m < m1; m += 32) {
            const int32_t x = p0 + (m - m0) * F * kChunkNnz;
            items[m] = make_int4(m1 - m0 == 1 ? r | static_cast<int32_t>(0x80000000u) : m, x, c0 + (m - m0) * F, min(F * kChunkNnz, p1 - x));
        }
    }
}

__device__ __forceinline__ int32_t first_not_below(const int32_t *__restrict__ colind, int32_t lo, int32_t hi, int64_t col) {
    while (lo < hi) {
        const int32_t mid = lo + ((hi - lo) >> 1);
        if (colind[mid] < col) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// Column windows, one thread per (heavy row i, window w): the nonzeros of the row whose columns fall in the window are a
// contiguous range (columns ascend); counts its chunks into a row-major and a window-major table.
__global__ void __launch_bounds__(256)
window_count_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colind, const int32_t *__restrict__ rows,
                    int64_t nl, int32_t W, int32_t F, int64_t wcols, int32_t *__restrict__ start, int32_t *__restrict__ chunks,
                    int32_t *__restrict__ items, int32_t *__restrict__ items_by_window) {
    const int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (t > nl * W) return;
    if (t == nl * W) {
        chunks[t] = 0;
        items[t] = 0;
        items_by_window[t] = 0;
        return;
    }
    const int64_t i = t / W;
    const int32_t w = static_cast<int32_t>(t % W);
    const int32_t r = rows[i], p0 = rowptr[r], p1 = rowptr[r + 1];
    const int32_t lo = w == 0 ? p0 : first_not_below(colind, p0, p1, w * wcols);
    const int32_t hi = w == W - 1 ? p1 : first_not_below(colind, lo, p1, (w + 1) * wcols);
    const int32_t n = (hi - lo + kChunkNnz - 1) / kChunkNnz, k = (n + F - 1) / F;
    start[2 * t] = lo;
    start[2 * t + 1] = hi;
    chunks[t] = n;
    items[t] = k;
    items_by_window[static_cast<int64_t>(w) * nl + i] = k;
}

__global__ void __launch_bounds__(256)
window_items_kernel(const int32_t *__restrict__ rows, const int32_t *__restrict__ start, const int32_t *__restrict__ chunk_off,
                    const int32_t *__restrict__ item_off, const int32_t *__restrict__ win_off, int64_t nl, int32_t W, int32_t F,
                    int4 *__restrict__ items) {
    const int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (t >= nl * W) return;
    const int64_t i = t / W;
    const int32_t w = static_cast<int32_t>(t % W);
    const bool alone = item_off[(i + 1) * W] - item_off[i * W] == 1;
    int32_t c = chunk_off[t], m = item_off[t], o = win_off[static_cast<int64_t>(w) * nl + i];
    const int32_t hi = start[2 * t + 1], step = F * kChunkNnz;
    for (int32_t x = start[2 * t]; x < hi; x += step, c += F, ++m, ++o)
        items[o] = make_int4(alone ? rows[i] | static_cast<int32_t>(0x80000000u) : m, x, c, min(step, hi - x));
}

// Chunks per item: one while there are few of them (the chain of dependent gathers counts), up to four when they fill the
// GPU several times over (fewer scratch rows to write and add up again: 80 MB each way at 128 columns on R-MAT scale 20).
static int32_t chunks_per_item(int64_t chunks, int sms) {
    const int64_t groups = static_cast<int64_t>(sms) * 4 * 16;   // half-warp groups resident together
    return chunks >= 4 * groups ? 4 : (chunks >= 2 * groups ? 2 : 1);
}

sd_status_t build_schedule(sd_plan *p, int W, int32_t T, const ScanAccum &h, cudaStream_t st) {
    sd_status_t s;
    if (W < 1) W = 1;
    T = std::min<int32_t>(std::max<int32_t>(T, 2), kHybridHeavyMax);
    p->h_T = T;
    p->h_counts.chunks_long = h.chunks_long;
    p->h_counts.chunks_long2 = h.chunks_long2;
    p->h_counts.chunks_long4 = h.chunks_long4;
    p->h_counts.giants = h.giants;
    std::copy(h.len_hist, h.len_hist + 256, p->h_counts.len_hist);
    const int32_t F = p->h_F = W == 1 ? chunks_per_item(static_cast<int64_t>(h.chunks_long), p->info.sm_count) : 1;   // with windows, items that outlast their window cost more (1,122 against 918 us on the rank-size matrix)
    int64_t nl = static_cast<int64_t>(h.long_rows), nc = static_cast<int64_t>(h.chunks_long);
    int64_t ni = static_cast<int64_t>(F == 4 ? h.chunks_long4 : (F == 2 ? h.chunks_long2 : h.chunks_long));
    for (int l = T; l < 256; ++l) {
        const int64_t rows = static_cast<int64_t>(h.len_hist[l]), chunks = (l + kChunkNnz - 1) / kChunkNnz;
        nl += rows;
        nc += rows * chunks;
        ni += rows * ((chunks + F - 1) / F);
    }
    SortBases bases;
    bases.first[0] = 0;
    int64_t at = nl;
    p->h_nm = p->h_nw = 0;
    for (int l = T - 1; l >= 0; --l) {
        bases.first[T - l] = static_cast<int32_t>(at);
        at += static_cast<int64_t>(h.len_hist[l]);
        if (l >= kHybridMedium) p->h_nm = at - nl;
        if (l >= kHybridWide) p->h_nw = at - nl;
    }
    p->h_nl = nl;
    const bool fine = p->M <= 131072;
    const int32_t ntiles = static_cast<int32_t>((p->M + (fine ? 511 : 2047)) / (fine ? 512 : 2048));
    TempBuf hist(st), ngiant(st), start(st), counts(st), offs(st), tmp(st);
    if ((s = hist.get(sizeof(int32_t) * (T + 1) * static_cast<size_t>(ntiles), "length counts"))) return s;
    if ((s = dev_alloc(p, &p->h_rows, p->M, "rows by length", st))) return s;
    if ((s = dev_alloc(p, &p->h_desc, p->M - nl, "light row descriptors", st))) return s;
    auto count = fine ? sort_count_kernel<2> : sort_count_kernel<8>;
    auto place = fine ? sort_place_kernel<2> : sort_place_kernel<8>;
    count<<<ntiles, 32 * kSortWarps, 0, st>>>(p->rowptr, p->M, T, ntiles, hist.as<int32_t>());
    SD_CUDA_TRY(cudaGetLastError());
    SD_CUDA_TRY(launch_overlapped(sort_prefix_kernel, static_cast<unsigned>((T + 8) / 8), 256, 0, st, bases, T, ntiles, hist.as<int32_t>()));
    SD_CUDA_TRY(launch_overlapped(place, static_cast<unsigned>(ntiles), 32 * kSortWarps, 0, st, p->rowptr, p->colind, p->M, T, ntiles,
                                  hist.as<int32_t>(), static_cast<int32_t>(nl), p->h_rows, p->h_desc));
    p->h_nc = p->h_ni = p->h_ng = 0;
    p->info.launches = 1;
    if (nl > 0) {
        int64_t ng = static_cast<int64_t>(h.giants);
        if ((s = dev_alloc(p, &p->h_chunk_ptr, nl + 1, "chunk pointers", st))) return s;
        if ((s = dev_alloc(p, &p->h_giant, W == 1 ? ng : nl, "rows of many chunks", st))) return s;
        if ((s = ngiant.get(sizeof(int32_t), "count"))) return s;
        if ((s = dev_alloc(p, &p->h_item_ptr, nl + 1, "item pointers", st))) return s;
        if (W == 1) {
            SD_CUDA_TRY(launch_overlapped(chunk_ptr_kernel, 1u, 1024, 0, st, p->rowptr, p->h_rows, nullptr, nullptr, 1, F, nl, p->h_chunk_ptr,
                                          p->h_item_ptr, p->h_giant, ngiant.as<int32_t>()));
            if (F > 1 && ng > 0) {   // the scan counted the rows of many chunks, this one those of many items
                int32_t got = 0;
                SD_CUDA_TRY(cudaMemcpyAsync(&got, ngiant.p, sizeof got, cudaMemcpyDeviceToHost, st));
                SD_CUDA_TRY(cudaStreamSynchronize(st));
                ng = got;
            }
            if ((s = dev_alloc(p, &p->h_items, ni, "chunk descriptors", st))) return s;
            SD_CUDA_TRY(launch_overlapped(items_kernel, static_cast<unsigned>(ceil_div(std::min<int64_t>(nl, 148 * 64), 8)), 256, 0, st, p->rowptr,
                                          p->h_rows, p->h_chunk_ptr, p->h_item_ptr, F, nl, p->h_items));
        } else {
            const int64_t cells = nl * W, n = cells + 1;
            if (n > INT32_MAX) {
                set_error(SD_ERR_UNSUPPORTED, "too many (heavy row, window) pairs");
                return SD_ERR_UNSUPPORTED;
            }
            if ((s = start.get(sizeof(int32_t) * 2 * cells, "window ranges"))) return s;
            if ((s = counts.get(sizeof(int32_t) * 3 * n, "chunk counts"))) return s;
            if ((s = offs.get(sizeof(int32_t) * 3 * n, "chunk offsets"))) return s;
            int32_t *cnt = counts.as<int32_t>(), *off = offs.as<int32_t>();   // chunks by row, items by row, items by window
            window_count_kernel<<<ceil_div(n, 256), 256, 0, st>>>(p->rowptr, p->colind, p->h_rows, nl, W, F, (p->K + W - 1) / W,
                                                                 start.as<int32_t>(), cnt, cnt + n, cnt + 2 * n);
            SD_CUDA_TRY(cudaGetLastError());
            size_t tb = 0;
            SD_CUDA_TRY(cub::DeviceScan::ExclusiveSum(nullptr, tb, cnt, off, static_cast<int>(n), st));
            if ((s = tmp.get(tb, "scan scratch"))) return s;
            for (int k = 0; k < 3; ++k)
                SD_CUDA_TRY(cub::DeviceScan::ExclusiveSum(tmp.p, tb, cnt + k * n, off + k * n, static_cast<int>(n), st));
            chunk_ptr_kernel<<<1, 1024, 0, st>>>(p->rowptr, p->h_rows, off, off + n, W, F, nl, p->h_chunk_ptr, p->h_item_ptr, p->h_giant, ngiant.as<int32_t>());
            SD_CUDA_TRY(cudaGetLastError());
            int32_t got[3] = {0, 0, 0};
            SD_CUDA_TRY(cudaMemcpyAsync(&got[0], p->h_chunk_ptr + nl, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
            SD_CUDA_TRY(cudaMemcpyAsync(&got[1], ngiant.p, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
            SD_CUDA_TRY(cudaMemcpyAsync(&got[2], p->h_item_ptr + nl, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
            SD_CUDA_TRY(cudaStreamSynchronize(st));
            nc = got[0];
            ng = got[1];
            ni = got[2];
            if ((s = dev_alloc(p, &p->h_items, ni, "chunk descriptors", st))) return s;
            window_items_kernel<<<ceil_div(cells, 256), 256, 0, st>>>(p->h_rows, start.as<int32_t>(), off, off + n, off + 2 * n, nl, W, F, p->h_items);
            SD_CUDA_TRY(cudaGetLastError());
        }
        p->h_nc = nc;
        p->h_ni = ni;
        p->h_ng = ng;
        if ((s = dev_alloc(p, &p->chunk_out, static_cast<size_t>(ni) * p->N, "chunk sums", st))) return s;
        p->info.launches = 2 + (ng > 0 ? 1 : 0);   // the fused kernel, the chunk sums, the chunk sums of very long rows
    }
    return SD_OK;
}

// =====================================================================================
// narrow dense operands
// =====================================================================================
// The columns that are worth a place in shared memory: the most frequent ones, as many as fit, in ascending order.
constexpr int kDegreeBins = 1 << 16;

__global__ void column_degrees_kernel(const int32_t *__restrict__ colind, int64_t nnz, int32_t *__restrict__ degree) {
    for (int64_t k = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; k < nnz; k += static_cast<int64_t>(gridDim.x) * blockDim.x)
        atomicAdd(degree + __ldg(colind + k), 1);
}
// Most columns share a few small degrees: those are counted per CTA first (R-MAT scale 18: 78 us with all of them in global memory, now 5).
constexpr int kLowBins = 8192;
__global__ void __launch_bounds__(1024)
degree_bins_kernel(const int32_t *__restrict__ degree, int64_t K, int32_t *__restrict__ bins) {
    __shared__ int low[kLowBins];
    for (int i = threadIdx.x; i < kLowBins; i += 1024) low[i] = 0;
    __syncthreads();
    for (int64_t j = static_cast<int64_t>(blockIdx.x) * 1024 + threadIdx.x; j < K; j += static_cast<int64_t>(gridDim.x) * 1024) {
        const int d = min(degree[j], kDegreeBins - 1);
        if (d < kLowBins) atomicAdd(&low[d], 1);
        else atomicAdd(bins + d, 1);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kLowBins; i += 1024)
        if (low[i]) atomicAdd(bins + i, low[i]);
}
// The smallest degree that at most `most` columns reach; one CTA, the last bin first.
__global__ void __launch_bounds__(1024)
degree_threshold_kernel(const int32_t *__restrict__ bins, int64_t most, int32_t *__restrict__ threshold) {
    constexpr int PER = kDegreeBins / 1024;
    using Scan = cub::BlockScan<long long, 1024>;
    __shared__ typename Scan::TempStorage tmp;
    const int t = threadIdx.x, end = kDegreeBins - t * PER;   // this thread's bins: end - 1 down to end - PER
    long long sum = 0, run;
#pragma unroll
    for (int i = 4; i <= PER; i += 4) {
        const int4 v = *reinterpret_cast<const int4 *>(bins + end - i);
        sum += static_cast<long long>(v.x) + v.y + v.z + v.w;
    }
    Scan(tmp).ExclusiveSum(sum, run);
    if (run <= most && run + sum > most)
        for (int i = 1; i <= PER; ++i) {
            const long long with = run + bins[end - i];
            if (run <= most && with > most) *threshold = end - i + 1;
            run = with;
        }
    else if (t == 1023 && run + sum <= most)
        *threshold = 0;
}
__global__ void hot_flags_kernel(const int32_t *__restrict__ degree, int64_t K, const int32_t *__restrict__ threshold, int32_t *__restrict__ flag,
                                 unsigned long long *__restrict__ covered) {
    const int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    const int deg = j < K ? degree[j] : 0;
    const bool hot = j < K && deg > 0 && deg >= *threshold;
    if (j <= K) flag[j] = hot;
    const unsigned mine = hot ? static_cast<unsigned>(deg) : 0u, sum = __reduce_add_sync(0xffffffffu, mine);
    if ((threadIdx.x & 31) == 0 && sum) atomicAdd(covered, static_cast<unsigned long long>(sum));
}
// degree becomes the new name of the column: its slot with bit 31 set, or itself
__global__ void hot_names_kernel(int32_t *__restrict__ degree, int64_t K, const int32_t *__restrict__ slot, int32_t *__restrict__ hot_cols) {
    const int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (j >= K) return;
    const int s = slot[j];
    const bool hot = slot[j + 1] != s;
    if (hot) hot_cols[s] = static_cast<int32_t>(j);
    degree[j] = hot ? s | static_cast<int32_t>(0x80000000u) : static_cast<int32_t>(j);
}
__global__ void rename_columns_kernel(const int32_t *__restrict__ colind, int64_t nnz, const int32_t *__restrict__ name, int32_t *__restrict__ out) {
    for (int64_t k = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; k < nnz; k += static_cast<int64_t>(gridDim.x) * blockDim.x)
        out[k] = __ldg(name + __ldg(colind + k));
}

// Taken where 4,096 columns pay for being fetched by every SM (at most nnz / 600 of them, nnz / 1000 at
// one column) and if they cover a quarter of the nonzeros.  Without and with, us: R-MAT with 32.4 M nonzeros at one, two, three and four
// fp32 columns 107 -> 83, 131 -> 110, 220 -> 169, 172 -> 155, bf16 96 -> 84, 117 -> 96, 215 -> 155, 159 -> 137; with 7.9 M at one 24.2 ->
// 22.1, bf16 23.6 -> 22.7; with 4.6 M at one 18.2 and 18.5, bf16 17.0 and 17.3; with 3.9 M two bf16 16.1 and 16.4, four 23.1 and 21.5;
// four fp32 columns, one 16-byte gather, only on the largest (with 16 M 86 -> 80).  More than kCooHotColumns gain nothing (one bf16 column
// 87 us with 32,768, 89 with 54,000).  Plan creation takes longer for it: scale 18 at one column 437 us, 250 at 32 columns.
constexpr int64_t kCooHotColumns = 32768;
static sd_status_t coo_hot_columns(sd_plan *p, cudaStream_t st) {
    const int64_t row_bytes = p->N * (p->dtype == SD_F32 ? 4 : 2);
    const int64_t most = std::min<int64_t>({kCooHotBytes / row_bytes, kCooHotColumns, p->nnz / (p->N == 1 ? 1000 : 600), p->K});
    if (most < 4096 || (row_bytes == 16 && p->nnz < 16000000)) return SD_OK;
    sd_status_t s;
    TempBuf degree(st), bins(st), flag(st), scratch(st), small(st);
    const int64_t K = p->K;
    if ((s = degree.get(sizeof(int32_t) * K, "column degrees"))) return s;
    if ((s = bins.get(sizeof(int32_t) * kDegreeBins, "degree histogram"))) return s;
    if ((s = flag.get(sizeof(int32_t) * (K + 1), "frequent columns"))) return s;
    if ((s = small.get(16, "degree threshold"))) return s;
    int32_t *threshold = small.as<int32_t>() + 2;
    unsigned long long *covered = small.as<unsigned long long>();
    SD_CUDA_TRY(cudaMemsetAsync(degree.p, 0, sizeof(int32_t) * K, st));
    SD_CUDA_TRY(cudaMemsetAsync(bins.p, 0, sizeof(int32_t) * kDegreeBins, st));
    SD_CUDA_TRY(cudaMemsetAsync(small.p, 0, 16, st));
    const unsigned wide = static_cast<unsigned>(std::min<int64_t>((p->nnz + 255) / 256, p->info.sm_count * 32));
    const unsigned cols = static_cast<unsigned>((K + 256) / 256);   // one thread more than columns at least
    column_degrees_kernel<<<wide, 256, 0, st>>>(p->colind, p->nnz, degree.as<int32_t>());
    degree_bins_kernel<<<static_cast<unsigned>(std::min<int64_t>((K + 1023) / 1024, p->info.sm_count)), 1024, 0, st>>>(degree.as<int32_t>(), K, bins.as<int32_t>());
    degree_threshold_kernel<<<1, 1024, 0, st>>>(bins.as<int32_t>(), most, threshold);
    hot_flags_kernel<<<cols, 256, 0, st>>>(degree.as<int32_t>(), K, threshold, flag.as<int32_t>(), covered);
    SD_CUDA_TRY(cudaGetLastError());
    size_t tb = 0;
    SD_CUDA_TRY(cub::DeviceScan::ExclusiveSum(nullptr, tb, flag.as<int32_t>(), flag.as<int32_t>(), K + 1, st));
    if ((s = scratch.get(tb, "scan scratch"))) return s;
    SD_CUDA_TRY(cub::DeviceScan::ExclusiveSum(scratch.p, tb, flag.as<int32_t>(), flag.as<int32_t>(), K + 1, st));
    int32_t hot = 0;
    unsigned long long sum = 0;
    SD_CUDA_TRY(cudaMemcpyAsync(&hot, flag.as<int32_t>() + K, sizeof hot, cudaMemcpyDeviceToHost, st));
    SD_CUDA_TRY(cudaMemcpyAsync(&sum, covered, sizeof sum, cudaMemcpyDeviceToHost, st));
    SD_CUDA_TRY(cudaStreamSynchronize(st));
    if (hot < 1 || hot > most || 4 * static_cast<int64_t>(sum) < p->nnz) return SD_OK;
    if ((s = dev_alloc(p, &p->coo_hot_cols, hot, "frequent columns", st))) return s;
    p->coo_shift = coo_shift(p->vals, p->dtype == SD_F32 ? 4 : 2, static_cast<int>(p->N));   // the renamed columns can begin anywhere
    if ((s = dev_alloc(p, &p->coo_hot_colind, p->nnz + p->coo_shift, "renamed columns", st))) return s;
    hot_names_kernel<<<cols, 256, 0, st>>>(degree.as<int32_t>(), K, flag.as<int32_t>(), p->coo_hot_cols);
    rename_columns_kernel<<<wide, 256, 0, st>>>(p->colind, p->nnz, degree.as<int32_t>(), p->coo_hot_colind + p->coo_shift);
    SD_CUDA_TRY(cudaGetLastError());
    p->coo_hot = hot;
    return SD_OK;
}

sd_status_t build_coo(sd_plan *p, cudaStream_t st) {
    sd_status_t s;
    p->coo_shift = coo_shift(p->colind, sizeof(int32_t), static_cast<int>(p->N));   // values of the same slice then are one load too, or two
    if ((s = coo_hot_columns(p, st))) return s;
    const int64_t items = p->nnz + p->coo_shift, steps = coo_steps(items, static_cast<int>(p->N));
    const int64_t count2 = 2 * coo_most_ranges(steps, static_cast<int64_t>(kCooMaxWarps) * p->info.sm_count);
    const int64_t chunks2 = (count2 + kCooCarryChunk - 1) / kCooCarryChunk, count3 = 2 * chunks2;
    const bool bits = p->N == 1 && p->info.empty_rows == 0;
    if ((s = dev_alloc(p, &p->coo_row, bits ? 32 * steps : items, "rows of nonzeros", st))) return s;
    if (bits && (s = dev_alloc(p, &p->coo_starts, 32 * steps, "starts of rows", st))) return s;
    if ((s = dev_alloc(p, &p->coo_c1_row, count2, "carry rows", st))) return s;
    if ((s = dev_alloc(p, &p->coo_c1_val, count2 * p->N, "carry sums", st))) return s;
    if ((s = dev_alloc(p, &p->coo_c2_row, count3, "carry rows (level 2)", st))) return s;
    if ((s = dev_alloc(p, &p->coo_c2_val, count3 * p->N, "carry sums (level 2)", st))) return s;
    SD_CUDA_TRY(build_coo_rows(p->rowptr, p->M, p->nnz, p->coo_shift, steps, p->coo_row, p->coo_starts, st));
    p->info.launches = 2 + (count2 > kCooDirectFinal);
    return SD_OK;
}

// =====================================================================================
// 16x16 blocks
// =====================================================================================
// The occupied block columns of a block-row, ascending, from a bitmap in shared memory (a range of kMapBits block columns
// at a time).  Without `bcol` they are only counted.
constexpr int kMapWords = 4096, kMapBits = 32 * kMapWords, kMapThreads = 128;

__global__ void __launch_bounds__(kMapThreads)
block_cols_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colind, int64_t M, int64_t Kb, int32_t Mb,
                  const int32_t *__restrict__ browptr, int32_t *__restrict__ counts, int32_t *__restrict__ bcol) {
    using Scan = cub::BlockScan<int, kMapThreads>;
    __shared__ typename Scan::TempStorage tmp;
    __shared__ unsigned map[kMapWords];
    const int64_t I = blockIdx.x;
    const int64_t b = __ldg(rowptr + I * 16), e = __ldg(rowptr + min((I + 1) * 16, M));
    int found = 0;   // in earlier ranges
    for (int64_t j0 = 0; j0 < Kb; j0 += kMapBits) {
        const int words = static_cast<int>(min(static_cast<int64_t>(kMapWords), (Kb - j0 + 31) / 32));
        for (int i = threadIdx.x; i < words; i += kMapThreads) map[i] = 0;
        __syncthreads();
        for (int64_t p = b + threadIdx.x; p < e; p += kMapThreads) {
            const int64_t j = (__ldg(colind + p) >> 4) - j0;
            if (j >= 0 && j < static_cast<int64_t>(words) * 32) atomicOr(&map[j >> 5], 1u << (j & 31));
        }
        __syncthreads();
        for (int i0 = 0; i0 < words; i0 += kMapThreads) {
            unsigned m = i0 + threadIdx.x < words ? map[i0 + threadIdx.x] : 0u;
            int before, total;
            Scan(tmp).ExclusiveSum(__popc(m), before, total);
            if (bcol) {
                int32_t *out = bcol + browptr[I] + found + before;
                for (; m; m &= m - 1) *out++ = static_cast<int32_t>(j0 + (i0 + threadIdx.x) * 32 + __ffs(m) - 1);
            }
            found += total;
            __syncthreads();
        }
    }
    if (counts && threadIdx.x == 0) {
        counts[I] = found;
        if (I == Mb - 1) counts[Mb] = 0;
    }
}

// Where the values of a block's rows come from: of each row of 16 the first of its nonzeros in the caller's order and a mask of
// the columns that are there.  The first nonzero of a block in its row writes both (the masks are cleared before).
static __global__ void __launch_bounds__(256)
block_rows_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colind, int64_t M, const int32_t *__restrict__ browptr,
                  const int32_t *__restrict__ bcol, int32_t *__restrict__ first, uint16_t *__restrict__ mask) {
    const int64_t I = blockIdx.x;
    const int b0 = __ldg(browptr + I), b1 = __ldg(browptr + I + 1);
    for (int r = threadIdx.x >> 5; r < 16 && I * 16 + r < M; r += 8) {
        const int p1 = __ldg(rowptr + I * 16 + r + 1), p0 = __ldg(rowptr + I * 16 + r);
        for (int p = p0 + (threadIdx.x & 31); p < p1; p += 32) {
            const int j = __ldg(colind + p) >> 4;
            if (p > p0 && __ldg(colind + p - 1) >> 4 == j) continue;
            int lo = b0, hi = b1 - 1;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (__ldg(bcol + mid) < j) lo = mid + 1;
                else hi = mid;
            }
            uint32_t m = 0;
            for (int q = p; q < p1; ++q) {
                const int c = __ldg(colind + q);
                if (c >> 4 != j) break;
                m |= 1u << (c & 15);
            }
            first[static_cast<int64_t>(lo) * 16 + r] = p;
            mask[static_cast<int64_t>(lo) * 16 + r] = static_cast<uint16_t>(m);
        }
    }
}

// Values of the blocks, row-major 16x16, absent entries +0: a thread fetches one 16-byte vector of a block row, with one load if all
// of it is there and aligned in the caller's array.  Bound by memory: each value is read and written once.  16,777 full bf16 blocks
// with a product at 128 columns: 71 us per new set of values with a search of every nonzero's block and separate operand
// images, 37 with a search in shared memory, 24 with these tables; 16,384 blocks with values that the last calls have read too 20.9 with a
// load per entry, 16.7 with vectors, with values that come from DRAM level.
constexpr int kValThreads = 256;

template <typename T>
__global__ void __launch_bounds__(kValThreads)
block_values_kernel(const T *vals, const int32_t *__restrict__ first, const uint16_t *__restrict__ mask, int64_t vectors,
                    int4 *__restrict__ bval) {
    constexpr int V = 16 / sizeof(T), PER_ROW = 16 / V;
    const int64_t i = static_cast<int64_t>(blockIdx.x) * kValThreads + threadIdx.x;
    uint32_t m = 0;
    int p = 0;
    if (i < vectors) {
        const int at = static_cast<int>(i % PER_ROW) * V;
        const uint32_t whole = __ldg(mask + i / PER_ROW);
        p = __ldg(first + i / PER_ROW) + __popc(whole & ((1u << at) - 1u));
        m = whole >> at;
    }
    overlap_next();
    overlap_wait();
    if (i >= vectors) return;
    union {
        T v[V];
        int4 all;
    } out;
    constexpr uint32_t ALL = (1u << V) - 1u;
    if ((m & ALL) == ALL && (reinterpret_cast<uintptr_t>(vals + p) & 15u) == 0) {
        out.all = *reinterpret_cast<const int4 *>(vals + p);
    } else {
        out.all = make_int4(0, 0, 0, 0);
#pragma unroll
        for (int e = 0; e < V; ++e)
            if (m >> e & 1) out.v[e] = vals[p + __popc(m & ((1u << e) - 1u))];
    }
    bval[i] = out.all;
}

template <typename T>
static cudaError_t fill_blocks(const sd_plan *p, bool overlap, cudaStream_t st) {
    const int64_t vectors = p->nnzb * (256 * static_cast<int64_t>(sizeof(T)) / 16);
    if (vectors == 0) return cudaSuccess;
    const unsigned grid = static_cast<unsigned>((vectors + kValThreads - 1) / kValThreads);
    const T *vals = static_cast<const T *>(p->vals);
    int4 *bval = static_cast<int4 *>(p->bval);
    if (overlap) return launch_overlapped(block_values_kernel<T>, grid, kValThreads, 0, st, vals, p->brow_first, p->brow_mask, vectors, bval);
    block_values_kernel<T><<<grid, kValThreads, 0, st>>>(vals, p->brow_first, p->brow_mask, vectors, bval);
    return cudaGetLastError();
}

// overlap: the pattern's tables are complete, only values may still be in flight on `st`
cudaError_t fill_bsr(const sd_plan *p, bool overlap, cudaStream_t st) {
    return p->dtype == SD_F32 ? fill_blocks<float>(p, overlap, st) : fill_blocks<uint16_t>(p, overlap, st);
}

sd_status_t build_bsr(sd_plan *p, int64_t nnzb, cudaStream_t st) {
    const int32_t Mb = static_cast<int32_t>((p->M + 15) / 16);
    const int64_t Kb = (p->K + 15) / 16;
    p->nnzb = nnzb;
    sd_status_t s;
    TempBuf counts(st), tmp(st);
    if ((s = dev_alloc(p, &p->browptr, static_cast<size_t>(Mb) + 1, "browptr", st))) return s;
    if ((s = dev_alloc(p, &p->bcol, nnzb, "bcol", st))) return s;
    if ((s = dev_alloc_bytes(p, &p->bval, (p->dtype == SD_F32 ? 4 : 2) * 256 * static_cast<size_t>(nnzb), "bval", st))) return s;
    if ((s = dev_alloc(p, &p->dev_error, 1, "error word", st))) return s;
    SD_CUDA_TRY(cudaMemsetAsync(p->dev_error, 0, sizeof(int32_t), st));
    if (Mb > 0) {
        if ((s = counts.get(sizeof(int32_t) * (static_cast<size_t>(Mb) + 1), "block counts"))) return s;
        block_cols_kernel<<<Mb, kMapThreads, 0, st>>>(p->rowptr, p->colind, p->M, Kb, Mb, nullptr, counts.as<int32_t>(), nullptr);
        SD_CUDA_TRY(cudaGetLastError());
        size_t tb = 0;
        SD_CUDA_TRY(cub::DeviceScan::ExclusiveSum(nullptr, tb, counts.as<int32_t>(), p->browptr, Mb + 1, st));
        if ((s = tmp.get(tb, "scan scratch"))) return s;
        SD_CUDA_TRY(cub::DeviceScan::ExclusiveSum(tmp.p, tb, counts.as<int32_t>(), p->browptr, Mb + 1, st));
        block_cols_kernel<<<Mb, kMapThreads, 0, st>>>(p->rowptr, p->colind, p->M, Kb, Mb, p->browptr, nullptr, p->bcol);
        SD_CUDA_TRY(cudaGetLastError());
    } else {
        SD_CUDA_TRY(cudaMemsetAsync(p->browptr, 0, sizeof(int32_t), st));
    }
    const size_t block_rows = 16 * static_cast<size_t>(nnzb);
    if ((s = dev_alloc(p, &p->brow_first, block_rows, "first nonzeros of block rows", st))) return s;
    if ((s = dev_alloc(p, &p->brow_mask, block_rows, "columns of block rows", st))) return s;
    if (nnzb > 0) {
        SD_CUDA_TRY(cudaMemsetAsync(p->brow_first, 0, sizeof(int32_t) * block_rows, st));
        SD_CUDA_TRY(cudaMemsetAsync(p->brow_mask, 0, sizeof(uint16_t) * block_rows, st));
        block_rows_kernel<<<Mb, 256, 0, st>>>(p->rowptr, p->colind, p->M, p->browptr, p->bcol, p->brow_first, p->brow_mask);
        SD_CUDA_TRY(cudaGetLastError());
    }
    SD_CUDA_TRY(fill_bsr(p, false, st));
    return SD_OK;
}

}  // namespace sd
