// Structure scan of plan creation (paper Sec. 3.1, intrinsic pattern features; integers only): row-length histogram and
// moments, span, gap, diagonal, order, and the occupied 16x16 blocks with their fill.
//
// One pass over the column indices (plan creation on R-MAT scale 16, 1.9 M nonzeros: 174 -> 101 us, scale 17 287 -> 151, with the
// kernels below in place of one warp or one CTA of 512 threads per block-row, an entry per thread at a time).  A block-row (16 rows) is contiguous in colind, so its occupied blocks are counted in
// a table in shared memory keyed by block column, instead of by sorting a 64-bit block key per nonzero (1.9 M nonzeros:
// key pass, radix sort, run-length encoding and fill count took 290 us and 39 MB of scratch).  A warp takes a block-row of
// up to kSmallNnz nonzeros, a small or a large CTA the longer ones, and a last kernel, cut by column range, those whose
// blocks fit no table.
#include <algorithm>

#include "sd_plan.cuh"

namespace sd {

namespace {

constexpr int kSmallNnz = 1000, kSmallSlots = 2048;    // warp table: at most half full
constexpr int kCountBits = 10;                         // of its words; the other bits hold a block column
// CTA tables of ints: one counter per block column, or hashed (keys and counters, at most half full)
constexpr int kMediumNnz = 4096, kMediumSlots = 16384, kMediumThreads = 256;
constexpr int kLargeSlots = 32768, kLargeThreads = 1024;
constexpr int kScanWarps = 8;

__device__ __forceinline__ int hist_bin(long long v) { return v <= 0 ? 0 : 64 - __clzll(v); }

// Histograms of one CTA in shared memory, added to the global ones when it ends; the sums stay in the threads' registers until
// then (sums of 64 bits in shared memory are loops of compare-and-swap: with every thread of a CTA adding to a few of them the
// long block-rows of R-MAT scale 16 took 101 us, 77 without).
enum { S_R2, S_EMPTY, S_SPAN, S_GAP, S_DIAG, S_UNSORTED, S_LONG, S_NNZ_LONG, S_CHUNKS, S_GIANTS, S_DENSE, S_CHUNKS2, S_CHUNKS4, S_COUNT };
struct alignas(16) ScanShared {
    unsigned long long sum[32][S_COUNT];   // per warp, at the end
    unsigned int row_hist[32], reach[10], len_hist[256], mx[2];   // reach[k]: blocks of at least 2^k entries; mx: longest row, largest span
};
constexpr int kInRegisters = 3;
struct Counts {
    unsigned long long sum[S_COUNT] = {};
    unsigned mr = 0, ms = 0;
    unsigned reach[kInRegisters] = {};
};

__device__ void scan_clear(ScanShared &s) {
    for (int i = threadIdx.x; i < static_cast<int>(sizeof(ScanShared) / 4); i += blockDim.x) reinterpret_cast<unsigned int *>(&s)[i] = 0;
    __syncthreads();
}

__device__ __forceinline__ void scan_flush(ScanShared &s, Counts &n, ScanAccum *out) {
    constexpr unsigned FULL = 0xffffffffu;
    const int t = threadIdx.x, lane = t & 31;
#pragma unroll
    for (int i = 0; i < S_COUNT; ++i) {
        unsigned long long v = n.sum[i];
        if (__any_sync(FULL, v != 0)) {
#pragma unroll
            for (int d = 16; d >= 1; d >>= 1) v += __shfl_xor_sync(FULL, v, d);
        }
        if (lane == 0) s.sum[t >> 5][i] = v;
    }
    const unsigned mr = __reduce_max_sync(FULL, n.mr), ms = __reduce_max_sync(FULL, n.ms);
    if (lane == 0 && mr) atomicMax(&s.mx[0], mr);
    if (lane == 0 && ms) atomicMax(&s.mx[1], ms);
#pragma unroll
    for (int k = 0; k < kInRegisters; ++k) {
        const unsigned v = __reduce_add_sync(FULL, n.reach[k]);
        if (lane == 0 && v) atomicAdd(&s.reach[k], v);
    }
    __syncthreads();
    unsigned long long *const sums[S_COUNT] = {&out->sum_r2, &out->empty_rows, &out->sum_span, &out->sum_gap, &out->diag,
                                          &out->unsorted_rows, &out->long_rows, &out->nnz_long_rows, &out->chunks_long,
                                          &out->giants, &out->nnz_dense_blocks, &out->chunks_long2, &out->chunks_long4};
    if (t < S_COUNT) {
        unsigned long long v = 0;
        for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) v += s.sum[w][t];
        if (v) atomicAdd(sums[t], v);
    }
    if (t == 16 && s.mx[0]) atomicMax(&out->max_r, static_cast<unsigned long long>(s.mx[0]));
    if (t == 17 && s.mx[1]) atomicMax(&out->max_span, static_cast<unsigned long long>(s.mx[1]));
    if (t >= 32 && t < 64 && s.row_hist[t - 32]) atomicAdd(&out->row_hist[t - 32], static_cast<unsigned long long>(s.row_hist[t - 32]));
    if (t >= 64 && t < 73 && s.reach[t - 64] != s.reach[t - 63]) atomicAdd(&out->blk_hist[t - 64], static_cast<unsigned long long>(s.reach[t - 64] - s.reach[t - 63]));
    if (t == 18 && s.reach[0]) atomicAdd(&out->nnzb, static_cast<unsigned long long>(s.reach[0]));
    for (int i = t; i < 256; i += blockDim.x)
        if (s.len_hist[i]) atomicAdd(&out->len_hist[i], static_cast<unsigned long long>(s.len_hist[i]));
}

// The rows of a block-row, one per lane (`mine`: the lane has a row).
__device__ __forceinline__ void count_rows(ScanShared &s, Counts &n, bool mine, int r, unsigned span, bool unsorted) {
    if (!mine) return;
    atomicAdd(&s.row_hist[hist_bin(r)], 1u);
    if (static_cast<unsigned>(r) < 256u) atomicAdd(&s.len_hist[r], 1u);
    if (r <= 0) {
        n.sum[S_EMPTY] += r == 0;
        return;
    }
    n.sum[S_R2] += static_cast<unsigned long long>(r) * static_cast<unsigned long long>(r);
    n.sum[S_SPAN] += span;
    n.sum[S_GAP] += span - 1ull;
    n.sum[S_UNSORTED] += unsorted;
    n.mr = max(n.mr, static_cast<unsigned>(r));
    n.ms = max(n.ms, span);
    if (r >= 256) {
        const unsigned long long chunks = static_cast<unsigned long long>((static_cast<long long>(r) + kChunkNnz - 1) / kChunkNnz);
        n.sum[S_LONG] += 1;
        n.sum[S_NNZ_LONG] += static_cast<unsigned long long>(r);
        n.sum[S_CHUNKS] += chunks;
        n.sum[S_CHUNKS2] += (chunks + 1) / 2;
        n.sum[S_CHUNKS4] += (chunks + 3) / 4;
        n.sum[S_GIANTS] += chunks > kGiantChunks;
    }
}

// A block grew from `old` to `now` entries.  The histogram is kept as it grows (blocks of at least 2^k entries, in registers for
// the frequent k), so nothing has to read the table when it is full: with one counter per block column that pass cost as much as
// the walk.
__device__ __forceinline__ void count_block(ScanShared &s, Counts &n, unsigned old, unsigned now) {
#pragma unroll
    for (int k = 0; k < kInRegisters; ++k) n.reach[k] += old < (1u << k) && now >= (1u << k);
    if (now >= (1u << kInRegisters)) {
        for (int k = kInRegisters; k < 9; ++k)
            if (old < (1u << k) && now >= (1u << k)) atomicAdd(&s.reach[k], 1u);
        if (now >= 128) n.sum[S_DENSE] += old >= 128 ? now - old : now;
    }
}

// Adds n entries to block column j of a hash table with `mask` + 1 slots (never full); its count before.
__device__ __forceinline__ int table_add(int *key, int *cnt, unsigned mask, int j, int n) {
    unsigned h = (static_cast<unsigned>(j) * 2654435761u) >> 7 & mask;
    for (;;) {
        const int was = atomicCAS(key + h, -1, j);
        if (was == -1 || was == j) break;
        h = (h + 1) & mask;
    }
    return atomicAdd(cnt + h, n);
}

// The 16 rows of a block-row: row r holds the nonzeros bound[r] .. bound[r + 1] - 1.
struct Rows {
    int bound[17], lo[16], hi[16];
    int excess;     // entries not below their successor in the block-row, less those that end a row: inside rows
    unsigned uns;   // rows out of order
};
__device__ __forceinline__ int row_of(const Rows &w, int64_t p) {   // the last row that begins at or before p
    int r = 0;
#pragma unroll
    for (int d = 8; d >= 1; d >>= 1)
        if (w.bound[r + d] <= p) r += d;
    return r;
}

// First and last column of the rows, one per lane of a warp, before the walk.  Also how many entries at the end of a row are not
// below their successor, the first entry of the next row that has any.
__device__ __forceinline__ void row_ends(const int32_t *__restrict__ colind, Rows &w, int lane) {
    bool falls = false;
    if (lane < 16 && w.bound[lane] >= w.bound[0] && w.bound[lane] < w.bound[lane + 1] && w.bound[lane + 1] <= w.bound[16]) {
        const int b = w.bound[lane], lo = __ldg(colind + b);
        w.lo[lane] = lo;
        w.hi[lane] = __ldg(colind + w.bound[lane + 1] - 1);
        falls = b > w.bound[0] && lo <= __ldg(colind + b - 1);
    }
    const int ends = __popc(__ballot_sync(0xffffffffu, falls));
    if (lane == 0) {
        w.excess = -ends;
        w.uns = 0;
    }
}

// The nonzeros of a block-row walked by T threads, four consecutive ones a step and thread (one 16-byte load where all four belong
// to the block-row), equal block columns merged.  Bound by instructions (1.9 M nonzeros of R-MAT scale 16 with the row of every entry
// looked up and smallest and largest columns kept as it goes: 105 us), so an entry is only compared with its successor, and
// rows are looked at one by one only when the sum of those comparisons says that some row is out of order.  add(j, n): n entries in
// block column j.
// ALL: every lane of a warp calls add at the same time (n may be 0).
template <int T, bool ALL, typename Add>
__device__ __forceinline__ void walk_block_row(const int32_t *__restrict__ colind, Rows &w, int64_t I, int t, unsigned long long &diag, Add add) {
    const int64_t b = w.bound[0], e = w.bound[16];
    const int off = static_cast<int>(reinterpret_cast<uintptr_t>(colind) >> 2 & 3);   // the arrays are aligned to an entry
    int falls = 0;
    for (int64_t q0 = ((b + off) & ~int64_t{3}) - off + 4 * (t & ~31); q0 < e; q0 += 4 * T) {
        const int64_t p0 = q0 + 4 * (t & 31);   // entries p0 + at .. p0 + end - 1
        const int at = static_cast<int>(max(b - p0, int64_t{0})), end = static_cast<int>(max(min(e - p0, int64_t{4}), int64_t{0}));
        int c[5];
        if (p0 >= b && p0 + 4 < e) {
            const int4 v = __ldg(reinterpret_cast<const int4 *>(colind + p0));
            c[0] = v.x, c[1] = v.y, c[2] = v.z, c[3] = v.w;
            c[4] = __ldg(colind + p0 + 4);
        } else {   // an entry beyond the last is above all others
#pragma unroll
            for (int u = 0; u < 5; ++u) c[u] = u >= at && p0 + u < e ? __ldg(colind + p0 + u) : INT_MAX;
        }
        int n = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int x = c[u], j = x >> 4;
            bool leads = false;
            if (u >= at && u < end) {
                falls += c[u + 1] <= x;
                if (j == I) diag += x == I * 16 + row_of(w, p0 + u);
                ++n;
                leads = u + 1 == end || c[u + 1] >> 4 != j;
            }
            if (ALL || leads) {
                add(j, leads ? n : 0);
                if (leads) n = 0;
            }
        }
    }
    falls = __reduce_add_sync(0xffffffffu, falls);
    if ((threadIdx.x & 31) == 0 && falls) atomicAdd(&w.excess, falls);
}

// Some row is out of order: which, and their smallest and largest columns.
template <int T>
__device__ __forceinline__ void unordered_rows(const int32_t *__restrict__ colind, Rows &w, int t) {
    for (int64_t p = static_cast<int64_t>(w.bound[0]) + t; p < w.bound[16]; p += T) {
        const int r = row_of(w, p), x = __ldg(colind + p);
        if (p + 1 < w.bound[r + 1] && __ldg(colind + p + 1) <= x) atomicOr(&w.uns, 1u << r);
        atomicMin(&w.lo[r], x);
        atomicMax(&w.hi[r], x);
    }
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

// ---- a warp per shorter block-row, overlapped launch that waits at the end ---------------------------------
// The table belongs to one warp, so a slot is taken without an atomic operation, which in shared memory costs a cycle or two per
// lane: lanes write their block columns and read back which one stayed.
struct alignas(16) WarpTable {
    unsigned word[kSmallSlots];   // block column and count; all ones: free.  WIDE: block columns in the first half, counts in the second
    Rows rows;
};

// Adds k entries to block column j (every lane of the warp calls it, k == 0: none).
// WIDE: block columns that leave no room for a count in their word.  The table then has half the slots and takes half the nonzeros
// (creating row-split plans, 2^27 columns: 4 M rows of 3 1,756 -> 319 us, 1 M rows of 8 560 -> 140 with all of them in CTAs before).
template <bool WIDE>
__device__ __forceinline__ void warp_table_add(unsigned *word, unsigned mask, int j, int k, ScanShared &s, Counts &n) {
    constexpr unsigned FULL = 0xffffffffu;
    volatile unsigned *const slots = word;
    constexpr int KEY_AT = WIDE ? 0 : kCountBits;
    const unsigned key = static_cast<unsigned>(j) << KEY_AT;
    unsigned h = (static_cast<unsigned>(j) * 2654435761u) >> 7 & mask;
    bool looking = k > 0;
    while (__any_sync(FULL, looking)) {
        const bool is_free = looking && slots[h] == FULL;
        __syncwarp();
        if (is_free) slots[h] = key;
        __syncwarp();
        if (looking) {
            if ((slots[h] ^ key) >> KEY_AT == 0) looking = false;
            else h = (h + 1) & mask;
        }
    }
    if (k > 0) {
        const unsigned old = WIDE ? atomicAdd(word + kSmallSlots / 2 + h, static_cast<unsigned>(k))
                                  : atomicAdd(word + h, static_cast<unsigned>(k)) & ((1u << kCountBits) - 1u);
        count_block(s, n, old, old + k);
    }
    __syncwarp();
}

static_assert(sizeof(ScanShared) % 16 == 0 && sizeof(WarpTable) % 16 == 0, "tables are cleared with 16-byte stores");

template <bool WIDE>
__global__ void __launch_bounds__(32 * kScanWarps)
scan_small_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colind, int64_t M, int64_t most, ScanAccum *__restrict__ out) {
    extern __shared__ __align__(16) unsigned char smem[];
    ScanShared &s = *reinterpret_cast<ScanShared *>(smem);
    WarpTable &table = reinterpret_cast<WarpTable *>(smem + sizeof(ScanShared))[threadIdx.x >> 5];
    Rows &w = table.rows;
    const int lane = threadIdx.x & 31;
    scan_clear(s);
    const long long last = __ldg(rowptr + M);
    if (blockIdx.x == 0 && threadIdx.x == 0) out->nnz = last;
    if (last < 0) {   // the host refuses such a pattern
        overlap_wait();
        return;
    }
    const int64_t Mb = (M + 15) / 16, warps = static_cast<int64_t>(gridDim.x) * kScanWarps;
    Counts n;
    for (int64_t I = static_cast<int64_t>(blockIdx.x) * kScanWarps + (threadIdx.x >> 5); I < Mb; I += warps) {
        const int64_t r0 = I * 16;
        if (lane < 17) w.bound[lane] = __ldg(rowptr + min(r0 + lane, M));
        __syncwarp();
        const int64_t b = w.bound[0], e = w.bound[16];
        if (e - b > most) {   // left to a CTA
            __syncwarp();
            continue;
        }
        const int len = static_cast<int>(e - b);
        unsigned slots = 128;
        while (static_cast<int>(slots) < 2 * len) slots <<= 1;
        row_ends(colind, w, lane);
        for (unsigned i = lane * 4; i < slots; i += 128) {
            *reinterpret_cast<int4 *>(table.word + i) = make_int4(-1, -1, -1, -1);
            if (WIDE) *reinterpret_cast<int4 *>(table.word + kSmallSlots / 2 + i) = make_int4(0, 0, 0, 0);
        }
        __syncwarp();
        walk_block_row<32, true>(colind, w, I, lane, n.sum[S_DIAG], [&](int j, int k) { warp_table_add<WIDE>(table.word, slots - 1, j, k, s, n); });
        __syncwarp();
        if (w.excess) {
            unordered_rows<32>(colind, w, lane);
            __syncwarp();
        }
        const bool mine = lane < 16 && r0 + lane < M;
        const int r = mine ? w.bound[lane + 1] - w.bound[lane] : 0;
        count_rows(s, n, mine, r, r > 0 ? static_cast<unsigned>(w.hi[lane]) - static_cast<unsigned>(w.lo[lane]) + 1u : 0u,
                   (w.uns >> (lane & 15)) & 1u);
        __syncwarp();
    }
    overlap_wait();   // what follows in the stream waits for this kernel alone
    scan_flush(s, n, out);
}

// ---- second and third kernel: a CTA per longer block-row ----------------------------------------------------
// Block-rows of more than `above` and at most `most` nonzeros.  A block-row costs a chain of about five round trips to memory
// and block barriers whatever its length, and about a cycle per atomic operation on the table, so those of up to kMediumNnz
// nonzeros go to small CTAs, three to an SM (R-MAT scale 16, 794 block-rows of 1,950 nonzeros on average: 77 us with all of
// them in CTAs of 1,024 threads, one to an SM; now 32 for the longest, beside 33 for the others).  Every CTA looks through its share of
// the block-rows, a thread each.  The kernels read nothing that an earlier one writes and run beside it (overlapped launches
// that wait at the end).
template <int THREADS, int SLOTS> struct alignas(16) CtaTable {
    Rows rows;
    unsigned found;
    int list[THREADS];
    alignas(16) int cnt[SLOTS];   // hashed: the first half are keys
};

template <int THREADS, int SLOTS>
__global__ void __launch_bounds__(THREADS)
scan_cta_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colind, int64_t M, int64_t Kb, int64_t above, int64_t most,
                int32_t *__restrict__ huge, ScanAccum *__restrict__ out) {
    overlap_next();
    extern __shared__ __align__(16) unsigned char smem[];
    ScanShared &s = *reinterpret_cast<ScanShared *>(smem);
    CtaTable<THREADS, SLOTS> &table = *reinterpret_cast<CtaTable<THREADS, SLOTS> *>(smem + sizeof(ScanShared));
    Rows &w = table.rows;
    if (__ldg(rowptr + M) < 0) {
        overlap_wait();
        return;
    }
    Counts n;
    bool any = false;
    const int64_t Mb = (M + 15) / 16;
    for (int64_t I0 = blockIdx.x; I0 < Mb; I0 += static_cast<int64_t>(gridDim.x) * THREADS) {
        if (threadIdx.x == 0) table.found = 0;
        __syncthreads();
        const int64_t own = I0 + static_cast<int64_t>(threadIdx.x) * gridDim.x;
        if (own < Mb) {
            const int64_t len = static_cast<int64_t>(__ldg(rowptr + min((own + 1) * 16, M))) - __ldg(rowptr + own * 16);
            if (len > above && len <= most) table.list[atomicAdd(&table.found, 1u)] = static_cast<int>(own);
        }
        __syncthreads();
        const unsigned found = table.found;
        if (found && !any) scan_clear(s);
        any |= found != 0;
        for (unsigned k = 0; k < found; ++k) {
            const int64_t I = table.list[k], r0 = I * 16;
            if (threadIdx.x < 17) w.bound[threadIdx.x] = __ldg(rowptr + min(r0 + threadIdx.x, M));
            __syncthreads();
            const int64_t len = static_cast<int64_t>(w.bound[16]) - w.bound[0];
            unsigned slots = 64;
            if (4 * len <= SLOTS) while (slots < 2u * static_cast<unsigned>(len)) slots <<= 1;
            const bool dense = Kb <= SLOTS, hashed = !dense && 4 * len <= SLOTS;
            int *const key = table.cnt, *const cnt = dense ? table.cnt : table.cnt + SLOTS / 2;
            const unsigned used = dense ? static_cast<unsigned>(Kb) : (hashed ? slots : 0u);
            if (threadIdx.x < 32) row_ends(colind, w, threadIdx.x);
            for (unsigned i = threadIdx.x * 4; i < used; i += THREADS * 4) {
                *reinterpret_cast<int4 *>(cnt + i) = make_int4(0, 0, 0, 0);
                if (hashed) *reinterpret_cast<int4 *>(key + i) = make_int4(-1, -1, -1, -1);
            }
            __syncthreads();
            walk_block_row<THREADS, false>(colind, w, I, threadIdx.x, n.sum[S_DIAG], [&](int j, int k) {
                unsigned old;
                if (hashed) old = table_add(key, cnt, slots - 1, j, k);
                else if (dense && j >= 0 && j < Kb) old = atomicAdd(cnt + j, k);
                else return;
                count_block(s, n, old, old + k);
            });
            __syncthreads();
            if (w.excess) {
                unordered_rows<THREADS>(colind, w, threadIdx.x);
                __syncthreads();
            }
            if (threadIdx.x < 32) {
                const int t = threadIdx.x;
                const bool mine = t < 16 && r0 + t < M;
                const int r = mine ? w.bound[t + 1] - w.bound[t] : 0;
                count_rows(s, n, mine, r, r > 0 ? static_cast<unsigned>(w.hi[t]) - static_cast<unsigned>(w.lo[t]) + 1u : 0u, (w.uns >> (t & 15)) & 1u);
            }
            if (!dense && !hashed && threadIdx.x == 0)   // bit 31: rows out of order, every column range has to look at all of them
                huge[atomicAdd(&out->huge, 1u)] = static_cast<int32_t>(static_cast<uint32_t>(I) | (w.uns ? 0x80000000u : 0u));
            __syncthreads();
        }
    }
    overlap_wait();   // what follows in the stream waits for the last of these kernels alone
    if (any) scan_flush(s, n, out);
}

// ---- fourth kernel: blocks of the remaining block-rows, a CTA per (block-row, range of kLargeSlots block columns) -----------
__global__ void __launch_bounds__(kLargeThreads)
scan_huge_kernel(const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colind, int64_t M, int64_t Kb,
                 const int32_t *__restrict__ huge, ScanAccum *__restrict__ out) {
    extern __shared__ __align__(16) unsigned char smem[];
    ScanShared &s = *reinterpret_cast<ScanShared *>(smem);
    CtaTable<kLargeThreads, kLargeSlots> &table = *reinterpret_cast<CtaTable<kLargeThreads, kLargeSlots> *>(smem + sizeof(ScanShared));
    Rows &w = table.rows;
    const int64_t ranges = (Kb + kLargeSlots - 1) / kLargeSlots, items = static_cast<int64_t>(out->huge) * ranges;
    if (blockIdx.x >= items) return;
    scan_clear(s);
    Counts n;
    for (int64_t k = blockIdx.x; k < items; k += gridDim.x) {
        const uint32_t entry = static_cast<uint32_t>(huge[k / ranges]);
        const int64_t r0 = static_cast<int64_t>(entry & 0x7FFFFFFFu) * 16, j0 = k % ranges * kLargeSlots;
        const bool sorted = (entry >> 31) == 0;
        const int used = static_cast<int>(min(static_cast<int64_t>(kLargeSlots), Kb - j0));
        for (int i = threadIdx.x; i < used; i += kLargeThreads) table.cnt[i] = 0;
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
                if (run && j >= j0 && j < j0 + used) {
                    const unsigned old = atomicAdd(table.cnt + (j - j0), run);
                    count_block(s, n, old, old + run);
                }
            }
        }
        __syncthreads();
    }
    scan_flush(s, n, out);
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
    void *list = nullptr;   // block-rows for the last kernel
    if (Kb > kLargeSlots && (e = pool_alloc(&list, sizeof(int32_t) * Mb, st)) != cudaSuccess) return e;
    int32_t *huge = static_cast<int32_t *>(list);
    const int small_smem = static_cast<int>(sizeof(ScanShared) + kScanWarps * sizeof(WarpTable));
    const int large_smem = static_cast<int>(sizeof(ScanShared) + sizeof(CtaTable<kLargeThreads, kLargeSlots>));
    const int medium_smem = static_cast<int>(sizeof(ScanShared) + sizeof(CtaTable<kMediumThreads, kMediumSlots>));
    auto medium = scan_cta_kernel<kMediumThreads, kMediumSlots>;
    auto large = scan_cta_kernel<kLargeThreads, kLargeSlots>;
    const bool wide = Kb >= (int64_t{1} << (32 - kCountBits)) - 1;   // block columns do not fit a word beside a count
    auto warps = wide ? scan_small_kernel<true> : scan_small_kernel<false>;
    static std::atomic<int> attr_set[kMaxDevices];
    const int dev = current_device();
    if (dev >= kMaxDevices || !attr_set[dev].load(std::memory_order_acquire)) {
        if ((e = cudaFuncSetAttribute(scan_small_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, small_smem)) != cudaSuccess ||
            (e = cudaFuncSetAttribute(scan_small_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, small_smem)) != cudaSuccess ||
            (e = cudaFuncSetAttribute(medium, cudaFuncAttributeMaxDynamicSharedMemorySize, medium_smem)) != cudaSuccess ||
            (e = cudaFuncSetAttribute(large, cudaFuncAttributeMaxDynamicSharedMemorySize, large_smem)) != cudaSuccess ||
            (e = cudaFuncSetAttribute(scan_huge_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, large_smem)) != cudaSuccess) {
            if (list) cudaFreeAsync(list, st);
            return e;
        }
        if (dev < kMaxDevices) attr_set[dev].store(1, std::memory_order_release);
    }
    const int sms = sm_count_cached();
    const int64_t small = wide ? kSmallNnz / 2 : kSmallNnz;
    // the longest chains first; the others fill in beside them.  With a block-row per SM at most the large CTAs take the medium ones too
    // (one launch less: 2,048 rows 45 -> 42 us for the whole plan).
    const bool few = Mb <= sms;
    large<<<static_cast<unsigned>(std::min<int64_t>(Mb, sms)), kLargeThreads, large_smem, st>>>(rowptr, colind, M, Kb, few ? small : kMediumNnz,
                                                                                            INT64_MAX, huge, out);
    e = cudaGetLastError();
    if (e == cudaSuccess && !few)
        e = launch_overlapped(medium, static_cast<unsigned>(std::min<int64_t>(Mb, 3 * sms)), kMediumThreads, static_cast<size_t>(medium_smem), st, rowptr,
                              colind, M, Kb, small, kMediumNnz, nullptr, out);
    if (e == cudaSuccess)
        e = launch_overlapped(warps, static_cast<unsigned>(std::min<int64_t>((Mb + kScanWarps - 1) / kScanWarps, 3 * sms)),
                              32 * kScanWarps, static_cast<size_t>(small_smem), st, rowptr, colind, M, small, out);
    if (e == cudaSuccess && Kb > kLargeSlots) {
        scan_huge_kernel<<<static_cast<unsigned>(sms), kLargeThreads, large_smem, st>>>(rowptr, colind, M, Kb, huge, out);
        e = cudaGetLastError();
    }
    if (list) cudaFreeAsync(list, st);
    return e;
}

}  // namespace sd
