// C ABI of the SpMM library: plan creation (structure scan, decision, representation
// build), execution dispatch, teardown.  See include/sd.h for the contract.
#include <algorithm>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstddef>
#include <cstring>
#include <new>
#include <vector>

#include "sd_hybrid.cuh"
#include "sd_plan.cuh"

// =====================================================================================
// error state
// =====================================================================================
namespace sd {

static thread_local char g_err_text[512] = "";
static thread_local int g_err_code = SD_OK;

void set_error(sd_status_t code, const char *fmt, ...) {
    g_err_code = code;
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err_text, sizeof g_err_text, fmt, ap);
    va_end(ap);
}

sd_status_t cuda_fail(cudaError_t e, const char *what) {
    set_error(SD_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
    return SD_ERR_CUDA;
}

static int env_int(const char *name, int dflt) {
    const char *e = getenv(name);
    return e ? atoi(e) : dflt;
}

const Switches &switches() {
    static const Switches sw = [] {
        Switches s;
        s.no_coo = getenv("SD_NO_COO") != nullptr;
        s.bsr_simt = getenv("SD_BSR_SIMT") != nullptr;
        s.no_narrow = getenv("SD_NO_NARROW") != nullptr;
        s.geom_nv = env_int("SD_GEOM_NV", 0);
        s.ksplit_g = env_int("SD_KSPLIT_G", 0);
        s.narrow_g = env_int("SD_NARROW_G", 0);
        return s;
    }();
    return sw;
}

// Family rule on the integer summary.  The paper ranks templates with a learned model and a
// measured search (Sec. 3.2-3.3) and prints no thresholds; these are fixed integer rules:
//   BSR-TC    rows strictly ascending, N >= 64 and a multiple of 32 (fp32) / 64 (bf16) columns, and
//             rho_BSR(16) = 256 nnzb / nnz <= rho_max(dtype, N) (Eq. 4)
//   MERGE     (max r >= 256 and rows >= 256 hold >= 10 % of nnz) or CV(r)^2 >= 4
//   ROWSPLIT  otherwise
// rho_max is where an earlier block kernel stopped paying on this GPU (Sec. 3.1: dense tiles pay "when useful arithmetic outweighs
// compaction and fill-in costs"): its time went by blocks, the CSR kernels' by nonzeros, measured on random 16x16 blocks thinned to a
// given fill.  The present kernel is two to three times as fast and ahead far beyond these lines; they stay because a matrix that
// moves to blocks loses accuracy and the row kernels' way with non-finite rows of B (below).
//              N < 128   128 <= N < 256   N >= 256
//     fp32       9/8          2              3
//     bf16       3            7              10
static int decide_family(const sd_plan_info_t &s, int dtype) {
    int64_t num, den = 1;
    if (dtype == SD_BF16) {
        num = s.N < 128 ? 3 : (s.N < 256 ? 7 : 10);
    } else if (s.N < 128) {
        num = 9;
        den = 8;
    } else {
        num = s.N < 256 ? 2 : 3;
    }
    // Whole 128-byte groups of columns, from 64 on.  The block kernel serves any multiple of a 16-byte piece and is ahead of the
    // row kernels there too (4,400 full blocks, 32 fp32 columns 5.7 against 13.7 us), but other widths stay with the row kernels:
    // they keep a non-finite row of B out of rows that do not name it, and their error against 64 bits is smaller (there
    // 9e-8 against 3.5e-7; 32 bf16 columns 4.4e-8 against 4.9e-8).
    const int64_t group = dtype == SD_BF16 ? 64 : 32;
    const bool tc_width = s.N >= 64 && s.N % group == 0;
    if (tc_width && s.nnz > 0 && s.unsorted_rows == 0 && den * 256 * s.nnzb16 <= num * s.nnz) return SD_BSR_TC;
    const unsigned __int128 lhs = static_cast<unsigned __int128>(static_cast<uint64_t>(s.M)) * s.sum_r2;
    const unsigned __int128 rhs =
        static_cast<unsigned __int128>(5) * static_cast<uint64_t>(s.nnz) * static_cast<uint64_t>(s.nnz);
    const bool skew = (s.max_r >= 256 && 10 * s.nnz_long_rows >= s.nnz) || (s.nnz > 0 && lhs >= rhs);
    return skew ? SD_MERGE : SD_ROWSPLIT;
}

// Number of column windows, which order the chunks of the heavy rows (and cut them, with a scratch row per piece): none unless
// the rows are short on average (nnz < 16 M), the columns are sorted, and B does not fit in 60 % of L2; then the smallest power
// of two that makes one window's slab of B fit.
static int decide_windows(const sd_plan_info_t &s, int dtype) {
    const int64_t es = dtype == SD_F32 ? 4 : 2;
    const int64_t bbytes = s.K * s.N * es;
    const int64_t budget = s.l2_bytes / 10 * 6;
    if (s.unsorted_rows != 0 || s.nnz >= 16 * s.M || budget <= 0 || bbytes <= budget) return 1;
    int w = 1;
    while (w < 64 && bbytes > budget * w) w <<= 1;
    return w;
}

// Which introspection form describes a merge plan with one window: the window-major segments (true) or the merge-path tiles.
// No product depends on it: from five columns on merge plans run the hybrid schedule, and the rule begins at eight.
static bool decide_class_split(const sd_plan_info_t &s, int dtype) {
    const int64_t widest = dtype == SD_BF16 ? 32 : 64;
    const int64_t narrowest = dtype == SD_BF16 ? 8 : 16;
    return s.unsorted_rows == 0 && s.nnz > 0 && s.N >= narrowest && s.N <= widest;
}

// The family an automatic plan of skewed rows reports, SD_HYBRID or SD_MERGE.  Both run build_schedule's schedule from five columns
// on; what is left to decide are the accessors a caller may use (sd_plan_get_hybrid or _get_tiles / _get_segments) and, below
// kSmallPlan nonzeros, the length at which a row is heavy.  At up to four columns SD_MERGE without windows is the
// segmented reduction, which the first condition of each case keeps.  The bands are where the hybrid schedule was ahead of the
// executors that the merge family had at first; plans saved then and the callers' expectations of `family` keep them.
static bool decide_hybrid(const sd_plan_info_t &s, int dtype, int windows) {
    const bool f32 = dtype == SD_F32;
    const int64_t row_bytes = s.N * (f32 ? 4 : 2);
    if (s.unsorted_rows != 0) return false;
    if (windows > 1) return row_bytes >= 64 && row_bytes <= (f32 ? 192 : 128);
    return s.N > kCooMaxN && row_bytes <= (f32 ? 384 : 256) && s.nnz * row_bytes >= (int64_t{1} << 28);
}

static constexpr int64_t kSmallPlan = 1000000;   // nonzeros: below this the merge family's heavy rows begin at 129 nonzeros (one chunk
                                                 // each at first): 14 to 30 % less on R-MAT scale 14, level at 2 M nonzeros

static sd_status_t read_last(const int32_t *rowptr, int64_t M, cudaStream_t st, int64_t *nnz) {
    int32_t last = 0;
    SD_CUDA_TRY(cudaMemcpyAsync(&last, rowptr + M, sizeof last, cudaMemcpyDeviceToHost, st));
    SD_CUDA_TRY(cudaStreamSynchronize(st));
    if (last < 0) {
        set_error(SD_ERR_INVALID_ARG, "rowptr[M] = %d is negative", last);
        return SD_ERR_INVALID_ARG;
    }
    *nnz = last;
    return SD_OK;
}

// Two round trips to the device for most plans: the scan's counts, and the end.
static sd_status_t create_plan(const sd_plan_desc_t *d, sd_plan *p) {
    cudaStream_t st = static_cast<cudaStream_t>(d->stream);
    p->rowptr = d->rowptr;
    p->colind = d->colind;
    p->vals = d->vals;
    p->M = d->M;
    p->K = d->K;
    p->N = d->N;
    p->dtype = d->dtype;
    p->test_wait_expiry = d->test_wait_expiry;
    SD_CUDA_TRY(cudaGetDevice(&p->device));
    sd_plan_info_t &info = p->info;
    memset(&info, 0, sizeof info);
    info.M = p->M;
    info.K = p->K;
    info.N = p->N;
    info.dtype = p->dtype;
    info.windows = 1;
    info.sm_count = sm_count_cached();
    int l2 = 0;   // single attributes: cudaGetDeviceProperties takes 2.6 ms
    SD_CUDA_TRY(cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, p->device));
    info.l2_bytes = l2;

    sd_status_t s;
    HostBlock block;
    if (!block.p) {
        set_error(SD_ERR_ALLOC, "page-locked host allocation failed");
        return SD_ERR_ALLOC;
    }
    static_assert(sizeof(ScanAccum) <= HostBlock::kBytes, "the scan's counts are read back through one block");
    ScanAccum &h = *static_cast<ScanAccum *>(block.p);
    memset(&h, 0, sizeof h);
    TempBuf accum(st);
    if ((s = accum.get(sizeof(ScanAccum), "scan accumulators"))) return s;
    ScanAccum *dacc = accum.as<ScanAccum>();
    if (p->M > 0) {
        if (!p->colind || !p->vals || d->validate) {   // these need the number of nonzeros before anything reads colind
            if ((s = read_last(p->rowptr, p->M, st, &p->nnz))) return s;
            if (p->nnz > 0 && (!p->colind || !p->vals)) {
                set_error(SD_ERR_INVALID_ARG, "colind / vals are null but rowptr[M] = %lld", (long long)p->nnz);
                return SD_ERR_INVALID_ARG;
            }
        }
        if (d->validate) {
            SD_CUDA_TRY(cudaMemsetAsync(dacc, 0, sizeof(ScanAccum), st));
            SD_CUDA_TRY(validate_csr(p->rowptr, p->colind, p->M, p->K, p->nnz, dacc, st));
            SD_CUDA_TRY(cudaMemcpyAsync(&h, dacc, sizeof h, cudaMemcpyDeviceToHost, st));
            SD_CUDA_TRY(cudaStreamSynchronize(st));
            if (h.bad_csr) {
                set_error(SD_ERR_INVALID_ARG, "malformed CSR: %llu offending rowptr / colind entries", h.bad_csr);
                return SD_ERR_INVALID_ARG;
            }
        }
        SD_CUDA_TRY(scan_structure(p->rowptr, p->colind, p->M, p->K, dacc, st));
        SD_CUDA_TRY(cudaMemcpyAsync(&h, dacc, sizeof h, cudaMemcpyDeviceToHost, st));
        SD_CUDA_TRY(cudaStreamSynchronize(st));
        if (h.nnz < 0) {
            set_error(SD_ERR_INVALID_ARG, "rowptr[M] = %lld is negative", h.nnz);
            return SD_ERR_INVALID_ARG;
        }
        p->nnz = h.nnz;
    }
    info.nnz = p->nnz;
    for (int i = 0; i < 32; ++i) info.row_hist[i] = static_cast<int64_t>(h.row_hist[i]);
    info.sum_r2 = h.sum_r2;
    info.max_r = static_cast<int64_t>(h.max_r);
    info.empty_rows = static_cast<int64_t>(h.empty_rows);
    info.sum_span = h.sum_span;
    info.max_span = static_cast<int64_t>(h.max_span);
    info.sum_gap = h.sum_gap;
    info.diag = static_cast<int64_t>(h.diag);
    info.unsorted_rows = static_cast<int64_t>(h.unsorted_rows);
    info.long_rows = static_cast<int64_t>(h.long_rows);
    info.nnz_long_rows = static_cast<int64_t>(h.nnz_long_rows);
    info.nnzb16 = static_cast<int64_t>(h.nnzb);
    for (int i = 0; i < 9; ++i) info.blk_hist[i] = static_cast<int64_t>(h.blk_hist[i]);
    info.nnz_dense_blocks = static_cast<int64_t>(h.nnz_dense_blocks);
    const bool some = p->M > 0 && p->nnz > 0;

    // ---- decision ------------------------------------------------------------------------------
    int family = d->family == SD_AUTO ? decide_family(info, p->dtype) : d->family;
    if (d->family == SD_AUTO && family == SD_MERGE && d->windows == 0 && some &&
        decide_hybrid(info, p->dtype, decide_windows(info, p->dtype)))
        family = SD_HYBRID;
    if (family == SD_HYBRID && info.unsorted_rows != 0) {   // the chunks of a window are ranges of the rows only if columns ascend
        if (d->family == SD_HYBRID) {
            set_error(SD_ERR_UNSUPPORTED, "the hybrid family needs ascending columns in every row (%lld rows are not)",
                      (long long)info.unsorted_rows);
            return SD_ERR_UNSUPPORTED;
        }
        family = SD_MERGE;
    }
    if (family == SD_BSR_TC && (info.unsorted_rows != 0 || p->nnz == 0)) {
        if (d->family == SD_BSR_TC && info.unsorted_rows != 0) {
            set_error(SD_ERR_UNSUPPORTED, "BSR needs strictly ascending columns in every row (%lld rows are not)",
                      (long long)info.unsorted_rows);
            return SD_ERR_UNSUPPORTED;
        }
        family = SD_ROWSPLIT;
    }
    info.family = family;

    // ---- representation -----------------------------------------------------------------------
    info.launches = 1;
    if (family == SD_MERGE && some) {
        int W = d->windows == 0 ? decide_windows(info, p->dtype) : d->windows;
        bool split = W > 1 || W == -1 || (d->windows == 0 && decide_class_split(info, p->dtype));
        if (W < 1) W = 1;
        if (info.unsorted_rows != 0) {   // windows and the class split need ascending columns
            W = 1;
            split = false;
        }
        info.windows = W;
        info.class_split = split ? 1 : 0;
        info.tile_items = kMergeTile;
        info.num_tiles = split ? 0 : (p->M + p->nnz + kMergeTile - 1) / kMergeTile;
        info.num_segments = p->M;
        if (W > 1 && (s = count_segments(p, W, &info.num_segments, st))) return s;   // reported only: no kernel needs the count
        // narrow dense operands take the segmented reduction, everything else the hybrid schedule
        if (!split && p->N >= 1 && p->N <= kCooMaxN && !switches().no_coo) {
            if ((s = build_coo(p, st))) return s;
        } else if ((s = build_schedule(p, W, p->nnz < kSmallPlan ? kChunkNnz + 1 : kHybridHeavy, h, st))) {
            return s;
        }
    } else if (family == SD_BSR_TC) {
        if ((s = build_bsr(p, info.nnzb16, st))) return s;
    } else if (family == SD_HYBRID && some) {
        const int W = std::max(1, d->windows == 0 ? decide_windows(info, p->dtype) : d->windows);
        if ((s = build_schedule(p, W, d->heavy_len > 0 ? d->heavy_len : kHybridHeavy, h, st))) return s;
        info.windows = W;
        info.num_segments = p->h_nc;
        info.num_tiles = p->h_nl;
        info.heavy_len = p->h_T;
    }
    info.plan_bytes = p->owned;
    SD_CUDA_TRY(cudaStreamSynchronize(st));
    return SD_OK;
}

static cudaError_t host_give_back(sd_plan *p);

// Device work that still uses the plan's memory may be running on any stream: wait for it, then give the memory back.
static void free_plan(sd_plan *p) {
    if (!p) return;
    int prev = 0;
    const bool switched = cudaGetDevice(&prev) == cudaSuccess && prev != p->device && cudaSetDevice(p->device) == cudaSuccess;
    host_give_back(p);
    if (!p->allocs.empty()) cudaDeviceSynchronize();
    for (void *a : p->allocs) cudaFreeAsync(a, nullptr);
    if (p->values_ev) cudaEventDestroy(p->values_ev);
    if (switched) cudaSetDevice(prev);
    delete p;
}

static bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// ---- plan serialisation ---------------------------------------------------------------------------
// Position-dependent 64-bit hash of an int32 array: the sum over i of mix(i, x[i]) (a sum, so the order in which
// the threads add does not matter and the value is the same on every run and every grid size).
__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
__global__ void __launch_bounds__(256)
hash_array_kernel(const int32_t *__restrict__ x, int64_t n, unsigned long long salt, unsigned long long *__restrict__ out) {
    unsigned long long h = 0;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        h += mix64((static_cast<unsigned long long>(i) + 1) * 0x9E3779B97F4A7C15ull ^
                   (static_cast<unsigned long long>(static_cast<uint32_t>(x[i])) + salt));
    for (int off = 16; off > 0; off >>= 1) h += __shfl_xor_sync(0xffffffffu, h, off);
    if ((threadIdx.x & 31) == 0 && h) atomicAdd(out, h);
}

// Hash of the sparsity pattern (rowptr and colind; the values are not part of it).
static sd_status_t pattern_hash(const int32_t *rowptr, const int32_t *colind, int64_t M, int64_t nnz, cudaStream_t st,
                                uint64_t *out) {
    TempBuf acc(st);
    sd_status_t s;
    if ((s = acc.get(sizeof(unsigned long long), "pattern hash"))) return s;
    SD_CUDA_TRY(cudaMemsetAsync(acc.p, 0, sizeof(unsigned long long), st));
    auto *d = static_cast<unsigned long long *>(acc.p);
    if (M >= 0 && rowptr) {
        hash_array_kernel<<<static_cast<unsigned>(std::min<int64_t>((M + 256) / 256, 148 * 8)), 256, 0, st>>>(rowptr, M + 1, 0x51ull, d);
        SD_CUDA_TRY(cudaGetLastError());
    }
    if (nnz > 0) {
        hash_array_kernel<<<static_cast<unsigned>(std::min<int64_t>((nnz + 255) / 256, 148 * 8)), 256, 0, st>>>(colind, nnz, 0xC0ull, d);
        SD_CUDA_TRY(cudaGetLastError());
    }
    unsigned long long h = 0;
    SD_CUDA_TRY(cudaMemcpyAsync(&h, d, sizeof h, cudaMemcpyDeviceToHost, st));
    SD_CUDA_TRY(cudaStreamSynchronize(st));
    *out = h;
    return SD_OK;
}

constexpr uint64_t kBlobMagic = 0x31304E414C504453ull;   // "SDPLAN01"
constexpr uint32_t kBlobVersion = 6;

// What a plan was made for and what was decided; the representation is built again from the caller's arrays when the blob is
// loaded (no scan, no decision), which takes less time than copying it from the host.
struct BlobHeader {
    uint64_t magic;
    uint32_t version, header_bytes;
    uint64_t pattern;           // pattern_hash of (rowptr, colind)
    int64_t M, K, N, nnz;
    int32_t dtype, family;
    char device_name[128];      // the plan was tuned on this GPU model (window count, thresholds)
    int32_t sm_count, has_coo, has_blocks;
    int64_t l2_bytes;
    sd_plan_info_t info;
    int32_t h_T, reserved;
    unsigned long long chunks_long, chunks_long2, chunks_long4, giants, len_hist[256];   // the scan's counts that the schedule is built from
};

static BsrArgs block_args(const sd_plan *plan, const SpmmArgs &a) {
    BsrArgs b;
    b.browptr = plan->browptr;
    b.bcol = plan->bcol;
    b.bval = plan->bval;
    b.B = a.B;
    b.C = a.C;
    b.ldb = a.ldb;
    b.ldc = a.ldc;
    b.M = plan->M;
    b.K = plan->K;
    b.Mb = static_cast<int32_t>((plan->M + 15) / 16);
    b.N = a.N;
    b.alpha = a.alpha;
    b.beta = a.beta;
    return b;
}

// The product on N columns of B and C: all of the plan's, or a slice of them.
static sd_status_t run_product(const sd_plan_t *plan, int64_t N, const void *B, int64_t ldb, float *C, int64_t ldc, float alpha,
                               float beta, cudaStream_t st) {
    const int64_t M = plan->M;
    if (M == 0 || N == 0) return SD_OK;
    if (!C || ldc < N) {
        set_error(SD_ERR_INVALID_ARG, "C is null or ldc < N");
        return SD_ERR_INVALID_ARG;
    }
    if (alpha == 0.f || plan->nnz == 0) {
        SD_CUDA_TRY(run_scale_c(C, ldc, M, static_cast<int32_t>(N), beta, st));
        return SD_OK;
    }
    if (!B || ldb < N) {
        set_error(SD_ERR_INVALID_ARG, "B is null or ldb < N");
        return SD_ERR_INVALID_ARG;
    }
    if (ldb * (plan->dtype == SD_F32 ? 4 : 2) > static_cast<int64_t>(UINT32_MAX)) {
        set_error(SD_ERR_UNSUPPORTED, "row pitch of B must be below 4 GiB");
        return SD_ERR_UNSUPPORTED;
    }
    const int vw = plan->dtype == SD_F32 ? 4 : 8;
    const bool vec = aligned16(B) && aligned16(C) && N % vw == 0 && ldb % vw == 0 && ldc % 4 == 0;

    SpmmArgs a;
    a.ptr = plan->rowptr;
    a.colind = plan->colind;
    a.vals = plan->vals;
    a.B = B;
    a.C = C;
    a.ldb = ldb;
    a.ldc = ldc;
    a.ldb_bytes = static_cast<uint32_t>(ldb * (plan->dtype == SD_F32 ? 4 : 2));
    a.S = M;
    a.max_len = plan->info.max_r;
    a.mean_len = M > 0 ? (plan->nnz + M - 1) / M : 0;
    a.b_bytes = plan->K * N * (plan->dtype == SD_F32 ? 4 : 2);
    a.shared = plan->nnz >= 4 * plan->info.nnzb16;
    a.N = static_cast<int32_t>(N);
    a.alpha = alpha;
    a.beta = beta;

    switch (plan->info.family) {
    case SD_ROWSPLIT:
        SD_CUDA_TRY(run_rowsplit(a, plan->dtype, piece_width(plan->dtype, N, B, ldb, C, ldc), st));
        return SD_OK;
    case SD_MERGE: {
        if (plan->coo_row) {   // narrow dense operand: one writer per row
            a.colind = plan->colind;
            a.vals = plan->vals;
            CooPlan cp;
            cp.row = plan->coo_row;
            cp.starts = plan->coo_starts;
            cp.rowptr = plan->rowptr;
            cp.M = plan->info.empty_rows > 0 ? M : 0;   // no search for rows without nonzeros when the scan found none
            cp.nnz = plan->nnz;
            cp.shift = plan->coo_shift;
            cp.c1_row = plan->coo_c1_row;
            cp.c1_val = plan->coo_c1_val;
            cp.c2_row = plan->coo_c2_row;
            cp.c2_val = plan->coo_c2_val;
            cp.hot_colind = plan->coo_hot_colind;
            cp.hot_cols = plan->coo_hot_cols;
            cp.hot = plan->coo_hot;
            SD_CUDA_TRY(run_coo(cp, a, plan->dtype, plan->info.sm_count, st));
            return SD_OK;
        }
        [[fallthrough]];   // wider ones run the hybrid schedule
    }
    case SD_HYBRID: {
        // one launch for the chunks of the heavy rows and all light rows; then the chunk sums
        const int vw = piece_width(plan->dtype, N, B, ldb, C, ldc);
        HybridArgs h;
        h.colind = plan->colind;
        h.vals = plan->vals;
        h.B = B;
        h.C = C;
        h.scratch = plan->chunk_out;
        h.items = plan->h_items;
        h.desc = plan->h_desc;
        h.ldc = ldc;
        h.ldb_bytes = a.ldb_bytes;
        h.N = static_cast<int32_t>(N);
        h.chunks = static_cast<int32_t>(plan->h_ni);
        h.wide = static_cast<int32_t>(plan->h_nw);
        h.medium = static_cast<int32_t>(plan->h_nm - plan->h_nw);
        h.light = static_cast<int32_t>(M - plan->h_nl - plan->h_nm);
        h.gc = h.gm = 0;
        h.alpha = alpha;
        h.beta = beta;
        SD_CUDA_TRY(plan->dtype == SD_F32 ? run_hybrid_f32(h, vw, st) : run_hybrid_bf16(h, vw, st));
        if (plan->h_nl > 0) {
            SD_CUDA_TRY(run_chunk_reduce(plan->chunk_out, plan->h_item_ptr, plan->h_rows, plan->h_nl, C, ldc,
                                         static_cast<int32_t>(N), alpha, beta, st, plan->h_ng > 0 ? kGiantChunks : 0));
            if (plan->h_ng > 0)
                SD_CUDA_TRY(run_chunk_reduce_wide(plan->chunk_out, plan->h_item_ptr, plan->h_rows, plan->h_giant,
                                                  plan->h_ng, C, ldc, static_cast<int32_t>(N), alpha, beta, st));
        }
        return SD_OK;
    }
    case SD_BSR_TC:
        SD_CUDA_TRY(run_bsr(block_args(plan, a), plan->dtype, st));
        if (plan->test_wait_expiry) SD_CUDA_TRY(run_wait_expiry(plan->dev_error, st));
        return SD_OK;
    default:
        set_error(SD_ERR_INTERNAL, "plan has no family");
        return SD_ERR_INTERNAL;
    }
}

// ---- host operands ---------------------------------------------------------------------------------
// A rows x width rectangle between the host and a device matrix of the same shape.  Whole contiguous rectangles go as one
// run of bytes: the two-dimensional copy of the same bytes from a host pitch below 256 took up to 30 times as long.
static cudaError_t copy_rect(void *dst, int64_t dpitch, const void *src, int64_t spitch, int64_t width, int64_t rows, cudaMemcpyKind kind, cudaStream_t st) {
    if (dpitch == width && spitch == width) return cudaMemcpyAsync(dst, src, static_cast<size_t>(width) * rows, kind, st);
    return cudaMemcpy2DAsync(dst, dpitch, src, spitch, width, rows, kind, st);
}

// Column slices of a product with host operands: while one slice is multiplied, the next one's columns of B travel in and the
// previous one's columns of C out (the bus carries both directions at once: strided copies of 256-byte pieces 99 GB/s together,
// of 128-byte pieces 72, one direction alone 55).  Slice boundaries in columns: whole 256-byte pieces of a row of B, of a
// 256-byte row two halves; at most eight slices.  One slice, no overlap: rows of B not of whole 128-byte pieces or below two of
// them, or little data.
constexpr int kHostSlices = 8;
static int host_slices(const sd_plan *p, int64_t ldb, int64_t ldc, int64_t (&at)[kHostSlices + 1]) {
    const int64_t es = p->dtype == SD_F32 ? 4 : 2, row = p->N * es;
    at[0] = 0;
    at[1] = p->N;
    if (row % 128 != 0 || row < 256 || (ldb * es) % 128 != 0 || (ldc * 4) % 128 != 0 || p->K * row < (int64_t{1} << 20) ||
        p->M * p->N * 4 < (int64_t{1} << 20))
        return 1;
    int64_t piece = row < 512 ? 128 : 256;
    while (row / piece > kHostSlices) piece *= 2;
    const int n = static_cast<int>(row / piece);
    for (int i = 1; i < n; ++i) at[i] = i * piece / es;
    at[n] = p->N;
    return n;
}

static std::mutex g_host_mutex;
static std::vector<HostStreams *> g_host_idle;

static void host_destroy(HostStreams *h) {
    for (cudaStream_t st : {h->st, h->in, h->out})
        if (st) cudaStreamDestroy(st);
    for (cudaEvent_t e : {h->in_ev, h->out_ev, h->done_ev})
        if (e) cudaEventDestroy(e);
    delete h;
}

static sd_status_t host_create(HostStreams *h) {
    for (cudaStream_t *st : {&h->st, &h->in, &h->out}) SD_CUDA_TRY(cudaStreamCreateWithFlags(st, cudaStreamNonBlocking));
    for (cudaEvent_t *e : {&h->in_ev, &h->out_ev, &h->done_ev}) SD_CUDA_TRY(cudaEventCreateWithFlags(e, cudaEventDisableTiming));
    return SD_OK;
}

// A set for the plan's next host product; it keeps one that is still in flight.
static sd_status_t host_take(sd_plan *p) {
    if (p->host) return SD_OK;
    const int dev = current_device();
    {
        std::lock_guard<std::mutex> lock(g_host_mutex);
        for (size_t i = g_host_idle.size(); i-- > 0;)
            if (g_host_idle[i]->device == dev) {
                p->host = g_host_idle[i];
                g_host_idle.erase(g_host_idle.begin() + static_cast<std::ptrdiff_t>(i));
                return SD_OK;
            }
    }
    HostStreams *h = new (std::nothrow) HostStreams;
    if (!h) {
        set_error(SD_ERR_ALLOC, "host allocation failed");
        return SD_ERR_ALLOC;
    }
    h->device = dev;
    const sd_status_t s = host_create(h);
    if (s) host_destroy(h);
    else p->host = h;
    return s;
}

// Waits for the plan's host products and gives the set back.
static cudaError_t host_give_back(sd_plan *p) {
    HostStreams *h = p->host;
    if (!h) return cudaSuccess;
    cudaError_t e = cudaSuccess;
    for (cudaStream_t st : {h->in, h->out, h->st}) {
        const cudaError_t x = cudaStreamSynchronize(st);
        if (e == cudaSuccess) e = x;
    }
    p->host = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_host_mutex);
        if (e == cudaSuccess && g_host_idle.size() < kHostStreamSets) {
            g_host_idle.push_back(h);
            return e;
        }
    }
    host_destroy(h);
    return e;
}

static void host_release_idle() {
    std::lock_guard<std::mutex> lock(g_host_mutex);
    for (HostStreams *h : g_host_idle) host_destroy(h);
    g_host_idle.clear();
}

// Values and host products.  Products with host operands run on a stream of the library, new values arrive on the caller's: each
// waits for the other through an event (new values and a product: 20.8 us with the event between them and without, 16,384 blocks at
// 128 bf16 columns; 4.7 against 4.4 on 2,048 rows).  Inside a stream capture nothing is recorded: when the graph runs is known to the
// caller alone.
static bool capturing(cudaStream_t st) {
    cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
    return cudaStreamIsCapturing(st, &s) == cudaSuccess && s != cudaStreamCaptureStatusNone;
}
static sd_status_t order_after_host_product(sd_plan *p, cudaStream_t st) {
    if (!p->host || capturing(st)) return SD_OK;
    SD_CUDA_TRY(cudaEventRecord(p->host->done_ev, p->host->st));
    SD_CUDA_TRY(cudaStreamWaitEvent(st, p->host->done_ev, 0));
    return SD_OK;
}
static sd_status_t order_before_host_product(sd_plan *p, cudaStream_t st) {
    if (capturing(st)) return SD_OK;
    if (!p->values_ev) SD_CUDA_TRY(cudaEventCreateWithFlags(&p->values_ev, cudaEventDisableTiming));
    SD_CUDA_TRY(cudaEventRecord(p->values_ev, st));
    p->values_recorded = true;
    return SD_OK;
}
static sd_status_t wait_for_values(sd_plan *p) {
    if (p->values_recorded) SD_CUDA_TRY(cudaStreamWaitEvent(p->host->st, p->values_ev, 0));
    p->values_recorded = false;
    return SD_OK;
}

// Queues the copies and the kernels of a product with host operands.
static sd_status_t queue_host_product(sd_plan *plan, const void *B_host, int64_t ldb, float *C_host, int64_t ldc, float alpha,
                                      float beta) {
    const int64_t M = plan->M, N = plan->N, K = plan->K;
    if (M == 0 || N == 0) return SD_OK;
    if (!C_host || ldc < N || !B_host || ldb < N) {
        set_error(SD_ERR_INVALID_ARG, "null host buffer or leading dimension < N");
        return SD_ERR_INVALID_ARG;
    }
    const size_t es = plan->dtype == SD_F32 ? 4 : 2;
    sd_status_t s;
    if ((s = host_take(plan))) return s;
    cudaStream_t st = plan->host->st, in = plan->host->in, out = plan->host->out;
    if (!plan->stage_B && (s = dev_alloc_bytes(plan, &plan->stage_B, es * K * N, "B staging", st))) return s;
    if (!plan->stage_C && (s = dev_alloc(plan, &plan->stage_C, static_cast<size_t>(M) * N, "C staging", st))) return s;
    int64_t at[kHostSlices + 1];
    const int n = host_slices(plan, ldb, ldc, at);
    const char *bh = static_cast<const char *>(B_host);
    char *bd = static_cast<char *>(plan->stage_B);
    if (n == 1) {
        SD_CUDA_TRY(copy_rect(bd, es * N, bh, es * ldb, es * N, K, cudaMemcpyHostToDevice, st));
        if (beta != 0.f) SD_CUDA_TRY(copy_rect(plan->stage_C, 4 * N, C_host, 4 * ldc, 4 * N, M, cudaMemcpyHostToDevice, st));
        if ((s = wait_for_values(plan))) return s;
        if ((s = run_product(plan, N, bd, N, plan->stage_C, N, alpha, beta, st))) return s;
        SD_CUDA_TRY(copy_rect(C_host, 4 * ldc, plan->stage_C, 4 * N, 4 * N, M, cudaMemcpyDeviceToHost, st));
        return SD_OK;
    }
    // forked from the products' stream and joined back into it: the staging buffers belong to one call at a time
    cudaEvent_t ev = plan->host->in_ev, out_ev = plan->host->out_ev;
    SD_CUDA_TRY(cudaEventRecord(ev, st));
    SD_CUDA_TRY(cudaStreamWaitEvent(in, ev, 0));
    SD_CUDA_TRY(cudaStreamWaitEvent(out, ev, 0));
    if ((s = wait_for_values(plan))) return s;
    for (int i = 0; i < n; ++i) {
        const int64_t c = at[i], w = at[i + 1] - c;
        SD_CUDA_TRY(cudaMemcpy2DAsync(bd + es * c, es * N, bh + es * c, es * ldb, es * w, K, cudaMemcpyHostToDevice, in));
        if (beta != 0.f)
            SD_CUDA_TRY(cudaMemcpy2DAsync(plan->stage_C + c, 4 * N, C_host + c, 4 * ldc, 4 * w, M, cudaMemcpyHostToDevice, in));
        SD_CUDA_TRY(cudaEventRecord(ev, in));
        SD_CUDA_TRY(cudaStreamWaitEvent(st, ev, 0));
        if ((s = run_product(plan, w, bd + es * c, N, plan->stage_C + c, N, alpha, beta, st))) return s;
        SD_CUDA_TRY(cudaEventRecord(out_ev, st));
        SD_CUDA_TRY(cudaStreamWaitEvent(out, out_ev, 0));
        SD_CUDA_TRY(cudaMemcpy2DAsync(C_host + c, 4 * ldc, plan->stage_C + c, 4 * N, 4 * w, M, cudaMemcpyDeviceToHost, out));
    }
    SD_CUDA_TRY(cudaEventRecord(out_ev, out));
    SD_CUDA_TRY(cudaStreamWaitEvent(st, out_ev, 0));
    return SD_OK;
}

}  // namespace sd

// =====================================================================================
// extern "C"
// =====================================================================================
using namespace sd;

extern "C" {
#pragma GCC visibility push(default)

const char *sd_version(void) { return "0.1"; }

int sd_last_error(char *buf, size_t n) {
    if (buf && n) {
        strncpy(buf, g_err_text, n - 1);
        buf[n - 1] = '\0';
    }
    return g_err_code;
}

sd_status_t sd_plan_create_ex(const sd_plan_desc_t *d, sd_plan_t **out) {
    if (out) *out = nullptr;
    if (!d || !out) {
        set_error(SD_ERR_INVALID_ARG, "desc and out must not be null");
        return SD_ERR_INVALID_ARG;
    }
    if (d->M < 0 || d->K < 0 || d->N < 0 || d->M > INT32_MAX - 1 || d->K > INT32_MAX - 1 || d->N > INT32_MAX / 2) {
        set_error(SD_ERR_INVALID_ARG, "M, K, N must be in [0, 2^31)");
        return SD_ERR_INVALID_ARG;
    }
    if (d->M > 0 && !d->rowptr) {
        set_error(SD_ERR_INVALID_ARG, "rowptr is null");
        return SD_ERR_INVALID_ARG;
    }
    if (d->dtype != SD_F32 && d->dtype != SD_BF16) {
        set_error(SD_ERR_INVALID_ARG, "unknown dtype %d", d->dtype);
        return SD_ERR_INVALID_ARG;
    }
    if (d->family < SD_AUTO || d->family > SD_HYBRID) {
        set_error(SD_ERR_INVALID_ARG, "unknown family %d", d->family);
        return SD_ERR_INVALID_ARG;
    }
    if (d->windows < -1 || d->windows > 64) {
        set_error(SD_ERR_INVALID_ARG, "windows must be in [-1, 64]");
        return SD_ERR_INVALID_ARG;
    }
    sd_plan *p = new (std::nothrow) sd_plan;
    if (!p) {
        set_error(SD_ERR_ALLOC, "host allocation failed");
        return SD_ERR_ALLOC;
    }
    const sd_status_t s = create_plan(d, p);
    if (s != SD_OK) {
        free_plan(p);
        return s;
    }
    *out = p;
    return SD_OK;
}

sd_plan_t *sd_plan_create(const int32_t *rowptr, const int32_t *colind, const float *vals, int64_t M, int64_t K,
                          int64_t N) {
    sd_plan_desc_t d;
    memset(&d, 0, sizeof d);
    d.rowptr = rowptr;
    d.colind = colind;
    d.vals = vals;
    d.M = M;
    d.K = K;
    d.N = N;
    d.dtype = SD_F32;
    d.family = SD_AUTO;
    sd_plan_t *p = nullptr;
    sd_plan_create_ex(&d, &p);
    return p;
}

void sd_plan_destroy(sd_plan_t *plan) { free_plan(plan); }

sd_status_t sd_release_unused(void) {
    host_release_idle();
    host_blocks_release();
    return pool_release();
}

sd_status_t sd_plan_get_info(const sd_plan_t *plan, sd_plan_info_t *out) {
    if (!plan || !out) {
        set_error(SD_ERR_INVALID_ARG, "plan and out must not be null");
        return SD_ERR_INVALID_ARG;
    }
    *out = plan->info;
    return SD_OK;
}

// Row-length shape class on the integers of the summary (Sec. 3.1 names five classes and gives no
// cut-offs; the rule is stated beside sd_shape_t).  CV^2 = M sum r^2 / nnz^2 - 1.
static int shape_class_of(const sd_plan_info_t &s) {
    if (s.nnz <= 0 || s.M <= 0) return SD_SHAPE_UNIFORM;
    using u128 = unsigned __int128;
    const u128 m_r2 = static_cast<u128>(static_cast<uint64_t>(s.M)) * s.sum_r2;
    const u128 nnz2 = static_cast<u128>(static_cast<uint64_t>(s.nnz)) * static_cast<uint64_t>(s.nnz);
    if (16 * m_r2 <= 17 * nnz2) return SD_SHAPE_UNIFORM;
    const int64_t nonempty = s.M - s.empty_rows;
    int first = -1, last = -1;
    for (int b = 1; b < 32; ++b) {
        if (4 * s.row_hist[b] >= nonempty) {
            if (first < 0) first = b;
            last = b;
        }
    }
    if (first >= 0 && last - first >= 3) return SD_SHAPE_BIMODAL;
    if (m_r2 >= 5 * nnz2 && static_cast<u128>(static_cast<uint64_t>(s.max_r)) * static_cast<uint64_t>(s.M) >=
                                static_cast<u128>(64) * static_cast<uint64_t>(s.nnz))
        return SD_SHAPE_POWERLAW;
    if (m_r2 >= 2 * nnz2) return SD_SHAPE_SKEWED;
    return SD_SHAPE_MODERATE;
}

sd_status_t sd_plan_get_features(sd_plan_t *plan, sd_features_t *out) {
    if (!plan || !out) {
        set_error(SD_ERR_INVALID_ARG, "sd_plan_get_features: null argument");
        return SD_ERR_INVALID_ARG;
    }
    if (!plan->have_feat) {
        int prev = 0;
        SD_CUDA_TRY(cudaGetDevice(&prev));
        SD_CUDA_TRY(cudaSetDevice(plan->device));
        FeatureCounts fc;
        const sd_status_t s = compute_feature_counts(plan->rowptr, plan->colind, plan->M, plan->K, plan->nnz, nullptr, &fc);
        cudaSetDevice(prev);
        if (s) return s;
        const sd_plan_info_t &info = plan->info;
        sd_features_t f{};
        for (int k = 0; k < 3; ++k) {
            f.row_q[k] = fc.row_q[k];
            f.col_q[k] = fc.col_q[k];
            f.sell_slots[k] = fc.sell_slots[k];
        }
        f.col_max = fc.col_max;
        f.col_empty = fc.col_empty;
        f.sum_d2 = fc.sum_d2;
        f.ell_slots = info.M * info.max_r;
        f.nnzb[0] = fc.nnzb4;
        f.nnzb[1] = fc.nnzb8;
        f.nnzb[2] = info.nnzb16;
        const int64_t vb = plan->dtype == SD_BF16 ? 2 : 4;
        f.value_bytes = static_cast<int32_t>(vb);
        f.rep_bytes[0] = (vb + 4) * info.nnz + 4 * (info.M + 1);
        f.rep_bytes[1] = (vb + 4) * f.ell_slots;
        const int64_t heights[3] = {16, 32, 512};
        for (int k = 0; k < 3; ++k)
            f.rep_bytes[2 + k] = (vb + 4) * f.sell_slots[k] + 4 * ((info.M + heights[k] - 1) / heights[k] + 1);
        const int64_t bs[3] = {4, 8, 16};
        for (int k = 0; k < 3; ++k)
            f.rep_bytes[5 + k] = (vb * bs[k] * bs[k] + 4) * f.nnzb[k] + 4 * ((info.M + bs[k] - 1) / bs[k] + 1);
        f.shape_class = shape_class_of(info);
        f.borrowed_bytes = info.family == SD_BSR_TC ? 0 : f.rep_bytes[0];   // blocks hold all of A, every other family reads it in place
        f.plan_bytes = info.plan_bytes;
        f.d_r = info.K * info.N * vb;
        f.d_s = 4 * info.M * info.N;
        f.m_r = f.borrowed_bytes + f.plan_bytes + f.d_r;
        f.m_t = f.m_r + f.d_s;
        f.work_units = info.family == SD_MERGE ? (info.class_split ? info.num_segments : info.num_tiles)
                     : info.family == SD_BSR_TC ? (info.M + 15) / 16
                     : info.family == SD_HYBRID ? info.num_segments + (info.M - info.num_tiles)
                                                : info.M;
        f.sm_count = info.sm_count;
        f.l2_bytes = info.l2_bytes;
        plan->feat = f;
        plan->have_feat = true;
    }
    *out = plan->feat;
    return SD_OK;
}

sd_status_t sd_plan_get_bsr(const sd_plan_t *plan, int32_t *browptr, int32_t *bcol, void *bval) {
    if (!plan) {
        set_error(SD_ERR_INVALID_ARG, "plan is null");
        return SD_ERR_INVALID_ARG;
    }
    if (plan->info.family != SD_BSR_TC) {
        set_error(SD_ERR_UNSUPPORTED, "the plan holds no BSR representation");
        return SD_ERR_UNSUPPORTED;
    }
    const int64_t Mb = (plan->M + 15) / 16;
    const size_t es = plan->dtype == SD_F32 ? 4 : 2;
    if (browptr) SD_CUDA_TRY(cudaMemcpy(browptr, plan->browptr, sizeof(int32_t) * (Mb + 1), cudaMemcpyDeviceToHost));
    if (bcol && plan->nnzb)
        SD_CUDA_TRY(cudaMemcpy(bcol, plan->bcol, sizeof(int32_t) * plan->nnzb, cudaMemcpyDeviceToHost));
    if (bval && plan->nnzb) SD_CUDA_TRY(cudaMemcpy(bval, plan->bval, es * 256 * plan->nnzb, cudaMemcpyDeviceToHost));
    return SD_OK;
}

sd_status_t sd_plan_get_hybrid(const sd_plan_t *plan, int32_t *heavy_rows, int32_t *chunk_ptr, int32_t *ranges,
                               int32_t *order, int32_t *light_rows) {
    if (!plan) {
        set_error(SD_ERR_INVALID_ARG, "plan is null");
        return SD_ERR_INVALID_ARG;
    }
    if (plan->info.family != SD_HYBRID) {
        set_error(SD_ERR_UNSUPPORTED, "the plan's family is not SD_HYBRID");
        return SD_ERR_UNSUPPORTED;
    }
    const int64_t nl = plan->h_nl, nc = plan->h_nc, nlight = plan->h_T > 0 ? plan->M - nl : 0;
    if (heavy_rows && nl > 0) SD_CUDA_TRY(cudaMemcpy(heavy_rows, plan->h_rows, 4 * nl, cudaMemcpyDeviceToHost));
    if (chunk_ptr) {
        if (nl > 0) SD_CUDA_TRY(cudaMemcpy(chunk_ptr, plan->h_chunk_ptr, 4 * (nl + 1), cudaMemcpyDeviceToHost));
        else chunk_ptr[0] = 0;
    }
    if ((ranges || order) && nc > 0) {   // the descriptors sd_spmm reads, taken apart
        const int64_t ni = plan->h_ni;
        std::vector<int4> items(ni);
        SD_CUDA_TRY(cudaMemcpy(items.data(), plan->h_items, sizeof(int4) * ni, cudaMemcpyDeviceToHost));
        int64_t at = 0;
        for (int64_t i = 0; i < ni; ++i) {
            int32_t c = items[i].z;
            for (int32_t x = items[i].y, e = x + items[i].w; x < e; x += kChunkNnz, ++c) {
                if (order) order[at++] = c;
                if (ranges) {
                    ranges[2 * c] = x;
                    ranges[2 * c + 1] = std::min(x + kChunkNnz, e);
                }
            }
        }
    }
    if (light_rows && nlight > 0) SD_CUDA_TRY(cudaMemcpy(light_rows, plan->h_rows + nl, 4 * nlight, cudaMemcpyDeviceToHost));
    return SD_OK;
}

sd_status_t sd_plan_device_status(sd_plan_t *plan, int32_t *status) {
    if (!plan || !status) {
        set_error(SD_ERR_INVALID_ARG, "plan and status must not be null");
        return SD_ERR_INVALID_ARG;
    }
    *status = 0;
    SD_CUDA_TRY(cudaDeviceSynchronize());
    if (plan->dev_error) {
        SD_CUDA_TRY(cudaMemcpy(status, plan->dev_error, sizeof(int32_t), cudaMemcpyDeviceToHost));
        if (*status) SD_CUDA_TRY(cudaMemset(plan->dev_error, 0, sizeof(int32_t)));
    }
    return SD_OK;
}

sd_status_t sd_plan_get_tiles(const sd_plan_t *plan, int32_t *tile_seg, int64_t cap, int64_t *count) {
    if (!plan || !count) {
        set_error(SD_ERR_INVALID_ARG, "plan and count must not be null");
        return SD_ERR_INVALID_ARG;
    }
    if (plan->info.family != SD_MERGE) {
        set_error(SD_ERR_UNSUPPORTED, "the plan holds no merge-path tile table");
        return SD_ERR_UNSUPPORTED;
    }
    const int64_t n = plan->M == 0 || plan->nnz == 0 ? 0 : (plan->info.class_split ? plan->info.windows : plan->info.num_tiles + 1);
    *count = n;
    return tile_seg && cap >= n && n > 0 ? inspect_tiles(plan, tile_seg) : SD_OK;
}

sd_status_t sd_plan_get_segments(const sd_plan_t *plan, int32_t *seg_ptr, int32_t *seg_row, int32_t *colind,
                                 void *vals, int64_t *win_seg) {
    if (!plan) {
        set_error(SD_ERR_INVALID_ARG, "plan is null");
        return SD_ERR_INVALID_ARG;
    }
    if (plan->info.family != SD_MERGE || !plan->info.class_split) {
        set_error(SD_ERR_UNSUPPORTED, "the plan holds no window-major segment list");
        return SD_ERR_UNSUPPORTED;
    }
    return inspect_segments(plan, plan->info.windows, seg_ptr, seg_row, colind, vals, win_seg);
}

sd_status_t sd_spmm(const sd_plan_t *plan, const void *B, int64_t ldb, float *C, int64_t ldc, float alpha, float beta,
                    void *stream) {
    if (!plan) {
        set_error(SD_ERR_INVALID_ARG, "plan is null");
        return SD_ERR_INVALID_ARG;
    }
    return run_product(plan, plan->N, B, ldb, C, ldc, alpha, beta, static_cast<cudaStream_t>(stream));
}

sd_status_t sd_plan_update_values(sd_plan_t *plan, const void *vals, void *stream) {
    if (!plan) {
        set_error(SD_ERR_INVALID_ARG, "plan is null");
        return SD_ERR_INVALID_ARG;
    }
    if (plan->nnz == 0) return SD_OK;
    if (!vals) {
        set_error(SD_ERR_INVALID_ARG, "vals is null");
        return SD_ERR_INVALID_ARG;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    sd_status_t s;
    if ((s = order_after_host_product(plan, st))) return s;
    plan->vals = vals;
    if (plan->bval) SD_CUDA_TRY(fill_bsr(plan, true, st));   // the other families read the caller's array
    return order_before_host_product(plan, st);
}

sd_status_t sd_spmm_host_async(sd_plan_t *plan, const void *B_host, int64_t ldb, float *C_host, int64_t ldc, float alpha,
                         float beta) {
    if (!plan) {
        set_error(SD_ERR_INVALID_ARG, "plan is null");
        return SD_ERR_INVALID_ARG;
    }
    const sd_status_t s = queue_host_product(plan, B_host, ldb, C_host, ldc, alpha, beta);
    if (s) host_give_back(plan);   // the caller may free the host buffers now: no copy that was queued before the error may still run
    return s;
}

sd_status_t sd_plan_sync(sd_plan_t *plan) {
    if (!plan) {
        set_error(SD_ERR_INVALID_ARG, "plan is null");
        return SD_ERR_INVALID_ARG;
    }
    SD_CUDA_TRY(host_give_back(plan));
    return SD_OK;
}

sd_status_t sd_spmm_host(sd_plan_t *plan, const void *B_host, int64_t ldb, float *C_host, int64_t ldc, float alpha,
                         float beta) {
    const sd_status_t s = sd_spmm_host_async(plan, B_host, ldb, C_host, ldc, alpha, beta);
    return s ? s : sd_plan_sync(plan);
}

sd_status_t sd_plan_save(const sd_plan_t *plan, void *buf, size_t cap, size_t *bytes) {
    if (!plan || !bytes) {
        set_error(SD_ERR_INVALID_ARG, "sd_plan_save: plan and bytes must not be null");
        return SD_ERR_INVALID_ARG;
    }
    *bytes = sizeof(BlobHeader);
    if (!buf) return SD_OK;   // size query
    if (cap < sizeof(BlobHeader)) {
        set_error(SD_ERR_INVALID_ARG, "sd_plan_save: the buffer holds %zu bytes, the plan needs %zu", cap, sizeof(BlobHeader));
        return SD_ERR_INVALID_ARG;
    }
    int prev = 0;
    SD_CUDA_TRY(cudaGetDevice(&prev));
    SD_CUDA_TRY(cudaSetDevice(plan->device));
    BlobHeader h;
    memset(&h, 0, sizeof h);
    sd_status_t s = pattern_hash(plan->rowptr, plan->colind, plan->M, plan->nnz, nullptr, &h.pattern);
    if (s == SD_OK) {
        cudaDeviceProp prop;
        const cudaError_t e = cudaGetDeviceProperties(&prop, plan->device);
        if (e != cudaSuccess) s = cuda_fail(e, "cudaGetDeviceProperties");
        else strncpy(h.device_name, prop.name, sizeof h.device_name - 1);
    }
    cudaSetDevice(prev);
    if (s != SD_OK) return s;
    h.magic = kBlobMagic;
    h.version = kBlobVersion;
    h.header_bytes = static_cast<uint32_t>(sizeof(BlobHeader));
    h.M = plan->M; h.K = plan->K; h.N = plan->N; h.nnz = plan->nnz;
    h.dtype = plan->dtype;
    h.family = plan->info.family;
    h.sm_count = plan->info.sm_count;
    h.l2_bytes = plan->info.l2_bytes;
    h.info = plan->info;
    h.has_coo = plan->coo_row ? 1 : 0;
    h.has_blocks = plan->browptr ? 1 : 0;   // informative: the family decides
    h.h_T = plan->h_T;
    h.chunks_long = plan->h_counts.chunks_long;
    h.chunks_long2 = plan->h_counts.chunks_long2;
    h.chunks_long4 = plan->h_counts.chunks_long4;
    h.giants = plan->h_counts.giants;
    memcpy(h.len_hist, plan->h_counts.len_hist, sizeof h.len_hist);
    memcpy(buf, &h, sizeof h);
    return SD_OK;
}

sd_status_t sd_plan_load(const void *blob, size_t bytes, const int32_t *rowptr, const int32_t *colind, const void *vals,
                         sd_plan_t **out) {
    if (out) *out = nullptr;
    if (!blob || !out || bytes < sizeof(BlobHeader)) {
        set_error(SD_ERR_INVALID_ARG, "sd_plan_load: null argument or a blob shorter than its header");
        return SD_ERR_INVALID_ARG;
    }
    BlobHeader h;
    memcpy(&h, blob, sizeof h);
    if (h.magic != kBlobMagic || h.version != kBlobVersion || h.header_bytes != sizeof(BlobHeader) ||
        h.M < 0 || h.nnz < 0 || (h.dtype != SD_F32 && h.dtype != SD_BF16)) {
        set_error(SD_ERR_INVALID_ARG, "sd_plan_load: not a plan blob of this library version");
        return SD_ERR_INVALID_ARG;
    }
    if ((h.M > 0 && !rowptr) || (h.nnz > 0 && (!colind || !vals))) {
        set_error(SD_ERR_INVALID_ARG, "sd_plan_load: the CSR arrays the plan was made for must be given again");
        return SD_ERR_INVALID_ARG;
    }
    // key: device model, then the pattern itself
    int dev = 0;
    SD_CUDA_TRY(cudaGetDevice(&dev));
    cudaDeviceProp prop;
    SD_CUDA_TRY(cudaGetDeviceProperties(&prop, dev));
    if (strncmp(prop.name, h.device_name, sizeof h.device_name) != 0 || prop.multiProcessorCount != h.sm_count ||
        static_cast<int64_t>(prop.l2CacheSize) != h.l2_bytes) {
        set_error(SD_ERR_UNSUPPORTED, "sd_plan_load: the plan was made on '%s' (%d SMs), this device is '%s' (%d SMs)",
                  h.device_name, h.sm_count, prop.name, prop.multiProcessorCount);
        return SD_ERR_UNSUPPORTED;
    }
    if (h.M > 0) {
        int32_t last = 0;
        SD_CUDA_TRY(cudaMemcpy(&last, rowptr + h.M, sizeof last, cudaMemcpyDeviceToHost));
        if (last != h.nnz) {
            set_error(SD_ERR_INVALID_ARG, "sd_plan_load: rowptr[M] = %d, the plan was made for %lld nonzeros", last,
                      (long long)h.nnz);
            return SD_ERR_INVALID_ARG;
        }
    }
    uint64_t pat = 0;
    sd_status_t s = pattern_hash(rowptr, colind, h.M, h.nnz, nullptr, &pat);
    if (s != SD_OK) return s;
    if (pat != h.pattern) {
        set_error(SD_ERR_INVALID_ARG, "sd_plan_load: the sparsity pattern differs from the one the plan was made for");
        return SD_ERR_INVALID_ARG;
    }
    sd_plan *p = new (std::nothrow) sd_plan;
    if (!p) {
        set_error(SD_ERR_ALLOC, "host allocation failed");
        return SD_ERR_ALLOC;
    }
    auto fail = [&](sd_status_t code) {
        free_plan(p);
        return code;
    };
    p->rowptr = rowptr;
    p->colind = colind;
    p->vals = vals;
    p->M = h.M; p->K = h.K; p->N = h.N; p->nnz = h.nnz;
    p->dtype = h.dtype;
    p->device = dev;
    p->info = h.info;
    if (h.has_coo) {
        if ((s = build_coo(p, nullptr))) return fail(s);
    } else if (h.h_T > 0) {
        ScanAccum counts{};
        counts.long_rows = static_cast<unsigned long long>(h.info.long_rows);
        counts.chunks_long = h.chunks_long;
        counts.chunks_long2 = h.chunks_long2;
        counts.chunks_long4 = h.chunks_long4;
        counts.giants = h.giants;
        memcpy(counts.len_hist, h.len_hist, sizeof h.len_hist);
        if ((s = build_schedule(p, h.info.windows, h.h_T, counts, nullptr))) return fail(s);
    } else if (h.family == SD_BSR_TC) {
        if ((s = build_bsr(p, h.info.nnzb16, nullptr))) return fail(s);
    }
    const cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) return fail(cuda_fail(e, "cudaDeviceSynchronize"));
    p->info = h.info;
    *out = p;
    return SD_OK;
}

#pragma GCC visibility pop
}  // extern "C"
