// Narrow dense operands (N <= 4, SpMV included) of family (b): a segmented reduction over the nonzeros in storage order (the COO
// form that the paper's Sec. 3.1 lists for SpMV-like widths).
//
// With one to four columns a lane group per row has nothing to share.  Here the nonzeros are dealt out evenly: a warp owns a
// contiguous range of them and walks it 256 (three or four columns: 128) at a time; a lane adds up eight (four) consecutive
// nonzeros by itself, and one segmented scan over the warp's lanes joins the rows that run across lanes.  A row that lies inside
// the range is complete: its lane writes alpha * sum + beta * C.  The first and the last row of the range may continue in the
// neighbours': their sums go to a carry list, two entries per range in order, (first row, sum) and (last row, sum), or, where the
// range is one single row, (row, sum) and (row, 0), so that entries of one row stay adjacent.  The list is a row-sorted list
// of values itself: a second kernel reduces it the same way, and the few entries that leaves over are added one row per thread.
// Rows without nonzeros are found from the row pointers and get beta * C.  Every row is written by one thread and every sum has
// a fixed order: results repeat bit for bit, no float atomics.
//
// Where rows begin: a bit per item and the row of every eighth (0.6 bytes per nonzero; one column, no rows without nonzeros), else
// a row index per item (4 bytes).
//
// What bounds it: L1, a cycle per line of B that a gather touches, 32 for 32 unrelated rows.  Where a few columns hold much of the
// matrix, the HOT form keeps their rows of B in shared memory (one CTA per SM), where 32 unrelated words cost about five
// cycles; the plan owns a copy of the columns with those renamed to slots (coo_hot_columns).
//
// 32.4 M nonzeros, R-MAT scale 20, us, with a scan per 32 nonzeros and a carry per 256 before (one fp32 column and all with frequent
// columns kept: as far as that paid then), and now:
//     columns    1           2            3            4
//     fp32       116 -> 83   170 -> 111   225 -> 170   238 -> 157
//     bf16       102 -> 83   160 -> 98    237 -> 156   267 -> 137
// 60 M nonzeros in rank-size rows, uniform columns: one column 251 -> 262, two 390 -> 303, four 512 -> 393.  Small matrices at one
// column are level (scale 13 to 16 between 5.8 -> 6.2 and 11.2 -> 10.7), scale 17 16.4 -> 15.1, bf16 14.9 -> 14.7.  Tried: the next step's
// columns and values requested ahead (registers: 86 -> 97), the frequent columns' products formed in storage order and dealt out through
// shared memory (110), the next launch let in before the carries are written (scale 16 11.5 -> 12.1), the open sum folded in shared
// memory every 32 steps (86 -> 88).
#pragma once

#include <type_traits>

#include "sd_common.cuh"
#include "sd_launch.cuh"

namespace sd {

constexpr int kCooHotThreads = 1024;
constexpr int coo_threads(int N) { return N == 1 ? 128 : 256; }

struct CooArgs {
    // Items are the nonzeros after `shift` others that are nothing: so many that item 0 of the columns lies on a multiple of what a lane
    // loads at once.  The arrays start at item 0; those of the caller begin at item `shift`.
    const int32_t *row;      // [count] row of every item (ascending), or with `starts` of every eighth
    const uint8_t *starts;   // one column without empty rows: bit u of byte g: item 8g + u begins a row
    const int32_t *colind;   // [count] column of every nonzero
    const void *vals;        // [count] values of A; carry list: [count][N] float partial sums
    unsigned shift;
    const void *B;
    uint32_t ldb_bytes;
    int64_t count;           // items
    float *C;
    int64_t ldc;
    float alpha, beta;
    const int32_t *rowptr;   // [M + 1], to find the rows without nonzeros (they get beta * C)
    int64_t M;
    int warps, per_warp;     // that work, ranges of each
    uint64_t range;          // steps of a range, 32 bits of them behind the point: range r begins with the whole steps of r times this
    int spread;              // neighbouring ranges go to different CTAs
    int32_t *carry_row;      // [2 * warps * per_warp] out
    float *carry_val;        // [2 * warps * per_warp][N] out
    const int32_t *hot_cols; // HOT: ascending columns whose rows of B the kernel keeps; colind names slot i of them as i | bit 31
    int32_t hot;
};

template <typename T> __device__ __forceinline__ T from_float(float v);   // of a value that T holds
template <> __device__ __forceinline__ float from_float<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_float<__nv_bfloat16>(float v) {
    return __ushort_as_bfloat16(static_cast<unsigned short>(__float_as_uint(v) >> 16));
}

// N floats of row `col` of B with one load where VEC says that its alignment allows it.
template <typename T, int N, bool VEC>
__device__ __forceinline__ void coo_row_of_b(const T *p, float (&b)[N]) {
    if constexpr (VEC && N == 4 && sizeof(T) == 4) {
        RowLoad<T, 4>::ld(p, b);
    } else if constexpr (VEC && N == 2 && sizeof(T) == 4) {
        const float2 v = live_load(reinterpret_cast<const float2 *>(p));
        b[0] = v.x, b[1] = v.y;
    } else if constexpr (VEC && N == 4) {
        const uint2 v = live_load(reinterpret_cast<const uint2 *>(p));
        b[0] = __uint_as_float(v.x << 16), b[1] = __uint_as_float(v.x & 0xFFFF0000u);
        b[2] = __uint_as_float(v.y << 16), b[3] = __uint_as_float(v.y & 0xFFFF0000u);
    } else if constexpr (VEC && N == 2) {
        const uint32_t v = live_load(reinterpret_cast<const uint32_t *>(p));
        b[0] = __uint_as_float(v << 16), b[1] = __uint_as_float(v & 0xFFFF0000u);
    } else {
#pragma unroll
        for (int e = 0; e < N; ++e) {
            float t[1];
            RowLoad<T, 1>::ld(p + e, t);
            b[e] = t[0];
        }
    }
}

// U consecutive elements, widened: one load, from a multiple of its size.
template <typename T, int U>
__device__ __forceinline__ void load_wide(const T *p, float (&o)[U]) {
    if constexpr (U * sizeof(T) == 32) {
        const Words8 v = live_load(reinterpret_cast<const Words8 *>(p));
#pragma unroll
        for (int u = 0; u < U; ++u) o[u] = __uint_as_float(v.w[u]);
    } else if constexpr (U * sizeof(T) == 16) {
        RowLoad<T, U>::ld(p, o);
    } else {
        coo_row_of_b<T, U, true>(p, o);
    }
}
// ... or two, or one per element, as `align`, the address of the array, allows.
template <typename T, int U>
__device__ __forceinline__ void load_run(const T *p, unsigned align, float (&o)[U]) {
    if (align % (U * sizeof(T)) == 0) {
        load_wide<T, U>(p, o);
    } else if (align % (U / 2 * sizeof(T)) == 0) {
        float low[U / 2], high[U / 2];
        load_wide<T, U / 2>(p, low);
        load_wide<T, U / 2>(p + U / 2, high);
#pragma unroll
        for (int u = 0; u < U / 2; ++u) o[u] = low[u], o[U / 2 + u] = high[u];
    } else {
#pragma unroll
        for (int u = 0; u < U; ++u) o[u] = to_float(p[u]);
    }
}
template <int U>
__device__ __forceinline__ void load_ints(const int32_t *p, int (&o)[U]) {
    float t[U];
    load_wide<float, U>(reinterpret_cast<const float *>(p), t);
#pragma unroll
    for (int u = 0; u < U; ++u) o[u] = __float_as_int(t[u]);
}

// Rows without nonzeros have no writer among the runs: one share of them per warp.
template <int N>
__device__ __forceinline__ void coo_empty_rows(const CooArgs &a, int64_t share, int64_t shares) {
    const int64_t rpc = (a.M + shares - 1) / shares;
    for (int64_t rr = share * rpc + (threadIdx.x & 31); rr < min(a.M, (share + 1) * rpc); rr += 32)
        if (__ldg(a.rowptr + rr) == __ldg(a.rowptr + rr + 1)) {
#pragma unroll
            for (int e = 0; e < N; ++e) {
                float *pc = a.C + rr * a.ldc + e;
                *pc = (a.beta != 0.f) ? a.beta * *pc : 0.f;
            }
        }
}

template <typename T, int N, bool VEC, bool HOT, bool BITS, bool TURN = false>
__global__ void __launch_bounds__(HOT ? kCooHotThreads : coo_threads(N), HOT ? 1 : (TURN ? 8 : N == 1 ? 9 : 4))
coo_kernel(const CooArgs a) {
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int U = coo_items(N), STEP = 32 * U;
    static_assert(!TURN || (N == 1 && !HOT), "what a warp keeps to deal out its gathers");
    extern __shared__ __align__(16) char coo_hot_raw[];
    T *kept = reinterpret_cast<T *>(coo_hot_raw);
    overlap_wait();
    if constexpr (HOT) {
        constexpr int AT = 16 / N;   // a thread fetches them in batches: one by one, 32,768 columns took 30 us
        for (int i0 = threadIdx.x; i0 < a.hot; i0 += AT * kCooHotThreads) {
            int c[AT];
            float b[AT][N];
#pragma unroll
            for (int j = 0; j < AT; ++j) c[j] = i0 + j * kCooHotThreads < a.hot ? __ldg(a.hot_cols + i0 + j * kCooHotThreads) : -1;
#pragma unroll
            for (int j = 0; j < AT; ++j)
                if (c[j] >= 0) coo_row_of_b<T, N, VEC>(b_row(static_cast<const T *>(a.B), c[j], a.ldb_bytes), b[j]);
#pragma unroll
            for (int j = 0; j < AT; ++j)
                if (c[j] >= 0)
#pragma unroll
                    for (int e = 0; e < N; ++e) kept[(i0 + j * kCooHotThreads) * N + e] = from_float<T>(b[j][e]);
        }
        __syncthreads();
    }
    // TURN: one column of a large matrix without frequent columns.  A gather takes 32 consecutive nonzeros there and not every eighth: those of a
    // long row lie so close that some share a line of B (60 M nonzeros in rank-size rows, fp32 272 -> 262 us, 12 M in
    // rows of 30,000 fp32 59 -> 54, bf16 52 -> 45; with few steps per warp the way through shared memory costs more than that, R-MAT scale
    // 17 15.0 -> 16.5).
    __shared__ __align__(16) float turns[TURN ? coo_threads(N) / 32 : 1][TURN ? STEP : 4];
    [[maybe_unused]] float *const turn = turns[TURN ? threadIdx.x >> 5 : 0];
    const int lane = threadIdx.x & 31;
    const int w = a.spread ? (threadIdx.x >> 5) * gridDim.x + blockIdx.x : (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w >= a.warps) return;
    if (a.M > 0) coo_empty_rows<N>(a, w, a.warps);
    const T *vals = static_cast<const T *>(a.vals), *B = static_cast<const T *>(a.B);
    const unsigned va = static_cast<unsigned>(reinterpret_cast<uintptr_t>(vals));

    auto emit = [&](int row, const float (&v)[N]) {
#pragma unroll
        for (int e = 0; e < N; ++e) {
            float *pc = a.C + static_cast<int64_t>(row) * a.ldc + e;
            *pc = (a.beta != 0.f) ? fmaf(a.beta, *pc, a.alpha * v[e]) : a.alpha * v[e];
        }
    };
    // One range for most matrices.  The open sum below takes one addition per step, so a range is at most kCooRange steps long: one billion
    // nonzeros would make it 740, and the longest chain of sums with it.
    for (int n = 0; n < a.per_warp; ++n) {
        const int range = w + n * a.warps, s0 = static_cast<int>(range * a.range >> 32), s1 = static_cast<int>((range + 1) * a.range >> 32);
        auto carry = [&](int which, int row, const float (&v)[N]) {
            const int64_t at = 2 * range + which;
            a.carry_row[at] = row;
#pragma unroll
            for (int e = 0; e < N; ++e) a.carry_val[at * N + e] = v[e];
        };
        const int first_row = __ldg(a.row + static_cast<int64_t>(s0) * (BITS ? 32 : STEP));
        int open_row = first_row;   // the row that reached the end of the step before ...
        float open[N] = {};         // ... and its sum so far (both the same in all lanes)
        for (int s = s0; s < s1; ++s) {
            const unsigned k0 = static_cast<unsigned>(s) * STEP + lane * U, count = static_cast<unsigned>(a.count);   // below 2^31 + STEP
            int col[U], r[U];
            float av[U];
            unsigned starts = 0;    // items that begin a row
            int row_in = 0;         // the row that is open where the lane begins ...
            int row_out = 0;        // ... and where it ends
            const bool whole = k0 - lane * U >= a.shift && k0 - lane * U + STEP <= count;   // the same in all lanes: every item is a nonzero
            if (whole) {
                if constexpr (TURN) {
#pragma unroll
                    for (int u = 0; u < U; ++u) col[u] = __ldg(a.colind + (k0 - lane * U + u * 32 + lane));
                } else {
                    load_ints<U>(a.colind + k0, col);
                }
                if constexpr (!BITS) load_ints<U>(a.row + k0, r);
                load_run<T, U>(vals + k0, va, av);
            } else {                // items before the first nonzero are zeros of its row, those past the end of the last one's
                const int pad = BITS ? 0 : __ldg(a.row + a.count - 1);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const bool ok = k0 + u >= a.shift && k0 + u < count;
                    col[u] = ok ? __ldg(a.colind + k0 + u) : 0;
                    av[u] = ok ? to_float(vals[k0 + u]) : 0.f;
                    r[u] = BITS ? 0 : (k0 + u < count ? __ldg(a.row + k0 + u) : pad);
                }
            }
            if constexpr (BITS) {
                starts = __ldg(a.starts + s * 32 + lane);
                row_in = __ldg(a.row + s * 32 + lane);
                row_out = row_in + __popc(starts >> 1);
                row_in -= starts & 1u;
                if (s == s0 && lane == 0) {
                    row_in = first_row;
                    starts &= ~1u;
                }
            }
            float b[U][N];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if constexpr (HOT) {   // every lane reads a slot (the others slot 0), those outside also their row of B
                    const bool in = col[u] < 0;
                    const T *q = kept + (in ? col[u] & 0x7fffffff : 0) * N;
                    if constexpr (VEC && N == 2 && sizeof(T) == 4) {
                        const float2 v = *reinterpret_cast<const float2 *>(q);
                        b[u][0] = v.x, b[u][1] = v.y;
                    } else {
#pragma unroll
                        for (int e = 0; e < N; ++e) b[u][e] = to_float(q[e]);
                    }
                    if (!in) coo_row_of_b<T, N, VEC>(b_row(B, col[u], a.ldb_bytes), b[u]);
                } else {
                    coo_row_of_b<T, N, VEC>(b_row(B, col[u], a.ldb_bytes), b[u]);
                }
            }
            if constexpr (TURN) {
                if (whole) {   // dealt out in order
                    __syncwarp();
#pragma unroll
                    for (int u = 0; u < U; ++u) turn[u * 32 + lane] = b[u][0];
                    __syncwarp();
#pragma unroll
                    for (int u = 0; u < U; u += 4) {
                        const float4 v = *reinterpret_cast<const float4 *>(turn + lane * U + u);
                        b[u][0] = v.x, b[u + 1][0] = v.y, b[u + 2][0] = v.z, b[u + 3][0] = v.w;
                    }
                }
            }
            if (!whole)   // they gathered row 0: never let its contents (Inf, NaN) in
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (k0 + u < a.shift || k0 + u >= count)
#pragma unroll
                        for (int e = 0; e < N; ++e) b[u][e] = 0.f;
            if constexpr (!BITS) {
                const int before = __shfl_up_sync(FULL, r[U - 1], 1);
                row_in = lane == 0 ? open_row : before;
                row_out = r[U - 1];
                starts = r[0] != row_in;
#pragma unroll
                for (int u = 1; u < U; ++u) starts |= static_cast<unsigned>(r[u] != r[u - 1]) << u;
            }
            // The lane's runs: the first may have begun before, the last may go on; those between are complete rows.  UPDATE: one column with
            // beta, where a lane has up to seven of them: they wait for one round trip for the old values of C and not for one each (R-MAT
            // scale 20, 32.4 M nonzeros fp32 130 -> 102 us, bf16 127 -> 98, scale 17 22.5 -> 18.0).
            float sum[N] = {}, top[N] = {};
            [[maybe_unused]] float old_top = 0.f;
            bool closed = false;
            auto runs = [&](auto update_tag) {
                constexpr bool UPDATE = decltype(update_tag)::value;
                unsigned held = 0;
                int now = row_in;
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const bool begins = starts >> u & 1u;
                    float done[N];
                    if (begins) {
                        if (closed && !UPDATE) emit(now, sum);
                        if (closed) held |= 1u << u;
#pragma unroll
                        for (int e = 0; e < N; ++e) {
                            done[e] = sum[e];
                            if (!closed) top[e] = sum[e];
                            sum[e] = 0.f;
                        }
                        closed = true;
                        now = BITS ? now + 1 : r[u];
                    }
#pragma unroll
                    for (int e = 0; e < N; ++e) {
                        sum[e] = fmaf(av[u], b[u][e], sum[e]);
                        if (UPDATE && begins) b[u][e] = done[e];
                    }
                }
                if constexpr (UPDATE) {   // all old values are requested before the first is needed
                    auto c_of = [&](int u) {
                        return a.C + static_cast<int64_t>(BITS ? row_in + __popc(starts & ((1u << u) - 1u)) : r[u - 1]) * a.ldc;
                    };
                    float old[U];
#pragma unroll
                    for (int u = 1; u < U; ++u) old[u] = held >> u & 1u ? *c_of(u) : 0.f;
                    if (closed && row_in != first_row) old_top = a.C[static_cast<int64_t>(row_in) * a.ldc];
#pragma unroll
                    for (int u = 1; u < U; ++u)
                        if (held >> u & 1u) *c_of(u) = fmaf(a.beta, old[u], a.alpha * b[u][0]);
                }
            };
            if (N == 1 && a.beta != 0.f) runs(std::bool_constant<N == 1>{});
            else runs(std::false_type{});
            if (lane == 0) {
#pragma unroll
                for (int e = 0; e < N; ++e) (closed ? top[e] : sum[e]) += open[e];
            }
            const unsigned ends = __ballot_sync(FULL, closed) & (FULL >> (31 - lane));
            const int dist = lane - (ends ? 31 - __clz(ends) : 0);
#pragma unroll
            for (int d = 1; d < 32; d <<= 1)
#pragma unroll
                for (int e = 0; e < N; ++e) {
                    const float up = __shfl_up_sync(FULL, sum[e], d);
                    if (dist >= d) sum[e] += up;
                }
#pragma unroll
            for (int e = 0; e < N; ++e) {
                const float in = __shfl_up_sync(FULL, sum[e], 1);
                if (lane > 0) top[e] += in;
                open[e] = __shfl_sync(FULL, sum[e], 31);
            }
            open_row = __shfl_sync(FULL, row_out, 31);
            if (closed) {
                if (row_in == first_row) carry(0, row_in, top);
                else if (N == 1 && a.beta != 0.f) a.C[static_cast<int64_t>(row_in) * a.ldc] = fmaf(a.beta, old_top, a.alpha * top[0]);
                else emit(row_in, top);
            }
        }
        if (lane == 0) {   // what is still open at the end of the range; one single row: (row, sum), (row, 0)
            const float none[N] = {};
            if (open_row == first_row) {
                carry(0, open_row, open);
                carry(1, open_row, none);
            } else {
                carry(1, open_row, open);
            }
        }
    }
}

// The carry list, reduced the same way: a warp per 128 entries, one row-segmented scan per 32.  The entries it leaves over are
// two per warp again.
template <int N>
__global__ void __launch_bounds__(256)
coo_carry_kernel(const CooArgs a) {
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int PER = kCooCarryChunk / 32;
    overlap_wait();
    const int lane = threadIdx.x & 31;
    const int64_t c = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    if (c * kCooCarryChunk >= a.count) return;
    const float *pvals = static_cast<const float *>(a.vals);
    const int64_t k0 = c * kCooCarryChunk + lane, last = a.count - 1;
    int r[PER];
    float p[PER][N];
#pragma unroll
    for (int u = 0; u < PER; ++u) {   // written by the kernel before: no read-only loads; entries past the end continue the last row with zeros
        const int64_t k = k0 + u * 32;
        r[u] = a.row[min(k, last)];
#pragma unroll
        for (int e = 0; e < N; ++e) p[u][e] = k <= last ? pvals[k * N + e] : 0.f;
    }
    // A run is written when it closes: the run of the first row goes to the carry list (it may have begun earlier), every other
    // one is a complete row.
    const int first_row = __shfl_sync(FULL, r[0], 0);
    auto emit = [&](int row, const float (&v)[N]) {
        if (row == first_row) {
            a.carry_row[2 * c] = row;
#pragma unroll
            for (int e = 0; e < N; ++e) a.carry_val[(2 * c) * N + e] = v[e];
        } else {
#pragma unroll
            for (int e = 0; e < N; ++e) {
                float *pc = a.C + static_cast<int64_t>(row) * a.ldc + e;
                *pc = (a.beta != 0.f) ? fmaf(a.beta, *pc, a.alpha * v[e]) : a.alpha * v[e];
            }
        }
    };
    int crow = first_row;   // the run that reached the end of the previous 32 entries ...
    float cval[N] = {};     // ... and its sum so far (both warp-uniform)
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int rp = __shfl_up_sync(FULL, r[u], 1);
        const unsigned starts = __ballot_sync(FULL, lane == 0 || rp != r[u]);
        const int my_start = 31 - __clz(starts & (FULL >> (31 - lane)));   // first lane of this lane's run
        const int dist = lane - my_start;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
#pragma unroll
            for (int e = 0; e < N; ++e) {
                const float vu = __shfl_up_sync(FULL, p[u][e], d);
                if (dist >= d) p[u][e] += vu;
            }
        }
        const bool cont = __shfl_sync(FULL, r[u], 0) == crow;
        if (cont) {                 // the open run continues in the lanes of lane 0's run
            if (my_start == 0) {
#pragma unroll
                for (int e = 0; e < N; ++e) p[u][e] += cval[e];
            }
        } else if (lane == 0) {     // it ended exactly at the 32-entry boundary
            emit(crow, cval);
        }
        if (lane < 31 && ((starts >> (lane + 1)) & 1u)) emit(r[u], p[u]);   // runs that end inside these 32 entries
        crow = __shfl_sync(FULL, r[u], 31);                                  // the run reaching lane 31 stays open
#pragma unroll
        for (int e = 0; e < N; ++e) cval[e] = __shfl_sync(FULL, p[u][e], 31);
    }
    if (lane == 0) {   // what is still open; all one run: (row, sum), (row, 0)
        a.carry_row[2 * c + 1] = crow;
        const bool single = crow == first_row;
        if (single) a.carry_row[2 * c] = crow;
#pragma unroll
        for (int e = 0; e < N; ++e) {
            if (single) a.carry_val[(2 * c) * N + e] = cval[e];
            a.carry_val[(2 * c + 1) * N + e] = single ? 0.f : cval[e];
        }
    }
}

// Level 3: one thread per run of equal rows in a short carry list.
template <int N>
__global__ void coo_final_kernel(const int32_t *row, const float *val, int64_t count, float *C,
                                 int64_t ldc, float alpha, float beta) {
    const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    overlap_wait();
    if (i >= count) return;
    const int r = row[i];
    if (i > 0 && row[i - 1] == r) return;
    float s[N];
#pragma unroll
    for (int e = 0; e < N; ++e) s[e] = 0.f;
    for (int64_t j = i; j < count && row[j] == r; ++j)
#pragma unroll
        for (int e = 0; e < N; ++e) s[e] += val[j * N + e];
#pragma unroll
    for (int e = 0; e < N; ++e) {
        float *pc = C + static_cast<int64_t>(r) * ldc + e;
        *pc = (beta != 0.f) ? fmaf(beta, *pc, alpha * s[e]) : alpha * s[e];
    }
}

// Plan time: the row of every item, or of every eighth.
static __global__ void coo_rows_kernel(const int32_t *__restrict__ rowptr, int64_t M, int64_t nnz, int64_t shift, int64_t every, int64_t count,
                                       int32_t *__restrict__ row) {
    const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x, k = min(max(i * every - shift, int64_t{0}), nnz - 1);
    if (i >= count) return;
    int64_t lo = 0, hi = M;   // last row with rowptr[row] <= k
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (rowptr[mid] <= k) lo = mid;
        else hi = mid;
    }
    row[i] = static_cast<int32_t>(lo);
}
// A bit per item that begins a row after the first; every row has one (`starts` is cleared before).  Row pointers beyond the nonzeros, which
// nobody has checked unless the caller asked for it, set none: the bits end with the nonzeros.
static __global__ void coo_starts_kernel(const int32_t *__restrict__ rowptr, int64_t M, int64_t nnz, unsigned shift, unsigned *__restrict__ starts) {
    const int64_t r = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    const int first = r < M ? __ldg(rowptr + r) : 0;
    if (first <= 0 || first >= nnz) return;
    const unsigned k = static_cast<unsigned>(first) + shift;
    atomicOr(starts + (k >> 5), 1u << (k & 31));
}

}  // namespace sd
