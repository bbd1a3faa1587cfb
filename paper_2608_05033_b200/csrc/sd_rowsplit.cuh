// Family (a): row-split CSR SpMM.  One group of LPR lanes owns one row of A; each lane
// owns NV vectors of VW adjacent columns of the output row and gathers the matching
// 16-byte pieces of the rows of B (paper, case study on af_shell10: a few threads per
// row, several outputs per thread in registers, shuffles share the sparse entries).
#pragma once

#include <cstdlib>

#include "sd_common.cuh"
#include "sd_piece.cuh"

namespace sd {

constexpr int kRowsplitThreads = 256;

// LONG = false: no row exceeds 32 * LPR terms (the plan knows the longest row), so the block-wise
// second accumulator and its instructions are not needed: 9 % faster on the 5-point stencil.
template <typename T, int VW, int LPR, int NV, bool LONG>
__global__ void __launch_bounds__(kRowsplitThreads, LONG ? 5 : 6)
rowsplit_kernel(const SpmmArgs a) {
    constexpr unsigned FULL = 0xffffffffu;
    const int lg = threadIdx.x % LPR;  // lane inside the group
    const int64_t row = (static_cast<int64_t>(blockIdx.x) * kRowsplitThreads + threadIdx.x) / LPR;
    const int cbase = blockIdx.y * (LPR * NV * VW);
    const T *vals = static_cast<const T *>(a.vals);
    const T *B = static_cast<const T *>(a.B);

    int p0 = 0, len = 0;
    if (row < a.S) {
        p0 = __ldg(a.ptr + row);
        len = __ldg(a.ptr + row + 1) - p0;
    }
    // the columns of the first step do not depend on earlier work in the stream
    int myc = 0;
    if (lg < len) myc = __ldg(a.colind + p0 + lg);
    overlap_wait();
    float myv = 0.f;
    if (lg < len) myv = to_float(vals[p0 + lg]);
    // trip counts are made warp-uniform so that the shuffles below are always converged
    const int maxlen = (LPR == 32) ? len : __reduce_max_sync(FULL, len);

    // two-level accumulation: `acc` takes at most 32*LPR terms before it is folded into
    // `tot`, so that a very long row is summed in blocks rather than as one running sum
    float acc[NV][VW], tot[LONG ? NV : 1][LONG ? VW : 1];
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int e = 0; e < VW; ++e) {
            acc[v][e] = 0.f;
            if constexpr (LONG) tot[v][e] = 0.f;
        }

    bool colok[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) colok[v] = cbase + (v * LPR + lg) * VW < a.N;

    // beta != 0: fetch the old C row now so that its latency hides behind the gathers
    float cin[NV][VW];
    if (a.beta != 0.f && row < a.S) {
        const float *crow = a.C + row * a.ldc + cbase;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            if (colok[v]) {
                if constexpr (VW == 1) {
                    cin[v][0] = crow[(v * LPR + lg)];
                } else {
#pragma unroll
                    for (int q = 0; q < VW / 4; ++q) {
                        const float4 o = *(reinterpret_cast<const float4 *>(crow + (v * LPR + lg) * VW) + q);
                        cin[v][4 * q] = o.x; cin[v][4 * q + 1] = o.y; cin[v][4 * q + 2] = o.z; cin[v][4 * q + 3] = o.w;
                    }
                }
            }
        }
    }

    for (int base = 0; base < maxlen; base += LPR) {
        if constexpr (LONG) {
            if (base != 0 && (base / LPR) % 32 == 0) {
#pragma unroll
                for (int v = 0; v < NV; ++v)
#pragma unroll
                    for (int e = 0; e < VW; ++e) {
                        tot[v][e] += acc[v][e];
                        acc[v][e] = 0.f;
                    }
            }
        }
        // the group fetches LPR (column, value) pairs with one coalesced load each ...
        if (base != 0) {
            const bool in = base + lg < len;
            myc = in ? __ldg(a.colind + p0 + base + lg) : 0;
            myv = in ? to_float(vals[p0 + base + lg]) : 0.f;
        }
        const int cnt = min(LPR, maxlen - base);
        // ... and hands them round by shuffle
#pragma unroll 4
        for (int q = 0; q < cnt; ++q) {
            const int c = (LPR == 1) ? myc : __shfl_sync(FULL, myc, q, LPR);
            const float av = (LPR == 1) ? myv : __shfl_sync(FULL, myv, q, LPR);
            if (base + q < len) {
                const T *brow = b_row(B, c, a.ldb_bytes) + cbase;
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    if (colok[v]) {
                        float b[VW];
                        RowLoad<T, VW>::ld(brow + (v * LPR + lg) * VW, b);
                        if constexpr (VW == 1) {
                            acc[v][0] = fmaf(av, b[0], acc[v][0]);
                        } else {
#pragma unroll
                            for (int e = 0; e < VW; e += 2) fma_pair(acc[v][e], acc[v][e + 1], av, b[e], b[e + 1]);
                        }
                    }
                }
            }
        }
    }

    overlap_next();
    if (row < a.S) {
        float *crow = a.C + row * a.ldc + cbase;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
#pragma unroll
            for (int e = 0; e < VW; ++e) {
                float t = acc[v][e];
                if constexpr (LONG) t += tot[v][e];
                t *= a.alpha;
                if (a.beta != 0.f) t = fmaf(a.beta, cin[v][e], t);
                acc[v][e] = t;
            }
            if (colok[v]) store_cols<VW>(crow + (v * LPR + lg) * VW, acc[v], 1.f, 0.f);
        }
    }
}

// C = beta * C for an M x N matrix (alpha == 0, or a matrix without nonzeros).
static __global__ void scale_c_kernel(float *C, int64_t ldc, int64_t M, int32_t N, float beta) {
    const int64_t total = M * N;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < total;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        float *p = C + (i / N) * ldc + (i % N);
        *p = (beta == 0.f) ? 0.f : beta * *p;
    }
}

template <typename T, int VW, int LPR, int NV>
cudaError_t launch_rowsplit_one(const SpmmArgs &a, cudaStream_t st) {
    const int rows_per_cta = kRowsplitThreads / LPR;
    dim3 grid(static_cast<unsigned>((a.S + rows_per_cta - 1) / rows_per_cta),
              static_cast<unsigned>((a.N + LPR * NV * VW - 1) / (LPR * NV * VW)));
    if (a.max_len > 0 && a.max_len <= 32 * LPR) return launch_overlapped(rowsplit_kernel<T, VW, LPR, NV, false>, grid, kRowsplitThreads, 0, st, a);
    return launch_overlapped(rowsplit_kernel<T, VW, LPR, NV, true>, grid, kRowsplitThreads, 0, st, a);
}

// Lane geometry for a dense width: VW elements per 16-byte load when `vec`, LPR lanes per
// row (a power of two), NV vectors per lane; wider rows are covered by grid.y slabs.
// Two vectors per lane (from `two_from` vectors per row on; 0: never) halve the per-nonzero instruction overhead (index
// broadcast, address arithmetic) per byte gathered; the merge-path kernel measures faster with one vector and more lanes per row.
struct LaneGeom {
    int vw, lpr, nv;
};
inline int geom_nv_override() { return switches().geom_nv; }
inline LaneGeom lane_geometry(int64_t N, bool vec, int vecw, int two_from) {
    LaneGeom g;
    g.vw = vec ? vecw : 1;
    const int64_t units = (N + g.vw - 1) / g.vw;
    if (!vec) {
        int lpr = 1;
        while (lpr < 32 && lpr < units) lpr <<= 1;
        g.lpr = lpr;
        g.nv = units > 32 ? 4 : 1;
        return g;
    }
    const bool two = two_from > 0 && units >= two_from && geom_nv_override() != 1;
    const int64_t per = two ? (units + 1) / 2 : units;
    int lpr = 1;
    while (lpr < 32 && lpr < per) lpr <<= 1;
    g.lpr = lpr;
    g.nv = (two || units > 32) ? 2 : 1;
    return g;
}

// Two vectors per lane where they leave no more lanes idle and a group still covers a 128-byte line with one load (a gather costs a
// cycle of L1 per line it touches): from nine vectors on (1 M stencil rows at 48 fp32 columns 210 -> 143 us, at 64 also before).  fp32
// also at five to seven with C beyond 10 MB (24 columns: 1 M rows 107 -> 80, 160,000 rows 11.5 -> 10.9, 62,500 5.2 -> 5.6) and, where
// operands come from DRAM and the lines are the smaller cost, at four and eight: C beyond 40 MB (32 columns: 1 M rows 111 -> 89, 360,000
// rows 38.1 -> 31.6, 250,000 18.6 -> 19.0; 16 columns: 640,000 rows 36.6 -> 33.3, 360,000 14.4 -> 16.6).  bf16 lanes hold twice the sums:
// slower there (64 columns 137 -> 155).  Rows of more than 64 nonzeros, from 16 vectors on: fewer lanes request fewer pairs of a row at a
// time, and one long row is what such a matrix waits for (the longest 900: 24 fp32 columns 123 -> 255 us, 96 bf16 columns 187 -> 280).
inline int rowsplit_two_from(const SpmmArgs &a, bool bf16) {
    if (a.max_len <= 0 || a.max_len > 64) return 16;
    if (bf16) return 9;
    const int64_t units = (a.N + 3) / 4, c_bytes = a.S * a.N * 4;
    return units >= 4 && c_bytes >= (units > 4 && units < 8 ? 10000000 : 40000000) ? 4 : 9;
}

template <typename T>
cudaError_t launch_rowsplit(const SpmmArgs &a, bool vec, cudaStream_t st) {
    constexpr int VWV = vec_width<T>::value;
    const LaneGeom g = lane_geometry(a.N, vec, VWV, rowsplit_two_from(a, sizeof(T) == 2));
    if (vec && g.nv == 2) {
        switch (g.lpr) {
        case 2: return launch_rowsplit_one<T, VWV, 2, 2>(a, st);
        case 4: return launch_rowsplit_one<T, VWV, 4, 2>(a, st);
        case 8: return launch_rowsplit_one<T, VWV, 8, 2>(a, st);
        case 16: return launch_rowsplit_one<T, VWV, 16, 2>(a, st);
        case 32: return launch_rowsplit_one<T, VWV, 32, 2>(a, st);
        }
        return cudaErrorInvalidValue;
    }
#define SD_RS_CASE(L)                                                  \
    case L:                                                            \
        if (vec) return launch_rowsplit_one<T, VWV, L, 1>(a, st);      \
        return (g.nv == 4) ? launch_rowsplit_one<T, 1, 32, 4>(a, st)   \
                           : launch_rowsplit_one<T, 1, L, 1>(a, st);
    switch (g.lpr) {
        SD_RS_CASE(1)
        SD_RS_CASE(2)
        SD_RS_CASE(4)
        SD_RS_CASE(8)
        SD_RS_CASE(16)
        SD_RS_CASE(32)
    }
#undef SD_RS_CASE
    return cudaErrorInvalidValue;
}

}  // namespace sd
