// Sums of the nonzeros of a row (or of a part of one) by a group of lanes: some of them stand across the columns of B and C,
// the others share the nonzeros.  Used by the hybrid schedule and by the row-group kernel.
#pragma once

#include <type_traits>

#include "sd_common.cuh"
#include "sd_piece.cuh"

namespace sd {

// Per-lane view of B and C for one column slab.  EXACT: every lane has columns in every slab, so no gather is tested (a tested
// one clears its registers first: five instructions more).
template <typename T, int VW, int LPR, int NV, bool EXACT = false>
struct LaneCols {
    const T *B;
    int cbase;
    bool ok[NV];
    __device__ __forceinline__ LaneCols(const void *b, int32_t N, int lg) {
        const int slab = blockIdx.y * (LPR * NV * VW);
        cbase = slab + lg * VW;
        B = static_cast<const T *>(b) + cbase;
#pragma unroll
        for (int v = 0; v < NV; ++v) ok[v] = cbase + v * LPR * VW < N;
    }
    // gathers of one row of B; `use` = false gathers nothing (row 0 of B may hold non-finite values)
    __device__ __forceinline__ void gather(int col, uint32_t ldb_bytes, bool use, Piece<T, VW> (&b)[NV]) const {
        const T *row = b_row(B, col, ldb_bytes);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            if (use && (EXACT || ok[v])) b[v].ld(row + v * LPR * VW);
            else b[v].zero();
        }
    }
    __device__ __forceinline__ void fma(float w, const Piece<T, VW> (&b)[NV], float (&acc)[NV][VW]) const {
#pragma unroll
        for (int v = 0; v < NV; ++v) b[v].fma(w, acc[v]);
    }
    __device__ __forceinline__ void store(float *crow, const float (&acc)[NV][VW], float alpha, float beta) const {
#pragma unroll
        for (int v = 0; v < NV; ++v)
            if (EXACT || ok[v]) store_cols<VW>(crow + cbase + v * LPR * VW, acc[v], alpha, beta);
    }
};

template <int NV, int VW>
__device__ __forceinline__ void clear_acc(float (&acc)[NV][VW]) {
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int e = 0; e < VW; ++e) acc[v][e] = 0.f;
}

template <int NV, int VW>
__device__ __forceinline__ void add_acc(float (&acc)[NV][VW], const float (&more)[NV][VW]) {
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int e = 0; e < VW; ++e) acc[v][e] += more[v][e];
}

// Sum over the LANES / LPR lane sets of a group (a fixed order: results repeat bit for bit).
template <int LANES, int LPR, int NV, int VW>
__device__ __forceinline__ void sum_sets(float (&acc)[NV][VW], unsigned mask) {
#pragma unroll
    for (int d = LANES / 2; d >= LPR; d >>= 1)
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
            for (int e = 0; e < VW; ++e) acc[v][e] += __shfl_xor_sync(mask, acc[v][e], d);
}

// Nonzeros [p0, p1) by a group of LANES lanes.  A step loads NB x LANES (column, value) pairs, one coalesced load of each
// per NB, and requests the next step's before this step's gathers.  The pairs go round through shared memory: four columns or
// four values per 16-byte load, which all lanes of a set read together, cost a quarter of the instructions and of the L1 cycles of
// as many shuffles.  Q gathers of a lane are in flight together.  Whole steps run without any test; only the
// last, partly filled one tests every pair: nothing may be gathered for a pair beyond the end (row 0 of B may hold
// non-finite values, and 0 * Inf is NaN).
// FOLD: a set adds at most kGroupFold products in one accumulator before they go to a second one, so the longest chain of sums of a
// row of L nonzeros is kGroupFold + L / (G * kGroupFold) long, not L / G.  The second accumulator is up to 16 registers, so rows
// that are shorter do without it.
constexpr int kGroupFold = 64;
template <int LPR> constexpr int kGroupLoads = LPR >= 4 ? 1 : 4 / LPR;   // loads of pairs per step: at least four gathers per lane and step
template <int THREADS, int LPR>
struct GroupStage {   // of a CTA; with one lane across the columns every lane has its own nonzeros, with two shuffles are as good (5 % less at 8 columns)
    static constexpr int N = LPR <= 2 ? 1 : THREADS * kGroupLoads<LPR>;
    alignas(16) int col[N];
    alignas(16) float val[N];
};
template <typename T, int VW, int LPR, int NV, int LANES, bool EXACT, bool FOLD, typename Args, int THREADS>
__device__ __forceinline__ void group_sum(const Args &a, const LaneCols<T, VW, LPR, NV, EXACT> &lc, GroupStage<THREADS, LPR> &stage, int p0,
                                          int p1, unsigned mask, float (&acc)[NV][VW]) {
    constexpr int G = LANES / LPR;
    constexpr int NB = kGroupLoads<LPR>;
    constexpr int PER = NB * LPR;                       // gathers of a lane per step
    constexpr int QM = NV * VW * sizeof(T) > 16 ? 4 : 8;
    constexpr int Q = PER < QM ? PER : QM;
    const T *vals = static_cast<const T *>(a.vals);
    const int lg = threadIdx.x % LANES, k = lg / LPR;
    int *const cols = LPR <= 2 ? nullptr : stage.col + threadIdx.x / LANES * (LANES * NB);
    float *const ws = LPR <= 2 ? nullptr : stage.val + threadIdx.x / LANES * (LANES * NB);
    int c[NB];
    float w[NB];
    auto fetch = [&](int p) {
#pragma unroll
        for (int n = 0; n < NB; ++n) {
            const bool in = p + n * LANES + lg < p1;
            c[n] = in ? __ldg(a.colind + p + n * LANES + lg) : -1;
            w[n] = in ? to_float(vals[p + n * LANES + lg]) : 0.f;
        }
    };
    auto step = [&](int p, auto whole_tag) {
        constexpr bool WHOLE = decltype(whole_tag)::value;
        int4 own_col = make_int4(c[0], c[1 % NB], c[2 % NB], c[3 % NB]);
        float4 own_val = make_float4(w[0], w[1 % NB], w[2 % NB], w[3 % NB]);
        if constexpr (LPR == 2) {
            own_col = make_int4(__shfl_sync(mask, c[0], k, LANES), __shfl_sync(mask, c[0], G + k, LANES), __shfl_sync(mask, c[1], k, LANES),
                                __shfl_sync(mask, c[1], G + k, LANES));
            own_val = make_float4(__shfl_sync(mask, w[0], k, LANES), __shfl_sync(mask, w[0], G + k, LANES), __shfl_sync(mask, w[1], k, LANES),
                                  __shfl_sync(mask, w[1], G + k, LANES));
        }
        if constexpr (LPR > 2) {
            __syncwarp(mask);   // the step before has been read
#pragma unroll
            for (int n = 0; n < NB; ++n) {
                const int j = n * LANES + lg, at = (j / (4 * G) * G + j % G) * 4 + j / G % 4;
                cols[at] = c[n];
                ws[at] = w[n];
            }
            __syncwarp(mask);
        }
        constexpr int QS = WHOLE || Q < 4 ? Q : 4;
        if (WHOLE) fetch(p + NB * LANES);
#pragma unroll 1
        for (int i0 = 0; i0 < PER; i0 += QS) {   // one batch at a time: unrolled, the compiler starts all of them and spills
            if (!WHOLE && p + i0 * G >= p1) break;
            Piece<T, VW> b[QS][NV];
#pragma unroll
            for (int u = 0; u < QS; u += 4) {
                const int4 x = LPR <= 2 ? own_col : *reinterpret_cast<const int4 *>(cols + (i0 + u) * G + 4 * k);
                const int col[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                for (int v = 0; v < 4; ++v) lc.gather(col[v], a.ldb_bytes, WHOLE || col[v] >= 0, b[u + v]);
            }
#pragma unroll
            for (int u = 0; u < QS; u += 4) {
                const float4 x = LPR <= 2 ? own_val : *reinterpret_cast<const float4 *>(ws + (i0 + u) * G + 4 * k);
                const float wv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                for (int v = 0; v < 4; ++v) lc.fma(wv[v], b[u + v], acc);
            }
        }
    };
    float tot[FOLD ? NV : 1][FOLD ? VW : 1];
    if constexpr (FOLD) clear_acc(tot);
    [[maybe_unused]] int steps = 0;
    int p = p0;
    fetch(p);
#pragma unroll 1
    for (; p + NB * LANES <= p1; p += NB * LANES) {
        step(p, std::true_type{});
        if constexpr (FOLD) {
            if (++steps == kGroupFold / PER) {
                steps = 0;
                add_acc(tot, acc);
                clear_acc(acc);
            }
        }
    }
    if (p < p1) step(p, std::false_type{});
    if constexpr (FOLD) add_acc(acc, tot);
    sum_sets<LANES, LPR, NV, VW>(acc, mask);
}

}  // namespace sd
