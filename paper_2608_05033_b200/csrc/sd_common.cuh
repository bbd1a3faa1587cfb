// Shared device/host helpers of the SpMM library (sm_100a only).
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <atomic>

#include "../../include/sd.h"

namespace sd {

// ---- error reporting (thread-local text + code) --------------------------------
void set_error(sd_status_t code, const char *fmt, ...);
sd_status_t cuda_fail(cudaError_t e, const char *what);

#define SD_CUDA_TRY(expr)                                   \
    do {                                                    \
        cudaError_t e__ = (expr);                           \
        if (e__ != cudaSuccess) return cuda_fail(e__, #expr); \
    } while (0)

// ---- element access -------------------------------------------------------------
__device__ __forceinline__ float to_float(float v) { return v; }
__device__ __forceinline__ float to_float(__nv_bfloat16 v) { return __bfloat162float(v); }

// Vector width in elements of a 16-byte load of T.
template <typename T> struct vec_width;
template <> struct vec_width<float> { static constexpr int value = 4; };
template <> struct vec_width<__nv_bfloat16> { static constexpr int value = 8; };

// B is read with these.  With overlapped launches (below) the kernel that writes B may still run when the one that reads it
// has begun: the loads are coherent, not read-only (__ldg, ld.global.nc, const __restrict__ kernel parameters promise that nobody
// writes during the kernel), and volatile, so that none is moved to before overlap_wait().  A's values and the scratch of an
// earlier kernel are ordinary C++ loads, which the wait's memory clobber orders; what never changes during the life of a plan
// (row pointers, columns, plan tables) may take the read-only path.  Ordinary loads for B too cost 6 % at one column (R-MAT scale
// 20: 120.5 -> 128.5 us), these nothing.
#define SD_LIVE_LOAD(V, asm_load, ...)                                      \
    __device__ __forceinline__ V live_load(const V *p) {                    \
        V r;                                                                \
        asm volatile(asm_load : __VA_ARGS__ : "l"(p));                      \
        return r;                                                           \
    }
SD_LIVE_LOAD(float4, "ld.global.v4.f32 {%0, %1, %2, %3}, [%4];", "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w))
SD_LIVE_LOAD(float2, "ld.global.v2.f32 {%0, %1}, [%2];", "=f"(r.x), "=f"(r.y))
SD_LIVE_LOAD(float, "ld.global.f32 %0, [%1];", "=f"(r))
SD_LIVE_LOAD(uint4, "ld.global.v4.u32 {%0, %1, %2, %3}, [%4];", "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w))
SD_LIVE_LOAD(uint2, "ld.global.v2.u32 {%0, %1}, [%2];", "=r"(r.x), "=r"(r.y))
SD_LIVE_LOAD(uint32_t, "ld.global.u32 %0, [%1];", "=r"(r))
SD_LIVE_LOAD(uint16_t, "ld.global.u16 %0, [%1];", "=h"(r))
#undef SD_LIVE_LOAD

// 32 bytes in one load, from a multiple of 32: a warp that reads 1 KB of consecutive data, 32 bytes a lane, passes L1 in eight
// cycles, where two 16-byte loads a lane pass it in sixteen (each spans all of the 1 KB).
struct alignas(32) Words8 {
    uint32_t w[8];
};
__device__ __forceinline__ Words8 live_load(const Words8 *p) {
    Words8 r;
    asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r.w[0]), "=r"(r.w[1]), "=r"(r.w[2]), "=r"(r.w[3]), "=r"(r.w[4]), "=r"(r.w[5]), "=r"(r.w[6]), "=r"(r.w[7])
                 : "l"(p));
    return r;
}

// Load VW consecutive elements of T and widen to float.
template <typename T, int VW> struct RowLoad;

template <> struct RowLoad<float, 4> {
    __device__ __forceinline__ static void ld(const float *p, float (&o)[4]) {
        const float4 v = live_load(reinterpret_cast<const float4 *>(p));
        o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
    }
};
template <> struct RowLoad<float, 1> {
    __device__ __forceinline__ static void ld(const float *p, float (&o)[1]) { o[0] = live_load(p); }
};
template <> struct RowLoad<__nv_bfloat16, 8> {
    __device__ __forceinline__ static void ld(const __nv_bfloat16 *p, float (&o)[8]) {
        const uint4 v = live_load(reinterpret_cast<const uint4 *>(p));
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {       // bf16 is the upper half of a float
            o[2 * i] = __uint_as_float(w[i] << 16);
            o[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
        }
    }
};
template <> struct RowLoad<__nv_bfloat16, 1> {
    __device__ __forceinline__ static void ld(const __nv_bfloat16 *p, float (&o)[1]) {
        o[0] = __uint_as_float(static_cast<uint32_t>(live_load(reinterpret_cast<const uint16_t *>(p))) << 16);
    }
};

// Rows of B are what the kernels re-read: an L2 policy that evicts them last keeps more of B
// resident against the streams of A and C (measured on the GCN workload: 5 to 19 % less time).
__device__ __forceinline__ uint64_t l2_keep_policy() {
    uint64_t pol;
    asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
// RowLoad with that policy, read-only: for kernels that are launched without overlap.
template <typename T, int VW> struct RowLoadKeep;
template <> struct RowLoadKeep<float, 4> {
    __device__ __forceinline__ static void ld(const float *p, float (&o)[4], uint64_t pol) {
        asm("ld.global.nc.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
            : "=f"(o[0]), "=f"(o[1]), "=f"(o[2]), "=f"(o[3])
            : "l"(p), "l"(pol));
    }
};
template <> struct RowLoadKeep<float, 1> {
    __device__ __forceinline__ static void ld(const float *p, float (&o)[1], uint64_t pol) {
        asm("ld.global.nc.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(o[0]) : "l"(p), "l"(pol));
    }
};

// How one output row leaves the registers: C = alpha*acc + beta*C (beta == 0 never reads C).
template <int VW>
__device__ __forceinline__ void store_cols(float *c, const float (&acc)[VW], float alpha, float beta) {
    if constexpr (VW == 1) {
        float r = alpha * acc[0];
        if (beta != 0.f) r += beta * *c;
        *c = r;
    } else if constexpr (VW == 2) {
        float2 r = make_float2(alpha * acc[0], alpha * acc[1]);
        if (beta != 0.f) {
            const float2 o = *reinterpret_cast<const float2 *>(c);
            r.x += beta * o.x; r.y += beta * o.y;
        }
        __stcs(reinterpret_cast<float2 *>(c), r);
    } else {
#pragma unroll
        for (int q = 0; q < VW / 4; ++q) {
            float4 *p = reinterpret_cast<float4 *>(c) + q;
            float4 r = make_float4(alpha * acc[4 * q], alpha * acc[4 * q + 1], alpha * acc[4 * q + 2],
                                   alpha * acc[4 * q + 3]);
            if (beta != 0.f) {
                const float4 o = *p;
                r.x += beta * o.x; r.y += beta * o.y; r.z += beta * o.z; r.w += beta * o.w;
            }
            __stcs(p, r);   // C is written once and not read again: streaming store, first to leave L2
        }
    }
}

// Address of row `col` of B given a per-lane base pointer: one 32 x 32 -> 64 bit multiply-add
// (column indices are non-negative and the row pitch in bytes is below 2^32, checked on the host).
template <typename T>
__device__ __forceinline__ const T *b_row(const T *base, int col, uint32_t ldb_bytes) {
    return reinterpret_cast<const T *>(reinterpret_cast<const char *>(base) +
                                       static_cast<uint64_t>(static_cast<uint32_t>(col)) * ldb_bytes);
}

// Arguments common to the CSR kernels.
struct SpmmArgs {
    const int32_t *ptr;     // row pointer array, [S+1]
    const int32_t *colind;  // [nnz]
    const void *vals;       // [nnz] float or bf16
    const void *B;
    float *C;
    int64_t ldb, ldc;
    uint32_t ldb_bytes;     // ldb * sizeof(element of B)
    int64_t S;              // number of rows
    int32_t N;
    float alpha, beta;
    int64_t max_len;        // longest row if known (0: unknown); lets the row-split kernel drop its second accumulator
    int64_t mean_len;       // mean row length rounded up if known (0: unknown): lanes per row of the narrow row-split kernel
    int64_t b_bytes;        // of the rows and columns of B that the product reads
    bool shared;            // neighbouring rows name the same rows of B: four nonzeros per occupied 16x16 block at least
};

// A/B measurement switches (none is needed in normal use).  The environment is read once, at the
// first use in the process (thread-safe), never on the sd_spmm path.
struct Switches {
    bool no_coo;           // SD_NO_COO: generic merge kernel at one to four columns
    bool bsr_simt;         // SD_BSR_SIMT: SIMT block kernel instead of the tensor-core one
    bool no_narrow;        // SD_NO_NARROW: wide row-split kernel at one to four columns
    int geom_nv;           // SD_GEOM_NV: 1 forces one vector per lane
    int ksplit_g;          // SD_KSPLIT_G: lane sets per row (0: rule, 1: off)
    int narrow_g;          // SD_NARROW_G: lanes per row of the narrow row-split kernel (0: rule)
};
const Switches &switches();

// Per-device caches of launch facts (SM count, resident CTAs of a kernel instance, attributes already set):
// one slot per device ordinal, published with atomics, so that a process driving several GPUs, or several
// host threads making their first call together, never reads another device's value or a torn one.
constexpr int kMaxDevices = 64;
inline int current_device() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) dev = 0;
    return dev;
}
inline int sm_count_cached() {
    static std::atomic<int> cache[kMaxDevices];
    const int dev = current_device();
    int v = dev < kMaxDevices ? cache[dev].load(std::memory_order_relaxed) : 0;
    if (v > 0) return v;
    v = 148;
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    if (dev < kMaxDevices) cache[dev].store(v, std::memory_order_relaxed);
    return v;
}
// CTAs of `kernel` (threads per CTA, no dynamic shared memory) that are resident together on one SM of the current device.
template <typename Kernel>
inline int occupancy_cached(std::atomic<int> (&cache)[kMaxDevices], Kernel kernel, int threads) {
    const int dev = current_device();
    int v = dev < kMaxDevices ? cache[dev].load(std::memory_order_relaxed) : 0;
    if (v > 0) return v;
    v = 8;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, kernel, threads, 0) != cudaSuccess || v < 1) v = v < 1 ? 1 : 8;
    if (dev < kMaxDevices) cache[dev].store(v, std::memory_order_relaxed);
    return v;
}

// ---- overlapped launches ---------------------------------------------------------------------
// Kernels of this library that follow one another in a stream overlap their ends: a kernel launched with
// launch_overlapped starts once every CTA of the kernel before it has called overlap_next() or ended, and may
// read what never changes during the life of a plan (row pointers, columns, plan tables).  Before it touches
// anything that earlier work in the stream may write (values, B, C, scratch) every thread calls overlap_wait(), which
// returns when the earlier kernels have completed and their writes are visible.  Each kernel waits, so completion
// is transitive.  A small kernel (2,048 rows, 32 columns) repeats every 6.1 us without this.
//
// Where a kernel calls overlap_next() matters as much.  Called first thing, it lets several kernels wait side by side on SMs
// that still work, and on matrices between one CTA per SM and a full GPU that cost up to twice the time (products of 24
// plans in turn, 20,000 rows of 20 at four bf16 columns: 12.7 us, 6.7 without overlap).  So the row, hybrid and segmented
// kernels call it when their gathers are done (6.1 us there; 60,000 rows of 3 at two columns 5.2 -> 3.5, R-MAT scale 14 at 64
// columns 13.0 -> 12.3, at two columns 10.4 -> 7.9), or leave it to their end.  The block kernel and the chunk sums, whose next
// kernel has tables to fetch, stay with the start (128 block-rows at 256 bf16 columns 3.6 us, 4.3 at the end).
__device__ __forceinline__ void overlap_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void overlap_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename... Params, typename... Args>
inline cudaError_t launch_overlapped(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args &&...args) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, Params(args)...);
}

inline int ceil_div(int64_t a, int64_t b) { return static_cast<int>((a + b - 1) / b); }

}  // namespace sd
