// A lane's share of a row of B: VW adjacent elements, loaded with one instruction and kept as they come from
// memory until they are multiplied (bf16 pairs are widened at the multiply-add, so that a gather in flight holds
// half the registers of its widened form).
#pragma once

#include "sd_common.cuh"

namespace sd {

// (x, y) += a * (bx, by): one packed fp32 instruction, each half rounded like fmaf.
__device__ __forceinline__ void fma_pair(float &x, float &y, float a, float bx, float by) {
    asm("{\n\t.reg .b64 a2, b2, c2;\n\t"
        "mov.b64 a2, {%4, %4};\n\t"
        "mov.b64 b2, {%2, %3};\n\t"
        "mov.b64 c2, {%0, %1};\n\t"
        "fma.rn.f32x2 c2, a2, b2, c2;\n\t"
        "mov.b64 {%0, %1}, c2;\n\t}"
        : "+f"(x), "+f"(y)
        : "f"(bx), "f"(by), "f"(a));
}

template <typename T, int VW> struct Piece;

template <> struct Piece<float, 4> {
    float4 r;
    __device__ __forceinline__ void ld(const float *p) { r = live_load(reinterpret_cast<const float4 *>(p)); }
    __device__ __forceinline__ void zero() { r = make_float4(0.f, 0.f, 0.f, 0.f); }
    __device__ __forceinline__ void fma(float a, float (&acc)[4]) const {
        fma_pair(acc[0], acc[1], a, r.x, r.y);
        fma_pair(acc[2], acc[3], a, r.z, r.w);
    }
};
template <> struct Piece<float, 2> {
    float2 r;
    __device__ __forceinline__ void ld(const float *p) { r = live_load(reinterpret_cast<const float2 *>(p)); }
    __device__ __forceinline__ void zero() { r = make_float2(0.f, 0.f); }
    __device__ __forceinline__ void fma(float a, float (&acc)[2]) const {
        acc[0] = fmaf(a, r.x, acc[0]);
        acc[1] = fmaf(a, r.y, acc[1]);
    }
};
template <> struct Piece<float, 1> {
    float r;
    __device__ __forceinline__ void ld(const float *p) { r = live_load(p); }
    __device__ __forceinline__ void zero() { r = 0.f; }
    __device__ __forceinline__ void fma(float a, float (&acc)[1]) const { acc[0] = fmaf(a, r, acc[0]); }
};

// bf16 is the upper half of a float
__device__ __forceinline__ void fma_bf16x2(float &x, float &y, float a, uint32_t w) {
    fma_pair(x, y, a, __uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
}
template <> struct Piece<__nv_bfloat16, 8> {
    uint4 r;
    __device__ __forceinline__ void ld(const __nv_bfloat16 *p) { r = live_load(reinterpret_cast<const uint4 *>(p)); }
    __device__ __forceinline__ void zero() { r = make_uint4(0, 0, 0, 0); }
    __device__ __forceinline__ void fma(float a, float (&acc)[8]) const {
        fma_bf16x2(acc[0], acc[1], a, r.x);
        fma_bf16x2(acc[2], acc[3], a, r.y);
        fma_bf16x2(acc[4], acc[5], a, r.z);
        fma_bf16x2(acc[6], acc[7], a, r.w);
    }
};
template <> struct Piece<__nv_bfloat16, 4> {
    uint2 r;
    __device__ __forceinline__ void ld(const __nv_bfloat16 *p) { r = live_load(reinterpret_cast<const uint2 *>(p)); }
    __device__ __forceinline__ void zero() { r = make_uint2(0, 0); }
    __device__ __forceinline__ void fma(float a, float (&acc)[4]) const {
        fma_bf16x2(acc[0], acc[1], a, r.x);
        fma_bf16x2(acc[2], acc[3], a, r.y);
    }
};
template <> struct Piece<__nv_bfloat16, 2> {
    uint32_t r;
    __device__ __forceinline__ void ld(const __nv_bfloat16 *p) { r = live_load(reinterpret_cast<const uint32_t *>(p)); }
    __device__ __forceinline__ void zero() { r = 0; }
    __device__ __forceinline__ void fma(float a, float (&acc)[2]) const { fma_bf16x2(acc[0], acc[1], a, r); }
};
template <> struct Piece<__nv_bfloat16, 1> {
    unsigned short r;
    __device__ __forceinline__ void ld(const __nv_bfloat16 *p) { r = live_load(reinterpret_cast<const uint16_t *>(p)); }
    __device__ __forceinline__ void zero() { r = 0; }
    __device__ __forceinline__ void fma(float a, float (&acc)[1]) const {
        acc[0] = fmaf(a, __uint_as_float(static_cast<uint32_t>(r) << 16), acc[0]);
    }
};

// Elements per load that the operands allow: the widest of 16, 8, 4 (and, with bf16, 2) bytes of B such that every
// lane's share starts at a multiple of its size, with the matching store of C.
inline int piece_width(int dtype, int64_t N, const void *B, int64_t ldb, const float *C, int64_t ldc) {
    const int es = dtype == SD_F32 ? 4 : 2;
    for (int vw = 16 / es; vw > 1; vw >>= 1) {
        const int cb = vw >= 4 ? 4 : vw;   // floats per store of C
        if (N % vw == 0 && ldb % vw == 0 && ldc % cb == 0 && (reinterpret_cast<uintptr_t>(B) & (vw * es - 1)) == 0 &&
            (reinterpret_cast<uintptr_t>(C) & (cb * 4 - 1)) == 0)
            return vw;
    }
    return 1;
}

}  // namespace sd
