#include "sd_launch.cuh"
#include "sd_rowsplit.cuh"
#include "sd_rowsplit_narrow.cuh"
#include "sd_chunk_sums.cuh"

namespace sd {

cudaError_t run_rowsplit(const SpmmArgs &a, int dtype, bool vec, cudaStream_t st) {
    if (a.N >= 1 && a.N <= 4 && !switches().no_narrow) {   // one to four columns: lanes share a row, not its columns
        if (dtype == SD_F32) return launch_rowsplit_narrow<float>(a, vec, st);
        return launch_rowsplit_narrow<__nv_bfloat16>(a, vec, st);
    }
    // 8 to 64 columns (fp32; 8 to 128 bf16) as whole 16-byte vectors and long rows: several lane sets per row
    const int vw = dtype == SD_F32 ? 4 : 8;
    if (vec && a.N % vw == 0 && a.N / vw <= 16 && ((a.N / vw) & (a.N / vw - 1)) == 0) {
        const int lpr = a.N / vw;
        const int g = ksplit_group(a.mean_len, lpr);
        if (g > 1) {
            if (dtype == SD_F32) return launch_rowsplit_ksplit<float>(a, lpr, g, st);
            return launch_rowsplit_ksplit<__nv_bfloat16>(a, lpr, g, st);
        }
    }
    if (dtype == SD_F32) return launch_rowsplit<float>(a, vec, st);
    return launch_rowsplit<__nv_bfloat16>(a, vec, st);
}

cudaError_t run_chunk_reduce(const float *chunk_out, const int32_t *chunk_ptr, const int32_t *rows, int64_t nl, float *C,
                             int64_t ldc, int32_t N, float alpha, float beta, cudaStream_t st, int32_t skip_above) {
    auto kernel = N % 4 == 0 ? chunk_reduce_kernel<4> : chunk_reduce_kernel<1>;   // 4: scratch rows are then 16-byte aligned
    return launch_overlapped(kernel, static_cast<unsigned>((nl + 7) / 8), 256, 0, st, chunk_out, chunk_ptr, rows, nl, C, ldc, N,
                             alpha, beta, skip_above);
}

cudaError_t run_chunk_reduce_wide(const float *chunk_out, const int32_t *chunk_ptr, const int32_t *rows,
                                  const int32_t *list, int64_t count, float *C, int64_t ldc, int32_t N, float alpha,
                                  float beta, cudaStream_t st) {
    auto kernel = N % 4 == 0 ? chunk_reduce_wide_kernel<4> : chunk_reduce_wide_kernel<1>;
    return launch_overlapped(kernel, static_cast<unsigned>(count), 256, 0, st, chunk_out, chunk_ptr, rows, list, C, ldc, N,
                             alpha, beta);
}

cudaError_t run_scale_c(float *C, int64_t ldc, int64_t M, int32_t N, float beta, cudaStream_t st) {
    const int64_t total = M * N;
    const int blocks = static_cast<int>(std::min<int64_t>((total + 255) / 256, 148 * 16));
    scale_c_kernel<<<blocks, 256, 0, st>>>(C, ldc, M, N, beta);
    return cudaGetLastError();
}

}  // namespace sd
