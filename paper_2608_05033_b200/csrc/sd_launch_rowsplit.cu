#include "sd_launch.cuh"
#include "sd_rowgroup.cuh"
#include "sd_rowsplit.cuh"
#include "sd_rowsplit_narrow.cuh"
#include "sd_chunk_sums.cuh"

namespace sd {

// Lane sets per row of the row-group kernel, or 0 where the kernels below are ahead.  Measured on Poisson rows of 3 to 44 nonzeros
// (40,000 to 1 M of them), 5-point stencils and blocks (125 to 131 per row), 8 to 256 columns, both value types.  Some of it, us: the
// kernels below / one set / four sets
//   not whole 16-byte loads   always (41 columns: 1.8 to 3.9 times as fast as one scalar per lane)
//   few rows                  four sets as soon as rows are 8 long: one set leaves the GPU idle (5,000 rows of 30 at 64 columns
//                             17.9 -> 5.3 us, at 128 bf16 24.9 -> 6.7)
//   short rows of one length  the plain kernel, whose loop has no last, tested step, where neighbouring rows share rows of B, so that
//                             instructions are the bound, from five loads on (stencils, us plain / one set: 5 points, 360,000 rows at 32, 64
//                             fp32 columns 29.5, 48.8 / 39.9, 77.1, 1 M rows at 64 bf16 columns 115 / 129).  Others wait for their gathers:
//                             one set from 12 nonzeros (400,000 rows of 12, 15 at 64 fp32 columns 136, 163 / 131, 156), from 6 with up to
//                             four loads (60,000 rows of 6, 12 at 16 fp32 columns 4.7, 6.5 / 4.3, 5.6, 7-point stencils 30.0 / 28.2) and, but
//                             where the plain kernel takes two loads per lane, up to eight (60,000 rows of 6, 12 at 24 fp32 columns 6.6,
//                             10.9 / 5.9, 7.8, 400,000 33.0, 52.1 / 41.1, 50.6) and beyond 16; bf16 with one load always (1 M rows of 4
//                             26.3 / 24.8, of 15 105 / 81, 5-point stencils 14.8 / 13.7)
//   8 columns                 four sets from 8 to 63 nonzeros (24: fp32 - / 18.6 / 15.3, bf16 - / 17.4 / 13.2), one below (3: 10.9 / 8.9 / 17.7)
//   up to 8 loads             one set below 16 (32 columns, 3, 12: 24.0, 14.5 / 23.5, 14.5 / 71, 24); from there by the loads: 2: four to
//                             64 (16 bf16 columns, 24: 17.0 / 20.3 / 16.8), the set kernel with as many where B is beyond 8 MB, with fp32
//                             values below 40 nonzeros (16 bf16 columns, set kernel / four sets here, 400,000 rows of 16, 24, 44: 41.6, 56.2, 91.7 /
//                             46.0, 61.7, 95.0, 8 fp32 columns 37.9, 54.6, 88.1 / 40.6, 58.2, 89.0); 4: the set kernel below (16 columns, 24: 17.7 / 18.6 / 19.0; 1 M
//                             rows of 40 at 32 bf16 columns 349 / 346 / 406); others: one to 64 (24 columns, 24, 44: 18.7, 29.8 / 15.6,
//                             25.0 / -), then four (32 columns, 125: 41.6 / 34.8 / 27.3).  8: two, as many as in the set kernel, which has
//                             2,048 threads on an SM for 1,280: that is ahead where B is far from the SMs, beyond 16 MB with fp32 values and
//                             with bf16 on rows below 32, unless some row is much longer and walked faster here
//                             (32 columns, set kernel / two sets, 60,000 rows of 24, 44: 16.2, 25.3 / 15.3, 23.4, 200,000 47.1, 77.6 /
//                             49.9, 79.0, 400,000 104, 158 / 120, 174; 64 bf16 columns 20.5, 30.4 / 19.1, 26.8, 61.4, 92.3 / 62.3, 86.4,
//                             133, 195 / 141, 195)
//   9 to 16 loads             one set from 8 (64 columns, 12, 24: 27.7, 47.2 / 24.9, 38.9 / 29.4, 42.7; 128 bf16 columns, 24: 63.7 / 47.3
//                             / 54.6; 6: 56.3 / 58.2 / 86.0), and on shorter rows where the loads are no power of two (96 bf16 columns, 3: 83.7 /
//                             76.0 / 121); bf16 two of 16 loads from 32 and four from 40, of even length fp32 the set
//                             kernel to 64 (64 columns, 35, set kernel / two sets: 60,000 rows 32.7 / 32.8, 200,000 109 / 127, 400,000 302 / 345)
//   17 to 32 loads            one set (128 columns, 6, 24: 89.9, 82.9 / 83.5, 72.3 / 109, 77.2), bf16 from 16 (200 columns, 12, 24: 66.1, 66.7 /
//                             70.7, 57.8 / 72.1, 58.0); four from 40 (200 bf16 columns, 44: 77.5 / 64.4 / 58.8)
//   beyond 32                 the plain kernel has two loads per lane and half the warps: one set to 12, then four (256 columns, 6, 12:
//                             240, 109 / 179, 109 / 180, 113)
static int one_length_from(const SpmmArgs &a, int units, bool bf16) {
    if (bf16 && units == 1) return 1;
    if (units <= 4) return 6;
    if (a.shared || units > (bf16 ? 16 : 32)) return 16;
    const bool two = !bf16 && units >= rowsplit_two_from(a, bf16);
    return units > 16 || (units <= 8 && !two) ? 6 : 12;
}
// Products of a lane set in one accumulator: no more than in the kernels below where those would take the rows.  The set kernel and, of
// two lanes, the plain kernel add 64 before they fold, the plain kernel of four 128, of more at least 256.  Rows beyond are folded every 64
// (kGroupFold), in kernels with a second accumulator and four CTAs per SM for five (rows of 24, the longest 900, at 64 bf16 columns 42.9
// -> 46.5 us, at 128 60.1 -> 62.4; with 64 everywhere also 400,000 rows of 35, the longest about 70, at 48 fp32 columns 275 -> 312, and
// 6,000 rows of 150, the longest 300, at 64 and 200 bf16 columns 10.6 -> 11.7 and 45.3 -> 51.6).
struct RowGroupForm {
    int sets, terms;
};
static RowGroupForm rowgroup_form(const SpmmArgs &a, int dtype, int vw, bool vec) {
    const int units = (a.N + vw - 1) / vw;
    const int64_t mean = a.mean_len;
    int lanes = 1;
    while (lanes < 32 && lanes < units) lanes <<= 1;
    const bool fills = a.S * lanes >= static_cast<int64_t>(sm_count_cached()) * 5 * kRowGroupThreads;
    const bool pow2 = (units & (units - 1)) == 0, bf16 = dtype == SD_BF16;
    const bool even = a.max_len <= 4 * mean, far = a.b_bytes > 16000000 && even;
    const bool one_length = mean < 16 && a.max_len <= 2 * mean;
    int sets = 0;
    if (!vec) sets = mean >= 48 || (!fills && mean >= 8) ? 4 : 1;
    else if (!fills && mean >= 8) sets = 4;
    else if (one_length) sets = mean >= one_length_from(a, units, bf16) ? 1 : 0;
    else if (units == 2 && mean >= 16 && mean < (bf16 ? 64 : 40) && a.b_bytes > 8000000 && even) sets = 0;
    else if (a.N <= 8) sets = mean < 8 ? 1 : mean < 64 ? 4 : 0;
    else if (units == 8 && mean >= 16 && mean < 64) sets = far && (!bf16 || mean < 32) ? 0 : 2;
    else if (units <= 8) sets = mean < 16 ? 1 : units == 2 ? (mean < 64 ? 4 : 0) : units == 4 ? 0 : mean < 64 ? 1 : 4;
    else if (units == 16 && !bf16 && mean >= 32 && mean < 64 && even) sets = 0;
    else if (units <= 16) sets = mean >= 40 ? 4 : pow2 && mean >= 32 ? 2 : mean >= 8 || !pow2 ? 1 : 0;
    else if (units <= 32) sets = mean >= 40 ? 4 : !bf16 || mean >= 16 ? 1 : 0;
    else sets = mean >= 12 ? 4 : 1;
    if (a.max_len <= 0 || a.max_len > static_cast<int64_t>(kRowGroupTerms) * sets) sets = 0;
    const bool alone = !vec || (!fills && mean >= 8);
    const bool set_kernel = units <= 16 && pow2 && mean >= 16;
    return {sets, alone || units > 16 ? 256 : units <= 2 || set_kernel ? 64 : units <= 4 ? 128 : 256};
}

cudaError_t run_rowsplit(const SpmmArgs &a, int dtype, int vw_now, cudaStream_t st) {
    const int vw = dtype == SD_F32 ? 4 : 8;
    const bool vec = vw_now == vw;
    if (a.N >= 1 && a.N <= 4 && !switches().no_narrow) {   // one to four columns: lanes share a row, not its columns
        if (dtype == SD_F32) return launch_rowsplit_narrow<float>(a, st);
        return launch_rowsplit_narrow<__nv_bfloat16>(a, st);
    }
    const RowGroupForm form = rowgroup_form(a, dtype, vw_now, vec);
    if (form.sets > 0)
        return dtype == SD_F32 ? run_rowgroup_f32(a, vw_now, form.sets, form.terms, st) : run_rowgroup_bf16(a, vw_now, form.sets, form.terms, st);
    // 8 to 64 columns (fp32; 8 to 128 bf16) as whole 16-byte vectors and long rows: several lane sets per row
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
