#include "sd_launch.cuh"
#include "sd_hybrid.cuh"

namespace sd {

// `vw`: elements per load of B (piece_width)
cudaError_t run_hybrid_bf16(const HybridArgs &a, int vw, cudaStream_t st) {
    switch (vw) {
    case 8: return launch_hybrid<__nv_bfloat16, 8>(a, st);
    case 4: return launch_hybrid<__nv_bfloat16, 4>(a, st);
    case 2: return launch_hybrid<__nv_bfloat16, 2>(a, st);
    default: return launch_hybrid<__nv_bfloat16, 1>(a, st);
    }
}

}  // namespace sd
