#include "sd_launch.cuh"
#include "sd_hybrid.cuh"

namespace sd {

// `vw`: elements per load of B (piece_width)
cudaError_t run_hybrid_f32(const HybridArgs &a, int vw, cudaStream_t st) {
    switch (vw) {

    case 4: return launch_hybrid<float, 4>(a, st);
    case 2: return launch_hybrid<float, 2>(a, st);
    default: return launch_hybrid<float, 1>(a, st);
    }
}

}  // namespace sd
