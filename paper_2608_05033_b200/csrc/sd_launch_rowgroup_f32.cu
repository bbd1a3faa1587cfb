#include "sd_launch.cuh"
#include "sd_rowgroup.cuh"

namespace sd {

// `vw`: elements per load of B (piece_width); `sets`: lane sets per row; `terms`: products of a set in one accumulator
cudaError_t run_rowgroup_f32(const SpmmArgs &a, int vw, int sets, int terms, cudaStream_t st) {
    switch (vw) {
    case 4: return launch_rowgroup<float, 4>(a, sets, terms, st);
    case 2: return launch_rowgroup<float, 2>(a, sets, terms, st);
    default: return launch_rowgroup<float, 1>(a, sets, terms, st);
    }
}

}  // namespace sd
