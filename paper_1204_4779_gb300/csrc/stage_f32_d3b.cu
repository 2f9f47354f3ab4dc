// FP32 RK-stage kernels, dim 3: tiles 16x16, 32x16, 16x8 (see stage_f32_d3.cu); 16x16 and 16x8
// also in the manifest forms, 16x8 also with TMA plane staging.  16x8 with look-ahead staging and
// nothing stored, the default, runs the strip kernels (stage_strip3.cu).
#include "stage_launch.cuh"

namespace hydro {

cudaError_t stage_f32_d3b(const StageLaunch &L, cudaStream_t st, bool prepare_only) {
    HYDRO_STAGE_CASE_M(float, 3, 16, 16, true)
    HYDRO_STAGE_CASE(float, 3, 32, 16, true)
    if (L.tile_x == 16 && L.tile_y == 8) {
        if (L.prefetch == 1 && L.manifest == 0) return stage_strip3_f32(L, st, prepare_only);
        if (L.prefetch == 2)
            return L.occupancy == 3 ? run_or_prepare_tma<float, 3, 16, 8, 3>(L, st, prepare_only)
                                    : run_or_prepare_tma<float, 3, 16, 8, 2>(L, st, prepare_only);
        if (L.manifest == 1) return run_or_prepare<float, 3, 16, 8, 1, 3, 1>(L, st, prepare_only);
        if (L.manifest == 2) return run_or_prepare<float, 3, 16, 8, 1, 3, 2>(L, st, prepare_only);
        return L.occupancy == 3 ? run_or_prepare<float, 3, 16, 8, 0, 3>(L, st, prepare_only)
                                : run_or_prepare<float, 3, 16, 8, 0, 2>(L, st, prepare_only);
    }
    return cudaErrorInvalidValue;
}

}  // namespace hydro
