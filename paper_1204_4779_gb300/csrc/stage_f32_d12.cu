// FP32 RK-stage kernels, dims 1 and 2 (FMAs are written out; the compiler contracts none):
// one-plane tiles, and in dim 2 row tiles that march along y (stage_rows.cu).
#include "stage_launch.cuh"

namespace hydro {

cudaError_t stage_f32_d1(const StageLaunch &L, cudaStream_t st, bool prepare_only) {
    HYDRO_STAGE_CASE(float, 1, 128, 1, false)
    HYDRO_STAGE_CASE(float, 1, 256, 1, false)
    return cudaErrorInvalidValue;
}

cudaError_t stage_f32_d2(const StageLaunch &L, cudaStream_t st, bool prepare_only) {
    HYDRO_STAGE_CASE(float, 2, 32, 8, false)
    HYDRO_STAGE_CASE(float, 2, 64, 4, false)
    HYDRO_STAGE_CASE(float, 2, 16, 16, false)
    HYDRO_STAGE_CASE(float, 2, 32, 16, false)
    // row tiles: strips of 64 columns per warp, marching along y
    if (L.tile_y == 1) return stage_rows_f32(L, st, prepare_only);
    return cudaErrorInvalidValue;
}

}  // namespace hydro
