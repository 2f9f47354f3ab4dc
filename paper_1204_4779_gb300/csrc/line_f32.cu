// Whole runs of small 1D grids, FP32.
#include "hydro_internal.h"
#include "line_kernel.cuh"

namespace hydro {
int line_ctas_f32(int n) { return line_ctas<float>(n); }
cudaError_t launch_line_f32(const LineLaunch &L, cudaStream_t st) { return launch_line<float>(L, st); }
}  // namespace hydro
