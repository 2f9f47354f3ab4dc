// Whole runs of small 1D grids, FP64 (compiled with --fmad=false like the FP64 stage kernels).
#include "hydro_internal.h"
#include "line_kernel.cuh"

namespace hydro {
int line_ctas_f64(int n) { return line_ctas<double>(n); }
cudaError_t launch_line_f64(const LineLaunch &L, cudaStream_t st) { return launch_line<double>(L, st); }
}  // namespace hydro
