// Launches of the FP64 2D strip kernel (row64_kernel.cuh; compiled with --fmad=false).
#include <math.h>

#include "hydro_internal.h"
#include "row64_kernel.cuh"
#include "stage_launch.cuh"

namespace hydro {

cudaError_t stage_row64(const StageLaunch &L, cudaStream_t st) {
    StageArgs<double> A = make_stage_args<double>(L);
    const long long strips = (A.n[0] + kStrip64Cells - 1) / kStrip64Cells;
    A.tiles_x = (int)strips;
    A.march = L.rows;
    const long long items = strips * ((A.n[1] + A.march - 1) / A.march);
    if (items < 1 || items >= (1LL << 31) - 4) return cudaErrorInvalidValue;
    A.items = (int)items;
    constexpr int warps = kRow64Threads / 32;
    const auto k = L.stage == 1 ? row64_stage_kernel<1, false> : row64_stage_kernel<2, true>;
    k<<<(unsigned)((items + warps - 1) / warps), kRow64Threads, 0, st>>>(A);
    return cudaGetLastError();
}

// Rows a warp marches through on an nx x ny grid: the least (m + 0.7) x (warps the busiest
// scheduler gets), a chunk's prologue (two recoveries and a face) counted as 0.7 rows.  A warp
// alone on its scheduler leaves the FP64 pipe idle between its operations, so fewer than two
// count as 1.5; over many the schedulers even out.
int default_row64_rows(long long nx, long long ny, int sm_count) {
    const double strips = (double)((nx + kStrip64Cells - 1) / kStrip64Cells);
    const double schedulers = 4.0 * (sm_count > 0 ? sm_count : 1);
    int best = 1;
    double best_cost = 0.0;
    for (int m = 1; m <= 128; ++m) {
        const double share = strips * (double)((ny + m - 1) / m) / schedulers;
        const double warps = share > 16.0 ? share + 0.5 : ceil(share);
        const double cost = (m + 0.7) * (warps < 1.5 ? 1.5 : warps);
        if (best_cost == 0.0 || cost < best_cost) best = m, best_cost = cost;
    }
    return best;
}

}  // namespace hydro
