// Launches of the FP32 2D strip kernels (row_kernel.cuh).
#include "hydro_internal.h"
#include "row_kernel.cuh"
#include "stage_launch.cuh"

namespace hydro {

namespace {

template <int STAGE, bool CFL> struct RowKernels {
    // [vectorised][scheme options other than the default]
    static constexpr void (*k[2][2])(StageArgs<float>) = {
        {row_stage_kernel<STAGE, CFL, false, false>, row_stage_kernel<STAGE, CFL, false, true>},
        {row_stage_kernel<STAGE, CFL, true, false>,
         row_stage_kernel<STAGE, CFL, true, true>}};
    static constexpr int warp_bytes = RowRing<STAGE>::bytes;
    static cudaError_t prepare() {
        cudaError_t e = cudaSuccess;
        for (int i = 0; i < 4 && e == cudaSuccess; ++i)
            e = cudaFuncSetAttribute(k[i >> 1][i & 1], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     warp_bytes * (kRowThreads / 32));
        return e;
    }
};

// Warps of a CTA: at most those of the tile (one per 64 cells), the count whose CTAs leave the
// fewest warps without a strip.
int row_warps(long long strips, int most) {
    int best = 1;
    long long waste = -1;
    for (int w = 1; w <= most; ++w) {
        const long long idle = (strips + w - 1) / w * w - strips;
        if (waste < 0 || idle <= waste) best = w, waste = idle;
    }
    return best;
}

// Rows a warp marches through by default: the least (m + 2) x (waves of the resident warps, plus
// half a wave of tail once there is more than one).  A chunk's prologue (four rows recovered, one
// extra face, the first copies' latency) costs about two rows.  Measured on GB300, us per step,
// shear layer, m = 2 / 4 / 8 / 12 / 16 / 24 / 32 / 48 / 64, the rule's choice marked; it is within
// 2.5 % of the best of each row:
//   512^2     16.9* 17.9  20.2  21.1  24.8  31.3  38.1  52.1  66.2
//   1024^2    42.1  34.0  33.6* 32.8  38.8  40.6  50.3  53.0  66.7
//   2048^2    185   130   106   100   101   97.5  98.2* 107   104
//   3001x2003 217   158   142   137   133   137   138   136*  136
//   4096^2    545   369   312   300   295   292*  297   291   302
int row_march(long long strips, long long ny, int warp_slots) {
    static const int kRows[] = {2, 4, 6, 8, 12, 16, 24, 32, 48, 64};
    int best = 0;
    double best_cost = 0.0;
    for (int m : kRows) {
        const double waves = (double)strips * (double)((ny + m - 1) / m) / (double)warp_slots;
        const double cost = (m + 2.0) * (waves < 1.0 ? 1.0 : waves + 0.5);
        if (best == 0 || cost < best_cost) best = m, best_cost = cost;
    }
    return best;
}

}  // namespace

cudaError_t stage_rows_f32(const StageLaunch &L, cudaStream_t st, bool prepare_only) {
    if (L.tile_x % 64 != 0 || L.tile_x > 64 * (kRowThreads / 32)) return cudaErrorInvalidValue;
    if (prepare_only) {
        static PerDevice attributes;
        return attributes.once([] {
            cudaError_t e = RowKernels<1, false>::prepare();
            if (e == cudaSuccess) e = RowKernels<2, false>::prepare();
            return e == cudaSuccess ? RowKernels<2, true>::prepare() : e;
        });
    }
    StageArgs<float> A = make_stage_args<float>(L);
    const long long strips = (A.n[0] + kStripCells - 1) / kStripCells;
    const int warps = row_warps(strips, L.tile_x / 64);
    if (L.rows > 0) A.march = L.rows;
    A.tiles_x = (int)((strips + warps - 1) / warps);
    const long long ctas = (long long)A.tiles_x * ((A.n[1] + A.march - 1) / A.march);
    if (ctas >= (1LL << 31)) return cudaErrorInvalidValue;
    const bool vec = rows_vec(L.uin, 4, A.n[0]) && rows_vec(L.ubase, 4, A.n[0]) &&
                     rows_vec(const_cast<const void *const *>(L.uout), 4, A.n[0]);
    const bool gen = A.order != 2 || A.riemann != 0;
    const auto k = L.stage == 1 ? RowKernels<1, false>::k[vec][gen]
                                : (L.split ? RowKernels<2, false>::k[vec][gen]
                                           : RowKernels<2, true>::k[vec][gen]);
    const size_t smem = (size_t)warps * (L.stage == 1 ? RowRing<1>::bytes : RowRing<2>::bytes);
    k<<<(unsigned)ctas, 32 * warps, smem, st>>>(A);
    return cudaGetLastError();
}

int default_strip_rows(long long nx, long long ny, int sm_count) {
    return row_march((nx + kStripCells - 1) / kStripCells, ny, (sm_count > 0 ? sm_count : 1) * 16);
}

}  // namespace hydro
