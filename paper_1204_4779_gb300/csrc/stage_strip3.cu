// Launches of the FP32 3D strip kernels (strip3_kernel.cuh).
#include <math.h>

#include "hydro_internal.h"
#include "stage_launch.cuh"
#include "strip3_kernel.cuh"

namespace hydro {

namespace {

template <int SEG, int STAGE, bool CFL> struct Strip3Kernels {
    // [vectorised][scheme options other than the default]
    static constexpr void (*k[2][2])(StageArgs<float>) = {
        {strip3_kernel<SEG, STAGE, CFL, false, false>, strip3_kernel<SEG, STAGE, CFL, false, true>},
        {strip3_kernel<SEG, STAGE, CFL, true, false>, strip3_kernel<SEG, STAGE, CFL, true, true>}};
    static cudaError_t prepare() {
        cudaError_t e = cudaSuccess;
        for (int i = 0; i < 4 && e == cudaSuccess; ++i)
            e = cudaFuncSetAttribute(k[i >> 1][i & 1], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)Strip3<SEG>::bytes);
        return e;
    }
};

template <int SEG> long long strip3_tiles_x(long long nx) {
    return (nx + Strip3<SEG>::cells - 1) / Strip3<SEG>::cells;
}
template <int SEG> long long strip3_tiles_y(long long ny) {
    return (ny + Strip3<SEG>::NR - 1) / Strip3<SEG>::NR;
}
// Rows of 32 lanes unless the grid leaves more columns and rows of theirs unused than of the
// 16-lane ones: a CTA of either covers 448 cells of a plane.
bool strip3_half_rows(long long nx, long long ny) {
    return strip3_tiles_x<16>(nx) * strip3_tiles_y<16>(ny) < strip3_tiles_x<32>(nx) * strip3_tiles_y<32>(ny);
}

double strip3_tiles(long long nx, long long ny) {
    return strip3_half_rows(nx, ny) ? (double)(strip3_tiles_x<16>(nx) * strip3_tiles_y<16>(ny))
                                    : (double)(strip3_tiles_x<32>(nx) * strip3_tiles_y<32>(ny));
}

// Modelled time, in planes, of a launch whose CTAs march through m planes (the comment at
// default_strip_planes).
double strip3_cost(long long nx, long long ny, long long nz, int m, int sm_count) {
    const double slots = 2.0 * (sm_count > 0 ? sm_count : 1);
    const double chunks = (double)((nz + m - 1) / m);
    double waves = strip3_tiles(nx, ny) * chunks / slots;
    if (waves >= 6.0)  // by work: the last chunk may be short
        waves = strip3_tiles(nx, ny) * ((double)nz + 1.5 * chunks) / ((m + 1.5) * slots);
    const double whole = floor(waves), rest = waves - whole;
    return (m + 1.5) * (whole + (rest > 0.5 || whole == 0.0 ? 1.0 : (rest > 0.0 ? 0.62 : 0.0)));
}

template <int SEG> cudaError_t launch_strip3(const StageLaunch &L, StageArgs<float> &A, cudaStream_t st) {
    A.tiles_x = (int)strip3_tiles_x<SEG>(A.n[0]);
    A.tiles_y = (int)strip3_tiles_y<SEG>(A.n[1]);
    const int chunks = L.zchunks > 0 ? L.zchunks : (A.n[2] + A.march - 1) / A.march - L.zchunk0;
    const long long ctas = (long long)A.tiles_x * A.tiles_y * chunks;
    if (ctas < 1 || ctas >= (1LL << 31)) return cudaErrorInvalidValue;
    const bool vec = rows_vec(L.uin, 5, A.n[0]) && rows_vec(L.ubase, 5, A.n[0]) &&
                     rows_vec(const_cast<const void *const *>(L.uout), 5, A.n[0]);
    const bool gen = A.order != 2 || A.riemann != 0;
    const auto k = L.stage == 1 ? Strip3Kernels<SEG, 1, false>::k[vec][gen]
                                : (L.split ? Strip3Kernels<SEG, 2, false>::k[vec][gen]
                                           : Strip3Kernels<SEG, 2, true>::k[vec][gen]);
    k<<<(unsigned)ctas, kStripThreads, Strip3<SEG>::bytes, st>>>(A);
    return cudaGetLastError();
}

}  // namespace

cudaError_t stage_strip3_f32(const StageLaunch &L, cudaStream_t st, bool prepare_only) {
    if (prepare_only) {
        static PerDevice attributes;
        return attributes.once([] {
            cudaError_t e = Strip3Kernels<32, 1, false>::prepare();
            if (e == cudaSuccess) e = Strip3Kernels<32, 2, false>::prepare();
            if (e == cudaSuccess) e = Strip3Kernels<32, 2, true>::prepare();
            if (e == cudaSuccess) e = Strip3Kernels<16, 1, false>::prepare();
            if (e == cudaSuccess) e = Strip3Kernels<16, 2, false>::prepare();
            return e == cudaSuccess ? Strip3Kernels<16, 2, true>::prepare() : e;
        });
    }
    StageArgs<float> A = make_stage_args<float>(L);
    return strip3_half_rows(A.n[0], A.n[1]) ? launch_strip3<16>(L, A, st)
                                            : launch_strip3<32>(L, A, st);
}

// Planes a CTA marches through by default: the least (m + 1.5) x waves, a chunk's prologue counted
// as 1.5 planes, the last wave of the resident CTAs (two per SM) whole, or 0.62 where no SM gets a
// second CTA of it.  Measured on GB300, blast, us per step at m planes, the rule's choice marked;
// it is within 3 % of the best of each row:
//   64^3    1: 35.9  2: 31.0  4: 28.6*  6: 31.5  8: 30.3  16: 48.7
//   128^3   8: 114  12: 110  16: 112  22: 100*  24: 108  32: 139
//   192^3  16: 279  24: 303  32: 274  48: 310  64: 271*  96: 396
//   256^3  16: 669  24: 665  26: 671*  32: 653  52: 711  64: 654  86: 689
//   512^3  32: 4520  64: 4498  74: 4441  86: 4497  96: 4411  128: 4500*  171: 4644
int default_strip_planes(long long nx, long long ny, long long nz, int sm_count) {
    static const int kPlanes[] = {2, 4, 6, 8, 12, 16, 20, 24, 32, 40, 48, 64, 80, 96, 128};
    int best = 0;
    double best_cost = 0.0;
    for (int named : kPlanes) {
        const int m = fitted_strip_planes(nx, ny, nz, named, sm_count);
        const double cost = strip3_cost(nx, ny, nz, m, sm_count);
        if (best == 0 || cost < best_cost) best = m, best_cost = cost;
    }
    return best;
}

// Planes of a CTA for a march of m: over many waves of CTAs m itself (a short last chunk shortens
// the tail).  Where the chunks make few waves, the waves' rounding and the longest chunk set the
// time, so the march is an upper bound: of the numbers of chunks that take between m / 2 and m
// planes each, evenly, the one of least cost (160^3 at 64: three chunks of 54, 54 and 52 planes
// instead of 64, 64 and 32; at 32: seven of 23 instead of five, which made 1.13 waves).
int fitted_strip_planes(long long nx, long long ny, long long nz, int m, int sm_count) {
    const double slots = 2.0 * (sm_count > 0 ? sm_count : 1);
    const long long least = (nz + m - 1) / m;
    if (strip3_tiles(nx, ny) * (double)least >= 6.0 * slots) return m;
    int best = 0;
    double best_cost = 0.0;
    for (long long chunks = least; chunks <= 2 * least; ++chunks) {
        const int k = (int)((nz + chunks - 1) / chunks);
        const double cost = strip3_cost(nx, ny, nz, k, sm_count);
        if (best == 0 || cost < best_cost) best = k, best_cost = cost;
    }
    return best;
}

// Whether the 16 x 8 tile kernel (no look-ahead, m_tiles planes a CTA) is the faster one of a grid
// whose strips would march m_strips planes: grids so narrow that less than two thirds of a strip
// CTA's 448 lanes own a cell, and large enough to fill the GPU with tiles.  A tile launch of
// w waves (six CTAs an SM) takes (m + 1) x w, or (0.4 + 0.6 w) where w < 1, in units of 1.2 planes
// of the strips' strip3_cost; both models fitted to 113 grids, the choice at worst 7 % from the
// better one.  Measured on GB300, us per step, tiles of the earlier version / strips / tiles now:
//   29x200x200    88.0  101.5   80.5*     61x200x200   147   156   140*
//   32x200x200    87.4   92.7   78.8*     64x200x200   148   143*  143
//   33x200x200   116    100.8* 109.8      16x200x200   57.7  54.4  49.7*
//   4x384x384    133    204    120*       16x64x48     34.0  17.6* 31.8
bool strip3_narrow(long long nx, long long ny, long long nz, int m_strips, int m_tiles, int sm_count) {
    if ((double)nx * (double)ny >= 0.66 * 448.0 * strip3_tiles(nx, ny)) return false;
    const long long ctas = ((nx + 15) / 16) * ((ny + 7) / 8) * ((nz + m_tiles - 1) / m_tiles);
    const double waves = (double)ctas / (6.0 * (sm_count > 0 ? sm_count : 1));
    if (waves < 0.3) return false;
    const double planes = (double)(m_tiles < nz ? m_tiles : nz) + 1.0;
    return 1.2 * planes * (waves < 1.0 ? 0.4 + 0.6 * waves : waves) <
           strip3_cost(nx, ny, nz, m_strips, sm_count);
}

}  // namespace hydro
