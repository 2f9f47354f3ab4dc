// FP64 RK-stage kernel of 2D grids: warps that march along y with everything in registers.
//
// A warp owns 32 columns, one per lane, of which 28 are stored (the outer two on each side are the
// strip's halo), and marches through a chunk of rows: x-neighbours by shuffles, y-neighbours from
// the lane's own pipeline, every slope, state and face once, no shared memory and no barrier.
//
// Bound by the FP64 pipe, which one warp per scheduler fills: what counts is the number of FP64
// operations a warp issues per stored cell and that every scheduler has a warp to issue them.  The
// 32 x 8 tiles issue about 317 a warp and stage and leave the pipe idle for a quarter of the time
// (one CTA of eight warps an SM; two of them evaluate the tile's 40 extra faces while the others
// wait at the barrier); a strip issues 261 for 28 / 32 of a warp's cells, and the warps wait for
// nothing.  The values are those of the tiles, bit for bit.
#pragma once

#include "stage_kernel.cuh"

namespace hydro {

constexpr int kStrip64Cells = 28;    // columns a warp stores
constexpr int kRow64Threads = 128;   // four strips side by side

template <int STAGE, bool CFL>
__global__ void __launch_bounds__(kRow64Threads, 2) row64_stage_kernel(const StageArgs<double> A) {
    constexpr int NV = 4;
    constexpr unsigned kAll = 0xffffffffu;
    __shared__ double sred[kRow64Threads / 32];
    Ctrl *ctrl = A.ctrl;
    if (!step_pending(ctrl)) return;  // uniform over the grid: no step to take
    const Gas<double> G = A.gas;
    const Fma64 &X = G.x;
    const double cx = step_coef<double>(ctrl, STAGE, 0), cy = step_coef<double>(ctrl, STAGE, 1);
    const int nx = A.n[0], ny = A.n[1], py = A.periodic[1];
    // the CTA's warps (one per scheduler) take consecutive (chunk, strip) items
    const int item = blockIdx.x * (kRow64Threads / 32) + (threadIdx.x >> 5);
    const int chunk = item / A.tiles_x, strip = item - chunk * A.tiles_x;
    const int lane = threadIdx.x & 31;
    const int yb = chunk * A.march, ye = min(yb + A.march, ny);
    const bool order2 = A.order == 2;
    double smax = 0.0;
    bool bad = false;
    if (item < A.items) {  // (the same for the whole warp)
        const int x = strip * kStrip64Cells - 2 + lane;
        const bool active = lane >= 2 && lane < 2 + kStrip64Cells && x < nx;
        const int o = remap(x, nx, A.periodic[0]);
        auto load = [&](int row, double (&v)[NV]) {
            const long long i = (long long)row * nx + o;
            double u[NV];
#pragma unroll
            for (int k = 0; k < NV; ++k) u[k] = __ldg(A.uin[k] + i);
            prim_of_cons<double, 2>(u, v, G);
        };
        // y-face between a row's upper face state and the next row's lower one, in axis order
        auto y_flux = [&](const double (&H)[NV], const double (&W)[NV], double (&F)[NV]) {
            const double vl[2] = {H[2], H[1]}, vr[2] = {W[2], W[1]};
            double N[NV];
            hllc<2, true>(H[0], vl, H[3], W[0], vr, W[3], G, N, A.riemann);
            F[0] = N[0], F[1] = N[2], F[2] = N[1], F[3] = N[3];
        };
        auto slope = [&](double a, double b) { return order2 ? minbee(a, b) : 0.0; };
        double Vc[NV], Vn[NV], dy[NV], Hy[NV], Fm[NV];
        {
            double V0[NV], V1[NV], H[NV], W[NV];
            load(remap(yb - 2, ny, py), V0);
            load(remap(yb - 1, ny, py), V1);
            load(yb, Vc);
            load(remap_ahead(yb + 1, ny, py), Vn);
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                const double d0 = X.sub(V1[k], V0[k]), d1 = X.sub(Vc[k], V1[k]);
                dy[k] = X.sub(Vn[k], Vc[k]);
                H[k] = fma(0.5, slope(d0, d1), V1[k]);
                const double s = slope(d1, dy[k]);
                W[k] = fma(-0.5, s, Vc[k]);
                Hy[k] = fma(0.5, s, Vc[k]);
            }
            y_flux(H, W, Fm);
        }
#pragma unroll 1
        for (int j = yb; j < ye; ++j) {
            double Vnn[NV], F[NV], Fh[NV], Fp[NV], Hn[NV];
            load(remap_ahead(j + 2, ny, py), Vnn);
            {  // x: the face below each lane's cell; the one above is the next lane's
                double L[NV], R[NV];
#pragma unroll
                for (int k = 0; k < NV; ++k) {
                    const double d = X.sub(Vc[k], __shfl_up_sync(kAll, Vc[k], 1));
                    const double s = slope(d, __shfl_down_sync(kAll, d, 1));
                    R[k] = fma(-0.5, s, Vc[k]);
                    L[k] = __shfl_up_sync(kAll, fma(0.5, s, Vc[k]), 1);
                }
                const double vl[2] = {L[1], L[2]}, vr[2] = {R[1], R[2]};
                hllc<2, false>(L[0], vl, L[3], R[0], vr, R[3], G, F, A.riemann);
                __syncwarp();
#pragma unroll
                for (int k = 0; k < NV; ++k) Fh[k] = __shfl_down_sync(kAll, F[k], 1);
            }
            {
                double W[NV];
#pragma unroll
                for (int k = 0; k < NV; ++k) {
                    const double dn = X.sub(Vnn[k], Vn[k]);
                    const double s = slope(dy[k], dn);
                    W[k] = fma(-0.5, s, Vn[k]);
                    Hn[k] = fma(0.5, s, Vn[k]);
                    dy[k] = dn;
                }
                y_flux(Hy, W, Fp);
            }
            const long long i = (long long)j * nx + x;
            if (active) {
                double base[NV], un[NV];
#pragma unroll
                for (int k = 0; k < NV; ++k) base[k] = A.ubase[k][i];
                add_fluxes<double, NV, true, false>(base, cx, F, Fh, cy, Fm, Fp, 0.0, F, F, un, X);
#pragma unroll
                for (int k = 0; k < NV; ++k) A.uout[k][i] = un[k];
                if constexpr (CFL) cfl_signal<double, 2>(un, A, smax, bad);
            }
            __syncwarp();
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                Vc[k] = Vn[k];
                Vn[k] = Vnn[k];
                Hy[k] = Hn[k];
                Fm[k] = Fp[k];
            }
        }
    }
    if constexpr (CFL) reduce_signal_and_finalize<double, kRow64Threads>(ctrl, smax, bad, true, sred);
}

}  // namespace hydro
