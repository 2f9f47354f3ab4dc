// FP32 RK-stage kernels of 2D grids: warps that march along y with everything in registers.
//
// A warp owns a strip of 64 columns, two neighbouring ones per lane in packed f32x2 pairs, and
// marches through a chunk of rows.  The x-neighbours' values come by warp shuffles, the
// y-neighbours' from the lane's own register pipeline, so nothing waits on another warp, each
// slope is computed once, and most of the arithmetic serves two cells per instruction.  The rows
// ahead come by asynchronous copies into a ring in shared memory (a load into registers ahead of
// its use does not stay ahead: under the register budget it is scheduled back to its use).  The
// outer two columns on each side are the strip's halo: 60 of 64 columns are stored (the warp
// repeats its neighbours' work on four columns instead of exchanging them).
//
// The step is bound by instruction issue, not by HBM or the FP32 pipe: the shared-memory row
// tiles this replaced executed 380-408 instructions per cell and stage (one cell per thread,
// in-plane slopes computed for both of their faces, the row's extra face and halo on separate
// lanes, a barrier per row).
#pragma once

#include "hydro_internal.h"
#include "pair_device.cuh"
#include "stage_kernel.cuh"

namespace hydro {

constexpr int kStripCells = 60;  // columns a warp stores
static_assert(kStripCells == kBatchStripCols, "the batch's work items are strips");

// One grid as the strip kernels see it.
struct RowGrid {
    const float *uin[4];
    const float *ubase[4];
    float *uout[4];
    int nx, ny;
    int px, py;          // periodic axes (else outflow)
    int order, riemann;  // scheme options (GEN)
    float cx, cy;        // AddFlux coefficients of the stage
    float inv_dr[2];
};

// Asynchronous copies (cp.async) of a lane's two cells into its place of a shared-memory slot.
__device__ __forceinline__ void copy_async8(uint32_t dst, const float *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async4(uint32_t dst, const float *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void copy_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ F2 load_shared(uint32_t a) {
    F2 v;
    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(v.r) : "r"(a) : "memory");
    return v;
}

// The rows a warp has in flight: a ring of slots of one row (four fields x 64 columns) of U_in,
// and in stage 2 another of U_base.  Every lane copies and reads its own cells only, so nothing
// waits on another lane.  In stage 1 U_base is U_in, and the ring keeps a row until it has been
// the base.
template <int STAGE> struct RowRing {
    static constexpr int ahead = 3;            // rows copied ahead of the pipeline's last one
    static constexpr int slot = 4 * 64 * 4;    // bytes of a row
    static constexpr int in_slots = 8;         // >= 4 rows of the prologue + ahead
    static constexpr int base_slots = STAGE == 1 ? 0 : 4;
    static constexpr int bytes = (in_slots + base_slots) * slot;  // per warp
    // rows j (the base) ... j + 2 + ahead live in the stage-1 ring at once
    static_assert(ahead + 3 <= in_slots && 4 + ahead <= in_slots, "the ring holds the live rows");
    static_assert(base_slots == 0 || ahead < base_slots, "the base ring holds the live rows");
};

// Rows [yb, ye) of the strip whose first lane holds columns xs, xs + 1 (xs even, >= -2); the
// lanes 1 ... 30 store theirs.  Whole warps only.  CFL: the signal maximum and the smallest
// density or pressure of the stored cells are folded into smax and vmin (NaN propagates).
// GEN: scheme options other than the default (MinBee, Davis speeds) are looked at.
// smem: the warp's RowRing in shared memory.
template <int STAGE, bool CFL, bool VEC, bool GEN>
__device__ __forceinline__ void row_strip(const RowGrid &A, const PairGas &G, int xs, int yb, int ye,
                                          uint32_t smem, float &smax, float &vmin) {
    using Ring = RowRing<STAGE>;
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int nx = A.nx, ny = A.ny, py = A.py;
    const int x = xs + 2 * lane;
    const bool mid = lane >= 1 && lane <= 30;
    const bool act0 = mid && x < nx, act1 = mid && x + 1 < nx;
    const bool order2 = !GEN || A.order == 2;
    const int riemann = GEN ? A.riemann : 0;
    // columns of the two cells after the boundary remap.  A 64-bit access takes an even pair:
    // periodic wraps move pairs as a whole (even nx); beyond an outflow end both cells copy
    // the end cell, which is the inner cell of the end pair.
    int o0, o1;
    bool dup_lo = false, dup_hi = false;
    if constexpr (VEC) {
        o0 = min(max(A.px ? (x < 0 ? x + nx : (x >= nx ? x - nx : x)) : x, 0), nx - 2);
        o1 = o0 + 1;
        dup_lo = !A.px && x < 0;
        dup_hi = !A.px && x >= nx;
    } else {
        o0 = remap(x, nx, A.px);
        o1 = remap(x + 1, nx, A.px);
    }
    const bool fix = VEC && __any_sync(kAll, dup_lo || dup_hi);
    const uint32_t mine = smem + 8u * lane;
    // ring position i: row yb - 2 + i
    auto fetch = [&](int i) {
        const int row = yb - 2 + i;
        const long long row0 = (long long)(row < yb ? remap(row, ny, py) : remap_ahead(row, ny, py)) * nx;
        const uint32_t d = mine + (uint32_t)(i & (Ring::in_slots - 1)) * Ring::slot;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float *p = A.uin[k] + row0;
            if constexpr (VEC) {
                copy_async8(d + 256u * k, p + o0);
            } else {
                copy_async4(d + 256u * k, p + o0);
                copy_async4(d + 256u * k + 4u, p + o1);
            }
        }
    };
    // U_base of row yb + i: only the storing lane reads a cell of it (stage 2 writes in place)
    auto fetch_base = [&](int i) {
        if constexpr (STAGE == 2) {
            const long long row0 = (long long)(yb + i) * nx;
            const uint32_t d = mine + Ring::in_slots * Ring::slot +
                               (uint32_t)(i & (Ring::base_slots - 1)) * Ring::slot;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float *p = A.ubase[k] + row0 + x;
                if constexpr (VEC) {
                    if (act0) copy_async8(d + 256u * k, p);
                } else {
                    if (act0) copy_async4(d + 256u * k, p);
                    if (act1) copy_async4(d + 256u * k + 4u, p + 1);
                }
            }
        }
    };
    auto take = [&](int i, F2 (&u)[4]) {
        const uint32_t d = mine + (uint32_t)(i & (Ring::in_slots - 1)) * Ring::slot;
#pragma unroll
        for (int k = 0; k < 4; ++k) u[k] = load_shared(d + 256u * k);
        if constexpr (VEC) {
            if (fix) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    float a, b;
                    f2_unpack(u[k], a, b);
                    u[k] = f2_pack(dup_hi ? b : a, dup_lo ? a : b);
                }
            }
        }
    };
    auto slopes = [&](const F2 (&a)[4], const F2 (&b)[4], F2 (&s)[4]) {
#pragma unroll
        for (int k = 0; k < 4; ++k) s[k] = order2 ? f2_minbee(a[k], b[k]) : f2_splat(0.0f);
    };
    const F2 half = f2_splat(0.5f), mhalf = f2_splat(-0.5f);
    // y-face between a row's upper face state H and the next row's lower face state W, the flux
    // in axis order
    auto y_flux = [&](const F2 (&H)[4], const F2 (&W)[4], F2 (&F)[4]) {
        const F2 vl[2] = {H[2], H[1]}, vr[2] = {W[2], W[1]};
        F2 N[4];
        hllc_pair<2>(H[0], vl, H[3], W[0], vr, W[3], G, N, riemann);
        F[0] = N[0], F[1] = N[2], F[2] = N[1], F[3] = N[3];
    };

    // Pipeline along y at row j: V of rows j and j + 1, their difference dy, the upper face
    // state Hy of row j and the flux Fm of its lower face; the rows after j + 1 in the ring.
    F2 Vc[4], Vn[4], dy[4], Hy[4], Fm[4];
    const int rows = ye - yb;
    {
#pragma unroll
        for (int i = 0; i < 4; ++i) fetch(i);
        copy_commit();
#pragma unroll
        for (int i = 0; i < Ring::ahead; ++i) {
            if (i < rows) {
                fetch(4 + i);
                fetch_base(i);
            }
            copy_commit();
        }
        copy_wait<Ring::ahead>();
        F2 u0[4], u1[4], u2[4], u3[4], s[4], W[4], H[4], V0[4], V1[4], d0[4], d1[4];
        take(0, u0);
        take(1, u1);
        take(2, u2);
        take(3, u3);
        prim_of_cons_pair<2>(u0, V0, G);
        prim_of_cons_pair<2>(u1, V1, G);
        prim_of_cons_pair<2>(u2, Vc, G);
        prim_of_cons_pair<2>(u3, Vn, G);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            d0[k] = f2_sub(V1[k], V0[k]);
            d1[k] = f2_sub(Vc[k], V1[k]);
            dy[k] = f2_sub(Vn[k], Vc[k]);
        }
        slopes(d0, d1, s);
#pragma unroll
        for (int k = 0; k < 4; ++k) H[k] = f2_fma(half, s[k], V1[k]);
        slopes(d1, dy, s);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            W[k] = f2_fma(mhalf, s[k], Vc[k]);
            Hy[k] = f2_fma(half, s[k], Vc[k]);
        }
        y_flux(H, W, Fm);
    }
    const F2 cx2 = f2_splat(A.cx), cy2 = f2_splat(A.cy);

#pragma unroll 2
    for (int i = 0; i < rows; ++i) {
        const long long row0 = (long long)(yb + i) * nx;
        if (i + Ring::ahead < rows) {
            fetch(4 + i + Ring::ahead);
            fetch_base(i + Ring::ahead);
        }
        copy_commit();
        copy_wait<Ring::ahead>();  // row yb + i + 2 and the base of row yb + i are here
        F2 Vnn[4];
        {
            F2 u[4];
            take(4 + i, u);
            prim_of_cons_pair<2>(u, Vnn, G);
        }

        // x: the face below each of the lane's cells, then the difference of each cell's faces
        F2 dFx[4];
        {
            F2 L[4], R[4], F[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float v0, v1;
                f2_unpack(Vc[k], v0, v1);
                const float dm = __fadd_rn(v0, -__shfl_up_sync(kAll, v1, 1));
                const float d = __fadd_rn(v1, -v0);
                const float dp = __shfl_down_sync(kAll, dm, 1);
                const float s0 = order2 ? minbee(dm, d) : 0.0f;
                const float s1 = order2 ? minbee(d, dp) : 0.0f;
                R[k] = f2_fma(mhalf, f2_pack(s0, s1), Vc[k]);
                L[k] = f2_pack(__shfl_up_sync(kAll, fmaf(0.5f, s1, v1), 1), fmaf(0.5f, s0, v0));
            }
            const F2 vl[2] = {L[1], L[2]}, vr[2] = {R[1], R[2]};
            hllc_pair<2>(L[0], vl, L[3], R[0], vr, R[3], G, F, riemann);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float f0, f1;
                f2_unpack(F[k], f0, f1);
                dFx[k] = f2_sub(F[k], f2_pack(f1, __shfl_down_sync(kAll, f0, 1)));
            }
        }
        // y: the face above row j
        F2 dn[4], Hn[4], Fp[4];
        {
            F2 s[4], W[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) dn[k] = f2_sub(Vnn[k], Vn[k]);
            slopes(dy, dn, s);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                W[k] = f2_fma(mhalf, s[k], Vn[k]);
                Hn[k] = f2_fma(half, s[k], Vn[k]);
            }
            y_flux(Hy, W, Fp);
        }
        // AddFlux, the axes in order (add_fluxes)
        const uint32_t bd = mine + (STAGE == 1
                                        ? (uint32_t)((i + 2) & (Ring::in_slots - 1)) * Ring::slot
                                        : Ring::in_slots * Ring::slot +
                                              (uint32_t)(i & (Ring::base_slots - 1)) * Ring::slot);
        F2 un[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const F2 sum = f2_fma(cy2, f2_sub(Fm[k], Fp[k]), f2_mul(cx2, dFx[k]));
            un[k] = f2_add(load_shared(bd + 256u * k), sum);
            float *p = A.uout[k] + row0;
            float a, b;
            f2_unpack(un[k], a, b);
            if constexpr (VEC) {
                if (act0) *reinterpret_cast<float2 *>(p + x) = make_float2(a, b);
            } else {
                if (act0) p[x] = a;
                if (act1) p[x + 1] = b;
            }
        }
        if constexpr (CFL) {
            float s[2], low[2];
            cfl_signal_pair<2>(un, G, A.inv_dr, s, low);
            if (act0) max_nan(smax, s[0]), min_nan(vmin, low[0]);
            if (act1) max_nan(smax, s[1]), min_nan(vmin, low[1]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            Vc[k] = Vn[k];
            Vn[k] = Vnn[k];
            dy[k] = dn[k];
            Hy[k] = Hn[k];
            Fm[k] = Fp[k];
        }
    }
}

// 64-bit accesses to a grid's rows: even nx and planes on 8-byte boundaries.
__host__ __device__ inline bool rows_vec(const void *const *planes, int nplanes, int nx) {
    bool ok = nx % 2 == 0;
    for (int k = 0; k < nplanes; ++k) ok &= reinterpret_cast<uintptr_t>(planes[k]) % 8 == 0;
    return ok;
}

constexpr int kRowThreads = 128;  // most threads of a CTA: four strips side by side

// One RK stage of a 2D grid.  CTA b of A.tiles_x CTAs per row chunk: its warps take
// neighbouring strips and the same A.march rows.
template <int STAGE, bool CFL, bool VEC, bool GEN>
__global__ void __launch_bounds__(kRowThreads, 4) row_stage_kernel(const StageArgs<float> A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ float sred[2 * kRowThreads / 32];
    Ctrl *ctrl = A.ctrl;
    if (!step_pending(ctrl)) return;  // uniform over the grid: no step to take
    RowGrid R;
#pragma unroll
    for (int k = 0; k < 4; ++k) R.uin[k] = A.uin[k], R.ubase[k] = A.ubase[k], R.uout[k] = A.uout[k];
    R.nx = A.n[0], R.ny = A.n[1];
    R.px = A.periodic[0], R.py = A.periodic[1];
    R.order = A.order, R.riemann = A.riemann;
    R.cx = step_coef<float>(ctrl, STAGE, 0);
    R.cy = step_coef<float>(ctrl, STAGE, 1);
    R.inv_dr[0] = A.inv_dr[0], R.inv_dr[1] = A.inv_dr[1];
    const int chunk = blockIdx.x / A.tiles_x;
    const int strip = (blockIdx.x - chunk * A.tiles_x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int yb = chunk * A.march;
    const int ye = min(yb + A.march, A.n[1]);
    float smax = 0.0f, vmin = 1.0f;
    if ((long long)strip * kStripCells < A.n[0])
        row_strip<STAGE, CFL, VEC, GEN>(R, pair_gas(A.gas), strip * kStripCells - 2, yb, ye,
                                        smem_u32(smem_raw) + (threadIdx.x >> 5) * RowRing<STAGE>::bytes,
                                        smax, vmin);
    if constexpr (CFL)
        reduce_signal_and_finalize<float, 0>(ctrl, smax, !(vmin > 0.0f), true, sred);
}

}  // namespace hydro
