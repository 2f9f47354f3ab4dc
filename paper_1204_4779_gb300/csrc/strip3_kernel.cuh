// FP32 RK-stage kernel of 3D grids: CTAs of seven warps of rows that march along z.
//
// A warp owns 64 columns of one row, two neighbouring ones per lane in packed f32x2 pairs (60 are
// stored, as in row_kernel.cuh; or 32 columns of two rows, 28 stored), and marches through a chunk
// of z-planes; a CTA is seven such warps one above the other and a helper warp.  The
// x-neighbours' values come by warp shuffles, the z-neighbours' from the lane's own pipeline, the
// y-neighbours' through shared memory: each row's V, then the upper face states, then the fluxes
// of the rows' lower faces, two barriers a plane.  Every slope and every face is computed once.
// The helper warp does what belongs to the rows outside the CTA's (V of the two rows on each
// side, their face states, the face above the last row), so that the rows' warps run the same
// straight code and none is late at a barrier.
// Rows of U ahead (own and base) come by cp.async.
#pragma once

#include "row_kernel.cuh"

namespace hydro {

constexpr int kStripWarps = 7;                         // warps of a CTA that own rows
constexpr int kStripThreads = 32 * (kStripWarps + 1);  // and the helper warp

// Shape of a CTA whose rows are SEG lanes wide: 32 (64 columns, a row per warp) or 16 (32
// columns, two rows per warp: the better fit of narrow grids).  Shared memory, in rows of
// five values of 2 SEG columns:
template <int SEG> struct Strip3 {
    static constexpr int RPW = 32 / SEG;              // rows of a warp
    static constexpr int NR = kStripWarps * RPW;      // rows of the CTA
    static constexpr int cells = 2 * SEG - 4;         // columns stored
    static constexpr int row = 5 * 8 * SEG;           // bytes of a row
    static constexpr int V = 0;                       // V of rows -1 ... NR of the plane
    static constexpr int H = V + NR + 2;              // upper y-face states of rows -1 ... NR - 1
    static constexpr int F = H + NR + 1;              // fluxes of the y-faces below rows 0 ... NR
    static constexpr int own = F + NR + 1;            // U ahead: two planes of the own rows
    static constexpr int base = own + 2 * NR;         // and of the base
    static constexpr size_t bytes = (size_t)(base + 2 * NR) * row;

    // one row, this lane's pair: two 16-byte groups and one 8-byte group
    __device__ static __forceinline__ void put(uint32_t r, int l, const F2 (&v)[5]) {
        const uint32_t a = r + 16u * l;
        asm volatile("st.shared.v2.b64 [%0], {%1, %2};" ::"r"(a), "l"(v[0].r), "l"(v[1].r) : "memory");
        asm volatile("st.shared.v2.b64 [%0], {%1, %2};" ::"r"(a + 16u * SEG), "l"(v[2].r), "l"(v[3].r) : "memory");
        asm volatile("st.shared.b64 [%0], %1;" ::"r"(r + 32u * SEG + 8u * l), "l"(v[4].r) : "memory");
    }
    __device__ static __forceinline__ void get(uint32_t r, int l, F2 (&v)[5]) {
        const uint32_t a = r + 16u * l;
        asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(v[0].r), "=l"(v[1].r) : "r"(a) : "memory");
        asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(v[2].r), "=l"(v[3].r) : "r"(a + 16u * SEG) : "memory");
        v[4] = load_shared(r + 32u * SEG + 8u * l);
    }
};

template <int SEG, int STAGE, bool CFL, bool VEC, bool GEN>
__global__ void __launch_bounds__(kStripThreads, 2) strip3_kernel(const StageArgs<float> A) {
    using S = Strip3<SEG>;
    constexpr int NR = S::NR, RPW = S::RPW;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ float sred[2 * kStripThreads / 32];
    Ctrl *ctrl = A.ctrl;
    if (!step_pending(ctrl)) return;  // uniform over the grid: no step to take
    constexpr unsigned kAll = 0xffffffffu;
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & (SEG - 1);    // lane of the row
    const int part = (threadIdx.x & 31) / SEG;   // which of the warp's rows
    // the helper warps of CTAs that run side by side sit on different schedulers
    const int helper = kStripWarps - (int)(blockIdx.x & 1);
    const int w = (warp - (warp > helper)) * RPW + part;  // row of the CTA
    const int nx = A.n[0], ny = A.n[1], nz = A.n[2];
    const int px = A.periodic[0], py = A.periodic[1], pz = A.periodic[2];
    const int ps = nx * ny;  // cells per plane
    const bool order2 = !GEN || A.order == 2;
    const int riemann = GEN ? A.riemann : 0;
    const int t = blockIdx.x / A.tiles_x, strip = blockIdx.x - t * A.tiles_x;
    const int chunk = t / A.tiles_y, y0 = (t - chunk * A.tiles_y) * NR;
    const int zb = (chunk + A.zchunk0) * A.march;
    const int n = min(A.march, nz - zb);  // planes of the chunk
    const int x = strip * S::cells - 2 + 2 * lane, y = y0 + w;
    // columns after the boundary remap (row_strip)
    int o0, o1;
    bool dup_lo = false, dup_hi = false;
    if constexpr (VEC) {
        o0 = min(max(px ? (x < 0 ? x + nx : (x >= nx ? x - nx : x)) : x, 0), nx - 2);
        o1 = o0 + 1;
        dup_lo = !px && x < 0;
        dup_hi = !px && x >= nx;
    } else {
        o0 = remap(x, nx, px);
        o1 = remap(x + 1, nx, px);
    }
    const bool fix = VEC && __any_sync(kAll, dup_lo || dup_hi);
    auto fix_ends = [&](F2 (&u)[5]) {
        if constexpr (VEC) {
            if (fix) {
#pragma unroll
                for (int k = 0; k < 5; ++k) {
                    float a, b;
                    f2_unpack(u[k], a, b);
                    u[k] = f2_pack(dup_hi ? b : a, dup_lo ? a : b);
                }
            }
        }
    };
    const uint32_t sm = smem_u32(smem_raw);
    auto row_at = [&](int r) { return sm + (uint32_t)(r * S::row); };
    // this lane's cells of the row at yo (in cells from its plane's start) of plane zr
    auto load = [&](int zr, int yo, F2 (&u)[5]) {
        const int i = zr * ps + yo;
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            const float *p = A.uin[k] + i;
            if constexpr (VEC) {
                const float2 v = __ldg(reinterpret_cast<const float2 *>(p + o0));
                u[k] = f2_pack(v.x, v.y);
            } else {
                u[k] = f2_pack(__ldg(p + o0), __ldg(p + o1));
            }
        }
        fix_ends(u);
    };
    const PairGas G = pair_gas(A.gas);
    const F2 half = f2_splat(0.5f), mhalf = f2_splat(-0.5f);
    // face states of a row from its neighbours: lower W, upper H
    auto faces = [&](const F2 (&lo)[5], const F2 (&c)[5], const F2 (&hi)[5], F2 (&W)[5], F2 (&H)[5]) {
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            const F2 s = order2 ? f2_minbee(f2_sub(c[k], lo[k]), f2_sub(hi[k], c[k])) : f2_splat(0.0f);
            W[k] = f2_fma(mhalf, s, c[k]);
            H[k] = f2_fma(half, s, c[k]);
        }
    };
    // flux of a y- or z-face between the face states H (below) and W (above), in axis order
    auto y_flux = [&](const F2 (&H)[5], const F2 (&W)[5], F2 (&F)[5]) {
        const F2 vl[3] = {H[2], H[1], H[3]}, vr[3] = {W[2], W[1], W[3]};
        F2 N[5];
        hllc_pair<3>(H[0], vl, H[4], W[0], vr, W[4], G, N, riemann);
        F[0] = N[0], F[1] = N[2], F[2] = N[1], F[3] = N[3], F[4] = N[4];
    };
    auto z_flux = [&](const F2 (&H)[5], const F2 (&W)[5], F2 (&F)[5]) {
        const F2 vl[3] = {H[3], H[1], H[2]}, vr[3] = {W[3], W[1], W[2]};
        F2 N[5];
        hllc_pair<3>(H[0], vl, H[4], W[0], vr, W[4], G, N, riemann);
        F[0] = N[0], F[1] = N[2], F[2] = N[3], F[3] = N[1], F[4] = N[4];
    };
    float smax = 0.0f, vmin = 1.0f;

    if (warp == helper) {
        // Per side (below the CTA's rows, above them) the outer and the inner halo row.  Rows of
        // half a warp: each half takes a side; whole-warp rows: both sides in turn.
        constexpr int SIDES = RPW == 2 ? 1 : 2;
        F2 vo[SIDES][5], vi[SIDES][5];
        bool top[SIDES];
        int yo[SIDES], yi[SIDES];
#pragma unroll
        for (int j = 0; j < SIDES; ++j) {
            top[j] = RPW == 2 ? part == 1 : j == 1;
            yo[j] = remap(top[j] ? y0 + NR + 1 : y0 - 2, ny, py) * nx;
            yi[j] = remap(top[j] ? y0 + NR : y0 - 1, ny, py) * nx;
        }
        auto load_all = [&](int zr) {
#pragma unroll
            for (int j = 0; j < SIDES; ++j) {
                load(zr, yo[j], vo[j]);
                load(zr, yi[j], vi[j]);
            }
        };
        auto stage = [&] {
#pragma unroll
            for (int j = 0; j < SIDES; ++j) {
                F2 v[5];
                prim_of_cons_pair<3>(vo[j], v, G);
#pragma unroll
                for (int k = 0; k < 5; ++k) vo[j][k] = v[k];
                prim_of_cons_pair<3>(vi[j], v, G);
                S::put(row_at(S::V + (top[j] ? NR + 1 : 0)), lane, v);
#pragma unroll
                for (int k = 0; k < 5; ++k) vi[j][k] = v[k];
            }
        };
        load_all(zb);
        stage();
        __syncthreads();
        for (int i = 0; i < n; ++i) {
            F2 W[5];  // lower face state of the row above the CTA's
#pragma unroll
            for (int j = 0; j < SIDES; ++j) {
                F2 e[5], lo[5], hi[5], X[5], H[5];
                S::get(row_at(S::V + (top[j] ? NR : 1)), lane, e);
#pragma unroll
                for (int k = 0; k < 5; ++k) {
                    lo[k].r = top[j] ? e[k].r : vo[j][k].r;
                    hi[k].r = top[j] ? vo[j][k].r : e[k].r;
                }
                faces(lo, vi[j], hi, X, H);
                if (!top[j]) S::put(row_at(S::H), lane, H);
                if (j == SIDES - 1) {
#pragma unroll
                    for (int k = 0; k < 5; ++k) W[k] = X[k];
                }
            }
            load_all(remap_ahead(zb + i + 1, nz, pz));
            __syncthreads();
            F2 e[5], X[5];
            S::get(row_at(S::H + NR), lane, e);
            y_flux(e, W, X);
            if (top[SIDES - 1]) S::put(row_at(S::F + NR), lane, X);
            stage();
            __syncthreads();
        }
    } else {
        const bool mid = lane >= 1 && lane <= SEG - 2 && y < ny;
        const bool act0 = mid && x < nx, act1 = mid && x + 1 < nx;
        const int own_y = remap(y, ny, py) * nx;
        // the copies of step i of the march: U of plane zb + i + 2 and the base of plane zb + i
        auto fetch = [&](int i) {
            const int s = i & 1, z = zb + i;
            const int at = remap_ahead(z + 2, nz, pz) * ps + own_y;
            const uint32_t d = row_at(S::own + s * NR + w) + 8u * lane;
            const uint32_t e = row_at(S::base + s * NR + w) + 8u * lane;
            const int bt = z * ps + y * nx + x;
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                const float *p = A.uin[k] + at;
                const float *q = A.ubase[k] + bt;
                if constexpr (VEC) {
                    copy_async8(d + 8u * SEG * k, p + o0);
                    if (act0) copy_async8(e + 8u * SEG * k, q);
                } else {
                    copy_async4(d + 8u * SEG * k, p + o0);
                    copy_async4(d + 8u * SEG * k + 4u, p + o1);
                    if (act0) copy_async4(e + 8u * SEG * k, q);
                    if (act1) copy_async4(e + 8u * SEG * k + 4u, q + 1);
                }
            }
        };
        // Pipeline along z at plane z: V of planes z and z + 1, the upper z-face state Hz of
        // plane z, the flux Fm of its lower z-face.
        F2 Vc[5], Vn[5], Hz[5], Fm[5];
        fetch(0);
        copy_commit();
        {
            F2 u[5], V0[5], V1[5], W[5], H[5];
            load(remap(zb - 2, nz, pz), own_y, u);
            prim_of_cons_pair<3>(u, V0, G);
            load(remap(zb - 1, nz, pz), own_y, u);
            prim_of_cons_pair<3>(u, V1, G);
            load(zb, own_y, u);
            prim_of_cons_pair<3>(u, Vc, G);
            load(remap_ahead(zb + 1, nz, pz), own_y, u);
            prim_of_cons_pair<3>(u, Vn, G);
            S::put(row_at(S::V + w + 1), lane, Vc);
            faces(V0, V1, Vc, W, H);
            faces(V1, Vc, Vn, W, Hz);
            z_flux(H, W, Fm);
        }
        const float cx = step_coef<float>(ctrl, STAGE, 0), cy = step_coef<float>(ctrl, STAGE, 1),
                    cz = step_coef<float>(ctrl, STAGE, 2);
        __syncthreads();

        for (int i = 0; i < n; ++i) {
            // y: the face states of this row; the upper one to the row above
            F2 Wy[5];
            {
                F2 dn[5], up[5], H[5];
                S::get(row_at(S::V + w), lane, dn);
                S::get(row_at(S::V + w + 2), lane, up);
                faces(dn, Vc, up, Wy, H);
                S::put(row_at(S::H + w + 1), lane, H);
            }
            // x: the face below each of the lane's cells, then the difference of each cell's faces
            F2 dFx[5];
            {
                F2 L[5], R[5], F[5];
#pragma unroll
                for (int k = 0; k < 5; ++k) {
                    float v0, v1;
                    f2_unpack(Vc[k], v0, v1);
                    const float dm = __fadd_rn(v0, -__shfl_up_sync(kAll, v1, 1, SEG));
                    const float d = __fadd_rn(v1, -v0);
                    const float dp = __shfl_down_sync(kAll, dm, 1, SEG);
                    const float s0 = order2 ? minbee(dm, d) : 0.0f;
                    const float s1 = order2 ? minbee(d, dp) : 0.0f;
                    R[k] = f2_fma(mhalf, f2_pack(s0, s1), Vc[k]);
                    L[k] = f2_pack(__shfl_up_sync(kAll, fmaf(0.5f, s1, v1), 1, SEG), fmaf(0.5f, s0, v0));
                }
                const F2 vl[3] = {L[1], L[2], L[3]}, vr[3] = {R[1], R[2], R[3]};
                hllc_pair<3>(L[0], vl, L[4], R[0], vr, R[4], G, F, riemann);
#pragma unroll
                for (int k = 0; k < 5; ++k) {
                    float f0, f1;
                    f2_unpack(F[k], f0, f1);
                    dFx[k] = f2_sub(F[k], f2_pack(f1, __shfl_down_sync(kAll, f0, 1, SEG)));
                }
            }
            if (i + 1 < n) fetch(i + 1);
            copy_commit();
            copy_wait<1>();
            __syncthreads();  // the face states of every row are there; V of the plane is free
            // y: the face below this row
            F2 Fy[5];
            {
                F2 H[5];
                S::get(row_at(S::H + w), lane, H);
                y_flux(H, Wy, Fy);
                S::put(row_at(S::F + w), lane, Fy);
            }
            // z: the face above this plane
            F2 Vnn[5], dFz[5], Hn[5];
            {
                F2 u[5], W[5], F[5];
                const uint32_t d = row_at(S::own + (i & 1) * NR + w) + 8u * lane;
#pragma unroll
                for (int k = 0; k < 5; ++k) u[k] = load_shared(d + 8u * SEG * k);
                fix_ends(u);
                prim_of_cons_pair<3>(u, Vnn, G);
                S::put(row_at(S::V + w + 1), lane, Vn);
                faces(Vc, Vn, Vnn, W, Hn);
                z_flux(Hz, W, F);
#pragma unroll
                for (int k = 0; k < 5; ++k) {
                    dFz[k] = f2_sub(Fm[k], F[k]);
                    Fm[k] = F[k];
                }
            }
            __syncthreads();  // the y-fluxes and the next plane's V are there
            // AddFlux, the axes in order (add_fluxes)
            F2 un[5];
            {
                F2 up[5];
                S::get(row_at(S::F + w + 1), lane, up);
                const F2 cx2 = f2_splat(cx), cy2 = f2_splat(cy), cz2 = f2_splat(cz);
                const uint32_t bd = row_at(S::base + (i & 1) * NR + w) + 8u * lane;
                const int at = (zb + i) * ps + y * nx + x;
#pragma unroll
                for (int k = 0; k < 5; ++k) {
                    F2 sum = f2_mul(cx2, dFx[k]);
                    sum = f2_fma(cy2, f2_sub(Fy[k], up[k]), sum);
                    sum = f2_fma(cz2, dFz[k], sum);
                    un[k] = f2_add(load_shared(bd + 8u * SEG * k), sum);
                    float *p = A.uout[k] + at;
                    float a, b;
                    f2_unpack(un[k], a, b);
                    if constexpr (VEC) {
                        if (act0) *reinterpret_cast<float2 *>(p) = make_float2(a, b);
                    } else {
                        if (act0) p[0] = a;
                        if (act1) p[1] = b;
                    }
                }
            }
            if constexpr (CFL) {
                float s[2], low[2];
                cfl_signal_pair<3>(un, G, A.inv_dr, s, low);
                if (act0) max_nan(smax, s[0]), min_nan(vmin, low[0]);
                if (act1) max_nan(smax, s[1]), min_nan(vmin, low[1]);
            }
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                Vc[k] = Vn[k];
                Vn[k] = Vnn[k];
                Hz[k] = Hn[k];
            }
        }
    }
    if constexpr (CFL)
        reduce_signal_and_finalize<float, kStripThreads>(ctrl, smax, !(vmin > 0.0f), true, sred);
}

}  // namespace hydro
