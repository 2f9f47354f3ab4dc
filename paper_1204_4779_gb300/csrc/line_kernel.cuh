// Whole runs of small 1D grids in one launch of one thread-block cluster.
//
// A 1D grid of a thousand cells fills a few SMs, and a step through the grid kernels is three
// launches (two RK stages, the CFL pass), each reading back what the last one wrote: 48 us a step
// at 1024 cells in FP64, of which the arithmetic's own latency is a fifth.  Here every CTA of a
// cluster keeps its cells in registers, one per thread, and up to `n_steps` steps run without
// leaving the kernel: per RK stage the CTAs exchange the primitive states of their two end cells
// through distributed shared memory behind one cluster barrier, each face is evaluated once, and
// the CFL maximum of the new states travels with the next stage's exchange.  Every CTA derives the
// same dt from it.  The operations are those of the grid kernels (inplane_face, add_fluxes,
// prim_of_cons, the CFL pass, finalize_dt), so the states are the same bit for bit.
//
// Bound by latency: about 280 FP64 operations in a row per step, 64 cycles each.  A scheduler
// takes one warp's FP64 operations at full rate, so up to four warps an SM cost nothing.  Measured,
// us per step: FP64 1024 cells 14.0, 2048 16.0, FP32 2.5 and 2.6; the grid kernels at 2049 and 8192
// cells take 33.7 and 35.0, FP32 11.2 and 11.4.  The line to them is not where the two meet: a
// cluster of 16 CTAs of kLinePer threads would hold 4096 cells, but above 2048 a scheduler holds
// more than one warp, and that has not been measured.
#pragma once

#include <atomic>

#include "stage_kernel.cuh"

namespace hydro {

template <class T> struct LineArgs {
    T *u[3];
    int n, per;  // cells of the grid and of a CTA
    int periodic, order, riemann, n_steps;
    double dr, inv_dr;
    T inv_dr_t;
    Gas<T> gas;
    Fma64 x;
    Ctrl *ctrl;
};

constexpr int kLinePer = 256;               // most cells of a CTA
constexpr int kLineThreads = kLinePer + 32; // (the warp after the last cell evaluates its high face)
constexpr int kLineMaxCtas = 16;

__device__ __forceinline__ void line_cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t line_map(const void *p, unsigned rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(r)
                 : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ void line_store(uint32_t a, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void line_store(uint32_t a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}

// a / b, correctly rounded, with y = 1 / b where b is in range (any y otherwise)
__device__ __forceinline__ double line_div(double a, double b, double y, const Fma64 &X) {
    return in_range(a) && in_range(b) ? X.div(a, b, y) : div_plain(a, b);
}

template <class T>
__global__ void __launch_bounds__(kLineThreads) line_kernel(const LineArgs<T> A) {
    constexpr int NV = 3, PL = (kLinePer + 4 + 3) / 4 * 4, NF = (kLinePer + 1 + 3) / 4 * 4;
    __shared__ T sV[2][NV * PL];      // V of the CTA's cells, two halo cells on each side
    __shared__ T sF[NV * NF];
    __shared__ T sMax[2][kLineMaxCtas];  // the CTAs' CFL maxima (NaN: a bad cell)
    __shared__ T sWarp[kLineThreads / 32];
    __shared__ double sStep[6];       // t, dt, coefficients of the two stages, dt_last
    __shared__ int sInfo[3];          // clipped, steps, status
    const int C = gridDim.x, rank = blockIdx.x, tid = threadIdx.x;
    const int c0 = rank * A.per, mine = min(A.per, A.n - c0);
    const int left = rank == 0 ? C - 1 : rank - 1, right = rank == C - 1 ? 0 : rank + 1;
    const int left_mine = min(A.per, A.n - left * A.per);
    const bool cell = tid < mine, face = tid <= mine;
    const Gas<T> G = A.gas;
    Ctrl *c = A.ctrl;

    // V of this thread's cell into the CTA's plane and the halo of the neighbours (or, at an
    // outflow end, its own)
    auto stage = [&](T *plane, const T (&v)[NV]) {
        if (!cell) return;
        Cells<T, NV>::put(plane, PL, tid + 2, v);
        auto send = [&](int r, int at) {
#pragma unroll
            for (int k = 0; k < NV; ++k) line_store(line_map(plane + k * PL + at, r), v[k]);
        };
        if (tid < 2 && (rank > 0 || A.periodic)) send(left, left_mine + 2 + tid);
        if (tid >= mine - 2 && (rank < C - 1 || A.periodic)) send(right, tid - (mine - 2));
        if (!A.periodic && rank == 0 && tid == 0) {
            Cells<T, NV>::put(plane, PL, 0, v);
            Cells<T, NV>::put(plane, PL, 1, v);
        }
        if (!A.periodic && rank == C - 1 && tid == mine - 1) {
            Cells<T, NV>::put(plane, PL, mine + 2, v);
            Cells<T, NV>::put(plane, PL, mine + 3, v);
        }
    };
    // faces from the plane, then u = base + coef (F_low - F_high)
    auto advance = [&](const T *plane, const T (&base)[NV], T coef, T (&u)[NV]) {
        if (face) inplane_face<T, 1, PL, NF>(plane, sF, tid, 1, 0, tid, G, A.order, A.riemann);
        __syncthreads();
        if (cell) {
            T fw[NV], fe[NV];
            Cells<T, NV>::get(sF, NF, tid, fw);
            Cells<T, NV>::get(sF, NF, tid + 1, fe);
            add_fluxes<T, NV, false, false>(base, coef, fw, fe, T(0), fw, fw, T(0), fw, fw, u, G.x);
        }
    };

    T u0[NV], u1[NV], v[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) u0[k] = cell ? A.u[k][c0 + tid] : T(1);
    prim_of_cons<T, 1>(u0, v, G);
    if (tid == 0) {
        sStep[0] = c->t;
        sStep[1] = c->dt;
        sStep[2] = c->coef[0][0];
        sStep[3] = c->coef[1][0];
        sStep[4] = c->dt_last;
        sInfo[0] = c->clipped;
        sInfo[1] = c->steps;
        sInfo[2] = (int)c->status;
    }
    const double t_end = c->t_end, cfl = c->cfl;
    line_cluster_sync();  // every CTA runs before any writes to its shared memory
    stage(sV[0], v);
    line_cluster_sync();

    int s = 0;
    for (; s < A.n_steps && sStep[1] > 0.0; ++s) {
        advance(sV[0], u0, T(sStep[2]), u1);
        if (cell) prim_of_cons<T, 1>(u1, v, G);
        stage(sV[1], v);
        line_cluster_sync();
        advance(sV[1], u0, T(sStep[3]), u1);
        // new state, its V for the next step's exchange, and its CFL signal (the CFL pass)
        T sig = T(0);
        if (cell) {
#pragma unroll
            for (int k = 0; k < NV; ++k) u0[k] = u1[k];
            prim_of_cons<T, 1>(u0, v, G);
            if constexpr (Arith<T>::exact) {
                sig = exact_signal<1>(v, G, &A.dr, &A.inv_dr);
            } else {
                const T cs = Arith<float>::sqrt_(G.g * v[2] * Arith<float>::rcp(v[0]));
                sig = (fabsf(v[1]) + cs) * A.inv_dr_t;
            }
            if (!(v[0] > T(0)) || !(v[2] > T(0))) sig = T(NAN);
        }
        stage(sV[0], v);
        // maxima on the bit patterns (signals are >= 0 or NaN, and NaN is the largest pattern)
        using U = typename std::conditional<sizeof(T) == 4, unsigned int, unsigned long long>::type;
        U bits;
        if constexpr (sizeof(T) == 4)
            bits = __float_as_uint(sig) & 0x7fffffffu;
        else
            bits = (unsigned long long)__double_as_longlong(sig) & 0x7fffffffffffffffull;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const U other = __shfl_xor_sync(0xffffffffu, bits, o);
            bits = other > bits ? other : bits;
        }
        U *const sw = reinterpret_cast<U *>(sWarp);
        if ((tid & 31) == 0) sw[tid >> 5] = bits;
        __syncthreads();
        if (tid < C) {
            U m = 0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = sw[w] > m ? sw[w] : m;
            T mv;
            if constexpr (sizeof(T) == 4)
                mv = __uint_as_float(m);
            else
                mv = __longlong_as_double((long long)m);
            line_store(line_map(&sMax[s & 1][rank], tid), mv);
        }
        line_cluster_sync();
        if (tid < 32) {  // the next step, as finalize_dt sets it (every CTA the same)
            const U *mx = reinterpret_cast<const U *>(sMax[s & 1]);
            U m = 0;
            for (int r = 0; r < C; ++r) m = mx[r] > m ? mx[r] : m;
            double sg;
            if constexpr (sizeof(T) == 4)
                sg = (double)__uint_as_float(m);
            else
                sg = __longlong_as_double((long long)m);
            const double last = sStep[1];
            const double t = sInfo[0] ? t_end : sStep[0] + last;
            double dt = 0.0;
            int clipped = 0, status = sInfo[2];
            if (!(sg <= 1.7976931348623157e308) || !(sg > 0.0)) {
                status |= (int)STATUS_NONFINITE;
            } else if (status == 0) {
                dt = line_div(cfl, sg, in_range(sg) ? recip64(sg) : 0.0, A.x);
                if (t_end > 0.0) {
                    if (t >= t_end) {
                        dt = 0.0;
                    } else if (dt >= t_end - t) {
                        dt = t_end - t;
                        clipped = 1;
                    }
                }
            }
            const double ca = dt > 0.0 ? line_div(tid == 0 ? 0.5 * dt : dt, A.dr, A.inv_dr, A.x) : 0.0;
            __syncwarp();
            if (tid < 2) sStep[2 + tid] = ca;
            if (tid == 0) {
                sStep[0] = t;
                sStep[1] = dt;
                sStep[4] = last;
                sInfo[0] = clipped;
                sInfo[1] += 1;
                sInfo[2] = status;
            }
        }
        __syncthreads();
    }
    if (s > 0 && cell) {
#pragma unroll
        for (int k = 0; k < NV; ++k) A.u[k][c0 + tid] = u0[k];
    }
    if (s > 0 && rank == 0 && tid == 0) {
        c->t = sStep[0];
        c->dt = sStep[1];
        c->dt_last = sStep[4];
        c->clipped = sInfo[0];
        c->steps = sInfo[1];
        if (sInfo[2]) atomicOr(&c->status, (unsigned)sInfo[2]);
        for (int st = 0; st < 2; ++st) {
            c->coef[st][0] = sStep[2 + st];
            c->coef32[st][0] = (float)sStep[2 + st];
        }
    }
    line_cluster_sync();  // no CTA leaves while another may write to its shared memory
}

// The largest cluster of full CTAs the device runs (a property of the kernel and device, asked
// once per device); 0 if none.
template <class T> int line_max_ctas() {
    static std::atomic<int> known[64];  // 1 + the answer
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (dev < 64 && known[dev].load() > 0) return known[dev].load() - 1;
    const auto k = line_kernel<T>;
    int C = 0;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess)
        for (C = kLineMaxCtas; C >= 1; C /= 2) {
            cudaLaunchAttribute at;
            at.id = cudaLaunchAttributeClusterDimension;
            at.val.clusterDim.x = (unsigned)C;
            at.val.clusterDim.y = at.val.clusterDim.z = 1;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((unsigned)C);
            cfg.blockDim = dim3(kLineThreads);
            cfg.attrs = &at;
            cfg.numAttrs = 1;
            int fit = 0;
            if (cudaOccupancyMaxActiveClusters(&fit, k, &cfg) == cudaSuccess && fit > 0) break;
        }
    cudaGetLastError();
    if (dev < 64) known[dev].store(C + 1);
    return C;
}

// Cluster of the grid: at most one CTA per 32 cells, a power of two, one cell per thread; 0 if
// the grid does not fit one.
template <class T> int line_ctas(int n) {
    const int most = line_max_ctas<T>();
    int C = 1;
    while (2 * C <= most && n >= 64 * C) C *= 2;
    return most >= 1 && (n + C - 1) / C <= kLinePer ? C : 0;
}

template <class T> cudaError_t launch_line(const LineLaunch &L, cudaStream_t st) {
    LineArgs<T> A;
    for (int k = 0; k < 3; ++k) A.u[k] = static_cast<T *>(L.u[k]);
    A.n = L.n;
    A.per = (L.n + L.ctas - 1) / L.ctas;
    A.periodic = L.periodic;
    A.order = L.order;
    A.riemann = L.riemann;
    A.n_steps = L.n_steps;
    A.dr = L.dr;
    A.inv_dr = 1.0 / L.dr;
    A.inv_dr_t = T(1.0 / L.dr);
    A.gas = make_gas<T>(L.gamma);
    A.x = A.gas.x;
    A.ctrl = static_cast<Ctrl *>(L.ctrl);
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)L.ctas;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)L.ctas);
    cfg.blockDim = dim3((unsigned)(A.per / 32 * 32 + 32));  // A.per + 1 threads at least
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, line_kernel<T>, A);
}

}  // namespace hydro
