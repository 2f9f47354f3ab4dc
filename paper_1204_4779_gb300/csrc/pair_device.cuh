// FP32 building blocks on pairs: two neighbouring cells (or two faces) share one 64-bit register
// pair per value, so that one add, multiply or FMA instruction (f32x2) serves both.  The steps
// the hardware has no packed form of (reciprocal, square root, minimum, selection) are done per
// lane on the halves of the pair.  Every operation is named by its rounding (no expression the
// compiler could contract differently in different kernels), so a cell's result does not depend
// on which half of a pair, which lane or which kernel it was computed in.
#pragma once

#include "hydro_device.cuh"

namespace hydro {

__device__ __forceinline__ F2 f2_splat(float a) { return f2_pack(a, a); }
__device__ __forceinline__ float f2_lo(F2 v) {
    float a, b;
    f2_unpack(v, a, b);
    return a;
}
__device__ __forceinline__ float f2_hi(F2 v) {
    float a, b;
    f2_unpack(v, a, b);
    return b;
}
__device__ __forceinline__ F2 f2_rcp(F2 v) {
    float a, b;
    f2_unpack(v, a, b);
    return f2_pack(Arith<float>::rcp(a), Arith<float>::rcp(b));
}
__device__ __forceinline__ F2 f2_sqrt(F2 v) {
    float a, b;
    f2_unpack(v, a, b);
    return f2_pack(Arith<float>::sqrt_(a), Arith<float>::sqrt_(b));
}
// MinBee slopes of both lanes from the one-sided differences (zero for first order)
__device__ __forceinline__ F2 f2_minbee(F2 a, F2 b) {
    float a0, a1, b0, b1;
    f2_unpack(a, a0, a1);
    f2_unpack(b, b0, b1);
    return f2_pack(minbee(a0, b0), minbee(a1, b1));
}

// The constants of the gas, once per lane.
struct PairGas {
    F2 g, gm1, inv_gm1;
};
__device__ __forceinline__ PairGas pair_gas(const Gas<float> &G) {
    return {f2_splat(G.g), f2_splat(G.gm1), f2_splat(G.inv_gm1)};
}

// V(U) of a pair of cells (prim_of_cons).
template <int D>
__device__ __forceinline__ void prim_of_cons_pair(const F2 (&u)[D + 2], F2 (&v)[D + 2],
                                                  const PairGas &G) {
    const F2 ir = f2_rcp(u[0]);
    v[0] = u[0];
    v[1] = f2_mul(u[1], ir);
    F2 kin = f2_mul(u[1], v[1]);
#pragma unroll
    for (int a = 1; a < D; ++a) {
        v[1 + a] = f2_mul(u[1 + a], ir);
        kin = f2_fma(u[1 + a], v[1 + a], kin);
    }
    v[D + 1] = f2_mul(G.gm1, f2_fma(f2_splat(-0.5f), kin, u[D + 1]));
}

// HLLC flux of a pair of faces; velocities and flux normal-first.  The operations of the FP32
// hllc(), on both lanes.
template <int D>
__device__ __forceinline__ void hllc_pair(F2 rl, const F2 (&vl)[D], F2 pl, F2 rr,
                                          const F2 (&vr)[D], F2 pr, const PairGas &G,
                                          F2 (&F)[D + 2], int riemann = 0) {
    const F2 ul = vl[0], ur = vr[0];
    const F2 al = f2_sqrt(f2_mul(f2_mul(G.g, pl), f2_rcp(rl)));
    const F2 ar = f2_sqrt(f2_mul(f2_mul(G.g, pr), f2_rcp(rr)));
    float SL[2], SR[2];
    if (riemann == 0) {
        float a0, a1, b0, b1;
        f2_unpack(f2_sub(ul, al), a0, a1);
        f2_unpack(f2_sub(ur, ar), b0, b1);
        SL[0] = fminf(fminf(a0, b0), 0.0f);
        SL[1] = fminf(fminf(a1, b1), 0.0f);
        f2_unpack(f2_add(ul, al), a0, a1);
        f2_unpack(f2_add(ur, ar), b0, b1);
        SR[0] = fmaxf(fmaxf(a0, b0), 0.0f);
        SR[1] = fmaxf(fmaxf(a1, b1), 0.0f);
    } else {
        float l[2], r[2], p1[2], p2[2], c1[2], c2[2], u1[2], u2[2];
        f2_unpack(rl, l[0], l[1]);
        f2_unpack(rr, r[0], r[1]);
        f2_unpack(pl, p1[0], p1[1]);
        f2_unpack(pr, p2[0], p2[1]);
        f2_unpack(al, c1[0], c1[1]);
        f2_unpack(ar, c2[0], c2[1]);
        f2_unpack(ul, u1[0], u1[1]);
        f2_unpack(ur, u2[0], u2[1]);
#pragma unroll
        for (int i = 0; i < 2; ++i)
            pvrs_speeds(l[i], u1[i], p1[i], c1[i], r[i], u2[i], p2[i], c2[i], f2_lo(G.g), SL[i], SR[i]);
    }
    const F2 ml = f2_mul(rl, f2_sub(f2_pack(SL[0], SL[1]), ul));
    const F2 nr = f2_mul(rr, f2_sub(ur, f2_pack(SR[0], SR[1])));  // -m_R
    const F2 num = f2_fma(ur, nr, f2_fma(ul, ml, f2_sub(pr, pl)));
    const F2 Ss = f2_mul(num, f2_rcp(f2_add(ml, nr)));
    float ss[2], s[2];
    f2_unpack(Ss, ss[0], ss[1]);
    bool left[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        left[i] = SL[i] >= 0.0f || ss[i] >= 0.0f;
        if (riemann != 0) SL[i] = fminf(SL[i], 0.0f), SR[i] = fmaxf(SR[i], 0.0f);
        s[i] = left[i] ? SL[i] : SR[i];
    }
    auto side = [&](F2 a, F2 b) {
        float a0, a1, b0, b1;
        f2_unpack(a, a0, a1);
        f2_unpack(b, b0, b1);
        return f2_pack(left[0] ? a0 : b0, left[1] ? a1 : b1);
    };
    const F2 p = side(pl, pr), S = f2_pack(s[0], s[1]);
    F2 v[D];
#pragma unroll
    for (int b = 0; b < D; ++b) v[b] = side(vl[b], vr[b]);
    const F2 u = v[0];
    const F2 us = f2_sub(u, S);
    F2 m;  // r (u - S)
    if (riemann == 0) {
        float l[2], r[2];
        f2_unpack(ml, l[0], l[1]);
        f2_unpack(nr, r[0], r[1]);
        m = f2_pack(left[0] ? -l[0] : r[0], left[1] ? -l[1] : r[1]);
    } else {
        m = f2_mul(side(rl, rr), us);
    }
    const F2 ps = f2_fma(m, f2_sub(u, Ss), p);
    float q[2];
    f2_unpack(f2_mul(Ss, f2_rcp(f2_sub(Ss, S))), q[0], q[1]);
    const F2 Q = f2_pack(s[0] == 0.0f ? 1.0f : q[0], s[1] == 0.0f ? 1.0f : q[1]);
    F2 v2 = f2_mul(u, u);
#pragma unroll
    for (int b = 1; b < D; ++b) v2 = f2_fma(v[b], v[b], v2);
    F[0] = f2_mul(m, Q);
    F[1] = f2_fma(F[0], Ss, ps);
#pragma unroll
    for (int b = 1; b < D; ++b) F[1 + b] = f2_mul(F[0], v[b]);
    const F2 x = f2_mul(ps, Ss);
    const F2 t = f2_fma(f2_mul(f2_splat(0.5f), m), v2, f2_mul(p, f2_fma(us, G.inv_gm1, u)));
    F[D + 1] = f2_fma(Q, f2_sub(t, x), x);
}

// CFL signal sum_a (|v_a| + c_s) / dr_a of a pair of new states (cfl_signal), per lane in s[],
// and the smaller of rho and p in low[] (NaN propagates into both).
template <int D>
__device__ __forceinline__ void cfl_signal_pair(const F2 (&un)[D + 2], const PairGas &G,
                                                const float *inv_dr, float (&s)[2],
                                                float (&low)[2]) {
    F2 v[D + 2];
    prim_of_cons_pair<D>(un, v, G);
    float c[2], a[2], r[2], p[2];
    const F2 cs = f2_sqrt(f2_mul(f2_mul(G.g, v[D + 1]), f2_rcp(v[0])));
    f2_unpack(cs, c[0], c[1]);
    f2_unpack(v[0], r[0], r[1]);
    f2_unpack(v[D + 1], p[0], p[1]);
#pragma unroll
    for (int i = 0; i < 2; ++i)
        asm("min.NaN.f32 %0, %1, %2;" : "=f"(low[i]) : "f"(r[i]), "f"(p[i]));
    s[0] = s[1] = 0.0f;
#pragma unroll
    for (int d = 0; d < D; ++d) {
        f2_unpack(v[1 + d], a[0], a[1]);
#pragma unroll
        for (int i = 0; i < 2; ++i) s[i] = fmaf(__fadd_rn(fabsf(a[i]), c[i]), inv_dr[d], s[i]);
    }
}
__device__ __forceinline__ void max_nan(float &m, float s) {
    asm("max.NaN.f32 %0, %0, %1;" : "+f"(m) : "f"(s));
}
__device__ __forceinline__ void min_nan(float &m, float s) {
    asm("min.NaN.f32 %0, %0, %1;" : "+f"(m) : "f"(s));
}

}  // namespace hydro
