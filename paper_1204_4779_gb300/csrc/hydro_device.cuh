// Device building blocks of the compressible-Euler step (arXiv:1204.4779, section 4.1):
// primitive recovery, the MinBee slope, the HLLC face flux, boundary index remapping and the
// on-device dt control block.
//
// Two arithmetic modes, chosen by the element type:
//  * double: the results of the plain formulas, each operation correctly rounded in the formulas'
//    order.  The FP64 translation units are compiled with --fmad=false; quotients, roots and
//    comparisons are those of exact64.cuh, which give the IEEE results by fewer FP64 operations;
//  * float:  the stencil runs in FP32 with fused multiply-adds and the approximate MUFU
//    reciprocal and square root (rcp.approx / sqrt.approx).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "exact64.cuh"

namespace hydro {

// ----------------------------------------------------------------- control block ----------

// One per context, in the workspace.  Written by the CFL pass and by the last CTA of every
// RK stage-2 launch; read by every CTA of the stage kernels.
struct Ctrl {
    double t;               // time of the state the next step starts from
    double dt;              // dt of the next step; 0 = no further step in this call
    double t_end;           // <= 0: no clipping
    double cfl;
    double dt_last;         // dt of the last completed step
    unsigned long long sig64;  // running max of the CFL signal, FP64 bit pattern
    unsigned int sig32;        // running max of the CFL signal, FP32 bit pattern
    unsigned int blocks_done;  // CTAs finished in the current reduction launch
    unsigned int status;       // bit 0: non-finite / non-positive value seen
    int steps;              // steps completed since the CFL pass
    int clipped;            // the next step is clipped onto t_end
    unsigned int claim;       // persistent stage launches: work items claimed beyond the first
    unsigned int claim_done;  // CTAs of the current persistent launch that stopped claiming
    int pad;
    double totals[5];       // output of the totals reduction
    double dr[3];           // cell sizes (set by the host with t, t_end, cfl)
    double coef[2][3];      // (dt/2)/dr_a and dt/dr_a of the next step, for RK stages 1 and 2
    float coef32[2][3];     // the same rounded to FP32 (a conversion costs a kernel's every warp
                            // as much as an FP64 operation)
};
static_assert(sizeof(Ctrl) <= 256, "the control block has 256 bytes in every workspace");

enum : unsigned int {
    STATUS_NONFINITE = 1u,  // non-finite, rho <= 0 or p <= 0 seen
    STATUS_TIMEOUT = 2u,    // a bounded wait on an mbarrier gave up
};

// ------------------------------------------------------------------- arithmetic -----------

template <class T> struct Arith;

template <> struct Arith<double> {
    static constexpr bool exact = true;
    __device__ static __forceinline__ double div(double a, double b) { return a / b; }
    __device__ static __forceinline__ double sqrt_(double a) { return sqrt(a); }
};

template <> struct Arith<float> {
    static constexpr bool exact = false;
    __device__ static __forceinline__ float rcp(float a) {
        float r;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
        return r;
    }
    __device__ static __forceinline__ float div(float a, float b) { return a * rcp(b); }
    __device__ static __forceinline__ float sqrt_(float a) {
        float r;
        asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
        return r;
    }
};

// Packed FP32 pairs: Blackwell's f32x2 add/sub/mul/fma apply one operation to two FP32 values
// held in a 64-bit register pair, so one issued instruction does the work of two.  Each lane
// rounds as the scalar instruction would (round to nearest, flush-to-zero like the FP32 units).
struct F2 {
    unsigned long long r;
};
__device__ __forceinline__ F2 f2_pack(float a, float b) {
    F2 v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v.r) : "f"(a), "f"(b));
    return v;
}
__device__ __forceinline__ void f2_unpack(F2 v, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v.r));
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
    F2 d;
    asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(d.r) : "l"(a.r), "l"(b.r));
    return d;
}
__device__ __forceinline__ F2 f2_sub(F2 a, F2 b) {
    F2 d;
    asm("sub.rn.ftz.f32x2 %0, %1, %2;" : "=l"(d.r) : "l"(a.r), "l"(b.r));
    return d;
}
// A product as a * b + 0 (the same but for the sign of a zero): the assembler fuses a packed
// multiplication with a packed addition that follows, .rn or not and whatever -fmad says, and
// does so in one copy of inlined code and not in another; a product that must be rounded by
// itself in every kernel is therefore not written as one.
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
    F2 d;
    asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(d.r) : "l"(a.r), "l"(b.r), "l"(0ull));
    return d;
}
// a * b + c, one rounding per lane
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c) {
    F2 d;
    asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(d.r) : "l"(a.r), "l"(b.r), "l"(c.r));
    return d;
}

// Double-float arithmetic: a value carried as an unevaluated sum hi + lo of two FP32 numbers
// (Dekker's and Knuth's error-free transformations, as used in double-double arithmetic).  The
// additions are plain IEEE operations in the order written; the translation units that use
// them either compile with --fmad=false or use no contractible product next to them.
struct DF {
    float hi, lo;
};
// a + b exactly as hi + lo (Knuth's TwoSum, six operations, any magnitudes)
__device__ __forceinline__ DF two_sum(float a, float b) {
    const float s = a + b;
    const float bb = s - a;
    const float e = (a - (s - bb)) + (b - bb);
    return {s, e};
}
// (hi + lo)^2 as a pair: hi^2 exactly by TwoProduct with an FMA, plus 2 hi lo (lo^2 dropped)
__device__ __forceinline__ DF square(DF x) {
    const float p = x.hi * x.hi;
    float e = fmaf(x.hi, x.hi, -p);
    e = fmaf(x.hi + x.hi, x.lo, e);
    return {p, e};
}
// running sum s += x: TwoSum of the high parts, low parts added, then renormalised so that
// |lo| <= ulp(hi) / 2 (Fast2Sum)
__device__ __forceinline__ void acc_add(DF &s, DF x) {
    const DF t = two_sum(s.hi, x.hi);
    const float e = t.lo + (s.lo + x.lo);
    const float h = t.hi + e;
    s.lo = e - (h - t.hi);
    s.hi = h;
}

template <class T> struct Gas {
    T g;        // gamma
    T gm1;      // gamma - 1
    T inv_gm1;  // 1 / (gamma - 1)
    Fma64 x;    // FP64 mode's constants
};

template <class T> __host__ __device__ inline Gas<T> make_gas(double gamma) {
    Gas<T> G;
    G.g = T(gamma);
    G.gm1 = T(gamma - 1.0);
    G.inv_gm1 = T(1.0 / (gamma - 1.0));
    G.x.one = 1.0;
    G.x.mzero = -0.0;
    return G;
}

// FP64 operations for operands the arithmetic of exact64.cuh leaves out, out of line (scalars
// only: the callers' arrays stay in registers).
static __device__ __noinline__ double div_plain(double a, double b) { return a / b; }
static __device__ __noinline__ double root_plain(double a) { return sqrt(a); }

// V(U) for one cell: v_a = m_a / rho, p = (gamma - 1)(E - rho v^2 / 2), the kinetic term
// summed in axis order as m_a v_a.
template <class T, int D>
__device__ __forceinline__ void prim_of_cons(const T (&u)[D + 2], T (&v)[D + 2], const Gas<T> &G) {
    const T rho = u[0];
    v[0] = rho;
    if constexpr (Arith<T>::exact) {
        // the plain form's values (0.5 kin is exact, so the FMA rounds once, as the difference)
        bool ok = in_range(rho) && positive(rho);
        const T y = recip64(rho);
        T kin = T(0);
#pragma unroll
        for (int a = 0; a < D; ++a) {
            ok &= in_range(u[1 + a]) || is_zero(u[1 + a]);
            v[1 + a] = G.x.div(u[1 + a], rho, y);
            const T e = G.x.mul(u[1 + a], v[1 + a]);
            kin = a == 0 ? e : G.x.add(kin, e);
        }
        v[D + 1] = G.x.mul(G.gm1, fma(-0.5, kin, u[D + 1]));
        if (!ok) {
            kin = T(0);
#pragma unroll
            for (int a = 0; a < D; ++a) {
                v[1 + a] = div_plain(u[1 + a], rho);
                kin = kin + u[1 + a] * v[1 + a];
            }
            v[D + 1] = G.gm1 * (u[D + 1] - T(0.5) * kin);
        }
    } else {
        const T ir = Arith<float>::rcp(rho);
        T kin = T(0);
#pragma unroll
        for (int a = 0; a < D; ++a) {
            v[1 + a] = u[1 + a] * ir;
            kin = fmaf(u[1 + a], v[1 + a], kin);
        }
        v[D + 1] = G.gm1 * fmaf(-0.5f, kin, u[D + 1]);
    }
}

// MinBee slope of Eq. eqInterpolateSingle from the two one-sided differences:
// 0 if d01 d12 < 0, else the one of smaller magnitude (d12 on a tie).
// FP64 on the bit patterns.  d01 d12 < 0: the signs differ, neither is zero or NaN, and the
// product does not underflow (differences that small are multiplied out).
__device__ __forceinline__ double minbee(double d01, double d12) {
    const unsigned long long a = (unsigned long long)__double_as_longlong(d01) & 0x7fffffffffffffffull;
    const unsigned long long b = (unsigned long long)__double_as_longlong(d12) & 0x7fffffffffffffffull;
    const int ah = (int)(a >> 32), bh = (int)(b >> 32);
    constexpr int kNan = 0x7ff80000;
    bool opposite = (__double2hiint(d01) ^ __double2hiint(d12)) < 0 && a != 0ull && b != 0ull &&
                    max(ah, bh) < kNan;
    if (opposite && (ah >> 20) + (bh >> 20) < 1100) opposite = d01 * d12 < 0.0;
    return opposite ? 0.0 : (a < b && bh < kNan ? d01 : d12);
}
// FP32 form in three ALU operations: min.xorsign.abs gives min(|a|, |b|) carrying a negative
// sign exactly when the signs of a and b differ; clamping at zero yields 0 for opposite signs;
// the sign of a restores the slope's sign.  Same values as the form above (up to the sign of
// a zero slope).
__device__ __forceinline__ float minbee(float d01, float d12) {
    float m;
    asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(m) : "f"(d01), "f"(d12));
    return copysignf(fmaxf(m, 0.0f), d01);
}

// HLLC flux through a face whose normal is axis a (Toro, Spruce & Speares; Davis wave-speed
// estimates), from the reconstructed primitive states on its lower (L) and upper (R) side.
// Velocities and the returned flux are in NORMAL-FIRST order: (normal, tangential in
// increasing axis order).  Flux components: (mass, normal momentum, tangential momenta,
// energy).  NLAST: the normal axis is the last axis (only the kinetic-energy summation order
// of the exact mode depends on it: v^2 is summed in axis order).
// riemann: wave-speed estimate, 0 = Davis, 1 = pressure-based (Toro's PVRS: p_pv from the
// arithmetic means, p* = max(0, p_pv), q_K = 1 or sqrt(1 + (g+1)/(2g) (p*/p_K - 1)) behind a
// shock, S_L = u_L - a_L q_L, S_R = u_R + a_R q_R).
//
// FP64: F_L if S_L >= 0; F*_L if S* >= 0; F*_R if S_R > 0; else F_R, with the formulas' own
// operations in their order.  The plain form, for operands the fast one below leaves out and
// the pressure-based speeds.
template <int D, bool NLAST>
__device__ __forceinline__ void hllc_plain(double rl, const double (&vl)[D], double pl, double rr,
                                           const double (&vr)[D], double pr, const Gas<double> &G,
                                           double (&F)[D + 2], int riemann) {
    using T = double;
    const T ul = vl[0], ur = vr[0];
    const T al = root_plain(div_plain(G.g * pl, rl));
    const T ar = root_plain(div_plain(G.g * pr, rr));
    T SL, SR;
    if (riemann == 0) {
        SL = fmin(ul - al, ur - ar);
        SR = fmax(ul + al, ur + ar);
    } else {
        const T rbar = T(0.5) * (rl + rr);
        const T abar = T(0.5) * (al + ar);
        const T ppv = T(0.5) * (pl + pr) - T(0.5) * (ur - ul) * rbar * abar;
        const T ps = fmax(T(0), ppv);
        T ql = T(1), qr = T(1);
        const T c = div_plain(G.g + T(1), T(2) * G.g);
        if (!(ps <= pl)) ql = root_plain(T(1) + c * (div_plain(ps, pl) - T(1)));
        if (!(ps <= pr)) qr = root_plain(T(1) + c * (div_plain(ps, pr) - T(1)));
        SL = ul - al * ql;
        SR = ur + ar * qr;
    }
    const T ml = rl * (SL - ul);
    const T mr = rr * (SR - ur);
    const T Ss = div_plain(pr - pl + rl * ul * (SL - ul) - rr * ur * (SR - ur), ml - mr);

    const bool left = (T(0) <= SL) || (T(0) <= Ss);
    const bool star = !(T(0) <= SL) && ((T(0) <= Ss) || (T(0) < SR));
    const T r = left ? rl : rr;
    const T p = left ? pl : pr;
    const T S = left ? SL : SR;
    T v[D];
#pragma unroll
    for (int b = 0; b < D; ++b) v[b] = left ? vl[b] : vr[b];
    const T u = v[0];

    // kinetic energy in axis order
    T v2 = T(0);
    if constexpr (NLAST) {
#pragma unroll
        for (int b = 1; b < D; ++b) v2 = v2 + v[b] * v[b];
        v2 = v2 + v[0] * v[0];
    } else {
#pragma unroll
        for (int b = 0; b < D; ++b) v2 = v2 + v[b] * v[b];
    }

    T U[D + 2], FK[D + 2];
    U[0] = r;
    FK[0] = r * u;
#pragma unroll
    for (int b = 0; b < D; ++b) U[1 + b] = r * v[b];
    U[D + 1] = div_plain(p, G.gm1) + T(0.5) * r * v2;
    FK[1] = U[1] * u + p;
#pragma unroll
    for (int b = 1; b < D; ++b) FK[1 + b] = U[1 + b] * u;
    FK[D + 1] = u * (U[D + 1] + p);

    // star state: rho (S - u)/(S - S*) (1, S*, v_t, E/rho + (S* - u)(S* + p/(rho (S - u))))
    const T chi = div_plain(r * (S - u), S - Ss);
    const T eterm = div_plain(U[D + 1], r) + (Ss - u) * (Ss + div_plain(p, r * (S - u)));
    T Us[D + 2];
    Us[0] = chi;
    Us[1] = chi * Ss;
#pragma unroll
    for (int b = 1; b < D; ++b) Us[1 + b] = chi * v[b];
    Us[D + 1] = chi * eterm;
#pragma unroll
    for (int k = 0; k < D + 2; ++k) F[k] = star ? FK[k] + S * (Us[k] - U[k]) : FK[k];
}

// The same values by the arithmetic of exact64.cuh: about 105 FP64 operations a face in 3D
// where the plain form issues 150.  5 reciprocals serve 7 quotients; S - u, r (S - u) and r u of
// the chosen side are selected, not computed again; 0.5 r v^2 is added by an FMA (the half is
// exact).
template <int D, bool NLAST>
__device__ __forceinline__ void hllc(double rl, const double (&vl)[D], double pl, double rr,
                                     const double (&vr)[D], double pr, const Gas<double> &G,
                                     double (&F)[D + 2], int riemann = 0) {
    const Fma64 &X = G.x;
    const double ul = vl[0], ur = vr[0];
    bool ok = riemann == 0 && in_range(rl) && in_range(rr) && in_range(pl) && in_range(pr) &&
              positive(rl) && positive(rr) && positive(pl) && positive(pr);
    const double yl = recip64(rl), yr = recip64(rr);
    const double al = sqrt64(X.div(X.mul(G.g, pl), rl, yl), X);
    const double ar = sqrt64(X.div(X.mul(G.g, pr), rr, yr), X);
    const double la = X.sub(ul, al), lb = X.sub(ur, ar), ra = X.add(ul, al), rb = X.add(ur, ar);
    const double SL = less(lb, la) ? lb : la, SR = less(ra, rb) ? rb : ra;
    const double sl = X.sub(SL, ul), sr = X.sub(SR, ur);
    const double ml = X.mul(rl, sl), mr = X.mul(rr, sr);
    const double rul = X.mul(rl, ul), rur = X.mul(rr, ur);
    const double num = X.sub(X.add(X.sub(pr, pl), X.mul(rul, sl)), X.mul(rur, sr));
    const double den = X.sub(ml, mr);
    ok = ok && in_range(den) && (in_range(num) || is_zero(num));
    const double Ss = X.div_by_negative(num, den, recip64(den));
    const bool left = ge0(SL) || ge0(Ss);
    const bool star = !ge0(SL) && (ge0(Ss) || gt0(SR));
    const double r = left ? rl : rr, p = left ? pl : pr, S = left ? SL : SR;
    const double y = left ? yl : yr, m = left ? ml : mr;
    double v[D];
#pragma unroll
    for (int b = 0; b < D; ++b) v[b] = left ? vl[b] : vr[b];
    const double u = v[0];
    // v^2 in axis order
    double v2;
    if constexpr (NLAST && D > 1) {
        v2 = X.mul(v[1], v[1]);
#pragma unroll
        for (int b = 2; b < D; ++b) v2 = X.add(v2, X.mul(v[b], v[b]));
        v2 = X.add(v2, X.mul(u, u));
    } else {
        v2 = X.mul(u, u);
#pragma unroll
        for (int b = 1; b < D; ++b) v2 = X.add(v2, X.mul(v[b], v[b]));
    }
    double U[D + 2], FK[D + 2];
    U[0] = r;
    U[1] = left ? rul : rur;
    FK[0] = U[1];
#pragma unroll
    for (int b = 1; b < D; ++b) U[1 + b] = X.mul(r, v[b]);
    const double E = fma(0.5, X.mul(r, v2), X.div(p, G.gm1, G.inv_gm1));
    U[D + 1] = E;
    FK[1] = X.add(X.mul(U[1], u), p);
#pragma unroll
    for (int b = 1; b < D; ++b) FK[1 + b] = X.mul(U[1 + b], u);
    FK[D + 1] = X.mul(u, X.add(E, p));
    const double sd = X.sub(S, Ss);
    ok = ok && in_range(E) && (!star || (in_range(sd) && in_range(m)));
    const double chi = X.div(m, sd, recip64(sd));
    const double eterm = X.add(X.div(E, r, y),
                               X.mul(X.sub(Ss, u), X.add(Ss, X.div(p, m, recip64(m)))));
    double Us[D + 2];
    Us[0] = chi;
    Us[1] = X.mul(chi, Ss);
#pragma unroll
    for (int b = 1; b < D; ++b) Us[1 + b] = X.mul(chi, v[b]);
    Us[D + 1] = X.mul(chi, eterm);
#pragma unroll
    for (int k = 0; k < D + 2; ++k) {
        const double f = X.add(FK[k], X.mul(S, X.sub(Us[k], U[k])));
        F[k] = star ? f : FK[k];
    }
    if (!ok) hllc_plain<D, NLAST>(rl, vl, pl, rr, vr, pr, G, F, riemann);
}

// Pressure-based wave speeds of one face in FP32, every operation named by its rounding.
__device__ __forceinline__ void pvrs_speeds(float rl, float ul, float pl, float al, float rr,
                                            float ur, float pr, float ar, float g, float &SL,
                                            float &SR) {
    const float c = __fmul_rn(__fadd_rn(g, 1.0f), __fmul_rn(0.5f, Arith<float>::rcp(g)));
    const float ra = __fmul_rn(__fmul_rn(0.5f, __fadd_rn(rl, rr)), __fmul_rn(0.5f, __fadd_rn(al, ar)));
    const float ps = fmaxf(0.0f, fmaf(__fmul_rn(-0.5f, __fadd_rn(ur, -ul)), ra,
                                      __fmul_rn(0.5f, __fadd_rn(pl, pr))));
    float ql = 1.0f, qr = 1.0f;
    if (!(ps <= pl)) ql = Arith<float>::sqrt_(fmaf(c, fmaf(ps, Arith<float>::rcp(pl), -1.0f), 1.0f));
    if (!(ps <= pr)) qr = Arith<float>::sqrt_(fmaf(c, fmaf(ps, Arith<float>::rcp(pr), -1.0f), 1.0f));
    SL = fmaf(-al, ql, ul);
    SR = fmaf(ar, qr, ur);
}

// FP32: the star form with clamped wave speeds (S_L to <= 0, S_R to >= 0).  The jump condition
// F* = F_K + S (U* - U_K) then covers all four cases: on a supersonic face S is 0 and F* = F_K.
// Written in the star state it needs neither F_K nor U_K.  With m = r (u - S),
// p* = p + m (u - S*) and q = S* / (S* - S) (q = 1 where S = 0),
//     F_mass = m q,  F_normal = F_mass S* + p*,  F_tangential = F_mass v_t,
//     F_E    = p* S* + q (p ((u - S) / (gamma - 1) + u) + m v^2 / 2 - p* S*),
// 55 instructions a face in 3D where the form through F_K and U_K took 75.
// The clamped speeds also enter S*: it is then the same wherever no wave speed has passed zero,
// and its sign, which chooses the side, is the same everywhere (Davis speeds: if S_R <= 0, both
// sides' u <= -a, and the numerator of S* is at least (gamma - 1) p_L + (gamma + 1) p_R > 0 with
// either S_R, so S* < 0).  The pressure-based estimate bounds only its own side's velocity, so
// there S* comes from the unclamped speeds.
// Every operation is named by its rounding: hllc_pair (pair_device.cuh) does the same ones on
// two faces at once, and kernels that use either agree bit for bit.
template <int D, bool NLAST>
__device__ __forceinline__ void hllc(float rl, const float (&vl)[D], float pl, float rr,
                                     const float (&vr)[D], float pr, const Gas<float> &G,
                                     float (&F)[D + 2], int riemann = 0) {
    const float ul = vl[0], ur = vr[0];
    const float al = Arith<float>::sqrt_(__fmul_rn(__fmul_rn(G.g, pl), Arith<float>::rcp(rl)));
    const float ar = Arith<float>::sqrt_(__fmul_rn(__fmul_rn(G.g, pr), Arith<float>::rcp(rr)));
    float SL, SR;
    if (riemann == 0) {
        SL = fminf(fminf(__fadd_rn(ul, -al), __fadd_rn(ur, -ar)), 0.0f);
        SR = fmaxf(fmaxf(__fadd_rn(ul, al), __fadd_rn(ur, ar)), 0.0f);
    } else {
        pvrs_speeds(rl, ul, pl, al, rr, ur, pr, ar, G.g, SL, SR);
    }
    const float ml = __fmul_rn(rl, __fadd_rn(SL, -ul));
    const float nr = __fmul_rn(rr, __fadd_rn(ur, -SR));  // -m_R
    const float num = fmaf(ur, nr, fmaf(ul, ml, __fadd_rn(pr, -pl)));
    const float Ss = __fmul_rn(num, Arith<float>::rcp(__fadd_rn(ml, nr)));
    const bool left = SL >= 0.0f || Ss >= 0.0f;
    if (riemann != 0) SL = fminf(SL, 0.0f), SR = fmaxf(SR, 0.0f);
    const float S = left ? SL : SR;
    const float p = left ? pl : pr;
    float v[D];
#pragma unroll
    for (int b = 0; b < D; ++b) v[b] = left ? vl[b] : vr[b];
    const float u = v[0];
    const float us = __fadd_rn(u, -S);
    const float m = riemann == 0 ? (left ? -ml : nr) : __fmul_rn(left ? rl : rr, us);
    const float ps = fmaf(m, __fadd_rn(u, -Ss), p);
    const float q = S == 0.0f ? 1.0f : __fmul_rn(Ss, Arith<float>::rcp(__fadd_rn(Ss, -S)));
    float v2 = __fmul_rn(u, u);
#pragma unroll
    for (int b = 1; b < D; ++b) v2 = fmaf(v[b], v[b], v2);
    F[0] = __fmul_rn(m, q);
    F[1] = fmaf(F[0], Ss, ps);
#pragma unroll
    for (int b = 1; b < D; ++b) F[1 + b] = __fmul_rn(F[0], v[b]);
    const float x = __fmul_rn(ps, Ss);
    const float t = fmaf(__fmul_rn(0.5f, m), v2, __fmul_rn(p, fmaf(us, G.inv_gm1, u)));
    F[D + 1] = fmaf(q, __fadd_rn(t, -x), x);
}

// CFL signal sum_a (|v_a| + c_s) / dr_a of an FP64 primitive state, c_s = sqrt(gamma p / rho).
template <int D>
__device__ __forceinline__ double exact_signal(const double (&v)[D + 2], const Gas<double> &G,
                                               const double *dr, const double *inv_dr) {
    const Fma64 &X = G.x;
    bool ok = in_range(v[0]) && in_range(v[D + 1]) && positive(v[0]) && positive(v[D + 1]);
    const double cs = sqrt64(X.div(X.mul(G.g, v[D + 1]), v[0], recip64(v[0])), X);
    double s = 0.0;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const double w = X.add(fabs(v[1 + a]), cs);
        ok = ok && in_range(w) && in_range(dr[a]);
        const double q = X.div(w, dr[a], inv_dr[a]);
        s = a == 0 ? q : X.add(s, q);
    }
    if (!ok) {
        const double c = root_plain(div_plain(G.g * v[D + 1], v[0]));
        s = 0.0;
#pragma unroll
        for (int a = 0; a < D; ++a) s = s + div_plain(fabs(v[1 + a]) + c, dr[a]);
    }
    return s;
}

// Boundary remap of a cell index at most two cells outside [0, n): periodic wraps once,
// outflow (zero gradient) clamps; the final clamp also keeps the unused positions of a ragged
// tile (more than two cells outside) in bounds.
__device__ __forceinline__ int remap(int i, int n, int periodic) {
    if (periodic) i = i < 0 ? i + n : (i >= n ? i - n : i);
    return min(max(i, 0), n - 1);
}
// The same for an index known to be >= 0 (the planes ahead of a marching tile): only the
// upper side can be outside, and the result equals remap(i, n, periodic).
__device__ __forceinline__ int remap_ahead(int i, int n, int periodic) {
    return min((periodic && i >= n) ? i - n : i, n - 1);
}

// ------------------------------------------------------------- dt finalisation ------------

template <class T> __device__ __forceinline__ double take_signal(Ctrl *c);
template <> __device__ __forceinline__ double take_signal<float>(Ctrl *c) {
    unsigned int b = atomicExch(&c->sig32, 0u);
    return (double)__uint_as_float(b);
}
template <> __device__ __forceinline__ double take_signal<double>(Ctrl *c) {
    unsigned long long b = atomicExch(&c->sig64, 0ull);
    return __longlong_as_double((long long)b);
}

template <class T> __device__ __forceinline__ void push_signal(Ctrl *c, T s);
template <> __device__ __forceinline__ void push_signal<float>(Ctrl *c, float s) {
    atomicMax(&c->sig32, __float_as_uint(s));
}
template <> __device__ __forceinline__ void push_signal<double>(Ctrl *c, double s) {
    atomicMax(&c->sig64, (unsigned long long)__double_as_longlong(s));
}

// Whether the control block holds a step to take (dt > 0; dt is never NaN), without an FP64
// comparison.
__device__ __forceinline__ bool step_pending(const Ctrl *c) {
    return __ldcg(reinterpret_cast<const long long *>(&c->dt)) > 0;
}
// AddFlux coefficient of RK stage `stage` (1 or 2) along axis a.
template <class T> __device__ __forceinline__ T step_coef(const Ctrl *c, int stage, int a) {
    if constexpr (sizeof(T) == 4)
        return __ldcg(&c->coef32[stage - 1][a]);
    else
        return __ldcg(&c->coef[stage - 1][a]);
}

// Run by one whole warp of the last CTA of a reduction launch.  `advance`: a step with
// dt = c->dt has just completed (no step ran if that dt is 0, e.g. once t reached t_end).  Then
// dt of the next step = cfl / max signal, clipped onto t_end.  Lane 0 sets dt; the six
// coefficients are divided one per lane (an FP64 division takes a warp about 600 cycles however
// few lanes take part, and every step waits for this).
template <class T> __device__ void finalize_dt(Ctrl *c, bool advance) {
    volatile Ctrl *vc = c;
    const int lane = threadIdx.x & 31;
    double dt = 0.0;
    if (lane == 0) {
        if (advance && vc->dt > 0.0) {
            const double d = vc->dt;
            vc->t = vc->clipped ? vc->t_end : vc->t + d;
            vc->dt_last = d;
            vc->steps = vc->steps + 1;
        }
        const double s = take_signal<T>(c);
        const double t = vc->t, t_end = vc->t_end;
        int clipped = 0;
        if (!(s <= 1.7976931348623157e308) || !(s > 0.0)) {  // NaN, inf or no signal
            atomicOr(&c->status, STATUS_NONFINITE);
        } else if (vc->status == 0u) {
            dt = vc->cfl / s;
            if (t_end > 0.0) {
                if (t >= t_end) {
                    dt = 0.0;
                } else if (dt >= t_end - t) {
                    dt = t_end - t;
                    clipped = 1;
                }
            }
        }
        if (atomicOr(&c->status, 0u) != 0u) dt = 0.0;
        vc->dt = dt;
        vc->clipped = clipped;
    }
    dt = __shfl_sync(0xffffffffu, dt, 0);
    // AddFlux coefficients of both stages, in the order of Eq. eqAddFlux: (c dt) / dr_a
    if (lane < 6) {
        const int st = lane / 3, a = lane - 3 * st;
        const double q = (st == 0 ? 0.5 * dt : dt) / vc->dr[a];
        vc->coef[st][a] = q;
        vc->coef32[st][a] = (float)q;
    }
    __threadfence();
}

// Block-wide max of a non-negative value (NaN propagates as the largest bit pattern), then
// one atomic per CTA; the last of `nblocks` contributions (0: every CTA of the launch)
// finalises dt.  Call from all threads of the CTA (NT of them; NT = 0: blockDim.x).
template <class T, int NT>
__device__ __forceinline__ void reduce_signal_and_finalize(Ctrl *ctrl, T smax, bool bad,
                                                           bool advance, T *sred,
                                                           unsigned int nblocks = 0) {
    // warp max on the bit patterns (order-free and exact)
    using U = typename std::conditional<sizeof(T) == 4, unsigned int, unsigned long long>::type;
    U bits;
    if constexpr (sizeof(T) == 4)
        bits = __float_as_uint(smax);
    else
        bits = (unsigned long long)__double_as_longlong(smax);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        U other = __shfl_xor_sync(0xffffffffu, bits, o);
        bits = other > bits ? other : bits;
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int anybad = __syncthreads_or(bad ? 1 : 0);
    U *sb = reinterpret_cast<U *>(sred);
    if (lane == 0) sb[warp] = bits;
    __syncthreads();
    if (warp == 0) {
        unsigned int last = 0;
        if (lane == 0) {
            U m = 0;
#pragma unroll 1
            for (int w = 0; w < (NT ? NT : (int)blockDim.x) / 32; ++w) m = sb[w] > m ? sb[w] : m;
            T bm;
            if constexpr (sizeof(T) == 4)
                bm = __uint_as_float(m);
            else
                bm = __longlong_as_double((long long)m);
            push_signal<T>(ctrl, bm);
            if (anybad) atomicOr(&ctrl->status, STATUS_NONFINITE);
            __threadfence();
            if (nblocks == 0) nblocks = gridDim.x * gridDim.y * gridDim.z;
            last = atomicAdd(&ctrl->blocks_done, 1u) == nblocks - 1;
        }
        if (__shfl_sync(0xffffffffu, last, 0)) {
            __threadfence();
            finalize_dt<T>(ctrl, advance);
            if (lane == 0) atomicExch(&ctrl->blocks_done, 0u);
        }
    }
}

}  // namespace hydro
