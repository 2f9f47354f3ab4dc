// FP64 arithmetic for GB300's FP64 pipe, where every operation takes a warp 64 cycles of its
// scheduler (two lanes a clock and SM): the results of the plain IEEE operations, by fewer of
// them.
//
//  * comparisons, signs and minima are done on the bit patterns (some ten integer instructions
//    cost a sixth of one FP64 comparison);
//  * sums and products are issued as fused multiply-adds with a factor 1 or an addend -0, which
//    rounds alike and, measured, takes 64 cycles against 76 for an addition or a product (four
//    warps an SM);
//  * quotients by Markstein's method (Markstein, "Computation of elementary functions on the IBM
//    RISC System/6000 processor", IBM J. R&D 34, 1990): a reciprocal y of the divisor, then
//    q = a y, the exact remainder a - b q by a fused multiply-add, and q + r y, which is the
//    correctly rounded quotient.  The reciprocal starts from the FP32 one of the divisor's
//    leading 24 bits and takes one cubic step (1 - b y = e, y (1 + e + e^2)): six operations a
//    quotient against nine, and three more for each further quotient by the same divisor;
//  * square roots by the coupled iteration for sqrt and 1 / (2 sqrt) (Goldschmidt's) from the
//    FP32 reciprocal root, closed by the same exact-remainder step: six operations against nine
//    and a half.
//
// Reciprocals and roots end in an integer comparison that settles the last place: the FP64 value
// is within an ulp, so the exact integer remainder (B Y against a power of two for the
// reciprocal, A 2^k - Z^2 for the root) fits 64 bits and says whether the value, or which
// neighbour of it, is the correctly rounded one.  A quotient by a correctly rounded reciprocal is
// correctly rounded for every divisor (Markstein's theorem), so these are the IEEE results, not
// only nearly always: without the comparison roots within 2^-34 ulp of the middle of two doubles
// came out an ulp off, and so did quotients next to it by divisors just below a power of two.
// The integer instructions are ones the FP64 pipe's schedulers have to spare: 1024^2 stays at
// 27.4 ms for 20 steps (the reciprocal's last place by a Newton step under a branch instead:
// 28.2 ms); one warp alone waits for them (1024 cells, 1126 steps: 15.4 -> 15.7 ms).
// Operands outside the range where no step under- or overflows (exponents of +-400, or zero
// numerators other than a momentum or the numerator of S*) are the caller's to send to the plain
// operations.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace hydro {

// Bit patterns of the range in which the quotients and roots below are exact.
__device__ __forceinline__ bool in_range(double x) {
    return ((unsigned)__double2hiint(x) & 0x7fffffffu) - (623u << 20) < (800u << 20);
}
__device__ __forceinline__ bool is_zero(double x) {
    return ((((unsigned)__double2hiint(x)) << 1) | (unsigned)__double2loint(x)) == 0u;
}
__device__ __forceinline__ bool positive(double x) { return __double2hiint(x) >= 0; }  // sign bit
// 0 <= x, 0 < x and a < b of values that are not NaN
__device__ __forceinline__ bool ge0(double x) {
    const long long b = __double_as_longlong(x);
    return b >= 0 || b == (long long)0x8000000000000000ull;
}
__device__ __forceinline__ bool gt0(double x) { return __double_as_longlong(x) > 0; }
__device__ __forceinline__ bool less(double a, double b) {
    const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
    const long long u = x ^ ((x >> 63) & 0x7fffffffffffffffll);
    const long long v = y ^ ((y >> 63) & 0x7fffffffffffffffll);
    return u < v;
}

// Constants the compiler cannot see through (a kernel argument): x * 1 + y and x * y - 0 would
// otherwise be turned back into the addition and the product.
struct Fma64 {
    double one, mzero;  // 1 and -0
    __device__ __forceinline__ double add(double a, double b) const { return fma(a, one, b); }
    __device__ __forceinline__ double sub(double a, double b) const { return fma(-b, one, a); }
    __device__ __forceinline__ double mul(double a, double b) const { return fma(a, b, mzero); }
    // a / b with y = recip64(b); a zero numerator (of a positive divisor) keeps its sign: the
    // remainder's zero is subtracted, which leaves -0 as it is
    __device__ __forceinline__ double div(double a, double b, double y) const {
        const double q = mul(a, y);
        return fma(-fma(b, q, -a), y, q);
    }
    // the same where b < 0: there the remainder's zero has to be added
    __device__ __forceinline__ double div_by_negative(double a, double b, double y) const {
        const double q = mul(a, y);
        return fma(fma(-b, q, a), y, q);
    }
};

// 1 / b, correctly rounded, b in range.
__device__ __forceinline__ double recip64(double b) {
    const int hi = __double2hiint(b), lo = __double2loint(b);
    const float m = __int_as_float((__funnelshift_l(lo, hi, 3) & 0x7fffff) | 0x3f800000);
    float r;  // in (1/2, 1]
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(m));
    const int rb = __float_as_int(r);
    const int e = (hi >> 20) & 0x7ff;
    const int h = ((rb >> 3) + ((2 * 1023 - 127 - e) << 20)) | (hi & (int)0x80000000);
    const double y = __hiloint2double(h, rb << 29);
    const double d = fma(-b, y, 1.0);
    const long long z = __double_as_longlong(fma(y, fma(d, d, d), y));
    // B Y = 2^104 or 2^105 minus the remainder, whose low 64 bits are all of it; Y is the rounded
    // reciprocal if and only if |remainder| <= B / 2
    const unsigned long long B =
        ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)lo;
    const unsigned long long Y = ((unsigned long long)z & 0xfffffffffffffull) | 0x10000000000000ull;
    const long long R = (long long)(0ull - 2ull * (B * Y));
    return __longlong_as_double(z + (R > (long long)B) - (R < -(long long)B));
}

// sqrt(a), a > 0 in twice the range (a quotient of two values in range).
__device__ __forceinline__ double sqrt64(double a, const Fma64 &X) {
    const int hi = __double2hiint(a), lo = __double2loint(a);
    const int e = (hi >> 20) - 1023;
    const int odd = e & 1;
    const float m = __int_as_float((__funnelshift_l(lo, hi, 3) & 0x7fffff) | ((127 + odd) << 23));
    float r;  // 1 / sqrt of m in [1, 4): in (1/2, 1]
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(m));
    const int rb = __float_as_int(r);
    const int half = (e - odd) >> 1;
    const int yh = (rb >> 3) + ((1023 - 127 - half) << 20);
    const double y = __hiloint2double(yh, rb << 29);
    const double h0 = __hiloint2double(yh - (1 << 20), rb << 29);  // y / 2
    const double g0 = X.mul(a, y);
    const double d = fma(-g0, h0, 0.5);
    const double g = fma(g0, d, g0), h = fma(h0, d, h0);
    const double z = fma(fma(-g, g, a), h, g);
    // With a = A 2^(e - 52) and z = Z 2^(half - 52), z is the rounded root if and only if
    // -Z < A 2^(52 + odd) - Z^2 <= Z; the difference is small, so its low 64 bits are all of it.
    // (z = 2^half, rounded up from a mantissa of ones, is one too high by the same comparison.)
    const long long zb = __double_as_longlong(z);
    const unsigned long long Z = ((unsigned long long)zb & 0xfffffffffffffull) | 0x10000000000000ull;
    const long long R = (long long)(((unsigned long long)((unsigned)lo << (20 + odd)) << 32) - Z * Z);
    return __longlong_as_double(zb + (R > (long long)Z) - (R <= -(long long)Z));
}

}  // namespace hydro
