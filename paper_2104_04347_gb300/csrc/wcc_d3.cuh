// wcc_d3.cuh -- FP64 arithmetic in three-register fused multiply-adds.
//
// GB300's FP64 pipe takes a warp instruction every 16 SM cycles when all
// three operands of a DFMA come from general registers, and every 19 when
// an operand is missing (DADD, DMUL) or is a constant, an immediate or a
// uniform register (measured with chains of each form, 4 to 16 warps per SM;
// the FP64 kernels' own average was 18.5).  The FP64 kernels are bound by
// that pipe, so they compute with this type: a + b is fma(a, 1, b), a b is
// fma(a, b, -0), and 1, -0 and the scheme's constants are general registers.
// Both forms round once, exactly as the addition and the product (signed
// zeros included: x + -0 is x for either zero).
//
// A constant stays in a general register only if the compiler cannot know its
// value: its bits are combined with a zero that depends on the lane and on
// a word of constant memory, with one integer operation per half (the integer
// pipe is idle here) and nothing on the FP64 pipe.
#pragma once

#include <cuda_runtime.h>

namespace wcc {

static __constant__ unsigned k_opaque_mask = 0u;

__device__ __forceinline__ unsigned opaque_zero() {
    unsigned lane;
    asm("mov.u32 %0, %%laneid;" : "=r"(lane));
    return lane & k_opaque_mask;
}

struct d3 {
    double v;
    __device__ __forceinline__ d3() {}
    // any double as a value in general registers (constants included)
    __device__ __forceinline__ explicit d3(double x) {
        const unsigned z = opaque_zero();
        v = __hiloint2double((int)((unsigned)__double2hiint(x) ^ z), (int)((unsigned)__double2loint(x) ^ z));
    }
    __device__ __forceinline__ explicit d3(float x) : d3((double)x) {}
    __device__ __forceinline__ explicit d3(int x) : d3((double)x) {}
    static __device__ __forceinline__ d3 reg(double x) {  // already in a register (a load)
        d3 r;
        r.v = x;
        return r;
    }
};

__device__ __forceinline__ d3 operator-(d3 a) { return d3::reg(-a.v); }
__device__ __forceinline__ d3 fma(d3 a, d3 b, d3 c) { return d3::reg(::fma(a.v, b.v, c.v)); }
__device__ __forceinline__ d3 operator+(d3 a, d3 b) { return d3::reg(::fma(a.v, d3(1.0).v, b.v)); }
__device__ __forceinline__ d3 operator-(d3 a, d3 b) { return d3::reg(::fma(a.v, d3(1.0).v, -b.v)); }
__device__ __forceinline__ d3 operator*(d3 a, d3 b) { return d3::reg(::fma(a.v, b.v, d3(-0.0).v)); }
__device__ __forceinline__ d3& operator+=(d3& a, d3 b) { a = a + b; return a; }
__device__ __forceinline__ d3& operator*=(d3& a, d3 b) { a = a * b; return a; }
__device__ __forceinline__ d3 fabs(d3 a) { return d3::reg(::fabs(a.v)); }

// 2 a (exact)
__device__ __forceinline__ d3 twice(d3 a) { return a + a; }

// a > 0 (false for NaN), on the integer pipe
__device__ __forceinline__ bool all_pos(d3 a) {
    const long long b = __double_as_longlong(a.v);
    return b > 0 && b <= 0x7ff0000000000000ll;
}
// NaN / Inf test on the exponent bits
__device__ __forceinline__ bool not_finite(d3 x) { return (__double2hiint(x.v) & 0x7ff00000) == 0x7ff00000; }

// Exponent field (0: zero or subnormal, 2047: infinity or NaN).
__device__ __forceinline__ int exponent_of(d3 a) { return (int)(((unsigned)__double2hiint(a.v) >> 20) & 0x7ffu); }

// Exponent between 2^-1000 and 2^1000: where the estimates below are normal
// and their residuals exact to rounding.  Everything else (zeros, infinities,
// NaN, extreme values, negative roots) takes the compiler's operations.
__device__ __forceinline__ bool mid_range(double x) {
    const unsigned e = ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;
    return e - 23u <= 2000u;
}
// Exponent between 2^-240 and 2^240: quotients of two such numbers, and of the
// quotient and a third, neither overflow nor leave an inexact remainder.
__device__ __forceinline__ bool moderate(double x) {
    const unsigned e = ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;
    return e - 783u <= 480u;
}
static __device__ __noinline__ double recip_any(double x) { return 1.0 / x; }
static __device__ __noinline__ double sqrt_any(double x) { return ::sqrt(x); }
static __device__ __noinline__ double quotient_any(double a, double b) { return a / b; }

// x with all 52 fraction bits set
__device__ __forceinline__ bool fraction_full(double x) {
    return __double2loint(x) == -1 && (__double2hiint(x) & 0xfffff) == 0xfffff;
}

// 1/x correctly rounded: the special-function unit's estimate y (about 20
// bits), one step of the cubic iteration y (1 + e + e^2), e = 1 - x y, whose
// remaining error is e^3 (2^-60), and Markstein's closing step r + r (1 - x r)
// (IBM J. Res. Dev. 34, 1990: from an r within one unit in the last place it
// gives the rounded reciprocal unless the fraction of x is all ones).
__device__ __forceinline__ d3 recip(d3 x) {
    if (mid_range(x.v) && !fraction_full(x.v)) {
        double y;
        asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x.v));
        const d3 y0 = d3::reg(y);
        const d3 e = fma(-x, y0, d3(1.0));
        const d3 r = fma(y0, fma(e, e, e), y0);
        return fma(r, fma(-x, r, d3(1.0)), r);
    }
    return d3::reg(recip_any(x.v));
}

// a / b from the rounded reciprocal rb of b: the quotient's remainder added back
// (Markstein 1990: the rounded quotient while nothing leaves the normal range).
__device__ __forceinline__ d3 quotient(d3 a, d3 b, d3 rb) {
    const d3 q = a * rb;
    return fma(fma(-q, b, a), rb, q);
}

// a / b for any operands
__device__ __forceinline__ d3 quotient(d3 a, d3 b) {
    if (moderate(a.v) && moderate(b.v)) return quotient(a, b, recip(b));
    return d3::reg(quotient_any(a.v, b.v));
}

// the limiter's weights for an exponent other than 2
__device__ __forceinline__ d3 pow_any(d3 a, double p) { return d3::reg(::pow(a.v, p)); }
__device__ __forceinline__ d3 div_any(d3 a, d3 b) { return d3::reg(a.v / b.v); }

// the neighbours of a positive normal x
__device__ __forceinline__ d3 next_above(d3 x) { return d3::reg(__longlong_as_double(__double_as_longlong(x.v) + 1)); }
__device__ __forceinline__ d3 next_below(d3 x) { return d3::reg(__longlong_as_double(__double_as_longlong(x.v) - 1)); }

// sqrt(x) correctly rounded, for a positive mid-range x, and 1/sqrt(x) to about an
// ulp in y: from the estimate y of 1/sqrt(x) (about 20 bits), h = x y, e = 1 - h y and
// (1 - e)^(-1/2) = 1 + e/2 + 3 e^2/8 + ... (the next term is below 2^-60), so that
// g = h (1 + e/2 + 3 e^2/8) is within one unit in the last place; then Tuckerman's
// test (Markstein 1990): g is the rounded root if g (g - ulp) < x <= g (g + ulp), the signs
// of both residuals being exact in one fused multiply-add each.
__device__ __forceinline__ d3 sqrt_mid(d3 x, d3& y) {
    double y_;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y_) : "d"(x.v));
    const d3 y0 = d3::reg(y_), h = x * y0;
    const d3 e = fma(-h, y0, d3(1.0));
    const d3 t = e * fma(d3(0.375), e, d3(0.5));
    y = fma(y0, t, y0);
    const d3 g = fma(h, t, h), gb = next_below(g), ga = next_above(g);
    return !all_pos(fma(-g, gb, x)) ? gb : all_pos(fma(-g, ga, x)) ? ga : g;
}
__device__ __forceinline__ bool sqrt_in_range(d3 x) { return mid_range(x.v) && __double2hiint(x.v) > 0; }

__device__ __forceinline__ d3 sqrt(d3 x) {
    if (sqrt_in_range(x)) {
        d3 y;
        return sqrt_mid(x, y);
    }
    return d3::reg(sqrt_any(x.v));
}

// c = sqrt(x) and ic = 1/c, both correctly rounded.
__device__ __forceinline__ d3 sqrt_and_recip(d3 x, d3& ic) {
    if (sqrt_in_range(x)) {
        d3 y;
        const d3 c = sqrt_mid(x, y);
        if (!fraction_full(c.v)) {
            const d3 r = fma(y, fma(-c, y, d3(1.0)), y);
            ic = fma(r, fma(-c, r, d3(1.0)), r);
            return c;
        }
    }
    const double c = sqrt_any(x.v);
    ic = d3::reg(recip_any(c));
    return d3::reg(c);
}

}  // namespace wcc
