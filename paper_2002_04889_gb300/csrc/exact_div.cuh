// Correctly rounded FP64 division and halving for kernels bound by the FP64
// units (which issue two lane-operations per SM and cycle on this GPU).
//
// Quotients with a common divisor share its correctly rounded reciprocal
// y = RN(1/b).  With q0 = RN(a y) and the exact remainder r = a - b q0 (one fused
// multiply-add), RN(q0 + r y) is RN(a / b) (Markstein, "Computation of elementary
// functions on the IBM RISC System/6000 processor", 1990; Muller et al., "Handbook
// of Floating-Point Arithmetic", the chapter on division by fused multiply-add),
// as long as nothing underflows or overflows on the way: three operations a
// quotient.  y comes from the hardware's seed (about 2^-20), one cubic Newton
// step, y1 = y0 + y0 (e + e^2) with e = 1 - b y0, which is within one ulp, and the
// correction y1 + y1 (1 - b y1), which rounds correctly unless b's significand is
// all ones (Markstein's theorem for the reciprocal).  Divisors of that kind, and
// operands outside the ranges in which every intermediate value is normal, take
// the plain division.  The checks run on the integer units, which the FP64 kernels
// leave idle.
#pragma once

#include <cuda_runtime.h>

namespace vg {

struct Recip {
    double b, y;             // the divisor and, if ok, RN(1/b)
    bool ok;
};

__device__ __forceinline__ double rcp_seed(double b)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
    return y;
}

// |b| in [2^-300, 2^300) and b's significand not all ones.
__device__ __forceinline__ bool divisor_ok(double b)
{
    const int hi = __double2hiint(b);
    const unsigned e = ((unsigned)hi >> 20) & 0x7ffu;
    return e - 723u < 600u && !((hi & 0xfffff) == 0xfffff && __double2loint(b) == -1);
}

// |a| in [2^-600, 2^600): a / b and the remainder are then normal for a good divisor.
__device__ __forceinline__ bool dividend_ok(double a)
{
    return (((unsigned)__double2hiint(a) >> 20) & 0x7ffu) - 423u < 1200u;
}

__device__ __forceinline__ Recip recip(double b)
{
    Recip r;
    r.b = b;
    r.ok = divisor_ok(b);
    const double y0 = rcp_seed(b);
    const double e = __fma_rn(-b, y0, 1.0);
    const double y1 = __fma_rn(y0, __fma_rn(e, e, e), y0);
    r.y = __fma_rn(y1, __fma_rn(-b, y1, 1.0), y1);
    return r;
}

// The reciprocal of b given as RN(1/b) (formed once on the host).
__device__ __forceinline__ Recip recip_given(double b, double y)
{
    Recip r;
    r.b = b;
    r.y = y;
    r.ok = divisor_ok(b);
    return r;
}

// RN(1/b).
__device__ __forceinline__ double inverse(const Recip &r) { return r.ok ? r.y : 1.0 / r.b; }

// RN(a / b).
__device__ __forceinline__ double quot(double a, const Recip &r)
{
    const double q0 = a * r.y;
    const double q = __fma_rn(__fma_rn(-r.b, q0, a), r.y, q0);
    if (r.ok && dividend_ok(a)) return q;
    if (r.ok && (__double_as_longlong(a) << 1) == 0) return q0;      // +-0
    return a / r.b;
}

// x / 2 on the integer units where that is exact; 0.5 x is also RN(x / 2) there.
__device__ __forceinline__ double half_of(double x)
{
    const int hi = __double2hiint(x), lo = __double2loint(x);
    const unsigned e = ((unsigned)hi >> 20) & 0x7ffu;
    if (e - 2u < 2045u) return __hiloint2double(hi - 0x100000, lo);
    return (((unsigned)hi << 1) | (unsigned)lo) == 0u ? x : 0.5 * x;
}

// x / 2 + y / 2, each rounded once: (x + y) / 2 except where a half is not exact or the
// sum overflows, that is for sums below 2^-959 (a subnormal half may then decide a
// rounding) and at the top of the range.
__device__ __forceinline__ double half_sum(double x, double y)
{
    const double s = x + y;
    const int hi = __double2hiint(s), lo = __double2loint(s);
    const unsigned e = ((unsigned)hi >> 20) & 0x7ffu;
    const bool zero = (((unsigned)hi << 1) | (unsigned)lo) == 0u;
    if (__builtin_expect(e - 64u < 1983u || zero, 1)) return __hiloint2double(zero ? hi : hi - 0x100000, lo);
    return 0.5 * x + 0.5 * y;
}

}  // namespace vg
