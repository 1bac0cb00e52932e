// pair_f64.cuh -- the float64 pair value of P2P and direct summation.
//
// GB300 issues float64 at 1/64 of the float32 rate, so these loops are bound by the number of float64
// operations per pair and by nothing else: whatever the other pipes can do in less than some forty operations is
// moved there.  With y the float32 unit's 1/sqrt(s) and e = 1 - s y^2, |e| < 2^-21, the binomial series
//   s^(-3/2) = y^3 (1 - e)^(-3/2) = y^3 (1 + 3/2 e + 15/8 e^2 + ...),  s^(-1/2) = y (1 + e/2 + 3/8 e^2 + ...)
// (the dropped cubic terms are below 2^-61) takes four float64 operations for the force: e, y^3, the bracket and the
// product.  y^2 is exact and formed by an integer multiply, the e^2 term matters to 2^-11 of itself and is a
// float32 product, and the conversions are shifts.  Whether a pair is softened, or so close or far that y would
// leave float32's range, is decided on the bits of s.  (The library's rsqrt and two products: about twelve.)
// That range is 2^-120 <= s < 2^120 in the caller's units, separations of 1e-18 to 1e18; beyond it every pair takes
// the library's rsqrt, as exact but slower (a 100,003-particle kick pair's P2P: 16.6 ms, in units 2^66 times as large
// 22.2, in units 2^66 times as small 20.6).
// Measured over 2^-20 < s < 2^20: s^(-3/2) to 2.2e-16 (6.5e-17 rms), the cube of rsqrt() to 5.4e-16 (1.6e-16 rms).
#pragma once
#include "p2p_pair.cuh"

namespace tg {

// float32 bits of 1/sqrt(s) to 22 bits, 2^-120 <= s < 2^120: the low 29 mantissa bits are dropped and the exponent
// bias moved from 1023 to 127
__device__ __forceinline__ uint32_t rsqrt_seed(double s)
{
    const uint32_t hi = (uint32_t)__double2hiint(s), lo = (uint32_t)__double2loint(s);
    return __float_as_uint(rsqrt_ftz(__uint_as_float(__funnelshift_l(lo, hi - 0x38000000u, 3))));
}
// a positive float32's bits as float64 (exact; zero becomes 2^-127)
__device__ __forceinline__ double widen(uint32_t u) { return __hiloint2double((int)((u >> 3) + 0x38000000u), (int)(u << 29)); }
// the exact square of a float32 as float64: 24 x 24 bits, leading one moved to bit 52
__device__ __forceinline__ double square_exact(uint32_t u)
{
    const uint32_t m = (u & 0x7fffffu) | 0x800000u, top = u >> 23;
    const unsigned long long p = (unsigned long long)m * m;
    const uint32_t lz = (uint32_t)(p >> 47);
    const unsigned long long mant = p << (6 - lz);
    return __longlong_as_double((long long)(mant + ((unsigned long long)(2 * top + 768 + lz) << 52)));
}
// e^2 of |e| < 2^-20 in float32 (20 bits of e; e below 2^-126 counts as that)
__device__ __forceinline__ float square_small(double e)
{
    const uint32_t h = max((uint32_t)__double2hiint(e) & 0x7fffffffu, 0x38800000u);
    const float f = __uint_as_float((h - 0x38000000u) << 3);
    return f * f;
}

// constants of a launch: the range of s where the series is used
struct PairF64 {
    double eps, eps2, inv_eps, inv_eps3;
    unsigned long long lo, span;   // s is taken by the series when bits(s) - lo < span
    __device__ __forceinline__ void init(double e, bool plummer)
    {
        eps = e;
        eps2 = e * e;
        inv_eps = 1.0 / e;
        inv_eps3 = inv_eps * inv_eps * inv_eps;
        const double tiny = ldexp(1.0, -120), huge = ldexp(1.0, 120);
        const double first = (!plummer && eps2 > tiny) ? eps2 : tiny;
        lo = (unsigned long long)__double_as_longlong(first);
        const unsigned long long top = (unsigned long long)__double_as_longlong(huge);
        span = top > lo ? top - lo : 0ull;
    }
};

// Squared distance as pair_f64 takes it: with the softening added for the Plummer kernel.
template <int KERNEL>
__device__ __forceinline__ double pair_s2(double dx, double dy, double dz, const PairF64 &k)
{
    return fma(dx, dx, fma(dy, dy, KERNEL == TG_KERNEL_PLUMMER ? fma(dz, dz, k.eps2) : dz * dz));
}

// g = phi'(r)/r and ri = -phi of a unit mass (ri only with POT)
template <int KERNEL, bool POT>
__device__ __forceinline__ void pair_f64(double s, const PairF64 &k, double &g, double &ri)
{
    if ((unsigned long long)__double_as_longlong(s) - k.lo < k.span) {
        const uint32_t u = rsqrt_seed(s);
        const double y = widen(u), y2 = square_exact(u), e = fma(-s, y2, 1.0);
        const float e2 = square_small(e);
        if (POT) {
            ri = fma(y, fma(e, 0.5, widen(__float_as_uint(0.375f * e2))), y);
            g = ri * ri * ri;
        } else {
            const double y3 = y2 * y;
            g = fma(y3, fma(e, 1.5, widen(__float_as_uint(1.875f * e2))), y3);
            ri = 0.0;
        }
    } else if (KERNEL == TG_KERNEL_PLUMMER) {
        ri = rsqrt(s);
        g = ri * ri * ri;
    } else {
        double phi;
        pair_kernel<double, TG_KERNEL_WENDLAND_C2>(s, k.eps, k.eps2, k.inv_eps, k.inv_eps3, g, phi);
        ri = -phi;
    }
}

}  // namespace tg
