// pair_f64.cuh -- the float64 pair value of P2P and direct summation.
//
// GB300 issues float64 at 1/64 of the float32 rate, so these loops are bound by the number of float64
// operations per pair and by nothing else; everything that can be done on another pipe is.  CUDA's rsqrt() and
// its division cost about ten float64 operations each.  Here the seed y of 1/sqrt(s) comes from the special
// function unit (PTX rsqrt.approx.ftz.f64: about 20 bits, low word zero, so y*y is exact), and with
// e = 1 - s y^2 the binomial series gives s^(-3/2) = y^3 (1 - e)^(-3/2) = y^3 (1 + 3/2 e + 15/8 e^2 + ...)
// in six operations (seven with s^(-1/2) as well); the dropped cubic term is below 2^-53.
// Whether a pair is softened, or so close or far that y^3 would leave the range, is decided on the bits of s
// by the integer pipe.
#pragma once
#include "p2p_pair.cuh"

namespace tg {

__device__ __forceinline__ double rsqrt_seed(double s)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(s));
    return y;
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
        const double tiny = ldexp(1.0, -600), huge = ldexp(1.0, 600);
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
        const double y = rsqrt_seed(s), y2 = y * y, e = fma(-s, y2, 1.0);
        if (POT) {
            ri = fma(y, e * fma(e, 0.375, 0.5), y);
            g = ri * ri * ri;
        } else {
            const double y3 = y2 * y;
            g = fma(y3, e * fma(e, 1.875, 1.5), y3);
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
