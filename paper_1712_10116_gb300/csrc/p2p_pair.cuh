// p2p_pair.cuh -- the value of one particle pair (Sec. 2.1, Eq. 8): g = phi'(r)/r and phi of a unit mass.
#pragma once
#include "tg_common.cuh"

namespace tg {

// PTX rsqrt.approx.ftz.f32: the hardware approximate reciprocal square root with a subnormal
// argument flushed to zero.  Only used where the argument is at least eps^2 (or a squared
// distance between distinct leaves, which is larger), so the flush never applies and the
// subnormal handling of the non-flushing form is saved.
__device__ __forceinline__ float rsqrt_ftz(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

template <class T>
__device__ __forceinline__ T tg_rsqrt(T x);
// float: hardware reciprocal square root refined by one Newton step (relative error ~1e-7)
template <>
__device__ __forceinline__ float tg_rsqrt<float>(float x)
{
    const float y = rsqrtf(x);
    return y * fmaf(-0.5f * x, y * y, 1.5f);
}
template <>
__device__ __forceinline__ double tg_rsqrt<double>(double x) { return rsqrt(x); }

// pair kernel: g = phi'(r)/r and phi(r) of a unit mass, Wendland C2 (Eq. 8) or Plummer.
// For u = r/eps in [1/2, 1) the Wendland terms are evaluated in the equivalent forms
//   g = M(u)/r^3,  M(u) = 1 - (1-u)^5 (21u^3 + 15u^2 + 5u + 1)   (enclosed mass fraction),
//   phi = -(1 - (1-u)^6 (3u^2 + 3u + 1))/r,
// which avoid the cancellation of the expanded polynomial near u = 1 in float32; below u = 1/2
// the expanded (Horner) forms are well conditioned.
template <class T, int KERNEL>
__device__ __forceinline__ void pair_kernel(T r2, T eps, T eps2, T inv_eps, T inv_eps3, T &g, T &phi)
{
    if (KERNEL == TG_KERNEL_PLUMMER) {
        const T si = tg_rsqrt<T>(r2 + eps2);
        phi = -si;
        g = si * si * si;
    } else if (r2 >= eps2) {
        const T ri = tg_rsqrt<T>(r2);
        phi = -ri;
        g = ri * ri * ri;
    } else if (r2 >= T(0.25) * eps2) {
        const T ri = tg_rsqrt<T>(r2);
        const T u = r2 * ri * inv_eps, w = T(1) - u, w2 = w * w, w5 = w2 * w2 * w;
        const T mfrac = T(1) - w5 * (((T(21) * u + T(15)) * u + T(5)) * u + T(1));
        g = mfrac * ri * ri * ri;
        phi = -(T(1) - w5 * w * ((T(3) * u + T(3)) * u + T(1))) * ri;
    } else {
        const T u = sqrt(r2) * inv_eps, u2 = u * u;
        // phi = (1/eps)(3u^7 - 15u^6 + 28u^5 - 21u^4 + 7u^2 - 3); g = (1/eps^3)(21u^5 - 90u^4 + 140u^3 - 84u^2 + 14)
        phi = ((((((T(3) * u - T(15)) * u + T(28)) * u - T(21)) * u2 + T(7)) * u2) - T(3)) * inv_eps;
        g = ((((T(21) * u - T(90)) * u + T(140)) * u - T(84)) * u2 + T(14)) * inv_eps3;
    }
}

}  // namespace tg
