// Generated by gen_m2l.py -- fixed-order M2L building blocks (do not edit).
#pragma once

__device__ __forceinline__ float m2l_fma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float m2l_rsqrt(float s)
{
    const float y = rsqrtf(s);
    return y * fmaf(-0.5f * s, y * y, 1.5f);   // one Newton step
}
#ifdef __CUDACC__
__device__ __forceinline__ double m2l_fma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double m2l_rsqrt(double s) { return rsqrt(s); }
#endif

template <class T> __device__ __forceinline__ void m2l_dtensor_1(T dx, T dy, T dz, T soft2, T (&D)[4])
{
    const T s2 = m2l_fma(dx, dx, m2l_fma(dy, dy, m2l_fma(dz, dz, soft2)));
    const T si = m2l_rsqrt(s2);
    const T si2 = si * si;
    const T f0 = -si;
    const T f1 = T(-1) * f0 * si2;
    const T r_0_0 = f0;
    const T r_1_0 = f1;
    const T r_0_1 = dx * r_1_0;
    const T r_0_2 = dy * r_1_0;
    const T r_0_3 = dz * r_1_0;
    D[0] = r_0_0;
    D[1] = r_0_1;
    D[2] = r_0_2;
    D[3] = r_0_3;
}

template <class T> __device__ __forceinline__ void m2l_side_a_1(const T (&D)[4], const T *__restrict__ Ms, T rho, T (&L)[4])
{
    T rp = T(1);
    { const T m = __ldg(Ms + 0) * rp;
      L[0] = D[0] * m;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
    }
    rp *= rho;
    { const T m = -__ldg(Ms + 1) * rp;
      L[0] = m2l_fma(D[1], m, L[0]);
    }
    { const T m = -__ldg(Ms + 2) * rp;
      L[0] = m2l_fma(D[2], m, L[0]);
    }
    { const T m = -__ldg(Ms + 3) * rp;
      L[0] = m2l_fma(D[3], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_1(const T (&D)[4], const T *__restrict__ Ms, T (&L)[4])
{
    { const T m = __ldg(Ms + 0);
      L[0] = D[0] * m;
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
    }
    { const T m = __ldg(Ms + 1);
      L[0] = m2l_fma(D[1], m, L[0]);
    }
    { const T m = __ldg(Ms + 2);
      L[0] = m2l_fma(D[2], m, L[0]);
    }
    { const T m = __ldg(Ms + 3);
      L[0] = m2l_fma(D[3], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_a_forces_1(const T (&D)[4], const T *__restrict__ Ms, T rho, T (&L)[4])
{
    L[0] = T(0);
    T rp = T(1);
    { const T m = __ldg(Ms + 0) * rp;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_forces_1(const T (&D)[4], const T *__restrict__ Ms, T (&L)[4])
{
    L[0] = T(0);
    { const T m = __ldg(Ms + 0);
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
    }
}

template <class T> __device__ __forceinline__ void m2l_dtensor_2(T dx, T dy, T dz, T soft2, T (&D)[10])
{
    const T s2 = m2l_fma(dx, dx, m2l_fma(dy, dy, m2l_fma(dz, dz, soft2)));
    const T si = m2l_rsqrt(s2);
    const T si2 = si * si;
    const T f0 = -si;
    const T f1 = T(-1) * f0 * si2;
    const T f2 = T(-3) * f1 * si2;
    const T r_0_0 = f0;
    const T r_1_0 = f1;
    const T r_2_0 = f2;
    const T r_0_1 = dx * r_1_0;
    const T r_1_1 = dx * r_2_0;
    const T r_0_2 = dy * r_1_0;
    const T r_1_2 = dy * r_2_0;
    const T r_0_3 = dz * r_1_0;
    const T r_1_3 = dz * r_2_0;
    const T r_0_4 = m2l_fma(T(1), r_1_0, dx * r_1_1);
    const T r_0_5 = dx * r_1_2;
    const T r_0_6 = dx * r_1_3;
    const T r_0_7 = m2l_fma(T(1), r_1_0, dy * r_1_2);
    const T r_0_8 = dy * r_1_3;
    const T r_0_9 = m2l_fma(T(1), r_1_0, dz * r_1_3);
    D[0] = r_0_0;
    D[1] = r_0_1;
    D[2] = r_0_2;
    D[3] = r_0_3;
    D[4] = r_0_4;
    D[5] = r_0_5;
    D[6] = r_0_6;
    D[7] = r_0_7;
    D[8] = r_0_8;
    D[9] = r_0_9;
}

template <class T> __device__ __forceinline__ void m2l_side_a_2(const T (&D)[10], const T *__restrict__ Ms, T rho, T (&L)[10])
{
    T rp = T(1);
    { const T m = __ldg(Ms + 0) * rp;
      L[0] = D[0] * m;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[9] * m;
    }
    rp *= rho;
    { const T m = -__ldg(Ms + 1) * rp;
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
    }
    { const T m = -__ldg(Ms + 2) * rp;
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
    }
    { const T m = -__ldg(Ms + 3) * rp;
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
    }
    rp *= rho;
    { const T m = __ldg(Ms + 4) * rp;
      L[0] = m2l_fma(D[4], m, L[0]);
    }
    { const T m = __ldg(Ms + 5) * rp;
      L[0] = m2l_fma(D[5], m, L[0]);
    }
    { const T m = __ldg(Ms + 6) * rp;
      L[0] = m2l_fma(D[6], m, L[0]);
    }
    { const T m = __ldg(Ms + 7) * rp;
      L[0] = m2l_fma(D[7], m, L[0]);
    }
    { const T m = __ldg(Ms + 8) * rp;
      L[0] = m2l_fma(D[8], m, L[0]);
    }
    { const T m = __ldg(Ms + 9) * rp;
      L[0] = m2l_fma(D[9], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_2(const T (&D)[10], const T *__restrict__ Ms, T (&L)[10])
{
    { const T m = __ldg(Ms + 0);
      L[0] = D[0] * m;
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[9] * m;
    }
    { const T m = __ldg(Ms + 1);
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(-D[4], m, L[1]);
      L[2] = m2l_fma(-D[5], m, L[2]);
      L[3] = m2l_fma(-D[6], m, L[3]);
    }
    { const T m = __ldg(Ms + 2);
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(-D[5], m, L[1]);
      L[2] = m2l_fma(-D[7], m, L[2]);
      L[3] = m2l_fma(-D[8], m, L[3]);
    }
    { const T m = __ldg(Ms + 3);
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(-D[6], m, L[1]);
      L[2] = m2l_fma(-D[8], m, L[2]);
      L[3] = m2l_fma(-D[9], m, L[3]);
    }
    { const T m = __ldg(Ms + 4);
      L[0] = m2l_fma(D[4], m, L[0]);
    }
    { const T m = __ldg(Ms + 5);
      L[0] = m2l_fma(D[5], m, L[0]);
    }
    { const T m = __ldg(Ms + 6);
      L[0] = m2l_fma(D[6], m, L[0]);
    }
    { const T m = __ldg(Ms + 7);
      L[0] = m2l_fma(D[7], m, L[0]);
    }
    { const T m = __ldg(Ms + 8);
      L[0] = m2l_fma(D[8], m, L[0]);
    }
    { const T m = __ldg(Ms + 9);
      L[0] = m2l_fma(D[9], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_a_forces_2(const T (&D)[10], const T *__restrict__ Ms, T rho, T (&L)[10])
{
    L[0] = T(0);
    T rp = T(1);
    { const T m = __ldg(Ms + 0) * rp;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[9] * m;
    }
    rp *= rho;
    { const T m = -__ldg(Ms + 1) * rp;
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
    }
    { const T m = -__ldg(Ms + 2) * rp;
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
    }
    { const T m = -__ldg(Ms + 3) * rp;
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_forces_2(const T (&D)[10], const T *__restrict__ Ms, T (&L)[10])
{
    L[0] = T(0);
    { const T m = __ldg(Ms + 0);
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[9] * m;
    }
    { const T m = __ldg(Ms + 1);
      L[1] = m2l_fma(-D[4], m, L[1]);
      L[2] = m2l_fma(-D[5], m, L[2]);
      L[3] = m2l_fma(-D[6], m, L[3]);
    }
    { const T m = __ldg(Ms + 2);
      L[1] = m2l_fma(-D[5], m, L[1]);
      L[2] = m2l_fma(-D[7], m, L[2]);
      L[3] = m2l_fma(-D[8], m, L[3]);
    }
    { const T m = __ldg(Ms + 3);
      L[1] = m2l_fma(-D[6], m, L[1]);
      L[2] = m2l_fma(-D[8], m, L[2]);
      L[3] = m2l_fma(-D[9], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_dtensor_3(T dx, T dy, T dz, T soft2, T (&D)[20])
{
    const T s2 = m2l_fma(dx, dx, m2l_fma(dy, dy, m2l_fma(dz, dz, soft2)));
    const T si = m2l_rsqrt(s2);
    const T si2 = si * si;
    const T f0 = -si;
    const T f1 = T(-1) * f0 * si2;
    const T f2 = T(-3) * f1 * si2;
    const T f3 = T(-5) * f2 * si2;
    const T r_0_0 = f0;
    const T r_1_0 = f1;
    const T r_2_0 = f2;
    const T r_3_0 = f3;
    const T r_0_1 = dx * r_1_0;
    const T r_1_1 = dx * r_2_0;
    const T r_2_1 = dx * r_3_0;
    const T r_0_2 = dy * r_1_0;
    const T r_1_2 = dy * r_2_0;
    const T r_2_2 = dy * r_3_0;
    const T r_0_3 = dz * r_1_0;
    const T r_1_3 = dz * r_2_0;
    const T r_2_3 = dz * r_3_0;
    const T r_0_4 = m2l_fma(T(1), r_1_0, dx * r_1_1);
    const T r_1_4 = m2l_fma(T(1), r_2_0, dx * r_2_1);
    const T r_0_5 = dx * r_1_2;
    const T r_1_5 = dx * r_2_2;
    const T r_0_6 = dx * r_1_3;
    const T r_1_6 = dx * r_2_3;
    const T r_0_7 = m2l_fma(T(1), r_1_0, dy * r_1_2);
    const T r_1_7 = m2l_fma(T(1), r_2_0, dy * r_2_2);
    const T r_0_8 = dy * r_1_3;
    const T r_1_8 = dy * r_2_3;
    const T r_0_9 = m2l_fma(T(1), r_1_0, dz * r_1_3);
    const T r_1_9 = m2l_fma(T(1), r_2_0, dz * r_2_3);
    const T r_0_10 = m2l_fma(T(2), r_1_1, dx * r_1_4);
    const T r_0_11 = m2l_fma(T(1), r_1_2, dx * r_1_5);
    const T r_0_12 = m2l_fma(T(1), r_1_3, dx * r_1_6);
    const T r_0_13 = dx * r_1_7;
    const T r_0_14 = dx * r_1_8;
    const T r_0_15 = dx * r_1_9;
    const T r_0_16 = m2l_fma(T(2), r_1_2, dy * r_1_7);
    const T r_0_17 = m2l_fma(T(1), r_1_3, dy * r_1_8);
    const T r_0_18 = dy * r_1_9;
    const T r_0_19 = m2l_fma(T(2), r_1_3, dz * r_1_9);
    D[0] = r_0_0;
    D[1] = r_0_1;
    D[2] = r_0_2;
    D[3] = r_0_3;
    D[4] = r_0_4;
    D[5] = r_0_5;
    D[6] = r_0_6;
    D[7] = r_0_7;
    D[8] = r_0_8;
    D[9] = r_0_9;
    D[10] = r_0_10;
    D[11] = r_0_11;
    D[12] = r_0_12;
    D[13] = r_0_13;
    D[14] = r_0_14;
    D[15] = r_0_15;
    D[16] = r_0_16;
    D[17] = r_0_17;
    D[18] = r_0_18;
    D[19] = r_0_19;
}

template <class T> __device__ __forceinline__ void m2l_side_a_3(const T (&D)[20], const T *__restrict__ Ms, T rho, T (&L)[20])
{
    T rp = T(1);
    { const T m = __ldg(Ms + 0) * rp;
      L[0] = D[0] * m;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[9] * m;
      L[10] = D[10] * m;
      L[11] = D[11] * m;
      L[12] = D[12] * m;
      L[13] = D[13] * m;
      L[14] = D[14] * m;
      L[15] = D[15] * m;
      L[16] = D[16] * m;
      L[17] = D[17] * m;
      L[18] = D[18] * m;
      L[19] = D[19] * m;
    }
    rp *= rho;
    { const T m = -__ldg(Ms + 1) * rp;
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[15], m, L[9]);
    }
    { const T m = -__ldg(Ms + 2) * rp;
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[18], m, L[9]);
    }
    { const T m = -__ldg(Ms + 3) * rp;
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
    }
    rp *= rho;
    { const T m = __ldg(Ms + 4) * rp;
      L[0] = m2l_fma(D[4], m, L[0]);
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
    }
    { const T m = __ldg(Ms + 5) * rp;
      L[0] = m2l_fma(D[5], m, L[0]);
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
    }
    { const T m = __ldg(Ms + 6) * rp;
      L[0] = m2l_fma(D[6], m, L[0]);
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
    }
    { const T m = __ldg(Ms + 7) * rp;
      L[0] = m2l_fma(D[7], m, L[0]);
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
    }
    { const T m = __ldg(Ms + 8) * rp;
      L[0] = m2l_fma(D[8], m, L[0]);
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
    }
    { const T m = __ldg(Ms + 9) * rp;
      L[0] = m2l_fma(D[9], m, L[0]);
      L[1] = m2l_fma(D[15], m, L[1]);
      L[2] = m2l_fma(D[18], m, L[2]);
      L[3] = m2l_fma(D[19], m, L[3]);
    }
    rp *= rho;
    { const T m = -__ldg(Ms + 10) * rp;
      L[0] = m2l_fma(D[10], m, L[0]);
    }
    { const T m = -__ldg(Ms + 11) * rp;
      L[0] = m2l_fma(D[11], m, L[0]);
    }
    { const T m = -__ldg(Ms + 12) * rp;
      L[0] = m2l_fma(D[12], m, L[0]);
    }
    { const T m = -__ldg(Ms + 13) * rp;
      L[0] = m2l_fma(D[13], m, L[0]);
    }
    { const T m = -__ldg(Ms + 14) * rp;
      L[0] = m2l_fma(D[14], m, L[0]);
    }
    { const T m = -__ldg(Ms + 15) * rp;
      L[0] = m2l_fma(D[15], m, L[0]);
    }
    { const T m = -__ldg(Ms + 16) * rp;
      L[0] = m2l_fma(D[16], m, L[0]);
    }
    { const T m = -__ldg(Ms + 17) * rp;
      L[0] = m2l_fma(D[17], m, L[0]);
    }
    { const T m = -__ldg(Ms + 18) * rp;
      L[0] = m2l_fma(D[18], m, L[0]);
    }
    { const T m = -__ldg(Ms + 19) * rp;
      L[0] = m2l_fma(D[19], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_3(const T (&D)[20], const T *__restrict__ Ms, T (&L)[20])
{
    { const T m = __ldg(Ms + 0);
      L[0] = D[0] * m;
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[9] * m;
      L[10] = -D[10] * m;
      L[11] = -D[11] * m;
      L[12] = -D[12] * m;
      L[13] = -D[13] * m;
      L[14] = -D[14] * m;
      L[15] = -D[15] * m;
      L[16] = -D[16] * m;
      L[17] = -D[17] * m;
      L[18] = -D[18] * m;
      L[19] = -D[19] * m;
    }
    { const T m = __ldg(Ms + 1);
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(-D[4], m, L[1]);
      L[2] = m2l_fma(-D[5], m, L[2]);
      L[3] = m2l_fma(-D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[15], m, L[9]);
    }
    { const T m = __ldg(Ms + 2);
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(-D[5], m, L[1]);
      L[2] = m2l_fma(-D[7], m, L[2]);
      L[3] = m2l_fma(-D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[18], m, L[9]);
    }
    { const T m = __ldg(Ms + 3);
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(-D[6], m, L[1]);
      L[2] = m2l_fma(-D[8], m, L[2]);
      L[3] = m2l_fma(-D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
    }
    { const T m = __ldg(Ms + 4);
      L[0] = m2l_fma(D[4], m, L[0]);
      L[1] = m2l_fma(-D[10], m, L[1]);
      L[2] = m2l_fma(-D[11], m, L[2]);
      L[3] = m2l_fma(-D[12], m, L[3]);
    }
    { const T m = __ldg(Ms + 5);
      L[0] = m2l_fma(D[5], m, L[0]);
      L[1] = m2l_fma(-D[11], m, L[1]);
      L[2] = m2l_fma(-D[13], m, L[2]);
      L[3] = m2l_fma(-D[14], m, L[3]);
    }
    { const T m = __ldg(Ms + 6);
      L[0] = m2l_fma(D[6], m, L[0]);
      L[1] = m2l_fma(-D[12], m, L[1]);
      L[2] = m2l_fma(-D[14], m, L[2]);
      L[3] = m2l_fma(-D[15], m, L[3]);
    }
    { const T m = __ldg(Ms + 7);
      L[0] = m2l_fma(D[7], m, L[0]);
      L[1] = m2l_fma(-D[13], m, L[1]);
      L[2] = m2l_fma(-D[16], m, L[2]);
      L[3] = m2l_fma(-D[17], m, L[3]);
    }
    { const T m = __ldg(Ms + 8);
      L[0] = m2l_fma(D[8], m, L[0]);
      L[1] = m2l_fma(-D[14], m, L[1]);
      L[2] = m2l_fma(-D[17], m, L[2]);
      L[3] = m2l_fma(-D[18], m, L[3]);
    }
    { const T m = __ldg(Ms + 9);
      L[0] = m2l_fma(D[9], m, L[0]);
      L[1] = m2l_fma(-D[15], m, L[1]);
      L[2] = m2l_fma(-D[18], m, L[2]);
      L[3] = m2l_fma(-D[19], m, L[3]);
    }
    { const T m = __ldg(Ms + 10);
      L[0] = m2l_fma(D[10], m, L[0]);
    }
    { const T m = __ldg(Ms + 11);
      L[0] = m2l_fma(D[11], m, L[0]);
    }
    { const T m = __ldg(Ms + 12);
      L[0] = m2l_fma(D[12], m, L[0]);
    }
    { const T m = __ldg(Ms + 13);
      L[0] = m2l_fma(D[13], m, L[0]);
    }
    { const T m = __ldg(Ms + 14);
      L[0] = m2l_fma(D[14], m, L[0]);
    }
    { const T m = __ldg(Ms + 15);
      L[0] = m2l_fma(D[15], m, L[0]);
    }
    { const T m = __ldg(Ms + 16);
      L[0] = m2l_fma(D[16], m, L[0]);
    }
    { const T m = __ldg(Ms + 17);
      L[0] = m2l_fma(D[17], m, L[0]);
    }
    { const T m = __ldg(Ms + 18);
      L[0] = m2l_fma(D[18], m, L[0]);
    }
    { const T m = __ldg(Ms + 19);
      L[0] = m2l_fma(D[19], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_a_forces_3(const T (&D)[20], const T *__restrict__ Ms, T rho, T (&L)[20])
{
    L[0] = T(0);
    T rp = T(1);
    { const T m = __ldg(Ms + 0) * rp;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[9] * m;
      L[10] = D[10] * m;
      L[11] = D[11] * m;
      L[12] = D[12] * m;
      L[13] = D[13] * m;
      L[14] = D[14] * m;
      L[15] = D[15] * m;
      L[16] = D[16] * m;
      L[17] = D[17] * m;
      L[18] = D[18] * m;
      L[19] = D[19] * m;
    }
    rp *= rho;
    { const T m = -__ldg(Ms + 1) * rp;
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[15], m, L[9]);
    }
    { const T m = -__ldg(Ms + 2) * rp;
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[18], m, L[9]);
    }
    { const T m = -__ldg(Ms + 3) * rp;
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
    }
    rp *= rho;
    { const T m = __ldg(Ms + 4) * rp;
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
    }
    { const T m = __ldg(Ms + 5) * rp;
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
    }
    { const T m = __ldg(Ms + 6) * rp;
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
    }
    { const T m = __ldg(Ms + 7) * rp;
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
    }
    { const T m = __ldg(Ms + 8) * rp;
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
    }
    { const T m = __ldg(Ms + 9) * rp;
      L[1] = m2l_fma(D[15], m, L[1]);
      L[2] = m2l_fma(D[18], m, L[2]);
      L[3] = m2l_fma(D[19], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_forces_3(const T (&D)[20], const T *__restrict__ Ms, T (&L)[20])
{
    L[0] = T(0);
    { const T m = __ldg(Ms + 0);
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[9] * m;
      L[10] = -D[10] * m;
      L[11] = -D[11] * m;
      L[12] = -D[12] * m;
      L[13] = -D[13] * m;
      L[14] = -D[14] * m;
      L[15] = -D[15] * m;
      L[16] = -D[16] * m;
      L[17] = -D[17] * m;
      L[18] = -D[18] * m;
      L[19] = -D[19] * m;
    }
    { const T m = __ldg(Ms + 1);
      L[1] = m2l_fma(-D[4], m, L[1]);
      L[2] = m2l_fma(-D[5], m, L[2]);
      L[3] = m2l_fma(-D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[15], m, L[9]);
    }
    { const T m = __ldg(Ms + 2);
      L[1] = m2l_fma(-D[5], m, L[1]);
      L[2] = m2l_fma(-D[7], m, L[2]);
      L[3] = m2l_fma(-D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[18], m, L[9]);
    }
    { const T m = __ldg(Ms + 3);
      L[1] = m2l_fma(-D[6], m, L[1]);
      L[2] = m2l_fma(-D[8], m, L[2]);
      L[3] = m2l_fma(-D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
    }
    { const T m = __ldg(Ms + 4);
      L[1] = m2l_fma(-D[10], m, L[1]);
      L[2] = m2l_fma(-D[11], m, L[2]);
      L[3] = m2l_fma(-D[12], m, L[3]);
    }
    { const T m = __ldg(Ms + 5);
      L[1] = m2l_fma(-D[11], m, L[1]);
      L[2] = m2l_fma(-D[13], m, L[2]);
      L[3] = m2l_fma(-D[14], m, L[3]);
    }
    { const T m = __ldg(Ms + 6);
      L[1] = m2l_fma(-D[12], m, L[1]);
      L[2] = m2l_fma(-D[14], m, L[2]);
      L[3] = m2l_fma(-D[15], m, L[3]);
    }
    { const T m = __ldg(Ms + 7);
      L[1] = m2l_fma(-D[13], m, L[1]);
      L[2] = m2l_fma(-D[16], m, L[2]);
      L[3] = m2l_fma(-D[17], m, L[3]);
    }
    { const T m = __ldg(Ms + 8);
      L[1] = m2l_fma(-D[14], m, L[1]);
      L[2] = m2l_fma(-D[17], m, L[2]);
      L[3] = m2l_fma(-D[18], m, L[3]);
    }
    { const T m = __ldg(Ms + 9);
      L[1] = m2l_fma(-D[15], m, L[1]);
      L[2] = m2l_fma(-D[18], m, L[2]);
      L[3] = m2l_fma(-D[19], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_dtensor_4(T dx, T dy, T dz, T soft2, T (&D)[35])
{
    const T s2 = m2l_fma(dx, dx, m2l_fma(dy, dy, m2l_fma(dz, dz, soft2)));
    const T si = m2l_rsqrt(s2);
    const T si2 = si * si;
    const T f0 = -si;
    const T f1 = T(-1) * f0 * si2;
    const T f2 = T(-3) * f1 * si2;
    const T f3 = T(-5) * f2 * si2;
    const T f4 = T(-7) * f3 * si2;
    const T r_0_0 = f0;
    const T r_1_0 = f1;
    const T r_2_0 = f2;
    const T r_3_0 = f3;
    const T r_4_0 = f4;
    const T r_0_1 = dx * r_1_0;
    const T r_1_1 = dx * r_2_0;
    const T r_2_1 = dx * r_3_0;
    const T r_3_1 = dx * r_4_0;
    const T r_0_2 = dy * r_1_0;
    const T r_1_2 = dy * r_2_0;
    const T r_2_2 = dy * r_3_0;
    const T r_3_2 = dy * r_4_0;
    const T r_0_3 = dz * r_1_0;
    const T r_1_3 = dz * r_2_0;
    const T r_2_3 = dz * r_3_0;
    const T r_3_3 = dz * r_4_0;
    const T r_0_4 = m2l_fma(T(1), r_1_0, dx * r_1_1);
    const T r_1_4 = m2l_fma(T(1), r_2_0, dx * r_2_1);
    const T r_2_4 = m2l_fma(T(1), r_3_0, dx * r_3_1);
    const T r_0_5 = dx * r_1_2;
    const T r_1_5 = dx * r_2_2;
    const T r_2_5 = dx * r_3_2;
    const T r_0_6 = dx * r_1_3;
    const T r_1_6 = dx * r_2_3;
    const T r_2_6 = dx * r_3_3;
    const T r_0_7 = m2l_fma(T(1), r_1_0, dy * r_1_2);
    const T r_1_7 = m2l_fma(T(1), r_2_0, dy * r_2_2);
    const T r_2_7 = m2l_fma(T(1), r_3_0, dy * r_3_2);
    const T r_0_8 = dy * r_1_3;
    const T r_1_8 = dy * r_2_3;
    const T r_2_8 = dy * r_3_3;
    const T r_0_9 = m2l_fma(T(1), r_1_0, dz * r_1_3);
    const T r_1_9 = m2l_fma(T(1), r_2_0, dz * r_2_3);
    const T r_2_9 = m2l_fma(T(1), r_3_0, dz * r_3_3);
    const T r_0_10 = m2l_fma(T(2), r_1_1, dx * r_1_4);
    const T r_1_10 = m2l_fma(T(2), r_2_1, dx * r_2_4);
    const T r_0_11 = m2l_fma(T(1), r_1_2, dx * r_1_5);
    const T r_1_11 = m2l_fma(T(1), r_2_2, dx * r_2_5);
    const T r_0_12 = m2l_fma(T(1), r_1_3, dx * r_1_6);
    const T r_1_12 = m2l_fma(T(1), r_2_3, dx * r_2_6);
    const T r_0_13 = dx * r_1_7;
    const T r_1_13 = dx * r_2_7;
    const T r_0_14 = dx * r_1_8;
    const T r_1_14 = dx * r_2_8;
    const T r_0_15 = dx * r_1_9;
    const T r_1_15 = dx * r_2_9;
    const T r_0_16 = m2l_fma(T(2), r_1_2, dy * r_1_7);
    const T r_1_16 = m2l_fma(T(2), r_2_2, dy * r_2_7);
    const T r_0_17 = m2l_fma(T(1), r_1_3, dy * r_1_8);
    const T r_1_17 = m2l_fma(T(1), r_2_3, dy * r_2_8);
    const T r_0_18 = dy * r_1_9;
    const T r_1_18 = dy * r_2_9;
    const T r_0_19 = m2l_fma(T(2), r_1_3, dz * r_1_9);
    const T r_1_19 = m2l_fma(T(2), r_2_3, dz * r_2_9);
    const T r_0_20 = m2l_fma(T(3), r_1_4, dx * r_1_10);
    const T r_0_21 = m2l_fma(T(2), r_1_5, dx * r_1_11);
    const T r_0_22 = m2l_fma(T(2), r_1_6, dx * r_1_12);
    const T r_0_23 = m2l_fma(T(1), r_1_7, dx * r_1_13);
    const T r_0_24 = m2l_fma(T(1), r_1_8, dx * r_1_14);
    const T r_0_25 = m2l_fma(T(1), r_1_9, dx * r_1_15);
    const T r_0_26 = dx * r_1_16;
    const T r_0_27 = dx * r_1_17;
    const T r_0_28 = dx * r_1_18;
    const T r_0_29 = dx * r_1_19;
    const T r_0_30 = m2l_fma(T(3), r_1_7, dy * r_1_16);
    const T r_0_31 = m2l_fma(T(2), r_1_8, dy * r_1_17);
    const T r_0_32 = m2l_fma(T(1), r_1_9, dy * r_1_18);
    const T r_0_33 = dy * r_1_19;
    const T r_0_34 = m2l_fma(T(3), r_1_9, dz * r_1_19);
    D[0] = r_0_0;
    D[1] = r_0_1;
    D[2] = r_0_2;
    D[3] = r_0_3;
    D[4] = r_0_4;
    D[5] = r_0_5;
    D[6] = r_0_6;
    D[7] = r_0_7;
    D[8] = r_0_8;
    D[9] = r_0_9;
    D[10] = r_0_10;
    D[11] = r_0_11;
    D[12] = r_0_12;
    D[13] = r_0_13;
    D[14] = r_0_14;
    D[15] = r_0_15;
    D[16] = r_0_16;
    D[17] = r_0_17;
    D[18] = r_0_18;
    D[19] = r_0_19;
    D[20] = r_0_20;
    D[21] = r_0_21;
    D[22] = r_0_22;
    D[23] = r_0_23;
    D[24] = r_0_24;
    D[25] = r_0_25;
    D[26] = r_0_26;
    D[27] = r_0_27;
    D[28] = r_0_28;
    D[29] = r_0_29;
    D[30] = r_0_30;
    D[31] = r_0_31;
    D[32] = r_0_32;
    D[33] = r_0_33;
    D[34] = r_0_34;
}

template <class T> __device__ __forceinline__ void m2l_side_a_4(const T (&D)[35], const T *__restrict__ Ms, T rho, T (&L)[35])
{
    T rp = T(1);
    { const T m = __ldg(Ms + 0) * rp;
      L[0] = D[0] * m;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[9] * m;
      L[10] = D[10] * m;
      L[11] = D[11] * m;
      L[12] = D[12] * m;
      L[13] = D[13] * m;
      L[14] = D[14] * m;
      L[15] = D[15] * m;
      L[16] = D[16] * m;
      L[17] = D[17] * m;
      L[18] = D[18] * m;
      L[19] = D[19] * m;
      L[20] = D[20] * m;
      L[21] = D[21] * m;
      L[22] = D[22] * m;
      L[23] = D[23] * m;
      L[24] = D[24] * m;
      L[25] = D[25] * m;
      L[26] = D[26] * m;
      L[27] = D[27] * m;
      L[28] = D[28] * m;
      L[29] = D[29] * m;
      L[30] = D[30] * m;
      L[31] = D[31] * m;
      L[32] = D[32] * m;
      L[33] = D[33] * m;
      L[34] = D[34] * m;
    }
    rp *= rho;
    { const T m = -__ldg(Ms + 1) * rp;
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[15], m, L[9]);
      L[10] = m2l_fma(D[20], m, L[10]);
      L[11] = m2l_fma(D[21], m, L[11]);
      L[12] = m2l_fma(D[22], m, L[12]);
      L[13] = m2l_fma(D[23], m, L[13]);
      L[14] = m2l_fma(D[24], m, L[14]);
      L[15] = m2l_fma(D[25], m, L[15]);
      L[16] = m2l_fma(D[26], m, L[16]);
      L[17] = m2l_fma(D[27], m, L[17]);
      L[18] = m2l_fma(D[28], m, L[18]);
      L[19] = m2l_fma(D[29], m, L[19]);
    }
    { const T m = -__ldg(Ms + 2) * rp;
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[18], m, L[9]);
      L[10] = m2l_fma(D[21], m, L[10]);
      L[11] = m2l_fma(D[23], m, L[11]);
      L[12] = m2l_fma(D[24], m, L[12]);
      L[13] = m2l_fma(D[26], m, L[13]);
      L[14] = m2l_fma(D[27], m, L[14]);
      L[15] = m2l_fma(D[28], m, L[15]);
      L[16] = m2l_fma(D[30], m, L[16]);
      L[17] = m2l_fma(D[31], m, L[17]);
      L[18] = m2l_fma(D[32], m, L[18]);
      L[19] = m2l_fma(D[33], m, L[19]);
    }
    { const T m = -__ldg(Ms + 3) * rp;
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(D[22], m, L[10]);
      L[11] = m2l_fma(D[24], m, L[11]);
      L[12] = m2l_fma(D[25], m, L[12]);
      L[13] = m2l_fma(D[27], m, L[13]);
      L[14] = m2l_fma(D[28], m, L[14]);
      L[15] = m2l_fma(D[29], m, L[15]);
      L[16] = m2l_fma(D[31], m, L[16]);
      L[17] = m2l_fma(D[32], m, L[17]);
      L[18] = m2l_fma(D[33], m, L[18]);
      L[19] = m2l_fma(D[34], m, L[19]);
    }
    rp *= rho;
    { const T m = __ldg(Ms + 4) * rp;
      L[0] = m2l_fma(D[4], m, L[0]);
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[21], m, L[5]);
      L[6] = m2l_fma(D[22], m, L[6]);
      L[7] = m2l_fma(D[23], m, L[7]);
      L[8] = m2l_fma(D[24], m, L[8]);
      L[9] = m2l_fma(D[25], m, L[9]);
    }
    { const T m = __ldg(Ms + 5) * rp;
      L[0] = m2l_fma(D[5], m, L[0]);
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(D[28], m, L[9]);
    }
    { const T m = __ldg(Ms + 6) * rp;
      L[0] = m2l_fma(D[6], m, L[0]);
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[24], m, L[5]);
      L[6] = m2l_fma(D[25], m, L[6]);
      L[7] = m2l_fma(D[27], m, L[7]);
      L[8] = m2l_fma(D[28], m, L[8]);
      L[9] = m2l_fma(D[29], m, L[9]);
    }
    { const T m = __ldg(Ms + 7) * rp;
      L[0] = m2l_fma(D[7], m, L[0]);
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[30], m, L[7]);
      L[8] = m2l_fma(D[31], m, L[8]);
      L[9] = m2l_fma(D[32], m, L[9]);
    }
    { const T m = __ldg(Ms + 8) * rp;
      L[0] = m2l_fma(D[8], m, L[0]);
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
      L[4] = m2l_fma(D[24], m, L[4]);
      L[5] = m2l_fma(D[27], m, L[5]);
      L[6] = m2l_fma(D[28], m, L[6]);
      L[7] = m2l_fma(D[31], m, L[7]);
      L[8] = m2l_fma(D[32], m, L[8]);
      L[9] = m2l_fma(D[33], m, L[9]);
    }
    { const T m = __ldg(Ms + 9) * rp;
      L[0] = m2l_fma(D[9], m, L[0]);
      L[1] = m2l_fma(D[15], m, L[1]);
      L[2] = m2l_fma(D[18], m, L[2]);
      L[3] = m2l_fma(D[19], m, L[3]);
      L[4] = m2l_fma(D[25], m, L[4]);
      L[5] = m2l_fma(D[28], m, L[5]);
      L[6] = m2l_fma(D[29], m, L[6]);
      L[7] = m2l_fma(D[32], m, L[7]);
      L[8] = m2l_fma(D[33], m, L[8]);
      L[9] = m2l_fma(D[34], m, L[9]);
    }
    rp *= rho;
    { const T m = -__ldg(Ms + 10) * rp;
      L[0] = m2l_fma(D[10], m, L[0]);
      L[1] = m2l_fma(D[20], m, L[1]);
      L[2] = m2l_fma(D[21], m, L[2]);
      L[3] = m2l_fma(D[22], m, L[3]);
    }
    { const T m = -__ldg(Ms + 11) * rp;
      L[0] = m2l_fma(D[11], m, L[0]);
      L[1] = m2l_fma(D[21], m, L[1]);
      L[2] = m2l_fma(D[23], m, L[2]);
      L[3] = m2l_fma(D[24], m, L[3]);
    }
    { const T m = -__ldg(Ms + 12) * rp;
      L[0] = m2l_fma(D[12], m, L[0]);
      L[1] = m2l_fma(D[22], m, L[1]);
      L[2] = m2l_fma(D[24], m, L[2]);
      L[3] = m2l_fma(D[25], m, L[3]);
    }
    { const T m = -__ldg(Ms + 13) * rp;
      L[0] = m2l_fma(D[13], m, L[0]);
      L[1] = m2l_fma(D[23], m, L[1]);
      L[2] = m2l_fma(D[26], m, L[2]);
      L[3] = m2l_fma(D[27], m, L[3]);
    }
    { const T m = -__ldg(Ms + 14) * rp;
      L[0] = m2l_fma(D[14], m, L[0]);
      L[1] = m2l_fma(D[24], m, L[1]);
      L[2] = m2l_fma(D[27], m, L[2]);
      L[3] = m2l_fma(D[28], m, L[3]);
    }
    { const T m = -__ldg(Ms + 15) * rp;
      L[0] = m2l_fma(D[15], m, L[0]);
      L[1] = m2l_fma(D[25], m, L[1]);
      L[2] = m2l_fma(D[28], m, L[2]);
      L[3] = m2l_fma(D[29], m, L[3]);
    }
    { const T m = -__ldg(Ms + 16) * rp;
      L[0] = m2l_fma(D[16], m, L[0]);
      L[1] = m2l_fma(D[26], m, L[1]);
      L[2] = m2l_fma(D[30], m, L[2]);
      L[3] = m2l_fma(D[31], m, L[3]);
    }
    { const T m = -__ldg(Ms + 17) * rp;
      L[0] = m2l_fma(D[17], m, L[0]);
      L[1] = m2l_fma(D[27], m, L[1]);
      L[2] = m2l_fma(D[31], m, L[2]);
      L[3] = m2l_fma(D[32], m, L[3]);
    }
    { const T m = -__ldg(Ms + 18) * rp;
      L[0] = m2l_fma(D[18], m, L[0]);
      L[1] = m2l_fma(D[28], m, L[1]);
      L[2] = m2l_fma(D[32], m, L[2]);
      L[3] = m2l_fma(D[33], m, L[3]);
    }
    { const T m = -__ldg(Ms + 19) * rp;
      L[0] = m2l_fma(D[19], m, L[0]);
      L[1] = m2l_fma(D[29], m, L[1]);
      L[2] = m2l_fma(D[33], m, L[2]);
      L[3] = m2l_fma(D[34], m, L[3]);
    }
    rp *= rho;
    { const T m = __ldg(Ms + 20) * rp;
      L[0] = m2l_fma(D[20], m, L[0]);
    }
    { const T m = __ldg(Ms + 21) * rp;
      L[0] = m2l_fma(D[21], m, L[0]);
    }
    { const T m = __ldg(Ms + 22) * rp;
      L[0] = m2l_fma(D[22], m, L[0]);
    }
    { const T m = __ldg(Ms + 23) * rp;
      L[0] = m2l_fma(D[23], m, L[0]);
    }
    { const T m = __ldg(Ms + 24) * rp;
      L[0] = m2l_fma(D[24], m, L[0]);
    }
    { const T m = __ldg(Ms + 25) * rp;
      L[0] = m2l_fma(D[25], m, L[0]);
    }
    { const T m = __ldg(Ms + 26) * rp;
      L[0] = m2l_fma(D[26], m, L[0]);
    }
    { const T m = __ldg(Ms + 27) * rp;
      L[0] = m2l_fma(D[27], m, L[0]);
    }
    { const T m = __ldg(Ms + 28) * rp;
      L[0] = m2l_fma(D[28], m, L[0]);
    }
    { const T m = __ldg(Ms + 29) * rp;
      L[0] = m2l_fma(D[29], m, L[0]);
    }
    { const T m = __ldg(Ms + 30) * rp;
      L[0] = m2l_fma(D[30], m, L[0]);
    }
    { const T m = __ldg(Ms + 31) * rp;
      L[0] = m2l_fma(D[31], m, L[0]);
    }
    { const T m = __ldg(Ms + 32) * rp;
      L[0] = m2l_fma(D[32], m, L[0]);
    }
    { const T m = __ldg(Ms + 33) * rp;
      L[0] = m2l_fma(D[33], m, L[0]);
    }
    { const T m = __ldg(Ms + 34) * rp;
      L[0] = m2l_fma(D[34], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_4(const T (&D)[35], const T *__restrict__ Ms, T (&L)[35])
{
    { const T m = __ldg(Ms + 0);
      L[0] = D[0] * m;
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[9] * m;
      L[10] = -D[10] * m;
      L[11] = -D[11] * m;
      L[12] = -D[12] * m;
      L[13] = -D[13] * m;
      L[14] = -D[14] * m;
      L[15] = -D[15] * m;
      L[16] = -D[16] * m;
      L[17] = -D[17] * m;
      L[18] = -D[18] * m;
      L[19] = -D[19] * m;
      L[20] = D[20] * m;
      L[21] = D[21] * m;
      L[22] = D[22] * m;
      L[23] = D[23] * m;
      L[24] = D[24] * m;
      L[25] = D[25] * m;
      L[26] = D[26] * m;
      L[27] = D[27] * m;
      L[28] = D[28] * m;
      L[29] = D[29] * m;
      L[30] = D[30] * m;
      L[31] = D[31] * m;
      L[32] = D[32] * m;
      L[33] = D[33] * m;
      L[34] = D[34] * m;
    }
    { const T m = __ldg(Ms + 1);
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(-D[4], m, L[1]);
      L[2] = m2l_fma(-D[5], m, L[2]);
      L[3] = m2l_fma(-D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[15], m, L[9]);
      L[10] = m2l_fma(-D[20], m, L[10]);
      L[11] = m2l_fma(-D[21], m, L[11]);
      L[12] = m2l_fma(-D[22], m, L[12]);
      L[13] = m2l_fma(-D[23], m, L[13]);
      L[14] = m2l_fma(-D[24], m, L[14]);
      L[15] = m2l_fma(-D[25], m, L[15]);
      L[16] = m2l_fma(-D[26], m, L[16]);
      L[17] = m2l_fma(-D[27], m, L[17]);
      L[18] = m2l_fma(-D[28], m, L[18]);
      L[19] = m2l_fma(-D[29], m, L[19]);
    }
    { const T m = __ldg(Ms + 2);
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(-D[5], m, L[1]);
      L[2] = m2l_fma(-D[7], m, L[2]);
      L[3] = m2l_fma(-D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[18], m, L[9]);
      L[10] = m2l_fma(-D[21], m, L[10]);
      L[11] = m2l_fma(-D[23], m, L[11]);
      L[12] = m2l_fma(-D[24], m, L[12]);
      L[13] = m2l_fma(-D[26], m, L[13]);
      L[14] = m2l_fma(-D[27], m, L[14]);
      L[15] = m2l_fma(-D[28], m, L[15]);
      L[16] = m2l_fma(-D[30], m, L[16]);
      L[17] = m2l_fma(-D[31], m, L[17]);
      L[18] = m2l_fma(-D[32], m, L[18]);
      L[19] = m2l_fma(-D[33], m, L[19]);
    }
    { const T m = __ldg(Ms + 3);
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(-D[6], m, L[1]);
      L[2] = m2l_fma(-D[8], m, L[2]);
      L[3] = m2l_fma(-D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(-D[22], m, L[10]);
      L[11] = m2l_fma(-D[24], m, L[11]);
      L[12] = m2l_fma(-D[25], m, L[12]);
      L[13] = m2l_fma(-D[27], m, L[13]);
      L[14] = m2l_fma(-D[28], m, L[14]);
      L[15] = m2l_fma(-D[29], m, L[15]);
      L[16] = m2l_fma(-D[31], m, L[16]);
      L[17] = m2l_fma(-D[32], m, L[17]);
      L[18] = m2l_fma(-D[33], m, L[18]);
      L[19] = m2l_fma(-D[34], m, L[19]);
    }
    { const T m = __ldg(Ms + 4);
      L[0] = m2l_fma(D[4], m, L[0]);
      L[1] = m2l_fma(-D[10], m, L[1]);
      L[2] = m2l_fma(-D[11], m, L[2]);
      L[3] = m2l_fma(-D[12], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[21], m, L[5]);
      L[6] = m2l_fma(D[22], m, L[6]);
      L[7] = m2l_fma(D[23], m, L[7]);
      L[8] = m2l_fma(D[24], m, L[8]);
      L[9] = m2l_fma(D[25], m, L[9]);
    }
    { const T m = __ldg(Ms + 5);
      L[0] = m2l_fma(D[5], m, L[0]);
      L[1] = m2l_fma(-D[11], m, L[1]);
      L[2] = m2l_fma(-D[13], m, L[2]);
      L[3] = m2l_fma(-D[14], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(D[28], m, L[9]);
    }
    { const T m = __ldg(Ms + 6);
      L[0] = m2l_fma(D[6], m, L[0]);
      L[1] = m2l_fma(-D[12], m, L[1]);
      L[2] = m2l_fma(-D[14], m, L[2]);
      L[3] = m2l_fma(-D[15], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[24], m, L[5]);
      L[6] = m2l_fma(D[25], m, L[6]);
      L[7] = m2l_fma(D[27], m, L[7]);
      L[8] = m2l_fma(D[28], m, L[8]);
      L[9] = m2l_fma(D[29], m, L[9]);
    }
    { const T m = __ldg(Ms + 7);
      L[0] = m2l_fma(D[7], m, L[0]);
      L[1] = m2l_fma(-D[13], m, L[1]);
      L[2] = m2l_fma(-D[16], m, L[2]);
      L[3] = m2l_fma(-D[17], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[30], m, L[7]);
      L[8] = m2l_fma(D[31], m, L[8]);
      L[9] = m2l_fma(D[32], m, L[9]);
    }
    { const T m = __ldg(Ms + 8);
      L[0] = m2l_fma(D[8], m, L[0]);
      L[1] = m2l_fma(-D[14], m, L[1]);
      L[2] = m2l_fma(-D[17], m, L[2]);
      L[3] = m2l_fma(-D[18], m, L[3]);
      L[4] = m2l_fma(D[24], m, L[4]);
      L[5] = m2l_fma(D[27], m, L[5]);
      L[6] = m2l_fma(D[28], m, L[6]);
      L[7] = m2l_fma(D[31], m, L[7]);
      L[8] = m2l_fma(D[32], m, L[8]);
      L[9] = m2l_fma(D[33], m, L[9]);
    }
    { const T m = __ldg(Ms + 9);
      L[0] = m2l_fma(D[9], m, L[0]);
      L[1] = m2l_fma(-D[15], m, L[1]);
      L[2] = m2l_fma(-D[18], m, L[2]);
      L[3] = m2l_fma(-D[19], m, L[3]);
      L[4] = m2l_fma(D[25], m, L[4]);
      L[5] = m2l_fma(D[28], m, L[5]);
      L[6] = m2l_fma(D[29], m, L[6]);
      L[7] = m2l_fma(D[32], m, L[7]);
      L[8] = m2l_fma(D[33], m, L[8]);
      L[9] = m2l_fma(D[34], m, L[9]);
    }
    { const T m = __ldg(Ms + 10);
      L[0] = m2l_fma(D[10], m, L[0]);
      L[1] = m2l_fma(-D[20], m, L[1]);
      L[2] = m2l_fma(-D[21], m, L[2]);
      L[3] = m2l_fma(-D[22], m, L[3]);
    }
    { const T m = __ldg(Ms + 11);
      L[0] = m2l_fma(D[11], m, L[0]);
      L[1] = m2l_fma(-D[21], m, L[1]);
      L[2] = m2l_fma(-D[23], m, L[2]);
      L[3] = m2l_fma(-D[24], m, L[3]);
    }
    { const T m = __ldg(Ms + 12);
      L[0] = m2l_fma(D[12], m, L[0]);
      L[1] = m2l_fma(-D[22], m, L[1]);
      L[2] = m2l_fma(-D[24], m, L[2]);
      L[3] = m2l_fma(-D[25], m, L[3]);
    }
    { const T m = __ldg(Ms + 13);
      L[0] = m2l_fma(D[13], m, L[0]);
      L[1] = m2l_fma(-D[23], m, L[1]);
      L[2] = m2l_fma(-D[26], m, L[2]);
      L[3] = m2l_fma(-D[27], m, L[3]);
    }
    { const T m = __ldg(Ms + 14);
      L[0] = m2l_fma(D[14], m, L[0]);
      L[1] = m2l_fma(-D[24], m, L[1]);
      L[2] = m2l_fma(-D[27], m, L[2]);
      L[3] = m2l_fma(-D[28], m, L[3]);
    }
    { const T m = __ldg(Ms + 15);
      L[0] = m2l_fma(D[15], m, L[0]);
      L[1] = m2l_fma(-D[25], m, L[1]);
      L[2] = m2l_fma(-D[28], m, L[2]);
      L[3] = m2l_fma(-D[29], m, L[3]);
    }
    { const T m = __ldg(Ms + 16);
      L[0] = m2l_fma(D[16], m, L[0]);
      L[1] = m2l_fma(-D[26], m, L[1]);
      L[2] = m2l_fma(-D[30], m, L[2]);
      L[3] = m2l_fma(-D[31], m, L[3]);
    }
    { const T m = __ldg(Ms + 17);
      L[0] = m2l_fma(D[17], m, L[0]);
      L[1] = m2l_fma(-D[27], m, L[1]);
      L[2] = m2l_fma(-D[31], m, L[2]);
      L[3] = m2l_fma(-D[32], m, L[3]);
    }
    { const T m = __ldg(Ms + 18);
      L[0] = m2l_fma(D[18], m, L[0]);
      L[1] = m2l_fma(-D[28], m, L[1]);
      L[2] = m2l_fma(-D[32], m, L[2]);
      L[3] = m2l_fma(-D[33], m, L[3]);
    }
    { const T m = __ldg(Ms + 19);
      L[0] = m2l_fma(D[19], m, L[0]);
      L[1] = m2l_fma(-D[29], m, L[1]);
      L[2] = m2l_fma(-D[33], m, L[2]);
      L[3] = m2l_fma(-D[34], m, L[3]);
    }
    { const T m = __ldg(Ms + 20);
      L[0] = m2l_fma(D[20], m, L[0]);
    }
    { const T m = __ldg(Ms + 21);
      L[0] = m2l_fma(D[21], m, L[0]);
    }
    { const T m = __ldg(Ms + 22);
      L[0] = m2l_fma(D[22], m, L[0]);
    }
    { const T m = __ldg(Ms + 23);
      L[0] = m2l_fma(D[23], m, L[0]);
    }
    { const T m = __ldg(Ms + 24);
      L[0] = m2l_fma(D[24], m, L[0]);
    }
    { const T m = __ldg(Ms + 25);
      L[0] = m2l_fma(D[25], m, L[0]);
    }
    { const T m = __ldg(Ms + 26);
      L[0] = m2l_fma(D[26], m, L[0]);
    }
    { const T m = __ldg(Ms + 27);
      L[0] = m2l_fma(D[27], m, L[0]);
    }
    { const T m = __ldg(Ms + 28);
      L[0] = m2l_fma(D[28], m, L[0]);
    }
    { const T m = __ldg(Ms + 29);
      L[0] = m2l_fma(D[29], m, L[0]);
    }
    { const T m = __ldg(Ms + 30);
      L[0] = m2l_fma(D[30], m, L[0]);
    }
    { const T m = __ldg(Ms + 31);
      L[0] = m2l_fma(D[31], m, L[0]);
    }
    { const T m = __ldg(Ms + 32);
      L[0] = m2l_fma(D[32], m, L[0]);
    }
    { const T m = __ldg(Ms + 33);
      L[0] = m2l_fma(D[33], m, L[0]);
    }
    { const T m = __ldg(Ms + 34);
      L[0] = m2l_fma(D[34], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_a_forces_4(const T (&D)[35], const T *__restrict__ Ms, T rho, T (&L)[35])
{
    L[0] = T(0);
    T rp = T(1);
    { const T m = __ldg(Ms + 0) * rp;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[9] * m;
      L[10] = D[10] * m;
      L[11] = D[11] * m;
      L[12] = D[12] * m;
      L[13] = D[13] * m;
      L[14] = D[14] * m;
      L[15] = D[15] * m;
      L[16] = D[16] * m;
      L[17] = D[17] * m;
      L[18] = D[18] * m;
      L[19] = D[19] * m;
      L[20] = D[20] * m;
      L[21] = D[21] * m;
      L[22] = D[22] * m;
      L[23] = D[23] * m;
      L[24] = D[24] * m;
      L[25] = D[25] * m;
      L[26] = D[26] * m;
      L[27] = D[27] * m;
      L[28] = D[28] * m;
      L[29] = D[29] * m;
      L[30] = D[30] * m;
      L[31] = D[31] * m;
      L[32] = D[32] * m;
      L[33] = D[33] * m;
      L[34] = D[34] * m;
    }
    rp *= rho;
    { const T m = -__ldg(Ms + 1) * rp;
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[15], m, L[9]);
      L[10] = m2l_fma(D[20], m, L[10]);
      L[11] = m2l_fma(D[21], m, L[11]);
      L[12] = m2l_fma(D[22], m, L[12]);
      L[13] = m2l_fma(D[23], m, L[13]);
      L[14] = m2l_fma(D[24], m, L[14]);
      L[15] = m2l_fma(D[25], m, L[15]);
      L[16] = m2l_fma(D[26], m, L[16]);
      L[17] = m2l_fma(D[27], m, L[17]);
      L[18] = m2l_fma(D[28], m, L[18]);
      L[19] = m2l_fma(D[29], m, L[19]);
    }
    { const T m = -__ldg(Ms + 2) * rp;
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[18], m, L[9]);
      L[10] = m2l_fma(D[21], m, L[10]);
      L[11] = m2l_fma(D[23], m, L[11]);
      L[12] = m2l_fma(D[24], m, L[12]);
      L[13] = m2l_fma(D[26], m, L[13]);
      L[14] = m2l_fma(D[27], m, L[14]);
      L[15] = m2l_fma(D[28], m, L[15]);
      L[16] = m2l_fma(D[30], m, L[16]);
      L[17] = m2l_fma(D[31], m, L[17]);
      L[18] = m2l_fma(D[32], m, L[18]);
      L[19] = m2l_fma(D[33], m, L[19]);
    }
    { const T m = -__ldg(Ms + 3) * rp;
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(D[22], m, L[10]);
      L[11] = m2l_fma(D[24], m, L[11]);
      L[12] = m2l_fma(D[25], m, L[12]);
      L[13] = m2l_fma(D[27], m, L[13]);
      L[14] = m2l_fma(D[28], m, L[14]);
      L[15] = m2l_fma(D[29], m, L[15]);
      L[16] = m2l_fma(D[31], m, L[16]);
      L[17] = m2l_fma(D[32], m, L[17]);
      L[18] = m2l_fma(D[33], m, L[18]);
      L[19] = m2l_fma(D[34], m, L[19]);
    }
    rp *= rho;
    { const T m = __ldg(Ms + 4) * rp;
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[21], m, L[5]);
      L[6] = m2l_fma(D[22], m, L[6]);
      L[7] = m2l_fma(D[23], m, L[7]);
      L[8] = m2l_fma(D[24], m, L[8]);
      L[9] = m2l_fma(D[25], m, L[9]);
    }
    { const T m = __ldg(Ms + 5) * rp;
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(D[28], m, L[9]);
    }
    { const T m = __ldg(Ms + 6) * rp;
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[24], m, L[5]);
      L[6] = m2l_fma(D[25], m, L[6]);
      L[7] = m2l_fma(D[27], m, L[7]);
      L[8] = m2l_fma(D[28], m, L[8]);
      L[9] = m2l_fma(D[29], m, L[9]);
    }
    { const T m = __ldg(Ms + 7) * rp;
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[30], m, L[7]);
      L[8] = m2l_fma(D[31], m, L[8]);
      L[9] = m2l_fma(D[32], m, L[9]);
    }
    { const T m = __ldg(Ms + 8) * rp;
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
      L[4] = m2l_fma(D[24], m, L[4]);
      L[5] = m2l_fma(D[27], m, L[5]);
      L[6] = m2l_fma(D[28], m, L[6]);
      L[7] = m2l_fma(D[31], m, L[7]);
      L[8] = m2l_fma(D[32], m, L[8]);
      L[9] = m2l_fma(D[33], m, L[9]);
    }
    { const T m = __ldg(Ms + 9) * rp;
      L[1] = m2l_fma(D[15], m, L[1]);
      L[2] = m2l_fma(D[18], m, L[2]);
      L[3] = m2l_fma(D[19], m, L[3]);
      L[4] = m2l_fma(D[25], m, L[4]);
      L[5] = m2l_fma(D[28], m, L[5]);
      L[6] = m2l_fma(D[29], m, L[6]);
      L[7] = m2l_fma(D[32], m, L[7]);
      L[8] = m2l_fma(D[33], m, L[8]);
      L[9] = m2l_fma(D[34], m, L[9]);
    }
    rp *= rho;
    { const T m = -__ldg(Ms + 10) * rp;
      L[1] = m2l_fma(D[20], m, L[1]);
      L[2] = m2l_fma(D[21], m, L[2]);
      L[3] = m2l_fma(D[22], m, L[3]);
    }
    { const T m = -__ldg(Ms + 11) * rp;
      L[1] = m2l_fma(D[21], m, L[1]);
      L[2] = m2l_fma(D[23], m, L[2]);
      L[3] = m2l_fma(D[24], m, L[3]);
    }
    { const T m = -__ldg(Ms + 12) * rp;
      L[1] = m2l_fma(D[22], m, L[1]);
      L[2] = m2l_fma(D[24], m, L[2]);
      L[3] = m2l_fma(D[25], m, L[3]);
    }
    { const T m = -__ldg(Ms + 13) * rp;
      L[1] = m2l_fma(D[23], m, L[1]);
      L[2] = m2l_fma(D[26], m, L[2]);
      L[3] = m2l_fma(D[27], m, L[3]);
    }
    { const T m = -__ldg(Ms + 14) * rp;
      L[1] = m2l_fma(D[24], m, L[1]);
      L[2] = m2l_fma(D[27], m, L[2]);
      L[3] = m2l_fma(D[28], m, L[3]);
    }
    { const T m = -__ldg(Ms + 15) * rp;
      L[1] = m2l_fma(D[25], m, L[1]);
      L[2] = m2l_fma(D[28], m, L[2]);
      L[3] = m2l_fma(D[29], m, L[3]);
    }
    { const T m = -__ldg(Ms + 16) * rp;
      L[1] = m2l_fma(D[26], m, L[1]);
      L[2] = m2l_fma(D[30], m, L[2]);
      L[3] = m2l_fma(D[31], m, L[3]);
    }
    { const T m = -__ldg(Ms + 17) * rp;
      L[1] = m2l_fma(D[27], m, L[1]);
      L[2] = m2l_fma(D[31], m, L[2]);
      L[3] = m2l_fma(D[32], m, L[3]);
    }
    { const T m = -__ldg(Ms + 18) * rp;
      L[1] = m2l_fma(D[28], m, L[1]);
      L[2] = m2l_fma(D[32], m, L[2]);
      L[3] = m2l_fma(D[33], m, L[3]);
    }
    { const T m = -__ldg(Ms + 19) * rp;
      L[1] = m2l_fma(D[29], m, L[1]);
      L[2] = m2l_fma(D[33], m, L[2]);
      L[3] = m2l_fma(D[34], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_forces_4(const T (&D)[35], const T *__restrict__ Ms, T (&L)[35])
{
    L[0] = T(0);
    { const T m = __ldg(Ms + 0);
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[9] * m;
      L[10] = -D[10] * m;
      L[11] = -D[11] * m;
      L[12] = -D[12] * m;
      L[13] = -D[13] * m;
      L[14] = -D[14] * m;
      L[15] = -D[15] * m;
      L[16] = -D[16] * m;
      L[17] = -D[17] * m;
      L[18] = -D[18] * m;
      L[19] = -D[19] * m;
      L[20] = D[20] * m;
      L[21] = D[21] * m;
      L[22] = D[22] * m;
      L[23] = D[23] * m;
      L[24] = D[24] * m;
      L[25] = D[25] * m;
      L[26] = D[26] * m;
      L[27] = D[27] * m;
      L[28] = D[28] * m;
      L[29] = D[29] * m;
      L[30] = D[30] * m;
      L[31] = D[31] * m;
      L[32] = D[32] * m;
      L[33] = D[33] * m;
      L[34] = D[34] * m;
    }
    { const T m = __ldg(Ms + 1);
      L[1] = m2l_fma(-D[4], m, L[1]);
      L[2] = m2l_fma(-D[5], m, L[2]);
      L[3] = m2l_fma(-D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[15], m, L[9]);
      L[10] = m2l_fma(-D[20], m, L[10]);
      L[11] = m2l_fma(-D[21], m, L[11]);
      L[12] = m2l_fma(-D[22], m, L[12]);
      L[13] = m2l_fma(-D[23], m, L[13]);
      L[14] = m2l_fma(-D[24], m, L[14]);
      L[15] = m2l_fma(-D[25], m, L[15]);
      L[16] = m2l_fma(-D[26], m, L[16]);
      L[17] = m2l_fma(-D[27], m, L[17]);
      L[18] = m2l_fma(-D[28], m, L[18]);
      L[19] = m2l_fma(-D[29], m, L[19]);
    }
    { const T m = __ldg(Ms + 2);
      L[1] = m2l_fma(-D[5], m, L[1]);
      L[2] = m2l_fma(-D[7], m, L[2]);
      L[3] = m2l_fma(-D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[18], m, L[9]);
      L[10] = m2l_fma(-D[21], m, L[10]);
      L[11] = m2l_fma(-D[23], m, L[11]);
      L[12] = m2l_fma(-D[24], m, L[12]);
      L[13] = m2l_fma(-D[26], m, L[13]);
      L[14] = m2l_fma(-D[27], m, L[14]);
      L[15] = m2l_fma(-D[28], m, L[15]);
      L[16] = m2l_fma(-D[30], m, L[16]);
      L[17] = m2l_fma(-D[31], m, L[17]);
      L[18] = m2l_fma(-D[32], m, L[18]);
      L[19] = m2l_fma(-D[33], m, L[19]);
    }
    { const T m = __ldg(Ms + 3);
      L[1] = m2l_fma(-D[6], m, L[1]);
      L[2] = m2l_fma(-D[8], m, L[2]);
      L[3] = m2l_fma(-D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(-D[22], m, L[10]);
      L[11] = m2l_fma(-D[24], m, L[11]);
      L[12] = m2l_fma(-D[25], m, L[12]);
      L[13] = m2l_fma(-D[27], m, L[13]);
      L[14] = m2l_fma(-D[28], m, L[14]);
      L[15] = m2l_fma(-D[29], m, L[15]);
      L[16] = m2l_fma(-D[31], m, L[16]);
      L[17] = m2l_fma(-D[32], m, L[17]);
      L[18] = m2l_fma(-D[33], m, L[18]);
      L[19] = m2l_fma(-D[34], m, L[19]);
    }
    { const T m = __ldg(Ms + 4);
      L[1] = m2l_fma(-D[10], m, L[1]);
      L[2] = m2l_fma(-D[11], m, L[2]);
      L[3] = m2l_fma(-D[12], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[21], m, L[5]);
      L[6] = m2l_fma(D[22], m, L[6]);
      L[7] = m2l_fma(D[23], m, L[7]);
      L[8] = m2l_fma(D[24], m, L[8]);
      L[9] = m2l_fma(D[25], m, L[9]);
    }
    { const T m = __ldg(Ms + 5);
      L[1] = m2l_fma(-D[11], m, L[1]);
      L[2] = m2l_fma(-D[13], m, L[2]);
      L[3] = m2l_fma(-D[14], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(D[28], m, L[9]);
    }
    { const T m = __ldg(Ms + 6);
      L[1] = m2l_fma(-D[12], m, L[1]);
      L[2] = m2l_fma(-D[14], m, L[2]);
      L[3] = m2l_fma(-D[15], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[24], m, L[5]);
      L[6] = m2l_fma(D[25], m, L[6]);
      L[7] = m2l_fma(D[27], m, L[7]);
      L[8] = m2l_fma(D[28], m, L[8]);
      L[9] = m2l_fma(D[29], m, L[9]);
    }
    { const T m = __ldg(Ms + 7);
      L[1] = m2l_fma(-D[13], m, L[1]);
      L[2] = m2l_fma(-D[16], m, L[2]);
      L[3] = m2l_fma(-D[17], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[30], m, L[7]);
      L[8] = m2l_fma(D[31], m, L[8]);
      L[9] = m2l_fma(D[32], m, L[9]);
    }
    { const T m = __ldg(Ms + 8);
      L[1] = m2l_fma(-D[14], m, L[1]);
      L[2] = m2l_fma(-D[17], m, L[2]);
      L[3] = m2l_fma(-D[18], m, L[3]);
      L[4] = m2l_fma(D[24], m, L[4]);
      L[5] = m2l_fma(D[27], m, L[5]);
      L[6] = m2l_fma(D[28], m, L[6]);
      L[7] = m2l_fma(D[31], m, L[7]);
      L[8] = m2l_fma(D[32], m, L[8]);
      L[9] = m2l_fma(D[33], m, L[9]);
    }
    { const T m = __ldg(Ms + 9);
      L[1] = m2l_fma(-D[15], m, L[1]);
      L[2] = m2l_fma(-D[18], m, L[2]);
      L[3] = m2l_fma(-D[19], m, L[3]);
      L[4] = m2l_fma(D[25], m, L[4]);
      L[5] = m2l_fma(D[28], m, L[5]);
      L[6] = m2l_fma(D[29], m, L[6]);
      L[7] = m2l_fma(D[32], m, L[7]);
      L[8] = m2l_fma(D[33], m, L[8]);
      L[9] = m2l_fma(D[34], m, L[9]);
    }
    { const T m = __ldg(Ms + 10);
      L[1] = m2l_fma(-D[20], m, L[1]);
      L[2] = m2l_fma(-D[21], m, L[2]);
      L[3] = m2l_fma(-D[22], m, L[3]);
    }
    { const T m = __ldg(Ms + 11);
      L[1] = m2l_fma(-D[21], m, L[1]);
      L[2] = m2l_fma(-D[23], m, L[2]);
      L[3] = m2l_fma(-D[24], m, L[3]);
    }
    { const T m = __ldg(Ms + 12);
      L[1] = m2l_fma(-D[22], m, L[1]);
      L[2] = m2l_fma(-D[24], m, L[2]);
      L[3] = m2l_fma(-D[25], m, L[3]);
    }
    { const T m = __ldg(Ms + 13);
      L[1] = m2l_fma(-D[23], m, L[1]);
      L[2] = m2l_fma(-D[26], m, L[2]);
      L[3] = m2l_fma(-D[27], m, L[3]);
    }
    { const T m = __ldg(Ms + 14);
      L[1] = m2l_fma(-D[24], m, L[1]);
      L[2] = m2l_fma(-D[27], m, L[2]);
      L[3] = m2l_fma(-D[28], m, L[3]);
    }
    { const T m = __ldg(Ms + 15);
      L[1] = m2l_fma(-D[25], m, L[1]);
      L[2] = m2l_fma(-D[28], m, L[2]);
      L[3] = m2l_fma(-D[29], m, L[3]);
    }
    { const T m = __ldg(Ms + 16);
      L[1] = m2l_fma(-D[26], m, L[1]);
      L[2] = m2l_fma(-D[30], m, L[2]);
      L[3] = m2l_fma(-D[31], m, L[3]);
    }
    { const T m = __ldg(Ms + 17);
      L[1] = m2l_fma(-D[27], m, L[1]);
      L[2] = m2l_fma(-D[31], m, L[2]);
      L[3] = m2l_fma(-D[32], m, L[3]);
    }
    { const T m = __ldg(Ms + 18);
      L[1] = m2l_fma(-D[28], m, L[1]);
      L[2] = m2l_fma(-D[32], m, L[2]);
      L[3] = m2l_fma(-D[33], m, L[3]);
    }
    { const T m = __ldg(Ms + 19);
      L[1] = m2l_fma(-D[29], m, L[1]);
      L[2] = m2l_fma(-D[33], m, L[2]);
      L[3] = m2l_fma(-D[34], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_dtensor_5(T dx, T dy, T dz, T soft2, T (&D)[56])
{
    const T s2 = m2l_fma(dx, dx, m2l_fma(dy, dy, m2l_fma(dz, dz, soft2)));
    const T si = m2l_rsqrt(s2);
    const T si2 = si * si;
    const T f0 = -si;
    const T f1 = T(-1) * f0 * si2;
    const T f2 = T(-3) * f1 * si2;
    const T f3 = T(-5) * f2 * si2;
    const T f4 = T(-7) * f3 * si2;
    const T f5 = T(-9) * f4 * si2;
    const T r_0_0 = f0;
    const T r_1_0 = f1;
    const T r_2_0 = f2;
    const T r_3_0 = f3;
    const T r_4_0 = f4;
    const T r_5_0 = f5;
    const T r_0_1 = dx * r_1_0;
    const T r_1_1 = dx * r_2_0;
    const T r_2_1 = dx * r_3_0;
    const T r_3_1 = dx * r_4_0;
    const T r_4_1 = dx * r_5_0;
    const T r_0_2 = dy * r_1_0;
    const T r_1_2 = dy * r_2_0;
    const T r_2_2 = dy * r_3_0;
    const T r_3_2 = dy * r_4_0;
    const T r_4_2 = dy * r_5_0;
    const T r_0_3 = dz * r_1_0;
    const T r_1_3 = dz * r_2_0;
    const T r_2_3 = dz * r_3_0;
    const T r_3_3 = dz * r_4_0;
    const T r_4_3 = dz * r_5_0;
    const T r_0_4 = m2l_fma(T(1), r_1_0, dx * r_1_1);
    const T r_1_4 = m2l_fma(T(1), r_2_0, dx * r_2_1);
    const T r_2_4 = m2l_fma(T(1), r_3_0, dx * r_3_1);
    const T r_3_4 = m2l_fma(T(1), r_4_0, dx * r_4_1);
    const T r_0_5 = dx * r_1_2;
    const T r_1_5 = dx * r_2_2;
    const T r_2_5 = dx * r_3_2;
    const T r_3_5 = dx * r_4_2;
    const T r_0_6 = dx * r_1_3;
    const T r_1_6 = dx * r_2_3;
    const T r_2_6 = dx * r_3_3;
    const T r_3_6 = dx * r_4_3;
    const T r_0_7 = m2l_fma(T(1), r_1_0, dy * r_1_2);
    const T r_1_7 = m2l_fma(T(1), r_2_0, dy * r_2_2);
    const T r_2_7 = m2l_fma(T(1), r_3_0, dy * r_3_2);
    const T r_3_7 = m2l_fma(T(1), r_4_0, dy * r_4_2);
    const T r_0_8 = dy * r_1_3;
    const T r_1_8 = dy * r_2_3;
    const T r_2_8 = dy * r_3_3;
    const T r_3_8 = dy * r_4_3;
    const T r_0_9 = m2l_fma(T(1), r_1_0, dz * r_1_3);
    const T r_1_9 = m2l_fma(T(1), r_2_0, dz * r_2_3);
    const T r_2_9 = m2l_fma(T(1), r_3_0, dz * r_3_3);
    const T r_3_9 = m2l_fma(T(1), r_4_0, dz * r_4_3);
    const T r_0_10 = m2l_fma(T(2), r_1_1, dx * r_1_4);
    const T r_1_10 = m2l_fma(T(2), r_2_1, dx * r_2_4);
    const T r_2_10 = m2l_fma(T(2), r_3_1, dx * r_3_4);
    const T r_0_11 = m2l_fma(T(1), r_1_2, dx * r_1_5);
    const T r_1_11 = m2l_fma(T(1), r_2_2, dx * r_2_5);
    const T r_2_11 = m2l_fma(T(1), r_3_2, dx * r_3_5);
    const T r_0_12 = m2l_fma(T(1), r_1_3, dx * r_1_6);
    const T r_1_12 = m2l_fma(T(1), r_2_3, dx * r_2_6);
    const T r_2_12 = m2l_fma(T(1), r_3_3, dx * r_3_6);
    const T r_0_13 = dx * r_1_7;
    const T r_1_13 = dx * r_2_7;
    const T r_2_13 = dx * r_3_7;
    const T r_0_14 = dx * r_1_8;
    const T r_1_14 = dx * r_2_8;
    const T r_2_14 = dx * r_3_8;
    const T r_0_15 = dx * r_1_9;
    const T r_1_15 = dx * r_2_9;
    const T r_2_15 = dx * r_3_9;
    const T r_0_16 = m2l_fma(T(2), r_1_2, dy * r_1_7);
    const T r_1_16 = m2l_fma(T(2), r_2_2, dy * r_2_7);
    const T r_2_16 = m2l_fma(T(2), r_3_2, dy * r_3_7);
    const T r_0_17 = m2l_fma(T(1), r_1_3, dy * r_1_8);
    const T r_1_17 = m2l_fma(T(1), r_2_3, dy * r_2_8);
    const T r_2_17 = m2l_fma(T(1), r_3_3, dy * r_3_8);
    const T r_0_18 = dy * r_1_9;
    const T r_1_18 = dy * r_2_9;
    const T r_2_18 = dy * r_3_9;
    const T r_0_19 = m2l_fma(T(2), r_1_3, dz * r_1_9);
    const T r_1_19 = m2l_fma(T(2), r_2_3, dz * r_2_9);
    const T r_2_19 = m2l_fma(T(2), r_3_3, dz * r_3_9);
    const T r_0_20 = m2l_fma(T(3), r_1_4, dx * r_1_10);
    const T r_1_20 = m2l_fma(T(3), r_2_4, dx * r_2_10);
    const T r_0_21 = m2l_fma(T(2), r_1_5, dx * r_1_11);
    const T r_1_21 = m2l_fma(T(2), r_2_5, dx * r_2_11);
    const T r_0_22 = m2l_fma(T(2), r_1_6, dx * r_1_12);
    const T r_1_22 = m2l_fma(T(2), r_2_6, dx * r_2_12);
    const T r_0_23 = m2l_fma(T(1), r_1_7, dx * r_1_13);
    const T r_1_23 = m2l_fma(T(1), r_2_7, dx * r_2_13);
    const T r_0_24 = m2l_fma(T(1), r_1_8, dx * r_1_14);
    const T r_1_24 = m2l_fma(T(1), r_2_8, dx * r_2_14);
    const T r_0_25 = m2l_fma(T(1), r_1_9, dx * r_1_15);
    const T r_1_25 = m2l_fma(T(1), r_2_9, dx * r_2_15);
    const T r_0_26 = dx * r_1_16;
    const T r_1_26 = dx * r_2_16;
    const T r_0_27 = dx * r_1_17;
    const T r_1_27 = dx * r_2_17;
    const T r_0_28 = dx * r_1_18;
    const T r_1_28 = dx * r_2_18;
    const T r_0_29 = dx * r_1_19;
    const T r_1_29 = dx * r_2_19;
    const T r_0_30 = m2l_fma(T(3), r_1_7, dy * r_1_16);
    const T r_1_30 = m2l_fma(T(3), r_2_7, dy * r_2_16);
    const T r_0_31 = m2l_fma(T(2), r_1_8, dy * r_1_17);
    const T r_1_31 = m2l_fma(T(2), r_2_8, dy * r_2_17);
    const T r_0_32 = m2l_fma(T(1), r_1_9, dy * r_1_18);
    const T r_1_32 = m2l_fma(T(1), r_2_9, dy * r_2_18);
    const T r_0_33 = dy * r_1_19;
    const T r_1_33 = dy * r_2_19;
    const T r_0_34 = m2l_fma(T(3), r_1_9, dz * r_1_19);
    const T r_1_34 = m2l_fma(T(3), r_2_9, dz * r_2_19);
    const T r_0_35 = m2l_fma(T(4), r_1_10, dx * r_1_20);
    const T r_0_36 = m2l_fma(T(3), r_1_11, dx * r_1_21);
    const T r_0_37 = m2l_fma(T(3), r_1_12, dx * r_1_22);
    const T r_0_38 = m2l_fma(T(2), r_1_13, dx * r_1_23);
    const T r_0_39 = m2l_fma(T(2), r_1_14, dx * r_1_24);
    const T r_0_40 = m2l_fma(T(2), r_1_15, dx * r_1_25);
    const T r_0_41 = m2l_fma(T(1), r_1_16, dx * r_1_26);
    const T r_0_42 = m2l_fma(T(1), r_1_17, dx * r_1_27);
    const T r_0_43 = m2l_fma(T(1), r_1_18, dx * r_1_28);
    const T r_0_44 = m2l_fma(T(1), r_1_19, dx * r_1_29);
    const T r_0_45 = dx * r_1_30;
    const T r_0_46 = dx * r_1_31;
    const T r_0_47 = dx * r_1_32;
    const T r_0_48 = dx * r_1_33;
    const T r_0_49 = dx * r_1_34;
    const T r_0_50 = m2l_fma(T(4), r_1_16, dy * r_1_30);
    const T r_0_51 = m2l_fma(T(3), r_1_17, dy * r_1_31);
    const T r_0_52 = m2l_fma(T(2), r_1_18, dy * r_1_32);
    const T r_0_53 = m2l_fma(T(1), r_1_19, dy * r_1_33);
    const T r_0_54 = dy * r_1_34;
    const T r_0_55 = m2l_fma(T(4), r_1_19, dz * r_1_34);
    D[0] = r_0_0;
    D[1] = r_0_1;
    D[2] = r_0_2;
    D[3] = r_0_3;
    D[4] = r_0_4;
    D[5] = r_0_5;
    D[6] = r_0_6;
    D[7] = r_0_7;
    D[8] = r_0_8;
    D[9] = r_0_9;
    D[10] = r_0_10;
    D[11] = r_0_11;
    D[12] = r_0_12;
    D[13] = r_0_13;
    D[14] = r_0_14;
    D[15] = r_0_15;
    D[16] = r_0_16;
    D[17] = r_0_17;
    D[18] = r_0_18;
    D[19] = r_0_19;
    D[20] = r_0_20;
    D[21] = r_0_21;
    D[22] = r_0_22;
    D[23] = r_0_23;
    D[24] = r_0_24;
    D[25] = r_0_25;
    D[26] = r_0_26;
    D[27] = r_0_27;
    D[28] = r_0_28;
    D[29] = r_0_29;
    D[30] = r_0_30;
    D[31] = r_0_31;
    D[32] = r_0_32;
    D[33] = r_0_33;
    D[34] = r_0_34;
    D[35] = r_0_35;
    D[36] = r_0_36;
    D[37] = r_0_37;
    D[38] = r_0_38;
    D[39] = r_0_39;
    D[40] = r_0_40;
    D[41] = r_0_41;
    D[42] = r_0_42;
    D[43] = r_0_43;
    D[44] = r_0_44;
    D[45] = r_0_45;
    D[46] = r_0_46;
    D[47] = r_0_47;
    D[48] = r_0_48;
    D[49] = r_0_49;
    D[50] = r_0_50;
    D[51] = r_0_51;
    D[52] = r_0_52;
    D[53] = r_0_53;
    D[54] = r_0_54;
    D[55] = r_0_55;
}

template <class T> __device__ __forceinline__ void m2l_side_a_5(const T (&D)[56], const T *__restrict__ Ms, T rho, T (&L)[56])
{
    T rp = T(1);
    { const T m = __ldg(Ms + 0) * rp;
      L[0] = D[0] * m;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[9] * m;
      L[10] = D[10] * m;
      L[11] = D[11] * m;
      L[12] = D[12] * m;
      L[13] = D[13] * m;
      L[14] = D[14] * m;
      L[15] = D[15] * m;
      L[16] = D[16] * m;
      L[17] = D[17] * m;
      L[18] = D[18] * m;
      L[19] = D[19] * m;
      L[20] = D[20] * m;
      L[21] = D[21] * m;
      L[22] = D[22] * m;
      L[23] = D[23] * m;
      L[24] = D[24] * m;
      L[25] = D[25] * m;
      L[26] = D[26] * m;
      L[27] = D[27] * m;
      L[28] = D[28] * m;
      L[29] = D[29] * m;
      L[30] = D[30] * m;
      L[31] = D[31] * m;
      L[32] = D[32] * m;
      L[33] = D[33] * m;
      L[34] = D[34] * m;
      L[35] = D[35] * m;
      L[36] = D[36] * m;
      L[37] = D[37] * m;
      L[38] = D[38] * m;
      L[39] = D[39] * m;
      L[40] = D[40] * m;
      L[41] = D[41] * m;
      L[42] = D[42] * m;
      L[43] = D[43] * m;
      L[44] = D[44] * m;
      L[45] = D[45] * m;
      L[46] = D[46] * m;
      L[47] = D[47] * m;
      L[48] = D[48] * m;
      L[49] = D[49] * m;
      L[50] = D[50] * m;
      L[51] = D[51] * m;
      L[52] = D[52] * m;
      L[53] = D[53] * m;
      L[54] = D[54] * m;
      L[55] = D[55] * m;
    }
    rp *= rho;
    { const T m = -__ldg(Ms + 1) * rp;
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[15], m, L[9]);
      L[10] = m2l_fma(D[20], m, L[10]);
      L[11] = m2l_fma(D[21], m, L[11]);
      L[12] = m2l_fma(D[22], m, L[12]);
      L[13] = m2l_fma(D[23], m, L[13]);
      L[14] = m2l_fma(D[24], m, L[14]);
      L[15] = m2l_fma(D[25], m, L[15]);
      L[16] = m2l_fma(D[26], m, L[16]);
      L[17] = m2l_fma(D[27], m, L[17]);
      L[18] = m2l_fma(D[28], m, L[18]);
      L[19] = m2l_fma(D[29], m, L[19]);
      L[20] = m2l_fma(D[35], m, L[20]);
      L[21] = m2l_fma(D[36], m, L[21]);
      L[22] = m2l_fma(D[37], m, L[22]);
      L[23] = m2l_fma(D[38], m, L[23]);
      L[24] = m2l_fma(D[39], m, L[24]);
      L[25] = m2l_fma(D[40], m, L[25]);
      L[26] = m2l_fma(D[41], m, L[26]);
      L[27] = m2l_fma(D[42], m, L[27]);
      L[28] = m2l_fma(D[43], m, L[28]);
      L[29] = m2l_fma(D[44], m, L[29]);
      L[30] = m2l_fma(D[45], m, L[30]);
      L[31] = m2l_fma(D[46], m, L[31]);
      L[32] = m2l_fma(D[47], m, L[32]);
      L[33] = m2l_fma(D[48], m, L[33]);
      L[34] = m2l_fma(D[49], m, L[34]);
    }
    { const T m = -__ldg(Ms + 2) * rp;
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[18], m, L[9]);
      L[10] = m2l_fma(D[21], m, L[10]);
      L[11] = m2l_fma(D[23], m, L[11]);
      L[12] = m2l_fma(D[24], m, L[12]);
      L[13] = m2l_fma(D[26], m, L[13]);
      L[14] = m2l_fma(D[27], m, L[14]);
      L[15] = m2l_fma(D[28], m, L[15]);
      L[16] = m2l_fma(D[30], m, L[16]);
      L[17] = m2l_fma(D[31], m, L[17]);
      L[18] = m2l_fma(D[32], m, L[18]);
      L[19] = m2l_fma(D[33], m, L[19]);
      L[20] = m2l_fma(D[36], m, L[20]);
      L[21] = m2l_fma(D[38], m, L[21]);
      L[22] = m2l_fma(D[39], m, L[22]);
      L[23] = m2l_fma(D[41], m, L[23]);
      L[24] = m2l_fma(D[42], m, L[24]);
      L[25] = m2l_fma(D[43], m, L[25]);
      L[26] = m2l_fma(D[45], m, L[26]);
      L[27] = m2l_fma(D[46], m, L[27]);
      L[28] = m2l_fma(D[47], m, L[28]);
      L[29] = m2l_fma(D[48], m, L[29]);
      L[30] = m2l_fma(D[50], m, L[30]);
      L[31] = m2l_fma(D[51], m, L[31]);
      L[32] = m2l_fma(D[52], m, L[32]);
      L[33] = m2l_fma(D[53], m, L[33]);
      L[34] = m2l_fma(D[54], m, L[34]);
    }
    { const T m = -__ldg(Ms + 3) * rp;
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(D[22], m, L[10]);
      L[11] = m2l_fma(D[24], m, L[11]);
      L[12] = m2l_fma(D[25], m, L[12]);
      L[13] = m2l_fma(D[27], m, L[13]);
      L[14] = m2l_fma(D[28], m, L[14]);
      L[15] = m2l_fma(D[29], m, L[15]);
      L[16] = m2l_fma(D[31], m, L[16]);
      L[17] = m2l_fma(D[32], m, L[17]);
      L[18] = m2l_fma(D[33], m, L[18]);
      L[19] = m2l_fma(D[34], m, L[19]);
      L[20] = m2l_fma(D[37], m, L[20]);
      L[21] = m2l_fma(D[39], m, L[21]);
      L[22] = m2l_fma(D[40], m, L[22]);
      L[23] = m2l_fma(D[42], m, L[23]);
      L[24] = m2l_fma(D[43], m, L[24]);
      L[25] = m2l_fma(D[44], m, L[25]);
      L[26] = m2l_fma(D[46], m, L[26]);
      L[27] = m2l_fma(D[47], m, L[27]);
      L[28] = m2l_fma(D[48], m, L[28]);
      L[29] = m2l_fma(D[49], m, L[29]);
      L[30] = m2l_fma(D[51], m, L[30]);
      L[31] = m2l_fma(D[52], m, L[31]);
      L[32] = m2l_fma(D[53], m, L[32]);
      L[33] = m2l_fma(D[54], m, L[33]);
      L[34] = m2l_fma(D[55], m, L[34]);
    }
    rp *= rho;
    { const T m = __ldg(Ms + 4) * rp;
      L[0] = m2l_fma(D[4], m, L[0]);
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[21], m, L[5]);
      L[6] = m2l_fma(D[22], m, L[6]);
      L[7] = m2l_fma(D[23], m, L[7]);
      L[8] = m2l_fma(D[24], m, L[8]);
      L[9] = m2l_fma(D[25], m, L[9]);
      L[10] = m2l_fma(D[35], m, L[10]);
      L[11] = m2l_fma(D[36], m, L[11]);
      L[12] = m2l_fma(D[37], m, L[12]);
      L[13] = m2l_fma(D[38], m, L[13]);
      L[14] = m2l_fma(D[39], m, L[14]);
      L[15] = m2l_fma(D[40], m, L[15]);
      L[16] = m2l_fma(D[41], m, L[16]);
      L[17] = m2l_fma(D[42], m, L[17]);
      L[18] = m2l_fma(D[43], m, L[18]);
      L[19] = m2l_fma(D[44], m, L[19]);
    }
    { const T m = __ldg(Ms + 5) * rp;
      L[0] = m2l_fma(D[5], m, L[0]);
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(D[28], m, L[9]);
      L[10] = m2l_fma(D[36], m, L[10]);
      L[11] = m2l_fma(D[38], m, L[11]);
      L[12] = m2l_fma(D[39], m, L[12]);
      L[13] = m2l_fma(D[41], m, L[13]);
      L[14] = m2l_fma(D[42], m, L[14]);
      L[15] = m2l_fma(D[43], m, L[15]);
      L[16] = m2l_fma(D[45], m, L[16]);
      L[17] = m2l_fma(D[46], m, L[17]);
      L[18] = m2l_fma(D[47], m, L[18]);
      L[19] = m2l_fma(D[48], m, L[19]);
    }
    { const T m = __ldg(Ms + 6) * rp;
      L[0] = m2l_fma(D[6], m, L[0]);
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[24], m, L[5]);
      L[6] = m2l_fma(D[25], m, L[6]);
      L[7] = m2l_fma(D[27], m, L[7]);
      L[8] = m2l_fma(D[28], m, L[8]);
      L[9] = m2l_fma(D[29], m, L[9]);
      L[10] = m2l_fma(D[37], m, L[10]);
      L[11] = m2l_fma(D[39], m, L[11]);
      L[12] = m2l_fma(D[40], m, L[12]);
      L[13] = m2l_fma(D[42], m, L[13]);
      L[14] = m2l_fma(D[43], m, L[14]);
      L[15] = m2l_fma(D[44], m, L[15]);
      L[16] = m2l_fma(D[46], m, L[16]);
      L[17] = m2l_fma(D[47], m, L[17]);
      L[18] = m2l_fma(D[48], m, L[18]);
      L[19] = m2l_fma(D[49], m, L[19]);
    }
    { const T m = __ldg(Ms + 7) * rp;
      L[0] = m2l_fma(D[7], m, L[0]);
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[30], m, L[7]);
      L[8] = m2l_fma(D[31], m, L[8]);
      L[9] = m2l_fma(D[32], m, L[9]);
      L[10] = m2l_fma(D[38], m, L[10]);
      L[11] = m2l_fma(D[41], m, L[11]);
      L[12] = m2l_fma(D[42], m, L[12]);
      L[13] = m2l_fma(D[45], m, L[13]);
      L[14] = m2l_fma(D[46], m, L[14]);
      L[15] = m2l_fma(D[47], m, L[15]);
      L[16] = m2l_fma(D[50], m, L[16]);
      L[17] = m2l_fma(D[51], m, L[17]);
      L[18] = m2l_fma(D[52], m, L[18]);
      L[19] = m2l_fma(D[53], m, L[19]);
    }
    { const T m = __ldg(Ms + 8) * rp;
      L[0] = m2l_fma(D[8], m, L[0]);
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
      L[4] = m2l_fma(D[24], m, L[4]);
      L[5] = m2l_fma(D[27], m, L[5]);
      L[6] = m2l_fma(D[28], m, L[6]);
      L[7] = m2l_fma(D[31], m, L[7]);
      L[8] = m2l_fma(D[32], m, L[8]);
      L[9] = m2l_fma(D[33], m, L[9]);
      L[10] = m2l_fma(D[39], m, L[10]);
      L[11] = m2l_fma(D[42], m, L[11]);
      L[12] = m2l_fma(D[43], m, L[12]);
      L[13] = m2l_fma(D[46], m, L[13]);
      L[14] = m2l_fma(D[47], m, L[14]);
      L[15] = m2l_fma(D[48], m, L[15]);
      L[16] = m2l_fma(D[51], m, L[16]);
      L[17] = m2l_fma(D[52], m, L[17]);
      L[18] = m2l_fma(D[53], m, L[18]);
      L[19] = m2l_fma(D[54], m, L[19]);
    }
    { const T m = __ldg(Ms + 9) * rp;
      L[0] = m2l_fma(D[9], m, L[0]);
      L[1] = m2l_fma(D[15], m, L[1]);
      L[2] = m2l_fma(D[18], m, L[2]);
      L[3] = m2l_fma(D[19], m, L[3]);
      L[4] = m2l_fma(D[25], m, L[4]);
      L[5] = m2l_fma(D[28], m, L[5]);
      L[6] = m2l_fma(D[29], m, L[6]);
      L[7] = m2l_fma(D[32], m, L[7]);
      L[8] = m2l_fma(D[33], m, L[8]);
      L[9] = m2l_fma(D[34], m, L[9]);
      L[10] = m2l_fma(D[40], m, L[10]);
      L[11] = m2l_fma(D[43], m, L[11]);
      L[12] = m2l_fma(D[44], m, L[12]);
      L[13] = m2l_fma(D[47], m, L[13]);
      L[14] = m2l_fma(D[48], m, L[14]);
      L[15] = m2l_fma(D[49], m, L[15]);
      L[16] = m2l_fma(D[52], m, L[16]);
      L[17] = m2l_fma(D[53], m, L[17]);
      L[18] = m2l_fma(D[54], m, L[18]);
      L[19] = m2l_fma(D[55], m, L[19]);
    }
    rp *= rho;
    { const T m = -__ldg(Ms + 10) * rp;
      L[0] = m2l_fma(D[10], m, L[0]);
      L[1] = m2l_fma(D[20], m, L[1]);
      L[2] = m2l_fma(D[21], m, L[2]);
      L[3] = m2l_fma(D[22], m, L[3]);
      L[4] = m2l_fma(D[35], m, L[4]);
      L[5] = m2l_fma(D[36], m, L[5]);
      L[6] = m2l_fma(D[37], m, L[6]);
      L[7] = m2l_fma(D[38], m, L[7]);
      L[8] = m2l_fma(D[39], m, L[8]);
      L[9] = m2l_fma(D[40], m, L[9]);
    }
    { const T m = -__ldg(Ms + 11) * rp;
      L[0] = m2l_fma(D[11], m, L[0]);
      L[1] = m2l_fma(D[21], m, L[1]);
      L[2] = m2l_fma(D[23], m, L[2]);
      L[3] = m2l_fma(D[24], m, L[3]);
      L[4] = m2l_fma(D[36], m, L[4]);
      L[5] = m2l_fma(D[38], m, L[5]);
      L[6] = m2l_fma(D[39], m, L[6]);
      L[7] = m2l_fma(D[41], m, L[7]);
      L[8] = m2l_fma(D[42], m, L[8]);
      L[9] = m2l_fma(D[43], m, L[9]);
    }
    { const T m = -__ldg(Ms + 12) * rp;
      L[0] = m2l_fma(D[12], m, L[0]);
      L[1] = m2l_fma(D[22], m, L[1]);
      L[2] = m2l_fma(D[24], m, L[2]);
      L[3] = m2l_fma(D[25], m, L[3]);
      L[4] = m2l_fma(D[37], m, L[4]);
      L[5] = m2l_fma(D[39], m, L[5]);
      L[6] = m2l_fma(D[40], m, L[6]);
      L[7] = m2l_fma(D[42], m, L[7]);
      L[8] = m2l_fma(D[43], m, L[8]);
      L[9] = m2l_fma(D[44], m, L[9]);
    }
    { const T m = -__ldg(Ms + 13) * rp;
      L[0] = m2l_fma(D[13], m, L[0]);
      L[1] = m2l_fma(D[23], m, L[1]);
      L[2] = m2l_fma(D[26], m, L[2]);
      L[3] = m2l_fma(D[27], m, L[3]);
      L[4] = m2l_fma(D[38], m, L[4]);
      L[5] = m2l_fma(D[41], m, L[5]);
      L[6] = m2l_fma(D[42], m, L[6]);
      L[7] = m2l_fma(D[45], m, L[7]);
      L[8] = m2l_fma(D[46], m, L[8]);
      L[9] = m2l_fma(D[47], m, L[9]);
    }
    { const T m = -__ldg(Ms + 14) * rp;
      L[0] = m2l_fma(D[14], m, L[0]);
      L[1] = m2l_fma(D[24], m, L[1]);
      L[2] = m2l_fma(D[27], m, L[2]);
      L[3] = m2l_fma(D[28], m, L[3]);
      L[4] = m2l_fma(D[39], m, L[4]);
      L[5] = m2l_fma(D[42], m, L[5]);
      L[6] = m2l_fma(D[43], m, L[6]);
      L[7] = m2l_fma(D[46], m, L[7]);
      L[8] = m2l_fma(D[47], m, L[8]);
      L[9] = m2l_fma(D[48], m, L[9]);
    }
    { const T m = -__ldg(Ms + 15) * rp;
      L[0] = m2l_fma(D[15], m, L[0]);
      L[1] = m2l_fma(D[25], m, L[1]);
      L[2] = m2l_fma(D[28], m, L[2]);
      L[3] = m2l_fma(D[29], m, L[3]);
      L[4] = m2l_fma(D[40], m, L[4]);
      L[5] = m2l_fma(D[43], m, L[5]);
      L[6] = m2l_fma(D[44], m, L[6]);
      L[7] = m2l_fma(D[47], m, L[7]);
      L[8] = m2l_fma(D[48], m, L[8]);
      L[9] = m2l_fma(D[49], m, L[9]);
    }
    { const T m = -__ldg(Ms + 16) * rp;
      L[0] = m2l_fma(D[16], m, L[0]);
      L[1] = m2l_fma(D[26], m, L[1]);
      L[2] = m2l_fma(D[30], m, L[2]);
      L[3] = m2l_fma(D[31], m, L[3]);
      L[4] = m2l_fma(D[41], m, L[4]);
      L[5] = m2l_fma(D[45], m, L[5]);
      L[6] = m2l_fma(D[46], m, L[6]);
      L[7] = m2l_fma(D[50], m, L[7]);
      L[8] = m2l_fma(D[51], m, L[8]);
      L[9] = m2l_fma(D[52], m, L[9]);
    }
    { const T m = -__ldg(Ms + 17) * rp;
      L[0] = m2l_fma(D[17], m, L[0]);
      L[1] = m2l_fma(D[27], m, L[1]);
      L[2] = m2l_fma(D[31], m, L[2]);
      L[3] = m2l_fma(D[32], m, L[3]);
      L[4] = m2l_fma(D[42], m, L[4]);
      L[5] = m2l_fma(D[46], m, L[5]);
      L[6] = m2l_fma(D[47], m, L[6]);
      L[7] = m2l_fma(D[51], m, L[7]);
      L[8] = m2l_fma(D[52], m, L[8]);
      L[9] = m2l_fma(D[53], m, L[9]);
    }
    { const T m = -__ldg(Ms + 18) * rp;
      L[0] = m2l_fma(D[18], m, L[0]);
      L[1] = m2l_fma(D[28], m, L[1]);
      L[2] = m2l_fma(D[32], m, L[2]);
      L[3] = m2l_fma(D[33], m, L[3]);
      L[4] = m2l_fma(D[43], m, L[4]);
      L[5] = m2l_fma(D[47], m, L[5]);
      L[6] = m2l_fma(D[48], m, L[6]);
      L[7] = m2l_fma(D[52], m, L[7]);
      L[8] = m2l_fma(D[53], m, L[8]);
      L[9] = m2l_fma(D[54], m, L[9]);
    }
    { const T m = -__ldg(Ms + 19) * rp;
      L[0] = m2l_fma(D[19], m, L[0]);
      L[1] = m2l_fma(D[29], m, L[1]);
      L[2] = m2l_fma(D[33], m, L[2]);
      L[3] = m2l_fma(D[34], m, L[3]);
      L[4] = m2l_fma(D[44], m, L[4]);
      L[5] = m2l_fma(D[48], m, L[5]);
      L[6] = m2l_fma(D[49], m, L[6]);
      L[7] = m2l_fma(D[53], m, L[7]);
      L[8] = m2l_fma(D[54], m, L[8]);
      L[9] = m2l_fma(D[55], m, L[9]);
    }
    rp *= rho;
    { const T m = __ldg(Ms + 20) * rp;
      L[0] = m2l_fma(D[20], m, L[0]);
      L[1] = m2l_fma(D[35], m, L[1]);
      L[2] = m2l_fma(D[36], m, L[2]);
      L[3] = m2l_fma(D[37], m, L[3]);
    }
    { const T m = __ldg(Ms + 21) * rp;
      L[0] = m2l_fma(D[21], m, L[0]);
      L[1] = m2l_fma(D[36], m, L[1]);
      L[2] = m2l_fma(D[38], m, L[2]);
      L[3] = m2l_fma(D[39], m, L[3]);
    }
    { const T m = __ldg(Ms + 22) * rp;
      L[0] = m2l_fma(D[22], m, L[0]);
      L[1] = m2l_fma(D[37], m, L[1]);
      L[2] = m2l_fma(D[39], m, L[2]);
      L[3] = m2l_fma(D[40], m, L[3]);
    }
    { const T m = __ldg(Ms + 23) * rp;
      L[0] = m2l_fma(D[23], m, L[0]);
      L[1] = m2l_fma(D[38], m, L[1]);
      L[2] = m2l_fma(D[41], m, L[2]);
      L[3] = m2l_fma(D[42], m, L[3]);
    }
    { const T m = __ldg(Ms + 24) * rp;
      L[0] = m2l_fma(D[24], m, L[0]);
      L[1] = m2l_fma(D[39], m, L[1]);
      L[2] = m2l_fma(D[42], m, L[2]);
      L[3] = m2l_fma(D[43], m, L[3]);
    }
    { const T m = __ldg(Ms + 25) * rp;
      L[0] = m2l_fma(D[25], m, L[0]);
      L[1] = m2l_fma(D[40], m, L[1]);
      L[2] = m2l_fma(D[43], m, L[2]);
      L[3] = m2l_fma(D[44], m, L[3]);
    }
    { const T m = __ldg(Ms + 26) * rp;
      L[0] = m2l_fma(D[26], m, L[0]);
      L[1] = m2l_fma(D[41], m, L[1]);
      L[2] = m2l_fma(D[45], m, L[2]);
      L[3] = m2l_fma(D[46], m, L[3]);
    }
    { const T m = __ldg(Ms + 27) * rp;
      L[0] = m2l_fma(D[27], m, L[0]);
      L[1] = m2l_fma(D[42], m, L[1]);
      L[2] = m2l_fma(D[46], m, L[2]);
      L[3] = m2l_fma(D[47], m, L[3]);
    }
    { const T m = __ldg(Ms + 28) * rp;
      L[0] = m2l_fma(D[28], m, L[0]);
      L[1] = m2l_fma(D[43], m, L[1]);
      L[2] = m2l_fma(D[47], m, L[2]);
      L[3] = m2l_fma(D[48], m, L[3]);
    }
    { const T m = __ldg(Ms + 29) * rp;
      L[0] = m2l_fma(D[29], m, L[0]);
      L[1] = m2l_fma(D[44], m, L[1]);
      L[2] = m2l_fma(D[48], m, L[2]);
      L[3] = m2l_fma(D[49], m, L[3]);
    }
    { const T m = __ldg(Ms + 30) * rp;
      L[0] = m2l_fma(D[30], m, L[0]);
      L[1] = m2l_fma(D[45], m, L[1]);
      L[2] = m2l_fma(D[50], m, L[2]);
      L[3] = m2l_fma(D[51], m, L[3]);
    }
    { const T m = __ldg(Ms + 31) * rp;
      L[0] = m2l_fma(D[31], m, L[0]);
      L[1] = m2l_fma(D[46], m, L[1]);
      L[2] = m2l_fma(D[51], m, L[2]);
      L[3] = m2l_fma(D[52], m, L[3]);
    }
    { const T m = __ldg(Ms + 32) * rp;
      L[0] = m2l_fma(D[32], m, L[0]);
      L[1] = m2l_fma(D[47], m, L[1]);
      L[2] = m2l_fma(D[52], m, L[2]);
      L[3] = m2l_fma(D[53], m, L[3]);
    }
    { const T m = __ldg(Ms + 33) * rp;
      L[0] = m2l_fma(D[33], m, L[0]);
      L[1] = m2l_fma(D[48], m, L[1]);
      L[2] = m2l_fma(D[53], m, L[2]);
      L[3] = m2l_fma(D[54], m, L[3]);
    }
    { const T m = __ldg(Ms + 34) * rp;
      L[0] = m2l_fma(D[34], m, L[0]);
      L[1] = m2l_fma(D[49], m, L[1]);
      L[2] = m2l_fma(D[54], m, L[2]);
      L[3] = m2l_fma(D[55], m, L[3]);
    }
    rp *= rho;
    { const T m = -__ldg(Ms + 35) * rp;
      L[0] = m2l_fma(D[35], m, L[0]);
    }
    { const T m = -__ldg(Ms + 36) * rp;
      L[0] = m2l_fma(D[36], m, L[0]);
    }
    { const T m = -__ldg(Ms + 37) * rp;
      L[0] = m2l_fma(D[37], m, L[0]);
    }
    { const T m = -__ldg(Ms + 38) * rp;
      L[0] = m2l_fma(D[38], m, L[0]);
    }
    { const T m = -__ldg(Ms + 39) * rp;
      L[0] = m2l_fma(D[39], m, L[0]);
    }
    { const T m = -__ldg(Ms + 40) * rp;
      L[0] = m2l_fma(D[40], m, L[0]);
    }
    { const T m = -__ldg(Ms + 41) * rp;
      L[0] = m2l_fma(D[41], m, L[0]);
    }
    { const T m = -__ldg(Ms + 42) * rp;
      L[0] = m2l_fma(D[42], m, L[0]);
    }
    { const T m = -__ldg(Ms + 43) * rp;
      L[0] = m2l_fma(D[43], m, L[0]);
    }
    { const T m = -__ldg(Ms + 44) * rp;
      L[0] = m2l_fma(D[44], m, L[0]);
    }
    { const T m = -__ldg(Ms + 45) * rp;
      L[0] = m2l_fma(D[45], m, L[0]);
    }
    { const T m = -__ldg(Ms + 46) * rp;
      L[0] = m2l_fma(D[46], m, L[0]);
    }
    { const T m = -__ldg(Ms + 47) * rp;
      L[0] = m2l_fma(D[47], m, L[0]);
    }
    { const T m = -__ldg(Ms + 48) * rp;
      L[0] = m2l_fma(D[48], m, L[0]);
    }
    { const T m = -__ldg(Ms + 49) * rp;
      L[0] = m2l_fma(D[49], m, L[0]);
    }
    { const T m = -__ldg(Ms + 50) * rp;
      L[0] = m2l_fma(D[50], m, L[0]);
    }
    { const T m = -__ldg(Ms + 51) * rp;
      L[0] = m2l_fma(D[51], m, L[0]);
    }
    { const T m = -__ldg(Ms + 52) * rp;
      L[0] = m2l_fma(D[52], m, L[0]);
    }
    { const T m = -__ldg(Ms + 53) * rp;
      L[0] = m2l_fma(D[53], m, L[0]);
    }
    { const T m = -__ldg(Ms + 54) * rp;
      L[0] = m2l_fma(D[54], m, L[0]);
    }
    { const T m = -__ldg(Ms + 55) * rp;
      L[0] = m2l_fma(D[55], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_5(const T (&D)[56], const T *__restrict__ Ms, T (&L)[56])
{
    { const T m = __ldg(Ms + 0);
      L[0] = D[0] * m;
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[9] * m;
      L[10] = -D[10] * m;
      L[11] = -D[11] * m;
      L[12] = -D[12] * m;
      L[13] = -D[13] * m;
      L[14] = -D[14] * m;
      L[15] = -D[15] * m;
      L[16] = -D[16] * m;
      L[17] = -D[17] * m;
      L[18] = -D[18] * m;
      L[19] = -D[19] * m;
      L[20] = D[20] * m;
      L[21] = D[21] * m;
      L[22] = D[22] * m;
      L[23] = D[23] * m;
      L[24] = D[24] * m;
      L[25] = D[25] * m;
      L[26] = D[26] * m;
      L[27] = D[27] * m;
      L[28] = D[28] * m;
      L[29] = D[29] * m;
      L[30] = D[30] * m;
      L[31] = D[31] * m;
      L[32] = D[32] * m;
      L[33] = D[33] * m;
      L[34] = D[34] * m;
      L[35] = -D[35] * m;
      L[36] = -D[36] * m;
      L[37] = -D[37] * m;
      L[38] = -D[38] * m;
      L[39] = -D[39] * m;
      L[40] = -D[40] * m;
      L[41] = -D[41] * m;
      L[42] = -D[42] * m;
      L[43] = -D[43] * m;
      L[44] = -D[44] * m;
      L[45] = -D[45] * m;
      L[46] = -D[46] * m;
      L[47] = -D[47] * m;
      L[48] = -D[48] * m;
      L[49] = -D[49] * m;
      L[50] = -D[50] * m;
      L[51] = -D[51] * m;
      L[52] = -D[52] * m;
      L[53] = -D[53] * m;
      L[54] = -D[54] * m;
      L[55] = -D[55] * m;
    }
    { const T m = __ldg(Ms + 1);
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(-D[4], m, L[1]);
      L[2] = m2l_fma(-D[5], m, L[2]);
      L[3] = m2l_fma(-D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[15], m, L[9]);
      L[10] = m2l_fma(-D[20], m, L[10]);
      L[11] = m2l_fma(-D[21], m, L[11]);
      L[12] = m2l_fma(-D[22], m, L[12]);
      L[13] = m2l_fma(-D[23], m, L[13]);
      L[14] = m2l_fma(-D[24], m, L[14]);
      L[15] = m2l_fma(-D[25], m, L[15]);
      L[16] = m2l_fma(-D[26], m, L[16]);
      L[17] = m2l_fma(-D[27], m, L[17]);
      L[18] = m2l_fma(-D[28], m, L[18]);
      L[19] = m2l_fma(-D[29], m, L[19]);
      L[20] = m2l_fma(D[35], m, L[20]);
      L[21] = m2l_fma(D[36], m, L[21]);
      L[22] = m2l_fma(D[37], m, L[22]);
      L[23] = m2l_fma(D[38], m, L[23]);
      L[24] = m2l_fma(D[39], m, L[24]);
      L[25] = m2l_fma(D[40], m, L[25]);
      L[26] = m2l_fma(D[41], m, L[26]);
      L[27] = m2l_fma(D[42], m, L[27]);
      L[28] = m2l_fma(D[43], m, L[28]);
      L[29] = m2l_fma(D[44], m, L[29]);
      L[30] = m2l_fma(D[45], m, L[30]);
      L[31] = m2l_fma(D[46], m, L[31]);
      L[32] = m2l_fma(D[47], m, L[32]);
      L[33] = m2l_fma(D[48], m, L[33]);
      L[34] = m2l_fma(D[49], m, L[34]);
    }
    { const T m = __ldg(Ms + 2);
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(-D[5], m, L[1]);
      L[2] = m2l_fma(-D[7], m, L[2]);
      L[3] = m2l_fma(-D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[18], m, L[9]);
      L[10] = m2l_fma(-D[21], m, L[10]);
      L[11] = m2l_fma(-D[23], m, L[11]);
      L[12] = m2l_fma(-D[24], m, L[12]);
      L[13] = m2l_fma(-D[26], m, L[13]);
      L[14] = m2l_fma(-D[27], m, L[14]);
      L[15] = m2l_fma(-D[28], m, L[15]);
      L[16] = m2l_fma(-D[30], m, L[16]);
      L[17] = m2l_fma(-D[31], m, L[17]);
      L[18] = m2l_fma(-D[32], m, L[18]);
      L[19] = m2l_fma(-D[33], m, L[19]);
      L[20] = m2l_fma(D[36], m, L[20]);
      L[21] = m2l_fma(D[38], m, L[21]);
      L[22] = m2l_fma(D[39], m, L[22]);
      L[23] = m2l_fma(D[41], m, L[23]);
      L[24] = m2l_fma(D[42], m, L[24]);
      L[25] = m2l_fma(D[43], m, L[25]);
      L[26] = m2l_fma(D[45], m, L[26]);
      L[27] = m2l_fma(D[46], m, L[27]);
      L[28] = m2l_fma(D[47], m, L[28]);
      L[29] = m2l_fma(D[48], m, L[29]);
      L[30] = m2l_fma(D[50], m, L[30]);
      L[31] = m2l_fma(D[51], m, L[31]);
      L[32] = m2l_fma(D[52], m, L[32]);
      L[33] = m2l_fma(D[53], m, L[33]);
      L[34] = m2l_fma(D[54], m, L[34]);
    }
    { const T m = __ldg(Ms + 3);
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(-D[6], m, L[1]);
      L[2] = m2l_fma(-D[8], m, L[2]);
      L[3] = m2l_fma(-D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(-D[22], m, L[10]);
      L[11] = m2l_fma(-D[24], m, L[11]);
      L[12] = m2l_fma(-D[25], m, L[12]);
      L[13] = m2l_fma(-D[27], m, L[13]);
      L[14] = m2l_fma(-D[28], m, L[14]);
      L[15] = m2l_fma(-D[29], m, L[15]);
      L[16] = m2l_fma(-D[31], m, L[16]);
      L[17] = m2l_fma(-D[32], m, L[17]);
      L[18] = m2l_fma(-D[33], m, L[18]);
      L[19] = m2l_fma(-D[34], m, L[19]);
      L[20] = m2l_fma(D[37], m, L[20]);
      L[21] = m2l_fma(D[39], m, L[21]);
      L[22] = m2l_fma(D[40], m, L[22]);
      L[23] = m2l_fma(D[42], m, L[23]);
      L[24] = m2l_fma(D[43], m, L[24]);
      L[25] = m2l_fma(D[44], m, L[25]);
      L[26] = m2l_fma(D[46], m, L[26]);
      L[27] = m2l_fma(D[47], m, L[27]);
      L[28] = m2l_fma(D[48], m, L[28]);
      L[29] = m2l_fma(D[49], m, L[29]);
      L[30] = m2l_fma(D[51], m, L[30]);
      L[31] = m2l_fma(D[52], m, L[31]);
      L[32] = m2l_fma(D[53], m, L[32]);
      L[33] = m2l_fma(D[54], m, L[33]);
      L[34] = m2l_fma(D[55], m, L[34]);
    }
    { const T m = __ldg(Ms + 4);
      L[0] = m2l_fma(D[4], m, L[0]);
      L[1] = m2l_fma(-D[10], m, L[1]);
      L[2] = m2l_fma(-D[11], m, L[2]);
      L[3] = m2l_fma(-D[12], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[21], m, L[5]);
      L[6] = m2l_fma(D[22], m, L[6]);
      L[7] = m2l_fma(D[23], m, L[7]);
      L[8] = m2l_fma(D[24], m, L[8]);
      L[9] = m2l_fma(D[25], m, L[9]);
      L[10] = m2l_fma(-D[35], m, L[10]);
      L[11] = m2l_fma(-D[36], m, L[11]);
      L[12] = m2l_fma(-D[37], m, L[12]);
      L[13] = m2l_fma(-D[38], m, L[13]);
      L[14] = m2l_fma(-D[39], m, L[14]);
      L[15] = m2l_fma(-D[40], m, L[15]);
      L[16] = m2l_fma(-D[41], m, L[16]);
      L[17] = m2l_fma(-D[42], m, L[17]);
      L[18] = m2l_fma(-D[43], m, L[18]);
      L[19] = m2l_fma(-D[44], m, L[19]);
    }
    { const T m = __ldg(Ms + 5);
      L[0] = m2l_fma(D[5], m, L[0]);
      L[1] = m2l_fma(-D[11], m, L[1]);
      L[2] = m2l_fma(-D[13], m, L[2]);
      L[3] = m2l_fma(-D[14], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(D[28], m, L[9]);
      L[10] = m2l_fma(-D[36], m, L[10]);
      L[11] = m2l_fma(-D[38], m, L[11]);
      L[12] = m2l_fma(-D[39], m, L[12]);
      L[13] = m2l_fma(-D[41], m, L[13]);
      L[14] = m2l_fma(-D[42], m, L[14]);
      L[15] = m2l_fma(-D[43], m, L[15]);
      L[16] = m2l_fma(-D[45], m, L[16]);
      L[17] = m2l_fma(-D[46], m, L[17]);
      L[18] = m2l_fma(-D[47], m, L[18]);
      L[19] = m2l_fma(-D[48], m, L[19]);
    }
    { const T m = __ldg(Ms + 6);
      L[0] = m2l_fma(D[6], m, L[0]);
      L[1] = m2l_fma(-D[12], m, L[1]);
      L[2] = m2l_fma(-D[14], m, L[2]);
      L[3] = m2l_fma(-D[15], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[24], m, L[5]);
      L[6] = m2l_fma(D[25], m, L[6]);
      L[7] = m2l_fma(D[27], m, L[7]);
      L[8] = m2l_fma(D[28], m, L[8]);
      L[9] = m2l_fma(D[29], m, L[9]);
      L[10] = m2l_fma(-D[37], m, L[10]);
      L[11] = m2l_fma(-D[39], m, L[11]);
      L[12] = m2l_fma(-D[40], m, L[12]);
      L[13] = m2l_fma(-D[42], m, L[13]);
      L[14] = m2l_fma(-D[43], m, L[14]);
      L[15] = m2l_fma(-D[44], m, L[15]);
      L[16] = m2l_fma(-D[46], m, L[16]);
      L[17] = m2l_fma(-D[47], m, L[17]);
      L[18] = m2l_fma(-D[48], m, L[18]);
      L[19] = m2l_fma(-D[49], m, L[19]);
    }
    { const T m = __ldg(Ms + 7);
      L[0] = m2l_fma(D[7], m, L[0]);
      L[1] = m2l_fma(-D[13], m, L[1]);
      L[2] = m2l_fma(-D[16], m, L[2]);
      L[3] = m2l_fma(-D[17], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[30], m, L[7]);
      L[8] = m2l_fma(D[31], m, L[8]);
      L[9] = m2l_fma(D[32], m, L[9]);
      L[10] = m2l_fma(-D[38], m, L[10]);
      L[11] = m2l_fma(-D[41], m, L[11]);
      L[12] = m2l_fma(-D[42], m, L[12]);
      L[13] = m2l_fma(-D[45], m, L[13]);
      L[14] = m2l_fma(-D[46], m, L[14]);
      L[15] = m2l_fma(-D[47], m, L[15]);
      L[16] = m2l_fma(-D[50], m, L[16]);
      L[17] = m2l_fma(-D[51], m, L[17]);
      L[18] = m2l_fma(-D[52], m, L[18]);
      L[19] = m2l_fma(-D[53], m, L[19]);
    }
    { const T m = __ldg(Ms + 8);
      L[0] = m2l_fma(D[8], m, L[0]);
      L[1] = m2l_fma(-D[14], m, L[1]);
      L[2] = m2l_fma(-D[17], m, L[2]);
      L[3] = m2l_fma(-D[18], m, L[3]);
      L[4] = m2l_fma(D[24], m, L[4]);
      L[5] = m2l_fma(D[27], m, L[5]);
      L[6] = m2l_fma(D[28], m, L[6]);
      L[7] = m2l_fma(D[31], m, L[7]);
      L[8] = m2l_fma(D[32], m, L[8]);
      L[9] = m2l_fma(D[33], m, L[9]);
      L[10] = m2l_fma(-D[39], m, L[10]);
      L[11] = m2l_fma(-D[42], m, L[11]);
      L[12] = m2l_fma(-D[43], m, L[12]);
      L[13] = m2l_fma(-D[46], m, L[13]);
      L[14] = m2l_fma(-D[47], m, L[14]);
      L[15] = m2l_fma(-D[48], m, L[15]);
      L[16] = m2l_fma(-D[51], m, L[16]);
      L[17] = m2l_fma(-D[52], m, L[17]);
      L[18] = m2l_fma(-D[53], m, L[18]);
      L[19] = m2l_fma(-D[54], m, L[19]);
    }
    { const T m = __ldg(Ms + 9);
      L[0] = m2l_fma(D[9], m, L[0]);
      L[1] = m2l_fma(-D[15], m, L[1]);
      L[2] = m2l_fma(-D[18], m, L[2]);
      L[3] = m2l_fma(-D[19], m, L[3]);
      L[4] = m2l_fma(D[25], m, L[4]);
      L[5] = m2l_fma(D[28], m, L[5]);
      L[6] = m2l_fma(D[29], m, L[6]);
      L[7] = m2l_fma(D[32], m, L[7]);
      L[8] = m2l_fma(D[33], m, L[8]);
      L[9] = m2l_fma(D[34], m, L[9]);
      L[10] = m2l_fma(-D[40], m, L[10]);
      L[11] = m2l_fma(-D[43], m, L[11]);
      L[12] = m2l_fma(-D[44], m, L[12]);
      L[13] = m2l_fma(-D[47], m, L[13]);
      L[14] = m2l_fma(-D[48], m, L[14]);
      L[15] = m2l_fma(-D[49], m, L[15]);
      L[16] = m2l_fma(-D[52], m, L[16]);
      L[17] = m2l_fma(-D[53], m, L[17]);
      L[18] = m2l_fma(-D[54], m, L[18]);
      L[19] = m2l_fma(-D[55], m, L[19]);
    }
    { const T m = __ldg(Ms + 10);
      L[0] = m2l_fma(D[10], m, L[0]);
      L[1] = m2l_fma(-D[20], m, L[1]);
      L[2] = m2l_fma(-D[21], m, L[2]);
      L[3] = m2l_fma(-D[22], m, L[3]);
      L[4] = m2l_fma(D[35], m, L[4]);
      L[5] = m2l_fma(D[36], m, L[5]);
      L[6] = m2l_fma(D[37], m, L[6]);
      L[7] = m2l_fma(D[38], m, L[7]);
      L[8] = m2l_fma(D[39], m, L[8]);
      L[9] = m2l_fma(D[40], m, L[9]);
    }
    { const T m = __ldg(Ms + 11);
      L[0] = m2l_fma(D[11], m, L[0]);
      L[1] = m2l_fma(-D[21], m, L[1]);
      L[2] = m2l_fma(-D[23], m, L[2]);
      L[3] = m2l_fma(-D[24], m, L[3]);
      L[4] = m2l_fma(D[36], m, L[4]);
      L[5] = m2l_fma(D[38], m, L[5]);
      L[6] = m2l_fma(D[39], m, L[6]);
      L[7] = m2l_fma(D[41], m, L[7]);
      L[8] = m2l_fma(D[42], m, L[8]);
      L[9] = m2l_fma(D[43], m, L[9]);
    }
    { const T m = __ldg(Ms + 12);
      L[0] = m2l_fma(D[12], m, L[0]);
      L[1] = m2l_fma(-D[22], m, L[1]);
      L[2] = m2l_fma(-D[24], m, L[2]);
      L[3] = m2l_fma(-D[25], m, L[3]);
      L[4] = m2l_fma(D[37], m, L[4]);
      L[5] = m2l_fma(D[39], m, L[5]);
      L[6] = m2l_fma(D[40], m, L[6]);
      L[7] = m2l_fma(D[42], m, L[7]);
      L[8] = m2l_fma(D[43], m, L[8]);
      L[9] = m2l_fma(D[44], m, L[9]);
    }
    { const T m = __ldg(Ms + 13);
      L[0] = m2l_fma(D[13], m, L[0]);
      L[1] = m2l_fma(-D[23], m, L[1]);
      L[2] = m2l_fma(-D[26], m, L[2]);
      L[3] = m2l_fma(-D[27], m, L[3]);
      L[4] = m2l_fma(D[38], m, L[4]);
      L[5] = m2l_fma(D[41], m, L[5]);
      L[6] = m2l_fma(D[42], m, L[6]);
      L[7] = m2l_fma(D[45], m, L[7]);
      L[8] = m2l_fma(D[46], m, L[8]);
      L[9] = m2l_fma(D[47], m, L[9]);
    }
    { const T m = __ldg(Ms + 14);
      L[0] = m2l_fma(D[14], m, L[0]);
      L[1] = m2l_fma(-D[24], m, L[1]);
      L[2] = m2l_fma(-D[27], m, L[2]);
      L[3] = m2l_fma(-D[28], m, L[3]);
      L[4] = m2l_fma(D[39], m, L[4]);
      L[5] = m2l_fma(D[42], m, L[5]);
      L[6] = m2l_fma(D[43], m, L[6]);
      L[7] = m2l_fma(D[46], m, L[7]);
      L[8] = m2l_fma(D[47], m, L[8]);
      L[9] = m2l_fma(D[48], m, L[9]);
    }
    { const T m = __ldg(Ms + 15);
      L[0] = m2l_fma(D[15], m, L[0]);
      L[1] = m2l_fma(-D[25], m, L[1]);
      L[2] = m2l_fma(-D[28], m, L[2]);
      L[3] = m2l_fma(-D[29], m, L[3]);
      L[4] = m2l_fma(D[40], m, L[4]);
      L[5] = m2l_fma(D[43], m, L[5]);
      L[6] = m2l_fma(D[44], m, L[6]);
      L[7] = m2l_fma(D[47], m, L[7]);
      L[8] = m2l_fma(D[48], m, L[8]);
      L[9] = m2l_fma(D[49], m, L[9]);
    }
    { const T m = __ldg(Ms + 16);
      L[0] = m2l_fma(D[16], m, L[0]);
      L[1] = m2l_fma(-D[26], m, L[1]);
      L[2] = m2l_fma(-D[30], m, L[2]);
      L[3] = m2l_fma(-D[31], m, L[3]);
      L[4] = m2l_fma(D[41], m, L[4]);
      L[5] = m2l_fma(D[45], m, L[5]);
      L[6] = m2l_fma(D[46], m, L[6]);
      L[7] = m2l_fma(D[50], m, L[7]);
      L[8] = m2l_fma(D[51], m, L[8]);
      L[9] = m2l_fma(D[52], m, L[9]);
    }
    { const T m = __ldg(Ms + 17);
      L[0] = m2l_fma(D[17], m, L[0]);
      L[1] = m2l_fma(-D[27], m, L[1]);
      L[2] = m2l_fma(-D[31], m, L[2]);
      L[3] = m2l_fma(-D[32], m, L[3]);
      L[4] = m2l_fma(D[42], m, L[4]);
      L[5] = m2l_fma(D[46], m, L[5]);
      L[6] = m2l_fma(D[47], m, L[6]);
      L[7] = m2l_fma(D[51], m, L[7]);
      L[8] = m2l_fma(D[52], m, L[8]);
      L[9] = m2l_fma(D[53], m, L[9]);
    }
    { const T m = __ldg(Ms + 18);
      L[0] = m2l_fma(D[18], m, L[0]);
      L[1] = m2l_fma(-D[28], m, L[1]);
      L[2] = m2l_fma(-D[32], m, L[2]);
      L[3] = m2l_fma(-D[33], m, L[3]);
      L[4] = m2l_fma(D[43], m, L[4]);
      L[5] = m2l_fma(D[47], m, L[5]);
      L[6] = m2l_fma(D[48], m, L[6]);
      L[7] = m2l_fma(D[52], m, L[7]);
      L[8] = m2l_fma(D[53], m, L[8]);
      L[9] = m2l_fma(D[54], m, L[9]);
    }
    { const T m = __ldg(Ms + 19);
      L[0] = m2l_fma(D[19], m, L[0]);
      L[1] = m2l_fma(-D[29], m, L[1]);
      L[2] = m2l_fma(-D[33], m, L[2]);
      L[3] = m2l_fma(-D[34], m, L[3]);
      L[4] = m2l_fma(D[44], m, L[4]);
      L[5] = m2l_fma(D[48], m, L[5]);
      L[6] = m2l_fma(D[49], m, L[6]);
      L[7] = m2l_fma(D[53], m, L[7]);
      L[8] = m2l_fma(D[54], m, L[8]);
      L[9] = m2l_fma(D[55], m, L[9]);
    }
    { const T m = __ldg(Ms + 20);
      L[0] = m2l_fma(D[20], m, L[0]);
      L[1] = m2l_fma(-D[35], m, L[1]);
      L[2] = m2l_fma(-D[36], m, L[2]);
      L[3] = m2l_fma(-D[37], m, L[3]);
    }
    { const T m = __ldg(Ms + 21);
      L[0] = m2l_fma(D[21], m, L[0]);
      L[1] = m2l_fma(-D[36], m, L[1]);
      L[2] = m2l_fma(-D[38], m, L[2]);
      L[3] = m2l_fma(-D[39], m, L[3]);
    }
    { const T m = __ldg(Ms + 22);
      L[0] = m2l_fma(D[22], m, L[0]);
      L[1] = m2l_fma(-D[37], m, L[1]);
      L[2] = m2l_fma(-D[39], m, L[2]);
      L[3] = m2l_fma(-D[40], m, L[3]);
    }
    { const T m = __ldg(Ms + 23);
      L[0] = m2l_fma(D[23], m, L[0]);
      L[1] = m2l_fma(-D[38], m, L[1]);
      L[2] = m2l_fma(-D[41], m, L[2]);
      L[3] = m2l_fma(-D[42], m, L[3]);
    }
    { const T m = __ldg(Ms + 24);
      L[0] = m2l_fma(D[24], m, L[0]);
      L[1] = m2l_fma(-D[39], m, L[1]);
      L[2] = m2l_fma(-D[42], m, L[2]);
      L[3] = m2l_fma(-D[43], m, L[3]);
    }
    { const T m = __ldg(Ms + 25);
      L[0] = m2l_fma(D[25], m, L[0]);
      L[1] = m2l_fma(-D[40], m, L[1]);
      L[2] = m2l_fma(-D[43], m, L[2]);
      L[3] = m2l_fma(-D[44], m, L[3]);
    }
    { const T m = __ldg(Ms + 26);
      L[0] = m2l_fma(D[26], m, L[0]);
      L[1] = m2l_fma(-D[41], m, L[1]);
      L[2] = m2l_fma(-D[45], m, L[2]);
      L[3] = m2l_fma(-D[46], m, L[3]);
    }
    { const T m = __ldg(Ms + 27);
      L[0] = m2l_fma(D[27], m, L[0]);
      L[1] = m2l_fma(-D[42], m, L[1]);
      L[2] = m2l_fma(-D[46], m, L[2]);
      L[3] = m2l_fma(-D[47], m, L[3]);
    }
    { const T m = __ldg(Ms + 28);
      L[0] = m2l_fma(D[28], m, L[0]);
      L[1] = m2l_fma(-D[43], m, L[1]);
      L[2] = m2l_fma(-D[47], m, L[2]);
      L[3] = m2l_fma(-D[48], m, L[3]);
    }
    { const T m = __ldg(Ms + 29);
      L[0] = m2l_fma(D[29], m, L[0]);
      L[1] = m2l_fma(-D[44], m, L[1]);
      L[2] = m2l_fma(-D[48], m, L[2]);
      L[3] = m2l_fma(-D[49], m, L[3]);
    }
    { const T m = __ldg(Ms + 30);
      L[0] = m2l_fma(D[30], m, L[0]);
      L[1] = m2l_fma(-D[45], m, L[1]);
      L[2] = m2l_fma(-D[50], m, L[2]);
      L[3] = m2l_fma(-D[51], m, L[3]);
    }
    { const T m = __ldg(Ms + 31);
      L[0] = m2l_fma(D[31], m, L[0]);
      L[1] = m2l_fma(-D[46], m, L[1]);
      L[2] = m2l_fma(-D[51], m, L[2]);
      L[3] = m2l_fma(-D[52], m, L[3]);
    }
    { const T m = __ldg(Ms + 32);
      L[0] = m2l_fma(D[32], m, L[0]);
      L[1] = m2l_fma(-D[47], m, L[1]);
      L[2] = m2l_fma(-D[52], m, L[2]);
      L[3] = m2l_fma(-D[53], m, L[3]);
    }
    { const T m = __ldg(Ms + 33);
      L[0] = m2l_fma(D[33], m, L[0]);
      L[1] = m2l_fma(-D[48], m, L[1]);
      L[2] = m2l_fma(-D[53], m, L[2]);
      L[3] = m2l_fma(-D[54], m, L[3]);
    }
    { const T m = __ldg(Ms + 34);
      L[0] = m2l_fma(D[34], m, L[0]);
      L[1] = m2l_fma(-D[49], m, L[1]);
      L[2] = m2l_fma(-D[54], m, L[2]);
      L[3] = m2l_fma(-D[55], m, L[3]);
    }
    { const T m = __ldg(Ms + 35);
      L[0] = m2l_fma(D[35], m, L[0]);
    }
    { const T m = __ldg(Ms + 36);
      L[0] = m2l_fma(D[36], m, L[0]);
    }
    { const T m = __ldg(Ms + 37);
      L[0] = m2l_fma(D[37], m, L[0]);
    }
    { const T m = __ldg(Ms + 38);
      L[0] = m2l_fma(D[38], m, L[0]);
    }
    { const T m = __ldg(Ms + 39);
      L[0] = m2l_fma(D[39], m, L[0]);
    }
    { const T m = __ldg(Ms + 40);
      L[0] = m2l_fma(D[40], m, L[0]);
    }
    { const T m = __ldg(Ms + 41);
      L[0] = m2l_fma(D[41], m, L[0]);
    }
    { const T m = __ldg(Ms + 42);
      L[0] = m2l_fma(D[42], m, L[0]);
    }
    { const T m = __ldg(Ms + 43);
      L[0] = m2l_fma(D[43], m, L[0]);
    }
    { const T m = __ldg(Ms + 44);
      L[0] = m2l_fma(D[44], m, L[0]);
    }
    { const T m = __ldg(Ms + 45);
      L[0] = m2l_fma(D[45], m, L[0]);
    }
    { const T m = __ldg(Ms + 46);
      L[0] = m2l_fma(D[46], m, L[0]);
    }
    { const T m = __ldg(Ms + 47);
      L[0] = m2l_fma(D[47], m, L[0]);
    }
    { const T m = __ldg(Ms + 48);
      L[0] = m2l_fma(D[48], m, L[0]);
    }
    { const T m = __ldg(Ms + 49);
      L[0] = m2l_fma(D[49], m, L[0]);
    }
    { const T m = __ldg(Ms + 50);
      L[0] = m2l_fma(D[50], m, L[0]);
    }
    { const T m = __ldg(Ms + 51);
      L[0] = m2l_fma(D[51], m, L[0]);
    }
    { const T m = __ldg(Ms + 52);
      L[0] = m2l_fma(D[52], m, L[0]);
    }
    { const T m = __ldg(Ms + 53);
      L[0] = m2l_fma(D[53], m, L[0]);
    }
    { const T m = __ldg(Ms + 54);
      L[0] = m2l_fma(D[54], m, L[0]);
    }
    { const T m = __ldg(Ms + 55);
      L[0] = m2l_fma(D[55], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_a_forces_5(const T (&D)[56], const T *__restrict__ Ms, T rho, T (&L)[56])
{
    L[0] = T(0);
    T rp = T(1);
    { const T m = __ldg(Ms + 0) * rp;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[9] * m;
      L[10] = D[10] * m;
      L[11] = D[11] * m;
      L[12] = D[12] * m;
      L[13] = D[13] * m;
      L[14] = D[14] * m;
      L[15] = D[15] * m;
      L[16] = D[16] * m;
      L[17] = D[17] * m;
      L[18] = D[18] * m;
      L[19] = D[19] * m;
      L[20] = D[20] * m;
      L[21] = D[21] * m;
      L[22] = D[22] * m;
      L[23] = D[23] * m;
      L[24] = D[24] * m;
      L[25] = D[25] * m;
      L[26] = D[26] * m;
      L[27] = D[27] * m;
      L[28] = D[28] * m;
      L[29] = D[29] * m;
      L[30] = D[30] * m;
      L[31] = D[31] * m;
      L[32] = D[32] * m;
      L[33] = D[33] * m;
      L[34] = D[34] * m;
      L[35] = D[35] * m;
      L[36] = D[36] * m;
      L[37] = D[37] * m;
      L[38] = D[38] * m;
      L[39] = D[39] * m;
      L[40] = D[40] * m;
      L[41] = D[41] * m;
      L[42] = D[42] * m;
      L[43] = D[43] * m;
      L[44] = D[44] * m;
      L[45] = D[45] * m;
      L[46] = D[46] * m;
      L[47] = D[47] * m;
      L[48] = D[48] * m;
      L[49] = D[49] * m;
      L[50] = D[50] * m;
      L[51] = D[51] * m;
      L[52] = D[52] * m;
      L[53] = D[53] * m;
      L[54] = D[54] * m;
      L[55] = D[55] * m;
    }
    rp *= rho;
    { const T m = -__ldg(Ms + 1) * rp;
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[15], m, L[9]);
      L[10] = m2l_fma(D[20], m, L[10]);
      L[11] = m2l_fma(D[21], m, L[11]);
      L[12] = m2l_fma(D[22], m, L[12]);
      L[13] = m2l_fma(D[23], m, L[13]);
      L[14] = m2l_fma(D[24], m, L[14]);
      L[15] = m2l_fma(D[25], m, L[15]);
      L[16] = m2l_fma(D[26], m, L[16]);
      L[17] = m2l_fma(D[27], m, L[17]);
      L[18] = m2l_fma(D[28], m, L[18]);
      L[19] = m2l_fma(D[29], m, L[19]);
      L[20] = m2l_fma(D[35], m, L[20]);
      L[21] = m2l_fma(D[36], m, L[21]);
      L[22] = m2l_fma(D[37], m, L[22]);
      L[23] = m2l_fma(D[38], m, L[23]);
      L[24] = m2l_fma(D[39], m, L[24]);
      L[25] = m2l_fma(D[40], m, L[25]);
      L[26] = m2l_fma(D[41], m, L[26]);
      L[27] = m2l_fma(D[42], m, L[27]);
      L[28] = m2l_fma(D[43], m, L[28]);
      L[29] = m2l_fma(D[44], m, L[29]);
      L[30] = m2l_fma(D[45], m, L[30]);
      L[31] = m2l_fma(D[46], m, L[31]);
      L[32] = m2l_fma(D[47], m, L[32]);
      L[33] = m2l_fma(D[48], m, L[33]);
      L[34] = m2l_fma(D[49], m, L[34]);
    }
    { const T m = -__ldg(Ms + 2) * rp;
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[18], m, L[9]);
      L[10] = m2l_fma(D[21], m, L[10]);
      L[11] = m2l_fma(D[23], m, L[11]);
      L[12] = m2l_fma(D[24], m, L[12]);
      L[13] = m2l_fma(D[26], m, L[13]);
      L[14] = m2l_fma(D[27], m, L[14]);
      L[15] = m2l_fma(D[28], m, L[15]);
      L[16] = m2l_fma(D[30], m, L[16]);
      L[17] = m2l_fma(D[31], m, L[17]);
      L[18] = m2l_fma(D[32], m, L[18]);
      L[19] = m2l_fma(D[33], m, L[19]);
      L[20] = m2l_fma(D[36], m, L[20]);
      L[21] = m2l_fma(D[38], m, L[21]);
      L[22] = m2l_fma(D[39], m, L[22]);
      L[23] = m2l_fma(D[41], m, L[23]);
      L[24] = m2l_fma(D[42], m, L[24]);
      L[25] = m2l_fma(D[43], m, L[25]);
      L[26] = m2l_fma(D[45], m, L[26]);
      L[27] = m2l_fma(D[46], m, L[27]);
      L[28] = m2l_fma(D[47], m, L[28]);
      L[29] = m2l_fma(D[48], m, L[29]);
      L[30] = m2l_fma(D[50], m, L[30]);
      L[31] = m2l_fma(D[51], m, L[31]);
      L[32] = m2l_fma(D[52], m, L[32]);
      L[33] = m2l_fma(D[53], m, L[33]);
      L[34] = m2l_fma(D[54], m, L[34]);
    }
    { const T m = -__ldg(Ms + 3) * rp;
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(D[22], m, L[10]);
      L[11] = m2l_fma(D[24], m, L[11]);
      L[12] = m2l_fma(D[25], m, L[12]);
      L[13] = m2l_fma(D[27], m, L[13]);
      L[14] = m2l_fma(D[28], m, L[14]);
      L[15] = m2l_fma(D[29], m, L[15]);
      L[16] = m2l_fma(D[31], m, L[16]);
      L[17] = m2l_fma(D[32], m, L[17]);
      L[18] = m2l_fma(D[33], m, L[18]);
      L[19] = m2l_fma(D[34], m, L[19]);
      L[20] = m2l_fma(D[37], m, L[20]);
      L[21] = m2l_fma(D[39], m, L[21]);
      L[22] = m2l_fma(D[40], m, L[22]);
      L[23] = m2l_fma(D[42], m, L[23]);
      L[24] = m2l_fma(D[43], m, L[24]);
      L[25] = m2l_fma(D[44], m, L[25]);
      L[26] = m2l_fma(D[46], m, L[26]);
      L[27] = m2l_fma(D[47], m, L[27]);
      L[28] = m2l_fma(D[48], m, L[28]);
      L[29] = m2l_fma(D[49], m, L[29]);
      L[30] = m2l_fma(D[51], m, L[30]);
      L[31] = m2l_fma(D[52], m, L[31]);
      L[32] = m2l_fma(D[53], m, L[32]);
      L[33] = m2l_fma(D[54], m, L[33]);
      L[34] = m2l_fma(D[55], m, L[34]);
    }
    rp *= rho;
    { const T m = __ldg(Ms + 4) * rp;
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[21], m, L[5]);
      L[6] = m2l_fma(D[22], m, L[6]);
      L[7] = m2l_fma(D[23], m, L[7]);
      L[8] = m2l_fma(D[24], m, L[8]);
      L[9] = m2l_fma(D[25], m, L[9]);
      L[10] = m2l_fma(D[35], m, L[10]);
      L[11] = m2l_fma(D[36], m, L[11]);
      L[12] = m2l_fma(D[37], m, L[12]);
      L[13] = m2l_fma(D[38], m, L[13]);
      L[14] = m2l_fma(D[39], m, L[14]);
      L[15] = m2l_fma(D[40], m, L[15]);
      L[16] = m2l_fma(D[41], m, L[16]);
      L[17] = m2l_fma(D[42], m, L[17]);
      L[18] = m2l_fma(D[43], m, L[18]);
      L[19] = m2l_fma(D[44], m, L[19]);
    }
    { const T m = __ldg(Ms + 5) * rp;
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(D[28], m, L[9]);
      L[10] = m2l_fma(D[36], m, L[10]);
      L[11] = m2l_fma(D[38], m, L[11]);
      L[12] = m2l_fma(D[39], m, L[12]);
      L[13] = m2l_fma(D[41], m, L[13]);
      L[14] = m2l_fma(D[42], m, L[14]);
      L[15] = m2l_fma(D[43], m, L[15]);
      L[16] = m2l_fma(D[45], m, L[16]);
      L[17] = m2l_fma(D[46], m, L[17]);
      L[18] = m2l_fma(D[47], m, L[18]);
      L[19] = m2l_fma(D[48], m, L[19]);
    }
    { const T m = __ldg(Ms + 6) * rp;
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[24], m, L[5]);
      L[6] = m2l_fma(D[25], m, L[6]);
      L[7] = m2l_fma(D[27], m, L[7]);
      L[8] = m2l_fma(D[28], m, L[8]);
      L[9] = m2l_fma(D[29], m, L[9]);
      L[10] = m2l_fma(D[37], m, L[10]);
      L[11] = m2l_fma(D[39], m, L[11]);
      L[12] = m2l_fma(D[40], m, L[12]);
      L[13] = m2l_fma(D[42], m, L[13]);
      L[14] = m2l_fma(D[43], m, L[14]);
      L[15] = m2l_fma(D[44], m, L[15]);
      L[16] = m2l_fma(D[46], m, L[16]);
      L[17] = m2l_fma(D[47], m, L[17]);
      L[18] = m2l_fma(D[48], m, L[18]);
      L[19] = m2l_fma(D[49], m, L[19]);
    }
    { const T m = __ldg(Ms + 7) * rp;
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[30], m, L[7]);
      L[8] = m2l_fma(D[31], m, L[8]);
      L[9] = m2l_fma(D[32], m, L[9]);
      L[10] = m2l_fma(D[38], m, L[10]);
      L[11] = m2l_fma(D[41], m, L[11]);
      L[12] = m2l_fma(D[42], m, L[12]);
      L[13] = m2l_fma(D[45], m, L[13]);
      L[14] = m2l_fma(D[46], m, L[14]);
      L[15] = m2l_fma(D[47], m, L[15]);
      L[16] = m2l_fma(D[50], m, L[16]);
      L[17] = m2l_fma(D[51], m, L[17]);
      L[18] = m2l_fma(D[52], m, L[18]);
      L[19] = m2l_fma(D[53], m, L[19]);
    }
    { const T m = __ldg(Ms + 8) * rp;
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
      L[4] = m2l_fma(D[24], m, L[4]);
      L[5] = m2l_fma(D[27], m, L[5]);
      L[6] = m2l_fma(D[28], m, L[6]);
      L[7] = m2l_fma(D[31], m, L[7]);
      L[8] = m2l_fma(D[32], m, L[8]);
      L[9] = m2l_fma(D[33], m, L[9]);
      L[10] = m2l_fma(D[39], m, L[10]);
      L[11] = m2l_fma(D[42], m, L[11]);
      L[12] = m2l_fma(D[43], m, L[12]);
      L[13] = m2l_fma(D[46], m, L[13]);
      L[14] = m2l_fma(D[47], m, L[14]);
      L[15] = m2l_fma(D[48], m, L[15]);
      L[16] = m2l_fma(D[51], m, L[16]);
      L[17] = m2l_fma(D[52], m, L[17]);
      L[18] = m2l_fma(D[53], m, L[18]);
      L[19] = m2l_fma(D[54], m, L[19]);
    }
    { const T m = __ldg(Ms + 9) * rp;
      L[1] = m2l_fma(D[15], m, L[1]);
      L[2] = m2l_fma(D[18], m, L[2]);
      L[3] = m2l_fma(D[19], m, L[3]);
      L[4] = m2l_fma(D[25], m, L[4]);
      L[5] = m2l_fma(D[28], m, L[5]);
      L[6] = m2l_fma(D[29], m, L[6]);
      L[7] = m2l_fma(D[32], m, L[7]);
      L[8] = m2l_fma(D[33], m, L[8]);
      L[9] = m2l_fma(D[34], m, L[9]);
      L[10] = m2l_fma(D[40], m, L[10]);
      L[11] = m2l_fma(D[43], m, L[11]);
      L[12] = m2l_fma(D[44], m, L[12]);
      L[13] = m2l_fma(D[47], m, L[13]);
      L[14] = m2l_fma(D[48], m, L[14]);
      L[15] = m2l_fma(D[49], m, L[15]);
      L[16] = m2l_fma(D[52], m, L[16]);
      L[17] = m2l_fma(D[53], m, L[17]);
      L[18] = m2l_fma(D[54], m, L[18]);
      L[19] = m2l_fma(D[55], m, L[19]);
    }
    rp *= rho;
    { const T m = -__ldg(Ms + 10) * rp;
      L[1] = m2l_fma(D[20], m, L[1]);
      L[2] = m2l_fma(D[21], m, L[2]);
      L[3] = m2l_fma(D[22], m, L[3]);
      L[4] = m2l_fma(D[35], m, L[4]);
      L[5] = m2l_fma(D[36], m, L[5]);
      L[6] = m2l_fma(D[37], m, L[6]);
      L[7] = m2l_fma(D[38], m, L[7]);
      L[8] = m2l_fma(D[39], m, L[8]);
      L[9] = m2l_fma(D[40], m, L[9]);
    }
    { const T m = -__ldg(Ms + 11) * rp;
      L[1] = m2l_fma(D[21], m, L[1]);
      L[2] = m2l_fma(D[23], m, L[2]);
      L[3] = m2l_fma(D[24], m, L[3]);
      L[4] = m2l_fma(D[36], m, L[4]);
      L[5] = m2l_fma(D[38], m, L[5]);
      L[6] = m2l_fma(D[39], m, L[6]);
      L[7] = m2l_fma(D[41], m, L[7]);
      L[8] = m2l_fma(D[42], m, L[8]);
      L[9] = m2l_fma(D[43], m, L[9]);
    }
    { const T m = -__ldg(Ms + 12) * rp;
      L[1] = m2l_fma(D[22], m, L[1]);
      L[2] = m2l_fma(D[24], m, L[2]);
      L[3] = m2l_fma(D[25], m, L[3]);
      L[4] = m2l_fma(D[37], m, L[4]);
      L[5] = m2l_fma(D[39], m, L[5]);
      L[6] = m2l_fma(D[40], m, L[6]);
      L[7] = m2l_fma(D[42], m, L[7]);
      L[8] = m2l_fma(D[43], m, L[8]);
      L[9] = m2l_fma(D[44], m, L[9]);
    }
    { const T m = -__ldg(Ms + 13) * rp;
      L[1] = m2l_fma(D[23], m, L[1]);
      L[2] = m2l_fma(D[26], m, L[2]);
      L[3] = m2l_fma(D[27], m, L[3]);
      L[4] = m2l_fma(D[38], m, L[4]);
      L[5] = m2l_fma(D[41], m, L[5]);
      L[6] = m2l_fma(D[42], m, L[6]);
      L[7] = m2l_fma(D[45], m, L[7]);
      L[8] = m2l_fma(D[46], m, L[8]);
      L[9] = m2l_fma(D[47], m, L[9]);
    }
    { const T m = -__ldg(Ms + 14) * rp;
      L[1] = m2l_fma(D[24], m, L[1]);
      L[2] = m2l_fma(D[27], m, L[2]);
      L[3] = m2l_fma(D[28], m, L[3]);
      L[4] = m2l_fma(D[39], m, L[4]);
      L[5] = m2l_fma(D[42], m, L[5]);
      L[6] = m2l_fma(D[43], m, L[6]);
      L[7] = m2l_fma(D[46], m, L[7]);
      L[8] = m2l_fma(D[47], m, L[8]);
      L[9] = m2l_fma(D[48], m, L[9]);
    }
    { const T m = -__ldg(Ms + 15) * rp;
      L[1] = m2l_fma(D[25], m, L[1]);
      L[2] = m2l_fma(D[28], m, L[2]);
      L[3] = m2l_fma(D[29], m, L[3]);
      L[4] = m2l_fma(D[40], m, L[4]);
      L[5] = m2l_fma(D[43], m, L[5]);
      L[6] = m2l_fma(D[44], m, L[6]);
      L[7] = m2l_fma(D[47], m, L[7]);
      L[8] = m2l_fma(D[48], m, L[8]);
      L[9] = m2l_fma(D[49], m, L[9]);
    }
    { const T m = -__ldg(Ms + 16) * rp;
      L[1] = m2l_fma(D[26], m, L[1]);
      L[2] = m2l_fma(D[30], m, L[2]);
      L[3] = m2l_fma(D[31], m, L[3]);
      L[4] = m2l_fma(D[41], m, L[4]);
      L[5] = m2l_fma(D[45], m, L[5]);
      L[6] = m2l_fma(D[46], m, L[6]);
      L[7] = m2l_fma(D[50], m, L[7]);
      L[8] = m2l_fma(D[51], m, L[8]);
      L[9] = m2l_fma(D[52], m, L[9]);
    }
    { const T m = -__ldg(Ms + 17) * rp;
      L[1] = m2l_fma(D[27], m, L[1]);
      L[2] = m2l_fma(D[31], m, L[2]);
      L[3] = m2l_fma(D[32], m, L[3]);
      L[4] = m2l_fma(D[42], m, L[4]);
      L[5] = m2l_fma(D[46], m, L[5]);
      L[6] = m2l_fma(D[47], m, L[6]);
      L[7] = m2l_fma(D[51], m, L[7]);
      L[8] = m2l_fma(D[52], m, L[8]);
      L[9] = m2l_fma(D[53], m, L[9]);
    }
    { const T m = -__ldg(Ms + 18) * rp;
      L[1] = m2l_fma(D[28], m, L[1]);
      L[2] = m2l_fma(D[32], m, L[2]);
      L[3] = m2l_fma(D[33], m, L[3]);
      L[4] = m2l_fma(D[43], m, L[4]);
      L[5] = m2l_fma(D[47], m, L[5]);
      L[6] = m2l_fma(D[48], m, L[6]);
      L[7] = m2l_fma(D[52], m, L[7]);
      L[8] = m2l_fma(D[53], m, L[8]);
      L[9] = m2l_fma(D[54], m, L[9]);
    }
    { const T m = -__ldg(Ms + 19) * rp;
      L[1] = m2l_fma(D[29], m, L[1]);
      L[2] = m2l_fma(D[33], m, L[2]);
      L[3] = m2l_fma(D[34], m, L[3]);
      L[4] = m2l_fma(D[44], m, L[4]);
      L[5] = m2l_fma(D[48], m, L[5]);
      L[6] = m2l_fma(D[49], m, L[6]);
      L[7] = m2l_fma(D[53], m, L[7]);
      L[8] = m2l_fma(D[54], m, L[8]);
      L[9] = m2l_fma(D[55], m, L[9]);
    }
    rp *= rho;
    { const T m = __ldg(Ms + 20) * rp;
      L[1] = m2l_fma(D[35], m, L[1]);
      L[2] = m2l_fma(D[36], m, L[2]);
      L[3] = m2l_fma(D[37], m, L[3]);
    }
    { const T m = __ldg(Ms + 21) * rp;
      L[1] = m2l_fma(D[36], m, L[1]);
      L[2] = m2l_fma(D[38], m, L[2]);
      L[3] = m2l_fma(D[39], m, L[3]);
    }
    { const T m = __ldg(Ms + 22) * rp;
      L[1] = m2l_fma(D[37], m, L[1]);
      L[2] = m2l_fma(D[39], m, L[2]);
      L[3] = m2l_fma(D[40], m, L[3]);
    }
    { const T m = __ldg(Ms + 23) * rp;
      L[1] = m2l_fma(D[38], m, L[1]);
      L[2] = m2l_fma(D[41], m, L[2]);
      L[3] = m2l_fma(D[42], m, L[3]);
    }
    { const T m = __ldg(Ms + 24) * rp;
      L[1] = m2l_fma(D[39], m, L[1]);
      L[2] = m2l_fma(D[42], m, L[2]);
      L[3] = m2l_fma(D[43], m, L[3]);
    }
    { const T m = __ldg(Ms + 25) * rp;
      L[1] = m2l_fma(D[40], m, L[1]);
      L[2] = m2l_fma(D[43], m, L[2]);
      L[3] = m2l_fma(D[44], m, L[3]);
    }
    { const T m = __ldg(Ms + 26) * rp;
      L[1] = m2l_fma(D[41], m, L[1]);
      L[2] = m2l_fma(D[45], m, L[2]);
      L[3] = m2l_fma(D[46], m, L[3]);
    }
    { const T m = __ldg(Ms + 27) * rp;
      L[1] = m2l_fma(D[42], m, L[1]);
      L[2] = m2l_fma(D[46], m, L[2]);
      L[3] = m2l_fma(D[47], m, L[3]);
    }
    { const T m = __ldg(Ms + 28) * rp;
      L[1] = m2l_fma(D[43], m, L[1]);
      L[2] = m2l_fma(D[47], m, L[2]);
      L[3] = m2l_fma(D[48], m, L[3]);
    }
    { const T m = __ldg(Ms + 29) * rp;
      L[1] = m2l_fma(D[44], m, L[1]);
      L[2] = m2l_fma(D[48], m, L[2]);
      L[3] = m2l_fma(D[49], m, L[3]);
    }
    { const T m = __ldg(Ms + 30) * rp;
      L[1] = m2l_fma(D[45], m, L[1]);
      L[2] = m2l_fma(D[50], m, L[2]);
      L[3] = m2l_fma(D[51], m, L[3]);
    }
    { const T m = __ldg(Ms + 31) * rp;
      L[1] = m2l_fma(D[46], m, L[1]);
      L[2] = m2l_fma(D[51], m, L[2]);
      L[3] = m2l_fma(D[52], m, L[3]);
    }
    { const T m = __ldg(Ms + 32) * rp;
      L[1] = m2l_fma(D[47], m, L[1]);
      L[2] = m2l_fma(D[52], m, L[2]);
      L[3] = m2l_fma(D[53], m, L[3]);
    }
    { const T m = __ldg(Ms + 33) * rp;
      L[1] = m2l_fma(D[48], m, L[1]);
      L[2] = m2l_fma(D[53], m, L[2]);
      L[3] = m2l_fma(D[54], m, L[3]);
    }
    { const T m = __ldg(Ms + 34) * rp;
      L[1] = m2l_fma(D[49], m, L[1]);
      L[2] = m2l_fma(D[54], m, L[2]);
      L[3] = m2l_fma(D[55], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_forces_5(const T (&D)[56], const T *__restrict__ Ms, T (&L)[56])
{
    L[0] = T(0);
    { const T m = __ldg(Ms + 0);
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[9] * m;
      L[10] = -D[10] * m;
      L[11] = -D[11] * m;
      L[12] = -D[12] * m;
      L[13] = -D[13] * m;
      L[14] = -D[14] * m;
      L[15] = -D[15] * m;
      L[16] = -D[16] * m;
      L[17] = -D[17] * m;
      L[18] = -D[18] * m;
      L[19] = -D[19] * m;
      L[20] = D[20] * m;
      L[21] = D[21] * m;
      L[22] = D[22] * m;
      L[23] = D[23] * m;
      L[24] = D[24] * m;
      L[25] = D[25] * m;
      L[26] = D[26] * m;
      L[27] = D[27] * m;
      L[28] = D[28] * m;
      L[29] = D[29] * m;
      L[30] = D[30] * m;
      L[31] = D[31] * m;
      L[32] = D[32] * m;
      L[33] = D[33] * m;
      L[34] = D[34] * m;
      L[35] = -D[35] * m;
      L[36] = -D[36] * m;
      L[37] = -D[37] * m;
      L[38] = -D[38] * m;
      L[39] = -D[39] * m;
      L[40] = -D[40] * m;
      L[41] = -D[41] * m;
      L[42] = -D[42] * m;
      L[43] = -D[43] * m;
      L[44] = -D[44] * m;
      L[45] = -D[45] * m;
      L[46] = -D[46] * m;
      L[47] = -D[47] * m;
      L[48] = -D[48] * m;
      L[49] = -D[49] * m;
      L[50] = -D[50] * m;
      L[51] = -D[51] * m;
      L[52] = -D[52] * m;
      L[53] = -D[53] * m;
      L[54] = -D[54] * m;
      L[55] = -D[55] * m;
    }
    { const T m = __ldg(Ms + 1);
      L[1] = m2l_fma(-D[4], m, L[1]);
      L[2] = m2l_fma(-D[5], m, L[2]);
      L[3] = m2l_fma(-D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[15], m, L[9]);
      L[10] = m2l_fma(-D[20], m, L[10]);
      L[11] = m2l_fma(-D[21], m, L[11]);
      L[12] = m2l_fma(-D[22], m, L[12]);
      L[13] = m2l_fma(-D[23], m, L[13]);
      L[14] = m2l_fma(-D[24], m, L[14]);
      L[15] = m2l_fma(-D[25], m, L[15]);
      L[16] = m2l_fma(-D[26], m, L[16]);
      L[17] = m2l_fma(-D[27], m, L[17]);
      L[18] = m2l_fma(-D[28], m, L[18]);
      L[19] = m2l_fma(-D[29], m, L[19]);
      L[20] = m2l_fma(D[35], m, L[20]);
      L[21] = m2l_fma(D[36], m, L[21]);
      L[22] = m2l_fma(D[37], m, L[22]);
      L[23] = m2l_fma(D[38], m, L[23]);
      L[24] = m2l_fma(D[39], m, L[24]);
      L[25] = m2l_fma(D[40], m, L[25]);
      L[26] = m2l_fma(D[41], m, L[26]);
      L[27] = m2l_fma(D[42], m, L[27]);
      L[28] = m2l_fma(D[43], m, L[28]);
      L[29] = m2l_fma(D[44], m, L[29]);
      L[30] = m2l_fma(D[45], m, L[30]);
      L[31] = m2l_fma(D[46], m, L[31]);
      L[32] = m2l_fma(D[47], m, L[32]);
      L[33] = m2l_fma(D[48], m, L[33]);
      L[34] = m2l_fma(D[49], m, L[34]);
    }
    { const T m = __ldg(Ms + 2);
      L[1] = m2l_fma(-D[5], m, L[1]);
      L[2] = m2l_fma(-D[7], m, L[2]);
      L[3] = m2l_fma(-D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[18], m, L[9]);
      L[10] = m2l_fma(-D[21], m, L[10]);
      L[11] = m2l_fma(-D[23], m, L[11]);
      L[12] = m2l_fma(-D[24], m, L[12]);
      L[13] = m2l_fma(-D[26], m, L[13]);
      L[14] = m2l_fma(-D[27], m, L[14]);
      L[15] = m2l_fma(-D[28], m, L[15]);
      L[16] = m2l_fma(-D[30], m, L[16]);
      L[17] = m2l_fma(-D[31], m, L[17]);
      L[18] = m2l_fma(-D[32], m, L[18]);
      L[19] = m2l_fma(-D[33], m, L[19]);
      L[20] = m2l_fma(D[36], m, L[20]);
      L[21] = m2l_fma(D[38], m, L[21]);
      L[22] = m2l_fma(D[39], m, L[22]);
      L[23] = m2l_fma(D[41], m, L[23]);
      L[24] = m2l_fma(D[42], m, L[24]);
      L[25] = m2l_fma(D[43], m, L[25]);
      L[26] = m2l_fma(D[45], m, L[26]);
      L[27] = m2l_fma(D[46], m, L[27]);
      L[28] = m2l_fma(D[47], m, L[28]);
      L[29] = m2l_fma(D[48], m, L[29]);
      L[30] = m2l_fma(D[50], m, L[30]);
      L[31] = m2l_fma(D[51], m, L[31]);
      L[32] = m2l_fma(D[52], m, L[32]);
      L[33] = m2l_fma(D[53], m, L[33]);
      L[34] = m2l_fma(D[54], m, L[34]);
    }
    { const T m = __ldg(Ms + 3);
      L[1] = m2l_fma(-D[6], m, L[1]);
      L[2] = m2l_fma(-D[8], m, L[2]);
      L[3] = m2l_fma(-D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(-D[22], m, L[10]);
      L[11] = m2l_fma(-D[24], m, L[11]);
      L[12] = m2l_fma(-D[25], m, L[12]);
      L[13] = m2l_fma(-D[27], m, L[13]);
      L[14] = m2l_fma(-D[28], m, L[14]);
      L[15] = m2l_fma(-D[29], m, L[15]);
      L[16] = m2l_fma(-D[31], m, L[16]);
      L[17] = m2l_fma(-D[32], m, L[17]);
      L[18] = m2l_fma(-D[33], m, L[18]);
      L[19] = m2l_fma(-D[34], m, L[19]);
      L[20] = m2l_fma(D[37], m, L[20]);
      L[21] = m2l_fma(D[39], m, L[21]);
      L[22] = m2l_fma(D[40], m, L[22]);
      L[23] = m2l_fma(D[42], m, L[23]);
      L[24] = m2l_fma(D[43], m, L[24]);
      L[25] = m2l_fma(D[44], m, L[25]);
      L[26] = m2l_fma(D[46], m, L[26]);
      L[27] = m2l_fma(D[47], m, L[27]);
      L[28] = m2l_fma(D[48], m, L[28]);
      L[29] = m2l_fma(D[49], m, L[29]);
      L[30] = m2l_fma(D[51], m, L[30]);
      L[31] = m2l_fma(D[52], m, L[31]);
      L[32] = m2l_fma(D[53], m, L[32]);
      L[33] = m2l_fma(D[54], m, L[33]);
      L[34] = m2l_fma(D[55], m, L[34]);
    }
    { const T m = __ldg(Ms + 4);
      L[1] = m2l_fma(-D[10], m, L[1]);
      L[2] = m2l_fma(-D[11], m, L[2]);
      L[3] = m2l_fma(-D[12], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[21], m, L[5]);
      L[6] = m2l_fma(D[22], m, L[6]);
      L[7] = m2l_fma(D[23], m, L[7]);
      L[8] = m2l_fma(D[24], m, L[8]);
      L[9] = m2l_fma(D[25], m, L[9]);
      L[10] = m2l_fma(-D[35], m, L[10]);
      L[11] = m2l_fma(-D[36], m, L[11]);
      L[12] = m2l_fma(-D[37], m, L[12]);
      L[13] = m2l_fma(-D[38], m, L[13]);
      L[14] = m2l_fma(-D[39], m, L[14]);
      L[15] = m2l_fma(-D[40], m, L[15]);
      L[16] = m2l_fma(-D[41], m, L[16]);
      L[17] = m2l_fma(-D[42], m, L[17]);
      L[18] = m2l_fma(-D[43], m, L[18]);
      L[19] = m2l_fma(-D[44], m, L[19]);
    }
    { const T m = __ldg(Ms + 5);
      L[1] = m2l_fma(-D[11], m, L[1]);
      L[2] = m2l_fma(-D[13], m, L[2]);
      L[3] = m2l_fma(-D[14], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(D[28], m, L[9]);
      L[10] = m2l_fma(-D[36], m, L[10]);
      L[11] = m2l_fma(-D[38], m, L[11]);
      L[12] = m2l_fma(-D[39], m, L[12]);
      L[13] = m2l_fma(-D[41], m, L[13]);
      L[14] = m2l_fma(-D[42], m, L[14]);
      L[15] = m2l_fma(-D[43], m, L[15]);
      L[16] = m2l_fma(-D[45], m, L[16]);
      L[17] = m2l_fma(-D[46], m, L[17]);
      L[18] = m2l_fma(-D[47], m, L[18]);
      L[19] = m2l_fma(-D[48], m, L[19]);
    }
    { const T m = __ldg(Ms + 6);
      L[1] = m2l_fma(-D[12], m, L[1]);
      L[2] = m2l_fma(-D[14], m, L[2]);
      L[3] = m2l_fma(-D[15], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[24], m, L[5]);
      L[6] = m2l_fma(D[25], m, L[6]);
      L[7] = m2l_fma(D[27], m, L[7]);
      L[8] = m2l_fma(D[28], m, L[8]);
      L[9] = m2l_fma(D[29], m, L[9]);
      L[10] = m2l_fma(-D[37], m, L[10]);
      L[11] = m2l_fma(-D[39], m, L[11]);
      L[12] = m2l_fma(-D[40], m, L[12]);
      L[13] = m2l_fma(-D[42], m, L[13]);
      L[14] = m2l_fma(-D[43], m, L[14]);
      L[15] = m2l_fma(-D[44], m, L[15]);
      L[16] = m2l_fma(-D[46], m, L[16]);
      L[17] = m2l_fma(-D[47], m, L[17]);
      L[18] = m2l_fma(-D[48], m, L[18]);
      L[19] = m2l_fma(-D[49], m, L[19]);
    }
    { const T m = __ldg(Ms + 7);
      L[1] = m2l_fma(-D[13], m, L[1]);
      L[2] = m2l_fma(-D[16], m, L[2]);
      L[3] = m2l_fma(-D[17], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[30], m, L[7]);
      L[8] = m2l_fma(D[31], m, L[8]);
      L[9] = m2l_fma(D[32], m, L[9]);
      L[10] = m2l_fma(-D[38], m, L[10]);
      L[11] = m2l_fma(-D[41], m, L[11]);
      L[12] = m2l_fma(-D[42], m, L[12]);
      L[13] = m2l_fma(-D[45], m, L[13]);
      L[14] = m2l_fma(-D[46], m, L[14]);
      L[15] = m2l_fma(-D[47], m, L[15]);
      L[16] = m2l_fma(-D[50], m, L[16]);
      L[17] = m2l_fma(-D[51], m, L[17]);
      L[18] = m2l_fma(-D[52], m, L[18]);
      L[19] = m2l_fma(-D[53], m, L[19]);
    }
    { const T m = __ldg(Ms + 8);
      L[1] = m2l_fma(-D[14], m, L[1]);
      L[2] = m2l_fma(-D[17], m, L[2]);
      L[3] = m2l_fma(-D[18], m, L[3]);
      L[4] = m2l_fma(D[24], m, L[4]);
      L[5] = m2l_fma(D[27], m, L[5]);
      L[6] = m2l_fma(D[28], m, L[6]);
      L[7] = m2l_fma(D[31], m, L[7]);
      L[8] = m2l_fma(D[32], m, L[8]);
      L[9] = m2l_fma(D[33], m, L[9]);
      L[10] = m2l_fma(-D[39], m, L[10]);
      L[11] = m2l_fma(-D[42], m, L[11]);
      L[12] = m2l_fma(-D[43], m, L[12]);
      L[13] = m2l_fma(-D[46], m, L[13]);
      L[14] = m2l_fma(-D[47], m, L[14]);
      L[15] = m2l_fma(-D[48], m, L[15]);
      L[16] = m2l_fma(-D[51], m, L[16]);
      L[17] = m2l_fma(-D[52], m, L[17]);
      L[18] = m2l_fma(-D[53], m, L[18]);
      L[19] = m2l_fma(-D[54], m, L[19]);
    }
    { const T m = __ldg(Ms + 9);
      L[1] = m2l_fma(-D[15], m, L[1]);
      L[2] = m2l_fma(-D[18], m, L[2]);
      L[3] = m2l_fma(-D[19], m, L[3]);
      L[4] = m2l_fma(D[25], m, L[4]);
      L[5] = m2l_fma(D[28], m, L[5]);
      L[6] = m2l_fma(D[29], m, L[6]);
      L[7] = m2l_fma(D[32], m, L[7]);
      L[8] = m2l_fma(D[33], m, L[8]);
      L[9] = m2l_fma(D[34], m, L[9]);
      L[10] = m2l_fma(-D[40], m, L[10]);
      L[11] = m2l_fma(-D[43], m, L[11]);
      L[12] = m2l_fma(-D[44], m, L[12]);
      L[13] = m2l_fma(-D[47], m, L[13]);
      L[14] = m2l_fma(-D[48], m, L[14]);
      L[15] = m2l_fma(-D[49], m, L[15]);
      L[16] = m2l_fma(-D[52], m, L[16]);
      L[17] = m2l_fma(-D[53], m, L[17]);
      L[18] = m2l_fma(-D[54], m, L[18]);
      L[19] = m2l_fma(-D[55], m, L[19]);
    }
    { const T m = __ldg(Ms + 10);
      L[1] = m2l_fma(-D[20], m, L[1]);
      L[2] = m2l_fma(-D[21], m, L[2]);
      L[3] = m2l_fma(-D[22], m, L[3]);
      L[4] = m2l_fma(D[35], m, L[4]);
      L[5] = m2l_fma(D[36], m, L[5]);
      L[6] = m2l_fma(D[37], m, L[6]);
      L[7] = m2l_fma(D[38], m, L[7]);
      L[8] = m2l_fma(D[39], m, L[8]);
      L[9] = m2l_fma(D[40], m, L[9]);
    }
    { const T m = __ldg(Ms + 11);
      L[1] = m2l_fma(-D[21], m, L[1]);
      L[2] = m2l_fma(-D[23], m, L[2]);
      L[3] = m2l_fma(-D[24], m, L[3]);
      L[4] = m2l_fma(D[36], m, L[4]);
      L[5] = m2l_fma(D[38], m, L[5]);
      L[6] = m2l_fma(D[39], m, L[6]);
      L[7] = m2l_fma(D[41], m, L[7]);
      L[8] = m2l_fma(D[42], m, L[8]);
      L[9] = m2l_fma(D[43], m, L[9]);
    }
    { const T m = __ldg(Ms + 12);
      L[1] = m2l_fma(-D[22], m, L[1]);
      L[2] = m2l_fma(-D[24], m, L[2]);
      L[3] = m2l_fma(-D[25], m, L[3]);
      L[4] = m2l_fma(D[37], m, L[4]);
      L[5] = m2l_fma(D[39], m, L[5]);
      L[6] = m2l_fma(D[40], m, L[6]);
      L[7] = m2l_fma(D[42], m, L[7]);
      L[8] = m2l_fma(D[43], m, L[8]);
      L[9] = m2l_fma(D[44], m, L[9]);
    }
    { const T m = __ldg(Ms + 13);
      L[1] = m2l_fma(-D[23], m, L[1]);
      L[2] = m2l_fma(-D[26], m, L[2]);
      L[3] = m2l_fma(-D[27], m, L[3]);
      L[4] = m2l_fma(D[38], m, L[4]);
      L[5] = m2l_fma(D[41], m, L[5]);
      L[6] = m2l_fma(D[42], m, L[6]);
      L[7] = m2l_fma(D[45], m, L[7]);
      L[8] = m2l_fma(D[46], m, L[8]);
      L[9] = m2l_fma(D[47], m, L[9]);
    }
    { const T m = __ldg(Ms + 14);
      L[1] = m2l_fma(-D[24], m, L[1]);
      L[2] = m2l_fma(-D[27], m, L[2]);
      L[3] = m2l_fma(-D[28], m, L[3]);
      L[4] = m2l_fma(D[39], m, L[4]);
      L[5] = m2l_fma(D[42], m, L[5]);
      L[6] = m2l_fma(D[43], m, L[6]);
      L[7] = m2l_fma(D[46], m, L[7]);
      L[8] = m2l_fma(D[47], m, L[8]);
      L[9] = m2l_fma(D[48], m, L[9]);
    }
    { const T m = __ldg(Ms + 15);
      L[1] = m2l_fma(-D[25], m, L[1]);
      L[2] = m2l_fma(-D[28], m, L[2]);
      L[3] = m2l_fma(-D[29], m, L[3]);
      L[4] = m2l_fma(D[40], m, L[4]);
      L[5] = m2l_fma(D[43], m, L[5]);
      L[6] = m2l_fma(D[44], m, L[6]);
      L[7] = m2l_fma(D[47], m, L[7]);
      L[8] = m2l_fma(D[48], m, L[8]);
      L[9] = m2l_fma(D[49], m, L[9]);
    }
    { const T m = __ldg(Ms + 16);
      L[1] = m2l_fma(-D[26], m, L[1]);
      L[2] = m2l_fma(-D[30], m, L[2]);
      L[3] = m2l_fma(-D[31], m, L[3]);
      L[4] = m2l_fma(D[41], m, L[4]);
      L[5] = m2l_fma(D[45], m, L[5]);
      L[6] = m2l_fma(D[46], m, L[6]);
      L[7] = m2l_fma(D[50], m, L[7]);
      L[8] = m2l_fma(D[51], m, L[8]);
      L[9] = m2l_fma(D[52], m, L[9]);
    }
    { const T m = __ldg(Ms + 17);
      L[1] = m2l_fma(-D[27], m, L[1]);
      L[2] = m2l_fma(-D[31], m, L[2]);
      L[3] = m2l_fma(-D[32], m, L[3]);
      L[4] = m2l_fma(D[42], m, L[4]);
      L[5] = m2l_fma(D[46], m, L[5]);
      L[6] = m2l_fma(D[47], m, L[6]);
      L[7] = m2l_fma(D[51], m, L[7]);
      L[8] = m2l_fma(D[52], m, L[8]);
      L[9] = m2l_fma(D[53], m, L[9]);
    }
    { const T m = __ldg(Ms + 18);
      L[1] = m2l_fma(-D[28], m, L[1]);
      L[2] = m2l_fma(-D[32], m, L[2]);
      L[3] = m2l_fma(-D[33], m, L[3]);
      L[4] = m2l_fma(D[43], m, L[4]);
      L[5] = m2l_fma(D[47], m, L[5]);
      L[6] = m2l_fma(D[48], m, L[6]);
      L[7] = m2l_fma(D[52], m, L[7]);
      L[8] = m2l_fma(D[53], m, L[8]);
      L[9] = m2l_fma(D[54], m, L[9]);
    }
    { const T m = __ldg(Ms + 19);
      L[1] = m2l_fma(-D[29], m, L[1]);
      L[2] = m2l_fma(-D[33], m, L[2]);
      L[3] = m2l_fma(-D[34], m, L[3]);
      L[4] = m2l_fma(D[44], m, L[4]);
      L[5] = m2l_fma(D[48], m, L[5]);
      L[6] = m2l_fma(D[49], m, L[6]);
      L[7] = m2l_fma(D[53], m, L[7]);
      L[8] = m2l_fma(D[54], m, L[8]);
      L[9] = m2l_fma(D[55], m, L[9]);
    }
    { const T m = __ldg(Ms + 20);
      L[1] = m2l_fma(-D[35], m, L[1]);
      L[2] = m2l_fma(-D[36], m, L[2]);
      L[3] = m2l_fma(-D[37], m, L[3]);
    }
    { const T m = __ldg(Ms + 21);
      L[1] = m2l_fma(-D[36], m, L[1]);
      L[2] = m2l_fma(-D[38], m, L[2]);
      L[3] = m2l_fma(-D[39], m, L[3]);
    }
    { const T m = __ldg(Ms + 22);
      L[1] = m2l_fma(-D[37], m, L[1]);
      L[2] = m2l_fma(-D[39], m, L[2]);
      L[3] = m2l_fma(-D[40], m, L[3]);
    }
    { const T m = __ldg(Ms + 23);
      L[1] = m2l_fma(-D[38], m, L[1]);
      L[2] = m2l_fma(-D[41], m, L[2]);
      L[3] = m2l_fma(-D[42], m, L[3]);
    }
    { const T m = __ldg(Ms + 24);
      L[1] = m2l_fma(-D[39], m, L[1]);
      L[2] = m2l_fma(-D[42], m, L[2]);
      L[3] = m2l_fma(-D[43], m, L[3]);
    }
    { const T m = __ldg(Ms + 25);
      L[1] = m2l_fma(-D[40], m, L[1]);
      L[2] = m2l_fma(-D[43], m, L[2]);
      L[3] = m2l_fma(-D[44], m, L[3]);
    }
    { const T m = __ldg(Ms + 26);
      L[1] = m2l_fma(-D[41], m, L[1]);
      L[2] = m2l_fma(-D[45], m, L[2]);
      L[3] = m2l_fma(-D[46], m, L[3]);
    }
    { const T m = __ldg(Ms + 27);
      L[1] = m2l_fma(-D[42], m, L[1]);
      L[2] = m2l_fma(-D[46], m, L[2]);
      L[3] = m2l_fma(-D[47], m, L[3]);
    }
    { const T m = __ldg(Ms + 28);
      L[1] = m2l_fma(-D[43], m, L[1]);
      L[2] = m2l_fma(-D[47], m, L[2]);
      L[3] = m2l_fma(-D[48], m, L[3]);
    }
    { const T m = __ldg(Ms + 29);
      L[1] = m2l_fma(-D[44], m, L[1]);
      L[2] = m2l_fma(-D[48], m, L[2]);
      L[3] = m2l_fma(-D[49], m, L[3]);
    }
    { const T m = __ldg(Ms + 30);
      L[1] = m2l_fma(-D[45], m, L[1]);
      L[2] = m2l_fma(-D[50], m, L[2]);
      L[3] = m2l_fma(-D[51], m, L[3]);
    }
    { const T m = __ldg(Ms + 31);
      L[1] = m2l_fma(-D[46], m, L[1]);
      L[2] = m2l_fma(-D[51], m, L[2]);
      L[3] = m2l_fma(-D[52], m, L[3]);
    }
    { const T m = __ldg(Ms + 32);
      L[1] = m2l_fma(-D[47], m, L[1]);
      L[2] = m2l_fma(-D[52], m, L[2]);
      L[3] = m2l_fma(-D[53], m, L[3]);
    }
    { const T m = __ldg(Ms + 33);
      L[1] = m2l_fma(-D[48], m, L[1]);
      L[2] = m2l_fma(-D[53], m, L[2]);
      L[3] = m2l_fma(-D[54], m, L[3]);
    }
    { const T m = __ldg(Ms + 34);
      L[1] = m2l_fma(-D[49], m, L[1]);
      L[2] = m2l_fma(-D[54], m, L[2]);
      L[3] = m2l_fma(-D[55], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_dtensor_6(T dx, T dy, T dz, T soft2, T (&D)[84])
{
    const T s2 = m2l_fma(dx, dx, m2l_fma(dy, dy, m2l_fma(dz, dz, soft2)));
    const T si = m2l_rsqrt(s2);
    const T si2 = si * si;
    const T f0 = -si;
    const T f1 = T(-1) * f0 * si2;
    const T f2 = T(-3) * f1 * si2;
    const T f3 = T(-5) * f2 * si2;
    const T f4 = T(-7) * f3 * si2;
    const T f5 = T(-9) * f4 * si2;
    const T f6 = T(-11) * f5 * si2;
    const T r_0_0 = f0;
    const T r_1_0 = f1;
    const T r_2_0 = f2;
    const T r_3_0 = f3;
    const T r_4_0 = f4;
    const T r_5_0 = f5;
    const T r_6_0 = f6;
    const T r_0_1 = dx * r_1_0;
    const T r_1_1 = dx * r_2_0;
    const T r_2_1 = dx * r_3_0;
    const T r_3_1 = dx * r_4_0;
    const T r_4_1 = dx * r_5_0;
    const T r_5_1 = dx * r_6_0;
    const T r_0_2 = dy * r_1_0;
    const T r_1_2 = dy * r_2_0;
    const T r_2_2 = dy * r_3_0;
    const T r_3_2 = dy * r_4_0;
    const T r_4_2 = dy * r_5_0;
    const T r_5_2 = dy * r_6_0;
    const T r_0_3 = dz * r_1_0;
    const T r_1_3 = dz * r_2_0;
    const T r_2_3 = dz * r_3_0;
    const T r_3_3 = dz * r_4_0;
    const T r_4_3 = dz * r_5_0;
    const T r_5_3 = dz * r_6_0;
    const T r_0_4 = m2l_fma(T(1), r_1_0, dx * r_1_1);
    const T r_1_4 = m2l_fma(T(1), r_2_0, dx * r_2_1);
    const T r_2_4 = m2l_fma(T(1), r_3_0, dx * r_3_1);
    const T r_3_4 = m2l_fma(T(1), r_4_0, dx * r_4_1);
    const T r_4_4 = m2l_fma(T(1), r_5_0, dx * r_5_1);
    const T r_0_5 = dx * r_1_2;
    const T r_1_5 = dx * r_2_2;
    const T r_2_5 = dx * r_3_2;
    const T r_3_5 = dx * r_4_2;
    const T r_4_5 = dx * r_5_2;
    const T r_0_6 = dx * r_1_3;
    const T r_1_6 = dx * r_2_3;
    const T r_2_6 = dx * r_3_3;
    const T r_3_6 = dx * r_4_3;
    const T r_4_6 = dx * r_5_3;
    const T r_0_7 = m2l_fma(T(1), r_1_0, dy * r_1_2);
    const T r_1_7 = m2l_fma(T(1), r_2_0, dy * r_2_2);
    const T r_2_7 = m2l_fma(T(1), r_3_0, dy * r_3_2);
    const T r_3_7 = m2l_fma(T(1), r_4_0, dy * r_4_2);
    const T r_4_7 = m2l_fma(T(1), r_5_0, dy * r_5_2);
    const T r_0_8 = dy * r_1_3;
    const T r_1_8 = dy * r_2_3;
    const T r_2_8 = dy * r_3_3;
    const T r_3_8 = dy * r_4_3;
    const T r_4_8 = dy * r_5_3;
    const T r_0_9 = m2l_fma(T(1), r_1_0, dz * r_1_3);
    const T r_1_9 = m2l_fma(T(1), r_2_0, dz * r_2_3);
    const T r_2_9 = m2l_fma(T(1), r_3_0, dz * r_3_3);
    const T r_3_9 = m2l_fma(T(1), r_4_0, dz * r_4_3);
    const T r_4_9 = m2l_fma(T(1), r_5_0, dz * r_5_3);
    const T r_0_10 = m2l_fma(T(2), r_1_1, dx * r_1_4);
    const T r_1_10 = m2l_fma(T(2), r_2_1, dx * r_2_4);
    const T r_2_10 = m2l_fma(T(2), r_3_1, dx * r_3_4);
    const T r_3_10 = m2l_fma(T(2), r_4_1, dx * r_4_4);
    const T r_0_11 = m2l_fma(T(1), r_1_2, dx * r_1_5);
    const T r_1_11 = m2l_fma(T(1), r_2_2, dx * r_2_5);
    const T r_2_11 = m2l_fma(T(1), r_3_2, dx * r_3_5);
    const T r_3_11 = m2l_fma(T(1), r_4_2, dx * r_4_5);
    const T r_0_12 = m2l_fma(T(1), r_1_3, dx * r_1_6);
    const T r_1_12 = m2l_fma(T(1), r_2_3, dx * r_2_6);
    const T r_2_12 = m2l_fma(T(1), r_3_3, dx * r_3_6);
    const T r_3_12 = m2l_fma(T(1), r_4_3, dx * r_4_6);
    const T r_0_13 = dx * r_1_7;
    const T r_1_13 = dx * r_2_7;
    const T r_2_13 = dx * r_3_7;
    const T r_3_13 = dx * r_4_7;
    const T r_0_14 = dx * r_1_8;
    const T r_1_14 = dx * r_2_8;
    const T r_2_14 = dx * r_3_8;
    const T r_3_14 = dx * r_4_8;
    const T r_0_15 = dx * r_1_9;
    const T r_1_15 = dx * r_2_9;
    const T r_2_15 = dx * r_3_9;
    const T r_3_15 = dx * r_4_9;
    const T r_0_16 = m2l_fma(T(2), r_1_2, dy * r_1_7);
    const T r_1_16 = m2l_fma(T(2), r_2_2, dy * r_2_7);
    const T r_2_16 = m2l_fma(T(2), r_3_2, dy * r_3_7);
    const T r_3_16 = m2l_fma(T(2), r_4_2, dy * r_4_7);
    const T r_0_17 = m2l_fma(T(1), r_1_3, dy * r_1_8);
    const T r_1_17 = m2l_fma(T(1), r_2_3, dy * r_2_8);
    const T r_2_17 = m2l_fma(T(1), r_3_3, dy * r_3_8);
    const T r_3_17 = m2l_fma(T(1), r_4_3, dy * r_4_8);
    const T r_0_18 = dy * r_1_9;
    const T r_1_18 = dy * r_2_9;
    const T r_2_18 = dy * r_3_9;
    const T r_3_18 = dy * r_4_9;
    const T r_0_19 = m2l_fma(T(2), r_1_3, dz * r_1_9);
    const T r_1_19 = m2l_fma(T(2), r_2_3, dz * r_2_9);
    const T r_2_19 = m2l_fma(T(2), r_3_3, dz * r_3_9);
    const T r_3_19 = m2l_fma(T(2), r_4_3, dz * r_4_9);
    const T r_0_20 = m2l_fma(T(3), r_1_4, dx * r_1_10);
    const T r_1_20 = m2l_fma(T(3), r_2_4, dx * r_2_10);
    const T r_2_20 = m2l_fma(T(3), r_3_4, dx * r_3_10);
    const T r_0_21 = m2l_fma(T(2), r_1_5, dx * r_1_11);
    const T r_1_21 = m2l_fma(T(2), r_2_5, dx * r_2_11);
    const T r_2_21 = m2l_fma(T(2), r_3_5, dx * r_3_11);
    const T r_0_22 = m2l_fma(T(2), r_1_6, dx * r_1_12);
    const T r_1_22 = m2l_fma(T(2), r_2_6, dx * r_2_12);
    const T r_2_22 = m2l_fma(T(2), r_3_6, dx * r_3_12);
    const T r_0_23 = m2l_fma(T(1), r_1_7, dx * r_1_13);
    const T r_1_23 = m2l_fma(T(1), r_2_7, dx * r_2_13);
    const T r_2_23 = m2l_fma(T(1), r_3_7, dx * r_3_13);
    const T r_0_24 = m2l_fma(T(1), r_1_8, dx * r_1_14);
    const T r_1_24 = m2l_fma(T(1), r_2_8, dx * r_2_14);
    const T r_2_24 = m2l_fma(T(1), r_3_8, dx * r_3_14);
    const T r_0_25 = m2l_fma(T(1), r_1_9, dx * r_1_15);
    const T r_1_25 = m2l_fma(T(1), r_2_9, dx * r_2_15);
    const T r_2_25 = m2l_fma(T(1), r_3_9, dx * r_3_15);
    const T r_0_26 = dx * r_1_16;
    const T r_1_26 = dx * r_2_16;
    const T r_2_26 = dx * r_3_16;
    const T r_0_27 = dx * r_1_17;
    const T r_1_27 = dx * r_2_17;
    const T r_2_27 = dx * r_3_17;
    const T r_0_28 = dx * r_1_18;
    const T r_1_28 = dx * r_2_18;
    const T r_2_28 = dx * r_3_18;
    const T r_0_29 = dx * r_1_19;
    const T r_1_29 = dx * r_2_19;
    const T r_2_29 = dx * r_3_19;
    const T r_0_30 = m2l_fma(T(3), r_1_7, dy * r_1_16);
    const T r_1_30 = m2l_fma(T(3), r_2_7, dy * r_2_16);
    const T r_2_30 = m2l_fma(T(3), r_3_7, dy * r_3_16);
    const T r_0_31 = m2l_fma(T(2), r_1_8, dy * r_1_17);
    const T r_1_31 = m2l_fma(T(2), r_2_8, dy * r_2_17);
    const T r_2_31 = m2l_fma(T(2), r_3_8, dy * r_3_17);
    const T r_0_32 = m2l_fma(T(1), r_1_9, dy * r_1_18);
    const T r_1_32 = m2l_fma(T(1), r_2_9, dy * r_2_18);
    const T r_2_32 = m2l_fma(T(1), r_3_9, dy * r_3_18);
    const T r_0_33 = dy * r_1_19;
    const T r_1_33 = dy * r_2_19;
    const T r_2_33 = dy * r_3_19;
    const T r_0_34 = m2l_fma(T(3), r_1_9, dz * r_1_19);
    const T r_1_34 = m2l_fma(T(3), r_2_9, dz * r_2_19);
    const T r_2_34 = m2l_fma(T(3), r_3_9, dz * r_3_19);
    const T r_0_35 = m2l_fma(T(4), r_1_10, dx * r_1_20);
    const T r_1_35 = m2l_fma(T(4), r_2_10, dx * r_2_20);
    const T r_0_36 = m2l_fma(T(3), r_1_11, dx * r_1_21);
    const T r_1_36 = m2l_fma(T(3), r_2_11, dx * r_2_21);
    const T r_0_37 = m2l_fma(T(3), r_1_12, dx * r_1_22);
    const T r_1_37 = m2l_fma(T(3), r_2_12, dx * r_2_22);
    const T r_0_38 = m2l_fma(T(2), r_1_13, dx * r_1_23);
    const T r_1_38 = m2l_fma(T(2), r_2_13, dx * r_2_23);
    const T r_0_39 = m2l_fma(T(2), r_1_14, dx * r_1_24);
    const T r_1_39 = m2l_fma(T(2), r_2_14, dx * r_2_24);
    const T r_0_40 = m2l_fma(T(2), r_1_15, dx * r_1_25);
    const T r_1_40 = m2l_fma(T(2), r_2_15, dx * r_2_25);
    const T r_0_41 = m2l_fma(T(1), r_1_16, dx * r_1_26);
    const T r_1_41 = m2l_fma(T(1), r_2_16, dx * r_2_26);
    const T r_0_42 = m2l_fma(T(1), r_1_17, dx * r_1_27);
    const T r_1_42 = m2l_fma(T(1), r_2_17, dx * r_2_27);
    const T r_0_43 = m2l_fma(T(1), r_1_18, dx * r_1_28);
    const T r_1_43 = m2l_fma(T(1), r_2_18, dx * r_2_28);
    const T r_0_44 = m2l_fma(T(1), r_1_19, dx * r_1_29);
    const T r_1_44 = m2l_fma(T(1), r_2_19, dx * r_2_29);
    const T r_0_45 = dx * r_1_30;
    const T r_1_45 = dx * r_2_30;
    const T r_0_46 = dx * r_1_31;
    const T r_1_46 = dx * r_2_31;
    const T r_0_47 = dx * r_1_32;
    const T r_1_47 = dx * r_2_32;
    const T r_0_48 = dx * r_1_33;
    const T r_1_48 = dx * r_2_33;
    const T r_0_49 = dx * r_1_34;
    const T r_1_49 = dx * r_2_34;
    const T r_0_50 = m2l_fma(T(4), r_1_16, dy * r_1_30);
    const T r_1_50 = m2l_fma(T(4), r_2_16, dy * r_2_30);
    const T r_0_51 = m2l_fma(T(3), r_1_17, dy * r_1_31);
    const T r_1_51 = m2l_fma(T(3), r_2_17, dy * r_2_31);
    const T r_0_52 = m2l_fma(T(2), r_1_18, dy * r_1_32);
    const T r_1_52 = m2l_fma(T(2), r_2_18, dy * r_2_32);
    const T r_0_53 = m2l_fma(T(1), r_1_19, dy * r_1_33);
    const T r_1_53 = m2l_fma(T(1), r_2_19, dy * r_2_33);
    const T r_0_54 = dy * r_1_34;
    const T r_1_54 = dy * r_2_34;
    const T r_0_55 = m2l_fma(T(4), r_1_19, dz * r_1_34);
    const T r_1_55 = m2l_fma(T(4), r_2_19, dz * r_2_34);
    const T r_0_56 = m2l_fma(T(5), r_1_20, dx * r_1_35);
    const T r_0_57 = m2l_fma(T(4), r_1_21, dx * r_1_36);
    const T r_0_58 = m2l_fma(T(4), r_1_22, dx * r_1_37);
    const T r_0_59 = m2l_fma(T(3), r_1_23, dx * r_1_38);
    const T r_0_60 = m2l_fma(T(3), r_1_24, dx * r_1_39);
    const T r_0_61 = m2l_fma(T(3), r_1_25, dx * r_1_40);
    const T r_0_62 = m2l_fma(T(2), r_1_26, dx * r_1_41);
    const T r_0_63 = m2l_fma(T(2), r_1_27, dx * r_1_42);
    const T r_0_64 = m2l_fma(T(2), r_1_28, dx * r_1_43);
    const T r_0_65 = m2l_fma(T(2), r_1_29, dx * r_1_44);
    const T r_0_66 = m2l_fma(T(1), r_1_30, dx * r_1_45);
    const T r_0_67 = m2l_fma(T(1), r_1_31, dx * r_1_46);
    const T r_0_68 = m2l_fma(T(1), r_1_32, dx * r_1_47);
    const T r_0_69 = m2l_fma(T(1), r_1_33, dx * r_1_48);
    const T r_0_70 = m2l_fma(T(1), r_1_34, dx * r_1_49);
    const T r_0_71 = dx * r_1_50;
    const T r_0_72 = dx * r_1_51;
    const T r_0_73 = dx * r_1_52;
    const T r_0_74 = dx * r_1_53;
    const T r_0_75 = dx * r_1_54;
    const T r_0_76 = dx * r_1_55;
    const T r_0_77 = m2l_fma(T(5), r_1_30, dy * r_1_50);
    const T r_0_78 = m2l_fma(T(4), r_1_31, dy * r_1_51);
    const T r_0_79 = m2l_fma(T(3), r_1_32, dy * r_1_52);
    const T r_0_80 = m2l_fma(T(2), r_1_33, dy * r_1_53);
    const T r_0_81 = m2l_fma(T(1), r_1_34, dy * r_1_54);
    const T r_0_82 = dy * r_1_55;
    const T r_0_83 = m2l_fma(T(5), r_1_34, dz * r_1_55);
    D[0] = r_0_0;
    D[1] = r_0_1;
    D[2] = r_0_2;
    D[3] = r_0_3;
    D[4] = r_0_4;
    D[5] = r_0_5;
    D[6] = r_0_6;
    D[7] = r_0_7;
    D[8] = r_0_8;
    D[9] = r_0_9;
    D[10] = r_0_10;
    D[11] = r_0_11;
    D[12] = r_0_12;
    D[13] = r_0_13;
    D[14] = r_0_14;
    D[15] = r_0_15;
    D[16] = r_0_16;
    D[17] = r_0_17;
    D[18] = r_0_18;
    D[19] = r_0_19;
    D[20] = r_0_20;
    D[21] = r_0_21;
    D[22] = r_0_22;
    D[23] = r_0_23;
    D[24] = r_0_24;
    D[25] = r_0_25;
    D[26] = r_0_26;
    D[27] = r_0_27;
    D[28] = r_0_28;
    D[29] = r_0_29;
    D[30] = r_0_30;
    D[31] = r_0_31;
    D[32] = r_0_32;
    D[33] = r_0_33;
    D[34] = r_0_34;
    D[35] = r_0_35;
    D[36] = r_0_36;
    D[37] = r_0_37;
    D[38] = r_0_38;
    D[39] = r_0_39;
    D[40] = r_0_40;
    D[41] = r_0_41;
    D[42] = r_0_42;
    D[43] = r_0_43;
    D[44] = r_0_44;
    D[45] = r_0_45;
    D[46] = r_0_46;
    D[47] = r_0_47;
    D[48] = r_0_48;
    D[49] = r_0_49;
    D[50] = r_0_50;
    D[51] = r_0_51;
    D[52] = r_0_52;
    D[53] = r_0_53;
    D[54] = r_0_54;
    D[55] = r_0_55;
    D[56] = r_0_56;
    D[57] = r_0_57;
    D[58] = r_0_58;
    D[59] = r_0_59;
    D[60] = r_0_60;
    D[61] = r_0_61;
    D[62] = r_0_62;
    D[63] = r_0_63;
    D[64] = r_0_64;
    D[65] = r_0_65;
    D[66] = r_0_66;
    D[67] = r_0_67;
    D[68] = r_0_68;
    D[69] = r_0_69;
    D[70] = r_0_70;
    D[71] = r_0_71;
    D[72] = r_0_72;
    D[73] = r_0_73;
    D[74] = r_0_74;
    D[75] = r_0_75;
    D[76] = r_0_76;
    D[77] = r_0_77;
    D[78] = r_0_78;
    D[79] = r_0_79;
    D[80] = r_0_80;
    D[81] = r_0_81;
    D[82] = r_0_82;
    D[83] = r_0_83;
}

template <class T> __device__ __forceinline__ void m2l_side_a_6(const T (&D)[84], const T *__restrict__ Ms, T rho, T (&L)[84])
{
    T rp = T(1);
    { const T m = __ldg(Ms + 0) * rp;
      L[0] = D[0] * m;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[9] * m;
      L[10] = D[10] * m;
      L[11] = D[11] * m;
      L[12] = D[12] * m;
      L[13] = D[13] * m;
      L[14] = D[14] * m;
      L[15] = D[15] * m;
      L[16] = D[16] * m;
      L[17] = D[17] * m;
      L[18] = D[18] * m;
      L[19] = D[19] * m;
      L[20] = D[20] * m;
      L[21] = D[21] * m;
      L[22] = D[22] * m;
      L[23] = D[23] * m;
      L[24] = D[24] * m;
      L[25] = D[25] * m;
      L[26] = D[26] * m;
      L[27] = D[27] * m;
      L[28] = D[28] * m;
      L[29] = D[29] * m;
      L[30] = D[30] * m;
      L[31] = D[31] * m;
      L[32] = D[32] * m;
      L[33] = D[33] * m;
      L[34] = D[34] * m;
      L[35] = D[35] * m;
      L[36] = D[36] * m;
      L[37] = D[37] * m;
      L[38] = D[38] * m;
      L[39] = D[39] * m;
      L[40] = D[40] * m;
      L[41] = D[41] * m;
      L[42] = D[42] * m;
      L[43] = D[43] * m;
      L[44] = D[44] * m;
      L[45] = D[45] * m;
      L[46] = D[46] * m;
      L[47] = D[47] * m;
      L[48] = D[48] * m;
      L[49] = D[49] * m;
      L[50] = D[50] * m;
      L[51] = D[51] * m;
      L[52] = D[52] * m;
      L[53] = D[53] * m;
      L[54] = D[54] * m;
      L[55] = D[55] * m;
      L[56] = D[56] * m;
      L[57] = D[57] * m;
      L[58] = D[58] * m;
      L[59] = D[59] * m;
      L[60] = D[60] * m;
      L[61] = D[61] * m;
      L[62] = D[62] * m;
      L[63] = D[63] * m;
      L[64] = D[64] * m;
      L[65] = D[65] * m;
      L[66] = D[66] * m;
      L[67] = D[67] * m;
      L[68] = D[68] * m;
      L[69] = D[69] * m;
      L[70] = D[70] * m;
      L[71] = D[71] * m;
      L[72] = D[72] * m;
      L[73] = D[73] * m;
      L[74] = D[74] * m;
      L[75] = D[75] * m;
      L[76] = D[76] * m;
      L[77] = D[77] * m;
      L[78] = D[78] * m;
      L[79] = D[79] * m;
      L[80] = D[80] * m;
      L[81] = D[81] * m;
      L[82] = D[82] * m;
      L[83] = D[83] * m;
    }
    rp *= rho;
    { const T m = -__ldg(Ms + 1) * rp;
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[15], m, L[9]);
      L[10] = m2l_fma(D[20], m, L[10]);
      L[11] = m2l_fma(D[21], m, L[11]);
      L[12] = m2l_fma(D[22], m, L[12]);
      L[13] = m2l_fma(D[23], m, L[13]);
      L[14] = m2l_fma(D[24], m, L[14]);
      L[15] = m2l_fma(D[25], m, L[15]);
      L[16] = m2l_fma(D[26], m, L[16]);
      L[17] = m2l_fma(D[27], m, L[17]);
      L[18] = m2l_fma(D[28], m, L[18]);
      L[19] = m2l_fma(D[29], m, L[19]);
      L[20] = m2l_fma(D[35], m, L[20]);
      L[21] = m2l_fma(D[36], m, L[21]);
      L[22] = m2l_fma(D[37], m, L[22]);
      L[23] = m2l_fma(D[38], m, L[23]);
      L[24] = m2l_fma(D[39], m, L[24]);
      L[25] = m2l_fma(D[40], m, L[25]);
      L[26] = m2l_fma(D[41], m, L[26]);
      L[27] = m2l_fma(D[42], m, L[27]);
      L[28] = m2l_fma(D[43], m, L[28]);
      L[29] = m2l_fma(D[44], m, L[29]);
      L[30] = m2l_fma(D[45], m, L[30]);
      L[31] = m2l_fma(D[46], m, L[31]);
      L[32] = m2l_fma(D[47], m, L[32]);
      L[33] = m2l_fma(D[48], m, L[33]);
      L[34] = m2l_fma(D[49], m, L[34]);
      L[35] = m2l_fma(D[56], m, L[35]);
      L[36] = m2l_fma(D[57], m, L[36]);
      L[37] = m2l_fma(D[58], m, L[37]);
      L[38] = m2l_fma(D[59], m, L[38]);
      L[39] = m2l_fma(D[60], m, L[39]);
      L[40] = m2l_fma(D[61], m, L[40]);
      L[41] = m2l_fma(D[62], m, L[41]);
      L[42] = m2l_fma(D[63], m, L[42]);
      L[43] = m2l_fma(D[64], m, L[43]);
      L[44] = m2l_fma(D[65], m, L[44]);
      L[45] = m2l_fma(D[66], m, L[45]);
      L[46] = m2l_fma(D[67], m, L[46]);
      L[47] = m2l_fma(D[68], m, L[47]);
      L[48] = m2l_fma(D[69], m, L[48]);
      L[49] = m2l_fma(D[70], m, L[49]);
      L[50] = m2l_fma(D[71], m, L[50]);
      L[51] = m2l_fma(D[72], m, L[51]);
      L[52] = m2l_fma(D[73], m, L[52]);
      L[53] = m2l_fma(D[74], m, L[53]);
      L[54] = m2l_fma(D[75], m, L[54]);
      L[55] = m2l_fma(D[76], m, L[55]);
    }
    { const T m = -__ldg(Ms + 2) * rp;
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[18], m, L[9]);
      L[10] = m2l_fma(D[21], m, L[10]);
      L[11] = m2l_fma(D[23], m, L[11]);
      L[12] = m2l_fma(D[24], m, L[12]);
      L[13] = m2l_fma(D[26], m, L[13]);
      L[14] = m2l_fma(D[27], m, L[14]);
      L[15] = m2l_fma(D[28], m, L[15]);
      L[16] = m2l_fma(D[30], m, L[16]);
      L[17] = m2l_fma(D[31], m, L[17]);
      L[18] = m2l_fma(D[32], m, L[18]);
      L[19] = m2l_fma(D[33], m, L[19]);
      L[20] = m2l_fma(D[36], m, L[20]);
      L[21] = m2l_fma(D[38], m, L[21]);
      L[22] = m2l_fma(D[39], m, L[22]);
      L[23] = m2l_fma(D[41], m, L[23]);
      L[24] = m2l_fma(D[42], m, L[24]);
      L[25] = m2l_fma(D[43], m, L[25]);
      L[26] = m2l_fma(D[45], m, L[26]);
      L[27] = m2l_fma(D[46], m, L[27]);
      L[28] = m2l_fma(D[47], m, L[28]);
      L[29] = m2l_fma(D[48], m, L[29]);
      L[30] = m2l_fma(D[50], m, L[30]);
      L[31] = m2l_fma(D[51], m, L[31]);
      L[32] = m2l_fma(D[52], m, L[32]);
      L[33] = m2l_fma(D[53], m, L[33]);
      L[34] = m2l_fma(D[54], m, L[34]);
      L[35] = m2l_fma(D[57], m, L[35]);
      L[36] = m2l_fma(D[59], m, L[36]);
      L[37] = m2l_fma(D[60], m, L[37]);
      L[38] = m2l_fma(D[62], m, L[38]);
      L[39] = m2l_fma(D[63], m, L[39]);
      L[40] = m2l_fma(D[64], m, L[40]);
      L[41] = m2l_fma(D[66], m, L[41]);
      L[42] = m2l_fma(D[67], m, L[42]);
      L[43] = m2l_fma(D[68], m, L[43]);
      L[44] = m2l_fma(D[69], m, L[44]);
      L[45] = m2l_fma(D[71], m, L[45]);
      L[46] = m2l_fma(D[72], m, L[46]);
      L[47] = m2l_fma(D[73], m, L[47]);
      L[48] = m2l_fma(D[74], m, L[48]);
      L[49] = m2l_fma(D[75], m, L[49]);
      L[50] = m2l_fma(D[77], m, L[50]);
      L[51] = m2l_fma(D[78], m, L[51]);
      L[52] = m2l_fma(D[79], m, L[52]);
      L[53] = m2l_fma(D[80], m, L[53]);
      L[54] = m2l_fma(D[81], m, L[54]);
      L[55] = m2l_fma(D[82], m, L[55]);
    }
    { const T m = -__ldg(Ms + 3) * rp;
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(D[22], m, L[10]);
      L[11] = m2l_fma(D[24], m, L[11]);
      L[12] = m2l_fma(D[25], m, L[12]);
      L[13] = m2l_fma(D[27], m, L[13]);
      L[14] = m2l_fma(D[28], m, L[14]);
      L[15] = m2l_fma(D[29], m, L[15]);
      L[16] = m2l_fma(D[31], m, L[16]);
      L[17] = m2l_fma(D[32], m, L[17]);
      L[18] = m2l_fma(D[33], m, L[18]);
      L[19] = m2l_fma(D[34], m, L[19]);
      L[20] = m2l_fma(D[37], m, L[20]);
      L[21] = m2l_fma(D[39], m, L[21]);
      L[22] = m2l_fma(D[40], m, L[22]);
      L[23] = m2l_fma(D[42], m, L[23]);
      L[24] = m2l_fma(D[43], m, L[24]);
      L[25] = m2l_fma(D[44], m, L[25]);
      L[26] = m2l_fma(D[46], m, L[26]);
      L[27] = m2l_fma(D[47], m, L[27]);
      L[28] = m2l_fma(D[48], m, L[28]);
      L[29] = m2l_fma(D[49], m, L[29]);
      L[30] = m2l_fma(D[51], m, L[30]);
      L[31] = m2l_fma(D[52], m, L[31]);
      L[32] = m2l_fma(D[53], m, L[32]);
      L[33] = m2l_fma(D[54], m, L[33]);
      L[34] = m2l_fma(D[55], m, L[34]);
      L[35] = m2l_fma(D[58], m, L[35]);
      L[36] = m2l_fma(D[60], m, L[36]);
      L[37] = m2l_fma(D[61], m, L[37]);
      L[38] = m2l_fma(D[63], m, L[38]);
      L[39] = m2l_fma(D[64], m, L[39]);
      L[40] = m2l_fma(D[65], m, L[40]);
      L[41] = m2l_fma(D[67], m, L[41]);
      L[42] = m2l_fma(D[68], m, L[42]);
      L[43] = m2l_fma(D[69], m, L[43]);
      L[44] = m2l_fma(D[70], m, L[44]);
      L[45] = m2l_fma(D[72], m, L[45]);
      L[46] = m2l_fma(D[73], m, L[46]);
      L[47] = m2l_fma(D[74], m, L[47]);
      L[48] = m2l_fma(D[75], m, L[48]);
      L[49] = m2l_fma(D[76], m, L[49]);
      L[50] = m2l_fma(D[78], m, L[50]);
      L[51] = m2l_fma(D[79], m, L[51]);
      L[52] = m2l_fma(D[80], m, L[52]);
      L[53] = m2l_fma(D[81], m, L[53]);
      L[54] = m2l_fma(D[82], m, L[54]);
      L[55] = m2l_fma(D[83], m, L[55]);
    }
    rp *= rho;
    { const T m = __ldg(Ms + 4) * rp;
      L[0] = m2l_fma(D[4], m, L[0]);
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[21], m, L[5]);
      L[6] = m2l_fma(D[22], m, L[6]);
      L[7] = m2l_fma(D[23], m, L[7]);
      L[8] = m2l_fma(D[24], m, L[8]);
      L[9] = m2l_fma(D[25], m, L[9]);
      L[10] = m2l_fma(D[35], m, L[10]);
      L[11] = m2l_fma(D[36], m, L[11]);
      L[12] = m2l_fma(D[37], m, L[12]);
      L[13] = m2l_fma(D[38], m, L[13]);
      L[14] = m2l_fma(D[39], m, L[14]);
      L[15] = m2l_fma(D[40], m, L[15]);
      L[16] = m2l_fma(D[41], m, L[16]);
      L[17] = m2l_fma(D[42], m, L[17]);
      L[18] = m2l_fma(D[43], m, L[18]);
      L[19] = m2l_fma(D[44], m, L[19]);
      L[20] = m2l_fma(D[56], m, L[20]);
      L[21] = m2l_fma(D[57], m, L[21]);
      L[22] = m2l_fma(D[58], m, L[22]);
      L[23] = m2l_fma(D[59], m, L[23]);
      L[24] = m2l_fma(D[60], m, L[24]);
      L[25] = m2l_fma(D[61], m, L[25]);
      L[26] = m2l_fma(D[62], m, L[26]);
      L[27] = m2l_fma(D[63], m, L[27]);
      L[28] = m2l_fma(D[64], m, L[28]);
      L[29] = m2l_fma(D[65], m, L[29]);
      L[30] = m2l_fma(D[66], m, L[30]);
      L[31] = m2l_fma(D[67], m, L[31]);
      L[32] = m2l_fma(D[68], m, L[32]);
      L[33] = m2l_fma(D[69], m, L[33]);
      L[34] = m2l_fma(D[70], m, L[34]);
    }
    { const T m = __ldg(Ms + 5) * rp;
      L[0] = m2l_fma(D[5], m, L[0]);
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(D[28], m, L[9]);
      L[10] = m2l_fma(D[36], m, L[10]);
      L[11] = m2l_fma(D[38], m, L[11]);
      L[12] = m2l_fma(D[39], m, L[12]);
      L[13] = m2l_fma(D[41], m, L[13]);
      L[14] = m2l_fma(D[42], m, L[14]);
      L[15] = m2l_fma(D[43], m, L[15]);
      L[16] = m2l_fma(D[45], m, L[16]);
      L[17] = m2l_fma(D[46], m, L[17]);
      L[18] = m2l_fma(D[47], m, L[18]);
      L[19] = m2l_fma(D[48], m, L[19]);
      L[20] = m2l_fma(D[57], m, L[20]);
      L[21] = m2l_fma(D[59], m, L[21]);
      L[22] = m2l_fma(D[60], m, L[22]);
      L[23] = m2l_fma(D[62], m, L[23]);
      L[24] = m2l_fma(D[63], m, L[24]);
      L[25] = m2l_fma(D[64], m, L[25]);
      L[26] = m2l_fma(D[66], m, L[26]);
      L[27] = m2l_fma(D[67], m, L[27]);
      L[28] = m2l_fma(D[68], m, L[28]);
      L[29] = m2l_fma(D[69], m, L[29]);
      L[30] = m2l_fma(D[71], m, L[30]);
      L[31] = m2l_fma(D[72], m, L[31]);
      L[32] = m2l_fma(D[73], m, L[32]);
      L[33] = m2l_fma(D[74], m, L[33]);
      L[34] = m2l_fma(D[75], m, L[34]);
    }
    { const T m = __ldg(Ms + 6) * rp;
      L[0] = m2l_fma(D[6], m, L[0]);
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[24], m, L[5]);
      L[6] = m2l_fma(D[25], m, L[6]);
      L[7] = m2l_fma(D[27], m, L[7]);
      L[8] = m2l_fma(D[28], m, L[8]);
      L[9] = m2l_fma(D[29], m, L[9]);
      L[10] = m2l_fma(D[37], m, L[10]);
      L[11] = m2l_fma(D[39], m, L[11]);
      L[12] = m2l_fma(D[40], m, L[12]);
      L[13] = m2l_fma(D[42], m, L[13]);
      L[14] = m2l_fma(D[43], m, L[14]);
      L[15] = m2l_fma(D[44], m, L[15]);
      L[16] = m2l_fma(D[46], m, L[16]);
      L[17] = m2l_fma(D[47], m, L[17]);
      L[18] = m2l_fma(D[48], m, L[18]);
      L[19] = m2l_fma(D[49], m, L[19]);
      L[20] = m2l_fma(D[58], m, L[20]);
      L[21] = m2l_fma(D[60], m, L[21]);
      L[22] = m2l_fma(D[61], m, L[22]);
      L[23] = m2l_fma(D[63], m, L[23]);
      L[24] = m2l_fma(D[64], m, L[24]);
      L[25] = m2l_fma(D[65], m, L[25]);
      L[26] = m2l_fma(D[67], m, L[26]);
      L[27] = m2l_fma(D[68], m, L[27]);
      L[28] = m2l_fma(D[69], m, L[28]);
      L[29] = m2l_fma(D[70], m, L[29]);
      L[30] = m2l_fma(D[72], m, L[30]);
      L[31] = m2l_fma(D[73], m, L[31]);
      L[32] = m2l_fma(D[74], m, L[32]);
      L[33] = m2l_fma(D[75], m, L[33]);
      L[34] = m2l_fma(D[76], m, L[34]);
    }
    { const T m = __ldg(Ms + 7) * rp;
      L[0] = m2l_fma(D[7], m, L[0]);
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[30], m, L[7]);
      L[8] = m2l_fma(D[31], m, L[8]);
      L[9] = m2l_fma(D[32], m, L[9]);
      L[10] = m2l_fma(D[38], m, L[10]);
      L[11] = m2l_fma(D[41], m, L[11]);
      L[12] = m2l_fma(D[42], m, L[12]);
      L[13] = m2l_fma(D[45], m, L[13]);
      L[14] = m2l_fma(D[46], m, L[14]);
      L[15] = m2l_fma(D[47], m, L[15]);
      L[16] = m2l_fma(D[50], m, L[16]);
      L[17] = m2l_fma(D[51], m, L[17]);
      L[18] = m2l_fma(D[52], m, L[18]);
      L[19] = m2l_fma(D[53], m, L[19]);
      L[20] = m2l_fma(D[59], m, L[20]);
      L[21] = m2l_fma(D[62], m, L[21]);
      L[22] = m2l_fma(D[63], m, L[22]);
      L[23] = m2l_fma(D[66], m, L[23]);
      L[24] = m2l_fma(D[67], m, L[24]);
      L[25] = m2l_fma(D[68], m, L[25]);
      L[26] = m2l_fma(D[71], m, L[26]);
      L[27] = m2l_fma(D[72], m, L[27]);
      L[28] = m2l_fma(D[73], m, L[28]);
      L[29] = m2l_fma(D[74], m, L[29]);
      L[30] = m2l_fma(D[77], m, L[30]);
      L[31] = m2l_fma(D[78], m, L[31]);
      L[32] = m2l_fma(D[79], m, L[32]);
      L[33] = m2l_fma(D[80], m, L[33]);
      L[34] = m2l_fma(D[81], m, L[34]);
    }
    { const T m = __ldg(Ms + 8) * rp;
      L[0] = m2l_fma(D[8], m, L[0]);
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
      L[4] = m2l_fma(D[24], m, L[4]);
      L[5] = m2l_fma(D[27], m, L[5]);
      L[6] = m2l_fma(D[28], m, L[6]);
      L[7] = m2l_fma(D[31], m, L[7]);
      L[8] = m2l_fma(D[32], m, L[8]);
      L[9] = m2l_fma(D[33], m, L[9]);
      L[10] = m2l_fma(D[39], m, L[10]);
      L[11] = m2l_fma(D[42], m, L[11]);
      L[12] = m2l_fma(D[43], m, L[12]);
      L[13] = m2l_fma(D[46], m, L[13]);
      L[14] = m2l_fma(D[47], m, L[14]);
      L[15] = m2l_fma(D[48], m, L[15]);
      L[16] = m2l_fma(D[51], m, L[16]);
      L[17] = m2l_fma(D[52], m, L[17]);
      L[18] = m2l_fma(D[53], m, L[18]);
      L[19] = m2l_fma(D[54], m, L[19]);
      L[20] = m2l_fma(D[60], m, L[20]);
      L[21] = m2l_fma(D[63], m, L[21]);
      L[22] = m2l_fma(D[64], m, L[22]);
      L[23] = m2l_fma(D[67], m, L[23]);
      L[24] = m2l_fma(D[68], m, L[24]);
      L[25] = m2l_fma(D[69], m, L[25]);
      L[26] = m2l_fma(D[72], m, L[26]);
      L[27] = m2l_fma(D[73], m, L[27]);
      L[28] = m2l_fma(D[74], m, L[28]);
      L[29] = m2l_fma(D[75], m, L[29]);
      L[30] = m2l_fma(D[78], m, L[30]);
      L[31] = m2l_fma(D[79], m, L[31]);
      L[32] = m2l_fma(D[80], m, L[32]);
      L[33] = m2l_fma(D[81], m, L[33]);
      L[34] = m2l_fma(D[82], m, L[34]);
    }
    { const T m = __ldg(Ms + 9) * rp;
      L[0] = m2l_fma(D[9], m, L[0]);
      L[1] = m2l_fma(D[15], m, L[1]);
      L[2] = m2l_fma(D[18], m, L[2]);
      L[3] = m2l_fma(D[19], m, L[3]);
      L[4] = m2l_fma(D[25], m, L[4]);
      L[5] = m2l_fma(D[28], m, L[5]);
      L[6] = m2l_fma(D[29], m, L[6]);
      L[7] = m2l_fma(D[32], m, L[7]);
      L[8] = m2l_fma(D[33], m, L[8]);
      L[9] = m2l_fma(D[34], m, L[9]);
      L[10] = m2l_fma(D[40], m, L[10]);
      L[11] = m2l_fma(D[43], m, L[11]);
      L[12] = m2l_fma(D[44], m, L[12]);
      L[13] = m2l_fma(D[47], m, L[13]);
      L[14] = m2l_fma(D[48], m, L[14]);
      L[15] = m2l_fma(D[49], m, L[15]);
      L[16] = m2l_fma(D[52], m, L[16]);
      L[17] = m2l_fma(D[53], m, L[17]);
      L[18] = m2l_fma(D[54], m, L[18]);
      L[19] = m2l_fma(D[55], m, L[19]);
      L[20] = m2l_fma(D[61], m, L[20]);
      L[21] = m2l_fma(D[64], m, L[21]);
      L[22] = m2l_fma(D[65], m, L[22]);
      L[23] = m2l_fma(D[68], m, L[23]);
      L[24] = m2l_fma(D[69], m, L[24]);
      L[25] = m2l_fma(D[70], m, L[25]);
      L[26] = m2l_fma(D[73], m, L[26]);
      L[27] = m2l_fma(D[74], m, L[27]);
      L[28] = m2l_fma(D[75], m, L[28]);
      L[29] = m2l_fma(D[76], m, L[29]);
      L[30] = m2l_fma(D[79], m, L[30]);
      L[31] = m2l_fma(D[80], m, L[31]);
      L[32] = m2l_fma(D[81], m, L[32]);
      L[33] = m2l_fma(D[82], m, L[33]);
      L[34] = m2l_fma(D[83], m, L[34]);
    }
    rp *= rho;
    { const T m = -__ldg(Ms + 10) * rp;
      L[0] = m2l_fma(D[10], m, L[0]);
      L[1] = m2l_fma(D[20], m, L[1]);
      L[2] = m2l_fma(D[21], m, L[2]);
      L[3] = m2l_fma(D[22], m, L[3]);
      L[4] = m2l_fma(D[35], m, L[4]);
      L[5] = m2l_fma(D[36], m, L[5]);
      L[6] = m2l_fma(D[37], m, L[6]);
      L[7] = m2l_fma(D[38], m, L[7]);
      L[8] = m2l_fma(D[39], m, L[8]);
      L[9] = m2l_fma(D[40], m, L[9]);
      L[10] = m2l_fma(D[56], m, L[10]);
      L[11] = m2l_fma(D[57], m, L[11]);
      L[12] = m2l_fma(D[58], m, L[12]);
      L[13] = m2l_fma(D[59], m, L[13]);
      L[14] = m2l_fma(D[60], m, L[14]);
      L[15] = m2l_fma(D[61], m, L[15]);
      L[16] = m2l_fma(D[62], m, L[16]);
      L[17] = m2l_fma(D[63], m, L[17]);
      L[18] = m2l_fma(D[64], m, L[18]);
      L[19] = m2l_fma(D[65], m, L[19]);
    }
    { const T m = -__ldg(Ms + 11) * rp;
      L[0] = m2l_fma(D[11], m, L[0]);
      L[1] = m2l_fma(D[21], m, L[1]);
      L[2] = m2l_fma(D[23], m, L[2]);
      L[3] = m2l_fma(D[24], m, L[3]);
      L[4] = m2l_fma(D[36], m, L[4]);
      L[5] = m2l_fma(D[38], m, L[5]);
      L[6] = m2l_fma(D[39], m, L[6]);
      L[7] = m2l_fma(D[41], m, L[7]);
      L[8] = m2l_fma(D[42], m, L[8]);
      L[9] = m2l_fma(D[43], m, L[9]);
      L[10] = m2l_fma(D[57], m, L[10]);
      L[11] = m2l_fma(D[59], m, L[11]);
      L[12] = m2l_fma(D[60], m, L[12]);
      L[13] = m2l_fma(D[62], m, L[13]);
      L[14] = m2l_fma(D[63], m, L[14]);
      L[15] = m2l_fma(D[64], m, L[15]);
      L[16] = m2l_fma(D[66], m, L[16]);
      L[17] = m2l_fma(D[67], m, L[17]);
      L[18] = m2l_fma(D[68], m, L[18]);
      L[19] = m2l_fma(D[69], m, L[19]);
    }
    { const T m = -__ldg(Ms + 12) * rp;
      L[0] = m2l_fma(D[12], m, L[0]);
      L[1] = m2l_fma(D[22], m, L[1]);
      L[2] = m2l_fma(D[24], m, L[2]);
      L[3] = m2l_fma(D[25], m, L[3]);
      L[4] = m2l_fma(D[37], m, L[4]);
      L[5] = m2l_fma(D[39], m, L[5]);
      L[6] = m2l_fma(D[40], m, L[6]);
      L[7] = m2l_fma(D[42], m, L[7]);
      L[8] = m2l_fma(D[43], m, L[8]);
      L[9] = m2l_fma(D[44], m, L[9]);
      L[10] = m2l_fma(D[58], m, L[10]);
      L[11] = m2l_fma(D[60], m, L[11]);
      L[12] = m2l_fma(D[61], m, L[12]);
      L[13] = m2l_fma(D[63], m, L[13]);
      L[14] = m2l_fma(D[64], m, L[14]);
      L[15] = m2l_fma(D[65], m, L[15]);
      L[16] = m2l_fma(D[67], m, L[16]);
      L[17] = m2l_fma(D[68], m, L[17]);
      L[18] = m2l_fma(D[69], m, L[18]);
      L[19] = m2l_fma(D[70], m, L[19]);
    }
    { const T m = -__ldg(Ms + 13) * rp;
      L[0] = m2l_fma(D[13], m, L[0]);
      L[1] = m2l_fma(D[23], m, L[1]);
      L[2] = m2l_fma(D[26], m, L[2]);
      L[3] = m2l_fma(D[27], m, L[3]);
      L[4] = m2l_fma(D[38], m, L[4]);
      L[5] = m2l_fma(D[41], m, L[5]);
      L[6] = m2l_fma(D[42], m, L[6]);
      L[7] = m2l_fma(D[45], m, L[7]);
      L[8] = m2l_fma(D[46], m, L[8]);
      L[9] = m2l_fma(D[47], m, L[9]);
      L[10] = m2l_fma(D[59], m, L[10]);
      L[11] = m2l_fma(D[62], m, L[11]);
      L[12] = m2l_fma(D[63], m, L[12]);
      L[13] = m2l_fma(D[66], m, L[13]);
      L[14] = m2l_fma(D[67], m, L[14]);
      L[15] = m2l_fma(D[68], m, L[15]);
      L[16] = m2l_fma(D[71], m, L[16]);
      L[17] = m2l_fma(D[72], m, L[17]);
      L[18] = m2l_fma(D[73], m, L[18]);
      L[19] = m2l_fma(D[74], m, L[19]);
    }
    { const T m = -__ldg(Ms + 14) * rp;
      L[0] = m2l_fma(D[14], m, L[0]);
      L[1] = m2l_fma(D[24], m, L[1]);
      L[2] = m2l_fma(D[27], m, L[2]);
      L[3] = m2l_fma(D[28], m, L[3]);
      L[4] = m2l_fma(D[39], m, L[4]);
      L[5] = m2l_fma(D[42], m, L[5]);
      L[6] = m2l_fma(D[43], m, L[6]);
      L[7] = m2l_fma(D[46], m, L[7]);
      L[8] = m2l_fma(D[47], m, L[8]);
      L[9] = m2l_fma(D[48], m, L[9]);
      L[10] = m2l_fma(D[60], m, L[10]);
      L[11] = m2l_fma(D[63], m, L[11]);
      L[12] = m2l_fma(D[64], m, L[12]);
      L[13] = m2l_fma(D[67], m, L[13]);
      L[14] = m2l_fma(D[68], m, L[14]);
      L[15] = m2l_fma(D[69], m, L[15]);
      L[16] = m2l_fma(D[72], m, L[16]);
      L[17] = m2l_fma(D[73], m, L[17]);
      L[18] = m2l_fma(D[74], m, L[18]);
      L[19] = m2l_fma(D[75], m, L[19]);
    }
    { const T m = -__ldg(Ms + 15) * rp;
      L[0] = m2l_fma(D[15], m, L[0]);
      L[1] = m2l_fma(D[25], m, L[1]);
      L[2] = m2l_fma(D[28], m, L[2]);
      L[3] = m2l_fma(D[29], m, L[3]);
      L[4] = m2l_fma(D[40], m, L[4]);
      L[5] = m2l_fma(D[43], m, L[5]);
      L[6] = m2l_fma(D[44], m, L[6]);
      L[7] = m2l_fma(D[47], m, L[7]);
      L[8] = m2l_fma(D[48], m, L[8]);
      L[9] = m2l_fma(D[49], m, L[9]);
      L[10] = m2l_fma(D[61], m, L[10]);
      L[11] = m2l_fma(D[64], m, L[11]);
      L[12] = m2l_fma(D[65], m, L[12]);
      L[13] = m2l_fma(D[68], m, L[13]);
      L[14] = m2l_fma(D[69], m, L[14]);
      L[15] = m2l_fma(D[70], m, L[15]);
      L[16] = m2l_fma(D[73], m, L[16]);
      L[17] = m2l_fma(D[74], m, L[17]);
      L[18] = m2l_fma(D[75], m, L[18]);
      L[19] = m2l_fma(D[76], m, L[19]);
    }
    { const T m = -__ldg(Ms + 16) * rp;
      L[0] = m2l_fma(D[16], m, L[0]);
      L[1] = m2l_fma(D[26], m, L[1]);
      L[2] = m2l_fma(D[30], m, L[2]);
      L[3] = m2l_fma(D[31], m, L[3]);
      L[4] = m2l_fma(D[41], m, L[4]);
      L[5] = m2l_fma(D[45], m, L[5]);
      L[6] = m2l_fma(D[46], m, L[6]);
      L[7] = m2l_fma(D[50], m, L[7]);
      L[8] = m2l_fma(D[51], m, L[8]);
      L[9] = m2l_fma(D[52], m, L[9]);
      L[10] = m2l_fma(D[62], m, L[10]);
      L[11] = m2l_fma(D[66], m, L[11]);
      L[12] = m2l_fma(D[67], m, L[12]);
      L[13] = m2l_fma(D[71], m, L[13]);
      L[14] = m2l_fma(D[72], m, L[14]);
      L[15] = m2l_fma(D[73], m, L[15]);
      L[16] = m2l_fma(D[77], m, L[16]);
      L[17] = m2l_fma(D[78], m, L[17]);
      L[18] = m2l_fma(D[79], m, L[18]);
      L[19] = m2l_fma(D[80], m, L[19]);
    }
    { const T m = -__ldg(Ms + 17) * rp;
      L[0] = m2l_fma(D[17], m, L[0]);
      L[1] = m2l_fma(D[27], m, L[1]);
      L[2] = m2l_fma(D[31], m, L[2]);
      L[3] = m2l_fma(D[32], m, L[3]);
      L[4] = m2l_fma(D[42], m, L[4]);
      L[5] = m2l_fma(D[46], m, L[5]);
      L[6] = m2l_fma(D[47], m, L[6]);
      L[7] = m2l_fma(D[51], m, L[7]);
      L[8] = m2l_fma(D[52], m, L[8]);
      L[9] = m2l_fma(D[53], m, L[9]);
      L[10] = m2l_fma(D[63], m, L[10]);
      L[11] = m2l_fma(D[67], m, L[11]);
      L[12] = m2l_fma(D[68], m, L[12]);
      L[13] = m2l_fma(D[72], m, L[13]);
      L[14] = m2l_fma(D[73], m, L[14]);
      L[15] = m2l_fma(D[74], m, L[15]);
      L[16] = m2l_fma(D[78], m, L[16]);
      L[17] = m2l_fma(D[79], m, L[17]);
      L[18] = m2l_fma(D[80], m, L[18]);
      L[19] = m2l_fma(D[81], m, L[19]);
    }
    { const T m = -__ldg(Ms + 18) * rp;
      L[0] = m2l_fma(D[18], m, L[0]);
      L[1] = m2l_fma(D[28], m, L[1]);
      L[2] = m2l_fma(D[32], m, L[2]);
      L[3] = m2l_fma(D[33], m, L[3]);
      L[4] = m2l_fma(D[43], m, L[4]);
      L[5] = m2l_fma(D[47], m, L[5]);
      L[6] = m2l_fma(D[48], m, L[6]);
      L[7] = m2l_fma(D[52], m, L[7]);
      L[8] = m2l_fma(D[53], m, L[8]);
      L[9] = m2l_fma(D[54], m, L[9]);
      L[10] = m2l_fma(D[64], m, L[10]);
      L[11] = m2l_fma(D[68], m, L[11]);
      L[12] = m2l_fma(D[69], m, L[12]);
      L[13] = m2l_fma(D[73], m, L[13]);
      L[14] = m2l_fma(D[74], m, L[14]);
      L[15] = m2l_fma(D[75], m, L[15]);
      L[16] = m2l_fma(D[79], m, L[16]);
      L[17] = m2l_fma(D[80], m, L[17]);
      L[18] = m2l_fma(D[81], m, L[18]);
      L[19] = m2l_fma(D[82], m, L[19]);
    }
    { const T m = -__ldg(Ms + 19) * rp;
      L[0] = m2l_fma(D[19], m, L[0]);
      L[1] = m2l_fma(D[29], m, L[1]);
      L[2] = m2l_fma(D[33], m, L[2]);
      L[3] = m2l_fma(D[34], m, L[3]);
      L[4] = m2l_fma(D[44], m, L[4]);
      L[5] = m2l_fma(D[48], m, L[5]);
      L[6] = m2l_fma(D[49], m, L[6]);
      L[7] = m2l_fma(D[53], m, L[7]);
      L[8] = m2l_fma(D[54], m, L[8]);
      L[9] = m2l_fma(D[55], m, L[9]);
      L[10] = m2l_fma(D[65], m, L[10]);
      L[11] = m2l_fma(D[69], m, L[11]);
      L[12] = m2l_fma(D[70], m, L[12]);
      L[13] = m2l_fma(D[74], m, L[13]);
      L[14] = m2l_fma(D[75], m, L[14]);
      L[15] = m2l_fma(D[76], m, L[15]);
      L[16] = m2l_fma(D[80], m, L[16]);
      L[17] = m2l_fma(D[81], m, L[17]);
      L[18] = m2l_fma(D[82], m, L[18]);
      L[19] = m2l_fma(D[83], m, L[19]);
    }
    rp *= rho;
    { const T m = __ldg(Ms + 20) * rp;
      L[0] = m2l_fma(D[20], m, L[0]);
      L[1] = m2l_fma(D[35], m, L[1]);
      L[2] = m2l_fma(D[36], m, L[2]);
      L[3] = m2l_fma(D[37], m, L[3]);
      L[4] = m2l_fma(D[56], m, L[4]);
      L[5] = m2l_fma(D[57], m, L[5]);
      L[6] = m2l_fma(D[58], m, L[6]);
      L[7] = m2l_fma(D[59], m, L[7]);
      L[8] = m2l_fma(D[60], m, L[8]);
      L[9] = m2l_fma(D[61], m, L[9]);
    }
    { const T m = __ldg(Ms + 21) * rp;
      L[0] = m2l_fma(D[21], m, L[0]);
      L[1] = m2l_fma(D[36], m, L[1]);
      L[2] = m2l_fma(D[38], m, L[2]);
      L[3] = m2l_fma(D[39], m, L[3]);
      L[4] = m2l_fma(D[57], m, L[4]);
      L[5] = m2l_fma(D[59], m, L[5]);
      L[6] = m2l_fma(D[60], m, L[6]);
      L[7] = m2l_fma(D[62], m, L[7]);
      L[8] = m2l_fma(D[63], m, L[8]);
      L[9] = m2l_fma(D[64], m, L[9]);
    }
    { const T m = __ldg(Ms + 22) * rp;
      L[0] = m2l_fma(D[22], m, L[0]);
      L[1] = m2l_fma(D[37], m, L[1]);
      L[2] = m2l_fma(D[39], m, L[2]);
      L[3] = m2l_fma(D[40], m, L[3]);
      L[4] = m2l_fma(D[58], m, L[4]);
      L[5] = m2l_fma(D[60], m, L[5]);
      L[6] = m2l_fma(D[61], m, L[6]);
      L[7] = m2l_fma(D[63], m, L[7]);
      L[8] = m2l_fma(D[64], m, L[8]);
      L[9] = m2l_fma(D[65], m, L[9]);
    }
    { const T m = __ldg(Ms + 23) * rp;
      L[0] = m2l_fma(D[23], m, L[0]);
      L[1] = m2l_fma(D[38], m, L[1]);
      L[2] = m2l_fma(D[41], m, L[2]);
      L[3] = m2l_fma(D[42], m, L[3]);
      L[4] = m2l_fma(D[59], m, L[4]);
      L[5] = m2l_fma(D[62], m, L[5]);
      L[6] = m2l_fma(D[63], m, L[6]);
      L[7] = m2l_fma(D[66], m, L[7]);
      L[8] = m2l_fma(D[67], m, L[8]);
      L[9] = m2l_fma(D[68], m, L[9]);
    }
    { const T m = __ldg(Ms + 24) * rp;
      L[0] = m2l_fma(D[24], m, L[0]);
      L[1] = m2l_fma(D[39], m, L[1]);
      L[2] = m2l_fma(D[42], m, L[2]);
      L[3] = m2l_fma(D[43], m, L[3]);
      L[4] = m2l_fma(D[60], m, L[4]);
      L[5] = m2l_fma(D[63], m, L[5]);
      L[6] = m2l_fma(D[64], m, L[6]);
      L[7] = m2l_fma(D[67], m, L[7]);
      L[8] = m2l_fma(D[68], m, L[8]);
      L[9] = m2l_fma(D[69], m, L[9]);
    }
    { const T m = __ldg(Ms + 25) * rp;
      L[0] = m2l_fma(D[25], m, L[0]);
      L[1] = m2l_fma(D[40], m, L[1]);
      L[2] = m2l_fma(D[43], m, L[2]);
      L[3] = m2l_fma(D[44], m, L[3]);
      L[4] = m2l_fma(D[61], m, L[4]);
      L[5] = m2l_fma(D[64], m, L[5]);
      L[6] = m2l_fma(D[65], m, L[6]);
      L[7] = m2l_fma(D[68], m, L[7]);
      L[8] = m2l_fma(D[69], m, L[8]);
      L[9] = m2l_fma(D[70], m, L[9]);
    }
    { const T m = __ldg(Ms + 26) * rp;
      L[0] = m2l_fma(D[26], m, L[0]);
      L[1] = m2l_fma(D[41], m, L[1]);
      L[2] = m2l_fma(D[45], m, L[2]);
      L[3] = m2l_fma(D[46], m, L[3]);
      L[4] = m2l_fma(D[62], m, L[4]);
      L[5] = m2l_fma(D[66], m, L[5]);
      L[6] = m2l_fma(D[67], m, L[6]);
      L[7] = m2l_fma(D[71], m, L[7]);
      L[8] = m2l_fma(D[72], m, L[8]);
      L[9] = m2l_fma(D[73], m, L[9]);
    }
    { const T m = __ldg(Ms + 27) * rp;
      L[0] = m2l_fma(D[27], m, L[0]);
      L[1] = m2l_fma(D[42], m, L[1]);
      L[2] = m2l_fma(D[46], m, L[2]);
      L[3] = m2l_fma(D[47], m, L[3]);
      L[4] = m2l_fma(D[63], m, L[4]);
      L[5] = m2l_fma(D[67], m, L[5]);
      L[6] = m2l_fma(D[68], m, L[6]);
      L[7] = m2l_fma(D[72], m, L[7]);
      L[8] = m2l_fma(D[73], m, L[8]);
      L[9] = m2l_fma(D[74], m, L[9]);
    }
    { const T m = __ldg(Ms + 28) * rp;
      L[0] = m2l_fma(D[28], m, L[0]);
      L[1] = m2l_fma(D[43], m, L[1]);
      L[2] = m2l_fma(D[47], m, L[2]);
      L[3] = m2l_fma(D[48], m, L[3]);
      L[4] = m2l_fma(D[64], m, L[4]);
      L[5] = m2l_fma(D[68], m, L[5]);
      L[6] = m2l_fma(D[69], m, L[6]);
      L[7] = m2l_fma(D[73], m, L[7]);
      L[8] = m2l_fma(D[74], m, L[8]);
      L[9] = m2l_fma(D[75], m, L[9]);
    }
    { const T m = __ldg(Ms + 29) * rp;
      L[0] = m2l_fma(D[29], m, L[0]);
      L[1] = m2l_fma(D[44], m, L[1]);
      L[2] = m2l_fma(D[48], m, L[2]);
      L[3] = m2l_fma(D[49], m, L[3]);
      L[4] = m2l_fma(D[65], m, L[4]);
      L[5] = m2l_fma(D[69], m, L[5]);
      L[6] = m2l_fma(D[70], m, L[6]);
      L[7] = m2l_fma(D[74], m, L[7]);
      L[8] = m2l_fma(D[75], m, L[8]);
      L[9] = m2l_fma(D[76], m, L[9]);
    }
    { const T m = __ldg(Ms + 30) * rp;
      L[0] = m2l_fma(D[30], m, L[0]);
      L[1] = m2l_fma(D[45], m, L[1]);
      L[2] = m2l_fma(D[50], m, L[2]);
      L[3] = m2l_fma(D[51], m, L[3]);
      L[4] = m2l_fma(D[66], m, L[4]);
      L[5] = m2l_fma(D[71], m, L[5]);
      L[6] = m2l_fma(D[72], m, L[6]);
      L[7] = m2l_fma(D[77], m, L[7]);
      L[8] = m2l_fma(D[78], m, L[8]);
      L[9] = m2l_fma(D[79], m, L[9]);
    }
    { const T m = __ldg(Ms + 31) * rp;
      L[0] = m2l_fma(D[31], m, L[0]);
      L[1] = m2l_fma(D[46], m, L[1]);
      L[2] = m2l_fma(D[51], m, L[2]);
      L[3] = m2l_fma(D[52], m, L[3]);
      L[4] = m2l_fma(D[67], m, L[4]);
      L[5] = m2l_fma(D[72], m, L[5]);
      L[6] = m2l_fma(D[73], m, L[6]);
      L[7] = m2l_fma(D[78], m, L[7]);
      L[8] = m2l_fma(D[79], m, L[8]);
      L[9] = m2l_fma(D[80], m, L[9]);
    }
    { const T m = __ldg(Ms + 32) * rp;
      L[0] = m2l_fma(D[32], m, L[0]);
      L[1] = m2l_fma(D[47], m, L[1]);
      L[2] = m2l_fma(D[52], m, L[2]);
      L[3] = m2l_fma(D[53], m, L[3]);
      L[4] = m2l_fma(D[68], m, L[4]);
      L[5] = m2l_fma(D[73], m, L[5]);
      L[6] = m2l_fma(D[74], m, L[6]);
      L[7] = m2l_fma(D[79], m, L[7]);
      L[8] = m2l_fma(D[80], m, L[8]);
      L[9] = m2l_fma(D[81], m, L[9]);
    }
    { const T m = __ldg(Ms + 33) * rp;
      L[0] = m2l_fma(D[33], m, L[0]);
      L[1] = m2l_fma(D[48], m, L[1]);
      L[2] = m2l_fma(D[53], m, L[2]);
      L[3] = m2l_fma(D[54], m, L[3]);
      L[4] = m2l_fma(D[69], m, L[4]);
      L[5] = m2l_fma(D[74], m, L[5]);
      L[6] = m2l_fma(D[75], m, L[6]);
      L[7] = m2l_fma(D[80], m, L[7]);
      L[8] = m2l_fma(D[81], m, L[8]);
      L[9] = m2l_fma(D[82], m, L[9]);
    }
    { const T m = __ldg(Ms + 34) * rp;
      L[0] = m2l_fma(D[34], m, L[0]);
      L[1] = m2l_fma(D[49], m, L[1]);
      L[2] = m2l_fma(D[54], m, L[2]);
      L[3] = m2l_fma(D[55], m, L[3]);
      L[4] = m2l_fma(D[70], m, L[4]);
      L[5] = m2l_fma(D[75], m, L[5]);
      L[6] = m2l_fma(D[76], m, L[6]);
      L[7] = m2l_fma(D[81], m, L[7]);
      L[8] = m2l_fma(D[82], m, L[8]);
      L[9] = m2l_fma(D[83], m, L[9]);
    }
    rp *= rho;
    { const T m = -__ldg(Ms + 35) * rp;
      L[0] = m2l_fma(D[35], m, L[0]);
      L[1] = m2l_fma(D[56], m, L[1]);
      L[2] = m2l_fma(D[57], m, L[2]);
      L[3] = m2l_fma(D[58], m, L[3]);
    }
    { const T m = -__ldg(Ms + 36) * rp;
      L[0] = m2l_fma(D[36], m, L[0]);
      L[1] = m2l_fma(D[57], m, L[1]);
      L[2] = m2l_fma(D[59], m, L[2]);
      L[3] = m2l_fma(D[60], m, L[3]);
    }
    { const T m = -__ldg(Ms + 37) * rp;
      L[0] = m2l_fma(D[37], m, L[0]);
      L[1] = m2l_fma(D[58], m, L[1]);
      L[2] = m2l_fma(D[60], m, L[2]);
      L[3] = m2l_fma(D[61], m, L[3]);
    }
    { const T m = -__ldg(Ms + 38) * rp;
      L[0] = m2l_fma(D[38], m, L[0]);
      L[1] = m2l_fma(D[59], m, L[1]);
      L[2] = m2l_fma(D[62], m, L[2]);
      L[3] = m2l_fma(D[63], m, L[3]);
    }
    { const T m = -__ldg(Ms + 39) * rp;
      L[0] = m2l_fma(D[39], m, L[0]);
      L[1] = m2l_fma(D[60], m, L[1]);
      L[2] = m2l_fma(D[63], m, L[2]);
      L[3] = m2l_fma(D[64], m, L[3]);
    }
    { const T m = -__ldg(Ms + 40) * rp;
      L[0] = m2l_fma(D[40], m, L[0]);
      L[1] = m2l_fma(D[61], m, L[1]);
      L[2] = m2l_fma(D[64], m, L[2]);
      L[3] = m2l_fma(D[65], m, L[3]);
    }
    { const T m = -__ldg(Ms + 41) * rp;
      L[0] = m2l_fma(D[41], m, L[0]);
      L[1] = m2l_fma(D[62], m, L[1]);
      L[2] = m2l_fma(D[66], m, L[2]);
      L[3] = m2l_fma(D[67], m, L[3]);
    }
    { const T m = -__ldg(Ms + 42) * rp;
      L[0] = m2l_fma(D[42], m, L[0]);
      L[1] = m2l_fma(D[63], m, L[1]);
      L[2] = m2l_fma(D[67], m, L[2]);
      L[3] = m2l_fma(D[68], m, L[3]);
    }
    { const T m = -__ldg(Ms + 43) * rp;
      L[0] = m2l_fma(D[43], m, L[0]);
      L[1] = m2l_fma(D[64], m, L[1]);
      L[2] = m2l_fma(D[68], m, L[2]);
      L[3] = m2l_fma(D[69], m, L[3]);
    }
    { const T m = -__ldg(Ms + 44) * rp;
      L[0] = m2l_fma(D[44], m, L[0]);
      L[1] = m2l_fma(D[65], m, L[1]);
      L[2] = m2l_fma(D[69], m, L[2]);
      L[3] = m2l_fma(D[70], m, L[3]);
    }
    { const T m = -__ldg(Ms + 45) * rp;
      L[0] = m2l_fma(D[45], m, L[0]);
      L[1] = m2l_fma(D[66], m, L[1]);
      L[2] = m2l_fma(D[71], m, L[2]);
      L[3] = m2l_fma(D[72], m, L[3]);
    }
    { const T m = -__ldg(Ms + 46) * rp;
      L[0] = m2l_fma(D[46], m, L[0]);
      L[1] = m2l_fma(D[67], m, L[1]);
      L[2] = m2l_fma(D[72], m, L[2]);
      L[3] = m2l_fma(D[73], m, L[3]);
    }
    { const T m = -__ldg(Ms + 47) * rp;
      L[0] = m2l_fma(D[47], m, L[0]);
      L[1] = m2l_fma(D[68], m, L[1]);
      L[2] = m2l_fma(D[73], m, L[2]);
      L[3] = m2l_fma(D[74], m, L[3]);
    }
    { const T m = -__ldg(Ms + 48) * rp;
      L[0] = m2l_fma(D[48], m, L[0]);
      L[1] = m2l_fma(D[69], m, L[1]);
      L[2] = m2l_fma(D[74], m, L[2]);
      L[3] = m2l_fma(D[75], m, L[3]);
    }
    { const T m = -__ldg(Ms + 49) * rp;
      L[0] = m2l_fma(D[49], m, L[0]);
      L[1] = m2l_fma(D[70], m, L[1]);
      L[2] = m2l_fma(D[75], m, L[2]);
      L[3] = m2l_fma(D[76], m, L[3]);
    }
    { const T m = -__ldg(Ms + 50) * rp;
      L[0] = m2l_fma(D[50], m, L[0]);
      L[1] = m2l_fma(D[71], m, L[1]);
      L[2] = m2l_fma(D[77], m, L[2]);
      L[3] = m2l_fma(D[78], m, L[3]);
    }
    { const T m = -__ldg(Ms + 51) * rp;
      L[0] = m2l_fma(D[51], m, L[0]);
      L[1] = m2l_fma(D[72], m, L[1]);
      L[2] = m2l_fma(D[78], m, L[2]);
      L[3] = m2l_fma(D[79], m, L[3]);
    }
    { const T m = -__ldg(Ms + 52) * rp;
      L[0] = m2l_fma(D[52], m, L[0]);
      L[1] = m2l_fma(D[73], m, L[1]);
      L[2] = m2l_fma(D[79], m, L[2]);
      L[3] = m2l_fma(D[80], m, L[3]);
    }
    { const T m = -__ldg(Ms + 53) * rp;
      L[0] = m2l_fma(D[53], m, L[0]);
      L[1] = m2l_fma(D[74], m, L[1]);
      L[2] = m2l_fma(D[80], m, L[2]);
      L[3] = m2l_fma(D[81], m, L[3]);
    }
    { const T m = -__ldg(Ms + 54) * rp;
      L[0] = m2l_fma(D[54], m, L[0]);
      L[1] = m2l_fma(D[75], m, L[1]);
      L[2] = m2l_fma(D[81], m, L[2]);
      L[3] = m2l_fma(D[82], m, L[3]);
    }
    { const T m = -__ldg(Ms + 55) * rp;
      L[0] = m2l_fma(D[55], m, L[0]);
      L[1] = m2l_fma(D[76], m, L[1]);
      L[2] = m2l_fma(D[82], m, L[2]);
      L[3] = m2l_fma(D[83], m, L[3]);
    }
    rp *= rho;
    { const T m = __ldg(Ms + 56) * rp;
      L[0] = m2l_fma(D[56], m, L[0]);
    }
    { const T m = __ldg(Ms + 57) * rp;
      L[0] = m2l_fma(D[57], m, L[0]);
    }
    { const T m = __ldg(Ms + 58) * rp;
      L[0] = m2l_fma(D[58], m, L[0]);
    }
    { const T m = __ldg(Ms + 59) * rp;
      L[0] = m2l_fma(D[59], m, L[0]);
    }
    { const T m = __ldg(Ms + 60) * rp;
      L[0] = m2l_fma(D[60], m, L[0]);
    }
    { const T m = __ldg(Ms + 61) * rp;
      L[0] = m2l_fma(D[61], m, L[0]);
    }
    { const T m = __ldg(Ms + 62) * rp;
      L[0] = m2l_fma(D[62], m, L[0]);
    }
    { const T m = __ldg(Ms + 63) * rp;
      L[0] = m2l_fma(D[63], m, L[0]);
    }
    { const T m = __ldg(Ms + 64) * rp;
      L[0] = m2l_fma(D[64], m, L[0]);
    }
    { const T m = __ldg(Ms + 65) * rp;
      L[0] = m2l_fma(D[65], m, L[0]);
    }
    { const T m = __ldg(Ms + 66) * rp;
      L[0] = m2l_fma(D[66], m, L[0]);
    }
    { const T m = __ldg(Ms + 67) * rp;
      L[0] = m2l_fma(D[67], m, L[0]);
    }
    { const T m = __ldg(Ms + 68) * rp;
      L[0] = m2l_fma(D[68], m, L[0]);
    }
    { const T m = __ldg(Ms + 69) * rp;
      L[0] = m2l_fma(D[69], m, L[0]);
    }
    { const T m = __ldg(Ms + 70) * rp;
      L[0] = m2l_fma(D[70], m, L[0]);
    }
    { const T m = __ldg(Ms + 71) * rp;
      L[0] = m2l_fma(D[71], m, L[0]);
    }
    { const T m = __ldg(Ms + 72) * rp;
      L[0] = m2l_fma(D[72], m, L[0]);
    }
    { const T m = __ldg(Ms + 73) * rp;
      L[0] = m2l_fma(D[73], m, L[0]);
    }
    { const T m = __ldg(Ms + 74) * rp;
      L[0] = m2l_fma(D[74], m, L[0]);
    }
    { const T m = __ldg(Ms + 75) * rp;
      L[0] = m2l_fma(D[75], m, L[0]);
    }
    { const T m = __ldg(Ms + 76) * rp;
      L[0] = m2l_fma(D[76], m, L[0]);
    }
    { const T m = __ldg(Ms + 77) * rp;
      L[0] = m2l_fma(D[77], m, L[0]);
    }
    { const T m = __ldg(Ms + 78) * rp;
      L[0] = m2l_fma(D[78], m, L[0]);
    }
    { const T m = __ldg(Ms + 79) * rp;
      L[0] = m2l_fma(D[79], m, L[0]);
    }
    { const T m = __ldg(Ms + 80) * rp;
      L[0] = m2l_fma(D[80], m, L[0]);
    }
    { const T m = __ldg(Ms + 81) * rp;
      L[0] = m2l_fma(D[81], m, L[0]);
    }
    { const T m = __ldg(Ms + 82) * rp;
      L[0] = m2l_fma(D[82], m, L[0]);
    }
    { const T m = __ldg(Ms + 83) * rp;
      L[0] = m2l_fma(D[83], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_6(const T (&D)[84], const T *__restrict__ Ms, T (&L)[84])
{
    { const T m = __ldg(Ms + 0);
      L[0] = D[0] * m;
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[9] * m;
      L[10] = -D[10] * m;
      L[11] = -D[11] * m;
      L[12] = -D[12] * m;
      L[13] = -D[13] * m;
      L[14] = -D[14] * m;
      L[15] = -D[15] * m;
      L[16] = -D[16] * m;
      L[17] = -D[17] * m;
      L[18] = -D[18] * m;
      L[19] = -D[19] * m;
      L[20] = D[20] * m;
      L[21] = D[21] * m;
      L[22] = D[22] * m;
      L[23] = D[23] * m;
      L[24] = D[24] * m;
      L[25] = D[25] * m;
      L[26] = D[26] * m;
      L[27] = D[27] * m;
      L[28] = D[28] * m;
      L[29] = D[29] * m;
      L[30] = D[30] * m;
      L[31] = D[31] * m;
      L[32] = D[32] * m;
      L[33] = D[33] * m;
      L[34] = D[34] * m;
      L[35] = -D[35] * m;
      L[36] = -D[36] * m;
      L[37] = -D[37] * m;
      L[38] = -D[38] * m;
      L[39] = -D[39] * m;
      L[40] = -D[40] * m;
      L[41] = -D[41] * m;
      L[42] = -D[42] * m;
      L[43] = -D[43] * m;
      L[44] = -D[44] * m;
      L[45] = -D[45] * m;
      L[46] = -D[46] * m;
      L[47] = -D[47] * m;
      L[48] = -D[48] * m;
      L[49] = -D[49] * m;
      L[50] = -D[50] * m;
      L[51] = -D[51] * m;
      L[52] = -D[52] * m;
      L[53] = -D[53] * m;
      L[54] = -D[54] * m;
      L[55] = -D[55] * m;
      L[56] = D[56] * m;
      L[57] = D[57] * m;
      L[58] = D[58] * m;
      L[59] = D[59] * m;
      L[60] = D[60] * m;
      L[61] = D[61] * m;
      L[62] = D[62] * m;
      L[63] = D[63] * m;
      L[64] = D[64] * m;
      L[65] = D[65] * m;
      L[66] = D[66] * m;
      L[67] = D[67] * m;
      L[68] = D[68] * m;
      L[69] = D[69] * m;
      L[70] = D[70] * m;
      L[71] = D[71] * m;
      L[72] = D[72] * m;
      L[73] = D[73] * m;
      L[74] = D[74] * m;
      L[75] = D[75] * m;
      L[76] = D[76] * m;
      L[77] = D[77] * m;
      L[78] = D[78] * m;
      L[79] = D[79] * m;
      L[80] = D[80] * m;
      L[81] = D[81] * m;
      L[82] = D[82] * m;
      L[83] = D[83] * m;
    }
    { const T m = __ldg(Ms + 1);
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(-D[4], m, L[1]);
      L[2] = m2l_fma(-D[5], m, L[2]);
      L[3] = m2l_fma(-D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[15], m, L[9]);
      L[10] = m2l_fma(-D[20], m, L[10]);
      L[11] = m2l_fma(-D[21], m, L[11]);
      L[12] = m2l_fma(-D[22], m, L[12]);
      L[13] = m2l_fma(-D[23], m, L[13]);
      L[14] = m2l_fma(-D[24], m, L[14]);
      L[15] = m2l_fma(-D[25], m, L[15]);
      L[16] = m2l_fma(-D[26], m, L[16]);
      L[17] = m2l_fma(-D[27], m, L[17]);
      L[18] = m2l_fma(-D[28], m, L[18]);
      L[19] = m2l_fma(-D[29], m, L[19]);
      L[20] = m2l_fma(D[35], m, L[20]);
      L[21] = m2l_fma(D[36], m, L[21]);
      L[22] = m2l_fma(D[37], m, L[22]);
      L[23] = m2l_fma(D[38], m, L[23]);
      L[24] = m2l_fma(D[39], m, L[24]);
      L[25] = m2l_fma(D[40], m, L[25]);
      L[26] = m2l_fma(D[41], m, L[26]);
      L[27] = m2l_fma(D[42], m, L[27]);
      L[28] = m2l_fma(D[43], m, L[28]);
      L[29] = m2l_fma(D[44], m, L[29]);
      L[30] = m2l_fma(D[45], m, L[30]);
      L[31] = m2l_fma(D[46], m, L[31]);
      L[32] = m2l_fma(D[47], m, L[32]);
      L[33] = m2l_fma(D[48], m, L[33]);
      L[34] = m2l_fma(D[49], m, L[34]);
      L[35] = m2l_fma(-D[56], m, L[35]);
      L[36] = m2l_fma(-D[57], m, L[36]);
      L[37] = m2l_fma(-D[58], m, L[37]);
      L[38] = m2l_fma(-D[59], m, L[38]);
      L[39] = m2l_fma(-D[60], m, L[39]);
      L[40] = m2l_fma(-D[61], m, L[40]);
      L[41] = m2l_fma(-D[62], m, L[41]);
      L[42] = m2l_fma(-D[63], m, L[42]);
      L[43] = m2l_fma(-D[64], m, L[43]);
      L[44] = m2l_fma(-D[65], m, L[44]);
      L[45] = m2l_fma(-D[66], m, L[45]);
      L[46] = m2l_fma(-D[67], m, L[46]);
      L[47] = m2l_fma(-D[68], m, L[47]);
      L[48] = m2l_fma(-D[69], m, L[48]);
      L[49] = m2l_fma(-D[70], m, L[49]);
      L[50] = m2l_fma(-D[71], m, L[50]);
      L[51] = m2l_fma(-D[72], m, L[51]);
      L[52] = m2l_fma(-D[73], m, L[52]);
      L[53] = m2l_fma(-D[74], m, L[53]);
      L[54] = m2l_fma(-D[75], m, L[54]);
      L[55] = m2l_fma(-D[76], m, L[55]);
    }
    { const T m = __ldg(Ms + 2);
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(-D[5], m, L[1]);
      L[2] = m2l_fma(-D[7], m, L[2]);
      L[3] = m2l_fma(-D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[18], m, L[9]);
      L[10] = m2l_fma(-D[21], m, L[10]);
      L[11] = m2l_fma(-D[23], m, L[11]);
      L[12] = m2l_fma(-D[24], m, L[12]);
      L[13] = m2l_fma(-D[26], m, L[13]);
      L[14] = m2l_fma(-D[27], m, L[14]);
      L[15] = m2l_fma(-D[28], m, L[15]);
      L[16] = m2l_fma(-D[30], m, L[16]);
      L[17] = m2l_fma(-D[31], m, L[17]);
      L[18] = m2l_fma(-D[32], m, L[18]);
      L[19] = m2l_fma(-D[33], m, L[19]);
      L[20] = m2l_fma(D[36], m, L[20]);
      L[21] = m2l_fma(D[38], m, L[21]);
      L[22] = m2l_fma(D[39], m, L[22]);
      L[23] = m2l_fma(D[41], m, L[23]);
      L[24] = m2l_fma(D[42], m, L[24]);
      L[25] = m2l_fma(D[43], m, L[25]);
      L[26] = m2l_fma(D[45], m, L[26]);
      L[27] = m2l_fma(D[46], m, L[27]);
      L[28] = m2l_fma(D[47], m, L[28]);
      L[29] = m2l_fma(D[48], m, L[29]);
      L[30] = m2l_fma(D[50], m, L[30]);
      L[31] = m2l_fma(D[51], m, L[31]);
      L[32] = m2l_fma(D[52], m, L[32]);
      L[33] = m2l_fma(D[53], m, L[33]);
      L[34] = m2l_fma(D[54], m, L[34]);
      L[35] = m2l_fma(-D[57], m, L[35]);
      L[36] = m2l_fma(-D[59], m, L[36]);
      L[37] = m2l_fma(-D[60], m, L[37]);
      L[38] = m2l_fma(-D[62], m, L[38]);
      L[39] = m2l_fma(-D[63], m, L[39]);
      L[40] = m2l_fma(-D[64], m, L[40]);
      L[41] = m2l_fma(-D[66], m, L[41]);
      L[42] = m2l_fma(-D[67], m, L[42]);
      L[43] = m2l_fma(-D[68], m, L[43]);
      L[44] = m2l_fma(-D[69], m, L[44]);
      L[45] = m2l_fma(-D[71], m, L[45]);
      L[46] = m2l_fma(-D[72], m, L[46]);
      L[47] = m2l_fma(-D[73], m, L[47]);
      L[48] = m2l_fma(-D[74], m, L[48]);
      L[49] = m2l_fma(-D[75], m, L[49]);
      L[50] = m2l_fma(-D[77], m, L[50]);
      L[51] = m2l_fma(-D[78], m, L[51]);
      L[52] = m2l_fma(-D[79], m, L[52]);
      L[53] = m2l_fma(-D[80], m, L[53]);
      L[54] = m2l_fma(-D[81], m, L[54]);
      L[55] = m2l_fma(-D[82], m, L[55]);
    }
    { const T m = __ldg(Ms + 3);
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(-D[6], m, L[1]);
      L[2] = m2l_fma(-D[8], m, L[2]);
      L[3] = m2l_fma(-D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(-D[22], m, L[10]);
      L[11] = m2l_fma(-D[24], m, L[11]);
      L[12] = m2l_fma(-D[25], m, L[12]);
      L[13] = m2l_fma(-D[27], m, L[13]);
      L[14] = m2l_fma(-D[28], m, L[14]);
      L[15] = m2l_fma(-D[29], m, L[15]);
      L[16] = m2l_fma(-D[31], m, L[16]);
      L[17] = m2l_fma(-D[32], m, L[17]);
      L[18] = m2l_fma(-D[33], m, L[18]);
      L[19] = m2l_fma(-D[34], m, L[19]);
      L[20] = m2l_fma(D[37], m, L[20]);
      L[21] = m2l_fma(D[39], m, L[21]);
      L[22] = m2l_fma(D[40], m, L[22]);
      L[23] = m2l_fma(D[42], m, L[23]);
      L[24] = m2l_fma(D[43], m, L[24]);
      L[25] = m2l_fma(D[44], m, L[25]);
      L[26] = m2l_fma(D[46], m, L[26]);
      L[27] = m2l_fma(D[47], m, L[27]);
      L[28] = m2l_fma(D[48], m, L[28]);
      L[29] = m2l_fma(D[49], m, L[29]);
      L[30] = m2l_fma(D[51], m, L[30]);
      L[31] = m2l_fma(D[52], m, L[31]);
      L[32] = m2l_fma(D[53], m, L[32]);
      L[33] = m2l_fma(D[54], m, L[33]);
      L[34] = m2l_fma(D[55], m, L[34]);
      L[35] = m2l_fma(-D[58], m, L[35]);
      L[36] = m2l_fma(-D[60], m, L[36]);
      L[37] = m2l_fma(-D[61], m, L[37]);
      L[38] = m2l_fma(-D[63], m, L[38]);
      L[39] = m2l_fma(-D[64], m, L[39]);
      L[40] = m2l_fma(-D[65], m, L[40]);
      L[41] = m2l_fma(-D[67], m, L[41]);
      L[42] = m2l_fma(-D[68], m, L[42]);
      L[43] = m2l_fma(-D[69], m, L[43]);
      L[44] = m2l_fma(-D[70], m, L[44]);
      L[45] = m2l_fma(-D[72], m, L[45]);
      L[46] = m2l_fma(-D[73], m, L[46]);
      L[47] = m2l_fma(-D[74], m, L[47]);
      L[48] = m2l_fma(-D[75], m, L[48]);
      L[49] = m2l_fma(-D[76], m, L[49]);
      L[50] = m2l_fma(-D[78], m, L[50]);
      L[51] = m2l_fma(-D[79], m, L[51]);
      L[52] = m2l_fma(-D[80], m, L[52]);
      L[53] = m2l_fma(-D[81], m, L[53]);
      L[54] = m2l_fma(-D[82], m, L[54]);
      L[55] = m2l_fma(-D[83], m, L[55]);
    }
    { const T m = __ldg(Ms + 4);
      L[0] = m2l_fma(D[4], m, L[0]);
      L[1] = m2l_fma(-D[10], m, L[1]);
      L[2] = m2l_fma(-D[11], m, L[2]);
      L[3] = m2l_fma(-D[12], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[21], m, L[5]);
      L[6] = m2l_fma(D[22], m, L[6]);
      L[7] = m2l_fma(D[23], m, L[7]);
      L[8] = m2l_fma(D[24], m, L[8]);
      L[9] = m2l_fma(D[25], m, L[9]);
      L[10] = m2l_fma(-D[35], m, L[10]);
      L[11] = m2l_fma(-D[36], m, L[11]);
      L[12] = m2l_fma(-D[37], m, L[12]);
      L[13] = m2l_fma(-D[38], m, L[13]);
      L[14] = m2l_fma(-D[39], m, L[14]);
      L[15] = m2l_fma(-D[40], m, L[15]);
      L[16] = m2l_fma(-D[41], m, L[16]);
      L[17] = m2l_fma(-D[42], m, L[17]);
      L[18] = m2l_fma(-D[43], m, L[18]);
      L[19] = m2l_fma(-D[44], m, L[19]);
      L[20] = m2l_fma(D[56], m, L[20]);
      L[21] = m2l_fma(D[57], m, L[21]);
      L[22] = m2l_fma(D[58], m, L[22]);
      L[23] = m2l_fma(D[59], m, L[23]);
      L[24] = m2l_fma(D[60], m, L[24]);
      L[25] = m2l_fma(D[61], m, L[25]);
      L[26] = m2l_fma(D[62], m, L[26]);
      L[27] = m2l_fma(D[63], m, L[27]);
      L[28] = m2l_fma(D[64], m, L[28]);
      L[29] = m2l_fma(D[65], m, L[29]);
      L[30] = m2l_fma(D[66], m, L[30]);
      L[31] = m2l_fma(D[67], m, L[31]);
      L[32] = m2l_fma(D[68], m, L[32]);
      L[33] = m2l_fma(D[69], m, L[33]);
      L[34] = m2l_fma(D[70], m, L[34]);
    }
    { const T m = __ldg(Ms + 5);
      L[0] = m2l_fma(D[5], m, L[0]);
      L[1] = m2l_fma(-D[11], m, L[1]);
      L[2] = m2l_fma(-D[13], m, L[2]);
      L[3] = m2l_fma(-D[14], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(D[28], m, L[9]);
      L[10] = m2l_fma(-D[36], m, L[10]);
      L[11] = m2l_fma(-D[38], m, L[11]);
      L[12] = m2l_fma(-D[39], m, L[12]);
      L[13] = m2l_fma(-D[41], m, L[13]);
      L[14] = m2l_fma(-D[42], m, L[14]);
      L[15] = m2l_fma(-D[43], m, L[15]);
      L[16] = m2l_fma(-D[45], m, L[16]);
      L[17] = m2l_fma(-D[46], m, L[17]);
      L[18] = m2l_fma(-D[47], m, L[18]);
      L[19] = m2l_fma(-D[48], m, L[19]);
      L[20] = m2l_fma(D[57], m, L[20]);
      L[21] = m2l_fma(D[59], m, L[21]);
      L[22] = m2l_fma(D[60], m, L[22]);
      L[23] = m2l_fma(D[62], m, L[23]);
      L[24] = m2l_fma(D[63], m, L[24]);
      L[25] = m2l_fma(D[64], m, L[25]);
      L[26] = m2l_fma(D[66], m, L[26]);
      L[27] = m2l_fma(D[67], m, L[27]);
      L[28] = m2l_fma(D[68], m, L[28]);
      L[29] = m2l_fma(D[69], m, L[29]);
      L[30] = m2l_fma(D[71], m, L[30]);
      L[31] = m2l_fma(D[72], m, L[31]);
      L[32] = m2l_fma(D[73], m, L[32]);
      L[33] = m2l_fma(D[74], m, L[33]);
      L[34] = m2l_fma(D[75], m, L[34]);
    }
    { const T m = __ldg(Ms + 6);
      L[0] = m2l_fma(D[6], m, L[0]);
      L[1] = m2l_fma(-D[12], m, L[1]);
      L[2] = m2l_fma(-D[14], m, L[2]);
      L[3] = m2l_fma(-D[15], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[24], m, L[5]);
      L[6] = m2l_fma(D[25], m, L[6]);
      L[7] = m2l_fma(D[27], m, L[7]);
      L[8] = m2l_fma(D[28], m, L[8]);
      L[9] = m2l_fma(D[29], m, L[9]);
      L[10] = m2l_fma(-D[37], m, L[10]);
      L[11] = m2l_fma(-D[39], m, L[11]);
      L[12] = m2l_fma(-D[40], m, L[12]);
      L[13] = m2l_fma(-D[42], m, L[13]);
      L[14] = m2l_fma(-D[43], m, L[14]);
      L[15] = m2l_fma(-D[44], m, L[15]);
      L[16] = m2l_fma(-D[46], m, L[16]);
      L[17] = m2l_fma(-D[47], m, L[17]);
      L[18] = m2l_fma(-D[48], m, L[18]);
      L[19] = m2l_fma(-D[49], m, L[19]);
      L[20] = m2l_fma(D[58], m, L[20]);
      L[21] = m2l_fma(D[60], m, L[21]);
      L[22] = m2l_fma(D[61], m, L[22]);
      L[23] = m2l_fma(D[63], m, L[23]);
      L[24] = m2l_fma(D[64], m, L[24]);
      L[25] = m2l_fma(D[65], m, L[25]);
      L[26] = m2l_fma(D[67], m, L[26]);
      L[27] = m2l_fma(D[68], m, L[27]);
      L[28] = m2l_fma(D[69], m, L[28]);
      L[29] = m2l_fma(D[70], m, L[29]);
      L[30] = m2l_fma(D[72], m, L[30]);
      L[31] = m2l_fma(D[73], m, L[31]);
      L[32] = m2l_fma(D[74], m, L[32]);
      L[33] = m2l_fma(D[75], m, L[33]);
      L[34] = m2l_fma(D[76], m, L[34]);
    }
    { const T m = __ldg(Ms + 7);
      L[0] = m2l_fma(D[7], m, L[0]);
      L[1] = m2l_fma(-D[13], m, L[1]);
      L[2] = m2l_fma(-D[16], m, L[2]);
      L[3] = m2l_fma(-D[17], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[30], m, L[7]);
      L[8] = m2l_fma(D[31], m, L[8]);
      L[9] = m2l_fma(D[32], m, L[9]);
      L[10] = m2l_fma(-D[38], m, L[10]);
      L[11] = m2l_fma(-D[41], m, L[11]);
      L[12] = m2l_fma(-D[42], m, L[12]);
      L[13] = m2l_fma(-D[45], m, L[13]);
      L[14] = m2l_fma(-D[46], m, L[14]);
      L[15] = m2l_fma(-D[47], m, L[15]);
      L[16] = m2l_fma(-D[50], m, L[16]);
      L[17] = m2l_fma(-D[51], m, L[17]);
      L[18] = m2l_fma(-D[52], m, L[18]);
      L[19] = m2l_fma(-D[53], m, L[19]);
      L[20] = m2l_fma(D[59], m, L[20]);
      L[21] = m2l_fma(D[62], m, L[21]);
      L[22] = m2l_fma(D[63], m, L[22]);
      L[23] = m2l_fma(D[66], m, L[23]);
      L[24] = m2l_fma(D[67], m, L[24]);
      L[25] = m2l_fma(D[68], m, L[25]);
      L[26] = m2l_fma(D[71], m, L[26]);
      L[27] = m2l_fma(D[72], m, L[27]);
      L[28] = m2l_fma(D[73], m, L[28]);
      L[29] = m2l_fma(D[74], m, L[29]);
      L[30] = m2l_fma(D[77], m, L[30]);
      L[31] = m2l_fma(D[78], m, L[31]);
      L[32] = m2l_fma(D[79], m, L[32]);
      L[33] = m2l_fma(D[80], m, L[33]);
      L[34] = m2l_fma(D[81], m, L[34]);
    }
    { const T m = __ldg(Ms + 8);
      L[0] = m2l_fma(D[8], m, L[0]);
      L[1] = m2l_fma(-D[14], m, L[1]);
      L[2] = m2l_fma(-D[17], m, L[2]);
      L[3] = m2l_fma(-D[18], m, L[3]);
      L[4] = m2l_fma(D[24], m, L[4]);
      L[5] = m2l_fma(D[27], m, L[5]);
      L[6] = m2l_fma(D[28], m, L[6]);
      L[7] = m2l_fma(D[31], m, L[7]);
      L[8] = m2l_fma(D[32], m, L[8]);
      L[9] = m2l_fma(D[33], m, L[9]);
      L[10] = m2l_fma(-D[39], m, L[10]);
      L[11] = m2l_fma(-D[42], m, L[11]);
      L[12] = m2l_fma(-D[43], m, L[12]);
      L[13] = m2l_fma(-D[46], m, L[13]);
      L[14] = m2l_fma(-D[47], m, L[14]);
      L[15] = m2l_fma(-D[48], m, L[15]);
      L[16] = m2l_fma(-D[51], m, L[16]);
      L[17] = m2l_fma(-D[52], m, L[17]);
      L[18] = m2l_fma(-D[53], m, L[18]);
      L[19] = m2l_fma(-D[54], m, L[19]);
      L[20] = m2l_fma(D[60], m, L[20]);
      L[21] = m2l_fma(D[63], m, L[21]);
      L[22] = m2l_fma(D[64], m, L[22]);
      L[23] = m2l_fma(D[67], m, L[23]);
      L[24] = m2l_fma(D[68], m, L[24]);
      L[25] = m2l_fma(D[69], m, L[25]);
      L[26] = m2l_fma(D[72], m, L[26]);
      L[27] = m2l_fma(D[73], m, L[27]);
      L[28] = m2l_fma(D[74], m, L[28]);
      L[29] = m2l_fma(D[75], m, L[29]);
      L[30] = m2l_fma(D[78], m, L[30]);
      L[31] = m2l_fma(D[79], m, L[31]);
      L[32] = m2l_fma(D[80], m, L[32]);
      L[33] = m2l_fma(D[81], m, L[33]);
      L[34] = m2l_fma(D[82], m, L[34]);
    }
    { const T m = __ldg(Ms + 9);
      L[0] = m2l_fma(D[9], m, L[0]);
      L[1] = m2l_fma(-D[15], m, L[1]);
      L[2] = m2l_fma(-D[18], m, L[2]);
      L[3] = m2l_fma(-D[19], m, L[3]);
      L[4] = m2l_fma(D[25], m, L[4]);
      L[5] = m2l_fma(D[28], m, L[5]);
      L[6] = m2l_fma(D[29], m, L[6]);
      L[7] = m2l_fma(D[32], m, L[7]);
      L[8] = m2l_fma(D[33], m, L[8]);
      L[9] = m2l_fma(D[34], m, L[9]);
      L[10] = m2l_fma(-D[40], m, L[10]);
      L[11] = m2l_fma(-D[43], m, L[11]);
      L[12] = m2l_fma(-D[44], m, L[12]);
      L[13] = m2l_fma(-D[47], m, L[13]);
      L[14] = m2l_fma(-D[48], m, L[14]);
      L[15] = m2l_fma(-D[49], m, L[15]);
      L[16] = m2l_fma(-D[52], m, L[16]);
      L[17] = m2l_fma(-D[53], m, L[17]);
      L[18] = m2l_fma(-D[54], m, L[18]);
      L[19] = m2l_fma(-D[55], m, L[19]);
      L[20] = m2l_fma(D[61], m, L[20]);
      L[21] = m2l_fma(D[64], m, L[21]);
      L[22] = m2l_fma(D[65], m, L[22]);
      L[23] = m2l_fma(D[68], m, L[23]);
      L[24] = m2l_fma(D[69], m, L[24]);
      L[25] = m2l_fma(D[70], m, L[25]);
      L[26] = m2l_fma(D[73], m, L[26]);
      L[27] = m2l_fma(D[74], m, L[27]);
      L[28] = m2l_fma(D[75], m, L[28]);
      L[29] = m2l_fma(D[76], m, L[29]);
      L[30] = m2l_fma(D[79], m, L[30]);
      L[31] = m2l_fma(D[80], m, L[31]);
      L[32] = m2l_fma(D[81], m, L[32]);
      L[33] = m2l_fma(D[82], m, L[33]);
      L[34] = m2l_fma(D[83], m, L[34]);
    }
    { const T m = __ldg(Ms + 10);
      L[0] = m2l_fma(D[10], m, L[0]);
      L[1] = m2l_fma(-D[20], m, L[1]);
      L[2] = m2l_fma(-D[21], m, L[2]);
      L[3] = m2l_fma(-D[22], m, L[3]);
      L[4] = m2l_fma(D[35], m, L[4]);
      L[5] = m2l_fma(D[36], m, L[5]);
      L[6] = m2l_fma(D[37], m, L[6]);
      L[7] = m2l_fma(D[38], m, L[7]);
      L[8] = m2l_fma(D[39], m, L[8]);
      L[9] = m2l_fma(D[40], m, L[9]);
      L[10] = m2l_fma(-D[56], m, L[10]);
      L[11] = m2l_fma(-D[57], m, L[11]);
      L[12] = m2l_fma(-D[58], m, L[12]);
      L[13] = m2l_fma(-D[59], m, L[13]);
      L[14] = m2l_fma(-D[60], m, L[14]);
      L[15] = m2l_fma(-D[61], m, L[15]);
      L[16] = m2l_fma(-D[62], m, L[16]);
      L[17] = m2l_fma(-D[63], m, L[17]);
      L[18] = m2l_fma(-D[64], m, L[18]);
      L[19] = m2l_fma(-D[65], m, L[19]);
    }
    { const T m = __ldg(Ms + 11);
      L[0] = m2l_fma(D[11], m, L[0]);
      L[1] = m2l_fma(-D[21], m, L[1]);
      L[2] = m2l_fma(-D[23], m, L[2]);
      L[3] = m2l_fma(-D[24], m, L[3]);
      L[4] = m2l_fma(D[36], m, L[4]);
      L[5] = m2l_fma(D[38], m, L[5]);
      L[6] = m2l_fma(D[39], m, L[6]);
      L[7] = m2l_fma(D[41], m, L[7]);
      L[8] = m2l_fma(D[42], m, L[8]);
      L[9] = m2l_fma(D[43], m, L[9]);
      L[10] = m2l_fma(-D[57], m, L[10]);
      L[11] = m2l_fma(-D[59], m, L[11]);
      L[12] = m2l_fma(-D[60], m, L[12]);
      L[13] = m2l_fma(-D[62], m, L[13]);
      L[14] = m2l_fma(-D[63], m, L[14]);
      L[15] = m2l_fma(-D[64], m, L[15]);
      L[16] = m2l_fma(-D[66], m, L[16]);
      L[17] = m2l_fma(-D[67], m, L[17]);
      L[18] = m2l_fma(-D[68], m, L[18]);
      L[19] = m2l_fma(-D[69], m, L[19]);
    }
    { const T m = __ldg(Ms + 12);
      L[0] = m2l_fma(D[12], m, L[0]);
      L[1] = m2l_fma(-D[22], m, L[1]);
      L[2] = m2l_fma(-D[24], m, L[2]);
      L[3] = m2l_fma(-D[25], m, L[3]);
      L[4] = m2l_fma(D[37], m, L[4]);
      L[5] = m2l_fma(D[39], m, L[5]);
      L[6] = m2l_fma(D[40], m, L[6]);
      L[7] = m2l_fma(D[42], m, L[7]);
      L[8] = m2l_fma(D[43], m, L[8]);
      L[9] = m2l_fma(D[44], m, L[9]);
      L[10] = m2l_fma(-D[58], m, L[10]);
      L[11] = m2l_fma(-D[60], m, L[11]);
      L[12] = m2l_fma(-D[61], m, L[12]);
      L[13] = m2l_fma(-D[63], m, L[13]);
      L[14] = m2l_fma(-D[64], m, L[14]);
      L[15] = m2l_fma(-D[65], m, L[15]);
      L[16] = m2l_fma(-D[67], m, L[16]);
      L[17] = m2l_fma(-D[68], m, L[17]);
      L[18] = m2l_fma(-D[69], m, L[18]);
      L[19] = m2l_fma(-D[70], m, L[19]);
    }
    { const T m = __ldg(Ms + 13);
      L[0] = m2l_fma(D[13], m, L[0]);
      L[1] = m2l_fma(-D[23], m, L[1]);
      L[2] = m2l_fma(-D[26], m, L[2]);
      L[3] = m2l_fma(-D[27], m, L[3]);
      L[4] = m2l_fma(D[38], m, L[4]);
      L[5] = m2l_fma(D[41], m, L[5]);
      L[6] = m2l_fma(D[42], m, L[6]);
      L[7] = m2l_fma(D[45], m, L[7]);
      L[8] = m2l_fma(D[46], m, L[8]);
      L[9] = m2l_fma(D[47], m, L[9]);
      L[10] = m2l_fma(-D[59], m, L[10]);
      L[11] = m2l_fma(-D[62], m, L[11]);
      L[12] = m2l_fma(-D[63], m, L[12]);
      L[13] = m2l_fma(-D[66], m, L[13]);
      L[14] = m2l_fma(-D[67], m, L[14]);
      L[15] = m2l_fma(-D[68], m, L[15]);
      L[16] = m2l_fma(-D[71], m, L[16]);
      L[17] = m2l_fma(-D[72], m, L[17]);
      L[18] = m2l_fma(-D[73], m, L[18]);
      L[19] = m2l_fma(-D[74], m, L[19]);
    }
    { const T m = __ldg(Ms + 14);
      L[0] = m2l_fma(D[14], m, L[0]);
      L[1] = m2l_fma(-D[24], m, L[1]);
      L[2] = m2l_fma(-D[27], m, L[2]);
      L[3] = m2l_fma(-D[28], m, L[3]);
      L[4] = m2l_fma(D[39], m, L[4]);
      L[5] = m2l_fma(D[42], m, L[5]);
      L[6] = m2l_fma(D[43], m, L[6]);
      L[7] = m2l_fma(D[46], m, L[7]);
      L[8] = m2l_fma(D[47], m, L[8]);
      L[9] = m2l_fma(D[48], m, L[9]);
      L[10] = m2l_fma(-D[60], m, L[10]);
      L[11] = m2l_fma(-D[63], m, L[11]);
      L[12] = m2l_fma(-D[64], m, L[12]);
      L[13] = m2l_fma(-D[67], m, L[13]);
      L[14] = m2l_fma(-D[68], m, L[14]);
      L[15] = m2l_fma(-D[69], m, L[15]);
      L[16] = m2l_fma(-D[72], m, L[16]);
      L[17] = m2l_fma(-D[73], m, L[17]);
      L[18] = m2l_fma(-D[74], m, L[18]);
      L[19] = m2l_fma(-D[75], m, L[19]);
    }
    { const T m = __ldg(Ms + 15);
      L[0] = m2l_fma(D[15], m, L[0]);
      L[1] = m2l_fma(-D[25], m, L[1]);
      L[2] = m2l_fma(-D[28], m, L[2]);
      L[3] = m2l_fma(-D[29], m, L[3]);
      L[4] = m2l_fma(D[40], m, L[4]);
      L[5] = m2l_fma(D[43], m, L[5]);
      L[6] = m2l_fma(D[44], m, L[6]);
      L[7] = m2l_fma(D[47], m, L[7]);
      L[8] = m2l_fma(D[48], m, L[8]);
      L[9] = m2l_fma(D[49], m, L[9]);
      L[10] = m2l_fma(-D[61], m, L[10]);
      L[11] = m2l_fma(-D[64], m, L[11]);
      L[12] = m2l_fma(-D[65], m, L[12]);
      L[13] = m2l_fma(-D[68], m, L[13]);
      L[14] = m2l_fma(-D[69], m, L[14]);
      L[15] = m2l_fma(-D[70], m, L[15]);
      L[16] = m2l_fma(-D[73], m, L[16]);
      L[17] = m2l_fma(-D[74], m, L[17]);
      L[18] = m2l_fma(-D[75], m, L[18]);
      L[19] = m2l_fma(-D[76], m, L[19]);
    }
    { const T m = __ldg(Ms + 16);
      L[0] = m2l_fma(D[16], m, L[0]);
      L[1] = m2l_fma(-D[26], m, L[1]);
      L[2] = m2l_fma(-D[30], m, L[2]);
      L[3] = m2l_fma(-D[31], m, L[3]);
      L[4] = m2l_fma(D[41], m, L[4]);
      L[5] = m2l_fma(D[45], m, L[5]);
      L[6] = m2l_fma(D[46], m, L[6]);
      L[7] = m2l_fma(D[50], m, L[7]);
      L[8] = m2l_fma(D[51], m, L[8]);
      L[9] = m2l_fma(D[52], m, L[9]);
      L[10] = m2l_fma(-D[62], m, L[10]);
      L[11] = m2l_fma(-D[66], m, L[11]);
      L[12] = m2l_fma(-D[67], m, L[12]);
      L[13] = m2l_fma(-D[71], m, L[13]);
      L[14] = m2l_fma(-D[72], m, L[14]);
      L[15] = m2l_fma(-D[73], m, L[15]);
      L[16] = m2l_fma(-D[77], m, L[16]);
      L[17] = m2l_fma(-D[78], m, L[17]);
      L[18] = m2l_fma(-D[79], m, L[18]);
      L[19] = m2l_fma(-D[80], m, L[19]);
    }
    { const T m = __ldg(Ms + 17);
      L[0] = m2l_fma(D[17], m, L[0]);
      L[1] = m2l_fma(-D[27], m, L[1]);
      L[2] = m2l_fma(-D[31], m, L[2]);
      L[3] = m2l_fma(-D[32], m, L[3]);
      L[4] = m2l_fma(D[42], m, L[4]);
      L[5] = m2l_fma(D[46], m, L[5]);
      L[6] = m2l_fma(D[47], m, L[6]);
      L[7] = m2l_fma(D[51], m, L[7]);
      L[8] = m2l_fma(D[52], m, L[8]);
      L[9] = m2l_fma(D[53], m, L[9]);
      L[10] = m2l_fma(-D[63], m, L[10]);
      L[11] = m2l_fma(-D[67], m, L[11]);
      L[12] = m2l_fma(-D[68], m, L[12]);
      L[13] = m2l_fma(-D[72], m, L[13]);
      L[14] = m2l_fma(-D[73], m, L[14]);
      L[15] = m2l_fma(-D[74], m, L[15]);
      L[16] = m2l_fma(-D[78], m, L[16]);
      L[17] = m2l_fma(-D[79], m, L[17]);
      L[18] = m2l_fma(-D[80], m, L[18]);
      L[19] = m2l_fma(-D[81], m, L[19]);
    }
    { const T m = __ldg(Ms + 18);
      L[0] = m2l_fma(D[18], m, L[0]);
      L[1] = m2l_fma(-D[28], m, L[1]);
      L[2] = m2l_fma(-D[32], m, L[2]);
      L[3] = m2l_fma(-D[33], m, L[3]);
      L[4] = m2l_fma(D[43], m, L[4]);
      L[5] = m2l_fma(D[47], m, L[5]);
      L[6] = m2l_fma(D[48], m, L[6]);
      L[7] = m2l_fma(D[52], m, L[7]);
      L[8] = m2l_fma(D[53], m, L[8]);
      L[9] = m2l_fma(D[54], m, L[9]);
      L[10] = m2l_fma(-D[64], m, L[10]);
      L[11] = m2l_fma(-D[68], m, L[11]);
      L[12] = m2l_fma(-D[69], m, L[12]);
      L[13] = m2l_fma(-D[73], m, L[13]);
      L[14] = m2l_fma(-D[74], m, L[14]);
      L[15] = m2l_fma(-D[75], m, L[15]);
      L[16] = m2l_fma(-D[79], m, L[16]);
      L[17] = m2l_fma(-D[80], m, L[17]);
      L[18] = m2l_fma(-D[81], m, L[18]);
      L[19] = m2l_fma(-D[82], m, L[19]);
    }
    { const T m = __ldg(Ms + 19);
      L[0] = m2l_fma(D[19], m, L[0]);
      L[1] = m2l_fma(-D[29], m, L[1]);
      L[2] = m2l_fma(-D[33], m, L[2]);
      L[3] = m2l_fma(-D[34], m, L[3]);
      L[4] = m2l_fma(D[44], m, L[4]);
      L[5] = m2l_fma(D[48], m, L[5]);
      L[6] = m2l_fma(D[49], m, L[6]);
      L[7] = m2l_fma(D[53], m, L[7]);
      L[8] = m2l_fma(D[54], m, L[8]);
      L[9] = m2l_fma(D[55], m, L[9]);
      L[10] = m2l_fma(-D[65], m, L[10]);
      L[11] = m2l_fma(-D[69], m, L[11]);
      L[12] = m2l_fma(-D[70], m, L[12]);
      L[13] = m2l_fma(-D[74], m, L[13]);
      L[14] = m2l_fma(-D[75], m, L[14]);
      L[15] = m2l_fma(-D[76], m, L[15]);
      L[16] = m2l_fma(-D[80], m, L[16]);
      L[17] = m2l_fma(-D[81], m, L[17]);
      L[18] = m2l_fma(-D[82], m, L[18]);
      L[19] = m2l_fma(-D[83], m, L[19]);
    }
    { const T m = __ldg(Ms + 20);
      L[0] = m2l_fma(D[20], m, L[0]);
      L[1] = m2l_fma(-D[35], m, L[1]);
      L[2] = m2l_fma(-D[36], m, L[2]);
      L[3] = m2l_fma(-D[37], m, L[3]);
      L[4] = m2l_fma(D[56], m, L[4]);
      L[5] = m2l_fma(D[57], m, L[5]);
      L[6] = m2l_fma(D[58], m, L[6]);
      L[7] = m2l_fma(D[59], m, L[7]);
      L[8] = m2l_fma(D[60], m, L[8]);
      L[9] = m2l_fma(D[61], m, L[9]);
    }
    { const T m = __ldg(Ms + 21);
      L[0] = m2l_fma(D[21], m, L[0]);
      L[1] = m2l_fma(-D[36], m, L[1]);
      L[2] = m2l_fma(-D[38], m, L[2]);
      L[3] = m2l_fma(-D[39], m, L[3]);
      L[4] = m2l_fma(D[57], m, L[4]);
      L[5] = m2l_fma(D[59], m, L[5]);
      L[6] = m2l_fma(D[60], m, L[6]);
      L[7] = m2l_fma(D[62], m, L[7]);
      L[8] = m2l_fma(D[63], m, L[8]);
      L[9] = m2l_fma(D[64], m, L[9]);
    }
    { const T m = __ldg(Ms + 22);
      L[0] = m2l_fma(D[22], m, L[0]);
      L[1] = m2l_fma(-D[37], m, L[1]);
      L[2] = m2l_fma(-D[39], m, L[2]);
      L[3] = m2l_fma(-D[40], m, L[3]);
      L[4] = m2l_fma(D[58], m, L[4]);
      L[5] = m2l_fma(D[60], m, L[5]);
      L[6] = m2l_fma(D[61], m, L[6]);
      L[7] = m2l_fma(D[63], m, L[7]);
      L[8] = m2l_fma(D[64], m, L[8]);
      L[9] = m2l_fma(D[65], m, L[9]);
    }
    { const T m = __ldg(Ms + 23);
      L[0] = m2l_fma(D[23], m, L[0]);
      L[1] = m2l_fma(-D[38], m, L[1]);
      L[2] = m2l_fma(-D[41], m, L[2]);
      L[3] = m2l_fma(-D[42], m, L[3]);
      L[4] = m2l_fma(D[59], m, L[4]);
      L[5] = m2l_fma(D[62], m, L[5]);
      L[6] = m2l_fma(D[63], m, L[6]);
      L[7] = m2l_fma(D[66], m, L[7]);
      L[8] = m2l_fma(D[67], m, L[8]);
      L[9] = m2l_fma(D[68], m, L[9]);
    }
    { const T m = __ldg(Ms + 24);
      L[0] = m2l_fma(D[24], m, L[0]);
      L[1] = m2l_fma(-D[39], m, L[1]);
      L[2] = m2l_fma(-D[42], m, L[2]);
      L[3] = m2l_fma(-D[43], m, L[3]);
      L[4] = m2l_fma(D[60], m, L[4]);
      L[5] = m2l_fma(D[63], m, L[5]);
      L[6] = m2l_fma(D[64], m, L[6]);
      L[7] = m2l_fma(D[67], m, L[7]);
      L[8] = m2l_fma(D[68], m, L[8]);
      L[9] = m2l_fma(D[69], m, L[9]);
    }
    { const T m = __ldg(Ms + 25);
      L[0] = m2l_fma(D[25], m, L[0]);
      L[1] = m2l_fma(-D[40], m, L[1]);
      L[2] = m2l_fma(-D[43], m, L[2]);
      L[3] = m2l_fma(-D[44], m, L[3]);
      L[4] = m2l_fma(D[61], m, L[4]);
      L[5] = m2l_fma(D[64], m, L[5]);
      L[6] = m2l_fma(D[65], m, L[6]);
      L[7] = m2l_fma(D[68], m, L[7]);
      L[8] = m2l_fma(D[69], m, L[8]);
      L[9] = m2l_fma(D[70], m, L[9]);
    }
    { const T m = __ldg(Ms + 26);
      L[0] = m2l_fma(D[26], m, L[0]);
      L[1] = m2l_fma(-D[41], m, L[1]);
      L[2] = m2l_fma(-D[45], m, L[2]);
      L[3] = m2l_fma(-D[46], m, L[3]);
      L[4] = m2l_fma(D[62], m, L[4]);
      L[5] = m2l_fma(D[66], m, L[5]);
      L[6] = m2l_fma(D[67], m, L[6]);
      L[7] = m2l_fma(D[71], m, L[7]);
      L[8] = m2l_fma(D[72], m, L[8]);
      L[9] = m2l_fma(D[73], m, L[9]);
    }
    { const T m = __ldg(Ms + 27);
      L[0] = m2l_fma(D[27], m, L[0]);
      L[1] = m2l_fma(-D[42], m, L[1]);
      L[2] = m2l_fma(-D[46], m, L[2]);
      L[3] = m2l_fma(-D[47], m, L[3]);
      L[4] = m2l_fma(D[63], m, L[4]);
      L[5] = m2l_fma(D[67], m, L[5]);
      L[6] = m2l_fma(D[68], m, L[6]);
      L[7] = m2l_fma(D[72], m, L[7]);
      L[8] = m2l_fma(D[73], m, L[8]);
      L[9] = m2l_fma(D[74], m, L[9]);
    }
    { const T m = __ldg(Ms + 28);
      L[0] = m2l_fma(D[28], m, L[0]);
      L[1] = m2l_fma(-D[43], m, L[1]);
      L[2] = m2l_fma(-D[47], m, L[2]);
      L[3] = m2l_fma(-D[48], m, L[3]);
      L[4] = m2l_fma(D[64], m, L[4]);
      L[5] = m2l_fma(D[68], m, L[5]);
      L[6] = m2l_fma(D[69], m, L[6]);
      L[7] = m2l_fma(D[73], m, L[7]);
      L[8] = m2l_fma(D[74], m, L[8]);
      L[9] = m2l_fma(D[75], m, L[9]);
    }
    { const T m = __ldg(Ms + 29);
      L[0] = m2l_fma(D[29], m, L[0]);
      L[1] = m2l_fma(-D[44], m, L[1]);
      L[2] = m2l_fma(-D[48], m, L[2]);
      L[3] = m2l_fma(-D[49], m, L[3]);
      L[4] = m2l_fma(D[65], m, L[4]);
      L[5] = m2l_fma(D[69], m, L[5]);
      L[6] = m2l_fma(D[70], m, L[6]);
      L[7] = m2l_fma(D[74], m, L[7]);
      L[8] = m2l_fma(D[75], m, L[8]);
      L[9] = m2l_fma(D[76], m, L[9]);
    }
    { const T m = __ldg(Ms + 30);
      L[0] = m2l_fma(D[30], m, L[0]);
      L[1] = m2l_fma(-D[45], m, L[1]);
      L[2] = m2l_fma(-D[50], m, L[2]);
      L[3] = m2l_fma(-D[51], m, L[3]);
      L[4] = m2l_fma(D[66], m, L[4]);
      L[5] = m2l_fma(D[71], m, L[5]);
      L[6] = m2l_fma(D[72], m, L[6]);
      L[7] = m2l_fma(D[77], m, L[7]);
      L[8] = m2l_fma(D[78], m, L[8]);
      L[9] = m2l_fma(D[79], m, L[9]);
    }
    { const T m = __ldg(Ms + 31);
      L[0] = m2l_fma(D[31], m, L[0]);
      L[1] = m2l_fma(-D[46], m, L[1]);
      L[2] = m2l_fma(-D[51], m, L[2]);
      L[3] = m2l_fma(-D[52], m, L[3]);
      L[4] = m2l_fma(D[67], m, L[4]);
      L[5] = m2l_fma(D[72], m, L[5]);
      L[6] = m2l_fma(D[73], m, L[6]);
      L[7] = m2l_fma(D[78], m, L[7]);
      L[8] = m2l_fma(D[79], m, L[8]);
      L[9] = m2l_fma(D[80], m, L[9]);
    }
    { const T m = __ldg(Ms + 32);
      L[0] = m2l_fma(D[32], m, L[0]);
      L[1] = m2l_fma(-D[47], m, L[1]);
      L[2] = m2l_fma(-D[52], m, L[2]);
      L[3] = m2l_fma(-D[53], m, L[3]);
      L[4] = m2l_fma(D[68], m, L[4]);
      L[5] = m2l_fma(D[73], m, L[5]);
      L[6] = m2l_fma(D[74], m, L[6]);
      L[7] = m2l_fma(D[79], m, L[7]);
      L[8] = m2l_fma(D[80], m, L[8]);
      L[9] = m2l_fma(D[81], m, L[9]);
    }
    { const T m = __ldg(Ms + 33);
      L[0] = m2l_fma(D[33], m, L[0]);
      L[1] = m2l_fma(-D[48], m, L[1]);
      L[2] = m2l_fma(-D[53], m, L[2]);
      L[3] = m2l_fma(-D[54], m, L[3]);
      L[4] = m2l_fma(D[69], m, L[4]);
      L[5] = m2l_fma(D[74], m, L[5]);
      L[6] = m2l_fma(D[75], m, L[6]);
      L[7] = m2l_fma(D[80], m, L[7]);
      L[8] = m2l_fma(D[81], m, L[8]);
      L[9] = m2l_fma(D[82], m, L[9]);
    }
    { const T m = __ldg(Ms + 34);
      L[0] = m2l_fma(D[34], m, L[0]);
      L[1] = m2l_fma(-D[49], m, L[1]);
      L[2] = m2l_fma(-D[54], m, L[2]);
      L[3] = m2l_fma(-D[55], m, L[3]);
      L[4] = m2l_fma(D[70], m, L[4]);
      L[5] = m2l_fma(D[75], m, L[5]);
      L[6] = m2l_fma(D[76], m, L[6]);
      L[7] = m2l_fma(D[81], m, L[7]);
      L[8] = m2l_fma(D[82], m, L[8]);
      L[9] = m2l_fma(D[83], m, L[9]);
    }
    { const T m = __ldg(Ms + 35);
      L[0] = m2l_fma(D[35], m, L[0]);
      L[1] = m2l_fma(-D[56], m, L[1]);
      L[2] = m2l_fma(-D[57], m, L[2]);
      L[3] = m2l_fma(-D[58], m, L[3]);
    }
    { const T m = __ldg(Ms + 36);
      L[0] = m2l_fma(D[36], m, L[0]);
      L[1] = m2l_fma(-D[57], m, L[1]);
      L[2] = m2l_fma(-D[59], m, L[2]);
      L[3] = m2l_fma(-D[60], m, L[3]);
    }
    { const T m = __ldg(Ms + 37);
      L[0] = m2l_fma(D[37], m, L[0]);
      L[1] = m2l_fma(-D[58], m, L[1]);
      L[2] = m2l_fma(-D[60], m, L[2]);
      L[3] = m2l_fma(-D[61], m, L[3]);
    }
    { const T m = __ldg(Ms + 38);
      L[0] = m2l_fma(D[38], m, L[0]);
      L[1] = m2l_fma(-D[59], m, L[1]);
      L[2] = m2l_fma(-D[62], m, L[2]);
      L[3] = m2l_fma(-D[63], m, L[3]);
    }
    { const T m = __ldg(Ms + 39);
      L[0] = m2l_fma(D[39], m, L[0]);
      L[1] = m2l_fma(-D[60], m, L[1]);
      L[2] = m2l_fma(-D[63], m, L[2]);
      L[3] = m2l_fma(-D[64], m, L[3]);
    }
    { const T m = __ldg(Ms + 40);
      L[0] = m2l_fma(D[40], m, L[0]);
      L[1] = m2l_fma(-D[61], m, L[1]);
      L[2] = m2l_fma(-D[64], m, L[2]);
      L[3] = m2l_fma(-D[65], m, L[3]);
    }
    { const T m = __ldg(Ms + 41);
      L[0] = m2l_fma(D[41], m, L[0]);
      L[1] = m2l_fma(-D[62], m, L[1]);
      L[2] = m2l_fma(-D[66], m, L[2]);
      L[3] = m2l_fma(-D[67], m, L[3]);
    }
    { const T m = __ldg(Ms + 42);
      L[0] = m2l_fma(D[42], m, L[0]);
      L[1] = m2l_fma(-D[63], m, L[1]);
      L[2] = m2l_fma(-D[67], m, L[2]);
      L[3] = m2l_fma(-D[68], m, L[3]);
    }
    { const T m = __ldg(Ms + 43);
      L[0] = m2l_fma(D[43], m, L[0]);
      L[1] = m2l_fma(-D[64], m, L[1]);
      L[2] = m2l_fma(-D[68], m, L[2]);
      L[3] = m2l_fma(-D[69], m, L[3]);
    }
    { const T m = __ldg(Ms + 44);
      L[0] = m2l_fma(D[44], m, L[0]);
      L[1] = m2l_fma(-D[65], m, L[1]);
      L[2] = m2l_fma(-D[69], m, L[2]);
      L[3] = m2l_fma(-D[70], m, L[3]);
    }
    { const T m = __ldg(Ms + 45);
      L[0] = m2l_fma(D[45], m, L[0]);
      L[1] = m2l_fma(-D[66], m, L[1]);
      L[2] = m2l_fma(-D[71], m, L[2]);
      L[3] = m2l_fma(-D[72], m, L[3]);
    }
    { const T m = __ldg(Ms + 46);
      L[0] = m2l_fma(D[46], m, L[0]);
      L[1] = m2l_fma(-D[67], m, L[1]);
      L[2] = m2l_fma(-D[72], m, L[2]);
      L[3] = m2l_fma(-D[73], m, L[3]);
    }
    { const T m = __ldg(Ms + 47);
      L[0] = m2l_fma(D[47], m, L[0]);
      L[1] = m2l_fma(-D[68], m, L[1]);
      L[2] = m2l_fma(-D[73], m, L[2]);
      L[3] = m2l_fma(-D[74], m, L[3]);
    }
    { const T m = __ldg(Ms + 48);
      L[0] = m2l_fma(D[48], m, L[0]);
      L[1] = m2l_fma(-D[69], m, L[1]);
      L[2] = m2l_fma(-D[74], m, L[2]);
      L[3] = m2l_fma(-D[75], m, L[3]);
    }
    { const T m = __ldg(Ms + 49);
      L[0] = m2l_fma(D[49], m, L[0]);
      L[1] = m2l_fma(-D[70], m, L[1]);
      L[2] = m2l_fma(-D[75], m, L[2]);
      L[3] = m2l_fma(-D[76], m, L[3]);
    }
    { const T m = __ldg(Ms + 50);
      L[0] = m2l_fma(D[50], m, L[0]);
      L[1] = m2l_fma(-D[71], m, L[1]);
      L[2] = m2l_fma(-D[77], m, L[2]);
      L[3] = m2l_fma(-D[78], m, L[3]);
    }
    { const T m = __ldg(Ms + 51);
      L[0] = m2l_fma(D[51], m, L[0]);
      L[1] = m2l_fma(-D[72], m, L[1]);
      L[2] = m2l_fma(-D[78], m, L[2]);
      L[3] = m2l_fma(-D[79], m, L[3]);
    }
    { const T m = __ldg(Ms + 52);
      L[0] = m2l_fma(D[52], m, L[0]);
      L[1] = m2l_fma(-D[73], m, L[1]);
      L[2] = m2l_fma(-D[79], m, L[2]);
      L[3] = m2l_fma(-D[80], m, L[3]);
    }
    { const T m = __ldg(Ms + 53);
      L[0] = m2l_fma(D[53], m, L[0]);
      L[1] = m2l_fma(-D[74], m, L[1]);
      L[2] = m2l_fma(-D[80], m, L[2]);
      L[3] = m2l_fma(-D[81], m, L[3]);
    }
    { const T m = __ldg(Ms + 54);
      L[0] = m2l_fma(D[54], m, L[0]);
      L[1] = m2l_fma(-D[75], m, L[1]);
      L[2] = m2l_fma(-D[81], m, L[2]);
      L[3] = m2l_fma(-D[82], m, L[3]);
    }
    { const T m = __ldg(Ms + 55);
      L[0] = m2l_fma(D[55], m, L[0]);
      L[1] = m2l_fma(-D[76], m, L[1]);
      L[2] = m2l_fma(-D[82], m, L[2]);
      L[3] = m2l_fma(-D[83], m, L[3]);
    }
    { const T m = __ldg(Ms + 56);
      L[0] = m2l_fma(D[56], m, L[0]);
    }
    { const T m = __ldg(Ms + 57);
      L[0] = m2l_fma(D[57], m, L[0]);
    }
    { const T m = __ldg(Ms + 58);
      L[0] = m2l_fma(D[58], m, L[0]);
    }
    { const T m = __ldg(Ms + 59);
      L[0] = m2l_fma(D[59], m, L[0]);
    }
    { const T m = __ldg(Ms + 60);
      L[0] = m2l_fma(D[60], m, L[0]);
    }
    { const T m = __ldg(Ms + 61);
      L[0] = m2l_fma(D[61], m, L[0]);
    }
    { const T m = __ldg(Ms + 62);
      L[0] = m2l_fma(D[62], m, L[0]);
    }
    { const T m = __ldg(Ms + 63);
      L[0] = m2l_fma(D[63], m, L[0]);
    }
    { const T m = __ldg(Ms + 64);
      L[0] = m2l_fma(D[64], m, L[0]);
    }
    { const T m = __ldg(Ms + 65);
      L[0] = m2l_fma(D[65], m, L[0]);
    }
    { const T m = __ldg(Ms + 66);
      L[0] = m2l_fma(D[66], m, L[0]);
    }
    { const T m = __ldg(Ms + 67);
      L[0] = m2l_fma(D[67], m, L[0]);
    }
    { const T m = __ldg(Ms + 68);
      L[0] = m2l_fma(D[68], m, L[0]);
    }
    { const T m = __ldg(Ms + 69);
      L[0] = m2l_fma(D[69], m, L[0]);
    }
    { const T m = __ldg(Ms + 70);
      L[0] = m2l_fma(D[70], m, L[0]);
    }
    { const T m = __ldg(Ms + 71);
      L[0] = m2l_fma(D[71], m, L[0]);
    }
    { const T m = __ldg(Ms + 72);
      L[0] = m2l_fma(D[72], m, L[0]);
    }
    { const T m = __ldg(Ms + 73);
      L[0] = m2l_fma(D[73], m, L[0]);
    }
    { const T m = __ldg(Ms + 74);
      L[0] = m2l_fma(D[74], m, L[0]);
    }
    { const T m = __ldg(Ms + 75);
      L[0] = m2l_fma(D[75], m, L[0]);
    }
    { const T m = __ldg(Ms + 76);
      L[0] = m2l_fma(D[76], m, L[0]);
    }
    { const T m = __ldg(Ms + 77);
      L[0] = m2l_fma(D[77], m, L[0]);
    }
    { const T m = __ldg(Ms + 78);
      L[0] = m2l_fma(D[78], m, L[0]);
    }
    { const T m = __ldg(Ms + 79);
      L[0] = m2l_fma(D[79], m, L[0]);
    }
    { const T m = __ldg(Ms + 80);
      L[0] = m2l_fma(D[80], m, L[0]);
    }
    { const T m = __ldg(Ms + 81);
      L[0] = m2l_fma(D[81], m, L[0]);
    }
    { const T m = __ldg(Ms + 82);
      L[0] = m2l_fma(D[82], m, L[0]);
    }
    { const T m = __ldg(Ms + 83);
      L[0] = m2l_fma(D[83], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_a_forces_6(const T (&D)[84], const T *__restrict__ Ms, T rho, T (&L)[84])
{
    L[0] = T(0);
    T rp = T(1);
    { const T m = __ldg(Ms + 0) * rp;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[9] * m;
      L[10] = D[10] * m;
      L[11] = D[11] * m;
      L[12] = D[12] * m;
      L[13] = D[13] * m;
      L[14] = D[14] * m;
      L[15] = D[15] * m;
      L[16] = D[16] * m;
      L[17] = D[17] * m;
      L[18] = D[18] * m;
      L[19] = D[19] * m;
      L[20] = D[20] * m;
      L[21] = D[21] * m;
      L[22] = D[22] * m;
      L[23] = D[23] * m;
      L[24] = D[24] * m;
      L[25] = D[25] * m;
      L[26] = D[26] * m;
      L[27] = D[27] * m;
      L[28] = D[28] * m;
      L[29] = D[29] * m;
      L[30] = D[30] * m;
      L[31] = D[31] * m;
      L[32] = D[32] * m;
      L[33] = D[33] * m;
      L[34] = D[34] * m;
      L[35] = D[35] * m;
      L[36] = D[36] * m;
      L[37] = D[37] * m;
      L[38] = D[38] * m;
      L[39] = D[39] * m;
      L[40] = D[40] * m;
      L[41] = D[41] * m;
      L[42] = D[42] * m;
      L[43] = D[43] * m;
      L[44] = D[44] * m;
      L[45] = D[45] * m;
      L[46] = D[46] * m;
      L[47] = D[47] * m;
      L[48] = D[48] * m;
      L[49] = D[49] * m;
      L[50] = D[50] * m;
      L[51] = D[51] * m;
      L[52] = D[52] * m;
      L[53] = D[53] * m;
      L[54] = D[54] * m;
      L[55] = D[55] * m;
      L[56] = D[56] * m;
      L[57] = D[57] * m;
      L[58] = D[58] * m;
      L[59] = D[59] * m;
      L[60] = D[60] * m;
      L[61] = D[61] * m;
      L[62] = D[62] * m;
      L[63] = D[63] * m;
      L[64] = D[64] * m;
      L[65] = D[65] * m;
      L[66] = D[66] * m;
      L[67] = D[67] * m;
      L[68] = D[68] * m;
      L[69] = D[69] * m;
      L[70] = D[70] * m;
      L[71] = D[71] * m;
      L[72] = D[72] * m;
      L[73] = D[73] * m;
      L[74] = D[74] * m;
      L[75] = D[75] * m;
      L[76] = D[76] * m;
      L[77] = D[77] * m;
      L[78] = D[78] * m;
      L[79] = D[79] * m;
      L[80] = D[80] * m;
      L[81] = D[81] * m;
      L[82] = D[82] * m;
      L[83] = D[83] * m;
    }
    rp *= rho;
    { const T m = -__ldg(Ms + 1) * rp;
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[15], m, L[9]);
      L[10] = m2l_fma(D[20], m, L[10]);
      L[11] = m2l_fma(D[21], m, L[11]);
      L[12] = m2l_fma(D[22], m, L[12]);
      L[13] = m2l_fma(D[23], m, L[13]);
      L[14] = m2l_fma(D[24], m, L[14]);
      L[15] = m2l_fma(D[25], m, L[15]);
      L[16] = m2l_fma(D[26], m, L[16]);
      L[17] = m2l_fma(D[27], m, L[17]);
      L[18] = m2l_fma(D[28], m, L[18]);
      L[19] = m2l_fma(D[29], m, L[19]);
      L[20] = m2l_fma(D[35], m, L[20]);
      L[21] = m2l_fma(D[36], m, L[21]);
      L[22] = m2l_fma(D[37], m, L[22]);
      L[23] = m2l_fma(D[38], m, L[23]);
      L[24] = m2l_fma(D[39], m, L[24]);
      L[25] = m2l_fma(D[40], m, L[25]);
      L[26] = m2l_fma(D[41], m, L[26]);
      L[27] = m2l_fma(D[42], m, L[27]);
      L[28] = m2l_fma(D[43], m, L[28]);
      L[29] = m2l_fma(D[44], m, L[29]);
      L[30] = m2l_fma(D[45], m, L[30]);
      L[31] = m2l_fma(D[46], m, L[31]);
      L[32] = m2l_fma(D[47], m, L[32]);
      L[33] = m2l_fma(D[48], m, L[33]);
      L[34] = m2l_fma(D[49], m, L[34]);
      L[35] = m2l_fma(D[56], m, L[35]);
      L[36] = m2l_fma(D[57], m, L[36]);
      L[37] = m2l_fma(D[58], m, L[37]);
      L[38] = m2l_fma(D[59], m, L[38]);
      L[39] = m2l_fma(D[60], m, L[39]);
      L[40] = m2l_fma(D[61], m, L[40]);
      L[41] = m2l_fma(D[62], m, L[41]);
      L[42] = m2l_fma(D[63], m, L[42]);
      L[43] = m2l_fma(D[64], m, L[43]);
      L[44] = m2l_fma(D[65], m, L[44]);
      L[45] = m2l_fma(D[66], m, L[45]);
      L[46] = m2l_fma(D[67], m, L[46]);
      L[47] = m2l_fma(D[68], m, L[47]);
      L[48] = m2l_fma(D[69], m, L[48]);
      L[49] = m2l_fma(D[70], m, L[49]);
      L[50] = m2l_fma(D[71], m, L[50]);
      L[51] = m2l_fma(D[72], m, L[51]);
      L[52] = m2l_fma(D[73], m, L[52]);
      L[53] = m2l_fma(D[74], m, L[53]);
      L[54] = m2l_fma(D[75], m, L[54]);
      L[55] = m2l_fma(D[76], m, L[55]);
    }
    { const T m = -__ldg(Ms + 2) * rp;
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[18], m, L[9]);
      L[10] = m2l_fma(D[21], m, L[10]);
      L[11] = m2l_fma(D[23], m, L[11]);
      L[12] = m2l_fma(D[24], m, L[12]);
      L[13] = m2l_fma(D[26], m, L[13]);
      L[14] = m2l_fma(D[27], m, L[14]);
      L[15] = m2l_fma(D[28], m, L[15]);
      L[16] = m2l_fma(D[30], m, L[16]);
      L[17] = m2l_fma(D[31], m, L[17]);
      L[18] = m2l_fma(D[32], m, L[18]);
      L[19] = m2l_fma(D[33], m, L[19]);
      L[20] = m2l_fma(D[36], m, L[20]);
      L[21] = m2l_fma(D[38], m, L[21]);
      L[22] = m2l_fma(D[39], m, L[22]);
      L[23] = m2l_fma(D[41], m, L[23]);
      L[24] = m2l_fma(D[42], m, L[24]);
      L[25] = m2l_fma(D[43], m, L[25]);
      L[26] = m2l_fma(D[45], m, L[26]);
      L[27] = m2l_fma(D[46], m, L[27]);
      L[28] = m2l_fma(D[47], m, L[28]);
      L[29] = m2l_fma(D[48], m, L[29]);
      L[30] = m2l_fma(D[50], m, L[30]);
      L[31] = m2l_fma(D[51], m, L[31]);
      L[32] = m2l_fma(D[52], m, L[32]);
      L[33] = m2l_fma(D[53], m, L[33]);
      L[34] = m2l_fma(D[54], m, L[34]);
      L[35] = m2l_fma(D[57], m, L[35]);
      L[36] = m2l_fma(D[59], m, L[36]);
      L[37] = m2l_fma(D[60], m, L[37]);
      L[38] = m2l_fma(D[62], m, L[38]);
      L[39] = m2l_fma(D[63], m, L[39]);
      L[40] = m2l_fma(D[64], m, L[40]);
      L[41] = m2l_fma(D[66], m, L[41]);
      L[42] = m2l_fma(D[67], m, L[42]);
      L[43] = m2l_fma(D[68], m, L[43]);
      L[44] = m2l_fma(D[69], m, L[44]);
      L[45] = m2l_fma(D[71], m, L[45]);
      L[46] = m2l_fma(D[72], m, L[46]);
      L[47] = m2l_fma(D[73], m, L[47]);
      L[48] = m2l_fma(D[74], m, L[48]);
      L[49] = m2l_fma(D[75], m, L[49]);
      L[50] = m2l_fma(D[77], m, L[50]);
      L[51] = m2l_fma(D[78], m, L[51]);
      L[52] = m2l_fma(D[79], m, L[52]);
      L[53] = m2l_fma(D[80], m, L[53]);
      L[54] = m2l_fma(D[81], m, L[54]);
      L[55] = m2l_fma(D[82], m, L[55]);
    }
    { const T m = -__ldg(Ms + 3) * rp;
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(D[22], m, L[10]);
      L[11] = m2l_fma(D[24], m, L[11]);
      L[12] = m2l_fma(D[25], m, L[12]);
      L[13] = m2l_fma(D[27], m, L[13]);
      L[14] = m2l_fma(D[28], m, L[14]);
      L[15] = m2l_fma(D[29], m, L[15]);
      L[16] = m2l_fma(D[31], m, L[16]);
      L[17] = m2l_fma(D[32], m, L[17]);
      L[18] = m2l_fma(D[33], m, L[18]);
      L[19] = m2l_fma(D[34], m, L[19]);
      L[20] = m2l_fma(D[37], m, L[20]);
      L[21] = m2l_fma(D[39], m, L[21]);
      L[22] = m2l_fma(D[40], m, L[22]);
      L[23] = m2l_fma(D[42], m, L[23]);
      L[24] = m2l_fma(D[43], m, L[24]);
      L[25] = m2l_fma(D[44], m, L[25]);
      L[26] = m2l_fma(D[46], m, L[26]);
      L[27] = m2l_fma(D[47], m, L[27]);
      L[28] = m2l_fma(D[48], m, L[28]);
      L[29] = m2l_fma(D[49], m, L[29]);
      L[30] = m2l_fma(D[51], m, L[30]);
      L[31] = m2l_fma(D[52], m, L[31]);
      L[32] = m2l_fma(D[53], m, L[32]);
      L[33] = m2l_fma(D[54], m, L[33]);
      L[34] = m2l_fma(D[55], m, L[34]);
      L[35] = m2l_fma(D[58], m, L[35]);
      L[36] = m2l_fma(D[60], m, L[36]);
      L[37] = m2l_fma(D[61], m, L[37]);
      L[38] = m2l_fma(D[63], m, L[38]);
      L[39] = m2l_fma(D[64], m, L[39]);
      L[40] = m2l_fma(D[65], m, L[40]);
      L[41] = m2l_fma(D[67], m, L[41]);
      L[42] = m2l_fma(D[68], m, L[42]);
      L[43] = m2l_fma(D[69], m, L[43]);
      L[44] = m2l_fma(D[70], m, L[44]);
      L[45] = m2l_fma(D[72], m, L[45]);
      L[46] = m2l_fma(D[73], m, L[46]);
      L[47] = m2l_fma(D[74], m, L[47]);
      L[48] = m2l_fma(D[75], m, L[48]);
      L[49] = m2l_fma(D[76], m, L[49]);
      L[50] = m2l_fma(D[78], m, L[50]);
      L[51] = m2l_fma(D[79], m, L[51]);
      L[52] = m2l_fma(D[80], m, L[52]);
      L[53] = m2l_fma(D[81], m, L[53]);
      L[54] = m2l_fma(D[82], m, L[54]);
      L[55] = m2l_fma(D[83], m, L[55]);
    }
    rp *= rho;
    { const T m = __ldg(Ms + 4) * rp;
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[21], m, L[5]);
      L[6] = m2l_fma(D[22], m, L[6]);
      L[7] = m2l_fma(D[23], m, L[7]);
      L[8] = m2l_fma(D[24], m, L[8]);
      L[9] = m2l_fma(D[25], m, L[9]);
      L[10] = m2l_fma(D[35], m, L[10]);
      L[11] = m2l_fma(D[36], m, L[11]);
      L[12] = m2l_fma(D[37], m, L[12]);
      L[13] = m2l_fma(D[38], m, L[13]);
      L[14] = m2l_fma(D[39], m, L[14]);
      L[15] = m2l_fma(D[40], m, L[15]);
      L[16] = m2l_fma(D[41], m, L[16]);
      L[17] = m2l_fma(D[42], m, L[17]);
      L[18] = m2l_fma(D[43], m, L[18]);
      L[19] = m2l_fma(D[44], m, L[19]);
      L[20] = m2l_fma(D[56], m, L[20]);
      L[21] = m2l_fma(D[57], m, L[21]);
      L[22] = m2l_fma(D[58], m, L[22]);
      L[23] = m2l_fma(D[59], m, L[23]);
      L[24] = m2l_fma(D[60], m, L[24]);
      L[25] = m2l_fma(D[61], m, L[25]);
      L[26] = m2l_fma(D[62], m, L[26]);
      L[27] = m2l_fma(D[63], m, L[27]);
      L[28] = m2l_fma(D[64], m, L[28]);
      L[29] = m2l_fma(D[65], m, L[29]);
      L[30] = m2l_fma(D[66], m, L[30]);
      L[31] = m2l_fma(D[67], m, L[31]);
      L[32] = m2l_fma(D[68], m, L[32]);
      L[33] = m2l_fma(D[69], m, L[33]);
      L[34] = m2l_fma(D[70], m, L[34]);
    }
    { const T m = __ldg(Ms + 5) * rp;
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(D[28], m, L[9]);
      L[10] = m2l_fma(D[36], m, L[10]);
      L[11] = m2l_fma(D[38], m, L[11]);
      L[12] = m2l_fma(D[39], m, L[12]);
      L[13] = m2l_fma(D[41], m, L[13]);
      L[14] = m2l_fma(D[42], m, L[14]);
      L[15] = m2l_fma(D[43], m, L[15]);
      L[16] = m2l_fma(D[45], m, L[16]);
      L[17] = m2l_fma(D[46], m, L[17]);
      L[18] = m2l_fma(D[47], m, L[18]);
      L[19] = m2l_fma(D[48], m, L[19]);
      L[20] = m2l_fma(D[57], m, L[20]);
      L[21] = m2l_fma(D[59], m, L[21]);
      L[22] = m2l_fma(D[60], m, L[22]);
      L[23] = m2l_fma(D[62], m, L[23]);
      L[24] = m2l_fma(D[63], m, L[24]);
      L[25] = m2l_fma(D[64], m, L[25]);
      L[26] = m2l_fma(D[66], m, L[26]);
      L[27] = m2l_fma(D[67], m, L[27]);
      L[28] = m2l_fma(D[68], m, L[28]);
      L[29] = m2l_fma(D[69], m, L[29]);
      L[30] = m2l_fma(D[71], m, L[30]);
      L[31] = m2l_fma(D[72], m, L[31]);
      L[32] = m2l_fma(D[73], m, L[32]);
      L[33] = m2l_fma(D[74], m, L[33]);
      L[34] = m2l_fma(D[75], m, L[34]);
    }
    { const T m = __ldg(Ms + 6) * rp;
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[24], m, L[5]);
      L[6] = m2l_fma(D[25], m, L[6]);
      L[7] = m2l_fma(D[27], m, L[7]);
      L[8] = m2l_fma(D[28], m, L[8]);
      L[9] = m2l_fma(D[29], m, L[9]);
      L[10] = m2l_fma(D[37], m, L[10]);
      L[11] = m2l_fma(D[39], m, L[11]);
      L[12] = m2l_fma(D[40], m, L[12]);
      L[13] = m2l_fma(D[42], m, L[13]);
      L[14] = m2l_fma(D[43], m, L[14]);
      L[15] = m2l_fma(D[44], m, L[15]);
      L[16] = m2l_fma(D[46], m, L[16]);
      L[17] = m2l_fma(D[47], m, L[17]);
      L[18] = m2l_fma(D[48], m, L[18]);
      L[19] = m2l_fma(D[49], m, L[19]);
      L[20] = m2l_fma(D[58], m, L[20]);
      L[21] = m2l_fma(D[60], m, L[21]);
      L[22] = m2l_fma(D[61], m, L[22]);
      L[23] = m2l_fma(D[63], m, L[23]);
      L[24] = m2l_fma(D[64], m, L[24]);
      L[25] = m2l_fma(D[65], m, L[25]);
      L[26] = m2l_fma(D[67], m, L[26]);
      L[27] = m2l_fma(D[68], m, L[27]);
      L[28] = m2l_fma(D[69], m, L[28]);
      L[29] = m2l_fma(D[70], m, L[29]);
      L[30] = m2l_fma(D[72], m, L[30]);
      L[31] = m2l_fma(D[73], m, L[31]);
      L[32] = m2l_fma(D[74], m, L[32]);
      L[33] = m2l_fma(D[75], m, L[33]);
      L[34] = m2l_fma(D[76], m, L[34]);
    }
    { const T m = __ldg(Ms + 7) * rp;
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[30], m, L[7]);
      L[8] = m2l_fma(D[31], m, L[8]);
      L[9] = m2l_fma(D[32], m, L[9]);
      L[10] = m2l_fma(D[38], m, L[10]);
      L[11] = m2l_fma(D[41], m, L[11]);
      L[12] = m2l_fma(D[42], m, L[12]);
      L[13] = m2l_fma(D[45], m, L[13]);
      L[14] = m2l_fma(D[46], m, L[14]);
      L[15] = m2l_fma(D[47], m, L[15]);
      L[16] = m2l_fma(D[50], m, L[16]);
      L[17] = m2l_fma(D[51], m, L[17]);
      L[18] = m2l_fma(D[52], m, L[18]);
      L[19] = m2l_fma(D[53], m, L[19]);
      L[20] = m2l_fma(D[59], m, L[20]);
      L[21] = m2l_fma(D[62], m, L[21]);
      L[22] = m2l_fma(D[63], m, L[22]);
      L[23] = m2l_fma(D[66], m, L[23]);
      L[24] = m2l_fma(D[67], m, L[24]);
      L[25] = m2l_fma(D[68], m, L[25]);
      L[26] = m2l_fma(D[71], m, L[26]);
      L[27] = m2l_fma(D[72], m, L[27]);
      L[28] = m2l_fma(D[73], m, L[28]);
      L[29] = m2l_fma(D[74], m, L[29]);
      L[30] = m2l_fma(D[77], m, L[30]);
      L[31] = m2l_fma(D[78], m, L[31]);
      L[32] = m2l_fma(D[79], m, L[32]);
      L[33] = m2l_fma(D[80], m, L[33]);
      L[34] = m2l_fma(D[81], m, L[34]);
    }
    { const T m = __ldg(Ms + 8) * rp;
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
      L[4] = m2l_fma(D[24], m, L[4]);
      L[5] = m2l_fma(D[27], m, L[5]);
      L[6] = m2l_fma(D[28], m, L[6]);
      L[7] = m2l_fma(D[31], m, L[7]);
      L[8] = m2l_fma(D[32], m, L[8]);
      L[9] = m2l_fma(D[33], m, L[9]);
      L[10] = m2l_fma(D[39], m, L[10]);
      L[11] = m2l_fma(D[42], m, L[11]);
      L[12] = m2l_fma(D[43], m, L[12]);
      L[13] = m2l_fma(D[46], m, L[13]);
      L[14] = m2l_fma(D[47], m, L[14]);
      L[15] = m2l_fma(D[48], m, L[15]);
      L[16] = m2l_fma(D[51], m, L[16]);
      L[17] = m2l_fma(D[52], m, L[17]);
      L[18] = m2l_fma(D[53], m, L[18]);
      L[19] = m2l_fma(D[54], m, L[19]);
      L[20] = m2l_fma(D[60], m, L[20]);
      L[21] = m2l_fma(D[63], m, L[21]);
      L[22] = m2l_fma(D[64], m, L[22]);
      L[23] = m2l_fma(D[67], m, L[23]);
      L[24] = m2l_fma(D[68], m, L[24]);
      L[25] = m2l_fma(D[69], m, L[25]);
      L[26] = m2l_fma(D[72], m, L[26]);
      L[27] = m2l_fma(D[73], m, L[27]);
      L[28] = m2l_fma(D[74], m, L[28]);
      L[29] = m2l_fma(D[75], m, L[29]);
      L[30] = m2l_fma(D[78], m, L[30]);
      L[31] = m2l_fma(D[79], m, L[31]);
      L[32] = m2l_fma(D[80], m, L[32]);
      L[33] = m2l_fma(D[81], m, L[33]);
      L[34] = m2l_fma(D[82], m, L[34]);
    }
    { const T m = __ldg(Ms + 9) * rp;
      L[1] = m2l_fma(D[15], m, L[1]);
      L[2] = m2l_fma(D[18], m, L[2]);
      L[3] = m2l_fma(D[19], m, L[3]);
      L[4] = m2l_fma(D[25], m, L[4]);
      L[5] = m2l_fma(D[28], m, L[5]);
      L[6] = m2l_fma(D[29], m, L[6]);
      L[7] = m2l_fma(D[32], m, L[7]);
      L[8] = m2l_fma(D[33], m, L[8]);
      L[9] = m2l_fma(D[34], m, L[9]);
      L[10] = m2l_fma(D[40], m, L[10]);
      L[11] = m2l_fma(D[43], m, L[11]);
      L[12] = m2l_fma(D[44], m, L[12]);
      L[13] = m2l_fma(D[47], m, L[13]);
      L[14] = m2l_fma(D[48], m, L[14]);
      L[15] = m2l_fma(D[49], m, L[15]);
      L[16] = m2l_fma(D[52], m, L[16]);
      L[17] = m2l_fma(D[53], m, L[17]);
      L[18] = m2l_fma(D[54], m, L[18]);
      L[19] = m2l_fma(D[55], m, L[19]);
      L[20] = m2l_fma(D[61], m, L[20]);
      L[21] = m2l_fma(D[64], m, L[21]);
      L[22] = m2l_fma(D[65], m, L[22]);
      L[23] = m2l_fma(D[68], m, L[23]);
      L[24] = m2l_fma(D[69], m, L[24]);
      L[25] = m2l_fma(D[70], m, L[25]);
      L[26] = m2l_fma(D[73], m, L[26]);
      L[27] = m2l_fma(D[74], m, L[27]);
      L[28] = m2l_fma(D[75], m, L[28]);
      L[29] = m2l_fma(D[76], m, L[29]);
      L[30] = m2l_fma(D[79], m, L[30]);
      L[31] = m2l_fma(D[80], m, L[31]);
      L[32] = m2l_fma(D[81], m, L[32]);
      L[33] = m2l_fma(D[82], m, L[33]);
      L[34] = m2l_fma(D[83], m, L[34]);
    }
    rp *= rho;
    { const T m = -__ldg(Ms + 10) * rp;
      L[1] = m2l_fma(D[20], m, L[1]);
      L[2] = m2l_fma(D[21], m, L[2]);
      L[3] = m2l_fma(D[22], m, L[3]);
      L[4] = m2l_fma(D[35], m, L[4]);
      L[5] = m2l_fma(D[36], m, L[5]);
      L[6] = m2l_fma(D[37], m, L[6]);
      L[7] = m2l_fma(D[38], m, L[7]);
      L[8] = m2l_fma(D[39], m, L[8]);
      L[9] = m2l_fma(D[40], m, L[9]);
      L[10] = m2l_fma(D[56], m, L[10]);
      L[11] = m2l_fma(D[57], m, L[11]);
      L[12] = m2l_fma(D[58], m, L[12]);
      L[13] = m2l_fma(D[59], m, L[13]);
      L[14] = m2l_fma(D[60], m, L[14]);
      L[15] = m2l_fma(D[61], m, L[15]);
      L[16] = m2l_fma(D[62], m, L[16]);
      L[17] = m2l_fma(D[63], m, L[17]);
      L[18] = m2l_fma(D[64], m, L[18]);
      L[19] = m2l_fma(D[65], m, L[19]);
    }
    { const T m = -__ldg(Ms + 11) * rp;
      L[1] = m2l_fma(D[21], m, L[1]);
      L[2] = m2l_fma(D[23], m, L[2]);
      L[3] = m2l_fma(D[24], m, L[3]);
      L[4] = m2l_fma(D[36], m, L[4]);
      L[5] = m2l_fma(D[38], m, L[5]);
      L[6] = m2l_fma(D[39], m, L[6]);
      L[7] = m2l_fma(D[41], m, L[7]);
      L[8] = m2l_fma(D[42], m, L[8]);
      L[9] = m2l_fma(D[43], m, L[9]);
      L[10] = m2l_fma(D[57], m, L[10]);
      L[11] = m2l_fma(D[59], m, L[11]);
      L[12] = m2l_fma(D[60], m, L[12]);
      L[13] = m2l_fma(D[62], m, L[13]);
      L[14] = m2l_fma(D[63], m, L[14]);
      L[15] = m2l_fma(D[64], m, L[15]);
      L[16] = m2l_fma(D[66], m, L[16]);
      L[17] = m2l_fma(D[67], m, L[17]);
      L[18] = m2l_fma(D[68], m, L[18]);
      L[19] = m2l_fma(D[69], m, L[19]);
    }
    { const T m = -__ldg(Ms + 12) * rp;
      L[1] = m2l_fma(D[22], m, L[1]);
      L[2] = m2l_fma(D[24], m, L[2]);
      L[3] = m2l_fma(D[25], m, L[3]);
      L[4] = m2l_fma(D[37], m, L[4]);
      L[5] = m2l_fma(D[39], m, L[5]);
      L[6] = m2l_fma(D[40], m, L[6]);
      L[7] = m2l_fma(D[42], m, L[7]);
      L[8] = m2l_fma(D[43], m, L[8]);
      L[9] = m2l_fma(D[44], m, L[9]);
      L[10] = m2l_fma(D[58], m, L[10]);
      L[11] = m2l_fma(D[60], m, L[11]);
      L[12] = m2l_fma(D[61], m, L[12]);
      L[13] = m2l_fma(D[63], m, L[13]);
      L[14] = m2l_fma(D[64], m, L[14]);
      L[15] = m2l_fma(D[65], m, L[15]);
      L[16] = m2l_fma(D[67], m, L[16]);
      L[17] = m2l_fma(D[68], m, L[17]);
      L[18] = m2l_fma(D[69], m, L[18]);
      L[19] = m2l_fma(D[70], m, L[19]);
    }
    { const T m = -__ldg(Ms + 13) * rp;
      L[1] = m2l_fma(D[23], m, L[1]);
      L[2] = m2l_fma(D[26], m, L[2]);
      L[3] = m2l_fma(D[27], m, L[3]);
      L[4] = m2l_fma(D[38], m, L[4]);
      L[5] = m2l_fma(D[41], m, L[5]);
      L[6] = m2l_fma(D[42], m, L[6]);
      L[7] = m2l_fma(D[45], m, L[7]);
      L[8] = m2l_fma(D[46], m, L[8]);
      L[9] = m2l_fma(D[47], m, L[9]);
      L[10] = m2l_fma(D[59], m, L[10]);
      L[11] = m2l_fma(D[62], m, L[11]);
      L[12] = m2l_fma(D[63], m, L[12]);
      L[13] = m2l_fma(D[66], m, L[13]);
      L[14] = m2l_fma(D[67], m, L[14]);
      L[15] = m2l_fma(D[68], m, L[15]);
      L[16] = m2l_fma(D[71], m, L[16]);
      L[17] = m2l_fma(D[72], m, L[17]);
      L[18] = m2l_fma(D[73], m, L[18]);
      L[19] = m2l_fma(D[74], m, L[19]);
    }
    { const T m = -__ldg(Ms + 14) * rp;
      L[1] = m2l_fma(D[24], m, L[1]);
      L[2] = m2l_fma(D[27], m, L[2]);
      L[3] = m2l_fma(D[28], m, L[3]);
      L[4] = m2l_fma(D[39], m, L[4]);
      L[5] = m2l_fma(D[42], m, L[5]);
      L[6] = m2l_fma(D[43], m, L[6]);
      L[7] = m2l_fma(D[46], m, L[7]);
      L[8] = m2l_fma(D[47], m, L[8]);
      L[9] = m2l_fma(D[48], m, L[9]);
      L[10] = m2l_fma(D[60], m, L[10]);
      L[11] = m2l_fma(D[63], m, L[11]);
      L[12] = m2l_fma(D[64], m, L[12]);
      L[13] = m2l_fma(D[67], m, L[13]);
      L[14] = m2l_fma(D[68], m, L[14]);
      L[15] = m2l_fma(D[69], m, L[15]);
      L[16] = m2l_fma(D[72], m, L[16]);
      L[17] = m2l_fma(D[73], m, L[17]);
      L[18] = m2l_fma(D[74], m, L[18]);
      L[19] = m2l_fma(D[75], m, L[19]);
    }
    { const T m = -__ldg(Ms + 15) * rp;
      L[1] = m2l_fma(D[25], m, L[1]);
      L[2] = m2l_fma(D[28], m, L[2]);
      L[3] = m2l_fma(D[29], m, L[3]);
      L[4] = m2l_fma(D[40], m, L[4]);
      L[5] = m2l_fma(D[43], m, L[5]);
      L[6] = m2l_fma(D[44], m, L[6]);
      L[7] = m2l_fma(D[47], m, L[7]);
      L[8] = m2l_fma(D[48], m, L[8]);
      L[9] = m2l_fma(D[49], m, L[9]);
      L[10] = m2l_fma(D[61], m, L[10]);
      L[11] = m2l_fma(D[64], m, L[11]);
      L[12] = m2l_fma(D[65], m, L[12]);
      L[13] = m2l_fma(D[68], m, L[13]);
      L[14] = m2l_fma(D[69], m, L[14]);
      L[15] = m2l_fma(D[70], m, L[15]);
      L[16] = m2l_fma(D[73], m, L[16]);
      L[17] = m2l_fma(D[74], m, L[17]);
      L[18] = m2l_fma(D[75], m, L[18]);
      L[19] = m2l_fma(D[76], m, L[19]);
    }
    { const T m = -__ldg(Ms + 16) * rp;
      L[1] = m2l_fma(D[26], m, L[1]);
      L[2] = m2l_fma(D[30], m, L[2]);
      L[3] = m2l_fma(D[31], m, L[3]);
      L[4] = m2l_fma(D[41], m, L[4]);
      L[5] = m2l_fma(D[45], m, L[5]);
      L[6] = m2l_fma(D[46], m, L[6]);
      L[7] = m2l_fma(D[50], m, L[7]);
      L[8] = m2l_fma(D[51], m, L[8]);
      L[9] = m2l_fma(D[52], m, L[9]);
      L[10] = m2l_fma(D[62], m, L[10]);
      L[11] = m2l_fma(D[66], m, L[11]);
      L[12] = m2l_fma(D[67], m, L[12]);
      L[13] = m2l_fma(D[71], m, L[13]);
      L[14] = m2l_fma(D[72], m, L[14]);
      L[15] = m2l_fma(D[73], m, L[15]);
      L[16] = m2l_fma(D[77], m, L[16]);
      L[17] = m2l_fma(D[78], m, L[17]);
      L[18] = m2l_fma(D[79], m, L[18]);
      L[19] = m2l_fma(D[80], m, L[19]);
    }
    { const T m = -__ldg(Ms + 17) * rp;
      L[1] = m2l_fma(D[27], m, L[1]);
      L[2] = m2l_fma(D[31], m, L[2]);
      L[3] = m2l_fma(D[32], m, L[3]);
      L[4] = m2l_fma(D[42], m, L[4]);
      L[5] = m2l_fma(D[46], m, L[5]);
      L[6] = m2l_fma(D[47], m, L[6]);
      L[7] = m2l_fma(D[51], m, L[7]);
      L[8] = m2l_fma(D[52], m, L[8]);
      L[9] = m2l_fma(D[53], m, L[9]);
      L[10] = m2l_fma(D[63], m, L[10]);
      L[11] = m2l_fma(D[67], m, L[11]);
      L[12] = m2l_fma(D[68], m, L[12]);
      L[13] = m2l_fma(D[72], m, L[13]);
      L[14] = m2l_fma(D[73], m, L[14]);
      L[15] = m2l_fma(D[74], m, L[15]);
      L[16] = m2l_fma(D[78], m, L[16]);
      L[17] = m2l_fma(D[79], m, L[17]);
      L[18] = m2l_fma(D[80], m, L[18]);
      L[19] = m2l_fma(D[81], m, L[19]);
    }
    { const T m = -__ldg(Ms + 18) * rp;
      L[1] = m2l_fma(D[28], m, L[1]);
      L[2] = m2l_fma(D[32], m, L[2]);
      L[3] = m2l_fma(D[33], m, L[3]);
      L[4] = m2l_fma(D[43], m, L[4]);
      L[5] = m2l_fma(D[47], m, L[5]);
      L[6] = m2l_fma(D[48], m, L[6]);
      L[7] = m2l_fma(D[52], m, L[7]);
      L[8] = m2l_fma(D[53], m, L[8]);
      L[9] = m2l_fma(D[54], m, L[9]);
      L[10] = m2l_fma(D[64], m, L[10]);
      L[11] = m2l_fma(D[68], m, L[11]);
      L[12] = m2l_fma(D[69], m, L[12]);
      L[13] = m2l_fma(D[73], m, L[13]);
      L[14] = m2l_fma(D[74], m, L[14]);
      L[15] = m2l_fma(D[75], m, L[15]);
      L[16] = m2l_fma(D[79], m, L[16]);
      L[17] = m2l_fma(D[80], m, L[17]);
      L[18] = m2l_fma(D[81], m, L[18]);
      L[19] = m2l_fma(D[82], m, L[19]);
    }
    { const T m = -__ldg(Ms + 19) * rp;
      L[1] = m2l_fma(D[29], m, L[1]);
      L[2] = m2l_fma(D[33], m, L[2]);
      L[3] = m2l_fma(D[34], m, L[3]);
      L[4] = m2l_fma(D[44], m, L[4]);
      L[5] = m2l_fma(D[48], m, L[5]);
      L[6] = m2l_fma(D[49], m, L[6]);
      L[7] = m2l_fma(D[53], m, L[7]);
      L[8] = m2l_fma(D[54], m, L[8]);
      L[9] = m2l_fma(D[55], m, L[9]);
      L[10] = m2l_fma(D[65], m, L[10]);
      L[11] = m2l_fma(D[69], m, L[11]);
      L[12] = m2l_fma(D[70], m, L[12]);
      L[13] = m2l_fma(D[74], m, L[13]);
      L[14] = m2l_fma(D[75], m, L[14]);
      L[15] = m2l_fma(D[76], m, L[15]);
      L[16] = m2l_fma(D[80], m, L[16]);
      L[17] = m2l_fma(D[81], m, L[17]);
      L[18] = m2l_fma(D[82], m, L[18]);
      L[19] = m2l_fma(D[83], m, L[19]);
    }
    rp *= rho;
    { const T m = __ldg(Ms + 20) * rp;
      L[1] = m2l_fma(D[35], m, L[1]);
      L[2] = m2l_fma(D[36], m, L[2]);
      L[3] = m2l_fma(D[37], m, L[3]);
      L[4] = m2l_fma(D[56], m, L[4]);
      L[5] = m2l_fma(D[57], m, L[5]);
      L[6] = m2l_fma(D[58], m, L[6]);
      L[7] = m2l_fma(D[59], m, L[7]);
      L[8] = m2l_fma(D[60], m, L[8]);
      L[9] = m2l_fma(D[61], m, L[9]);
    }
    { const T m = __ldg(Ms + 21) * rp;
      L[1] = m2l_fma(D[36], m, L[1]);
      L[2] = m2l_fma(D[38], m, L[2]);
      L[3] = m2l_fma(D[39], m, L[3]);
      L[4] = m2l_fma(D[57], m, L[4]);
      L[5] = m2l_fma(D[59], m, L[5]);
      L[6] = m2l_fma(D[60], m, L[6]);
      L[7] = m2l_fma(D[62], m, L[7]);
      L[8] = m2l_fma(D[63], m, L[8]);
      L[9] = m2l_fma(D[64], m, L[9]);
    }
    { const T m = __ldg(Ms + 22) * rp;
      L[1] = m2l_fma(D[37], m, L[1]);
      L[2] = m2l_fma(D[39], m, L[2]);
      L[3] = m2l_fma(D[40], m, L[3]);
      L[4] = m2l_fma(D[58], m, L[4]);
      L[5] = m2l_fma(D[60], m, L[5]);
      L[6] = m2l_fma(D[61], m, L[6]);
      L[7] = m2l_fma(D[63], m, L[7]);
      L[8] = m2l_fma(D[64], m, L[8]);
      L[9] = m2l_fma(D[65], m, L[9]);
    }
    { const T m = __ldg(Ms + 23) * rp;
      L[1] = m2l_fma(D[38], m, L[1]);
      L[2] = m2l_fma(D[41], m, L[2]);
      L[3] = m2l_fma(D[42], m, L[3]);
      L[4] = m2l_fma(D[59], m, L[4]);
      L[5] = m2l_fma(D[62], m, L[5]);
      L[6] = m2l_fma(D[63], m, L[6]);
      L[7] = m2l_fma(D[66], m, L[7]);
      L[8] = m2l_fma(D[67], m, L[8]);
      L[9] = m2l_fma(D[68], m, L[9]);
    }
    { const T m = __ldg(Ms + 24) * rp;
      L[1] = m2l_fma(D[39], m, L[1]);
      L[2] = m2l_fma(D[42], m, L[2]);
      L[3] = m2l_fma(D[43], m, L[3]);
      L[4] = m2l_fma(D[60], m, L[4]);
      L[5] = m2l_fma(D[63], m, L[5]);
      L[6] = m2l_fma(D[64], m, L[6]);
      L[7] = m2l_fma(D[67], m, L[7]);
      L[8] = m2l_fma(D[68], m, L[8]);
      L[9] = m2l_fma(D[69], m, L[9]);
    }
    { const T m = __ldg(Ms + 25) * rp;
      L[1] = m2l_fma(D[40], m, L[1]);
      L[2] = m2l_fma(D[43], m, L[2]);
      L[3] = m2l_fma(D[44], m, L[3]);
      L[4] = m2l_fma(D[61], m, L[4]);
      L[5] = m2l_fma(D[64], m, L[5]);
      L[6] = m2l_fma(D[65], m, L[6]);
      L[7] = m2l_fma(D[68], m, L[7]);
      L[8] = m2l_fma(D[69], m, L[8]);
      L[9] = m2l_fma(D[70], m, L[9]);
    }
    { const T m = __ldg(Ms + 26) * rp;
      L[1] = m2l_fma(D[41], m, L[1]);
      L[2] = m2l_fma(D[45], m, L[2]);
      L[3] = m2l_fma(D[46], m, L[3]);
      L[4] = m2l_fma(D[62], m, L[4]);
      L[5] = m2l_fma(D[66], m, L[5]);
      L[6] = m2l_fma(D[67], m, L[6]);
      L[7] = m2l_fma(D[71], m, L[7]);
      L[8] = m2l_fma(D[72], m, L[8]);
      L[9] = m2l_fma(D[73], m, L[9]);
    }
    { const T m = __ldg(Ms + 27) * rp;
      L[1] = m2l_fma(D[42], m, L[1]);
      L[2] = m2l_fma(D[46], m, L[2]);
      L[3] = m2l_fma(D[47], m, L[3]);
      L[4] = m2l_fma(D[63], m, L[4]);
      L[5] = m2l_fma(D[67], m, L[5]);
      L[6] = m2l_fma(D[68], m, L[6]);
      L[7] = m2l_fma(D[72], m, L[7]);
      L[8] = m2l_fma(D[73], m, L[8]);
      L[9] = m2l_fma(D[74], m, L[9]);
    }
    { const T m = __ldg(Ms + 28) * rp;
      L[1] = m2l_fma(D[43], m, L[1]);
      L[2] = m2l_fma(D[47], m, L[2]);
      L[3] = m2l_fma(D[48], m, L[3]);
      L[4] = m2l_fma(D[64], m, L[4]);
      L[5] = m2l_fma(D[68], m, L[5]);
      L[6] = m2l_fma(D[69], m, L[6]);
      L[7] = m2l_fma(D[73], m, L[7]);
      L[8] = m2l_fma(D[74], m, L[8]);
      L[9] = m2l_fma(D[75], m, L[9]);
    }
    { const T m = __ldg(Ms + 29) * rp;
      L[1] = m2l_fma(D[44], m, L[1]);
      L[2] = m2l_fma(D[48], m, L[2]);
      L[3] = m2l_fma(D[49], m, L[3]);
      L[4] = m2l_fma(D[65], m, L[4]);
      L[5] = m2l_fma(D[69], m, L[5]);
      L[6] = m2l_fma(D[70], m, L[6]);
      L[7] = m2l_fma(D[74], m, L[7]);
      L[8] = m2l_fma(D[75], m, L[8]);
      L[9] = m2l_fma(D[76], m, L[9]);
    }
    { const T m = __ldg(Ms + 30) * rp;
      L[1] = m2l_fma(D[45], m, L[1]);
      L[2] = m2l_fma(D[50], m, L[2]);
      L[3] = m2l_fma(D[51], m, L[3]);
      L[4] = m2l_fma(D[66], m, L[4]);
      L[5] = m2l_fma(D[71], m, L[5]);
      L[6] = m2l_fma(D[72], m, L[6]);
      L[7] = m2l_fma(D[77], m, L[7]);
      L[8] = m2l_fma(D[78], m, L[8]);
      L[9] = m2l_fma(D[79], m, L[9]);
    }
    { const T m = __ldg(Ms + 31) * rp;
      L[1] = m2l_fma(D[46], m, L[1]);
      L[2] = m2l_fma(D[51], m, L[2]);
      L[3] = m2l_fma(D[52], m, L[3]);
      L[4] = m2l_fma(D[67], m, L[4]);
      L[5] = m2l_fma(D[72], m, L[5]);
      L[6] = m2l_fma(D[73], m, L[6]);
      L[7] = m2l_fma(D[78], m, L[7]);
      L[8] = m2l_fma(D[79], m, L[8]);
      L[9] = m2l_fma(D[80], m, L[9]);
    }
    { const T m = __ldg(Ms + 32) * rp;
      L[1] = m2l_fma(D[47], m, L[1]);
      L[2] = m2l_fma(D[52], m, L[2]);
      L[3] = m2l_fma(D[53], m, L[3]);
      L[4] = m2l_fma(D[68], m, L[4]);
      L[5] = m2l_fma(D[73], m, L[5]);
      L[6] = m2l_fma(D[74], m, L[6]);
      L[7] = m2l_fma(D[79], m, L[7]);
      L[8] = m2l_fma(D[80], m, L[8]);
      L[9] = m2l_fma(D[81], m, L[9]);
    }
    { const T m = __ldg(Ms + 33) * rp;
      L[1] = m2l_fma(D[48], m, L[1]);
      L[2] = m2l_fma(D[53], m, L[2]);
      L[3] = m2l_fma(D[54], m, L[3]);
      L[4] = m2l_fma(D[69], m, L[4]);
      L[5] = m2l_fma(D[74], m, L[5]);
      L[6] = m2l_fma(D[75], m, L[6]);
      L[7] = m2l_fma(D[80], m, L[7]);
      L[8] = m2l_fma(D[81], m, L[8]);
      L[9] = m2l_fma(D[82], m, L[9]);
    }
    { const T m = __ldg(Ms + 34) * rp;
      L[1] = m2l_fma(D[49], m, L[1]);
      L[2] = m2l_fma(D[54], m, L[2]);
      L[3] = m2l_fma(D[55], m, L[3]);
      L[4] = m2l_fma(D[70], m, L[4]);
      L[5] = m2l_fma(D[75], m, L[5]);
      L[6] = m2l_fma(D[76], m, L[6]);
      L[7] = m2l_fma(D[81], m, L[7]);
      L[8] = m2l_fma(D[82], m, L[8]);
      L[9] = m2l_fma(D[83], m, L[9]);
    }
    rp *= rho;
    { const T m = -__ldg(Ms + 35) * rp;
      L[1] = m2l_fma(D[56], m, L[1]);
      L[2] = m2l_fma(D[57], m, L[2]);
      L[3] = m2l_fma(D[58], m, L[3]);
    }
    { const T m = -__ldg(Ms + 36) * rp;
      L[1] = m2l_fma(D[57], m, L[1]);
      L[2] = m2l_fma(D[59], m, L[2]);
      L[3] = m2l_fma(D[60], m, L[3]);
    }
    { const T m = -__ldg(Ms + 37) * rp;
      L[1] = m2l_fma(D[58], m, L[1]);
      L[2] = m2l_fma(D[60], m, L[2]);
      L[3] = m2l_fma(D[61], m, L[3]);
    }
    { const T m = -__ldg(Ms + 38) * rp;
      L[1] = m2l_fma(D[59], m, L[1]);
      L[2] = m2l_fma(D[62], m, L[2]);
      L[3] = m2l_fma(D[63], m, L[3]);
    }
    { const T m = -__ldg(Ms + 39) * rp;
      L[1] = m2l_fma(D[60], m, L[1]);
      L[2] = m2l_fma(D[63], m, L[2]);
      L[3] = m2l_fma(D[64], m, L[3]);
    }
    { const T m = -__ldg(Ms + 40) * rp;
      L[1] = m2l_fma(D[61], m, L[1]);
      L[2] = m2l_fma(D[64], m, L[2]);
      L[3] = m2l_fma(D[65], m, L[3]);
    }
    { const T m = -__ldg(Ms + 41) * rp;
      L[1] = m2l_fma(D[62], m, L[1]);
      L[2] = m2l_fma(D[66], m, L[2]);
      L[3] = m2l_fma(D[67], m, L[3]);
    }
    { const T m = -__ldg(Ms + 42) * rp;
      L[1] = m2l_fma(D[63], m, L[1]);
      L[2] = m2l_fma(D[67], m, L[2]);
      L[3] = m2l_fma(D[68], m, L[3]);
    }
    { const T m = -__ldg(Ms + 43) * rp;
      L[1] = m2l_fma(D[64], m, L[1]);
      L[2] = m2l_fma(D[68], m, L[2]);
      L[3] = m2l_fma(D[69], m, L[3]);
    }
    { const T m = -__ldg(Ms + 44) * rp;
      L[1] = m2l_fma(D[65], m, L[1]);
      L[2] = m2l_fma(D[69], m, L[2]);
      L[3] = m2l_fma(D[70], m, L[3]);
    }
    { const T m = -__ldg(Ms + 45) * rp;
      L[1] = m2l_fma(D[66], m, L[1]);
      L[2] = m2l_fma(D[71], m, L[2]);
      L[3] = m2l_fma(D[72], m, L[3]);
    }
    { const T m = -__ldg(Ms + 46) * rp;
      L[1] = m2l_fma(D[67], m, L[1]);
      L[2] = m2l_fma(D[72], m, L[2]);
      L[3] = m2l_fma(D[73], m, L[3]);
    }
    { const T m = -__ldg(Ms + 47) * rp;
      L[1] = m2l_fma(D[68], m, L[1]);
      L[2] = m2l_fma(D[73], m, L[2]);
      L[3] = m2l_fma(D[74], m, L[3]);
    }
    { const T m = -__ldg(Ms + 48) * rp;
      L[1] = m2l_fma(D[69], m, L[1]);
      L[2] = m2l_fma(D[74], m, L[2]);
      L[3] = m2l_fma(D[75], m, L[3]);
    }
    { const T m = -__ldg(Ms + 49) * rp;
      L[1] = m2l_fma(D[70], m, L[1]);
      L[2] = m2l_fma(D[75], m, L[2]);
      L[3] = m2l_fma(D[76], m, L[3]);
    }
    { const T m = -__ldg(Ms + 50) * rp;
      L[1] = m2l_fma(D[71], m, L[1]);
      L[2] = m2l_fma(D[77], m, L[2]);
      L[3] = m2l_fma(D[78], m, L[3]);
    }
    { const T m = -__ldg(Ms + 51) * rp;
      L[1] = m2l_fma(D[72], m, L[1]);
      L[2] = m2l_fma(D[78], m, L[2]);
      L[3] = m2l_fma(D[79], m, L[3]);
    }
    { const T m = -__ldg(Ms + 52) * rp;
      L[1] = m2l_fma(D[73], m, L[1]);
      L[2] = m2l_fma(D[79], m, L[2]);
      L[3] = m2l_fma(D[80], m, L[3]);
    }
    { const T m = -__ldg(Ms + 53) * rp;
      L[1] = m2l_fma(D[74], m, L[1]);
      L[2] = m2l_fma(D[80], m, L[2]);
      L[3] = m2l_fma(D[81], m, L[3]);
    }
    { const T m = -__ldg(Ms + 54) * rp;
      L[1] = m2l_fma(D[75], m, L[1]);
      L[2] = m2l_fma(D[81], m, L[2]);
      L[3] = m2l_fma(D[82], m, L[3]);
    }
    { const T m = -__ldg(Ms + 55) * rp;
      L[1] = m2l_fma(D[76], m, L[1]);
      L[2] = m2l_fma(D[82], m, L[2]);
      L[3] = m2l_fma(D[83], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_forces_6(const T (&D)[84], const T *__restrict__ Ms, T (&L)[84])
{
    L[0] = T(0);
    { const T m = __ldg(Ms + 0);
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[9] * m;
      L[10] = -D[10] * m;
      L[11] = -D[11] * m;
      L[12] = -D[12] * m;
      L[13] = -D[13] * m;
      L[14] = -D[14] * m;
      L[15] = -D[15] * m;
      L[16] = -D[16] * m;
      L[17] = -D[17] * m;
      L[18] = -D[18] * m;
      L[19] = -D[19] * m;
      L[20] = D[20] * m;
      L[21] = D[21] * m;
      L[22] = D[22] * m;
      L[23] = D[23] * m;
      L[24] = D[24] * m;
      L[25] = D[25] * m;
      L[26] = D[26] * m;
      L[27] = D[27] * m;
      L[28] = D[28] * m;
      L[29] = D[29] * m;
      L[30] = D[30] * m;
      L[31] = D[31] * m;
      L[32] = D[32] * m;
      L[33] = D[33] * m;
      L[34] = D[34] * m;
      L[35] = -D[35] * m;
      L[36] = -D[36] * m;
      L[37] = -D[37] * m;
      L[38] = -D[38] * m;
      L[39] = -D[39] * m;
      L[40] = -D[40] * m;
      L[41] = -D[41] * m;
      L[42] = -D[42] * m;
      L[43] = -D[43] * m;
      L[44] = -D[44] * m;
      L[45] = -D[45] * m;
      L[46] = -D[46] * m;
      L[47] = -D[47] * m;
      L[48] = -D[48] * m;
      L[49] = -D[49] * m;
      L[50] = -D[50] * m;
      L[51] = -D[51] * m;
      L[52] = -D[52] * m;
      L[53] = -D[53] * m;
      L[54] = -D[54] * m;
      L[55] = -D[55] * m;
      L[56] = D[56] * m;
      L[57] = D[57] * m;
      L[58] = D[58] * m;
      L[59] = D[59] * m;
      L[60] = D[60] * m;
      L[61] = D[61] * m;
      L[62] = D[62] * m;
      L[63] = D[63] * m;
      L[64] = D[64] * m;
      L[65] = D[65] * m;
      L[66] = D[66] * m;
      L[67] = D[67] * m;
      L[68] = D[68] * m;
      L[69] = D[69] * m;
      L[70] = D[70] * m;
      L[71] = D[71] * m;
      L[72] = D[72] * m;
      L[73] = D[73] * m;
      L[74] = D[74] * m;
      L[75] = D[75] * m;
      L[76] = D[76] * m;
      L[77] = D[77] * m;
      L[78] = D[78] * m;
      L[79] = D[79] * m;
      L[80] = D[80] * m;
      L[81] = D[81] * m;
      L[82] = D[82] * m;
      L[83] = D[83] * m;
    }
    { const T m = __ldg(Ms + 1);
      L[1] = m2l_fma(-D[4], m, L[1]);
      L[2] = m2l_fma(-D[5], m, L[2]);
      L[3] = m2l_fma(-D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[15], m, L[9]);
      L[10] = m2l_fma(-D[20], m, L[10]);
      L[11] = m2l_fma(-D[21], m, L[11]);
      L[12] = m2l_fma(-D[22], m, L[12]);
      L[13] = m2l_fma(-D[23], m, L[13]);
      L[14] = m2l_fma(-D[24], m, L[14]);
      L[15] = m2l_fma(-D[25], m, L[15]);
      L[16] = m2l_fma(-D[26], m, L[16]);
      L[17] = m2l_fma(-D[27], m, L[17]);
      L[18] = m2l_fma(-D[28], m, L[18]);
      L[19] = m2l_fma(-D[29], m, L[19]);
      L[20] = m2l_fma(D[35], m, L[20]);
      L[21] = m2l_fma(D[36], m, L[21]);
      L[22] = m2l_fma(D[37], m, L[22]);
      L[23] = m2l_fma(D[38], m, L[23]);
      L[24] = m2l_fma(D[39], m, L[24]);
      L[25] = m2l_fma(D[40], m, L[25]);
      L[26] = m2l_fma(D[41], m, L[26]);
      L[27] = m2l_fma(D[42], m, L[27]);
      L[28] = m2l_fma(D[43], m, L[28]);
      L[29] = m2l_fma(D[44], m, L[29]);
      L[30] = m2l_fma(D[45], m, L[30]);
      L[31] = m2l_fma(D[46], m, L[31]);
      L[32] = m2l_fma(D[47], m, L[32]);
      L[33] = m2l_fma(D[48], m, L[33]);
      L[34] = m2l_fma(D[49], m, L[34]);
      L[35] = m2l_fma(-D[56], m, L[35]);
      L[36] = m2l_fma(-D[57], m, L[36]);
      L[37] = m2l_fma(-D[58], m, L[37]);
      L[38] = m2l_fma(-D[59], m, L[38]);
      L[39] = m2l_fma(-D[60], m, L[39]);
      L[40] = m2l_fma(-D[61], m, L[40]);
      L[41] = m2l_fma(-D[62], m, L[41]);
      L[42] = m2l_fma(-D[63], m, L[42]);
      L[43] = m2l_fma(-D[64], m, L[43]);
      L[44] = m2l_fma(-D[65], m, L[44]);
      L[45] = m2l_fma(-D[66], m, L[45]);
      L[46] = m2l_fma(-D[67], m, L[46]);
      L[47] = m2l_fma(-D[68], m, L[47]);
      L[48] = m2l_fma(-D[69], m, L[48]);
      L[49] = m2l_fma(-D[70], m, L[49]);
      L[50] = m2l_fma(-D[71], m, L[50]);
      L[51] = m2l_fma(-D[72], m, L[51]);
      L[52] = m2l_fma(-D[73], m, L[52]);
      L[53] = m2l_fma(-D[74], m, L[53]);
      L[54] = m2l_fma(-D[75], m, L[54]);
      L[55] = m2l_fma(-D[76], m, L[55]);
    }
    { const T m = __ldg(Ms + 2);
      L[1] = m2l_fma(-D[5], m, L[1]);
      L[2] = m2l_fma(-D[7], m, L[2]);
      L[3] = m2l_fma(-D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[18], m, L[9]);
      L[10] = m2l_fma(-D[21], m, L[10]);
      L[11] = m2l_fma(-D[23], m, L[11]);
      L[12] = m2l_fma(-D[24], m, L[12]);
      L[13] = m2l_fma(-D[26], m, L[13]);
      L[14] = m2l_fma(-D[27], m, L[14]);
      L[15] = m2l_fma(-D[28], m, L[15]);
      L[16] = m2l_fma(-D[30], m, L[16]);
      L[17] = m2l_fma(-D[31], m, L[17]);
      L[18] = m2l_fma(-D[32], m, L[18]);
      L[19] = m2l_fma(-D[33], m, L[19]);
      L[20] = m2l_fma(D[36], m, L[20]);
      L[21] = m2l_fma(D[38], m, L[21]);
      L[22] = m2l_fma(D[39], m, L[22]);
      L[23] = m2l_fma(D[41], m, L[23]);
      L[24] = m2l_fma(D[42], m, L[24]);
      L[25] = m2l_fma(D[43], m, L[25]);
      L[26] = m2l_fma(D[45], m, L[26]);
      L[27] = m2l_fma(D[46], m, L[27]);
      L[28] = m2l_fma(D[47], m, L[28]);
      L[29] = m2l_fma(D[48], m, L[29]);
      L[30] = m2l_fma(D[50], m, L[30]);
      L[31] = m2l_fma(D[51], m, L[31]);
      L[32] = m2l_fma(D[52], m, L[32]);
      L[33] = m2l_fma(D[53], m, L[33]);
      L[34] = m2l_fma(D[54], m, L[34]);
      L[35] = m2l_fma(-D[57], m, L[35]);
      L[36] = m2l_fma(-D[59], m, L[36]);
      L[37] = m2l_fma(-D[60], m, L[37]);
      L[38] = m2l_fma(-D[62], m, L[38]);
      L[39] = m2l_fma(-D[63], m, L[39]);
      L[40] = m2l_fma(-D[64], m, L[40]);
      L[41] = m2l_fma(-D[66], m, L[41]);
      L[42] = m2l_fma(-D[67], m, L[42]);
      L[43] = m2l_fma(-D[68], m, L[43]);
      L[44] = m2l_fma(-D[69], m, L[44]);
      L[45] = m2l_fma(-D[71], m, L[45]);
      L[46] = m2l_fma(-D[72], m, L[46]);
      L[47] = m2l_fma(-D[73], m, L[47]);
      L[48] = m2l_fma(-D[74], m, L[48]);
      L[49] = m2l_fma(-D[75], m, L[49]);
      L[50] = m2l_fma(-D[77], m, L[50]);
      L[51] = m2l_fma(-D[78], m, L[51]);
      L[52] = m2l_fma(-D[79], m, L[52]);
      L[53] = m2l_fma(-D[80], m, L[53]);
      L[54] = m2l_fma(-D[81], m, L[54]);
      L[55] = m2l_fma(-D[82], m, L[55]);
    }
    { const T m = __ldg(Ms + 3);
      L[1] = m2l_fma(-D[6], m, L[1]);
      L[2] = m2l_fma(-D[8], m, L[2]);
      L[3] = m2l_fma(-D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(-D[22], m, L[10]);
      L[11] = m2l_fma(-D[24], m, L[11]);
      L[12] = m2l_fma(-D[25], m, L[12]);
      L[13] = m2l_fma(-D[27], m, L[13]);
      L[14] = m2l_fma(-D[28], m, L[14]);
      L[15] = m2l_fma(-D[29], m, L[15]);
      L[16] = m2l_fma(-D[31], m, L[16]);
      L[17] = m2l_fma(-D[32], m, L[17]);
      L[18] = m2l_fma(-D[33], m, L[18]);
      L[19] = m2l_fma(-D[34], m, L[19]);
      L[20] = m2l_fma(D[37], m, L[20]);
      L[21] = m2l_fma(D[39], m, L[21]);
      L[22] = m2l_fma(D[40], m, L[22]);
      L[23] = m2l_fma(D[42], m, L[23]);
      L[24] = m2l_fma(D[43], m, L[24]);
      L[25] = m2l_fma(D[44], m, L[25]);
      L[26] = m2l_fma(D[46], m, L[26]);
      L[27] = m2l_fma(D[47], m, L[27]);
      L[28] = m2l_fma(D[48], m, L[28]);
      L[29] = m2l_fma(D[49], m, L[29]);
      L[30] = m2l_fma(D[51], m, L[30]);
      L[31] = m2l_fma(D[52], m, L[31]);
      L[32] = m2l_fma(D[53], m, L[32]);
      L[33] = m2l_fma(D[54], m, L[33]);
      L[34] = m2l_fma(D[55], m, L[34]);
      L[35] = m2l_fma(-D[58], m, L[35]);
      L[36] = m2l_fma(-D[60], m, L[36]);
      L[37] = m2l_fma(-D[61], m, L[37]);
      L[38] = m2l_fma(-D[63], m, L[38]);
      L[39] = m2l_fma(-D[64], m, L[39]);
      L[40] = m2l_fma(-D[65], m, L[40]);
      L[41] = m2l_fma(-D[67], m, L[41]);
      L[42] = m2l_fma(-D[68], m, L[42]);
      L[43] = m2l_fma(-D[69], m, L[43]);
      L[44] = m2l_fma(-D[70], m, L[44]);
      L[45] = m2l_fma(-D[72], m, L[45]);
      L[46] = m2l_fma(-D[73], m, L[46]);
      L[47] = m2l_fma(-D[74], m, L[47]);
      L[48] = m2l_fma(-D[75], m, L[48]);
      L[49] = m2l_fma(-D[76], m, L[49]);
      L[50] = m2l_fma(-D[78], m, L[50]);
      L[51] = m2l_fma(-D[79], m, L[51]);
      L[52] = m2l_fma(-D[80], m, L[52]);
      L[53] = m2l_fma(-D[81], m, L[53]);
      L[54] = m2l_fma(-D[82], m, L[54]);
      L[55] = m2l_fma(-D[83], m, L[55]);
    }
    { const T m = __ldg(Ms + 4);
      L[1] = m2l_fma(-D[10], m, L[1]);
      L[2] = m2l_fma(-D[11], m, L[2]);
      L[3] = m2l_fma(-D[12], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[21], m, L[5]);
      L[6] = m2l_fma(D[22], m, L[6]);
      L[7] = m2l_fma(D[23], m, L[7]);
      L[8] = m2l_fma(D[24], m, L[8]);
      L[9] = m2l_fma(D[25], m, L[9]);
      L[10] = m2l_fma(-D[35], m, L[10]);
      L[11] = m2l_fma(-D[36], m, L[11]);
      L[12] = m2l_fma(-D[37], m, L[12]);
      L[13] = m2l_fma(-D[38], m, L[13]);
      L[14] = m2l_fma(-D[39], m, L[14]);
      L[15] = m2l_fma(-D[40], m, L[15]);
      L[16] = m2l_fma(-D[41], m, L[16]);
      L[17] = m2l_fma(-D[42], m, L[17]);
      L[18] = m2l_fma(-D[43], m, L[18]);
      L[19] = m2l_fma(-D[44], m, L[19]);
      L[20] = m2l_fma(D[56], m, L[20]);
      L[21] = m2l_fma(D[57], m, L[21]);
      L[22] = m2l_fma(D[58], m, L[22]);
      L[23] = m2l_fma(D[59], m, L[23]);
      L[24] = m2l_fma(D[60], m, L[24]);
      L[25] = m2l_fma(D[61], m, L[25]);
      L[26] = m2l_fma(D[62], m, L[26]);
      L[27] = m2l_fma(D[63], m, L[27]);
      L[28] = m2l_fma(D[64], m, L[28]);
      L[29] = m2l_fma(D[65], m, L[29]);
      L[30] = m2l_fma(D[66], m, L[30]);
      L[31] = m2l_fma(D[67], m, L[31]);
      L[32] = m2l_fma(D[68], m, L[32]);
      L[33] = m2l_fma(D[69], m, L[33]);
      L[34] = m2l_fma(D[70], m, L[34]);
    }
    { const T m = __ldg(Ms + 5);
      L[1] = m2l_fma(-D[11], m, L[1]);
      L[2] = m2l_fma(-D[13], m, L[2]);
      L[3] = m2l_fma(-D[14], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(D[28], m, L[9]);
      L[10] = m2l_fma(-D[36], m, L[10]);
      L[11] = m2l_fma(-D[38], m, L[11]);
      L[12] = m2l_fma(-D[39], m, L[12]);
      L[13] = m2l_fma(-D[41], m, L[13]);
      L[14] = m2l_fma(-D[42], m, L[14]);
      L[15] = m2l_fma(-D[43], m, L[15]);
      L[16] = m2l_fma(-D[45], m, L[16]);
      L[17] = m2l_fma(-D[46], m, L[17]);
      L[18] = m2l_fma(-D[47], m, L[18]);
      L[19] = m2l_fma(-D[48], m, L[19]);
      L[20] = m2l_fma(D[57], m, L[20]);
      L[21] = m2l_fma(D[59], m, L[21]);
      L[22] = m2l_fma(D[60], m, L[22]);
      L[23] = m2l_fma(D[62], m, L[23]);
      L[24] = m2l_fma(D[63], m, L[24]);
      L[25] = m2l_fma(D[64], m, L[25]);
      L[26] = m2l_fma(D[66], m, L[26]);
      L[27] = m2l_fma(D[67], m, L[27]);
      L[28] = m2l_fma(D[68], m, L[28]);
      L[29] = m2l_fma(D[69], m, L[29]);
      L[30] = m2l_fma(D[71], m, L[30]);
      L[31] = m2l_fma(D[72], m, L[31]);
      L[32] = m2l_fma(D[73], m, L[32]);
      L[33] = m2l_fma(D[74], m, L[33]);
      L[34] = m2l_fma(D[75], m, L[34]);
    }
    { const T m = __ldg(Ms + 6);
      L[1] = m2l_fma(-D[12], m, L[1]);
      L[2] = m2l_fma(-D[14], m, L[2]);
      L[3] = m2l_fma(-D[15], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[24], m, L[5]);
      L[6] = m2l_fma(D[25], m, L[6]);
      L[7] = m2l_fma(D[27], m, L[7]);
      L[8] = m2l_fma(D[28], m, L[8]);
      L[9] = m2l_fma(D[29], m, L[9]);
      L[10] = m2l_fma(-D[37], m, L[10]);
      L[11] = m2l_fma(-D[39], m, L[11]);
      L[12] = m2l_fma(-D[40], m, L[12]);
      L[13] = m2l_fma(-D[42], m, L[13]);
      L[14] = m2l_fma(-D[43], m, L[14]);
      L[15] = m2l_fma(-D[44], m, L[15]);
      L[16] = m2l_fma(-D[46], m, L[16]);
      L[17] = m2l_fma(-D[47], m, L[17]);
      L[18] = m2l_fma(-D[48], m, L[18]);
      L[19] = m2l_fma(-D[49], m, L[19]);
      L[20] = m2l_fma(D[58], m, L[20]);
      L[21] = m2l_fma(D[60], m, L[21]);
      L[22] = m2l_fma(D[61], m, L[22]);
      L[23] = m2l_fma(D[63], m, L[23]);
      L[24] = m2l_fma(D[64], m, L[24]);
      L[25] = m2l_fma(D[65], m, L[25]);
      L[26] = m2l_fma(D[67], m, L[26]);
      L[27] = m2l_fma(D[68], m, L[27]);
      L[28] = m2l_fma(D[69], m, L[28]);
      L[29] = m2l_fma(D[70], m, L[29]);
      L[30] = m2l_fma(D[72], m, L[30]);
      L[31] = m2l_fma(D[73], m, L[31]);
      L[32] = m2l_fma(D[74], m, L[32]);
      L[33] = m2l_fma(D[75], m, L[33]);
      L[34] = m2l_fma(D[76], m, L[34]);
    }
    { const T m = __ldg(Ms + 7);
      L[1] = m2l_fma(-D[13], m, L[1]);
      L[2] = m2l_fma(-D[16], m, L[2]);
      L[3] = m2l_fma(-D[17], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[30], m, L[7]);
      L[8] = m2l_fma(D[31], m, L[8]);
      L[9] = m2l_fma(D[32], m, L[9]);
      L[10] = m2l_fma(-D[38], m, L[10]);
      L[11] = m2l_fma(-D[41], m, L[11]);
      L[12] = m2l_fma(-D[42], m, L[12]);
      L[13] = m2l_fma(-D[45], m, L[13]);
      L[14] = m2l_fma(-D[46], m, L[14]);
      L[15] = m2l_fma(-D[47], m, L[15]);
      L[16] = m2l_fma(-D[50], m, L[16]);
      L[17] = m2l_fma(-D[51], m, L[17]);
      L[18] = m2l_fma(-D[52], m, L[18]);
      L[19] = m2l_fma(-D[53], m, L[19]);
      L[20] = m2l_fma(D[59], m, L[20]);
      L[21] = m2l_fma(D[62], m, L[21]);
      L[22] = m2l_fma(D[63], m, L[22]);
      L[23] = m2l_fma(D[66], m, L[23]);
      L[24] = m2l_fma(D[67], m, L[24]);
      L[25] = m2l_fma(D[68], m, L[25]);
      L[26] = m2l_fma(D[71], m, L[26]);
      L[27] = m2l_fma(D[72], m, L[27]);
      L[28] = m2l_fma(D[73], m, L[28]);
      L[29] = m2l_fma(D[74], m, L[29]);
      L[30] = m2l_fma(D[77], m, L[30]);
      L[31] = m2l_fma(D[78], m, L[31]);
      L[32] = m2l_fma(D[79], m, L[32]);
      L[33] = m2l_fma(D[80], m, L[33]);
      L[34] = m2l_fma(D[81], m, L[34]);
    }
    { const T m = __ldg(Ms + 8);
      L[1] = m2l_fma(-D[14], m, L[1]);
      L[2] = m2l_fma(-D[17], m, L[2]);
      L[3] = m2l_fma(-D[18], m, L[3]);
      L[4] = m2l_fma(D[24], m, L[4]);
      L[5] = m2l_fma(D[27], m, L[5]);
      L[6] = m2l_fma(D[28], m, L[6]);
      L[7] = m2l_fma(D[31], m, L[7]);
      L[8] = m2l_fma(D[32], m, L[8]);
      L[9] = m2l_fma(D[33], m, L[9]);
      L[10] = m2l_fma(-D[39], m, L[10]);
      L[11] = m2l_fma(-D[42], m, L[11]);
      L[12] = m2l_fma(-D[43], m, L[12]);
      L[13] = m2l_fma(-D[46], m, L[13]);
      L[14] = m2l_fma(-D[47], m, L[14]);
      L[15] = m2l_fma(-D[48], m, L[15]);
      L[16] = m2l_fma(-D[51], m, L[16]);
      L[17] = m2l_fma(-D[52], m, L[17]);
      L[18] = m2l_fma(-D[53], m, L[18]);
      L[19] = m2l_fma(-D[54], m, L[19]);
      L[20] = m2l_fma(D[60], m, L[20]);
      L[21] = m2l_fma(D[63], m, L[21]);
      L[22] = m2l_fma(D[64], m, L[22]);
      L[23] = m2l_fma(D[67], m, L[23]);
      L[24] = m2l_fma(D[68], m, L[24]);
      L[25] = m2l_fma(D[69], m, L[25]);
      L[26] = m2l_fma(D[72], m, L[26]);
      L[27] = m2l_fma(D[73], m, L[27]);
      L[28] = m2l_fma(D[74], m, L[28]);
      L[29] = m2l_fma(D[75], m, L[29]);
      L[30] = m2l_fma(D[78], m, L[30]);
      L[31] = m2l_fma(D[79], m, L[31]);
      L[32] = m2l_fma(D[80], m, L[32]);
      L[33] = m2l_fma(D[81], m, L[33]);
      L[34] = m2l_fma(D[82], m, L[34]);
    }
    { const T m = __ldg(Ms + 9);
      L[1] = m2l_fma(-D[15], m, L[1]);
      L[2] = m2l_fma(-D[18], m, L[2]);
      L[3] = m2l_fma(-D[19], m, L[3]);
      L[4] = m2l_fma(D[25], m, L[4]);
      L[5] = m2l_fma(D[28], m, L[5]);
      L[6] = m2l_fma(D[29], m, L[6]);
      L[7] = m2l_fma(D[32], m, L[7]);
      L[8] = m2l_fma(D[33], m, L[8]);
      L[9] = m2l_fma(D[34], m, L[9]);
      L[10] = m2l_fma(-D[40], m, L[10]);
      L[11] = m2l_fma(-D[43], m, L[11]);
      L[12] = m2l_fma(-D[44], m, L[12]);
      L[13] = m2l_fma(-D[47], m, L[13]);
      L[14] = m2l_fma(-D[48], m, L[14]);
      L[15] = m2l_fma(-D[49], m, L[15]);
      L[16] = m2l_fma(-D[52], m, L[16]);
      L[17] = m2l_fma(-D[53], m, L[17]);
      L[18] = m2l_fma(-D[54], m, L[18]);
      L[19] = m2l_fma(-D[55], m, L[19]);
      L[20] = m2l_fma(D[61], m, L[20]);
      L[21] = m2l_fma(D[64], m, L[21]);
      L[22] = m2l_fma(D[65], m, L[22]);
      L[23] = m2l_fma(D[68], m, L[23]);
      L[24] = m2l_fma(D[69], m, L[24]);
      L[25] = m2l_fma(D[70], m, L[25]);
      L[26] = m2l_fma(D[73], m, L[26]);
      L[27] = m2l_fma(D[74], m, L[27]);
      L[28] = m2l_fma(D[75], m, L[28]);
      L[29] = m2l_fma(D[76], m, L[29]);
      L[30] = m2l_fma(D[79], m, L[30]);
      L[31] = m2l_fma(D[80], m, L[31]);
      L[32] = m2l_fma(D[81], m, L[32]);
      L[33] = m2l_fma(D[82], m, L[33]);
      L[34] = m2l_fma(D[83], m, L[34]);
    }
    { const T m = __ldg(Ms + 10);
      L[1] = m2l_fma(-D[20], m, L[1]);
      L[2] = m2l_fma(-D[21], m, L[2]);
      L[3] = m2l_fma(-D[22], m, L[3]);
      L[4] = m2l_fma(D[35], m, L[4]);
      L[5] = m2l_fma(D[36], m, L[5]);
      L[6] = m2l_fma(D[37], m, L[6]);
      L[7] = m2l_fma(D[38], m, L[7]);
      L[8] = m2l_fma(D[39], m, L[8]);
      L[9] = m2l_fma(D[40], m, L[9]);
      L[10] = m2l_fma(-D[56], m, L[10]);
      L[11] = m2l_fma(-D[57], m, L[11]);
      L[12] = m2l_fma(-D[58], m, L[12]);
      L[13] = m2l_fma(-D[59], m, L[13]);
      L[14] = m2l_fma(-D[60], m, L[14]);
      L[15] = m2l_fma(-D[61], m, L[15]);
      L[16] = m2l_fma(-D[62], m, L[16]);
      L[17] = m2l_fma(-D[63], m, L[17]);
      L[18] = m2l_fma(-D[64], m, L[18]);
      L[19] = m2l_fma(-D[65], m, L[19]);
    }
    { const T m = __ldg(Ms + 11);
      L[1] = m2l_fma(-D[21], m, L[1]);
      L[2] = m2l_fma(-D[23], m, L[2]);
      L[3] = m2l_fma(-D[24], m, L[3]);
      L[4] = m2l_fma(D[36], m, L[4]);
      L[5] = m2l_fma(D[38], m, L[5]);
      L[6] = m2l_fma(D[39], m, L[6]);
      L[7] = m2l_fma(D[41], m, L[7]);
      L[8] = m2l_fma(D[42], m, L[8]);
      L[9] = m2l_fma(D[43], m, L[9]);
      L[10] = m2l_fma(-D[57], m, L[10]);
      L[11] = m2l_fma(-D[59], m, L[11]);
      L[12] = m2l_fma(-D[60], m, L[12]);
      L[13] = m2l_fma(-D[62], m, L[13]);
      L[14] = m2l_fma(-D[63], m, L[14]);
      L[15] = m2l_fma(-D[64], m, L[15]);
      L[16] = m2l_fma(-D[66], m, L[16]);
      L[17] = m2l_fma(-D[67], m, L[17]);
      L[18] = m2l_fma(-D[68], m, L[18]);
      L[19] = m2l_fma(-D[69], m, L[19]);
    }
    { const T m = __ldg(Ms + 12);
      L[1] = m2l_fma(-D[22], m, L[1]);
      L[2] = m2l_fma(-D[24], m, L[2]);
      L[3] = m2l_fma(-D[25], m, L[3]);
      L[4] = m2l_fma(D[37], m, L[4]);
      L[5] = m2l_fma(D[39], m, L[5]);
      L[6] = m2l_fma(D[40], m, L[6]);
      L[7] = m2l_fma(D[42], m, L[7]);
      L[8] = m2l_fma(D[43], m, L[8]);
      L[9] = m2l_fma(D[44], m, L[9]);
      L[10] = m2l_fma(-D[58], m, L[10]);
      L[11] = m2l_fma(-D[60], m, L[11]);
      L[12] = m2l_fma(-D[61], m, L[12]);
      L[13] = m2l_fma(-D[63], m, L[13]);
      L[14] = m2l_fma(-D[64], m, L[14]);
      L[15] = m2l_fma(-D[65], m, L[15]);
      L[16] = m2l_fma(-D[67], m, L[16]);
      L[17] = m2l_fma(-D[68], m, L[17]);
      L[18] = m2l_fma(-D[69], m, L[18]);
      L[19] = m2l_fma(-D[70], m, L[19]);
    }
    { const T m = __ldg(Ms + 13);
      L[1] = m2l_fma(-D[23], m, L[1]);
      L[2] = m2l_fma(-D[26], m, L[2]);
      L[3] = m2l_fma(-D[27], m, L[3]);
      L[4] = m2l_fma(D[38], m, L[4]);
      L[5] = m2l_fma(D[41], m, L[5]);
      L[6] = m2l_fma(D[42], m, L[6]);
      L[7] = m2l_fma(D[45], m, L[7]);
      L[8] = m2l_fma(D[46], m, L[8]);
      L[9] = m2l_fma(D[47], m, L[9]);
      L[10] = m2l_fma(-D[59], m, L[10]);
      L[11] = m2l_fma(-D[62], m, L[11]);
      L[12] = m2l_fma(-D[63], m, L[12]);
      L[13] = m2l_fma(-D[66], m, L[13]);
      L[14] = m2l_fma(-D[67], m, L[14]);
      L[15] = m2l_fma(-D[68], m, L[15]);
      L[16] = m2l_fma(-D[71], m, L[16]);
      L[17] = m2l_fma(-D[72], m, L[17]);
      L[18] = m2l_fma(-D[73], m, L[18]);
      L[19] = m2l_fma(-D[74], m, L[19]);
    }
    { const T m = __ldg(Ms + 14);
      L[1] = m2l_fma(-D[24], m, L[1]);
      L[2] = m2l_fma(-D[27], m, L[2]);
      L[3] = m2l_fma(-D[28], m, L[3]);
      L[4] = m2l_fma(D[39], m, L[4]);
      L[5] = m2l_fma(D[42], m, L[5]);
      L[6] = m2l_fma(D[43], m, L[6]);
      L[7] = m2l_fma(D[46], m, L[7]);
      L[8] = m2l_fma(D[47], m, L[8]);
      L[9] = m2l_fma(D[48], m, L[9]);
      L[10] = m2l_fma(-D[60], m, L[10]);
      L[11] = m2l_fma(-D[63], m, L[11]);
      L[12] = m2l_fma(-D[64], m, L[12]);
      L[13] = m2l_fma(-D[67], m, L[13]);
      L[14] = m2l_fma(-D[68], m, L[14]);
      L[15] = m2l_fma(-D[69], m, L[15]);
      L[16] = m2l_fma(-D[72], m, L[16]);
      L[17] = m2l_fma(-D[73], m, L[17]);
      L[18] = m2l_fma(-D[74], m, L[18]);
      L[19] = m2l_fma(-D[75], m, L[19]);
    }
    { const T m = __ldg(Ms + 15);
      L[1] = m2l_fma(-D[25], m, L[1]);
      L[2] = m2l_fma(-D[28], m, L[2]);
      L[3] = m2l_fma(-D[29], m, L[3]);
      L[4] = m2l_fma(D[40], m, L[4]);
      L[5] = m2l_fma(D[43], m, L[5]);
      L[6] = m2l_fma(D[44], m, L[6]);
      L[7] = m2l_fma(D[47], m, L[7]);
      L[8] = m2l_fma(D[48], m, L[8]);
      L[9] = m2l_fma(D[49], m, L[9]);
      L[10] = m2l_fma(-D[61], m, L[10]);
      L[11] = m2l_fma(-D[64], m, L[11]);
      L[12] = m2l_fma(-D[65], m, L[12]);
      L[13] = m2l_fma(-D[68], m, L[13]);
      L[14] = m2l_fma(-D[69], m, L[14]);
      L[15] = m2l_fma(-D[70], m, L[15]);
      L[16] = m2l_fma(-D[73], m, L[16]);
      L[17] = m2l_fma(-D[74], m, L[17]);
      L[18] = m2l_fma(-D[75], m, L[18]);
      L[19] = m2l_fma(-D[76], m, L[19]);
    }
    { const T m = __ldg(Ms + 16);
      L[1] = m2l_fma(-D[26], m, L[1]);
      L[2] = m2l_fma(-D[30], m, L[2]);
      L[3] = m2l_fma(-D[31], m, L[3]);
      L[4] = m2l_fma(D[41], m, L[4]);
      L[5] = m2l_fma(D[45], m, L[5]);
      L[6] = m2l_fma(D[46], m, L[6]);
      L[7] = m2l_fma(D[50], m, L[7]);
      L[8] = m2l_fma(D[51], m, L[8]);
      L[9] = m2l_fma(D[52], m, L[9]);
      L[10] = m2l_fma(-D[62], m, L[10]);
      L[11] = m2l_fma(-D[66], m, L[11]);
      L[12] = m2l_fma(-D[67], m, L[12]);
      L[13] = m2l_fma(-D[71], m, L[13]);
      L[14] = m2l_fma(-D[72], m, L[14]);
      L[15] = m2l_fma(-D[73], m, L[15]);
      L[16] = m2l_fma(-D[77], m, L[16]);
      L[17] = m2l_fma(-D[78], m, L[17]);
      L[18] = m2l_fma(-D[79], m, L[18]);
      L[19] = m2l_fma(-D[80], m, L[19]);
    }
    { const T m = __ldg(Ms + 17);
      L[1] = m2l_fma(-D[27], m, L[1]);
      L[2] = m2l_fma(-D[31], m, L[2]);
      L[3] = m2l_fma(-D[32], m, L[3]);
      L[4] = m2l_fma(D[42], m, L[4]);
      L[5] = m2l_fma(D[46], m, L[5]);
      L[6] = m2l_fma(D[47], m, L[6]);
      L[7] = m2l_fma(D[51], m, L[7]);
      L[8] = m2l_fma(D[52], m, L[8]);
      L[9] = m2l_fma(D[53], m, L[9]);
      L[10] = m2l_fma(-D[63], m, L[10]);
      L[11] = m2l_fma(-D[67], m, L[11]);
      L[12] = m2l_fma(-D[68], m, L[12]);
      L[13] = m2l_fma(-D[72], m, L[13]);
      L[14] = m2l_fma(-D[73], m, L[14]);
      L[15] = m2l_fma(-D[74], m, L[15]);
      L[16] = m2l_fma(-D[78], m, L[16]);
      L[17] = m2l_fma(-D[79], m, L[17]);
      L[18] = m2l_fma(-D[80], m, L[18]);
      L[19] = m2l_fma(-D[81], m, L[19]);
    }
    { const T m = __ldg(Ms + 18);
      L[1] = m2l_fma(-D[28], m, L[1]);
      L[2] = m2l_fma(-D[32], m, L[2]);
      L[3] = m2l_fma(-D[33], m, L[3]);
      L[4] = m2l_fma(D[43], m, L[4]);
      L[5] = m2l_fma(D[47], m, L[5]);
      L[6] = m2l_fma(D[48], m, L[6]);
      L[7] = m2l_fma(D[52], m, L[7]);
      L[8] = m2l_fma(D[53], m, L[8]);
      L[9] = m2l_fma(D[54], m, L[9]);
      L[10] = m2l_fma(-D[64], m, L[10]);
      L[11] = m2l_fma(-D[68], m, L[11]);
      L[12] = m2l_fma(-D[69], m, L[12]);
      L[13] = m2l_fma(-D[73], m, L[13]);
      L[14] = m2l_fma(-D[74], m, L[14]);
      L[15] = m2l_fma(-D[75], m, L[15]);
      L[16] = m2l_fma(-D[79], m, L[16]);
      L[17] = m2l_fma(-D[80], m, L[17]);
      L[18] = m2l_fma(-D[81], m, L[18]);
      L[19] = m2l_fma(-D[82], m, L[19]);
    }
    { const T m = __ldg(Ms + 19);
      L[1] = m2l_fma(-D[29], m, L[1]);
      L[2] = m2l_fma(-D[33], m, L[2]);
      L[3] = m2l_fma(-D[34], m, L[3]);
      L[4] = m2l_fma(D[44], m, L[4]);
      L[5] = m2l_fma(D[48], m, L[5]);
      L[6] = m2l_fma(D[49], m, L[6]);
      L[7] = m2l_fma(D[53], m, L[7]);
      L[8] = m2l_fma(D[54], m, L[8]);
      L[9] = m2l_fma(D[55], m, L[9]);
      L[10] = m2l_fma(-D[65], m, L[10]);
      L[11] = m2l_fma(-D[69], m, L[11]);
      L[12] = m2l_fma(-D[70], m, L[12]);
      L[13] = m2l_fma(-D[74], m, L[13]);
      L[14] = m2l_fma(-D[75], m, L[14]);
      L[15] = m2l_fma(-D[76], m, L[15]);
      L[16] = m2l_fma(-D[80], m, L[16]);
      L[17] = m2l_fma(-D[81], m, L[17]);
      L[18] = m2l_fma(-D[82], m, L[18]);
      L[19] = m2l_fma(-D[83], m, L[19]);
    }
    { const T m = __ldg(Ms + 20);
      L[1] = m2l_fma(-D[35], m, L[1]);
      L[2] = m2l_fma(-D[36], m, L[2]);
      L[3] = m2l_fma(-D[37], m, L[3]);
      L[4] = m2l_fma(D[56], m, L[4]);
      L[5] = m2l_fma(D[57], m, L[5]);
      L[6] = m2l_fma(D[58], m, L[6]);
      L[7] = m2l_fma(D[59], m, L[7]);
      L[8] = m2l_fma(D[60], m, L[8]);
      L[9] = m2l_fma(D[61], m, L[9]);
    }
    { const T m = __ldg(Ms + 21);
      L[1] = m2l_fma(-D[36], m, L[1]);
      L[2] = m2l_fma(-D[38], m, L[2]);
      L[3] = m2l_fma(-D[39], m, L[3]);
      L[4] = m2l_fma(D[57], m, L[4]);
      L[5] = m2l_fma(D[59], m, L[5]);
      L[6] = m2l_fma(D[60], m, L[6]);
      L[7] = m2l_fma(D[62], m, L[7]);
      L[8] = m2l_fma(D[63], m, L[8]);
      L[9] = m2l_fma(D[64], m, L[9]);
    }
    { const T m = __ldg(Ms + 22);
      L[1] = m2l_fma(-D[37], m, L[1]);
      L[2] = m2l_fma(-D[39], m, L[2]);
      L[3] = m2l_fma(-D[40], m, L[3]);
      L[4] = m2l_fma(D[58], m, L[4]);
      L[5] = m2l_fma(D[60], m, L[5]);
      L[6] = m2l_fma(D[61], m, L[6]);
      L[7] = m2l_fma(D[63], m, L[7]);
      L[8] = m2l_fma(D[64], m, L[8]);
      L[9] = m2l_fma(D[65], m, L[9]);
    }
    { const T m = __ldg(Ms + 23);
      L[1] = m2l_fma(-D[38], m, L[1]);
      L[2] = m2l_fma(-D[41], m, L[2]);
      L[3] = m2l_fma(-D[42], m, L[3]);
      L[4] = m2l_fma(D[59], m, L[4]);
      L[5] = m2l_fma(D[62], m, L[5]);
      L[6] = m2l_fma(D[63], m, L[6]);
      L[7] = m2l_fma(D[66], m, L[7]);
      L[8] = m2l_fma(D[67], m, L[8]);
      L[9] = m2l_fma(D[68], m, L[9]);
    }
    { const T m = __ldg(Ms + 24);
      L[1] = m2l_fma(-D[39], m, L[1]);
      L[2] = m2l_fma(-D[42], m, L[2]);
      L[3] = m2l_fma(-D[43], m, L[3]);
      L[4] = m2l_fma(D[60], m, L[4]);
      L[5] = m2l_fma(D[63], m, L[5]);
      L[6] = m2l_fma(D[64], m, L[6]);
      L[7] = m2l_fma(D[67], m, L[7]);
      L[8] = m2l_fma(D[68], m, L[8]);
      L[9] = m2l_fma(D[69], m, L[9]);
    }
    { const T m = __ldg(Ms + 25);
      L[1] = m2l_fma(-D[40], m, L[1]);
      L[2] = m2l_fma(-D[43], m, L[2]);
      L[3] = m2l_fma(-D[44], m, L[3]);
      L[4] = m2l_fma(D[61], m, L[4]);
      L[5] = m2l_fma(D[64], m, L[5]);
      L[6] = m2l_fma(D[65], m, L[6]);
      L[7] = m2l_fma(D[68], m, L[7]);
      L[8] = m2l_fma(D[69], m, L[8]);
      L[9] = m2l_fma(D[70], m, L[9]);
    }
    { const T m = __ldg(Ms + 26);
      L[1] = m2l_fma(-D[41], m, L[1]);
      L[2] = m2l_fma(-D[45], m, L[2]);
      L[3] = m2l_fma(-D[46], m, L[3]);
      L[4] = m2l_fma(D[62], m, L[4]);
      L[5] = m2l_fma(D[66], m, L[5]);
      L[6] = m2l_fma(D[67], m, L[6]);
      L[7] = m2l_fma(D[71], m, L[7]);
      L[8] = m2l_fma(D[72], m, L[8]);
      L[9] = m2l_fma(D[73], m, L[9]);
    }
    { const T m = __ldg(Ms + 27);
      L[1] = m2l_fma(-D[42], m, L[1]);
      L[2] = m2l_fma(-D[46], m, L[2]);
      L[3] = m2l_fma(-D[47], m, L[3]);
      L[4] = m2l_fma(D[63], m, L[4]);
      L[5] = m2l_fma(D[67], m, L[5]);
      L[6] = m2l_fma(D[68], m, L[6]);
      L[7] = m2l_fma(D[72], m, L[7]);
      L[8] = m2l_fma(D[73], m, L[8]);
      L[9] = m2l_fma(D[74], m, L[9]);
    }
    { const T m = __ldg(Ms + 28);
      L[1] = m2l_fma(-D[43], m, L[1]);
      L[2] = m2l_fma(-D[47], m, L[2]);
      L[3] = m2l_fma(-D[48], m, L[3]);
      L[4] = m2l_fma(D[64], m, L[4]);
      L[5] = m2l_fma(D[68], m, L[5]);
      L[6] = m2l_fma(D[69], m, L[6]);
      L[7] = m2l_fma(D[73], m, L[7]);
      L[8] = m2l_fma(D[74], m, L[8]);
      L[9] = m2l_fma(D[75], m, L[9]);
    }
    { const T m = __ldg(Ms + 29);
      L[1] = m2l_fma(-D[44], m, L[1]);
      L[2] = m2l_fma(-D[48], m, L[2]);
      L[3] = m2l_fma(-D[49], m, L[3]);
      L[4] = m2l_fma(D[65], m, L[4]);
      L[5] = m2l_fma(D[69], m, L[5]);
      L[6] = m2l_fma(D[70], m, L[6]);
      L[7] = m2l_fma(D[74], m, L[7]);
      L[8] = m2l_fma(D[75], m, L[8]);
      L[9] = m2l_fma(D[76], m, L[9]);
    }
    { const T m = __ldg(Ms + 30);
      L[1] = m2l_fma(-D[45], m, L[1]);
      L[2] = m2l_fma(-D[50], m, L[2]);
      L[3] = m2l_fma(-D[51], m, L[3]);
      L[4] = m2l_fma(D[66], m, L[4]);
      L[5] = m2l_fma(D[71], m, L[5]);
      L[6] = m2l_fma(D[72], m, L[6]);
      L[7] = m2l_fma(D[77], m, L[7]);
      L[8] = m2l_fma(D[78], m, L[8]);
      L[9] = m2l_fma(D[79], m, L[9]);
    }
    { const T m = __ldg(Ms + 31);
      L[1] = m2l_fma(-D[46], m, L[1]);
      L[2] = m2l_fma(-D[51], m, L[2]);
      L[3] = m2l_fma(-D[52], m, L[3]);
      L[4] = m2l_fma(D[67], m, L[4]);
      L[5] = m2l_fma(D[72], m, L[5]);
      L[6] = m2l_fma(D[73], m, L[6]);
      L[7] = m2l_fma(D[78], m, L[7]);
      L[8] = m2l_fma(D[79], m, L[8]);
      L[9] = m2l_fma(D[80], m, L[9]);
    }
    { const T m = __ldg(Ms + 32);
      L[1] = m2l_fma(-D[47], m, L[1]);
      L[2] = m2l_fma(-D[52], m, L[2]);
      L[3] = m2l_fma(-D[53], m, L[3]);
      L[4] = m2l_fma(D[68], m, L[4]);
      L[5] = m2l_fma(D[73], m, L[5]);
      L[6] = m2l_fma(D[74], m, L[6]);
      L[7] = m2l_fma(D[79], m, L[7]);
      L[8] = m2l_fma(D[80], m, L[8]);
      L[9] = m2l_fma(D[81], m, L[9]);
    }
    { const T m = __ldg(Ms + 33);
      L[1] = m2l_fma(-D[48], m, L[1]);
      L[2] = m2l_fma(-D[53], m, L[2]);
      L[3] = m2l_fma(-D[54], m, L[3]);
      L[4] = m2l_fma(D[69], m, L[4]);
      L[5] = m2l_fma(D[74], m, L[5]);
      L[6] = m2l_fma(D[75], m, L[6]);
      L[7] = m2l_fma(D[80], m, L[7]);
      L[8] = m2l_fma(D[81], m, L[8]);
      L[9] = m2l_fma(D[82], m, L[9]);
    }
    { const T m = __ldg(Ms + 34);
      L[1] = m2l_fma(-D[49], m, L[1]);
      L[2] = m2l_fma(-D[54], m, L[2]);
      L[3] = m2l_fma(-D[55], m, L[3]);
      L[4] = m2l_fma(D[70], m, L[4]);
      L[5] = m2l_fma(D[75], m, L[5]);
      L[6] = m2l_fma(D[76], m, L[6]);
      L[7] = m2l_fma(D[81], m, L[7]);
      L[8] = m2l_fma(D[82], m, L[8]);
      L[9] = m2l_fma(D[83], m, L[9]);
    }
    { const T m = __ldg(Ms + 35);
      L[1] = m2l_fma(-D[56], m, L[1]);
      L[2] = m2l_fma(-D[57], m, L[2]);
      L[3] = m2l_fma(-D[58], m, L[3]);
    }
    { const T m = __ldg(Ms + 36);
      L[1] = m2l_fma(-D[57], m, L[1]);
      L[2] = m2l_fma(-D[59], m, L[2]);
      L[3] = m2l_fma(-D[60], m, L[3]);
    }
    { const T m = __ldg(Ms + 37);
      L[1] = m2l_fma(-D[58], m, L[1]);
      L[2] = m2l_fma(-D[60], m, L[2]);
      L[3] = m2l_fma(-D[61], m, L[3]);
    }
    { const T m = __ldg(Ms + 38);
      L[1] = m2l_fma(-D[59], m, L[1]);
      L[2] = m2l_fma(-D[62], m, L[2]);
      L[3] = m2l_fma(-D[63], m, L[3]);
    }
    { const T m = __ldg(Ms + 39);
      L[1] = m2l_fma(-D[60], m, L[1]);
      L[2] = m2l_fma(-D[63], m, L[2]);
      L[3] = m2l_fma(-D[64], m, L[3]);
    }
    { const T m = __ldg(Ms + 40);
      L[1] = m2l_fma(-D[61], m, L[1]);
      L[2] = m2l_fma(-D[64], m, L[2]);
      L[3] = m2l_fma(-D[65], m, L[3]);
    }
    { const T m = __ldg(Ms + 41);
      L[1] = m2l_fma(-D[62], m, L[1]);
      L[2] = m2l_fma(-D[66], m, L[2]);
      L[3] = m2l_fma(-D[67], m, L[3]);
    }
    { const T m = __ldg(Ms + 42);
      L[1] = m2l_fma(-D[63], m, L[1]);
      L[2] = m2l_fma(-D[67], m, L[2]);
      L[3] = m2l_fma(-D[68], m, L[3]);
    }
    { const T m = __ldg(Ms + 43);
      L[1] = m2l_fma(-D[64], m, L[1]);
      L[2] = m2l_fma(-D[68], m, L[2]);
      L[3] = m2l_fma(-D[69], m, L[3]);
    }
    { const T m = __ldg(Ms + 44);
      L[1] = m2l_fma(-D[65], m, L[1]);
      L[2] = m2l_fma(-D[69], m, L[2]);
      L[3] = m2l_fma(-D[70], m, L[3]);
    }
    { const T m = __ldg(Ms + 45);
      L[1] = m2l_fma(-D[66], m, L[1]);
      L[2] = m2l_fma(-D[71], m, L[2]);
      L[3] = m2l_fma(-D[72], m, L[3]);
    }
    { const T m = __ldg(Ms + 46);
      L[1] = m2l_fma(-D[67], m, L[1]);
      L[2] = m2l_fma(-D[72], m, L[2]);
      L[3] = m2l_fma(-D[73], m, L[3]);
    }
    { const T m = __ldg(Ms + 47);
      L[1] = m2l_fma(-D[68], m, L[1]);
      L[2] = m2l_fma(-D[73], m, L[2]);
      L[3] = m2l_fma(-D[74], m, L[3]);
    }
    { const T m = __ldg(Ms + 48);
      L[1] = m2l_fma(-D[69], m, L[1]);
      L[2] = m2l_fma(-D[74], m, L[2]);
      L[3] = m2l_fma(-D[75], m, L[3]);
    }
    { const T m = __ldg(Ms + 49);
      L[1] = m2l_fma(-D[70], m, L[1]);
      L[2] = m2l_fma(-D[75], m, L[2]);
      L[3] = m2l_fma(-D[76], m, L[3]);
    }
    { const T m = __ldg(Ms + 50);
      L[1] = m2l_fma(-D[71], m, L[1]);
      L[2] = m2l_fma(-D[77], m, L[2]);
      L[3] = m2l_fma(-D[78], m, L[3]);
    }
    { const T m = __ldg(Ms + 51);
      L[1] = m2l_fma(-D[72], m, L[1]);
      L[2] = m2l_fma(-D[78], m, L[2]);
      L[3] = m2l_fma(-D[79], m, L[3]);
    }
    { const T m = __ldg(Ms + 52);
      L[1] = m2l_fma(-D[73], m, L[1]);
      L[2] = m2l_fma(-D[79], m, L[2]);
      L[3] = m2l_fma(-D[80], m, L[3]);
    }
    { const T m = __ldg(Ms + 53);
      L[1] = m2l_fma(-D[74], m, L[1]);
      L[2] = m2l_fma(-D[80], m, L[2]);
      L[3] = m2l_fma(-D[81], m, L[3]);
    }
    { const T m = __ldg(Ms + 54);
      L[1] = m2l_fma(-D[75], m, L[1]);
      L[2] = m2l_fma(-D[81], m, L[2]);
      L[3] = m2l_fma(-D[82], m, L[3]);
    }
    { const T m = __ldg(Ms + 55);
      L[1] = m2l_fma(-D[76], m, L[1]);
      L[2] = m2l_fma(-D[82], m, L[2]);
      L[3] = m2l_fma(-D[83], m, L[3]);
    }
}

template <int P> struct M2LGen;
template <> struct M2LGen<1> {
    static constexpr int NC = 4;
    template <class T> static __device__ __forceinline__ void dtensor(T dx, T dy, T dz, T s, T (&D)[4]) { m2l_dtensor_1(dx, dy, dz, s, D); }
    template <class T> static __device__ __forceinline__ void side_a(const T (&D)[4], const T *Ms, T rho, T (&L)[4]) { m2l_side_a_1(D, Ms, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b(const T (&D)[4], const T *Ms, T (&L)[4]) { m2l_side_b_1(D, Ms, L); }
    template <class T> static __device__ __forceinline__ void side_a_forces(const T (&D)[4], const T *Ms, T rho, T (&L)[4]) { m2l_side_a_forces_1(D, Ms, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b_forces(const T (&D)[4], const T *Ms, T (&L)[4]) { m2l_side_b_forces_1(D, Ms, L); }
};
template <> struct M2LGen<2> {
    static constexpr int NC = 10;
    template <class T> static __device__ __forceinline__ void dtensor(T dx, T dy, T dz, T s, T (&D)[10]) { m2l_dtensor_2(dx, dy, dz, s, D); }
    template <class T> static __device__ __forceinline__ void side_a(const T (&D)[10], const T *Ms, T rho, T (&L)[10]) { m2l_side_a_2(D, Ms, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b(const T (&D)[10], const T *Ms, T (&L)[10]) { m2l_side_b_2(D, Ms, L); }
    template <class T> static __device__ __forceinline__ void side_a_forces(const T (&D)[10], const T *Ms, T rho, T (&L)[10]) { m2l_side_a_forces_2(D, Ms, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b_forces(const T (&D)[10], const T *Ms, T (&L)[10]) { m2l_side_b_forces_2(D, Ms, L); }
};
template <> struct M2LGen<3> {
    static constexpr int NC = 20;
    template <class T> static __device__ __forceinline__ void dtensor(T dx, T dy, T dz, T s, T (&D)[20]) { m2l_dtensor_3(dx, dy, dz, s, D); }
    template <class T> static __device__ __forceinline__ void side_a(const T (&D)[20], const T *Ms, T rho, T (&L)[20]) { m2l_side_a_3(D, Ms, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b(const T (&D)[20], const T *Ms, T (&L)[20]) { m2l_side_b_3(D, Ms, L); }
    template <class T> static __device__ __forceinline__ void side_a_forces(const T (&D)[20], const T *Ms, T rho, T (&L)[20]) { m2l_side_a_forces_3(D, Ms, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b_forces(const T (&D)[20], const T *Ms, T (&L)[20]) { m2l_side_b_forces_3(D, Ms, L); }
};
template <> struct M2LGen<4> {
    static constexpr int NC = 35;
    template <class T> static __device__ __forceinline__ void dtensor(T dx, T dy, T dz, T s, T (&D)[35]) { m2l_dtensor_4(dx, dy, dz, s, D); }
    template <class T> static __device__ __forceinline__ void side_a(const T (&D)[35], const T *Ms, T rho, T (&L)[35]) { m2l_side_a_4(D, Ms, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b(const T (&D)[35], const T *Ms, T (&L)[35]) { m2l_side_b_4(D, Ms, L); }
    template <class T> static __device__ __forceinline__ void side_a_forces(const T (&D)[35], const T *Ms, T rho, T (&L)[35]) { m2l_side_a_forces_4(D, Ms, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b_forces(const T (&D)[35], const T *Ms, T (&L)[35]) { m2l_side_b_forces_4(D, Ms, L); }
};
template <> struct M2LGen<5> {
    static constexpr int NC = 56;
    template <class T> static __device__ __forceinline__ void dtensor(T dx, T dy, T dz, T s, T (&D)[56]) { m2l_dtensor_5(dx, dy, dz, s, D); }
    template <class T> static __device__ __forceinline__ void side_a(const T (&D)[56], const T *Ms, T rho, T (&L)[56]) { m2l_side_a_5(D, Ms, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b(const T (&D)[56], const T *Ms, T (&L)[56]) { m2l_side_b_5(D, Ms, L); }
    template <class T> static __device__ __forceinline__ void side_a_forces(const T (&D)[56], const T *Ms, T rho, T (&L)[56]) { m2l_side_a_forces_5(D, Ms, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b_forces(const T (&D)[56], const T *Ms, T (&L)[56]) { m2l_side_b_forces_5(D, Ms, L); }
};
template <> struct M2LGen<6> {
    static constexpr int NC = 84;
    template <class T> static __device__ __forceinline__ void dtensor(T dx, T dy, T dz, T s, T (&D)[84]) { m2l_dtensor_6(dx, dy, dz, s, D); }
    template <class T> static __device__ __forceinline__ void side_a(const T (&D)[84], const T *Ms, T rho, T (&L)[84]) { m2l_side_a_6(D, Ms, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b(const T (&D)[84], const T *Ms, T (&L)[84]) { m2l_side_b_6(D, Ms, L); }
    template <class T> static __device__ __forceinline__ void side_a_forces(const T (&D)[84], const T *Ms, T rho, T (&L)[84]) { m2l_side_a_forces_6(D, Ms, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b_forces(const T (&D)[84], const T *Ms, T (&L)[84]) { m2l_side_b_forces_6(D, Ms, L); }
};
template <class T> __device__ __forceinline__ void m2l_dtensor_h_1(T dx, T dy, T dz, T (&D)[4])
{
    const T s2 = m2l_fma(dx, dx, m2l_fma(dy, dy, dz * dz));
    const T si = m2l_rsqrt(s2);
    const T si2 = si * si;
    const T f0 = -si;
    const T f1 = T(-1) * f0 * si2;
    const T r_0_0 = f0;
    const T r_1_0 = f1;
    const T r_0_1 = dx * r_1_0;
    const T r_0_2 = dy * r_1_0;
    D[0] = r_0_0;
    D[1] = r_0_1;
    D[2] = r_0_2;
    D[3] = dz * r_1_0;
}

template <class T> __device__ __forceinline__ void m2l_side_a_h_1(const T (&D)[4], const T *__restrict__ Mr, T rho, T (&L)[4])
{
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[0] = D[0] * m;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 1) * rp;
      L[0] = m2l_fma(D[1], m, L[0]);
    }
    { const T m = -__ldg(Mr + 2) * rp;
      L[0] = m2l_fma(D[2], m, L[0]);
    }
    { const T m = -__ldg(Mr + 3) * rp;
      L[0] = m2l_fma(D[3], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_acc_h_1(const T (&D)[4], const T *__restrict__ Mr, T rho, T (&L)[4])
{
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[0] = m2l_fma(D[0], m, L[0]);
      L[1] = m2l_fma(D[1], m, L[1]);
      L[2] = m2l_fma(D[2], m, L[2]);
      L[3] = m2l_fma(D[3], m, L[3]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 1) * rp;
      L[0] = m2l_fma(D[1], m, L[0]);
    }
    { const T m = -__ldg(Mr + 2) * rp;
      L[0] = m2l_fma(D[2], m, L[0]);
    }
    { const T m = -__ldg(Mr + 3) * rp;
      L[0] = m2l_fma(D[3], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_h_1(const T (&D)[4], const T *__restrict__ Mr, T (&L)[4])
{
    { const T m = __ldg(Mr + 0);
      L[0] = D[0] * m;
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
    }
    { const T m = __ldg(Mr + 1);
      L[0] = m2l_fma(D[1], m, L[0]);
    }
    { const T m = __ldg(Mr + 2);
      L[0] = m2l_fma(D[2], m, L[0]);
    }
    { const T m = __ldg(Mr + 3);
      L[0] = m2l_fma(D[3], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_a_h_forces_1(const T (&D)[4], const T *__restrict__ Mr, T rho, T (&L)[4])
{
    L[0] = T(0);
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
    }
}

template <class T> __device__ __forceinline__ void m2l_acc_h_forces_1(const T (&D)[4], const T *__restrict__ Mr, T rho, T (&L)[4])
{
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[1] = m2l_fma(D[1], m, L[1]);
      L[2] = m2l_fma(D[2], m, L[2]);
      L[3] = m2l_fma(D[3], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_h_forces_1(const T (&D)[4], const T *__restrict__ Mr, T (&L)[4])
{
    L[0] = T(0);
    { const T m = __ldg(Mr + 0);
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
    }
}

template <class T> __device__ __forceinline__ void m2l_reduce_moments_h_1(const T *__restrict__ Ms, T *__restrict__ Mr)
{
    T v0 = Ms[0];
    T v1 = Ms[1];
    T v2 = Ms[2];
    T v3 = Ms[3];
    Mr[0] = v0;
    Mr[1] = v1;
    Mr[2] = v2;
    Mr[3] = v3;
}

template <class T> __device__ __forceinline__ void m2l_complete_locals_h_1(const T *__restrict__ Lr, T *__restrict__ L)
{
    const T v0 = Lr[0];
    L[0] = v0;
    const T v1 = Lr[1];
    L[1] = v1;
    const T v2 = Lr[2];
    L[2] = v2;
    const T v3 = Lr[3];
    L[3] = v3;
}

template <class T> __device__ __forceinline__ void m2l_dtensor_h_2(T dx, T dy, T dz, T (&D)[10])
{
    const T s2 = m2l_fma(dx, dx, m2l_fma(dy, dy, dz * dz));
    const T si = m2l_rsqrt(s2);
    const T si2 = si * si;
    const T f0 = -si;
    const T f1 = T(-1) * f0 * si2;
    const T f2 = T(-3) * f1 * si2;
    const T r_0_0 = f0;
    const T r_1_0 = f1;
    const T r_2_0 = f2;
    const T r_0_1 = dx * r_1_0;
    const T r_1_1 = dx * r_2_0;
    const T r_0_2 = dy * r_1_0;
    const T r_1_2 = dy * r_2_0;
    const T r_0_4 = m2l_fma(T(1), r_1_0, dx * r_1_1);
    const T r_0_5 = dx * r_1_2;
    const T r_0_7 = m2l_fma(T(1), r_1_0, dy * r_1_2);
    D[0] = r_0_0;
    D[1] = r_0_1;
    D[2] = r_0_2;
    D[3] = dz * r_1_0;
    D[4] = r_0_4;
    D[5] = r_0_5;
    D[6] = dz * r_1_1;
    D[7] = r_0_7;
    D[8] = dz * r_1_2;
    D[9] = -D[4] - D[7];
}

template <class T> __device__ __forceinline__ void m2l_side_a_h_2(const T (&D)[10], const T *__restrict__ Mr, T rho, T (&L)[9])
{
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[0] = D[0] * m;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 1) * rp;
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
    }
    { const T m = -__ldg(Mr + 2) * rp;
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
    }
    { const T m = -__ldg(Mr + 3) * rp;
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 4) * rp;
      L[0] = m2l_fma(D[4], m, L[0]);
    }
    { const T m = __ldg(Mr + 5) * rp;
      L[0] = m2l_fma(D[5], m, L[0]);
    }
    { const T m = __ldg(Mr + 6) * rp;
      L[0] = m2l_fma(D[6], m, L[0]);
    }
    { const T m = __ldg(Mr + 7) * rp;
      L[0] = m2l_fma(D[7], m, L[0]);
    }
    { const T m = __ldg(Mr + 8) * rp;
      L[0] = m2l_fma(D[8], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_acc_h_2(const T (&D)[10], const T *__restrict__ Mr, T rho, T (&L)[9])
{
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[0] = m2l_fma(D[0], m, L[0]);
      L[1] = m2l_fma(D[1], m, L[1]);
      L[2] = m2l_fma(D[2], m, L[2]);
      L[3] = m2l_fma(D[3], m, L[3]);
      L[4] = m2l_fma(D[4], m, L[4]);
      L[5] = m2l_fma(D[5], m, L[5]);
      L[6] = m2l_fma(D[6], m, L[6]);
      L[7] = m2l_fma(D[7], m, L[7]);
      L[8] = m2l_fma(D[8], m, L[8]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 1) * rp;
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
    }
    { const T m = -__ldg(Mr + 2) * rp;
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
    }
    { const T m = -__ldg(Mr + 3) * rp;
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 4) * rp;
      L[0] = m2l_fma(D[4], m, L[0]);
    }
    { const T m = __ldg(Mr + 5) * rp;
      L[0] = m2l_fma(D[5], m, L[0]);
    }
    { const T m = __ldg(Mr + 6) * rp;
      L[0] = m2l_fma(D[6], m, L[0]);
    }
    { const T m = __ldg(Mr + 7) * rp;
      L[0] = m2l_fma(D[7], m, L[0]);
    }
    { const T m = __ldg(Mr + 8) * rp;
      L[0] = m2l_fma(D[8], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_h_2(const T (&D)[10], const T *__restrict__ Mr, T (&L)[9])
{
    { const T m = __ldg(Mr + 0);
      L[0] = D[0] * m;
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
    }
    { const T m = __ldg(Mr + 1);
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(-D[4], m, L[1]);
      L[2] = m2l_fma(-D[5], m, L[2]);
      L[3] = m2l_fma(-D[6], m, L[3]);
    }
    { const T m = __ldg(Mr + 2);
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(-D[5], m, L[1]);
      L[2] = m2l_fma(-D[7], m, L[2]);
      L[3] = m2l_fma(-D[8], m, L[3]);
    }
    { const T m = __ldg(Mr + 3);
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(-D[6], m, L[1]);
      L[2] = m2l_fma(-D[8], m, L[2]);
      L[3] = m2l_fma(-D[9], m, L[3]);
    }
    { const T m = __ldg(Mr + 4);
      L[0] = m2l_fma(D[4], m, L[0]);
    }
    { const T m = __ldg(Mr + 5);
      L[0] = m2l_fma(D[5], m, L[0]);
    }
    { const T m = __ldg(Mr + 6);
      L[0] = m2l_fma(D[6], m, L[0]);
    }
    { const T m = __ldg(Mr + 7);
      L[0] = m2l_fma(D[7], m, L[0]);
    }
    { const T m = __ldg(Mr + 8);
      L[0] = m2l_fma(D[8], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_a_h_forces_2(const T (&D)[10], const T *__restrict__ Mr, T rho, T (&L)[9])
{
    L[0] = T(0);
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 1) * rp;
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
    }
    { const T m = -__ldg(Mr + 2) * rp;
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
    }
    { const T m = -__ldg(Mr + 3) * rp;
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_acc_h_forces_2(const T (&D)[10], const T *__restrict__ Mr, T rho, T (&L)[9])
{
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[1] = m2l_fma(D[1], m, L[1]);
      L[2] = m2l_fma(D[2], m, L[2]);
      L[3] = m2l_fma(D[3], m, L[3]);
      L[4] = m2l_fma(D[4], m, L[4]);
      L[5] = m2l_fma(D[5], m, L[5]);
      L[6] = m2l_fma(D[6], m, L[6]);
      L[7] = m2l_fma(D[7], m, L[7]);
      L[8] = m2l_fma(D[8], m, L[8]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 1) * rp;
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
    }
    { const T m = -__ldg(Mr + 2) * rp;
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
    }
    { const T m = -__ldg(Mr + 3) * rp;
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_h_forces_2(const T (&D)[10], const T *__restrict__ Mr, T (&L)[9])
{
    L[0] = T(0);
    { const T m = __ldg(Mr + 0);
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
    }
    { const T m = __ldg(Mr + 1);
      L[1] = m2l_fma(-D[4], m, L[1]);
      L[2] = m2l_fma(-D[5], m, L[2]);
      L[3] = m2l_fma(-D[6], m, L[3]);
    }
    { const T m = __ldg(Mr + 2);
      L[1] = m2l_fma(-D[5], m, L[1]);
      L[2] = m2l_fma(-D[7], m, L[2]);
      L[3] = m2l_fma(-D[8], m, L[3]);
    }
    { const T m = __ldg(Mr + 3);
      L[1] = m2l_fma(-D[6], m, L[1]);
      L[2] = m2l_fma(-D[8], m, L[2]);
      L[3] = m2l_fma(-D[9], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_reduce_moments_h_2(const T *__restrict__ Ms, T *__restrict__ Mr)
{
    T v0 = Ms[0];
    T v1 = Ms[1];
    T v2 = Ms[2];
    T v3 = Ms[3];
    T v4 = Ms[4];
    T v5 = Ms[5];
    T v6 = Ms[6];
    T v7 = Ms[7];
    T v8 = Ms[8];
    T v9 = Ms[9];
    v4 -= v9;
    v7 -= v9;
    Mr[0] = v0;
    Mr[1] = v1;
    Mr[2] = v2;
    Mr[3] = v3;
    Mr[4] = v4;
    Mr[5] = v5;
    Mr[6] = v6;
    Mr[7] = v7;
    Mr[8] = v8;
}

template <class T> __device__ __forceinline__ void m2l_complete_locals_h_2(const T *__restrict__ Lr, T *__restrict__ L)
{
    const T v0 = Lr[0];
    L[0] = v0;
    const T v1 = Lr[1];
    L[1] = v1;
    const T v2 = Lr[2];
    L[2] = v2;
    const T v3 = Lr[3];
    L[3] = v3;
    const T v4 = Lr[4];
    L[4] = v4;
    const T v5 = Lr[5];
    L[5] = v5;
    const T v6 = Lr[6];
    L[6] = v6;
    const T v7 = Lr[7];
    L[7] = v7;
    const T v8 = Lr[8];
    L[8] = v8;
    const T v9 = -v4 - v7;
    L[9] = v9;
}

template <class T> __device__ __forceinline__ void m2l_dtensor_h_3(T dx, T dy, T dz, T (&D)[19])
{
    const T s2 = m2l_fma(dx, dx, m2l_fma(dy, dy, dz * dz));
    const T si = m2l_rsqrt(s2);
    const T si2 = si * si;
    const T f0 = -si;
    const T f1 = T(-1) * f0 * si2;
    const T f2 = T(-3) * f1 * si2;
    const T f3 = T(-5) * f2 * si2;
    const T r_0_0 = f0;
    const T r_1_0 = f1;
    const T r_2_0 = f2;
    const T r_3_0 = f3;
    const T r_0_1 = dx * r_1_0;
    const T r_1_1 = dx * r_2_0;
    const T r_2_1 = dx * r_3_0;
    const T r_0_2 = dy * r_1_0;
    const T r_1_2 = dy * r_2_0;
    const T r_2_2 = dy * r_3_0;
    const T r_0_4 = m2l_fma(T(1), r_1_0, dx * r_1_1);
    const T r_1_4 = m2l_fma(T(1), r_2_0, dx * r_2_1);
    const T r_0_5 = dx * r_1_2;
    const T r_1_5 = dx * r_2_2;
    const T r_0_7 = m2l_fma(T(1), r_1_0, dy * r_1_2);
    const T r_1_7 = m2l_fma(T(1), r_2_0, dy * r_2_2);
    const T r_0_10 = m2l_fma(T(2), r_1_1, dx * r_1_4);
    const T r_0_11 = m2l_fma(T(1), r_1_2, dx * r_1_5);
    const T r_0_13 = dx * r_1_7;
    const T r_0_16 = m2l_fma(T(2), r_1_2, dy * r_1_7);
    D[0] = r_0_0;
    D[1] = r_0_1;
    D[2] = r_0_2;
    D[3] = dz * r_1_0;
    D[4] = r_0_4;
    D[5] = r_0_5;
    D[6] = dz * r_1_1;
    D[7] = r_0_7;
    D[8] = dz * r_1_2;
    D[10] = r_0_10;
    D[11] = r_0_11;
    D[12] = dz * r_1_4;
    D[13] = r_0_13;
    D[14] = dz * r_1_5;
    D[16] = r_0_16;
    D[17] = dz * r_1_7;
    D[9] = -D[4] - D[7];
    D[15] = -D[10] - D[13];
    D[18] = -D[11] - D[16];
}

template <class T> __device__ __forceinline__ void m2l_side_a_h_3(const T (&D)[19], const T *__restrict__ Mr, T rho, T (&L)[16])
{
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[0] = D[0] * m;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[10] * m;
      L[10] = D[11] * m;
      L[11] = D[12] * m;
      L[12] = D[13] * m;
      L[13] = D[14] * m;
      L[14] = D[16] * m;
      L[15] = D[17] * m;
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 1) * rp;
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
    }
    { const T m = -__ldg(Mr + 2) * rp;
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
    }
    { const T m = -__ldg(Mr + 3) * rp;
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 4) * rp;
      L[0] = m2l_fma(D[4], m, L[0]);
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
    }
    { const T m = __ldg(Mr + 5) * rp;
      L[0] = m2l_fma(D[5], m, L[0]);
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
    }
    { const T m = __ldg(Mr + 6) * rp;
      L[0] = m2l_fma(D[6], m, L[0]);
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
    }
    { const T m = __ldg(Mr + 7) * rp;
      L[0] = m2l_fma(D[7], m, L[0]);
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
    }
    { const T m = __ldg(Mr + 8) * rp;
      L[0] = m2l_fma(D[8], m, L[0]);
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 9) * rp;
      L[0] = m2l_fma(D[10], m, L[0]);
    }
    { const T m = -__ldg(Mr + 10) * rp;
      L[0] = m2l_fma(D[11], m, L[0]);
    }
    { const T m = -__ldg(Mr + 11) * rp;
      L[0] = m2l_fma(D[12], m, L[0]);
    }
    { const T m = -__ldg(Mr + 12) * rp;
      L[0] = m2l_fma(D[13], m, L[0]);
    }
    { const T m = -__ldg(Mr + 13) * rp;
      L[0] = m2l_fma(D[14], m, L[0]);
    }
    { const T m = -__ldg(Mr + 14) * rp;
      L[0] = m2l_fma(D[16], m, L[0]);
    }
    { const T m = -__ldg(Mr + 15) * rp;
      L[0] = m2l_fma(D[17], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_acc_h_3(const T (&D)[19], const T *__restrict__ Mr, T rho, T (&L)[16])
{
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[0] = m2l_fma(D[0], m, L[0]);
      L[1] = m2l_fma(D[1], m, L[1]);
      L[2] = m2l_fma(D[2], m, L[2]);
      L[3] = m2l_fma(D[3], m, L[3]);
      L[4] = m2l_fma(D[4], m, L[4]);
      L[5] = m2l_fma(D[5], m, L[5]);
      L[6] = m2l_fma(D[6], m, L[6]);
      L[7] = m2l_fma(D[7], m, L[7]);
      L[8] = m2l_fma(D[8], m, L[8]);
      L[9] = m2l_fma(D[10], m, L[9]);
      L[10] = m2l_fma(D[11], m, L[10]);
      L[11] = m2l_fma(D[12], m, L[11]);
      L[12] = m2l_fma(D[13], m, L[12]);
      L[13] = m2l_fma(D[14], m, L[13]);
      L[14] = m2l_fma(D[16], m, L[14]);
      L[15] = m2l_fma(D[17], m, L[15]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 1) * rp;
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
    }
    { const T m = -__ldg(Mr + 2) * rp;
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
    }
    { const T m = -__ldg(Mr + 3) * rp;
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 4) * rp;
      L[0] = m2l_fma(D[4], m, L[0]);
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
    }
    { const T m = __ldg(Mr + 5) * rp;
      L[0] = m2l_fma(D[5], m, L[0]);
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
    }
    { const T m = __ldg(Mr + 6) * rp;
      L[0] = m2l_fma(D[6], m, L[0]);
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
    }
    { const T m = __ldg(Mr + 7) * rp;
      L[0] = m2l_fma(D[7], m, L[0]);
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
    }
    { const T m = __ldg(Mr + 8) * rp;
      L[0] = m2l_fma(D[8], m, L[0]);
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 9) * rp;
      L[0] = m2l_fma(D[10], m, L[0]);
    }
    { const T m = -__ldg(Mr + 10) * rp;
      L[0] = m2l_fma(D[11], m, L[0]);
    }
    { const T m = -__ldg(Mr + 11) * rp;
      L[0] = m2l_fma(D[12], m, L[0]);
    }
    { const T m = -__ldg(Mr + 12) * rp;
      L[0] = m2l_fma(D[13], m, L[0]);
    }
    { const T m = -__ldg(Mr + 13) * rp;
      L[0] = m2l_fma(D[14], m, L[0]);
    }
    { const T m = -__ldg(Mr + 14) * rp;
      L[0] = m2l_fma(D[16], m, L[0]);
    }
    { const T m = -__ldg(Mr + 15) * rp;
      L[0] = m2l_fma(D[17], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_h_3(const T (&D)[19], const T *__restrict__ Mr, T (&L)[16])
{
    { const T m = __ldg(Mr + 0);
      L[0] = D[0] * m;
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = -D[10] * m;
      L[10] = -D[11] * m;
      L[11] = -D[12] * m;
      L[12] = -D[13] * m;
      L[13] = -D[14] * m;
      L[14] = -D[16] * m;
      L[15] = -D[17] * m;
    }
    { const T m = __ldg(Mr + 1);
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(-D[4], m, L[1]);
      L[2] = m2l_fma(-D[5], m, L[2]);
      L[3] = m2l_fma(-D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
    }
    { const T m = __ldg(Mr + 2);
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(-D[5], m, L[1]);
      L[2] = m2l_fma(-D[7], m, L[2]);
      L[3] = m2l_fma(-D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
    }
    { const T m = __ldg(Mr + 3);
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(-D[6], m, L[1]);
      L[2] = m2l_fma(-D[8], m, L[2]);
      L[3] = m2l_fma(-D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
    }
    { const T m = __ldg(Mr + 4);
      L[0] = m2l_fma(D[4], m, L[0]);
      L[1] = m2l_fma(-D[10], m, L[1]);
      L[2] = m2l_fma(-D[11], m, L[2]);
      L[3] = m2l_fma(-D[12], m, L[3]);
    }
    { const T m = __ldg(Mr + 5);
      L[0] = m2l_fma(D[5], m, L[0]);
      L[1] = m2l_fma(-D[11], m, L[1]);
      L[2] = m2l_fma(-D[13], m, L[2]);
      L[3] = m2l_fma(-D[14], m, L[3]);
    }
    { const T m = __ldg(Mr + 6);
      L[0] = m2l_fma(D[6], m, L[0]);
      L[1] = m2l_fma(-D[12], m, L[1]);
      L[2] = m2l_fma(-D[14], m, L[2]);
      L[3] = m2l_fma(-D[15], m, L[3]);
    }
    { const T m = __ldg(Mr + 7);
      L[0] = m2l_fma(D[7], m, L[0]);
      L[1] = m2l_fma(-D[13], m, L[1]);
      L[2] = m2l_fma(-D[16], m, L[2]);
      L[3] = m2l_fma(-D[17], m, L[3]);
    }
    { const T m = __ldg(Mr + 8);
      L[0] = m2l_fma(D[8], m, L[0]);
      L[1] = m2l_fma(-D[14], m, L[1]);
      L[2] = m2l_fma(-D[17], m, L[2]);
      L[3] = m2l_fma(-D[18], m, L[3]);
    }
    { const T m = __ldg(Mr + 9);
      L[0] = m2l_fma(D[10], m, L[0]);
    }
    { const T m = __ldg(Mr + 10);
      L[0] = m2l_fma(D[11], m, L[0]);
    }
    { const T m = __ldg(Mr + 11);
      L[0] = m2l_fma(D[12], m, L[0]);
    }
    { const T m = __ldg(Mr + 12);
      L[0] = m2l_fma(D[13], m, L[0]);
    }
    { const T m = __ldg(Mr + 13);
      L[0] = m2l_fma(D[14], m, L[0]);
    }
    { const T m = __ldg(Mr + 14);
      L[0] = m2l_fma(D[16], m, L[0]);
    }
    { const T m = __ldg(Mr + 15);
      L[0] = m2l_fma(D[17], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_a_h_forces_3(const T (&D)[19], const T *__restrict__ Mr, T rho, T (&L)[16])
{
    L[0] = T(0);
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[10] * m;
      L[10] = D[11] * m;
      L[11] = D[12] * m;
      L[12] = D[13] * m;
      L[13] = D[14] * m;
      L[14] = D[16] * m;
      L[15] = D[17] * m;
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 1) * rp;
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
    }
    { const T m = -__ldg(Mr + 2) * rp;
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
    }
    { const T m = -__ldg(Mr + 3) * rp;
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 4) * rp;
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
    }
    { const T m = __ldg(Mr + 5) * rp;
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
    }
    { const T m = __ldg(Mr + 6) * rp;
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
    }
    { const T m = __ldg(Mr + 7) * rp;
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
    }
    { const T m = __ldg(Mr + 8) * rp;
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_acc_h_forces_3(const T (&D)[19], const T *__restrict__ Mr, T rho, T (&L)[16])
{
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[1] = m2l_fma(D[1], m, L[1]);
      L[2] = m2l_fma(D[2], m, L[2]);
      L[3] = m2l_fma(D[3], m, L[3]);
      L[4] = m2l_fma(D[4], m, L[4]);
      L[5] = m2l_fma(D[5], m, L[5]);
      L[6] = m2l_fma(D[6], m, L[6]);
      L[7] = m2l_fma(D[7], m, L[7]);
      L[8] = m2l_fma(D[8], m, L[8]);
      L[9] = m2l_fma(D[10], m, L[9]);
      L[10] = m2l_fma(D[11], m, L[10]);
      L[11] = m2l_fma(D[12], m, L[11]);
      L[12] = m2l_fma(D[13], m, L[12]);
      L[13] = m2l_fma(D[14], m, L[13]);
      L[14] = m2l_fma(D[16], m, L[14]);
      L[15] = m2l_fma(D[17], m, L[15]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 1) * rp;
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
    }
    { const T m = -__ldg(Mr + 2) * rp;
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
    }
    { const T m = -__ldg(Mr + 3) * rp;
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 4) * rp;
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
    }
    { const T m = __ldg(Mr + 5) * rp;
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
    }
    { const T m = __ldg(Mr + 6) * rp;
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
    }
    { const T m = __ldg(Mr + 7) * rp;
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
    }
    { const T m = __ldg(Mr + 8) * rp;
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_h_forces_3(const T (&D)[19], const T *__restrict__ Mr, T (&L)[16])
{
    L[0] = T(0);
    { const T m = __ldg(Mr + 0);
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = -D[10] * m;
      L[10] = -D[11] * m;
      L[11] = -D[12] * m;
      L[12] = -D[13] * m;
      L[13] = -D[14] * m;
      L[14] = -D[16] * m;
      L[15] = -D[17] * m;
    }
    { const T m = __ldg(Mr + 1);
      L[1] = m2l_fma(-D[4], m, L[1]);
      L[2] = m2l_fma(-D[5], m, L[2]);
      L[3] = m2l_fma(-D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
    }
    { const T m = __ldg(Mr + 2);
      L[1] = m2l_fma(-D[5], m, L[1]);
      L[2] = m2l_fma(-D[7], m, L[2]);
      L[3] = m2l_fma(-D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
    }
    { const T m = __ldg(Mr + 3);
      L[1] = m2l_fma(-D[6], m, L[1]);
      L[2] = m2l_fma(-D[8], m, L[2]);
      L[3] = m2l_fma(-D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
    }
    { const T m = __ldg(Mr + 4);
      L[1] = m2l_fma(-D[10], m, L[1]);
      L[2] = m2l_fma(-D[11], m, L[2]);
      L[3] = m2l_fma(-D[12], m, L[3]);
    }
    { const T m = __ldg(Mr + 5);
      L[1] = m2l_fma(-D[11], m, L[1]);
      L[2] = m2l_fma(-D[13], m, L[2]);
      L[3] = m2l_fma(-D[14], m, L[3]);
    }
    { const T m = __ldg(Mr + 6);
      L[1] = m2l_fma(-D[12], m, L[1]);
      L[2] = m2l_fma(-D[14], m, L[2]);
      L[3] = m2l_fma(-D[15], m, L[3]);
    }
    { const T m = __ldg(Mr + 7);
      L[1] = m2l_fma(-D[13], m, L[1]);
      L[2] = m2l_fma(-D[16], m, L[2]);
      L[3] = m2l_fma(-D[17], m, L[3]);
    }
    { const T m = __ldg(Mr + 8);
      L[1] = m2l_fma(-D[14], m, L[1]);
      L[2] = m2l_fma(-D[17], m, L[2]);
      L[3] = m2l_fma(-D[18], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_reduce_moments_h_3(const T *__restrict__ Ms, T *__restrict__ Mr)
{
    T v0 = Ms[0];
    T v1 = Ms[1];
    T v2 = Ms[2];
    T v3 = Ms[3];
    T v4 = Ms[4];
    T v5 = Ms[5];
    T v6 = Ms[6];
    T v7 = Ms[7];
    T v8 = Ms[8];
    T v9 = Ms[9];
    T v10 = Ms[10];
    T v11 = Ms[11];
    T v12 = Ms[12];
    T v13 = Ms[13];
    T v14 = Ms[14];
    T v15 = Ms[15];
    T v16 = Ms[16];
    T v17 = Ms[17];
    T v18 = Ms[18];
    T v19 = Ms[19];
    v12 -= v19;
    v17 -= v19;
    v4 -= v9;
    v7 -= v9;
    v10 -= v15;
    v13 -= v15;
    v11 -= v18;
    v16 -= v18;
    Mr[0] = v0;
    Mr[1] = v1;
    Mr[2] = v2;
    Mr[3] = v3;
    Mr[4] = v4;
    Mr[5] = v5;
    Mr[6] = v6;
    Mr[7] = v7;
    Mr[8] = v8;
    Mr[9] = v10;
    Mr[10] = v11;
    Mr[11] = v12;
    Mr[12] = v13;
    Mr[13] = v14;
    Mr[14] = v16;
    Mr[15] = v17;
}

template <class T> __device__ __forceinline__ void m2l_complete_locals_h_3(const T *__restrict__ Lr, T *__restrict__ L)
{
    const T v0 = Lr[0];
    L[0] = v0;
    const T v1 = Lr[1];
    L[1] = v1;
    const T v2 = Lr[2];
    L[2] = v2;
    const T v3 = Lr[3];
    L[3] = v3;
    const T v4 = Lr[4];
    L[4] = v4;
    const T v5 = Lr[5];
    L[5] = v5;
    const T v6 = Lr[6];
    L[6] = v6;
    const T v7 = Lr[7];
    L[7] = v7;
    const T v8 = Lr[8];
    L[8] = v8;
    const T v9 = -v4 - v7;
    L[9] = v9;
    const T v10 = Lr[9];
    L[10] = v10;
    const T v11 = Lr[10];
    L[11] = v11;
    const T v12 = Lr[11];
    L[12] = v12;
    const T v13 = Lr[12];
    L[13] = v13;
    const T v14 = Lr[13];
    L[14] = v14;
    const T v15 = -v10 - v13;
    L[15] = v15;
    const T v16 = Lr[14];
    L[16] = v16;
    const T v17 = Lr[15];
    L[17] = v17;
    const T v18 = -v11 - v16;
    L[18] = v18;
    const T v19 = -v12 - v17;
    L[19] = v19;
}

template <class T> __device__ __forceinline__ void m2l_dtensor_h_4(T dx, T dy, T dz, T (&D)[31])
{
    const T s2 = m2l_fma(dx, dx, m2l_fma(dy, dy, dz * dz));
    const T si = m2l_rsqrt(s2);
    const T si2 = si * si;
    const T f0 = -si;
    const T f1 = T(-1) * f0 * si2;
    const T f2 = T(-3) * f1 * si2;
    const T f3 = T(-5) * f2 * si2;
    const T f4 = T(-7) * f3 * si2;
    const T r_0_0 = f0;
    const T r_1_0 = f1;
    const T r_2_0 = f2;
    const T r_3_0 = f3;
    const T r_4_0 = f4;
    const T r_0_1 = dx * r_1_0;
    const T r_1_1 = dx * r_2_0;
    const T r_2_1 = dx * r_3_0;
    const T r_3_1 = dx * r_4_0;
    const T r_0_2 = dy * r_1_0;
    const T r_1_2 = dy * r_2_0;
    const T r_2_2 = dy * r_3_0;
    const T r_3_2 = dy * r_4_0;
    const T r_0_4 = m2l_fma(T(1), r_1_0, dx * r_1_1);
    const T r_1_4 = m2l_fma(T(1), r_2_0, dx * r_2_1);
    const T r_2_4 = m2l_fma(T(1), r_3_0, dx * r_3_1);
    const T r_0_5 = dx * r_1_2;
    const T r_1_5 = dx * r_2_2;
    const T r_2_5 = dx * r_3_2;
    const T r_0_7 = m2l_fma(T(1), r_1_0, dy * r_1_2);
    const T r_1_7 = m2l_fma(T(1), r_2_0, dy * r_2_2);
    const T r_2_7 = m2l_fma(T(1), r_3_0, dy * r_3_2);
    const T r_0_10 = m2l_fma(T(2), r_1_1, dx * r_1_4);
    const T r_1_10 = m2l_fma(T(2), r_2_1, dx * r_2_4);
    const T r_0_11 = m2l_fma(T(1), r_1_2, dx * r_1_5);
    const T r_1_11 = m2l_fma(T(1), r_2_2, dx * r_2_5);
    const T r_0_13 = dx * r_1_7;
    const T r_1_13 = dx * r_2_7;
    const T r_0_16 = m2l_fma(T(2), r_1_2, dy * r_1_7);
    const T r_1_16 = m2l_fma(T(2), r_2_2, dy * r_2_7);
    const T r_0_20 = m2l_fma(T(3), r_1_4, dx * r_1_10);
    const T r_0_21 = m2l_fma(T(2), r_1_5, dx * r_1_11);
    const T r_0_23 = m2l_fma(T(1), r_1_7, dx * r_1_13);
    const T r_0_26 = dx * r_1_16;
    const T r_0_30 = m2l_fma(T(3), r_1_7, dy * r_1_16);
    D[0] = r_0_0;
    D[1] = r_0_1;
    D[2] = r_0_2;
    D[3] = dz * r_1_0;
    D[4] = r_0_4;
    D[5] = r_0_5;
    D[6] = dz * r_1_1;
    D[7] = r_0_7;
    D[8] = dz * r_1_2;
    D[10] = r_0_10;
    D[11] = r_0_11;
    D[12] = dz * r_1_4;
    D[13] = r_0_13;
    D[14] = dz * r_1_5;
    D[16] = r_0_16;
    D[17] = dz * r_1_7;
    D[19] = r_0_20;
    D[20] = r_0_21;
    D[21] = dz * r_1_10;
    D[22] = r_0_23;
    D[23] = dz * r_1_11;
    D[25] = r_0_26;
    D[26] = dz * r_1_13;
    D[28] = r_0_30;
    D[29] = dz * r_1_16;
    D[9] = -D[4] - D[7];
    D[15] = -D[10] - D[13];
    D[18] = -D[11] - D[16];
    D[24] = -D[19] - D[22];
    D[27] = -D[20] - D[25];
    D[30] = -D[22] - D[28];
}

template <class T> __device__ __forceinline__ void m2l_side_a_h_4(const T (&D)[31], const T *__restrict__ Mr, T rho, T (&L)[25])
{
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[0] = D[0] * m;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[10] * m;
      L[10] = D[11] * m;
      L[11] = D[12] * m;
      L[12] = D[13] * m;
      L[13] = D[14] * m;
      L[14] = D[16] * m;
      L[15] = D[17] * m;
      L[16] = D[19] * m;
      L[17] = D[20] * m;
      L[18] = D[21] * m;
      L[19] = D[22] * m;
      L[20] = D[23] * m;
      L[21] = D[25] * m;
      L[22] = D[26] * m;
      L[23] = D[28] * m;
      L[24] = D[29] * m;
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 1) * rp;
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(D[20], m, L[10]);
      L[11] = m2l_fma(D[21], m, L[11]);
      L[12] = m2l_fma(D[22], m, L[12]);
      L[13] = m2l_fma(D[23], m, L[13]);
      L[14] = m2l_fma(D[25], m, L[14]);
      L[15] = m2l_fma(D[26], m, L[15]);
    }
    { const T m = -__ldg(Mr + 2) * rp;
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[20], m, L[9]);
      L[10] = m2l_fma(D[22], m, L[10]);
      L[11] = m2l_fma(D[23], m, L[11]);
      L[12] = m2l_fma(D[25], m, L[12]);
      L[13] = m2l_fma(D[26], m, L[13]);
      L[14] = m2l_fma(D[28], m, L[14]);
      L[15] = m2l_fma(D[29], m, L[15]);
    }
    { const T m = -__ldg(Mr + 3) * rp;
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[21], m, L[9]);
      L[10] = m2l_fma(D[23], m, L[10]);
      L[11] = m2l_fma(D[24], m, L[11]);
      L[12] = m2l_fma(D[26], m, L[12]);
      L[13] = m2l_fma(D[27], m, L[13]);
      L[14] = m2l_fma(D[29], m, L[14]);
      L[15] = m2l_fma(D[30], m, L[15]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 4) * rp;
      L[0] = m2l_fma(D[4], m, L[0]);
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
      L[4] = m2l_fma(D[19], m, L[4]);
      L[5] = m2l_fma(D[20], m, L[5]);
      L[6] = m2l_fma(D[21], m, L[6]);
      L[7] = m2l_fma(D[22], m, L[7]);
      L[8] = m2l_fma(D[23], m, L[8]);
    }
    { const T m = __ldg(Mr + 5) * rp;
      L[0] = m2l_fma(D[5], m, L[0]);
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[22], m, L[5]);
      L[6] = m2l_fma(D[23], m, L[6]);
      L[7] = m2l_fma(D[25], m, L[7]);
      L[8] = m2l_fma(D[26], m, L[8]);
    }
    { const T m = __ldg(Mr + 6) * rp;
      L[0] = m2l_fma(D[6], m, L[0]);
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
    }
    { const T m = __ldg(Mr + 7) * rp;
      L[0] = m2l_fma(D[7], m, L[0]);
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[25], m, L[5]);
      L[6] = m2l_fma(D[26], m, L[6]);
      L[7] = m2l_fma(D[28], m, L[7]);
      L[8] = m2l_fma(D[29], m, L[8]);
    }
    { const T m = __ldg(Mr + 8) * rp;
      L[0] = m2l_fma(D[8], m, L[0]);
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[29], m, L[7]);
      L[8] = m2l_fma(D[30], m, L[8]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 9) * rp;
      L[0] = m2l_fma(D[10], m, L[0]);
      L[1] = m2l_fma(D[19], m, L[1]);
      L[2] = m2l_fma(D[20], m, L[2]);
      L[3] = m2l_fma(D[21], m, L[3]);
    }
    { const T m = -__ldg(Mr + 10) * rp;
      L[0] = m2l_fma(D[11], m, L[0]);
      L[1] = m2l_fma(D[20], m, L[1]);
      L[2] = m2l_fma(D[22], m, L[2]);
      L[3] = m2l_fma(D[23], m, L[3]);
    }
    { const T m = -__ldg(Mr + 11) * rp;
      L[0] = m2l_fma(D[12], m, L[0]);
      L[1] = m2l_fma(D[21], m, L[1]);
      L[2] = m2l_fma(D[23], m, L[2]);
      L[3] = m2l_fma(D[24], m, L[3]);
    }
    { const T m = -__ldg(Mr + 12) * rp;
      L[0] = m2l_fma(D[13], m, L[0]);
      L[1] = m2l_fma(D[22], m, L[1]);
      L[2] = m2l_fma(D[25], m, L[2]);
      L[3] = m2l_fma(D[26], m, L[3]);
    }
    { const T m = -__ldg(Mr + 13) * rp;
      L[0] = m2l_fma(D[14], m, L[0]);
      L[1] = m2l_fma(D[23], m, L[1]);
      L[2] = m2l_fma(D[26], m, L[2]);
      L[3] = m2l_fma(D[27], m, L[3]);
    }
    { const T m = -__ldg(Mr + 14) * rp;
      L[0] = m2l_fma(D[16], m, L[0]);
      L[1] = m2l_fma(D[25], m, L[1]);
      L[2] = m2l_fma(D[28], m, L[2]);
      L[3] = m2l_fma(D[29], m, L[3]);
    }
    { const T m = -__ldg(Mr + 15) * rp;
      L[0] = m2l_fma(D[17], m, L[0]);
      L[1] = m2l_fma(D[26], m, L[1]);
      L[2] = m2l_fma(D[29], m, L[2]);
      L[3] = m2l_fma(D[30], m, L[3]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 16) * rp;
      L[0] = m2l_fma(D[19], m, L[0]);
    }
    { const T m = __ldg(Mr + 17) * rp;
      L[0] = m2l_fma(D[20], m, L[0]);
    }
    { const T m = __ldg(Mr + 18) * rp;
      L[0] = m2l_fma(D[21], m, L[0]);
    }
    { const T m = __ldg(Mr + 19) * rp;
      L[0] = m2l_fma(D[22], m, L[0]);
    }
    { const T m = __ldg(Mr + 20) * rp;
      L[0] = m2l_fma(D[23], m, L[0]);
    }
    { const T m = __ldg(Mr + 21) * rp;
      L[0] = m2l_fma(D[25], m, L[0]);
    }
    { const T m = __ldg(Mr + 22) * rp;
      L[0] = m2l_fma(D[26], m, L[0]);
    }
    { const T m = __ldg(Mr + 23) * rp;
      L[0] = m2l_fma(D[28], m, L[0]);
    }
    { const T m = __ldg(Mr + 24) * rp;
      L[0] = m2l_fma(D[29], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_acc_h_4(const T (&D)[31], const T *__restrict__ Mr, T rho, T (&L)[25])
{
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[0] = m2l_fma(D[0], m, L[0]);
      L[1] = m2l_fma(D[1], m, L[1]);
      L[2] = m2l_fma(D[2], m, L[2]);
      L[3] = m2l_fma(D[3], m, L[3]);
      L[4] = m2l_fma(D[4], m, L[4]);
      L[5] = m2l_fma(D[5], m, L[5]);
      L[6] = m2l_fma(D[6], m, L[6]);
      L[7] = m2l_fma(D[7], m, L[7]);
      L[8] = m2l_fma(D[8], m, L[8]);
      L[9] = m2l_fma(D[10], m, L[9]);
      L[10] = m2l_fma(D[11], m, L[10]);
      L[11] = m2l_fma(D[12], m, L[11]);
      L[12] = m2l_fma(D[13], m, L[12]);
      L[13] = m2l_fma(D[14], m, L[13]);
      L[14] = m2l_fma(D[16], m, L[14]);
      L[15] = m2l_fma(D[17], m, L[15]);
      L[16] = m2l_fma(D[19], m, L[16]);
      L[17] = m2l_fma(D[20], m, L[17]);
      L[18] = m2l_fma(D[21], m, L[18]);
      L[19] = m2l_fma(D[22], m, L[19]);
      L[20] = m2l_fma(D[23], m, L[20]);
      L[21] = m2l_fma(D[25], m, L[21]);
      L[22] = m2l_fma(D[26], m, L[22]);
      L[23] = m2l_fma(D[28], m, L[23]);
      L[24] = m2l_fma(D[29], m, L[24]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 1) * rp;
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(D[20], m, L[10]);
      L[11] = m2l_fma(D[21], m, L[11]);
      L[12] = m2l_fma(D[22], m, L[12]);
      L[13] = m2l_fma(D[23], m, L[13]);
      L[14] = m2l_fma(D[25], m, L[14]);
      L[15] = m2l_fma(D[26], m, L[15]);
    }
    { const T m = -__ldg(Mr + 2) * rp;
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[20], m, L[9]);
      L[10] = m2l_fma(D[22], m, L[10]);
      L[11] = m2l_fma(D[23], m, L[11]);
      L[12] = m2l_fma(D[25], m, L[12]);
      L[13] = m2l_fma(D[26], m, L[13]);
      L[14] = m2l_fma(D[28], m, L[14]);
      L[15] = m2l_fma(D[29], m, L[15]);
    }
    { const T m = -__ldg(Mr + 3) * rp;
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[21], m, L[9]);
      L[10] = m2l_fma(D[23], m, L[10]);
      L[11] = m2l_fma(D[24], m, L[11]);
      L[12] = m2l_fma(D[26], m, L[12]);
      L[13] = m2l_fma(D[27], m, L[13]);
      L[14] = m2l_fma(D[29], m, L[14]);
      L[15] = m2l_fma(D[30], m, L[15]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 4) * rp;
      L[0] = m2l_fma(D[4], m, L[0]);
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
      L[4] = m2l_fma(D[19], m, L[4]);
      L[5] = m2l_fma(D[20], m, L[5]);
      L[6] = m2l_fma(D[21], m, L[6]);
      L[7] = m2l_fma(D[22], m, L[7]);
      L[8] = m2l_fma(D[23], m, L[8]);
    }
    { const T m = __ldg(Mr + 5) * rp;
      L[0] = m2l_fma(D[5], m, L[0]);
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[22], m, L[5]);
      L[6] = m2l_fma(D[23], m, L[6]);
      L[7] = m2l_fma(D[25], m, L[7]);
      L[8] = m2l_fma(D[26], m, L[8]);
    }
    { const T m = __ldg(Mr + 6) * rp;
      L[0] = m2l_fma(D[6], m, L[0]);
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
    }
    { const T m = __ldg(Mr + 7) * rp;
      L[0] = m2l_fma(D[7], m, L[0]);
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[25], m, L[5]);
      L[6] = m2l_fma(D[26], m, L[6]);
      L[7] = m2l_fma(D[28], m, L[7]);
      L[8] = m2l_fma(D[29], m, L[8]);
    }
    { const T m = __ldg(Mr + 8) * rp;
      L[0] = m2l_fma(D[8], m, L[0]);
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[29], m, L[7]);
      L[8] = m2l_fma(D[30], m, L[8]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 9) * rp;
      L[0] = m2l_fma(D[10], m, L[0]);
      L[1] = m2l_fma(D[19], m, L[1]);
      L[2] = m2l_fma(D[20], m, L[2]);
      L[3] = m2l_fma(D[21], m, L[3]);
    }
    { const T m = -__ldg(Mr + 10) * rp;
      L[0] = m2l_fma(D[11], m, L[0]);
      L[1] = m2l_fma(D[20], m, L[1]);
      L[2] = m2l_fma(D[22], m, L[2]);
      L[3] = m2l_fma(D[23], m, L[3]);
    }
    { const T m = -__ldg(Mr + 11) * rp;
      L[0] = m2l_fma(D[12], m, L[0]);
      L[1] = m2l_fma(D[21], m, L[1]);
      L[2] = m2l_fma(D[23], m, L[2]);
      L[3] = m2l_fma(D[24], m, L[3]);
    }
    { const T m = -__ldg(Mr + 12) * rp;
      L[0] = m2l_fma(D[13], m, L[0]);
      L[1] = m2l_fma(D[22], m, L[1]);
      L[2] = m2l_fma(D[25], m, L[2]);
      L[3] = m2l_fma(D[26], m, L[3]);
    }
    { const T m = -__ldg(Mr + 13) * rp;
      L[0] = m2l_fma(D[14], m, L[0]);
      L[1] = m2l_fma(D[23], m, L[1]);
      L[2] = m2l_fma(D[26], m, L[2]);
      L[3] = m2l_fma(D[27], m, L[3]);
    }
    { const T m = -__ldg(Mr + 14) * rp;
      L[0] = m2l_fma(D[16], m, L[0]);
      L[1] = m2l_fma(D[25], m, L[1]);
      L[2] = m2l_fma(D[28], m, L[2]);
      L[3] = m2l_fma(D[29], m, L[3]);
    }
    { const T m = -__ldg(Mr + 15) * rp;
      L[0] = m2l_fma(D[17], m, L[0]);
      L[1] = m2l_fma(D[26], m, L[1]);
      L[2] = m2l_fma(D[29], m, L[2]);
      L[3] = m2l_fma(D[30], m, L[3]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 16) * rp;
      L[0] = m2l_fma(D[19], m, L[0]);
    }
    { const T m = __ldg(Mr + 17) * rp;
      L[0] = m2l_fma(D[20], m, L[0]);
    }
    { const T m = __ldg(Mr + 18) * rp;
      L[0] = m2l_fma(D[21], m, L[0]);
    }
    { const T m = __ldg(Mr + 19) * rp;
      L[0] = m2l_fma(D[22], m, L[0]);
    }
    { const T m = __ldg(Mr + 20) * rp;
      L[0] = m2l_fma(D[23], m, L[0]);
    }
    { const T m = __ldg(Mr + 21) * rp;
      L[0] = m2l_fma(D[25], m, L[0]);
    }
    { const T m = __ldg(Mr + 22) * rp;
      L[0] = m2l_fma(D[26], m, L[0]);
    }
    { const T m = __ldg(Mr + 23) * rp;
      L[0] = m2l_fma(D[28], m, L[0]);
    }
    { const T m = __ldg(Mr + 24) * rp;
      L[0] = m2l_fma(D[29], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_h_4(const T (&D)[31], const T *__restrict__ Mr, T (&L)[25])
{
    { const T m = __ldg(Mr + 0);
      L[0] = D[0] * m;
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = -D[10] * m;
      L[10] = -D[11] * m;
      L[11] = -D[12] * m;
      L[12] = -D[13] * m;
      L[13] = -D[14] * m;
      L[14] = -D[16] * m;
      L[15] = -D[17] * m;
      L[16] = D[19] * m;
      L[17] = D[20] * m;
      L[18] = D[21] * m;
      L[19] = D[22] * m;
      L[20] = D[23] * m;
      L[21] = D[25] * m;
      L[22] = D[26] * m;
      L[23] = D[28] * m;
      L[24] = D[29] * m;
    }
    { const T m = __ldg(Mr + 1);
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(-D[4], m, L[1]);
      L[2] = m2l_fma(-D[5], m, L[2]);
      L[3] = m2l_fma(-D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(-D[19], m, L[9]);
      L[10] = m2l_fma(-D[20], m, L[10]);
      L[11] = m2l_fma(-D[21], m, L[11]);
      L[12] = m2l_fma(-D[22], m, L[12]);
      L[13] = m2l_fma(-D[23], m, L[13]);
      L[14] = m2l_fma(-D[25], m, L[14]);
      L[15] = m2l_fma(-D[26], m, L[15]);
    }
    { const T m = __ldg(Mr + 2);
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(-D[5], m, L[1]);
      L[2] = m2l_fma(-D[7], m, L[2]);
      L[3] = m2l_fma(-D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(-D[20], m, L[9]);
      L[10] = m2l_fma(-D[22], m, L[10]);
      L[11] = m2l_fma(-D[23], m, L[11]);
      L[12] = m2l_fma(-D[25], m, L[12]);
      L[13] = m2l_fma(-D[26], m, L[13]);
      L[14] = m2l_fma(-D[28], m, L[14]);
      L[15] = m2l_fma(-D[29], m, L[15]);
    }
    { const T m = __ldg(Mr + 3);
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(-D[6], m, L[1]);
      L[2] = m2l_fma(-D[8], m, L[2]);
      L[3] = m2l_fma(-D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(-D[21], m, L[9]);
      L[10] = m2l_fma(-D[23], m, L[10]);
      L[11] = m2l_fma(-D[24], m, L[11]);
      L[12] = m2l_fma(-D[26], m, L[12]);
      L[13] = m2l_fma(-D[27], m, L[13]);
      L[14] = m2l_fma(-D[29], m, L[14]);
      L[15] = m2l_fma(-D[30], m, L[15]);
    }
    { const T m = __ldg(Mr + 4);
      L[0] = m2l_fma(D[4], m, L[0]);
      L[1] = m2l_fma(-D[10], m, L[1]);
      L[2] = m2l_fma(-D[11], m, L[2]);
      L[3] = m2l_fma(-D[12], m, L[3]);
      L[4] = m2l_fma(D[19], m, L[4]);
      L[5] = m2l_fma(D[20], m, L[5]);
      L[6] = m2l_fma(D[21], m, L[6]);
      L[7] = m2l_fma(D[22], m, L[7]);
      L[8] = m2l_fma(D[23], m, L[8]);
    }
    { const T m = __ldg(Mr + 5);
      L[0] = m2l_fma(D[5], m, L[0]);
      L[1] = m2l_fma(-D[11], m, L[1]);
      L[2] = m2l_fma(-D[13], m, L[2]);
      L[3] = m2l_fma(-D[14], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[22], m, L[5]);
      L[6] = m2l_fma(D[23], m, L[6]);
      L[7] = m2l_fma(D[25], m, L[7]);
      L[8] = m2l_fma(D[26], m, L[8]);
    }
    { const T m = __ldg(Mr + 6);
      L[0] = m2l_fma(D[6], m, L[0]);
      L[1] = m2l_fma(-D[12], m, L[1]);
      L[2] = m2l_fma(-D[14], m, L[2]);
      L[3] = m2l_fma(-D[15], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
    }
    { const T m = __ldg(Mr + 7);
      L[0] = m2l_fma(D[7], m, L[0]);
      L[1] = m2l_fma(-D[13], m, L[1]);
      L[2] = m2l_fma(-D[16], m, L[2]);
      L[3] = m2l_fma(-D[17], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[25], m, L[5]);
      L[6] = m2l_fma(D[26], m, L[6]);
      L[7] = m2l_fma(D[28], m, L[7]);
      L[8] = m2l_fma(D[29], m, L[8]);
    }
    { const T m = __ldg(Mr + 8);
      L[0] = m2l_fma(D[8], m, L[0]);
      L[1] = m2l_fma(-D[14], m, L[1]);
      L[2] = m2l_fma(-D[17], m, L[2]);
      L[3] = m2l_fma(-D[18], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[29], m, L[7]);
      L[8] = m2l_fma(D[30], m, L[8]);
    }
    { const T m = __ldg(Mr + 9);
      L[0] = m2l_fma(D[10], m, L[0]);
      L[1] = m2l_fma(-D[19], m, L[1]);
      L[2] = m2l_fma(-D[20], m, L[2]);
      L[3] = m2l_fma(-D[21], m, L[3]);
    }
    { const T m = __ldg(Mr + 10);
      L[0] = m2l_fma(D[11], m, L[0]);
      L[1] = m2l_fma(-D[20], m, L[1]);
      L[2] = m2l_fma(-D[22], m, L[2]);
      L[3] = m2l_fma(-D[23], m, L[3]);
    }
    { const T m = __ldg(Mr + 11);
      L[0] = m2l_fma(D[12], m, L[0]);
      L[1] = m2l_fma(-D[21], m, L[1]);
      L[2] = m2l_fma(-D[23], m, L[2]);
      L[3] = m2l_fma(-D[24], m, L[3]);
    }
    { const T m = __ldg(Mr + 12);
      L[0] = m2l_fma(D[13], m, L[0]);
      L[1] = m2l_fma(-D[22], m, L[1]);
      L[2] = m2l_fma(-D[25], m, L[2]);
      L[3] = m2l_fma(-D[26], m, L[3]);
    }
    { const T m = __ldg(Mr + 13);
      L[0] = m2l_fma(D[14], m, L[0]);
      L[1] = m2l_fma(-D[23], m, L[1]);
      L[2] = m2l_fma(-D[26], m, L[2]);
      L[3] = m2l_fma(-D[27], m, L[3]);
    }
    { const T m = __ldg(Mr + 14);
      L[0] = m2l_fma(D[16], m, L[0]);
      L[1] = m2l_fma(-D[25], m, L[1]);
      L[2] = m2l_fma(-D[28], m, L[2]);
      L[3] = m2l_fma(-D[29], m, L[3]);
    }
    { const T m = __ldg(Mr + 15);
      L[0] = m2l_fma(D[17], m, L[0]);
      L[1] = m2l_fma(-D[26], m, L[1]);
      L[2] = m2l_fma(-D[29], m, L[2]);
      L[3] = m2l_fma(-D[30], m, L[3]);
    }
    { const T m = __ldg(Mr + 16);
      L[0] = m2l_fma(D[19], m, L[0]);
    }
    { const T m = __ldg(Mr + 17);
      L[0] = m2l_fma(D[20], m, L[0]);
    }
    { const T m = __ldg(Mr + 18);
      L[0] = m2l_fma(D[21], m, L[0]);
    }
    { const T m = __ldg(Mr + 19);
      L[0] = m2l_fma(D[22], m, L[0]);
    }
    { const T m = __ldg(Mr + 20);
      L[0] = m2l_fma(D[23], m, L[0]);
    }
    { const T m = __ldg(Mr + 21);
      L[0] = m2l_fma(D[25], m, L[0]);
    }
    { const T m = __ldg(Mr + 22);
      L[0] = m2l_fma(D[26], m, L[0]);
    }
    { const T m = __ldg(Mr + 23);
      L[0] = m2l_fma(D[28], m, L[0]);
    }
    { const T m = __ldg(Mr + 24);
      L[0] = m2l_fma(D[29], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_a_h_forces_4(const T (&D)[31], const T *__restrict__ Mr, T rho, T (&L)[25])
{
    L[0] = T(0);
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[10] * m;
      L[10] = D[11] * m;
      L[11] = D[12] * m;
      L[12] = D[13] * m;
      L[13] = D[14] * m;
      L[14] = D[16] * m;
      L[15] = D[17] * m;
      L[16] = D[19] * m;
      L[17] = D[20] * m;
      L[18] = D[21] * m;
      L[19] = D[22] * m;
      L[20] = D[23] * m;
      L[21] = D[25] * m;
      L[22] = D[26] * m;
      L[23] = D[28] * m;
      L[24] = D[29] * m;
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 1) * rp;
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(D[20], m, L[10]);
      L[11] = m2l_fma(D[21], m, L[11]);
      L[12] = m2l_fma(D[22], m, L[12]);
      L[13] = m2l_fma(D[23], m, L[13]);
      L[14] = m2l_fma(D[25], m, L[14]);
      L[15] = m2l_fma(D[26], m, L[15]);
    }
    { const T m = -__ldg(Mr + 2) * rp;
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[20], m, L[9]);
      L[10] = m2l_fma(D[22], m, L[10]);
      L[11] = m2l_fma(D[23], m, L[11]);
      L[12] = m2l_fma(D[25], m, L[12]);
      L[13] = m2l_fma(D[26], m, L[13]);
      L[14] = m2l_fma(D[28], m, L[14]);
      L[15] = m2l_fma(D[29], m, L[15]);
    }
    { const T m = -__ldg(Mr + 3) * rp;
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[21], m, L[9]);
      L[10] = m2l_fma(D[23], m, L[10]);
      L[11] = m2l_fma(D[24], m, L[11]);
      L[12] = m2l_fma(D[26], m, L[12]);
      L[13] = m2l_fma(D[27], m, L[13]);
      L[14] = m2l_fma(D[29], m, L[14]);
      L[15] = m2l_fma(D[30], m, L[15]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 4) * rp;
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
      L[4] = m2l_fma(D[19], m, L[4]);
      L[5] = m2l_fma(D[20], m, L[5]);
      L[6] = m2l_fma(D[21], m, L[6]);
      L[7] = m2l_fma(D[22], m, L[7]);
      L[8] = m2l_fma(D[23], m, L[8]);
    }
    { const T m = __ldg(Mr + 5) * rp;
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[22], m, L[5]);
      L[6] = m2l_fma(D[23], m, L[6]);
      L[7] = m2l_fma(D[25], m, L[7]);
      L[8] = m2l_fma(D[26], m, L[8]);
    }
    { const T m = __ldg(Mr + 6) * rp;
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
    }
    { const T m = __ldg(Mr + 7) * rp;
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[25], m, L[5]);
      L[6] = m2l_fma(D[26], m, L[6]);
      L[7] = m2l_fma(D[28], m, L[7]);
      L[8] = m2l_fma(D[29], m, L[8]);
    }
    { const T m = __ldg(Mr + 8) * rp;
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[29], m, L[7]);
      L[8] = m2l_fma(D[30], m, L[8]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 9) * rp;
      L[1] = m2l_fma(D[19], m, L[1]);
      L[2] = m2l_fma(D[20], m, L[2]);
      L[3] = m2l_fma(D[21], m, L[3]);
    }
    { const T m = -__ldg(Mr + 10) * rp;
      L[1] = m2l_fma(D[20], m, L[1]);
      L[2] = m2l_fma(D[22], m, L[2]);
      L[3] = m2l_fma(D[23], m, L[3]);
    }
    { const T m = -__ldg(Mr + 11) * rp;
      L[1] = m2l_fma(D[21], m, L[1]);
      L[2] = m2l_fma(D[23], m, L[2]);
      L[3] = m2l_fma(D[24], m, L[3]);
    }
    { const T m = -__ldg(Mr + 12) * rp;
      L[1] = m2l_fma(D[22], m, L[1]);
      L[2] = m2l_fma(D[25], m, L[2]);
      L[3] = m2l_fma(D[26], m, L[3]);
    }
    { const T m = -__ldg(Mr + 13) * rp;
      L[1] = m2l_fma(D[23], m, L[1]);
      L[2] = m2l_fma(D[26], m, L[2]);
      L[3] = m2l_fma(D[27], m, L[3]);
    }
    { const T m = -__ldg(Mr + 14) * rp;
      L[1] = m2l_fma(D[25], m, L[1]);
      L[2] = m2l_fma(D[28], m, L[2]);
      L[3] = m2l_fma(D[29], m, L[3]);
    }
    { const T m = -__ldg(Mr + 15) * rp;
      L[1] = m2l_fma(D[26], m, L[1]);
      L[2] = m2l_fma(D[29], m, L[2]);
      L[3] = m2l_fma(D[30], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_acc_h_forces_4(const T (&D)[31], const T *__restrict__ Mr, T rho, T (&L)[25])
{
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[1] = m2l_fma(D[1], m, L[1]);
      L[2] = m2l_fma(D[2], m, L[2]);
      L[3] = m2l_fma(D[3], m, L[3]);
      L[4] = m2l_fma(D[4], m, L[4]);
      L[5] = m2l_fma(D[5], m, L[5]);
      L[6] = m2l_fma(D[6], m, L[6]);
      L[7] = m2l_fma(D[7], m, L[7]);
      L[8] = m2l_fma(D[8], m, L[8]);
      L[9] = m2l_fma(D[10], m, L[9]);
      L[10] = m2l_fma(D[11], m, L[10]);
      L[11] = m2l_fma(D[12], m, L[11]);
      L[12] = m2l_fma(D[13], m, L[12]);
      L[13] = m2l_fma(D[14], m, L[13]);
      L[14] = m2l_fma(D[16], m, L[14]);
      L[15] = m2l_fma(D[17], m, L[15]);
      L[16] = m2l_fma(D[19], m, L[16]);
      L[17] = m2l_fma(D[20], m, L[17]);
      L[18] = m2l_fma(D[21], m, L[18]);
      L[19] = m2l_fma(D[22], m, L[19]);
      L[20] = m2l_fma(D[23], m, L[20]);
      L[21] = m2l_fma(D[25], m, L[21]);
      L[22] = m2l_fma(D[26], m, L[22]);
      L[23] = m2l_fma(D[28], m, L[23]);
      L[24] = m2l_fma(D[29], m, L[24]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 1) * rp;
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(D[20], m, L[10]);
      L[11] = m2l_fma(D[21], m, L[11]);
      L[12] = m2l_fma(D[22], m, L[12]);
      L[13] = m2l_fma(D[23], m, L[13]);
      L[14] = m2l_fma(D[25], m, L[14]);
      L[15] = m2l_fma(D[26], m, L[15]);
    }
    { const T m = -__ldg(Mr + 2) * rp;
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[20], m, L[9]);
      L[10] = m2l_fma(D[22], m, L[10]);
      L[11] = m2l_fma(D[23], m, L[11]);
      L[12] = m2l_fma(D[25], m, L[12]);
      L[13] = m2l_fma(D[26], m, L[13]);
      L[14] = m2l_fma(D[28], m, L[14]);
      L[15] = m2l_fma(D[29], m, L[15]);
    }
    { const T m = -__ldg(Mr + 3) * rp;
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[21], m, L[9]);
      L[10] = m2l_fma(D[23], m, L[10]);
      L[11] = m2l_fma(D[24], m, L[11]);
      L[12] = m2l_fma(D[26], m, L[12]);
      L[13] = m2l_fma(D[27], m, L[13]);
      L[14] = m2l_fma(D[29], m, L[14]);
      L[15] = m2l_fma(D[30], m, L[15]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 4) * rp;
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
      L[4] = m2l_fma(D[19], m, L[4]);
      L[5] = m2l_fma(D[20], m, L[5]);
      L[6] = m2l_fma(D[21], m, L[6]);
      L[7] = m2l_fma(D[22], m, L[7]);
      L[8] = m2l_fma(D[23], m, L[8]);
    }
    { const T m = __ldg(Mr + 5) * rp;
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[22], m, L[5]);
      L[6] = m2l_fma(D[23], m, L[6]);
      L[7] = m2l_fma(D[25], m, L[7]);
      L[8] = m2l_fma(D[26], m, L[8]);
    }
    { const T m = __ldg(Mr + 6) * rp;
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
    }
    { const T m = __ldg(Mr + 7) * rp;
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[25], m, L[5]);
      L[6] = m2l_fma(D[26], m, L[6]);
      L[7] = m2l_fma(D[28], m, L[7]);
      L[8] = m2l_fma(D[29], m, L[8]);
    }
    { const T m = __ldg(Mr + 8) * rp;
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[29], m, L[7]);
      L[8] = m2l_fma(D[30], m, L[8]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 9) * rp;
      L[1] = m2l_fma(D[19], m, L[1]);
      L[2] = m2l_fma(D[20], m, L[2]);
      L[3] = m2l_fma(D[21], m, L[3]);
    }
    { const T m = -__ldg(Mr + 10) * rp;
      L[1] = m2l_fma(D[20], m, L[1]);
      L[2] = m2l_fma(D[22], m, L[2]);
      L[3] = m2l_fma(D[23], m, L[3]);
    }
    { const T m = -__ldg(Mr + 11) * rp;
      L[1] = m2l_fma(D[21], m, L[1]);
      L[2] = m2l_fma(D[23], m, L[2]);
      L[3] = m2l_fma(D[24], m, L[3]);
    }
    { const T m = -__ldg(Mr + 12) * rp;
      L[1] = m2l_fma(D[22], m, L[1]);
      L[2] = m2l_fma(D[25], m, L[2]);
      L[3] = m2l_fma(D[26], m, L[3]);
    }
    { const T m = -__ldg(Mr + 13) * rp;
      L[1] = m2l_fma(D[23], m, L[1]);
      L[2] = m2l_fma(D[26], m, L[2]);
      L[3] = m2l_fma(D[27], m, L[3]);
    }
    { const T m = -__ldg(Mr + 14) * rp;
      L[1] = m2l_fma(D[25], m, L[1]);
      L[2] = m2l_fma(D[28], m, L[2]);
      L[3] = m2l_fma(D[29], m, L[3]);
    }
    { const T m = -__ldg(Mr + 15) * rp;
      L[1] = m2l_fma(D[26], m, L[1]);
      L[2] = m2l_fma(D[29], m, L[2]);
      L[3] = m2l_fma(D[30], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_h_forces_4(const T (&D)[31], const T *__restrict__ Mr, T (&L)[25])
{
    L[0] = T(0);
    { const T m = __ldg(Mr + 0);
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = -D[10] * m;
      L[10] = -D[11] * m;
      L[11] = -D[12] * m;
      L[12] = -D[13] * m;
      L[13] = -D[14] * m;
      L[14] = -D[16] * m;
      L[15] = -D[17] * m;
      L[16] = D[19] * m;
      L[17] = D[20] * m;
      L[18] = D[21] * m;
      L[19] = D[22] * m;
      L[20] = D[23] * m;
      L[21] = D[25] * m;
      L[22] = D[26] * m;
      L[23] = D[28] * m;
      L[24] = D[29] * m;
    }
    { const T m = __ldg(Mr + 1);
      L[1] = m2l_fma(-D[4], m, L[1]);
      L[2] = m2l_fma(-D[5], m, L[2]);
      L[3] = m2l_fma(-D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(-D[19], m, L[9]);
      L[10] = m2l_fma(-D[20], m, L[10]);
      L[11] = m2l_fma(-D[21], m, L[11]);
      L[12] = m2l_fma(-D[22], m, L[12]);
      L[13] = m2l_fma(-D[23], m, L[13]);
      L[14] = m2l_fma(-D[25], m, L[14]);
      L[15] = m2l_fma(-D[26], m, L[15]);
    }
    { const T m = __ldg(Mr + 2);
      L[1] = m2l_fma(-D[5], m, L[1]);
      L[2] = m2l_fma(-D[7], m, L[2]);
      L[3] = m2l_fma(-D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(-D[20], m, L[9]);
      L[10] = m2l_fma(-D[22], m, L[10]);
      L[11] = m2l_fma(-D[23], m, L[11]);
      L[12] = m2l_fma(-D[25], m, L[12]);
      L[13] = m2l_fma(-D[26], m, L[13]);
      L[14] = m2l_fma(-D[28], m, L[14]);
      L[15] = m2l_fma(-D[29], m, L[15]);
    }
    { const T m = __ldg(Mr + 3);
      L[1] = m2l_fma(-D[6], m, L[1]);
      L[2] = m2l_fma(-D[8], m, L[2]);
      L[3] = m2l_fma(-D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(-D[21], m, L[9]);
      L[10] = m2l_fma(-D[23], m, L[10]);
      L[11] = m2l_fma(-D[24], m, L[11]);
      L[12] = m2l_fma(-D[26], m, L[12]);
      L[13] = m2l_fma(-D[27], m, L[13]);
      L[14] = m2l_fma(-D[29], m, L[14]);
      L[15] = m2l_fma(-D[30], m, L[15]);
    }
    { const T m = __ldg(Mr + 4);
      L[1] = m2l_fma(-D[10], m, L[1]);
      L[2] = m2l_fma(-D[11], m, L[2]);
      L[3] = m2l_fma(-D[12], m, L[3]);
      L[4] = m2l_fma(D[19], m, L[4]);
      L[5] = m2l_fma(D[20], m, L[5]);
      L[6] = m2l_fma(D[21], m, L[6]);
      L[7] = m2l_fma(D[22], m, L[7]);
      L[8] = m2l_fma(D[23], m, L[8]);
    }
    { const T m = __ldg(Mr + 5);
      L[1] = m2l_fma(-D[11], m, L[1]);
      L[2] = m2l_fma(-D[13], m, L[2]);
      L[3] = m2l_fma(-D[14], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[22], m, L[5]);
      L[6] = m2l_fma(D[23], m, L[6]);
      L[7] = m2l_fma(D[25], m, L[7]);
      L[8] = m2l_fma(D[26], m, L[8]);
    }
    { const T m = __ldg(Mr + 6);
      L[1] = m2l_fma(-D[12], m, L[1]);
      L[2] = m2l_fma(-D[14], m, L[2]);
      L[3] = m2l_fma(-D[15], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
    }
    { const T m = __ldg(Mr + 7);
      L[1] = m2l_fma(-D[13], m, L[1]);
      L[2] = m2l_fma(-D[16], m, L[2]);
      L[3] = m2l_fma(-D[17], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[25], m, L[5]);
      L[6] = m2l_fma(D[26], m, L[6]);
      L[7] = m2l_fma(D[28], m, L[7]);
      L[8] = m2l_fma(D[29], m, L[8]);
    }
    { const T m = __ldg(Mr + 8);
      L[1] = m2l_fma(-D[14], m, L[1]);
      L[2] = m2l_fma(-D[17], m, L[2]);
      L[3] = m2l_fma(-D[18], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[29], m, L[7]);
      L[8] = m2l_fma(D[30], m, L[8]);
    }
    { const T m = __ldg(Mr + 9);
      L[1] = m2l_fma(-D[19], m, L[1]);
      L[2] = m2l_fma(-D[20], m, L[2]);
      L[3] = m2l_fma(-D[21], m, L[3]);
    }
    { const T m = __ldg(Mr + 10);
      L[1] = m2l_fma(-D[20], m, L[1]);
      L[2] = m2l_fma(-D[22], m, L[2]);
      L[3] = m2l_fma(-D[23], m, L[3]);
    }
    { const T m = __ldg(Mr + 11);
      L[1] = m2l_fma(-D[21], m, L[1]);
      L[2] = m2l_fma(-D[23], m, L[2]);
      L[3] = m2l_fma(-D[24], m, L[3]);
    }
    { const T m = __ldg(Mr + 12);
      L[1] = m2l_fma(-D[22], m, L[1]);
      L[2] = m2l_fma(-D[25], m, L[2]);
      L[3] = m2l_fma(-D[26], m, L[3]);
    }
    { const T m = __ldg(Mr + 13);
      L[1] = m2l_fma(-D[23], m, L[1]);
      L[2] = m2l_fma(-D[26], m, L[2]);
      L[3] = m2l_fma(-D[27], m, L[3]);
    }
    { const T m = __ldg(Mr + 14);
      L[1] = m2l_fma(-D[25], m, L[1]);
      L[2] = m2l_fma(-D[28], m, L[2]);
      L[3] = m2l_fma(-D[29], m, L[3]);
    }
    { const T m = __ldg(Mr + 15);
      L[1] = m2l_fma(-D[26], m, L[1]);
      L[2] = m2l_fma(-D[29], m, L[2]);
      L[3] = m2l_fma(-D[30], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_reduce_moments_h_4(const T *__restrict__ Ms, T *__restrict__ Mr)
{
    T v0 = Ms[0];
    T v1 = Ms[1];
    T v2 = Ms[2];
    T v3 = Ms[3];
    T v4 = Ms[4];
    T v5 = Ms[5];
    T v6 = Ms[6];
    T v7 = Ms[7];
    T v8 = Ms[8];
    T v9 = Ms[9];
    T v10 = Ms[10];
    T v11 = Ms[11];
    T v12 = Ms[12];
    T v13 = Ms[13];
    T v14 = Ms[14];
    T v15 = Ms[15];
    T v16 = Ms[16];
    T v17 = Ms[17];
    T v18 = Ms[18];
    T v19 = Ms[19];
    T v20 = Ms[20];
    T v21 = Ms[21];
    T v22 = Ms[22];
    T v23 = Ms[23];
    T v24 = Ms[24];
    T v25 = Ms[25];
    T v26 = Ms[26];
    T v27 = Ms[27];
    T v28 = Ms[28];
    T v29 = Ms[29];
    T v30 = Ms[30];
    T v31 = Ms[31];
    T v32 = Ms[32];
    T v33 = Ms[33];
    T v34 = Ms[34];
    v25 -= v34;
    v32 -= v34;
    v12 -= v19;
    v17 -= v19;
    v22 -= v29;
    v27 -= v29;
    v24 -= v33;
    v31 -= v33;
    v4 -= v9;
    v7 -= v9;
    v10 -= v15;
    v13 -= v15;
    v11 -= v18;
    v16 -= v18;
    v20 -= v25;
    v23 -= v25;
    v21 -= v28;
    v26 -= v28;
    v23 -= v32;
    v30 -= v32;
    Mr[0] = v0;
    Mr[1] = v1;
    Mr[2] = v2;
    Mr[3] = v3;
    Mr[4] = v4;
    Mr[5] = v5;
    Mr[6] = v6;
    Mr[7] = v7;
    Mr[8] = v8;
    Mr[9] = v10;
    Mr[10] = v11;
    Mr[11] = v12;
    Mr[12] = v13;
    Mr[13] = v14;
    Mr[14] = v16;
    Mr[15] = v17;
    Mr[16] = v20;
    Mr[17] = v21;
    Mr[18] = v22;
    Mr[19] = v23;
    Mr[20] = v24;
    Mr[21] = v26;
    Mr[22] = v27;
    Mr[23] = v30;
    Mr[24] = v31;
}

template <class T> __device__ __forceinline__ void m2l_complete_locals_h_4(const T *__restrict__ Lr, T *__restrict__ L)
{
    const T v0 = Lr[0];
    L[0] = v0;
    const T v1 = Lr[1];
    L[1] = v1;
    const T v2 = Lr[2];
    L[2] = v2;
    const T v3 = Lr[3];
    L[3] = v3;
    const T v4 = Lr[4];
    L[4] = v4;
    const T v5 = Lr[5];
    L[5] = v5;
    const T v6 = Lr[6];
    L[6] = v6;
    const T v7 = Lr[7];
    L[7] = v7;
    const T v8 = Lr[8];
    L[8] = v8;
    const T v9 = -v4 - v7;
    L[9] = v9;
    const T v10 = Lr[9];
    L[10] = v10;
    const T v11 = Lr[10];
    L[11] = v11;
    const T v12 = Lr[11];
    L[12] = v12;
    const T v13 = Lr[12];
    L[13] = v13;
    const T v14 = Lr[13];
    L[14] = v14;
    const T v15 = -v10 - v13;
    L[15] = v15;
    const T v16 = Lr[14];
    L[16] = v16;
    const T v17 = Lr[15];
    L[17] = v17;
    const T v18 = -v11 - v16;
    L[18] = v18;
    const T v19 = -v12 - v17;
    L[19] = v19;
    const T v20 = Lr[16];
    L[20] = v20;
    const T v21 = Lr[17];
    L[21] = v21;
    const T v22 = Lr[18];
    L[22] = v22;
    const T v23 = Lr[19];
    L[23] = v23;
    const T v24 = Lr[20];
    L[24] = v24;
    const T v25 = -v20 - v23;
    L[25] = v25;
    const T v26 = Lr[21];
    L[26] = v26;
    const T v27 = Lr[22];
    L[27] = v27;
    const T v28 = -v21 - v26;
    L[28] = v28;
    const T v29 = -v22 - v27;
    L[29] = v29;
    const T v30 = Lr[23];
    L[30] = v30;
    const T v31 = Lr[24];
    L[31] = v31;
    const T v32 = -v23 - v30;
    L[32] = v32;
    const T v33 = -v24 - v31;
    L[33] = v33;
    const T v34 = -v25 - v32;
    L[34] = v34;
}

template <class T> __device__ __forceinline__ void m2l_dtensor_h_5(T dx, T dy, T dz, T (&D)[46])
{
    const T s2 = m2l_fma(dx, dx, m2l_fma(dy, dy, dz * dz));
    const T si = m2l_rsqrt(s2);
    const T si2 = si * si;
    const T f0 = -si;
    const T f1 = T(-1) * f0 * si2;
    const T f2 = T(-3) * f1 * si2;
    const T f3 = T(-5) * f2 * si2;
    const T f4 = T(-7) * f3 * si2;
    const T f5 = T(-9) * f4 * si2;
    const T r_0_0 = f0;
    const T r_1_0 = f1;
    const T r_2_0 = f2;
    const T r_3_0 = f3;
    const T r_4_0 = f4;
    const T r_5_0 = f5;
    const T r_0_1 = dx * r_1_0;
    const T r_1_1 = dx * r_2_0;
    const T r_2_1 = dx * r_3_0;
    const T r_3_1 = dx * r_4_0;
    const T r_4_1 = dx * r_5_0;
    const T r_0_2 = dy * r_1_0;
    const T r_1_2 = dy * r_2_0;
    const T r_2_2 = dy * r_3_0;
    const T r_3_2 = dy * r_4_0;
    const T r_4_2 = dy * r_5_0;
    const T r_0_4 = m2l_fma(T(1), r_1_0, dx * r_1_1);
    const T r_1_4 = m2l_fma(T(1), r_2_0, dx * r_2_1);
    const T r_2_4 = m2l_fma(T(1), r_3_0, dx * r_3_1);
    const T r_3_4 = m2l_fma(T(1), r_4_0, dx * r_4_1);
    const T r_0_5 = dx * r_1_2;
    const T r_1_5 = dx * r_2_2;
    const T r_2_5 = dx * r_3_2;
    const T r_3_5 = dx * r_4_2;
    const T r_0_7 = m2l_fma(T(1), r_1_0, dy * r_1_2);
    const T r_1_7 = m2l_fma(T(1), r_2_0, dy * r_2_2);
    const T r_2_7 = m2l_fma(T(1), r_3_0, dy * r_3_2);
    const T r_3_7 = m2l_fma(T(1), r_4_0, dy * r_4_2);
    const T r_0_10 = m2l_fma(T(2), r_1_1, dx * r_1_4);
    const T r_1_10 = m2l_fma(T(2), r_2_1, dx * r_2_4);
    const T r_2_10 = m2l_fma(T(2), r_3_1, dx * r_3_4);
    const T r_0_11 = m2l_fma(T(1), r_1_2, dx * r_1_5);
    const T r_1_11 = m2l_fma(T(1), r_2_2, dx * r_2_5);
    const T r_2_11 = m2l_fma(T(1), r_3_2, dx * r_3_5);
    const T r_0_13 = dx * r_1_7;
    const T r_1_13 = dx * r_2_7;
    const T r_2_13 = dx * r_3_7;
    const T r_0_16 = m2l_fma(T(2), r_1_2, dy * r_1_7);
    const T r_1_16 = m2l_fma(T(2), r_2_2, dy * r_2_7);
    const T r_2_16 = m2l_fma(T(2), r_3_2, dy * r_3_7);
    const T r_0_20 = m2l_fma(T(3), r_1_4, dx * r_1_10);
    const T r_1_20 = m2l_fma(T(3), r_2_4, dx * r_2_10);
    const T r_0_21 = m2l_fma(T(2), r_1_5, dx * r_1_11);
    const T r_1_21 = m2l_fma(T(2), r_2_5, dx * r_2_11);
    const T r_0_23 = m2l_fma(T(1), r_1_7, dx * r_1_13);
    const T r_1_23 = m2l_fma(T(1), r_2_7, dx * r_2_13);
    const T r_0_26 = dx * r_1_16;
    const T r_1_26 = dx * r_2_16;
    const T r_0_30 = m2l_fma(T(3), r_1_7, dy * r_1_16);
    const T r_1_30 = m2l_fma(T(3), r_2_7, dy * r_2_16);
    const T r_0_35 = m2l_fma(T(4), r_1_10, dx * r_1_20);
    const T r_0_36 = m2l_fma(T(3), r_1_11, dx * r_1_21);
    const T r_0_38 = m2l_fma(T(2), r_1_13, dx * r_1_23);
    const T r_0_41 = m2l_fma(T(1), r_1_16, dx * r_1_26);
    const T r_0_45 = dx * r_1_30;
    const T r_0_50 = m2l_fma(T(4), r_1_16, dy * r_1_30);
    D[0] = r_0_0;
    D[1] = r_0_1;
    D[2] = r_0_2;
    D[3] = dz * r_1_0;
    D[4] = r_0_4;
    D[5] = r_0_5;
    D[6] = dz * r_1_1;
    D[7] = r_0_7;
    D[8] = dz * r_1_2;
    D[10] = r_0_10;
    D[11] = r_0_11;
    D[12] = dz * r_1_4;
    D[13] = r_0_13;
    D[14] = dz * r_1_5;
    D[16] = r_0_16;
    D[17] = dz * r_1_7;
    D[19] = r_0_20;
    D[20] = r_0_21;
    D[21] = dz * r_1_10;
    D[22] = r_0_23;
    D[23] = dz * r_1_11;
    D[25] = r_0_26;
    D[26] = dz * r_1_13;
    D[28] = r_0_30;
    D[29] = dz * r_1_16;
    D[31] = r_0_35;
    D[32] = r_0_36;
    D[33] = dz * r_1_20;
    D[34] = r_0_38;
    D[35] = dz * r_1_21;
    D[37] = r_0_41;
    D[38] = dz * r_1_23;
    D[40] = r_0_45;
    D[41] = dz * r_1_26;
    D[43] = r_0_50;
    D[44] = dz * r_1_30;
    D[9] = -D[4] - D[7];
    D[15] = -D[10] - D[13];
    D[18] = -D[11] - D[16];
    D[24] = -D[19] - D[22];
    D[27] = -D[20] - D[25];
    D[30] = -D[22] - D[28];
    D[36] = -D[31] - D[34];
    D[39] = -D[32] - D[37];
    D[42] = -D[34] - D[40];
    D[45] = -D[37] - D[43];
}

template <class T> __device__ __forceinline__ void m2l_side_a_h_5(const T (&D)[46], const T *__restrict__ Mr, T rho, T (&L)[36])
{
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[0] = D[0] * m;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[10] * m;
      L[10] = D[11] * m;
      L[11] = D[12] * m;
      L[12] = D[13] * m;
      L[13] = D[14] * m;
      L[14] = D[16] * m;
      L[15] = D[17] * m;
      L[16] = D[19] * m;
      L[17] = D[20] * m;
      L[18] = D[21] * m;
      L[19] = D[22] * m;
      L[20] = D[23] * m;
      L[21] = D[25] * m;
      L[22] = D[26] * m;
      L[23] = D[28] * m;
      L[24] = D[29] * m;
      L[25] = D[31] * m;
      L[26] = D[32] * m;
      L[27] = D[33] * m;
      L[28] = D[34] * m;
      L[29] = D[35] * m;
      L[30] = D[37] * m;
      L[31] = D[38] * m;
      L[32] = D[40] * m;
      L[33] = D[41] * m;
      L[34] = D[43] * m;
      L[35] = D[44] * m;
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 1) * rp;
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(D[20], m, L[10]);
      L[11] = m2l_fma(D[21], m, L[11]);
      L[12] = m2l_fma(D[22], m, L[12]);
      L[13] = m2l_fma(D[23], m, L[13]);
      L[14] = m2l_fma(D[25], m, L[14]);
      L[15] = m2l_fma(D[26], m, L[15]);
      L[16] = m2l_fma(D[31], m, L[16]);
      L[17] = m2l_fma(D[32], m, L[17]);
      L[18] = m2l_fma(D[33], m, L[18]);
      L[19] = m2l_fma(D[34], m, L[19]);
      L[20] = m2l_fma(D[35], m, L[20]);
      L[21] = m2l_fma(D[37], m, L[21]);
      L[22] = m2l_fma(D[38], m, L[22]);
      L[23] = m2l_fma(D[40], m, L[23]);
      L[24] = m2l_fma(D[41], m, L[24]);
    }
    { const T m = -__ldg(Mr + 2) * rp;
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[20], m, L[9]);
      L[10] = m2l_fma(D[22], m, L[10]);
      L[11] = m2l_fma(D[23], m, L[11]);
      L[12] = m2l_fma(D[25], m, L[12]);
      L[13] = m2l_fma(D[26], m, L[13]);
      L[14] = m2l_fma(D[28], m, L[14]);
      L[15] = m2l_fma(D[29], m, L[15]);
      L[16] = m2l_fma(D[32], m, L[16]);
      L[17] = m2l_fma(D[34], m, L[17]);
      L[18] = m2l_fma(D[35], m, L[18]);
      L[19] = m2l_fma(D[37], m, L[19]);
      L[20] = m2l_fma(D[38], m, L[20]);
      L[21] = m2l_fma(D[40], m, L[21]);
      L[22] = m2l_fma(D[41], m, L[22]);
      L[23] = m2l_fma(D[43], m, L[23]);
      L[24] = m2l_fma(D[44], m, L[24]);
    }
    { const T m = -__ldg(Mr + 3) * rp;
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[21], m, L[9]);
      L[10] = m2l_fma(D[23], m, L[10]);
      L[11] = m2l_fma(D[24], m, L[11]);
      L[12] = m2l_fma(D[26], m, L[12]);
      L[13] = m2l_fma(D[27], m, L[13]);
      L[14] = m2l_fma(D[29], m, L[14]);
      L[15] = m2l_fma(D[30], m, L[15]);
      L[16] = m2l_fma(D[33], m, L[16]);
      L[17] = m2l_fma(D[35], m, L[17]);
      L[18] = m2l_fma(D[36], m, L[18]);
      L[19] = m2l_fma(D[38], m, L[19]);
      L[20] = m2l_fma(D[39], m, L[20]);
      L[21] = m2l_fma(D[41], m, L[21]);
      L[22] = m2l_fma(D[42], m, L[22]);
      L[23] = m2l_fma(D[44], m, L[23]);
      L[24] = m2l_fma(D[45], m, L[24]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 4) * rp;
      L[0] = m2l_fma(D[4], m, L[0]);
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
      L[4] = m2l_fma(D[19], m, L[4]);
      L[5] = m2l_fma(D[20], m, L[5]);
      L[6] = m2l_fma(D[21], m, L[6]);
      L[7] = m2l_fma(D[22], m, L[7]);
      L[8] = m2l_fma(D[23], m, L[8]);
      L[9] = m2l_fma(D[31], m, L[9]);
      L[10] = m2l_fma(D[32], m, L[10]);
      L[11] = m2l_fma(D[33], m, L[11]);
      L[12] = m2l_fma(D[34], m, L[12]);
      L[13] = m2l_fma(D[35], m, L[13]);
      L[14] = m2l_fma(D[37], m, L[14]);
      L[15] = m2l_fma(D[38], m, L[15]);
    }
    { const T m = __ldg(Mr + 5) * rp;
      L[0] = m2l_fma(D[5], m, L[0]);
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[22], m, L[5]);
      L[6] = m2l_fma(D[23], m, L[6]);
      L[7] = m2l_fma(D[25], m, L[7]);
      L[8] = m2l_fma(D[26], m, L[8]);
      L[9] = m2l_fma(D[32], m, L[9]);
      L[10] = m2l_fma(D[34], m, L[10]);
      L[11] = m2l_fma(D[35], m, L[11]);
      L[12] = m2l_fma(D[37], m, L[12]);
      L[13] = m2l_fma(D[38], m, L[13]);
      L[14] = m2l_fma(D[40], m, L[14]);
      L[15] = m2l_fma(D[41], m, L[15]);
    }
    { const T m = __ldg(Mr + 6) * rp;
      L[0] = m2l_fma(D[6], m, L[0]);
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(D[33], m, L[9]);
      L[10] = m2l_fma(D[35], m, L[10]);
      L[11] = m2l_fma(D[36], m, L[11]);
      L[12] = m2l_fma(D[38], m, L[12]);
      L[13] = m2l_fma(D[39], m, L[13]);
      L[14] = m2l_fma(D[41], m, L[14]);
      L[15] = m2l_fma(D[42], m, L[15]);
    }
    { const T m = __ldg(Mr + 7) * rp;
      L[0] = m2l_fma(D[7], m, L[0]);
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[25], m, L[5]);
      L[6] = m2l_fma(D[26], m, L[6]);
      L[7] = m2l_fma(D[28], m, L[7]);
      L[8] = m2l_fma(D[29], m, L[8]);
      L[9] = m2l_fma(D[34], m, L[9]);
      L[10] = m2l_fma(D[37], m, L[10]);
      L[11] = m2l_fma(D[38], m, L[11]);
      L[12] = m2l_fma(D[40], m, L[12]);
      L[13] = m2l_fma(D[41], m, L[13]);
      L[14] = m2l_fma(D[43], m, L[14]);
      L[15] = m2l_fma(D[44], m, L[15]);
    }
    { const T m = __ldg(Mr + 8) * rp;
      L[0] = m2l_fma(D[8], m, L[0]);
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[29], m, L[7]);
      L[8] = m2l_fma(D[30], m, L[8]);
      L[9] = m2l_fma(D[35], m, L[9]);
      L[10] = m2l_fma(D[38], m, L[10]);
      L[11] = m2l_fma(D[39], m, L[11]);
      L[12] = m2l_fma(D[41], m, L[12]);
      L[13] = m2l_fma(D[42], m, L[13]);
      L[14] = m2l_fma(D[44], m, L[14]);
      L[15] = m2l_fma(D[45], m, L[15]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 9) * rp;
      L[0] = m2l_fma(D[10], m, L[0]);
      L[1] = m2l_fma(D[19], m, L[1]);
      L[2] = m2l_fma(D[20], m, L[2]);
      L[3] = m2l_fma(D[21], m, L[3]);
      L[4] = m2l_fma(D[31], m, L[4]);
      L[5] = m2l_fma(D[32], m, L[5]);
      L[6] = m2l_fma(D[33], m, L[6]);
      L[7] = m2l_fma(D[34], m, L[7]);
      L[8] = m2l_fma(D[35], m, L[8]);
    }
    { const T m = -__ldg(Mr + 10) * rp;
      L[0] = m2l_fma(D[11], m, L[0]);
      L[1] = m2l_fma(D[20], m, L[1]);
      L[2] = m2l_fma(D[22], m, L[2]);
      L[3] = m2l_fma(D[23], m, L[3]);
      L[4] = m2l_fma(D[32], m, L[4]);
      L[5] = m2l_fma(D[34], m, L[5]);
      L[6] = m2l_fma(D[35], m, L[6]);
      L[7] = m2l_fma(D[37], m, L[7]);
      L[8] = m2l_fma(D[38], m, L[8]);
    }
    { const T m = -__ldg(Mr + 11) * rp;
      L[0] = m2l_fma(D[12], m, L[0]);
      L[1] = m2l_fma(D[21], m, L[1]);
      L[2] = m2l_fma(D[23], m, L[2]);
      L[3] = m2l_fma(D[24], m, L[3]);
      L[4] = m2l_fma(D[33], m, L[4]);
      L[5] = m2l_fma(D[35], m, L[5]);
      L[6] = m2l_fma(D[36], m, L[6]);
      L[7] = m2l_fma(D[38], m, L[7]);
      L[8] = m2l_fma(D[39], m, L[8]);
    }
    { const T m = -__ldg(Mr + 12) * rp;
      L[0] = m2l_fma(D[13], m, L[0]);
      L[1] = m2l_fma(D[22], m, L[1]);
      L[2] = m2l_fma(D[25], m, L[2]);
      L[3] = m2l_fma(D[26], m, L[3]);
      L[4] = m2l_fma(D[34], m, L[4]);
      L[5] = m2l_fma(D[37], m, L[5]);
      L[6] = m2l_fma(D[38], m, L[6]);
      L[7] = m2l_fma(D[40], m, L[7]);
      L[8] = m2l_fma(D[41], m, L[8]);
    }
    { const T m = -__ldg(Mr + 13) * rp;
      L[0] = m2l_fma(D[14], m, L[0]);
      L[1] = m2l_fma(D[23], m, L[1]);
      L[2] = m2l_fma(D[26], m, L[2]);
      L[3] = m2l_fma(D[27], m, L[3]);
      L[4] = m2l_fma(D[35], m, L[4]);
      L[5] = m2l_fma(D[38], m, L[5]);
      L[6] = m2l_fma(D[39], m, L[6]);
      L[7] = m2l_fma(D[41], m, L[7]);
      L[8] = m2l_fma(D[42], m, L[8]);
    }
    { const T m = -__ldg(Mr + 14) * rp;
      L[0] = m2l_fma(D[16], m, L[0]);
      L[1] = m2l_fma(D[25], m, L[1]);
      L[2] = m2l_fma(D[28], m, L[2]);
      L[3] = m2l_fma(D[29], m, L[3]);
      L[4] = m2l_fma(D[37], m, L[4]);
      L[5] = m2l_fma(D[40], m, L[5]);
      L[6] = m2l_fma(D[41], m, L[6]);
      L[7] = m2l_fma(D[43], m, L[7]);
      L[8] = m2l_fma(D[44], m, L[8]);
    }
    { const T m = -__ldg(Mr + 15) * rp;
      L[0] = m2l_fma(D[17], m, L[0]);
      L[1] = m2l_fma(D[26], m, L[1]);
      L[2] = m2l_fma(D[29], m, L[2]);
      L[3] = m2l_fma(D[30], m, L[3]);
      L[4] = m2l_fma(D[38], m, L[4]);
      L[5] = m2l_fma(D[41], m, L[5]);
      L[6] = m2l_fma(D[42], m, L[6]);
      L[7] = m2l_fma(D[44], m, L[7]);
      L[8] = m2l_fma(D[45], m, L[8]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 16) * rp;
      L[0] = m2l_fma(D[19], m, L[0]);
      L[1] = m2l_fma(D[31], m, L[1]);
      L[2] = m2l_fma(D[32], m, L[2]);
      L[3] = m2l_fma(D[33], m, L[3]);
    }
    { const T m = __ldg(Mr + 17) * rp;
      L[0] = m2l_fma(D[20], m, L[0]);
      L[1] = m2l_fma(D[32], m, L[1]);
      L[2] = m2l_fma(D[34], m, L[2]);
      L[3] = m2l_fma(D[35], m, L[3]);
    }
    { const T m = __ldg(Mr + 18) * rp;
      L[0] = m2l_fma(D[21], m, L[0]);
      L[1] = m2l_fma(D[33], m, L[1]);
      L[2] = m2l_fma(D[35], m, L[2]);
      L[3] = m2l_fma(D[36], m, L[3]);
    }
    { const T m = __ldg(Mr + 19) * rp;
      L[0] = m2l_fma(D[22], m, L[0]);
      L[1] = m2l_fma(D[34], m, L[1]);
      L[2] = m2l_fma(D[37], m, L[2]);
      L[3] = m2l_fma(D[38], m, L[3]);
    }
    { const T m = __ldg(Mr + 20) * rp;
      L[0] = m2l_fma(D[23], m, L[0]);
      L[1] = m2l_fma(D[35], m, L[1]);
      L[2] = m2l_fma(D[38], m, L[2]);
      L[3] = m2l_fma(D[39], m, L[3]);
    }
    { const T m = __ldg(Mr + 21) * rp;
      L[0] = m2l_fma(D[25], m, L[0]);
      L[1] = m2l_fma(D[37], m, L[1]);
      L[2] = m2l_fma(D[40], m, L[2]);
      L[3] = m2l_fma(D[41], m, L[3]);
    }
    { const T m = __ldg(Mr + 22) * rp;
      L[0] = m2l_fma(D[26], m, L[0]);
      L[1] = m2l_fma(D[38], m, L[1]);
      L[2] = m2l_fma(D[41], m, L[2]);
      L[3] = m2l_fma(D[42], m, L[3]);
    }
    { const T m = __ldg(Mr + 23) * rp;
      L[0] = m2l_fma(D[28], m, L[0]);
      L[1] = m2l_fma(D[40], m, L[1]);
      L[2] = m2l_fma(D[43], m, L[2]);
      L[3] = m2l_fma(D[44], m, L[3]);
    }
    { const T m = __ldg(Mr + 24) * rp;
      L[0] = m2l_fma(D[29], m, L[0]);
      L[1] = m2l_fma(D[41], m, L[1]);
      L[2] = m2l_fma(D[44], m, L[2]);
      L[3] = m2l_fma(D[45], m, L[3]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 25) * rp;
      L[0] = m2l_fma(D[31], m, L[0]);
    }
    { const T m = -__ldg(Mr + 26) * rp;
      L[0] = m2l_fma(D[32], m, L[0]);
    }
    { const T m = -__ldg(Mr + 27) * rp;
      L[0] = m2l_fma(D[33], m, L[0]);
    }
    { const T m = -__ldg(Mr + 28) * rp;
      L[0] = m2l_fma(D[34], m, L[0]);
    }
    { const T m = -__ldg(Mr + 29) * rp;
      L[0] = m2l_fma(D[35], m, L[0]);
    }
    { const T m = -__ldg(Mr + 30) * rp;
      L[0] = m2l_fma(D[37], m, L[0]);
    }
    { const T m = -__ldg(Mr + 31) * rp;
      L[0] = m2l_fma(D[38], m, L[0]);
    }
    { const T m = -__ldg(Mr + 32) * rp;
      L[0] = m2l_fma(D[40], m, L[0]);
    }
    { const T m = -__ldg(Mr + 33) * rp;
      L[0] = m2l_fma(D[41], m, L[0]);
    }
    { const T m = -__ldg(Mr + 34) * rp;
      L[0] = m2l_fma(D[43], m, L[0]);
    }
    { const T m = -__ldg(Mr + 35) * rp;
      L[0] = m2l_fma(D[44], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_acc_h_5(const T (&D)[46], const T *__restrict__ Mr, T rho, T (&L)[36])
{
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[0] = m2l_fma(D[0], m, L[0]);
      L[1] = m2l_fma(D[1], m, L[1]);
      L[2] = m2l_fma(D[2], m, L[2]);
      L[3] = m2l_fma(D[3], m, L[3]);
      L[4] = m2l_fma(D[4], m, L[4]);
      L[5] = m2l_fma(D[5], m, L[5]);
      L[6] = m2l_fma(D[6], m, L[6]);
      L[7] = m2l_fma(D[7], m, L[7]);
      L[8] = m2l_fma(D[8], m, L[8]);
      L[9] = m2l_fma(D[10], m, L[9]);
      L[10] = m2l_fma(D[11], m, L[10]);
      L[11] = m2l_fma(D[12], m, L[11]);
      L[12] = m2l_fma(D[13], m, L[12]);
      L[13] = m2l_fma(D[14], m, L[13]);
      L[14] = m2l_fma(D[16], m, L[14]);
      L[15] = m2l_fma(D[17], m, L[15]);
      L[16] = m2l_fma(D[19], m, L[16]);
      L[17] = m2l_fma(D[20], m, L[17]);
      L[18] = m2l_fma(D[21], m, L[18]);
      L[19] = m2l_fma(D[22], m, L[19]);
      L[20] = m2l_fma(D[23], m, L[20]);
      L[21] = m2l_fma(D[25], m, L[21]);
      L[22] = m2l_fma(D[26], m, L[22]);
      L[23] = m2l_fma(D[28], m, L[23]);
      L[24] = m2l_fma(D[29], m, L[24]);
      L[25] = m2l_fma(D[31], m, L[25]);
      L[26] = m2l_fma(D[32], m, L[26]);
      L[27] = m2l_fma(D[33], m, L[27]);
      L[28] = m2l_fma(D[34], m, L[28]);
      L[29] = m2l_fma(D[35], m, L[29]);
      L[30] = m2l_fma(D[37], m, L[30]);
      L[31] = m2l_fma(D[38], m, L[31]);
      L[32] = m2l_fma(D[40], m, L[32]);
      L[33] = m2l_fma(D[41], m, L[33]);
      L[34] = m2l_fma(D[43], m, L[34]);
      L[35] = m2l_fma(D[44], m, L[35]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 1) * rp;
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(D[20], m, L[10]);
      L[11] = m2l_fma(D[21], m, L[11]);
      L[12] = m2l_fma(D[22], m, L[12]);
      L[13] = m2l_fma(D[23], m, L[13]);
      L[14] = m2l_fma(D[25], m, L[14]);
      L[15] = m2l_fma(D[26], m, L[15]);
      L[16] = m2l_fma(D[31], m, L[16]);
      L[17] = m2l_fma(D[32], m, L[17]);
      L[18] = m2l_fma(D[33], m, L[18]);
      L[19] = m2l_fma(D[34], m, L[19]);
      L[20] = m2l_fma(D[35], m, L[20]);
      L[21] = m2l_fma(D[37], m, L[21]);
      L[22] = m2l_fma(D[38], m, L[22]);
      L[23] = m2l_fma(D[40], m, L[23]);
      L[24] = m2l_fma(D[41], m, L[24]);
    }
    { const T m = -__ldg(Mr + 2) * rp;
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[20], m, L[9]);
      L[10] = m2l_fma(D[22], m, L[10]);
      L[11] = m2l_fma(D[23], m, L[11]);
      L[12] = m2l_fma(D[25], m, L[12]);
      L[13] = m2l_fma(D[26], m, L[13]);
      L[14] = m2l_fma(D[28], m, L[14]);
      L[15] = m2l_fma(D[29], m, L[15]);
      L[16] = m2l_fma(D[32], m, L[16]);
      L[17] = m2l_fma(D[34], m, L[17]);
      L[18] = m2l_fma(D[35], m, L[18]);
      L[19] = m2l_fma(D[37], m, L[19]);
      L[20] = m2l_fma(D[38], m, L[20]);
      L[21] = m2l_fma(D[40], m, L[21]);
      L[22] = m2l_fma(D[41], m, L[22]);
      L[23] = m2l_fma(D[43], m, L[23]);
      L[24] = m2l_fma(D[44], m, L[24]);
    }
    { const T m = -__ldg(Mr + 3) * rp;
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[21], m, L[9]);
      L[10] = m2l_fma(D[23], m, L[10]);
      L[11] = m2l_fma(D[24], m, L[11]);
      L[12] = m2l_fma(D[26], m, L[12]);
      L[13] = m2l_fma(D[27], m, L[13]);
      L[14] = m2l_fma(D[29], m, L[14]);
      L[15] = m2l_fma(D[30], m, L[15]);
      L[16] = m2l_fma(D[33], m, L[16]);
      L[17] = m2l_fma(D[35], m, L[17]);
      L[18] = m2l_fma(D[36], m, L[18]);
      L[19] = m2l_fma(D[38], m, L[19]);
      L[20] = m2l_fma(D[39], m, L[20]);
      L[21] = m2l_fma(D[41], m, L[21]);
      L[22] = m2l_fma(D[42], m, L[22]);
      L[23] = m2l_fma(D[44], m, L[23]);
      L[24] = m2l_fma(D[45], m, L[24]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 4) * rp;
      L[0] = m2l_fma(D[4], m, L[0]);
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
      L[4] = m2l_fma(D[19], m, L[4]);
      L[5] = m2l_fma(D[20], m, L[5]);
      L[6] = m2l_fma(D[21], m, L[6]);
      L[7] = m2l_fma(D[22], m, L[7]);
      L[8] = m2l_fma(D[23], m, L[8]);
      L[9] = m2l_fma(D[31], m, L[9]);
      L[10] = m2l_fma(D[32], m, L[10]);
      L[11] = m2l_fma(D[33], m, L[11]);
      L[12] = m2l_fma(D[34], m, L[12]);
      L[13] = m2l_fma(D[35], m, L[13]);
      L[14] = m2l_fma(D[37], m, L[14]);
      L[15] = m2l_fma(D[38], m, L[15]);
    }
    { const T m = __ldg(Mr + 5) * rp;
      L[0] = m2l_fma(D[5], m, L[0]);
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[22], m, L[5]);
      L[6] = m2l_fma(D[23], m, L[6]);
      L[7] = m2l_fma(D[25], m, L[7]);
      L[8] = m2l_fma(D[26], m, L[8]);
      L[9] = m2l_fma(D[32], m, L[9]);
      L[10] = m2l_fma(D[34], m, L[10]);
      L[11] = m2l_fma(D[35], m, L[11]);
      L[12] = m2l_fma(D[37], m, L[12]);
      L[13] = m2l_fma(D[38], m, L[13]);
      L[14] = m2l_fma(D[40], m, L[14]);
      L[15] = m2l_fma(D[41], m, L[15]);
    }
    { const T m = __ldg(Mr + 6) * rp;
      L[0] = m2l_fma(D[6], m, L[0]);
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(D[33], m, L[9]);
      L[10] = m2l_fma(D[35], m, L[10]);
      L[11] = m2l_fma(D[36], m, L[11]);
      L[12] = m2l_fma(D[38], m, L[12]);
      L[13] = m2l_fma(D[39], m, L[13]);
      L[14] = m2l_fma(D[41], m, L[14]);
      L[15] = m2l_fma(D[42], m, L[15]);
    }
    { const T m = __ldg(Mr + 7) * rp;
      L[0] = m2l_fma(D[7], m, L[0]);
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[25], m, L[5]);
      L[6] = m2l_fma(D[26], m, L[6]);
      L[7] = m2l_fma(D[28], m, L[7]);
      L[8] = m2l_fma(D[29], m, L[8]);
      L[9] = m2l_fma(D[34], m, L[9]);
      L[10] = m2l_fma(D[37], m, L[10]);
      L[11] = m2l_fma(D[38], m, L[11]);
      L[12] = m2l_fma(D[40], m, L[12]);
      L[13] = m2l_fma(D[41], m, L[13]);
      L[14] = m2l_fma(D[43], m, L[14]);
      L[15] = m2l_fma(D[44], m, L[15]);
    }
    { const T m = __ldg(Mr + 8) * rp;
      L[0] = m2l_fma(D[8], m, L[0]);
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[29], m, L[7]);
      L[8] = m2l_fma(D[30], m, L[8]);
      L[9] = m2l_fma(D[35], m, L[9]);
      L[10] = m2l_fma(D[38], m, L[10]);
      L[11] = m2l_fma(D[39], m, L[11]);
      L[12] = m2l_fma(D[41], m, L[12]);
      L[13] = m2l_fma(D[42], m, L[13]);
      L[14] = m2l_fma(D[44], m, L[14]);
      L[15] = m2l_fma(D[45], m, L[15]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 9) * rp;
      L[0] = m2l_fma(D[10], m, L[0]);
      L[1] = m2l_fma(D[19], m, L[1]);
      L[2] = m2l_fma(D[20], m, L[2]);
      L[3] = m2l_fma(D[21], m, L[3]);
      L[4] = m2l_fma(D[31], m, L[4]);
      L[5] = m2l_fma(D[32], m, L[5]);
      L[6] = m2l_fma(D[33], m, L[6]);
      L[7] = m2l_fma(D[34], m, L[7]);
      L[8] = m2l_fma(D[35], m, L[8]);
    }
    { const T m = -__ldg(Mr + 10) * rp;
      L[0] = m2l_fma(D[11], m, L[0]);
      L[1] = m2l_fma(D[20], m, L[1]);
      L[2] = m2l_fma(D[22], m, L[2]);
      L[3] = m2l_fma(D[23], m, L[3]);
      L[4] = m2l_fma(D[32], m, L[4]);
      L[5] = m2l_fma(D[34], m, L[5]);
      L[6] = m2l_fma(D[35], m, L[6]);
      L[7] = m2l_fma(D[37], m, L[7]);
      L[8] = m2l_fma(D[38], m, L[8]);
    }
    { const T m = -__ldg(Mr + 11) * rp;
      L[0] = m2l_fma(D[12], m, L[0]);
      L[1] = m2l_fma(D[21], m, L[1]);
      L[2] = m2l_fma(D[23], m, L[2]);
      L[3] = m2l_fma(D[24], m, L[3]);
      L[4] = m2l_fma(D[33], m, L[4]);
      L[5] = m2l_fma(D[35], m, L[5]);
      L[6] = m2l_fma(D[36], m, L[6]);
      L[7] = m2l_fma(D[38], m, L[7]);
      L[8] = m2l_fma(D[39], m, L[8]);
    }
    { const T m = -__ldg(Mr + 12) * rp;
      L[0] = m2l_fma(D[13], m, L[0]);
      L[1] = m2l_fma(D[22], m, L[1]);
      L[2] = m2l_fma(D[25], m, L[2]);
      L[3] = m2l_fma(D[26], m, L[3]);
      L[4] = m2l_fma(D[34], m, L[4]);
      L[5] = m2l_fma(D[37], m, L[5]);
      L[6] = m2l_fma(D[38], m, L[6]);
      L[7] = m2l_fma(D[40], m, L[7]);
      L[8] = m2l_fma(D[41], m, L[8]);
    }
    { const T m = -__ldg(Mr + 13) * rp;
      L[0] = m2l_fma(D[14], m, L[0]);
      L[1] = m2l_fma(D[23], m, L[1]);
      L[2] = m2l_fma(D[26], m, L[2]);
      L[3] = m2l_fma(D[27], m, L[3]);
      L[4] = m2l_fma(D[35], m, L[4]);
      L[5] = m2l_fma(D[38], m, L[5]);
      L[6] = m2l_fma(D[39], m, L[6]);
      L[7] = m2l_fma(D[41], m, L[7]);
      L[8] = m2l_fma(D[42], m, L[8]);
    }
    { const T m = -__ldg(Mr + 14) * rp;
      L[0] = m2l_fma(D[16], m, L[0]);
      L[1] = m2l_fma(D[25], m, L[1]);
      L[2] = m2l_fma(D[28], m, L[2]);
      L[3] = m2l_fma(D[29], m, L[3]);
      L[4] = m2l_fma(D[37], m, L[4]);
      L[5] = m2l_fma(D[40], m, L[5]);
      L[6] = m2l_fma(D[41], m, L[6]);
      L[7] = m2l_fma(D[43], m, L[7]);
      L[8] = m2l_fma(D[44], m, L[8]);
    }
    { const T m = -__ldg(Mr + 15) * rp;
      L[0] = m2l_fma(D[17], m, L[0]);
      L[1] = m2l_fma(D[26], m, L[1]);
      L[2] = m2l_fma(D[29], m, L[2]);
      L[3] = m2l_fma(D[30], m, L[3]);
      L[4] = m2l_fma(D[38], m, L[4]);
      L[5] = m2l_fma(D[41], m, L[5]);
      L[6] = m2l_fma(D[42], m, L[6]);
      L[7] = m2l_fma(D[44], m, L[7]);
      L[8] = m2l_fma(D[45], m, L[8]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 16) * rp;
      L[0] = m2l_fma(D[19], m, L[0]);
      L[1] = m2l_fma(D[31], m, L[1]);
      L[2] = m2l_fma(D[32], m, L[2]);
      L[3] = m2l_fma(D[33], m, L[3]);
    }
    { const T m = __ldg(Mr + 17) * rp;
      L[0] = m2l_fma(D[20], m, L[0]);
      L[1] = m2l_fma(D[32], m, L[1]);
      L[2] = m2l_fma(D[34], m, L[2]);
      L[3] = m2l_fma(D[35], m, L[3]);
    }
    { const T m = __ldg(Mr + 18) * rp;
      L[0] = m2l_fma(D[21], m, L[0]);
      L[1] = m2l_fma(D[33], m, L[1]);
      L[2] = m2l_fma(D[35], m, L[2]);
      L[3] = m2l_fma(D[36], m, L[3]);
    }
    { const T m = __ldg(Mr + 19) * rp;
      L[0] = m2l_fma(D[22], m, L[0]);
      L[1] = m2l_fma(D[34], m, L[1]);
      L[2] = m2l_fma(D[37], m, L[2]);
      L[3] = m2l_fma(D[38], m, L[3]);
    }
    { const T m = __ldg(Mr + 20) * rp;
      L[0] = m2l_fma(D[23], m, L[0]);
      L[1] = m2l_fma(D[35], m, L[1]);
      L[2] = m2l_fma(D[38], m, L[2]);
      L[3] = m2l_fma(D[39], m, L[3]);
    }
    { const T m = __ldg(Mr + 21) * rp;
      L[0] = m2l_fma(D[25], m, L[0]);
      L[1] = m2l_fma(D[37], m, L[1]);
      L[2] = m2l_fma(D[40], m, L[2]);
      L[3] = m2l_fma(D[41], m, L[3]);
    }
    { const T m = __ldg(Mr + 22) * rp;
      L[0] = m2l_fma(D[26], m, L[0]);
      L[1] = m2l_fma(D[38], m, L[1]);
      L[2] = m2l_fma(D[41], m, L[2]);
      L[3] = m2l_fma(D[42], m, L[3]);
    }
    { const T m = __ldg(Mr + 23) * rp;
      L[0] = m2l_fma(D[28], m, L[0]);
      L[1] = m2l_fma(D[40], m, L[1]);
      L[2] = m2l_fma(D[43], m, L[2]);
      L[3] = m2l_fma(D[44], m, L[3]);
    }
    { const T m = __ldg(Mr + 24) * rp;
      L[0] = m2l_fma(D[29], m, L[0]);
      L[1] = m2l_fma(D[41], m, L[1]);
      L[2] = m2l_fma(D[44], m, L[2]);
      L[3] = m2l_fma(D[45], m, L[3]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 25) * rp;
      L[0] = m2l_fma(D[31], m, L[0]);
    }
    { const T m = -__ldg(Mr + 26) * rp;
      L[0] = m2l_fma(D[32], m, L[0]);
    }
    { const T m = -__ldg(Mr + 27) * rp;
      L[0] = m2l_fma(D[33], m, L[0]);
    }
    { const T m = -__ldg(Mr + 28) * rp;
      L[0] = m2l_fma(D[34], m, L[0]);
    }
    { const T m = -__ldg(Mr + 29) * rp;
      L[0] = m2l_fma(D[35], m, L[0]);
    }
    { const T m = -__ldg(Mr + 30) * rp;
      L[0] = m2l_fma(D[37], m, L[0]);
    }
    { const T m = -__ldg(Mr + 31) * rp;
      L[0] = m2l_fma(D[38], m, L[0]);
    }
    { const T m = -__ldg(Mr + 32) * rp;
      L[0] = m2l_fma(D[40], m, L[0]);
    }
    { const T m = -__ldg(Mr + 33) * rp;
      L[0] = m2l_fma(D[41], m, L[0]);
    }
    { const T m = -__ldg(Mr + 34) * rp;
      L[0] = m2l_fma(D[43], m, L[0]);
    }
    { const T m = -__ldg(Mr + 35) * rp;
      L[0] = m2l_fma(D[44], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_h_5(const T (&D)[46], const T *__restrict__ Mr, T (&L)[36])
{
    { const T m = __ldg(Mr + 0);
      L[0] = D[0] * m;
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = -D[10] * m;
      L[10] = -D[11] * m;
      L[11] = -D[12] * m;
      L[12] = -D[13] * m;
      L[13] = -D[14] * m;
      L[14] = -D[16] * m;
      L[15] = -D[17] * m;
      L[16] = D[19] * m;
      L[17] = D[20] * m;
      L[18] = D[21] * m;
      L[19] = D[22] * m;
      L[20] = D[23] * m;
      L[21] = D[25] * m;
      L[22] = D[26] * m;
      L[23] = D[28] * m;
      L[24] = D[29] * m;
      L[25] = -D[31] * m;
      L[26] = -D[32] * m;
      L[27] = -D[33] * m;
      L[28] = -D[34] * m;
      L[29] = -D[35] * m;
      L[30] = -D[37] * m;
      L[31] = -D[38] * m;
      L[32] = -D[40] * m;
      L[33] = -D[41] * m;
      L[34] = -D[43] * m;
      L[35] = -D[44] * m;
    }
    { const T m = __ldg(Mr + 1);
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(-D[4], m, L[1]);
      L[2] = m2l_fma(-D[5], m, L[2]);
      L[3] = m2l_fma(-D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(-D[19], m, L[9]);
      L[10] = m2l_fma(-D[20], m, L[10]);
      L[11] = m2l_fma(-D[21], m, L[11]);
      L[12] = m2l_fma(-D[22], m, L[12]);
      L[13] = m2l_fma(-D[23], m, L[13]);
      L[14] = m2l_fma(-D[25], m, L[14]);
      L[15] = m2l_fma(-D[26], m, L[15]);
      L[16] = m2l_fma(D[31], m, L[16]);
      L[17] = m2l_fma(D[32], m, L[17]);
      L[18] = m2l_fma(D[33], m, L[18]);
      L[19] = m2l_fma(D[34], m, L[19]);
      L[20] = m2l_fma(D[35], m, L[20]);
      L[21] = m2l_fma(D[37], m, L[21]);
      L[22] = m2l_fma(D[38], m, L[22]);
      L[23] = m2l_fma(D[40], m, L[23]);
      L[24] = m2l_fma(D[41], m, L[24]);
    }
    { const T m = __ldg(Mr + 2);
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(-D[5], m, L[1]);
      L[2] = m2l_fma(-D[7], m, L[2]);
      L[3] = m2l_fma(-D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(-D[20], m, L[9]);
      L[10] = m2l_fma(-D[22], m, L[10]);
      L[11] = m2l_fma(-D[23], m, L[11]);
      L[12] = m2l_fma(-D[25], m, L[12]);
      L[13] = m2l_fma(-D[26], m, L[13]);
      L[14] = m2l_fma(-D[28], m, L[14]);
      L[15] = m2l_fma(-D[29], m, L[15]);
      L[16] = m2l_fma(D[32], m, L[16]);
      L[17] = m2l_fma(D[34], m, L[17]);
      L[18] = m2l_fma(D[35], m, L[18]);
      L[19] = m2l_fma(D[37], m, L[19]);
      L[20] = m2l_fma(D[38], m, L[20]);
      L[21] = m2l_fma(D[40], m, L[21]);
      L[22] = m2l_fma(D[41], m, L[22]);
      L[23] = m2l_fma(D[43], m, L[23]);
      L[24] = m2l_fma(D[44], m, L[24]);
    }
    { const T m = __ldg(Mr + 3);
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(-D[6], m, L[1]);
      L[2] = m2l_fma(-D[8], m, L[2]);
      L[3] = m2l_fma(-D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(-D[21], m, L[9]);
      L[10] = m2l_fma(-D[23], m, L[10]);
      L[11] = m2l_fma(-D[24], m, L[11]);
      L[12] = m2l_fma(-D[26], m, L[12]);
      L[13] = m2l_fma(-D[27], m, L[13]);
      L[14] = m2l_fma(-D[29], m, L[14]);
      L[15] = m2l_fma(-D[30], m, L[15]);
      L[16] = m2l_fma(D[33], m, L[16]);
      L[17] = m2l_fma(D[35], m, L[17]);
      L[18] = m2l_fma(D[36], m, L[18]);
      L[19] = m2l_fma(D[38], m, L[19]);
      L[20] = m2l_fma(D[39], m, L[20]);
      L[21] = m2l_fma(D[41], m, L[21]);
      L[22] = m2l_fma(D[42], m, L[22]);
      L[23] = m2l_fma(D[44], m, L[23]);
      L[24] = m2l_fma(D[45], m, L[24]);
    }
    { const T m = __ldg(Mr + 4);
      L[0] = m2l_fma(D[4], m, L[0]);
      L[1] = m2l_fma(-D[10], m, L[1]);
      L[2] = m2l_fma(-D[11], m, L[2]);
      L[3] = m2l_fma(-D[12], m, L[3]);
      L[4] = m2l_fma(D[19], m, L[4]);
      L[5] = m2l_fma(D[20], m, L[5]);
      L[6] = m2l_fma(D[21], m, L[6]);
      L[7] = m2l_fma(D[22], m, L[7]);
      L[8] = m2l_fma(D[23], m, L[8]);
      L[9] = m2l_fma(-D[31], m, L[9]);
      L[10] = m2l_fma(-D[32], m, L[10]);
      L[11] = m2l_fma(-D[33], m, L[11]);
      L[12] = m2l_fma(-D[34], m, L[12]);
      L[13] = m2l_fma(-D[35], m, L[13]);
      L[14] = m2l_fma(-D[37], m, L[14]);
      L[15] = m2l_fma(-D[38], m, L[15]);
    }
    { const T m = __ldg(Mr + 5);
      L[0] = m2l_fma(D[5], m, L[0]);
      L[1] = m2l_fma(-D[11], m, L[1]);
      L[2] = m2l_fma(-D[13], m, L[2]);
      L[3] = m2l_fma(-D[14], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[22], m, L[5]);
      L[6] = m2l_fma(D[23], m, L[6]);
      L[7] = m2l_fma(D[25], m, L[7]);
      L[8] = m2l_fma(D[26], m, L[8]);
      L[9] = m2l_fma(-D[32], m, L[9]);
      L[10] = m2l_fma(-D[34], m, L[10]);
      L[11] = m2l_fma(-D[35], m, L[11]);
      L[12] = m2l_fma(-D[37], m, L[12]);
      L[13] = m2l_fma(-D[38], m, L[13]);
      L[14] = m2l_fma(-D[40], m, L[14]);
      L[15] = m2l_fma(-D[41], m, L[15]);
    }
    { const T m = __ldg(Mr + 6);
      L[0] = m2l_fma(D[6], m, L[0]);
      L[1] = m2l_fma(-D[12], m, L[1]);
      L[2] = m2l_fma(-D[14], m, L[2]);
      L[3] = m2l_fma(-D[15], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(-D[33], m, L[9]);
      L[10] = m2l_fma(-D[35], m, L[10]);
      L[11] = m2l_fma(-D[36], m, L[11]);
      L[12] = m2l_fma(-D[38], m, L[12]);
      L[13] = m2l_fma(-D[39], m, L[13]);
      L[14] = m2l_fma(-D[41], m, L[14]);
      L[15] = m2l_fma(-D[42], m, L[15]);
    }
    { const T m = __ldg(Mr + 7);
      L[0] = m2l_fma(D[7], m, L[0]);
      L[1] = m2l_fma(-D[13], m, L[1]);
      L[2] = m2l_fma(-D[16], m, L[2]);
      L[3] = m2l_fma(-D[17], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[25], m, L[5]);
      L[6] = m2l_fma(D[26], m, L[6]);
      L[7] = m2l_fma(D[28], m, L[7]);
      L[8] = m2l_fma(D[29], m, L[8]);
      L[9] = m2l_fma(-D[34], m, L[9]);
      L[10] = m2l_fma(-D[37], m, L[10]);
      L[11] = m2l_fma(-D[38], m, L[11]);
      L[12] = m2l_fma(-D[40], m, L[12]);
      L[13] = m2l_fma(-D[41], m, L[13]);
      L[14] = m2l_fma(-D[43], m, L[14]);
      L[15] = m2l_fma(-D[44], m, L[15]);
    }
    { const T m = __ldg(Mr + 8);
      L[0] = m2l_fma(D[8], m, L[0]);
      L[1] = m2l_fma(-D[14], m, L[1]);
      L[2] = m2l_fma(-D[17], m, L[2]);
      L[3] = m2l_fma(-D[18], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[29], m, L[7]);
      L[8] = m2l_fma(D[30], m, L[8]);
      L[9] = m2l_fma(-D[35], m, L[9]);
      L[10] = m2l_fma(-D[38], m, L[10]);
      L[11] = m2l_fma(-D[39], m, L[11]);
      L[12] = m2l_fma(-D[41], m, L[12]);
      L[13] = m2l_fma(-D[42], m, L[13]);
      L[14] = m2l_fma(-D[44], m, L[14]);
      L[15] = m2l_fma(-D[45], m, L[15]);
    }
    { const T m = __ldg(Mr + 9);
      L[0] = m2l_fma(D[10], m, L[0]);
      L[1] = m2l_fma(-D[19], m, L[1]);
      L[2] = m2l_fma(-D[20], m, L[2]);
      L[3] = m2l_fma(-D[21], m, L[3]);
      L[4] = m2l_fma(D[31], m, L[4]);
      L[5] = m2l_fma(D[32], m, L[5]);
      L[6] = m2l_fma(D[33], m, L[6]);
      L[7] = m2l_fma(D[34], m, L[7]);
      L[8] = m2l_fma(D[35], m, L[8]);
    }
    { const T m = __ldg(Mr + 10);
      L[0] = m2l_fma(D[11], m, L[0]);
      L[1] = m2l_fma(-D[20], m, L[1]);
      L[2] = m2l_fma(-D[22], m, L[2]);
      L[3] = m2l_fma(-D[23], m, L[3]);
      L[4] = m2l_fma(D[32], m, L[4]);
      L[5] = m2l_fma(D[34], m, L[5]);
      L[6] = m2l_fma(D[35], m, L[6]);
      L[7] = m2l_fma(D[37], m, L[7]);
      L[8] = m2l_fma(D[38], m, L[8]);
    }
    { const T m = __ldg(Mr + 11);
      L[0] = m2l_fma(D[12], m, L[0]);
      L[1] = m2l_fma(-D[21], m, L[1]);
      L[2] = m2l_fma(-D[23], m, L[2]);
      L[3] = m2l_fma(-D[24], m, L[3]);
      L[4] = m2l_fma(D[33], m, L[4]);
      L[5] = m2l_fma(D[35], m, L[5]);
      L[6] = m2l_fma(D[36], m, L[6]);
      L[7] = m2l_fma(D[38], m, L[7]);
      L[8] = m2l_fma(D[39], m, L[8]);
    }
    { const T m = __ldg(Mr + 12);
      L[0] = m2l_fma(D[13], m, L[0]);
      L[1] = m2l_fma(-D[22], m, L[1]);
      L[2] = m2l_fma(-D[25], m, L[2]);
      L[3] = m2l_fma(-D[26], m, L[3]);
      L[4] = m2l_fma(D[34], m, L[4]);
      L[5] = m2l_fma(D[37], m, L[5]);
      L[6] = m2l_fma(D[38], m, L[6]);
      L[7] = m2l_fma(D[40], m, L[7]);
      L[8] = m2l_fma(D[41], m, L[8]);
    }
    { const T m = __ldg(Mr + 13);
      L[0] = m2l_fma(D[14], m, L[0]);
      L[1] = m2l_fma(-D[23], m, L[1]);
      L[2] = m2l_fma(-D[26], m, L[2]);
      L[3] = m2l_fma(-D[27], m, L[3]);
      L[4] = m2l_fma(D[35], m, L[4]);
      L[5] = m2l_fma(D[38], m, L[5]);
      L[6] = m2l_fma(D[39], m, L[6]);
      L[7] = m2l_fma(D[41], m, L[7]);
      L[8] = m2l_fma(D[42], m, L[8]);
    }
    { const T m = __ldg(Mr + 14);
      L[0] = m2l_fma(D[16], m, L[0]);
      L[1] = m2l_fma(-D[25], m, L[1]);
      L[2] = m2l_fma(-D[28], m, L[2]);
      L[3] = m2l_fma(-D[29], m, L[3]);
      L[4] = m2l_fma(D[37], m, L[4]);
      L[5] = m2l_fma(D[40], m, L[5]);
      L[6] = m2l_fma(D[41], m, L[6]);
      L[7] = m2l_fma(D[43], m, L[7]);
      L[8] = m2l_fma(D[44], m, L[8]);
    }
    { const T m = __ldg(Mr + 15);
      L[0] = m2l_fma(D[17], m, L[0]);
      L[1] = m2l_fma(-D[26], m, L[1]);
      L[2] = m2l_fma(-D[29], m, L[2]);
      L[3] = m2l_fma(-D[30], m, L[3]);
      L[4] = m2l_fma(D[38], m, L[4]);
      L[5] = m2l_fma(D[41], m, L[5]);
      L[6] = m2l_fma(D[42], m, L[6]);
      L[7] = m2l_fma(D[44], m, L[7]);
      L[8] = m2l_fma(D[45], m, L[8]);
    }
    { const T m = __ldg(Mr + 16);
      L[0] = m2l_fma(D[19], m, L[0]);
      L[1] = m2l_fma(-D[31], m, L[1]);
      L[2] = m2l_fma(-D[32], m, L[2]);
      L[3] = m2l_fma(-D[33], m, L[3]);
    }
    { const T m = __ldg(Mr + 17);
      L[0] = m2l_fma(D[20], m, L[0]);
      L[1] = m2l_fma(-D[32], m, L[1]);
      L[2] = m2l_fma(-D[34], m, L[2]);
      L[3] = m2l_fma(-D[35], m, L[3]);
    }
    { const T m = __ldg(Mr + 18);
      L[0] = m2l_fma(D[21], m, L[0]);
      L[1] = m2l_fma(-D[33], m, L[1]);
      L[2] = m2l_fma(-D[35], m, L[2]);
      L[3] = m2l_fma(-D[36], m, L[3]);
    }
    { const T m = __ldg(Mr + 19);
      L[0] = m2l_fma(D[22], m, L[0]);
      L[1] = m2l_fma(-D[34], m, L[1]);
      L[2] = m2l_fma(-D[37], m, L[2]);
      L[3] = m2l_fma(-D[38], m, L[3]);
    }
    { const T m = __ldg(Mr + 20);
      L[0] = m2l_fma(D[23], m, L[0]);
      L[1] = m2l_fma(-D[35], m, L[1]);
      L[2] = m2l_fma(-D[38], m, L[2]);
      L[3] = m2l_fma(-D[39], m, L[3]);
    }
    { const T m = __ldg(Mr + 21);
      L[0] = m2l_fma(D[25], m, L[0]);
      L[1] = m2l_fma(-D[37], m, L[1]);
      L[2] = m2l_fma(-D[40], m, L[2]);
      L[3] = m2l_fma(-D[41], m, L[3]);
    }
    { const T m = __ldg(Mr + 22);
      L[0] = m2l_fma(D[26], m, L[0]);
      L[1] = m2l_fma(-D[38], m, L[1]);
      L[2] = m2l_fma(-D[41], m, L[2]);
      L[3] = m2l_fma(-D[42], m, L[3]);
    }
    { const T m = __ldg(Mr + 23);
      L[0] = m2l_fma(D[28], m, L[0]);
      L[1] = m2l_fma(-D[40], m, L[1]);
      L[2] = m2l_fma(-D[43], m, L[2]);
      L[3] = m2l_fma(-D[44], m, L[3]);
    }
    { const T m = __ldg(Mr + 24);
      L[0] = m2l_fma(D[29], m, L[0]);
      L[1] = m2l_fma(-D[41], m, L[1]);
      L[2] = m2l_fma(-D[44], m, L[2]);
      L[3] = m2l_fma(-D[45], m, L[3]);
    }
    { const T m = __ldg(Mr + 25);
      L[0] = m2l_fma(D[31], m, L[0]);
    }
    { const T m = __ldg(Mr + 26);
      L[0] = m2l_fma(D[32], m, L[0]);
    }
    { const T m = __ldg(Mr + 27);
      L[0] = m2l_fma(D[33], m, L[0]);
    }
    { const T m = __ldg(Mr + 28);
      L[0] = m2l_fma(D[34], m, L[0]);
    }
    { const T m = __ldg(Mr + 29);
      L[0] = m2l_fma(D[35], m, L[0]);
    }
    { const T m = __ldg(Mr + 30);
      L[0] = m2l_fma(D[37], m, L[0]);
    }
    { const T m = __ldg(Mr + 31);
      L[0] = m2l_fma(D[38], m, L[0]);
    }
    { const T m = __ldg(Mr + 32);
      L[0] = m2l_fma(D[40], m, L[0]);
    }
    { const T m = __ldg(Mr + 33);
      L[0] = m2l_fma(D[41], m, L[0]);
    }
    { const T m = __ldg(Mr + 34);
      L[0] = m2l_fma(D[43], m, L[0]);
    }
    { const T m = __ldg(Mr + 35);
      L[0] = m2l_fma(D[44], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_a_h_forces_5(const T (&D)[46], const T *__restrict__ Mr, T rho, T (&L)[36])
{
    L[0] = T(0);
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[10] * m;
      L[10] = D[11] * m;
      L[11] = D[12] * m;
      L[12] = D[13] * m;
      L[13] = D[14] * m;
      L[14] = D[16] * m;
      L[15] = D[17] * m;
      L[16] = D[19] * m;
      L[17] = D[20] * m;
      L[18] = D[21] * m;
      L[19] = D[22] * m;
      L[20] = D[23] * m;
      L[21] = D[25] * m;
      L[22] = D[26] * m;
      L[23] = D[28] * m;
      L[24] = D[29] * m;
      L[25] = D[31] * m;
      L[26] = D[32] * m;
      L[27] = D[33] * m;
      L[28] = D[34] * m;
      L[29] = D[35] * m;
      L[30] = D[37] * m;
      L[31] = D[38] * m;
      L[32] = D[40] * m;
      L[33] = D[41] * m;
      L[34] = D[43] * m;
      L[35] = D[44] * m;
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 1) * rp;
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(D[20], m, L[10]);
      L[11] = m2l_fma(D[21], m, L[11]);
      L[12] = m2l_fma(D[22], m, L[12]);
      L[13] = m2l_fma(D[23], m, L[13]);
      L[14] = m2l_fma(D[25], m, L[14]);
      L[15] = m2l_fma(D[26], m, L[15]);
      L[16] = m2l_fma(D[31], m, L[16]);
      L[17] = m2l_fma(D[32], m, L[17]);
      L[18] = m2l_fma(D[33], m, L[18]);
      L[19] = m2l_fma(D[34], m, L[19]);
      L[20] = m2l_fma(D[35], m, L[20]);
      L[21] = m2l_fma(D[37], m, L[21]);
      L[22] = m2l_fma(D[38], m, L[22]);
      L[23] = m2l_fma(D[40], m, L[23]);
      L[24] = m2l_fma(D[41], m, L[24]);
    }
    { const T m = -__ldg(Mr + 2) * rp;
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[20], m, L[9]);
      L[10] = m2l_fma(D[22], m, L[10]);
      L[11] = m2l_fma(D[23], m, L[11]);
      L[12] = m2l_fma(D[25], m, L[12]);
      L[13] = m2l_fma(D[26], m, L[13]);
      L[14] = m2l_fma(D[28], m, L[14]);
      L[15] = m2l_fma(D[29], m, L[15]);
      L[16] = m2l_fma(D[32], m, L[16]);
      L[17] = m2l_fma(D[34], m, L[17]);
      L[18] = m2l_fma(D[35], m, L[18]);
      L[19] = m2l_fma(D[37], m, L[19]);
      L[20] = m2l_fma(D[38], m, L[20]);
      L[21] = m2l_fma(D[40], m, L[21]);
      L[22] = m2l_fma(D[41], m, L[22]);
      L[23] = m2l_fma(D[43], m, L[23]);
      L[24] = m2l_fma(D[44], m, L[24]);
    }
    { const T m = -__ldg(Mr + 3) * rp;
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[21], m, L[9]);
      L[10] = m2l_fma(D[23], m, L[10]);
      L[11] = m2l_fma(D[24], m, L[11]);
      L[12] = m2l_fma(D[26], m, L[12]);
      L[13] = m2l_fma(D[27], m, L[13]);
      L[14] = m2l_fma(D[29], m, L[14]);
      L[15] = m2l_fma(D[30], m, L[15]);
      L[16] = m2l_fma(D[33], m, L[16]);
      L[17] = m2l_fma(D[35], m, L[17]);
      L[18] = m2l_fma(D[36], m, L[18]);
      L[19] = m2l_fma(D[38], m, L[19]);
      L[20] = m2l_fma(D[39], m, L[20]);
      L[21] = m2l_fma(D[41], m, L[21]);
      L[22] = m2l_fma(D[42], m, L[22]);
      L[23] = m2l_fma(D[44], m, L[23]);
      L[24] = m2l_fma(D[45], m, L[24]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 4) * rp;
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
      L[4] = m2l_fma(D[19], m, L[4]);
      L[5] = m2l_fma(D[20], m, L[5]);
      L[6] = m2l_fma(D[21], m, L[6]);
      L[7] = m2l_fma(D[22], m, L[7]);
      L[8] = m2l_fma(D[23], m, L[8]);
      L[9] = m2l_fma(D[31], m, L[9]);
      L[10] = m2l_fma(D[32], m, L[10]);
      L[11] = m2l_fma(D[33], m, L[11]);
      L[12] = m2l_fma(D[34], m, L[12]);
      L[13] = m2l_fma(D[35], m, L[13]);
      L[14] = m2l_fma(D[37], m, L[14]);
      L[15] = m2l_fma(D[38], m, L[15]);
    }
    { const T m = __ldg(Mr + 5) * rp;
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[22], m, L[5]);
      L[6] = m2l_fma(D[23], m, L[6]);
      L[7] = m2l_fma(D[25], m, L[7]);
      L[8] = m2l_fma(D[26], m, L[8]);
      L[9] = m2l_fma(D[32], m, L[9]);
      L[10] = m2l_fma(D[34], m, L[10]);
      L[11] = m2l_fma(D[35], m, L[11]);
      L[12] = m2l_fma(D[37], m, L[12]);
      L[13] = m2l_fma(D[38], m, L[13]);
      L[14] = m2l_fma(D[40], m, L[14]);
      L[15] = m2l_fma(D[41], m, L[15]);
    }
    { const T m = __ldg(Mr + 6) * rp;
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(D[33], m, L[9]);
      L[10] = m2l_fma(D[35], m, L[10]);
      L[11] = m2l_fma(D[36], m, L[11]);
      L[12] = m2l_fma(D[38], m, L[12]);
      L[13] = m2l_fma(D[39], m, L[13]);
      L[14] = m2l_fma(D[41], m, L[14]);
      L[15] = m2l_fma(D[42], m, L[15]);
    }
    { const T m = __ldg(Mr + 7) * rp;
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[25], m, L[5]);
      L[6] = m2l_fma(D[26], m, L[6]);
      L[7] = m2l_fma(D[28], m, L[7]);
      L[8] = m2l_fma(D[29], m, L[8]);
      L[9] = m2l_fma(D[34], m, L[9]);
      L[10] = m2l_fma(D[37], m, L[10]);
      L[11] = m2l_fma(D[38], m, L[11]);
      L[12] = m2l_fma(D[40], m, L[12]);
      L[13] = m2l_fma(D[41], m, L[13]);
      L[14] = m2l_fma(D[43], m, L[14]);
      L[15] = m2l_fma(D[44], m, L[15]);
    }
    { const T m = __ldg(Mr + 8) * rp;
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[29], m, L[7]);
      L[8] = m2l_fma(D[30], m, L[8]);
      L[9] = m2l_fma(D[35], m, L[9]);
      L[10] = m2l_fma(D[38], m, L[10]);
      L[11] = m2l_fma(D[39], m, L[11]);
      L[12] = m2l_fma(D[41], m, L[12]);
      L[13] = m2l_fma(D[42], m, L[13]);
      L[14] = m2l_fma(D[44], m, L[14]);
      L[15] = m2l_fma(D[45], m, L[15]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 9) * rp;
      L[1] = m2l_fma(D[19], m, L[1]);
      L[2] = m2l_fma(D[20], m, L[2]);
      L[3] = m2l_fma(D[21], m, L[3]);
      L[4] = m2l_fma(D[31], m, L[4]);
      L[5] = m2l_fma(D[32], m, L[5]);
      L[6] = m2l_fma(D[33], m, L[6]);
      L[7] = m2l_fma(D[34], m, L[7]);
      L[8] = m2l_fma(D[35], m, L[8]);
    }
    { const T m = -__ldg(Mr + 10) * rp;
      L[1] = m2l_fma(D[20], m, L[1]);
      L[2] = m2l_fma(D[22], m, L[2]);
      L[3] = m2l_fma(D[23], m, L[3]);
      L[4] = m2l_fma(D[32], m, L[4]);
      L[5] = m2l_fma(D[34], m, L[5]);
      L[6] = m2l_fma(D[35], m, L[6]);
      L[7] = m2l_fma(D[37], m, L[7]);
      L[8] = m2l_fma(D[38], m, L[8]);
    }
    { const T m = -__ldg(Mr + 11) * rp;
      L[1] = m2l_fma(D[21], m, L[1]);
      L[2] = m2l_fma(D[23], m, L[2]);
      L[3] = m2l_fma(D[24], m, L[3]);
      L[4] = m2l_fma(D[33], m, L[4]);
      L[5] = m2l_fma(D[35], m, L[5]);
      L[6] = m2l_fma(D[36], m, L[6]);
      L[7] = m2l_fma(D[38], m, L[7]);
      L[8] = m2l_fma(D[39], m, L[8]);
    }
    { const T m = -__ldg(Mr + 12) * rp;
      L[1] = m2l_fma(D[22], m, L[1]);
      L[2] = m2l_fma(D[25], m, L[2]);
      L[3] = m2l_fma(D[26], m, L[3]);
      L[4] = m2l_fma(D[34], m, L[4]);
      L[5] = m2l_fma(D[37], m, L[5]);
      L[6] = m2l_fma(D[38], m, L[6]);
      L[7] = m2l_fma(D[40], m, L[7]);
      L[8] = m2l_fma(D[41], m, L[8]);
    }
    { const T m = -__ldg(Mr + 13) * rp;
      L[1] = m2l_fma(D[23], m, L[1]);
      L[2] = m2l_fma(D[26], m, L[2]);
      L[3] = m2l_fma(D[27], m, L[3]);
      L[4] = m2l_fma(D[35], m, L[4]);
      L[5] = m2l_fma(D[38], m, L[5]);
      L[6] = m2l_fma(D[39], m, L[6]);
      L[7] = m2l_fma(D[41], m, L[7]);
      L[8] = m2l_fma(D[42], m, L[8]);
    }
    { const T m = -__ldg(Mr + 14) * rp;
      L[1] = m2l_fma(D[25], m, L[1]);
      L[2] = m2l_fma(D[28], m, L[2]);
      L[3] = m2l_fma(D[29], m, L[3]);
      L[4] = m2l_fma(D[37], m, L[4]);
      L[5] = m2l_fma(D[40], m, L[5]);
      L[6] = m2l_fma(D[41], m, L[6]);
      L[7] = m2l_fma(D[43], m, L[7]);
      L[8] = m2l_fma(D[44], m, L[8]);
    }
    { const T m = -__ldg(Mr + 15) * rp;
      L[1] = m2l_fma(D[26], m, L[1]);
      L[2] = m2l_fma(D[29], m, L[2]);
      L[3] = m2l_fma(D[30], m, L[3]);
      L[4] = m2l_fma(D[38], m, L[4]);
      L[5] = m2l_fma(D[41], m, L[5]);
      L[6] = m2l_fma(D[42], m, L[6]);
      L[7] = m2l_fma(D[44], m, L[7]);
      L[8] = m2l_fma(D[45], m, L[8]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 16) * rp;
      L[1] = m2l_fma(D[31], m, L[1]);
      L[2] = m2l_fma(D[32], m, L[2]);
      L[3] = m2l_fma(D[33], m, L[3]);
    }
    { const T m = __ldg(Mr + 17) * rp;
      L[1] = m2l_fma(D[32], m, L[1]);
      L[2] = m2l_fma(D[34], m, L[2]);
      L[3] = m2l_fma(D[35], m, L[3]);
    }
    { const T m = __ldg(Mr + 18) * rp;
      L[1] = m2l_fma(D[33], m, L[1]);
      L[2] = m2l_fma(D[35], m, L[2]);
      L[3] = m2l_fma(D[36], m, L[3]);
    }
    { const T m = __ldg(Mr + 19) * rp;
      L[1] = m2l_fma(D[34], m, L[1]);
      L[2] = m2l_fma(D[37], m, L[2]);
      L[3] = m2l_fma(D[38], m, L[3]);
    }
    { const T m = __ldg(Mr + 20) * rp;
      L[1] = m2l_fma(D[35], m, L[1]);
      L[2] = m2l_fma(D[38], m, L[2]);
      L[3] = m2l_fma(D[39], m, L[3]);
    }
    { const T m = __ldg(Mr + 21) * rp;
      L[1] = m2l_fma(D[37], m, L[1]);
      L[2] = m2l_fma(D[40], m, L[2]);
      L[3] = m2l_fma(D[41], m, L[3]);
    }
    { const T m = __ldg(Mr + 22) * rp;
      L[1] = m2l_fma(D[38], m, L[1]);
      L[2] = m2l_fma(D[41], m, L[2]);
      L[3] = m2l_fma(D[42], m, L[3]);
    }
    { const T m = __ldg(Mr + 23) * rp;
      L[1] = m2l_fma(D[40], m, L[1]);
      L[2] = m2l_fma(D[43], m, L[2]);
      L[3] = m2l_fma(D[44], m, L[3]);
    }
    { const T m = __ldg(Mr + 24) * rp;
      L[1] = m2l_fma(D[41], m, L[1]);
      L[2] = m2l_fma(D[44], m, L[2]);
      L[3] = m2l_fma(D[45], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_acc_h_forces_5(const T (&D)[46], const T *__restrict__ Mr, T rho, T (&L)[36])
{
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[1] = m2l_fma(D[1], m, L[1]);
      L[2] = m2l_fma(D[2], m, L[2]);
      L[3] = m2l_fma(D[3], m, L[3]);
      L[4] = m2l_fma(D[4], m, L[4]);
      L[5] = m2l_fma(D[5], m, L[5]);
      L[6] = m2l_fma(D[6], m, L[6]);
      L[7] = m2l_fma(D[7], m, L[7]);
      L[8] = m2l_fma(D[8], m, L[8]);
      L[9] = m2l_fma(D[10], m, L[9]);
      L[10] = m2l_fma(D[11], m, L[10]);
      L[11] = m2l_fma(D[12], m, L[11]);
      L[12] = m2l_fma(D[13], m, L[12]);
      L[13] = m2l_fma(D[14], m, L[13]);
      L[14] = m2l_fma(D[16], m, L[14]);
      L[15] = m2l_fma(D[17], m, L[15]);
      L[16] = m2l_fma(D[19], m, L[16]);
      L[17] = m2l_fma(D[20], m, L[17]);
      L[18] = m2l_fma(D[21], m, L[18]);
      L[19] = m2l_fma(D[22], m, L[19]);
      L[20] = m2l_fma(D[23], m, L[20]);
      L[21] = m2l_fma(D[25], m, L[21]);
      L[22] = m2l_fma(D[26], m, L[22]);
      L[23] = m2l_fma(D[28], m, L[23]);
      L[24] = m2l_fma(D[29], m, L[24]);
      L[25] = m2l_fma(D[31], m, L[25]);
      L[26] = m2l_fma(D[32], m, L[26]);
      L[27] = m2l_fma(D[33], m, L[27]);
      L[28] = m2l_fma(D[34], m, L[28]);
      L[29] = m2l_fma(D[35], m, L[29]);
      L[30] = m2l_fma(D[37], m, L[30]);
      L[31] = m2l_fma(D[38], m, L[31]);
      L[32] = m2l_fma(D[40], m, L[32]);
      L[33] = m2l_fma(D[41], m, L[33]);
      L[34] = m2l_fma(D[43], m, L[34]);
      L[35] = m2l_fma(D[44], m, L[35]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 1) * rp;
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(D[20], m, L[10]);
      L[11] = m2l_fma(D[21], m, L[11]);
      L[12] = m2l_fma(D[22], m, L[12]);
      L[13] = m2l_fma(D[23], m, L[13]);
      L[14] = m2l_fma(D[25], m, L[14]);
      L[15] = m2l_fma(D[26], m, L[15]);
      L[16] = m2l_fma(D[31], m, L[16]);
      L[17] = m2l_fma(D[32], m, L[17]);
      L[18] = m2l_fma(D[33], m, L[18]);
      L[19] = m2l_fma(D[34], m, L[19]);
      L[20] = m2l_fma(D[35], m, L[20]);
      L[21] = m2l_fma(D[37], m, L[21]);
      L[22] = m2l_fma(D[38], m, L[22]);
      L[23] = m2l_fma(D[40], m, L[23]);
      L[24] = m2l_fma(D[41], m, L[24]);
    }
    { const T m = -__ldg(Mr + 2) * rp;
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[20], m, L[9]);
      L[10] = m2l_fma(D[22], m, L[10]);
      L[11] = m2l_fma(D[23], m, L[11]);
      L[12] = m2l_fma(D[25], m, L[12]);
      L[13] = m2l_fma(D[26], m, L[13]);
      L[14] = m2l_fma(D[28], m, L[14]);
      L[15] = m2l_fma(D[29], m, L[15]);
      L[16] = m2l_fma(D[32], m, L[16]);
      L[17] = m2l_fma(D[34], m, L[17]);
      L[18] = m2l_fma(D[35], m, L[18]);
      L[19] = m2l_fma(D[37], m, L[19]);
      L[20] = m2l_fma(D[38], m, L[20]);
      L[21] = m2l_fma(D[40], m, L[21]);
      L[22] = m2l_fma(D[41], m, L[22]);
      L[23] = m2l_fma(D[43], m, L[23]);
      L[24] = m2l_fma(D[44], m, L[24]);
    }
    { const T m = -__ldg(Mr + 3) * rp;
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[21], m, L[9]);
      L[10] = m2l_fma(D[23], m, L[10]);
      L[11] = m2l_fma(D[24], m, L[11]);
      L[12] = m2l_fma(D[26], m, L[12]);
      L[13] = m2l_fma(D[27], m, L[13]);
      L[14] = m2l_fma(D[29], m, L[14]);
      L[15] = m2l_fma(D[30], m, L[15]);
      L[16] = m2l_fma(D[33], m, L[16]);
      L[17] = m2l_fma(D[35], m, L[17]);
      L[18] = m2l_fma(D[36], m, L[18]);
      L[19] = m2l_fma(D[38], m, L[19]);
      L[20] = m2l_fma(D[39], m, L[20]);
      L[21] = m2l_fma(D[41], m, L[21]);
      L[22] = m2l_fma(D[42], m, L[22]);
      L[23] = m2l_fma(D[44], m, L[23]);
      L[24] = m2l_fma(D[45], m, L[24]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 4) * rp;
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
      L[4] = m2l_fma(D[19], m, L[4]);
      L[5] = m2l_fma(D[20], m, L[5]);
      L[6] = m2l_fma(D[21], m, L[6]);
      L[7] = m2l_fma(D[22], m, L[7]);
      L[8] = m2l_fma(D[23], m, L[8]);
      L[9] = m2l_fma(D[31], m, L[9]);
      L[10] = m2l_fma(D[32], m, L[10]);
      L[11] = m2l_fma(D[33], m, L[11]);
      L[12] = m2l_fma(D[34], m, L[12]);
      L[13] = m2l_fma(D[35], m, L[13]);
      L[14] = m2l_fma(D[37], m, L[14]);
      L[15] = m2l_fma(D[38], m, L[15]);
    }
    { const T m = __ldg(Mr + 5) * rp;
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[22], m, L[5]);
      L[6] = m2l_fma(D[23], m, L[6]);
      L[7] = m2l_fma(D[25], m, L[7]);
      L[8] = m2l_fma(D[26], m, L[8]);
      L[9] = m2l_fma(D[32], m, L[9]);
      L[10] = m2l_fma(D[34], m, L[10]);
      L[11] = m2l_fma(D[35], m, L[11]);
      L[12] = m2l_fma(D[37], m, L[12]);
      L[13] = m2l_fma(D[38], m, L[13]);
      L[14] = m2l_fma(D[40], m, L[14]);
      L[15] = m2l_fma(D[41], m, L[15]);
    }
    { const T m = __ldg(Mr + 6) * rp;
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(D[33], m, L[9]);
      L[10] = m2l_fma(D[35], m, L[10]);
      L[11] = m2l_fma(D[36], m, L[11]);
      L[12] = m2l_fma(D[38], m, L[12]);
      L[13] = m2l_fma(D[39], m, L[13]);
      L[14] = m2l_fma(D[41], m, L[14]);
      L[15] = m2l_fma(D[42], m, L[15]);
    }
    { const T m = __ldg(Mr + 7) * rp;
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[25], m, L[5]);
      L[6] = m2l_fma(D[26], m, L[6]);
      L[7] = m2l_fma(D[28], m, L[7]);
      L[8] = m2l_fma(D[29], m, L[8]);
      L[9] = m2l_fma(D[34], m, L[9]);
      L[10] = m2l_fma(D[37], m, L[10]);
      L[11] = m2l_fma(D[38], m, L[11]);
      L[12] = m2l_fma(D[40], m, L[12]);
      L[13] = m2l_fma(D[41], m, L[13]);
      L[14] = m2l_fma(D[43], m, L[14]);
      L[15] = m2l_fma(D[44], m, L[15]);
    }
    { const T m = __ldg(Mr + 8) * rp;
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[29], m, L[7]);
      L[8] = m2l_fma(D[30], m, L[8]);
      L[9] = m2l_fma(D[35], m, L[9]);
      L[10] = m2l_fma(D[38], m, L[10]);
      L[11] = m2l_fma(D[39], m, L[11]);
      L[12] = m2l_fma(D[41], m, L[12]);
      L[13] = m2l_fma(D[42], m, L[13]);
      L[14] = m2l_fma(D[44], m, L[14]);
      L[15] = m2l_fma(D[45], m, L[15]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 9) * rp;
      L[1] = m2l_fma(D[19], m, L[1]);
      L[2] = m2l_fma(D[20], m, L[2]);
      L[3] = m2l_fma(D[21], m, L[3]);
      L[4] = m2l_fma(D[31], m, L[4]);
      L[5] = m2l_fma(D[32], m, L[5]);
      L[6] = m2l_fma(D[33], m, L[6]);
      L[7] = m2l_fma(D[34], m, L[7]);
      L[8] = m2l_fma(D[35], m, L[8]);
    }
    { const T m = -__ldg(Mr + 10) * rp;
      L[1] = m2l_fma(D[20], m, L[1]);
      L[2] = m2l_fma(D[22], m, L[2]);
      L[3] = m2l_fma(D[23], m, L[3]);
      L[4] = m2l_fma(D[32], m, L[4]);
      L[5] = m2l_fma(D[34], m, L[5]);
      L[6] = m2l_fma(D[35], m, L[6]);
      L[7] = m2l_fma(D[37], m, L[7]);
      L[8] = m2l_fma(D[38], m, L[8]);
    }
    { const T m = -__ldg(Mr + 11) * rp;
      L[1] = m2l_fma(D[21], m, L[1]);
      L[2] = m2l_fma(D[23], m, L[2]);
      L[3] = m2l_fma(D[24], m, L[3]);
      L[4] = m2l_fma(D[33], m, L[4]);
      L[5] = m2l_fma(D[35], m, L[5]);
      L[6] = m2l_fma(D[36], m, L[6]);
      L[7] = m2l_fma(D[38], m, L[7]);
      L[8] = m2l_fma(D[39], m, L[8]);
    }
    { const T m = -__ldg(Mr + 12) * rp;
      L[1] = m2l_fma(D[22], m, L[1]);
      L[2] = m2l_fma(D[25], m, L[2]);
      L[3] = m2l_fma(D[26], m, L[3]);
      L[4] = m2l_fma(D[34], m, L[4]);
      L[5] = m2l_fma(D[37], m, L[5]);
      L[6] = m2l_fma(D[38], m, L[6]);
      L[7] = m2l_fma(D[40], m, L[7]);
      L[8] = m2l_fma(D[41], m, L[8]);
    }
    { const T m = -__ldg(Mr + 13) * rp;
      L[1] = m2l_fma(D[23], m, L[1]);
      L[2] = m2l_fma(D[26], m, L[2]);
      L[3] = m2l_fma(D[27], m, L[3]);
      L[4] = m2l_fma(D[35], m, L[4]);
      L[5] = m2l_fma(D[38], m, L[5]);
      L[6] = m2l_fma(D[39], m, L[6]);
      L[7] = m2l_fma(D[41], m, L[7]);
      L[8] = m2l_fma(D[42], m, L[8]);
    }
    { const T m = -__ldg(Mr + 14) * rp;
      L[1] = m2l_fma(D[25], m, L[1]);
      L[2] = m2l_fma(D[28], m, L[2]);
      L[3] = m2l_fma(D[29], m, L[3]);
      L[4] = m2l_fma(D[37], m, L[4]);
      L[5] = m2l_fma(D[40], m, L[5]);
      L[6] = m2l_fma(D[41], m, L[6]);
      L[7] = m2l_fma(D[43], m, L[7]);
      L[8] = m2l_fma(D[44], m, L[8]);
    }
    { const T m = -__ldg(Mr + 15) * rp;
      L[1] = m2l_fma(D[26], m, L[1]);
      L[2] = m2l_fma(D[29], m, L[2]);
      L[3] = m2l_fma(D[30], m, L[3]);
      L[4] = m2l_fma(D[38], m, L[4]);
      L[5] = m2l_fma(D[41], m, L[5]);
      L[6] = m2l_fma(D[42], m, L[6]);
      L[7] = m2l_fma(D[44], m, L[7]);
      L[8] = m2l_fma(D[45], m, L[8]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 16) * rp;
      L[1] = m2l_fma(D[31], m, L[1]);
      L[2] = m2l_fma(D[32], m, L[2]);
      L[3] = m2l_fma(D[33], m, L[3]);
    }
    { const T m = __ldg(Mr + 17) * rp;
      L[1] = m2l_fma(D[32], m, L[1]);
      L[2] = m2l_fma(D[34], m, L[2]);
      L[3] = m2l_fma(D[35], m, L[3]);
    }
    { const T m = __ldg(Mr + 18) * rp;
      L[1] = m2l_fma(D[33], m, L[1]);
      L[2] = m2l_fma(D[35], m, L[2]);
      L[3] = m2l_fma(D[36], m, L[3]);
    }
    { const T m = __ldg(Mr + 19) * rp;
      L[1] = m2l_fma(D[34], m, L[1]);
      L[2] = m2l_fma(D[37], m, L[2]);
      L[3] = m2l_fma(D[38], m, L[3]);
    }
    { const T m = __ldg(Mr + 20) * rp;
      L[1] = m2l_fma(D[35], m, L[1]);
      L[2] = m2l_fma(D[38], m, L[2]);
      L[3] = m2l_fma(D[39], m, L[3]);
    }
    { const T m = __ldg(Mr + 21) * rp;
      L[1] = m2l_fma(D[37], m, L[1]);
      L[2] = m2l_fma(D[40], m, L[2]);
      L[3] = m2l_fma(D[41], m, L[3]);
    }
    { const T m = __ldg(Mr + 22) * rp;
      L[1] = m2l_fma(D[38], m, L[1]);
      L[2] = m2l_fma(D[41], m, L[2]);
      L[3] = m2l_fma(D[42], m, L[3]);
    }
    { const T m = __ldg(Mr + 23) * rp;
      L[1] = m2l_fma(D[40], m, L[1]);
      L[2] = m2l_fma(D[43], m, L[2]);
      L[3] = m2l_fma(D[44], m, L[3]);
    }
    { const T m = __ldg(Mr + 24) * rp;
      L[1] = m2l_fma(D[41], m, L[1]);
      L[2] = m2l_fma(D[44], m, L[2]);
      L[3] = m2l_fma(D[45], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_h_forces_5(const T (&D)[46], const T *__restrict__ Mr, T (&L)[36])
{
    L[0] = T(0);
    { const T m = __ldg(Mr + 0);
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = -D[10] * m;
      L[10] = -D[11] * m;
      L[11] = -D[12] * m;
      L[12] = -D[13] * m;
      L[13] = -D[14] * m;
      L[14] = -D[16] * m;
      L[15] = -D[17] * m;
      L[16] = D[19] * m;
      L[17] = D[20] * m;
      L[18] = D[21] * m;
      L[19] = D[22] * m;
      L[20] = D[23] * m;
      L[21] = D[25] * m;
      L[22] = D[26] * m;
      L[23] = D[28] * m;
      L[24] = D[29] * m;
      L[25] = -D[31] * m;
      L[26] = -D[32] * m;
      L[27] = -D[33] * m;
      L[28] = -D[34] * m;
      L[29] = -D[35] * m;
      L[30] = -D[37] * m;
      L[31] = -D[38] * m;
      L[32] = -D[40] * m;
      L[33] = -D[41] * m;
      L[34] = -D[43] * m;
      L[35] = -D[44] * m;
    }
    { const T m = __ldg(Mr + 1);
      L[1] = m2l_fma(-D[4], m, L[1]);
      L[2] = m2l_fma(-D[5], m, L[2]);
      L[3] = m2l_fma(-D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(-D[19], m, L[9]);
      L[10] = m2l_fma(-D[20], m, L[10]);
      L[11] = m2l_fma(-D[21], m, L[11]);
      L[12] = m2l_fma(-D[22], m, L[12]);
      L[13] = m2l_fma(-D[23], m, L[13]);
      L[14] = m2l_fma(-D[25], m, L[14]);
      L[15] = m2l_fma(-D[26], m, L[15]);
      L[16] = m2l_fma(D[31], m, L[16]);
      L[17] = m2l_fma(D[32], m, L[17]);
      L[18] = m2l_fma(D[33], m, L[18]);
      L[19] = m2l_fma(D[34], m, L[19]);
      L[20] = m2l_fma(D[35], m, L[20]);
      L[21] = m2l_fma(D[37], m, L[21]);
      L[22] = m2l_fma(D[38], m, L[22]);
      L[23] = m2l_fma(D[40], m, L[23]);
      L[24] = m2l_fma(D[41], m, L[24]);
    }
    { const T m = __ldg(Mr + 2);
      L[1] = m2l_fma(-D[5], m, L[1]);
      L[2] = m2l_fma(-D[7], m, L[2]);
      L[3] = m2l_fma(-D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(-D[20], m, L[9]);
      L[10] = m2l_fma(-D[22], m, L[10]);
      L[11] = m2l_fma(-D[23], m, L[11]);
      L[12] = m2l_fma(-D[25], m, L[12]);
      L[13] = m2l_fma(-D[26], m, L[13]);
      L[14] = m2l_fma(-D[28], m, L[14]);
      L[15] = m2l_fma(-D[29], m, L[15]);
      L[16] = m2l_fma(D[32], m, L[16]);
      L[17] = m2l_fma(D[34], m, L[17]);
      L[18] = m2l_fma(D[35], m, L[18]);
      L[19] = m2l_fma(D[37], m, L[19]);
      L[20] = m2l_fma(D[38], m, L[20]);
      L[21] = m2l_fma(D[40], m, L[21]);
      L[22] = m2l_fma(D[41], m, L[22]);
      L[23] = m2l_fma(D[43], m, L[23]);
      L[24] = m2l_fma(D[44], m, L[24]);
    }
    { const T m = __ldg(Mr + 3);
      L[1] = m2l_fma(-D[6], m, L[1]);
      L[2] = m2l_fma(-D[8], m, L[2]);
      L[3] = m2l_fma(-D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(-D[21], m, L[9]);
      L[10] = m2l_fma(-D[23], m, L[10]);
      L[11] = m2l_fma(-D[24], m, L[11]);
      L[12] = m2l_fma(-D[26], m, L[12]);
      L[13] = m2l_fma(-D[27], m, L[13]);
      L[14] = m2l_fma(-D[29], m, L[14]);
      L[15] = m2l_fma(-D[30], m, L[15]);
      L[16] = m2l_fma(D[33], m, L[16]);
      L[17] = m2l_fma(D[35], m, L[17]);
      L[18] = m2l_fma(D[36], m, L[18]);
      L[19] = m2l_fma(D[38], m, L[19]);
      L[20] = m2l_fma(D[39], m, L[20]);
      L[21] = m2l_fma(D[41], m, L[21]);
      L[22] = m2l_fma(D[42], m, L[22]);
      L[23] = m2l_fma(D[44], m, L[23]);
      L[24] = m2l_fma(D[45], m, L[24]);
    }
    { const T m = __ldg(Mr + 4);
      L[1] = m2l_fma(-D[10], m, L[1]);
      L[2] = m2l_fma(-D[11], m, L[2]);
      L[3] = m2l_fma(-D[12], m, L[3]);
      L[4] = m2l_fma(D[19], m, L[4]);
      L[5] = m2l_fma(D[20], m, L[5]);
      L[6] = m2l_fma(D[21], m, L[6]);
      L[7] = m2l_fma(D[22], m, L[7]);
      L[8] = m2l_fma(D[23], m, L[8]);
      L[9] = m2l_fma(-D[31], m, L[9]);
      L[10] = m2l_fma(-D[32], m, L[10]);
      L[11] = m2l_fma(-D[33], m, L[11]);
      L[12] = m2l_fma(-D[34], m, L[12]);
      L[13] = m2l_fma(-D[35], m, L[13]);
      L[14] = m2l_fma(-D[37], m, L[14]);
      L[15] = m2l_fma(-D[38], m, L[15]);
    }
    { const T m = __ldg(Mr + 5);
      L[1] = m2l_fma(-D[11], m, L[1]);
      L[2] = m2l_fma(-D[13], m, L[2]);
      L[3] = m2l_fma(-D[14], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[22], m, L[5]);
      L[6] = m2l_fma(D[23], m, L[6]);
      L[7] = m2l_fma(D[25], m, L[7]);
      L[8] = m2l_fma(D[26], m, L[8]);
      L[9] = m2l_fma(-D[32], m, L[9]);
      L[10] = m2l_fma(-D[34], m, L[10]);
      L[11] = m2l_fma(-D[35], m, L[11]);
      L[12] = m2l_fma(-D[37], m, L[12]);
      L[13] = m2l_fma(-D[38], m, L[13]);
      L[14] = m2l_fma(-D[40], m, L[14]);
      L[15] = m2l_fma(-D[41], m, L[15]);
    }
    { const T m = __ldg(Mr + 6);
      L[1] = m2l_fma(-D[12], m, L[1]);
      L[2] = m2l_fma(-D[14], m, L[2]);
      L[3] = m2l_fma(-D[15], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(-D[33], m, L[9]);
      L[10] = m2l_fma(-D[35], m, L[10]);
      L[11] = m2l_fma(-D[36], m, L[11]);
      L[12] = m2l_fma(-D[38], m, L[12]);
      L[13] = m2l_fma(-D[39], m, L[13]);
      L[14] = m2l_fma(-D[41], m, L[14]);
      L[15] = m2l_fma(-D[42], m, L[15]);
    }
    { const T m = __ldg(Mr + 7);
      L[1] = m2l_fma(-D[13], m, L[1]);
      L[2] = m2l_fma(-D[16], m, L[2]);
      L[3] = m2l_fma(-D[17], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[25], m, L[5]);
      L[6] = m2l_fma(D[26], m, L[6]);
      L[7] = m2l_fma(D[28], m, L[7]);
      L[8] = m2l_fma(D[29], m, L[8]);
      L[9] = m2l_fma(-D[34], m, L[9]);
      L[10] = m2l_fma(-D[37], m, L[10]);
      L[11] = m2l_fma(-D[38], m, L[11]);
      L[12] = m2l_fma(-D[40], m, L[12]);
      L[13] = m2l_fma(-D[41], m, L[13]);
      L[14] = m2l_fma(-D[43], m, L[14]);
      L[15] = m2l_fma(-D[44], m, L[15]);
    }
    { const T m = __ldg(Mr + 8);
      L[1] = m2l_fma(-D[14], m, L[1]);
      L[2] = m2l_fma(-D[17], m, L[2]);
      L[3] = m2l_fma(-D[18], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[29], m, L[7]);
      L[8] = m2l_fma(D[30], m, L[8]);
      L[9] = m2l_fma(-D[35], m, L[9]);
      L[10] = m2l_fma(-D[38], m, L[10]);
      L[11] = m2l_fma(-D[39], m, L[11]);
      L[12] = m2l_fma(-D[41], m, L[12]);
      L[13] = m2l_fma(-D[42], m, L[13]);
      L[14] = m2l_fma(-D[44], m, L[14]);
      L[15] = m2l_fma(-D[45], m, L[15]);
    }
    { const T m = __ldg(Mr + 9);
      L[1] = m2l_fma(-D[19], m, L[1]);
      L[2] = m2l_fma(-D[20], m, L[2]);
      L[3] = m2l_fma(-D[21], m, L[3]);
      L[4] = m2l_fma(D[31], m, L[4]);
      L[5] = m2l_fma(D[32], m, L[5]);
      L[6] = m2l_fma(D[33], m, L[6]);
      L[7] = m2l_fma(D[34], m, L[7]);
      L[8] = m2l_fma(D[35], m, L[8]);
    }
    { const T m = __ldg(Mr + 10);
      L[1] = m2l_fma(-D[20], m, L[1]);
      L[2] = m2l_fma(-D[22], m, L[2]);
      L[3] = m2l_fma(-D[23], m, L[3]);
      L[4] = m2l_fma(D[32], m, L[4]);
      L[5] = m2l_fma(D[34], m, L[5]);
      L[6] = m2l_fma(D[35], m, L[6]);
      L[7] = m2l_fma(D[37], m, L[7]);
      L[8] = m2l_fma(D[38], m, L[8]);
    }
    { const T m = __ldg(Mr + 11);
      L[1] = m2l_fma(-D[21], m, L[1]);
      L[2] = m2l_fma(-D[23], m, L[2]);
      L[3] = m2l_fma(-D[24], m, L[3]);
      L[4] = m2l_fma(D[33], m, L[4]);
      L[5] = m2l_fma(D[35], m, L[5]);
      L[6] = m2l_fma(D[36], m, L[6]);
      L[7] = m2l_fma(D[38], m, L[7]);
      L[8] = m2l_fma(D[39], m, L[8]);
    }
    { const T m = __ldg(Mr + 12);
      L[1] = m2l_fma(-D[22], m, L[1]);
      L[2] = m2l_fma(-D[25], m, L[2]);
      L[3] = m2l_fma(-D[26], m, L[3]);
      L[4] = m2l_fma(D[34], m, L[4]);
      L[5] = m2l_fma(D[37], m, L[5]);
      L[6] = m2l_fma(D[38], m, L[6]);
      L[7] = m2l_fma(D[40], m, L[7]);
      L[8] = m2l_fma(D[41], m, L[8]);
    }
    { const T m = __ldg(Mr + 13);
      L[1] = m2l_fma(-D[23], m, L[1]);
      L[2] = m2l_fma(-D[26], m, L[2]);
      L[3] = m2l_fma(-D[27], m, L[3]);
      L[4] = m2l_fma(D[35], m, L[4]);
      L[5] = m2l_fma(D[38], m, L[5]);
      L[6] = m2l_fma(D[39], m, L[6]);
      L[7] = m2l_fma(D[41], m, L[7]);
      L[8] = m2l_fma(D[42], m, L[8]);
    }
    { const T m = __ldg(Mr + 14);
      L[1] = m2l_fma(-D[25], m, L[1]);
      L[2] = m2l_fma(-D[28], m, L[2]);
      L[3] = m2l_fma(-D[29], m, L[3]);
      L[4] = m2l_fma(D[37], m, L[4]);
      L[5] = m2l_fma(D[40], m, L[5]);
      L[6] = m2l_fma(D[41], m, L[6]);
      L[7] = m2l_fma(D[43], m, L[7]);
      L[8] = m2l_fma(D[44], m, L[8]);
    }
    { const T m = __ldg(Mr + 15);
      L[1] = m2l_fma(-D[26], m, L[1]);
      L[2] = m2l_fma(-D[29], m, L[2]);
      L[3] = m2l_fma(-D[30], m, L[3]);
      L[4] = m2l_fma(D[38], m, L[4]);
      L[5] = m2l_fma(D[41], m, L[5]);
      L[6] = m2l_fma(D[42], m, L[6]);
      L[7] = m2l_fma(D[44], m, L[7]);
      L[8] = m2l_fma(D[45], m, L[8]);
    }
    { const T m = __ldg(Mr + 16);
      L[1] = m2l_fma(-D[31], m, L[1]);
      L[2] = m2l_fma(-D[32], m, L[2]);
      L[3] = m2l_fma(-D[33], m, L[3]);
    }
    { const T m = __ldg(Mr + 17);
      L[1] = m2l_fma(-D[32], m, L[1]);
      L[2] = m2l_fma(-D[34], m, L[2]);
      L[3] = m2l_fma(-D[35], m, L[3]);
    }
    { const T m = __ldg(Mr + 18);
      L[1] = m2l_fma(-D[33], m, L[1]);
      L[2] = m2l_fma(-D[35], m, L[2]);
      L[3] = m2l_fma(-D[36], m, L[3]);
    }
    { const T m = __ldg(Mr + 19);
      L[1] = m2l_fma(-D[34], m, L[1]);
      L[2] = m2l_fma(-D[37], m, L[2]);
      L[3] = m2l_fma(-D[38], m, L[3]);
    }
    { const T m = __ldg(Mr + 20);
      L[1] = m2l_fma(-D[35], m, L[1]);
      L[2] = m2l_fma(-D[38], m, L[2]);
      L[3] = m2l_fma(-D[39], m, L[3]);
    }
    { const T m = __ldg(Mr + 21);
      L[1] = m2l_fma(-D[37], m, L[1]);
      L[2] = m2l_fma(-D[40], m, L[2]);
      L[3] = m2l_fma(-D[41], m, L[3]);
    }
    { const T m = __ldg(Mr + 22);
      L[1] = m2l_fma(-D[38], m, L[1]);
      L[2] = m2l_fma(-D[41], m, L[2]);
      L[3] = m2l_fma(-D[42], m, L[3]);
    }
    { const T m = __ldg(Mr + 23);
      L[1] = m2l_fma(-D[40], m, L[1]);
      L[2] = m2l_fma(-D[43], m, L[2]);
      L[3] = m2l_fma(-D[44], m, L[3]);
    }
    { const T m = __ldg(Mr + 24);
      L[1] = m2l_fma(-D[41], m, L[1]);
      L[2] = m2l_fma(-D[44], m, L[2]);
      L[3] = m2l_fma(-D[45], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_reduce_moments_h_5(const T *__restrict__ Ms, T *__restrict__ Mr)
{
    T v0 = Ms[0];
    T v1 = Ms[1];
    T v2 = Ms[2];
    T v3 = Ms[3];
    T v4 = Ms[4];
    T v5 = Ms[5];
    T v6 = Ms[6];
    T v7 = Ms[7];
    T v8 = Ms[8];
    T v9 = Ms[9];
    T v10 = Ms[10];
    T v11 = Ms[11];
    T v12 = Ms[12];
    T v13 = Ms[13];
    T v14 = Ms[14];
    T v15 = Ms[15];
    T v16 = Ms[16];
    T v17 = Ms[17];
    T v18 = Ms[18];
    T v19 = Ms[19];
    T v20 = Ms[20];
    T v21 = Ms[21];
    T v22 = Ms[22];
    T v23 = Ms[23];
    T v24 = Ms[24];
    T v25 = Ms[25];
    T v26 = Ms[26];
    T v27 = Ms[27];
    T v28 = Ms[28];
    T v29 = Ms[29];
    T v30 = Ms[30];
    T v31 = Ms[31];
    T v32 = Ms[32];
    T v33 = Ms[33];
    T v34 = Ms[34];
    T v35 = Ms[35];
    T v36 = Ms[36];
    T v37 = Ms[37];
    T v38 = Ms[38];
    T v39 = Ms[39];
    T v40 = Ms[40];
    T v41 = Ms[41];
    T v42 = Ms[42];
    T v43 = Ms[43];
    T v44 = Ms[44];
    T v45 = Ms[45];
    T v46 = Ms[46];
    T v47 = Ms[47];
    T v48 = Ms[48];
    T v49 = Ms[49];
    T v50 = Ms[50];
    T v51 = Ms[51];
    T v52 = Ms[52];
    T v53 = Ms[53];
    T v54 = Ms[54];
    T v55 = Ms[55];
    v44 -= v55;
    v53 -= v55;
    v25 -= v34;
    v32 -= v34;
    v40 -= v49;
    v47 -= v49;
    v43 -= v54;
    v52 -= v54;
    v12 -= v19;
    v17 -= v19;
    v22 -= v29;
    v27 -= v29;
    v24 -= v33;
    v31 -= v33;
    v37 -= v44;
    v42 -= v44;
    v39 -= v48;
    v46 -= v48;
    v42 -= v53;
    v51 -= v53;
    v4 -= v9;
    v7 -= v9;
    v10 -= v15;
    v13 -= v15;
    v11 -= v18;
    v16 -= v18;
    v20 -= v25;
    v23 -= v25;
    v21 -= v28;
    v26 -= v28;
    v23 -= v32;
    v30 -= v32;
    v35 -= v40;
    v38 -= v40;
    v36 -= v43;
    v41 -= v43;
    v38 -= v47;
    v45 -= v47;
    v41 -= v52;
    v50 -= v52;
    Mr[0] = v0;
    Mr[1] = v1;
    Mr[2] = v2;
    Mr[3] = v3;
    Mr[4] = v4;
    Mr[5] = v5;
    Mr[6] = v6;
    Mr[7] = v7;
    Mr[8] = v8;
    Mr[9] = v10;
    Mr[10] = v11;
    Mr[11] = v12;
    Mr[12] = v13;
    Mr[13] = v14;
    Mr[14] = v16;
    Mr[15] = v17;
    Mr[16] = v20;
    Mr[17] = v21;
    Mr[18] = v22;
    Mr[19] = v23;
    Mr[20] = v24;
    Mr[21] = v26;
    Mr[22] = v27;
    Mr[23] = v30;
    Mr[24] = v31;
    Mr[25] = v35;
    Mr[26] = v36;
    Mr[27] = v37;
    Mr[28] = v38;
    Mr[29] = v39;
    Mr[30] = v41;
    Mr[31] = v42;
    Mr[32] = v45;
    Mr[33] = v46;
    Mr[34] = v50;
    Mr[35] = v51;
}

template <class T> __device__ __forceinline__ void m2l_complete_locals_h_5(const T *__restrict__ Lr, T *__restrict__ L)
{
    const T v0 = Lr[0];
    L[0] = v0;
    const T v1 = Lr[1];
    L[1] = v1;
    const T v2 = Lr[2];
    L[2] = v2;
    const T v3 = Lr[3];
    L[3] = v3;
    const T v4 = Lr[4];
    L[4] = v4;
    const T v5 = Lr[5];
    L[5] = v5;
    const T v6 = Lr[6];
    L[6] = v6;
    const T v7 = Lr[7];
    L[7] = v7;
    const T v8 = Lr[8];
    L[8] = v8;
    const T v9 = -v4 - v7;
    L[9] = v9;
    const T v10 = Lr[9];
    L[10] = v10;
    const T v11 = Lr[10];
    L[11] = v11;
    const T v12 = Lr[11];
    L[12] = v12;
    const T v13 = Lr[12];
    L[13] = v13;
    const T v14 = Lr[13];
    L[14] = v14;
    const T v15 = -v10 - v13;
    L[15] = v15;
    const T v16 = Lr[14];
    L[16] = v16;
    const T v17 = Lr[15];
    L[17] = v17;
    const T v18 = -v11 - v16;
    L[18] = v18;
    const T v19 = -v12 - v17;
    L[19] = v19;
    const T v20 = Lr[16];
    L[20] = v20;
    const T v21 = Lr[17];
    L[21] = v21;
    const T v22 = Lr[18];
    L[22] = v22;
    const T v23 = Lr[19];
    L[23] = v23;
    const T v24 = Lr[20];
    L[24] = v24;
    const T v25 = -v20 - v23;
    L[25] = v25;
    const T v26 = Lr[21];
    L[26] = v26;
    const T v27 = Lr[22];
    L[27] = v27;
    const T v28 = -v21 - v26;
    L[28] = v28;
    const T v29 = -v22 - v27;
    L[29] = v29;
    const T v30 = Lr[23];
    L[30] = v30;
    const T v31 = Lr[24];
    L[31] = v31;
    const T v32 = -v23 - v30;
    L[32] = v32;
    const T v33 = -v24 - v31;
    L[33] = v33;
    const T v34 = -v25 - v32;
    L[34] = v34;
    const T v35 = Lr[25];
    L[35] = v35;
    const T v36 = Lr[26];
    L[36] = v36;
    const T v37 = Lr[27];
    L[37] = v37;
    const T v38 = Lr[28];
    L[38] = v38;
    const T v39 = Lr[29];
    L[39] = v39;
    const T v40 = -v35 - v38;
    L[40] = v40;
    const T v41 = Lr[30];
    L[41] = v41;
    const T v42 = Lr[31];
    L[42] = v42;
    const T v43 = -v36 - v41;
    L[43] = v43;
    const T v44 = -v37 - v42;
    L[44] = v44;
    const T v45 = Lr[32];
    L[45] = v45;
    const T v46 = Lr[33];
    L[46] = v46;
    const T v47 = -v38 - v45;
    L[47] = v47;
    const T v48 = -v39 - v46;
    L[48] = v48;
    const T v49 = -v40 - v47;
    L[49] = v49;
    const T v50 = Lr[34];
    L[50] = v50;
    const T v51 = Lr[35];
    L[51] = v51;
    const T v52 = -v41 - v50;
    L[52] = v52;
    const T v53 = -v42 - v51;
    L[53] = v53;
    const T v54 = -v43 - v52;
    L[54] = v54;
    const T v55 = -v44 - v53;
    L[55] = v55;
}

template <class T> __device__ __forceinline__ void m2l_dtensor_h_6(T dx, T dy, T dz, T (&D)[64])
{
    const T s2 = m2l_fma(dx, dx, m2l_fma(dy, dy, dz * dz));
    const T si = m2l_rsqrt(s2);
    const T si2 = si * si;
    const T f0 = -si;
    const T f1 = T(-1) * f0 * si2;
    const T f2 = T(-3) * f1 * si2;
    const T f3 = T(-5) * f2 * si2;
    const T f4 = T(-7) * f3 * si2;
    const T f5 = T(-9) * f4 * si2;
    const T f6 = T(-11) * f5 * si2;
    const T r_0_0 = f0;
    const T r_1_0 = f1;
    const T r_2_0 = f2;
    const T r_3_0 = f3;
    const T r_4_0 = f4;
    const T r_5_0 = f5;
    const T r_6_0 = f6;
    const T r_0_1 = dx * r_1_0;
    const T r_1_1 = dx * r_2_0;
    const T r_2_1 = dx * r_3_0;
    const T r_3_1 = dx * r_4_0;
    const T r_4_1 = dx * r_5_0;
    const T r_5_1 = dx * r_6_0;
    const T r_0_2 = dy * r_1_0;
    const T r_1_2 = dy * r_2_0;
    const T r_2_2 = dy * r_3_0;
    const T r_3_2 = dy * r_4_0;
    const T r_4_2 = dy * r_5_0;
    const T r_5_2 = dy * r_6_0;
    const T r_0_4 = m2l_fma(T(1), r_1_0, dx * r_1_1);
    const T r_1_4 = m2l_fma(T(1), r_2_0, dx * r_2_1);
    const T r_2_4 = m2l_fma(T(1), r_3_0, dx * r_3_1);
    const T r_3_4 = m2l_fma(T(1), r_4_0, dx * r_4_1);
    const T r_4_4 = m2l_fma(T(1), r_5_0, dx * r_5_1);
    const T r_0_5 = dx * r_1_2;
    const T r_1_5 = dx * r_2_2;
    const T r_2_5 = dx * r_3_2;
    const T r_3_5 = dx * r_4_2;
    const T r_4_5 = dx * r_5_2;
    const T r_0_7 = m2l_fma(T(1), r_1_0, dy * r_1_2);
    const T r_1_7 = m2l_fma(T(1), r_2_0, dy * r_2_2);
    const T r_2_7 = m2l_fma(T(1), r_3_0, dy * r_3_2);
    const T r_3_7 = m2l_fma(T(1), r_4_0, dy * r_4_2);
    const T r_4_7 = m2l_fma(T(1), r_5_0, dy * r_5_2);
    const T r_0_10 = m2l_fma(T(2), r_1_1, dx * r_1_4);
    const T r_1_10 = m2l_fma(T(2), r_2_1, dx * r_2_4);
    const T r_2_10 = m2l_fma(T(2), r_3_1, dx * r_3_4);
    const T r_3_10 = m2l_fma(T(2), r_4_1, dx * r_4_4);
    const T r_0_11 = m2l_fma(T(1), r_1_2, dx * r_1_5);
    const T r_1_11 = m2l_fma(T(1), r_2_2, dx * r_2_5);
    const T r_2_11 = m2l_fma(T(1), r_3_2, dx * r_3_5);
    const T r_3_11 = m2l_fma(T(1), r_4_2, dx * r_4_5);
    const T r_0_13 = dx * r_1_7;
    const T r_1_13 = dx * r_2_7;
    const T r_2_13 = dx * r_3_7;
    const T r_3_13 = dx * r_4_7;
    const T r_0_16 = m2l_fma(T(2), r_1_2, dy * r_1_7);
    const T r_1_16 = m2l_fma(T(2), r_2_2, dy * r_2_7);
    const T r_2_16 = m2l_fma(T(2), r_3_2, dy * r_3_7);
    const T r_3_16 = m2l_fma(T(2), r_4_2, dy * r_4_7);
    const T r_0_20 = m2l_fma(T(3), r_1_4, dx * r_1_10);
    const T r_1_20 = m2l_fma(T(3), r_2_4, dx * r_2_10);
    const T r_2_20 = m2l_fma(T(3), r_3_4, dx * r_3_10);
    const T r_0_21 = m2l_fma(T(2), r_1_5, dx * r_1_11);
    const T r_1_21 = m2l_fma(T(2), r_2_5, dx * r_2_11);
    const T r_2_21 = m2l_fma(T(2), r_3_5, dx * r_3_11);
    const T r_0_23 = m2l_fma(T(1), r_1_7, dx * r_1_13);
    const T r_1_23 = m2l_fma(T(1), r_2_7, dx * r_2_13);
    const T r_2_23 = m2l_fma(T(1), r_3_7, dx * r_3_13);
    const T r_0_26 = dx * r_1_16;
    const T r_1_26 = dx * r_2_16;
    const T r_2_26 = dx * r_3_16;
    const T r_0_30 = m2l_fma(T(3), r_1_7, dy * r_1_16);
    const T r_1_30 = m2l_fma(T(3), r_2_7, dy * r_2_16);
    const T r_2_30 = m2l_fma(T(3), r_3_7, dy * r_3_16);
    const T r_0_35 = m2l_fma(T(4), r_1_10, dx * r_1_20);
    const T r_1_35 = m2l_fma(T(4), r_2_10, dx * r_2_20);
    const T r_0_36 = m2l_fma(T(3), r_1_11, dx * r_1_21);
    const T r_1_36 = m2l_fma(T(3), r_2_11, dx * r_2_21);
    const T r_0_38 = m2l_fma(T(2), r_1_13, dx * r_1_23);
    const T r_1_38 = m2l_fma(T(2), r_2_13, dx * r_2_23);
    const T r_0_41 = m2l_fma(T(1), r_1_16, dx * r_1_26);
    const T r_1_41 = m2l_fma(T(1), r_2_16, dx * r_2_26);
    const T r_0_45 = dx * r_1_30;
    const T r_1_45 = dx * r_2_30;
    const T r_0_50 = m2l_fma(T(4), r_1_16, dy * r_1_30);
    const T r_1_50 = m2l_fma(T(4), r_2_16, dy * r_2_30);
    const T r_0_56 = m2l_fma(T(5), r_1_20, dx * r_1_35);
    const T r_0_57 = m2l_fma(T(4), r_1_21, dx * r_1_36);
    const T r_0_59 = m2l_fma(T(3), r_1_23, dx * r_1_38);
    const T r_0_62 = m2l_fma(T(2), r_1_26, dx * r_1_41);
    const T r_0_66 = m2l_fma(T(1), r_1_30, dx * r_1_45);
    const T r_0_71 = dx * r_1_50;
    const T r_0_77 = m2l_fma(T(5), r_1_30, dy * r_1_50);
    D[0] = r_0_0;
    D[1] = r_0_1;
    D[2] = r_0_2;
    D[3] = dz * r_1_0;
    D[4] = r_0_4;
    D[5] = r_0_5;
    D[6] = dz * r_1_1;
    D[7] = r_0_7;
    D[8] = dz * r_1_2;
    D[10] = r_0_10;
    D[11] = r_0_11;
    D[12] = dz * r_1_4;
    D[13] = r_0_13;
    D[14] = dz * r_1_5;
    D[16] = r_0_16;
    D[17] = dz * r_1_7;
    D[19] = r_0_20;
    D[20] = r_0_21;
    D[21] = dz * r_1_10;
    D[22] = r_0_23;
    D[23] = dz * r_1_11;
    D[25] = r_0_26;
    D[26] = dz * r_1_13;
    D[28] = r_0_30;
    D[29] = dz * r_1_16;
    D[31] = r_0_35;
    D[32] = r_0_36;
    D[33] = dz * r_1_20;
    D[34] = r_0_38;
    D[35] = dz * r_1_21;
    D[37] = r_0_41;
    D[38] = dz * r_1_23;
    D[40] = r_0_45;
    D[41] = dz * r_1_26;
    D[43] = r_0_50;
    D[44] = dz * r_1_30;
    D[46] = r_0_56;
    D[47] = r_0_57;
    D[48] = dz * r_1_35;
    D[49] = r_0_59;
    D[50] = dz * r_1_36;
    D[52] = r_0_62;
    D[53] = dz * r_1_38;
    D[55] = r_0_66;
    D[56] = dz * r_1_41;
    D[58] = r_0_71;
    D[59] = dz * r_1_45;
    D[61] = r_0_77;
    D[62] = dz * r_1_50;
    D[9] = -D[4] - D[7];
    D[15] = -D[10] - D[13];
    D[18] = -D[11] - D[16];
    D[24] = -D[19] - D[22];
    D[27] = -D[20] - D[25];
    D[30] = -D[22] - D[28];
    D[36] = -D[31] - D[34];
    D[39] = -D[32] - D[37];
    D[42] = -D[34] - D[40];
    D[45] = -D[37] - D[43];
    D[51] = -D[46] - D[49];
    D[54] = -D[47] - D[52];
    D[57] = -D[49] - D[55];
    D[60] = -D[52] - D[58];
    D[63] = -D[55] - D[61];
}

template <class T> __device__ __forceinline__ void m2l_side_a_h_6(const T (&D)[64], const T *__restrict__ Mr, T rho, T (&L)[49])
{
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[0] = D[0] * m;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[10] * m;
      L[10] = D[11] * m;
      L[11] = D[12] * m;
      L[12] = D[13] * m;
      L[13] = D[14] * m;
      L[14] = D[16] * m;
      L[15] = D[17] * m;
      L[16] = D[19] * m;
      L[17] = D[20] * m;
      L[18] = D[21] * m;
      L[19] = D[22] * m;
      L[20] = D[23] * m;
      L[21] = D[25] * m;
      L[22] = D[26] * m;
      L[23] = D[28] * m;
      L[24] = D[29] * m;
      L[25] = D[31] * m;
      L[26] = D[32] * m;
      L[27] = D[33] * m;
      L[28] = D[34] * m;
      L[29] = D[35] * m;
      L[30] = D[37] * m;
      L[31] = D[38] * m;
      L[32] = D[40] * m;
      L[33] = D[41] * m;
      L[34] = D[43] * m;
      L[35] = D[44] * m;
      L[36] = D[46] * m;
      L[37] = D[47] * m;
      L[38] = D[48] * m;
      L[39] = D[49] * m;
      L[40] = D[50] * m;
      L[41] = D[52] * m;
      L[42] = D[53] * m;
      L[43] = D[55] * m;
      L[44] = D[56] * m;
      L[45] = D[58] * m;
      L[46] = D[59] * m;
      L[47] = D[61] * m;
      L[48] = D[62] * m;
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 1) * rp;
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(D[20], m, L[10]);
      L[11] = m2l_fma(D[21], m, L[11]);
      L[12] = m2l_fma(D[22], m, L[12]);
      L[13] = m2l_fma(D[23], m, L[13]);
      L[14] = m2l_fma(D[25], m, L[14]);
      L[15] = m2l_fma(D[26], m, L[15]);
      L[16] = m2l_fma(D[31], m, L[16]);
      L[17] = m2l_fma(D[32], m, L[17]);
      L[18] = m2l_fma(D[33], m, L[18]);
      L[19] = m2l_fma(D[34], m, L[19]);
      L[20] = m2l_fma(D[35], m, L[20]);
      L[21] = m2l_fma(D[37], m, L[21]);
      L[22] = m2l_fma(D[38], m, L[22]);
      L[23] = m2l_fma(D[40], m, L[23]);
      L[24] = m2l_fma(D[41], m, L[24]);
      L[25] = m2l_fma(D[46], m, L[25]);
      L[26] = m2l_fma(D[47], m, L[26]);
      L[27] = m2l_fma(D[48], m, L[27]);
      L[28] = m2l_fma(D[49], m, L[28]);
      L[29] = m2l_fma(D[50], m, L[29]);
      L[30] = m2l_fma(D[52], m, L[30]);
      L[31] = m2l_fma(D[53], m, L[31]);
      L[32] = m2l_fma(D[55], m, L[32]);
      L[33] = m2l_fma(D[56], m, L[33]);
      L[34] = m2l_fma(D[58], m, L[34]);
      L[35] = m2l_fma(D[59], m, L[35]);
    }
    { const T m = -__ldg(Mr + 2) * rp;
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[20], m, L[9]);
      L[10] = m2l_fma(D[22], m, L[10]);
      L[11] = m2l_fma(D[23], m, L[11]);
      L[12] = m2l_fma(D[25], m, L[12]);
      L[13] = m2l_fma(D[26], m, L[13]);
      L[14] = m2l_fma(D[28], m, L[14]);
      L[15] = m2l_fma(D[29], m, L[15]);
      L[16] = m2l_fma(D[32], m, L[16]);
      L[17] = m2l_fma(D[34], m, L[17]);
      L[18] = m2l_fma(D[35], m, L[18]);
      L[19] = m2l_fma(D[37], m, L[19]);
      L[20] = m2l_fma(D[38], m, L[20]);
      L[21] = m2l_fma(D[40], m, L[21]);
      L[22] = m2l_fma(D[41], m, L[22]);
      L[23] = m2l_fma(D[43], m, L[23]);
      L[24] = m2l_fma(D[44], m, L[24]);
      L[25] = m2l_fma(D[47], m, L[25]);
      L[26] = m2l_fma(D[49], m, L[26]);
      L[27] = m2l_fma(D[50], m, L[27]);
      L[28] = m2l_fma(D[52], m, L[28]);
      L[29] = m2l_fma(D[53], m, L[29]);
      L[30] = m2l_fma(D[55], m, L[30]);
      L[31] = m2l_fma(D[56], m, L[31]);
      L[32] = m2l_fma(D[58], m, L[32]);
      L[33] = m2l_fma(D[59], m, L[33]);
      L[34] = m2l_fma(D[61], m, L[34]);
      L[35] = m2l_fma(D[62], m, L[35]);
    }
    { const T m = -__ldg(Mr + 3) * rp;
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[21], m, L[9]);
      L[10] = m2l_fma(D[23], m, L[10]);
      L[11] = m2l_fma(D[24], m, L[11]);
      L[12] = m2l_fma(D[26], m, L[12]);
      L[13] = m2l_fma(D[27], m, L[13]);
      L[14] = m2l_fma(D[29], m, L[14]);
      L[15] = m2l_fma(D[30], m, L[15]);
      L[16] = m2l_fma(D[33], m, L[16]);
      L[17] = m2l_fma(D[35], m, L[17]);
      L[18] = m2l_fma(D[36], m, L[18]);
      L[19] = m2l_fma(D[38], m, L[19]);
      L[20] = m2l_fma(D[39], m, L[20]);
      L[21] = m2l_fma(D[41], m, L[21]);
      L[22] = m2l_fma(D[42], m, L[22]);
      L[23] = m2l_fma(D[44], m, L[23]);
      L[24] = m2l_fma(D[45], m, L[24]);
      L[25] = m2l_fma(D[48], m, L[25]);
      L[26] = m2l_fma(D[50], m, L[26]);
      L[27] = m2l_fma(D[51], m, L[27]);
      L[28] = m2l_fma(D[53], m, L[28]);
      L[29] = m2l_fma(D[54], m, L[29]);
      L[30] = m2l_fma(D[56], m, L[30]);
      L[31] = m2l_fma(D[57], m, L[31]);
      L[32] = m2l_fma(D[59], m, L[32]);
      L[33] = m2l_fma(D[60], m, L[33]);
      L[34] = m2l_fma(D[62], m, L[34]);
      L[35] = m2l_fma(D[63], m, L[35]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 4) * rp;
      L[0] = m2l_fma(D[4], m, L[0]);
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
      L[4] = m2l_fma(D[19], m, L[4]);
      L[5] = m2l_fma(D[20], m, L[5]);
      L[6] = m2l_fma(D[21], m, L[6]);
      L[7] = m2l_fma(D[22], m, L[7]);
      L[8] = m2l_fma(D[23], m, L[8]);
      L[9] = m2l_fma(D[31], m, L[9]);
      L[10] = m2l_fma(D[32], m, L[10]);
      L[11] = m2l_fma(D[33], m, L[11]);
      L[12] = m2l_fma(D[34], m, L[12]);
      L[13] = m2l_fma(D[35], m, L[13]);
      L[14] = m2l_fma(D[37], m, L[14]);
      L[15] = m2l_fma(D[38], m, L[15]);
      L[16] = m2l_fma(D[46], m, L[16]);
      L[17] = m2l_fma(D[47], m, L[17]);
      L[18] = m2l_fma(D[48], m, L[18]);
      L[19] = m2l_fma(D[49], m, L[19]);
      L[20] = m2l_fma(D[50], m, L[20]);
      L[21] = m2l_fma(D[52], m, L[21]);
      L[22] = m2l_fma(D[53], m, L[22]);
      L[23] = m2l_fma(D[55], m, L[23]);
      L[24] = m2l_fma(D[56], m, L[24]);
    }
    { const T m = __ldg(Mr + 5) * rp;
      L[0] = m2l_fma(D[5], m, L[0]);
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[22], m, L[5]);
      L[6] = m2l_fma(D[23], m, L[6]);
      L[7] = m2l_fma(D[25], m, L[7]);
      L[8] = m2l_fma(D[26], m, L[8]);
      L[9] = m2l_fma(D[32], m, L[9]);
      L[10] = m2l_fma(D[34], m, L[10]);
      L[11] = m2l_fma(D[35], m, L[11]);
      L[12] = m2l_fma(D[37], m, L[12]);
      L[13] = m2l_fma(D[38], m, L[13]);
      L[14] = m2l_fma(D[40], m, L[14]);
      L[15] = m2l_fma(D[41], m, L[15]);
      L[16] = m2l_fma(D[47], m, L[16]);
      L[17] = m2l_fma(D[49], m, L[17]);
      L[18] = m2l_fma(D[50], m, L[18]);
      L[19] = m2l_fma(D[52], m, L[19]);
      L[20] = m2l_fma(D[53], m, L[20]);
      L[21] = m2l_fma(D[55], m, L[21]);
      L[22] = m2l_fma(D[56], m, L[22]);
      L[23] = m2l_fma(D[58], m, L[23]);
      L[24] = m2l_fma(D[59], m, L[24]);
    }
    { const T m = __ldg(Mr + 6) * rp;
      L[0] = m2l_fma(D[6], m, L[0]);
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(D[33], m, L[9]);
      L[10] = m2l_fma(D[35], m, L[10]);
      L[11] = m2l_fma(D[36], m, L[11]);
      L[12] = m2l_fma(D[38], m, L[12]);
      L[13] = m2l_fma(D[39], m, L[13]);
      L[14] = m2l_fma(D[41], m, L[14]);
      L[15] = m2l_fma(D[42], m, L[15]);
      L[16] = m2l_fma(D[48], m, L[16]);
      L[17] = m2l_fma(D[50], m, L[17]);
      L[18] = m2l_fma(D[51], m, L[18]);
      L[19] = m2l_fma(D[53], m, L[19]);
      L[20] = m2l_fma(D[54], m, L[20]);
      L[21] = m2l_fma(D[56], m, L[21]);
      L[22] = m2l_fma(D[57], m, L[22]);
      L[23] = m2l_fma(D[59], m, L[23]);
      L[24] = m2l_fma(D[60], m, L[24]);
    }
    { const T m = __ldg(Mr + 7) * rp;
      L[0] = m2l_fma(D[7], m, L[0]);
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[25], m, L[5]);
      L[6] = m2l_fma(D[26], m, L[6]);
      L[7] = m2l_fma(D[28], m, L[7]);
      L[8] = m2l_fma(D[29], m, L[8]);
      L[9] = m2l_fma(D[34], m, L[9]);
      L[10] = m2l_fma(D[37], m, L[10]);
      L[11] = m2l_fma(D[38], m, L[11]);
      L[12] = m2l_fma(D[40], m, L[12]);
      L[13] = m2l_fma(D[41], m, L[13]);
      L[14] = m2l_fma(D[43], m, L[14]);
      L[15] = m2l_fma(D[44], m, L[15]);
      L[16] = m2l_fma(D[49], m, L[16]);
      L[17] = m2l_fma(D[52], m, L[17]);
      L[18] = m2l_fma(D[53], m, L[18]);
      L[19] = m2l_fma(D[55], m, L[19]);
      L[20] = m2l_fma(D[56], m, L[20]);
      L[21] = m2l_fma(D[58], m, L[21]);
      L[22] = m2l_fma(D[59], m, L[22]);
      L[23] = m2l_fma(D[61], m, L[23]);
      L[24] = m2l_fma(D[62], m, L[24]);
    }
    { const T m = __ldg(Mr + 8) * rp;
      L[0] = m2l_fma(D[8], m, L[0]);
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[29], m, L[7]);
      L[8] = m2l_fma(D[30], m, L[8]);
      L[9] = m2l_fma(D[35], m, L[9]);
      L[10] = m2l_fma(D[38], m, L[10]);
      L[11] = m2l_fma(D[39], m, L[11]);
      L[12] = m2l_fma(D[41], m, L[12]);
      L[13] = m2l_fma(D[42], m, L[13]);
      L[14] = m2l_fma(D[44], m, L[14]);
      L[15] = m2l_fma(D[45], m, L[15]);
      L[16] = m2l_fma(D[50], m, L[16]);
      L[17] = m2l_fma(D[53], m, L[17]);
      L[18] = m2l_fma(D[54], m, L[18]);
      L[19] = m2l_fma(D[56], m, L[19]);
      L[20] = m2l_fma(D[57], m, L[20]);
      L[21] = m2l_fma(D[59], m, L[21]);
      L[22] = m2l_fma(D[60], m, L[22]);
      L[23] = m2l_fma(D[62], m, L[23]);
      L[24] = m2l_fma(D[63], m, L[24]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 9) * rp;
      L[0] = m2l_fma(D[10], m, L[0]);
      L[1] = m2l_fma(D[19], m, L[1]);
      L[2] = m2l_fma(D[20], m, L[2]);
      L[3] = m2l_fma(D[21], m, L[3]);
      L[4] = m2l_fma(D[31], m, L[4]);
      L[5] = m2l_fma(D[32], m, L[5]);
      L[6] = m2l_fma(D[33], m, L[6]);
      L[7] = m2l_fma(D[34], m, L[7]);
      L[8] = m2l_fma(D[35], m, L[8]);
      L[9] = m2l_fma(D[46], m, L[9]);
      L[10] = m2l_fma(D[47], m, L[10]);
      L[11] = m2l_fma(D[48], m, L[11]);
      L[12] = m2l_fma(D[49], m, L[12]);
      L[13] = m2l_fma(D[50], m, L[13]);
      L[14] = m2l_fma(D[52], m, L[14]);
      L[15] = m2l_fma(D[53], m, L[15]);
    }
    { const T m = -__ldg(Mr + 10) * rp;
      L[0] = m2l_fma(D[11], m, L[0]);
      L[1] = m2l_fma(D[20], m, L[1]);
      L[2] = m2l_fma(D[22], m, L[2]);
      L[3] = m2l_fma(D[23], m, L[3]);
      L[4] = m2l_fma(D[32], m, L[4]);
      L[5] = m2l_fma(D[34], m, L[5]);
      L[6] = m2l_fma(D[35], m, L[6]);
      L[7] = m2l_fma(D[37], m, L[7]);
      L[8] = m2l_fma(D[38], m, L[8]);
      L[9] = m2l_fma(D[47], m, L[9]);
      L[10] = m2l_fma(D[49], m, L[10]);
      L[11] = m2l_fma(D[50], m, L[11]);
      L[12] = m2l_fma(D[52], m, L[12]);
      L[13] = m2l_fma(D[53], m, L[13]);
      L[14] = m2l_fma(D[55], m, L[14]);
      L[15] = m2l_fma(D[56], m, L[15]);
    }
    { const T m = -__ldg(Mr + 11) * rp;
      L[0] = m2l_fma(D[12], m, L[0]);
      L[1] = m2l_fma(D[21], m, L[1]);
      L[2] = m2l_fma(D[23], m, L[2]);
      L[3] = m2l_fma(D[24], m, L[3]);
      L[4] = m2l_fma(D[33], m, L[4]);
      L[5] = m2l_fma(D[35], m, L[5]);
      L[6] = m2l_fma(D[36], m, L[6]);
      L[7] = m2l_fma(D[38], m, L[7]);
      L[8] = m2l_fma(D[39], m, L[8]);
      L[9] = m2l_fma(D[48], m, L[9]);
      L[10] = m2l_fma(D[50], m, L[10]);
      L[11] = m2l_fma(D[51], m, L[11]);
      L[12] = m2l_fma(D[53], m, L[12]);
      L[13] = m2l_fma(D[54], m, L[13]);
      L[14] = m2l_fma(D[56], m, L[14]);
      L[15] = m2l_fma(D[57], m, L[15]);
    }
    { const T m = -__ldg(Mr + 12) * rp;
      L[0] = m2l_fma(D[13], m, L[0]);
      L[1] = m2l_fma(D[22], m, L[1]);
      L[2] = m2l_fma(D[25], m, L[2]);
      L[3] = m2l_fma(D[26], m, L[3]);
      L[4] = m2l_fma(D[34], m, L[4]);
      L[5] = m2l_fma(D[37], m, L[5]);
      L[6] = m2l_fma(D[38], m, L[6]);
      L[7] = m2l_fma(D[40], m, L[7]);
      L[8] = m2l_fma(D[41], m, L[8]);
      L[9] = m2l_fma(D[49], m, L[9]);
      L[10] = m2l_fma(D[52], m, L[10]);
      L[11] = m2l_fma(D[53], m, L[11]);
      L[12] = m2l_fma(D[55], m, L[12]);
      L[13] = m2l_fma(D[56], m, L[13]);
      L[14] = m2l_fma(D[58], m, L[14]);
      L[15] = m2l_fma(D[59], m, L[15]);
    }
    { const T m = -__ldg(Mr + 13) * rp;
      L[0] = m2l_fma(D[14], m, L[0]);
      L[1] = m2l_fma(D[23], m, L[1]);
      L[2] = m2l_fma(D[26], m, L[2]);
      L[3] = m2l_fma(D[27], m, L[3]);
      L[4] = m2l_fma(D[35], m, L[4]);
      L[5] = m2l_fma(D[38], m, L[5]);
      L[6] = m2l_fma(D[39], m, L[6]);
      L[7] = m2l_fma(D[41], m, L[7]);
      L[8] = m2l_fma(D[42], m, L[8]);
      L[9] = m2l_fma(D[50], m, L[9]);
      L[10] = m2l_fma(D[53], m, L[10]);
      L[11] = m2l_fma(D[54], m, L[11]);
      L[12] = m2l_fma(D[56], m, L[12]);
      L[13] = m2l_fma(D[57], m, L[13]);
      L[14] = m2l_fma(D[59], m, L[14]);
      L[15] = m2l_fma(D[60], m, L[15]);
    }
    { const T m = -__ldg(Mr + 14) * rp;
      L[0] = m2l_fma(D[16], m, L[0]);
      L[1] = m2l_fma(D[25], m, L[1]);
      L[2] = m2l_fma(D[28], m, L[2]);
      L[3] = m2l_fma(D[29], m, L[3]);
      L[4] = m2l_fma(D[37], m, L[4]);
      L[5] = m2l_fma(D[40], m, L[5]);
      L[6] = m2l_fma(D[41], m, L[6]);
      L[7] = m2l_fma(D[43], m, L[7]);
      L[8] = m2l_fma(D[44], m, L[8]);
      L[9] = m2l_fma(D[52], m, L[9]);
      L[10] = m2l_fma(D[55], m, L[10]);
      L[11] = m2l_fma(D[56], m, L[11]);
      L[12] = m2l_fma(D[58], m, L[12]);
      L[13] = m2l_fma(D[59], m, L[13]);
      L[14] = m2l_fma(D[61], m, L[14]);
      L[15] = m2l_fma(D[62], m, L[15]);
    }
    { const T m = -__ldg(Mr + 15) * rp;
      L[0] = m2l_fma(D[17], m, L[0]);
      L[1] = m2l_fma(D[26], m, L[1]);
      L[2] = m2l_fma(D[29], m, L[2]);
      L[3] = m2l_fma(D[30], m, L[3]);
      L[4] = m2l_fma(D[38], m, L[4]);
      L[5] = m2l_fma(D[41], m, L[5]);
      L[6] = m2l_fma(D[42], m, L[6]);
      L[7] = m2l_fma(D[44], m, L[7]);
      L[8] = m2l_fma(D[45], m, L[8]);
      L[9] = m2l_fma(D[53], m, L[9]);
      L[10] = m2l_fma(D[56], m, L[10]);
      L[11] = m2l_fma(D[57], m, L[11]);
      L[12] = m2l_fma(D[59], m, L[12]);
      L[13] = m2l_fma(D[60], m, L[13]);
      L[14] = m2l_fma(D[62], m, L[14]);
      L[15] = m2l_fma(D[63], m, L[15]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 16) * rp;
      L[0] = m2l_fma(D[19], m, L[0]);
      L[1] = m2l_fma(D[31], m, L[1]);
      L[2] = m2l_fma(D[32], m, L[2]);
      L[3] = m2l_fma(D[33], m, L[3]);
      L[4] = m2l_fma(D[46], m, L[4]);
      L[5] = m2l_fma(D[47], m, L[5]);
      L[6] = m2l_fma(D[48], m, L[6]);
      L[7] = m2l_fma(D[49], m, L[7]);
      L[8] = m2l_fma(D[50], m, L[8]);
    }
    { const T m = __ldg(Mr + 17) * rp;
      L[0] = m2l_fma(D[20], m, L[0]);
      L[1] = m2l_fma(D[32], m, L[1]);
      L[2] = m2l_fma(D[34], m, L[2]);
      L[3] = m2l_fma(D[35], m, L[3]);
      L[4] = m2l_fma(D[47], m, L[4]);
      L[5] = m2l_fma(D[49], m, L[5]);
      L[6] = m2l_fma(D[50], m, L[6]);
      L[7] = m2l_fma(D[52], m, L[7]);
      L[8] = m2l_fma(D[53], m, L[8]);
    }
    { const T m = __ldg(Mr + 18) * rp;
      L[0] = m2l_fma(D[21], m, L[0]);
      L[1] = m2l_fma(D[33], m, L[1]);
      L[2] = m2l_fma(D[35], m, L[2]);
      L[3] = m2l_fma(D[36], m, L[3]);
      L[4] = m2l_fma(D[48], m, L[4]);
      L[5] = m2l_fma(D[50], m, L[5]);
      L[6] = m2l_fma(D[51], m, L[6]);
      L[7] = m2l_fma(D[53], m, L[7]);
      L[8] = m2l_fma(D[54], m, L[8]);
    }
    { const T m = __ldg(Mr + 19) * rp;
      L[0] = m2l_fma(D[22], m, L[0]);
      L[1] = m2l_fma(D[34], m, L[1]);
      L[2] = m2l_fma(D[37], m, L[2]);
      L[3] = m2l_fma(D[38], m, L[3]);
      L[4] = m2l_fma(D[49], m, L[4]);
      L[5] = m2l_fma(D[52], m, L[5]);
      L[6] = m2l_fma(D[53], m, L[6]);
      L[7] = m2l_fma(D[55], m, L[7]);
      L[8] = m2l_fma(D[56], m, L[8]);
    }
    { const T m = __ldg(Mr + 20) * rp;
      L[0] = m2l_fma(D[23], m, L[0]);
      L[1] = m2l_fma(D[35], m, L[1]);
      L[2] = m2l_fma(D[38], m, L[2]);
      L[3] = m2l_fma(D[39], m, L[3]);
      L[4] = m2l_fma(D[50], m, L[4]);
      L[5] = m2l_fma(D[53], m, L[5]);
      L[6] = m2l_fma(D[54], m, L[6]);
      L[7] = m2l_fma(D[56], m, L[7]);
      L[8] = m2l_fma(D[57], m, L[8]);
    }
    { const T m = __ldg(Mr + 21) * rp;
      L[0] = m2l_fma(D[25], m, L[0]);
      L[1] = m2l_fma(D[37], m, L[1]);
      L[2] = m2l_fma(D[40], m, L[2]);
      L[3] = m2l_fma(D[41], m, L[3]);
      L[4] = m2l_fma(D[52], m, L[4]);
      L[5] = m2l_fma(D[55], m, L[5]);
      L[6] = m2l_fma(D[56], m, L[6]);
      L[7] = m2l_fma(D[58], m, L[7]);
      L[8] = m2l_fma(D[59], m, L[8]);
    }
    { const T m = __ldg(Mr + 22) * rp;
      L[0] = m2l_fma(D[26], m, L[0]);
      L[1] = m2l_fma(D[38], m, L[1]);
      L[2] = m2l_fma(D[41], m, L[2]);
      L[3] = m2l_fma(D[42], m, L[3]);
      L[4] = m2l_fma(D[53], m, L[4]);
      L[5] = m2l_fma(D[56], m, L[5]);
      L[6] = m2l_fma(D[57], m, L[6]);
      L[7] = m2l_fma(D[59], m, L[7]);
      L[8] = m2l_fma(D[60], m, L[8]);
    }
    { const T m = __ldg(Mr + 23) * rp;
      L[0] = m2l_fma(D[28], m, L[0]);
      L[1] = m2l_fma(D[40], m, L[1]);
      L[2] = m2l_fma(D[43], m, L[2]);
      L[3] = m2l_fma(D[44], m, L[3]);
      L[4] = m2l_fma(D[55], m, L[4]);
      L[5] = m2l_fma(D[58], m, L[5]);
      L[6] = m2l_fma(D[59], m, L[6]);
      L[7] = m2l_fma(D[61], m, L[7]);
      L[8] = m2l_fma(D[62], m, L[8]);
    }
    { const T m = __ldg(Mr + 24) * rp;
      L[0] = m2l_fma(D[29], m, L[0]);
      L[1] = m2l_fma(D[41], m, L[1]);
      L[2] = m2l_fma(D[44], m, L[2]);
      L[3] = m2l_fma(D[45], m, L[3]);
      L[4] = m2l_fma(D[56], m, L[4]);
      L[5] = m2l_fma(D[59], m, L[5]);
      L[6] = m2l_fma(D[60], m, L[6]);
      L[7] = m2l_fma(D[62], m, L[7]);
      L[8] = m2l_fma(D[63], m, L[8]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 25) * rp;
      L[0] = m2l_fma(D[31], m, L[0]);
      L[1] = m2l_fma(D[46], m, L[1]);
      L[2] = m2l_fma(D[47], m, L[2]);
      L[3] = m2l_fma(D[48], m, L[3]);
    }
    { const T m = -__ldg(Mr + 26) * rp;
      L[0] = m2l_fma(D[32], m, L[0]);
      L[1] = m2l_fma(D[47], m, L[1]);
      L[2] = m2l_fma(D[49], m, L[2]);
      L[3] = m2l_fma(D[50], m, L[3]);
    }
    { const T m = -__ldg(Mr + 27) * rp;
      L[0] = m2l_fma(D[33], m, L[0]);
      L[1] = m2l_fma(D[48], m, L[1]);
      L[2] = m2l_fma(D[50], m, L[2]);
      L[3] = m2l_fma(D[51], m, L[3]);
    }
    { const T m = -__ldg(Mr + 28) * rp;
      L[0] = m2l_fma(D[34], m, L[0]);
      L[1] = m2l_fma(D[49], m, L[1]);
      L[2] = m2l_fma(D[52], m, L[2]);
      L[3] = m2l_fma(D[53], m, L[3]);
    }
    { const T m = -__ldg(Mr + 29) * rp;
      L[0] = m2l_fma(D[35], m, L[0]);
      L[1] = m2l_fma(D[50], m, L[1]);
      L[2] = m2l_fma(D[53], m, L[2]);
      L[3] = m2l_fma(D[54], m, L[3]);
    }
    { const T m = -__ldg(Mr + 30) * rp;
      L[0] = m2l_fma(D[37], m, L[0]);
      L[1] = m2l_fma(D[52], m, L[1]);
      L[2] = m2l_fma(D[55], m, L[2]);
      L[3] = m2l_fma(D[56], m, L[3]);
    }
    { const T m = -__ldg(Mr + 31) * rp;
      L[0] = m2l_fma(D[38], m, L[0]);
      L[1] = m2l_fma(D[53], m, L[1]);
      L[2] = m2l_fma(D[56], m, L[2]);
      L[3] = m2l_fma(D[57], m, L[3]);
    }
    { const T m = -__ldg(Mr + 32) * rp;
      L[0] = m2l_fma(D[40], m, L[0]);
      L[1] = m2l_fma(D[55], m, L[1]);
      L[2] = m2l_fma(D[58], m, L[2]);
      L[3] = m2l_fma(D[59], m, L[3]);
    }
    { const T m = -__ldg(Mr + 33) * rp;
      L[0] = m2l_fma(D[41], m, L[0]);
      L[1] = m2l_fma(D[56], m, L[1]);
      L[2] = m2l_fma(D[59], m, L[2]);
      L[3] = m2l_fma(D[60], m, L[3]);
    }
    { const T m = -__ldg(Mr + 34) * rp;
      L[0] = m2l_fma(D[43], m, L[0]);
      L[1] = m2l_fma(D[58], m, L[1]);
      L[2] = m2l_fma(D[61], m, L[2]);
      L[3] = m2l_fma(D[62], m, L[3]);
    }
    { const T m = -__ldg(Mr + 35) * rp;
      L[0] = m2l_fma(D[44], m, L[0]);
      L[1] = m2l_fma(D[59], m, L[1]);
      L[2] = m2l_fma(D[62], m, L[2]);
      L[3] = m2l_fma(D[63], m, L[3]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 36) * rp;
      L[0] = m2l_fma(D[46], m, L[0]);
    }
    { const T m = __ldg(Mr + 37) * rp;
      L[0] = m2l_fma(D[47], m, L[0]);
    }
    { const T m = __ldg(Mr + 38) * rp;
      L[0] = m2l_fma(D[48], m, L[0]);
    }
    { const T m = __ldg(Mr + 39) * rp;
      L[0] = m2l_fma(D[49], m, L[0]);
    }
    { const T m = __ldg(Mr + 40) * rp;
      L[0] = m2l_fma(D[50], m, L[0]);
    }
    { const T m = __ldg(Mr + 41) * rp;
      L[0] = m2l_fma(D[52], m, L[0]);
    }
    { const T m = __ldg(Mr + 42) * rp;
      L[0] = m2l_fma(D[53], m, L[0]);
    }
    { const T m = __ldg(Mr + 43) * rp;
      L[0] = m2l_fma(D[55], m, L[0]);
    }
    { const T m = __ldg(Mr + 44) * rp;
      L[0] = m2l_fma(D[56], m, L[0]);
    }
    { const T m = __ldg(Mr + 45) * rp;
      L[0] = m2l_fma(D[58], m, L[0]);
    }
    { const T m = __ldg(Mr + 46) * rp;
      L[0] = m2l_fma(D[59], m, L[0]);
    }
    { const T m = __ldg(Mr + 47) * rp;
      L[0] = m2l_fma(D[61], m, L[0]);
    }
    { const T m = __ldg(Mr + 48) * rp;
      L[0] = m2l_fma(D[62], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_acc_h_6(const T (&D)[64], const T *__restrict__ Mr, T rho, T (&L)[49])
{
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[0] = m2l_fma(D[0], m, L[0]);
      L[1] = m2l_fma(D[1], m, L[1]);
      L[2] = m2l_fma(D[2], m, L[2]);
      L[3] = m2l_fma(D[3], m, L[3]);
      L[4] = m2l_fma(D[4], m, L[4]);
      L[5] = m2l_fma(D[5], m, L[5]);
      L[6] = m2l_fma(D[6], m, L[6]);
      L[7] = m2l_fma(D[7], m, L[7]);
      L[8] = m2l_fma(D[8], m, L[8]);
      L[9] = m2l_fma(D[10], m, L[9]);
      L[10] = m2l_fma(D[11], m, L[10]);
      L[11] = m2l_fma(D[12], m, L[11]);
      L[12] = m2l_fma(D[13], m, L[12]);
      L[13] = m2l_fma(D[14], m, L[13]);
      L[14] = m2l_fma(D[16], m, L[14]);
      L[15] = m2l_fma(D[17], m, L[15]);
      L[16] = m2l_fma(D[19], m, L[16]);
      L[17] = m2l_fma(D[20], m, L[17]);
      L[18] = m2l_fma(D[21], m, L[18]);
      L[19] = m2l_fma(D[22], m, L[19]);
      L[20] = m2l_fma(D[23], m, L[20]);
      L[21] = m2l_fma(D[25], m, L[21]);
      L[22] = m2l_fma(D[26], m, L[22]);
      L[23] = m2l_fma(D[28], m, L[23]);
      L[24] = m2l_fma(D[29], m, L[24]);
      L[25] = m2l_fma(D[31], m, L[25]);
      L[26] = m2l_fma(D[32], m, L[26]);
      L[27] = m2l_fma(D[33], m, L[27]);
      L[28] = m2l_fma(D[34], m, L[28]);
      L[29] = m2l_fma(D[35], m, L[29]);
      L[30] = m2l_fma(D[37], m, L[30]);
      L[31] = m2l_fma(D[38], m, L[31]);
      L[32] = m2l_fma(D[40], m, L[32]);
      L[33] = m2l_fma(D[41], m, L[33]);
      L[34] = m2l_fma(D[43], m, L[34]);
      L[35] = m2l_fma(D[44], m, L[35]);
      L[36] = m2l_fma(D[46], m, L[36]);
      L[37] = m2l_fma(D[47], m, L[37]);
      L[38] = m2l_fma(D[48], m, L[38]);
      L[39] = m2l_fma(D[49], m, L[39]);
      L[40] = m2l_fma(D[50], m, L[40]);
      L[41] = m2l_fma(D[52], m, L[41]);
      L[42] = m2l_fma(D[53], m, L[42]);
      L[43] = m2l_fma(D[55], m, L[43]);
      L[44] = m2l_fma(D[56], m, L[44]);
      L[45] = m2l_fma(D[58], m, L[45]);
      L[46] = m2l_fma(D[59], m, L[46]);
      L[47] = m2l_fma(D[61], m, L[47]);
      L[48] = m2l_fma(D[62], m, L[48]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 1) * rp;
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(D[20], m, L[10]);
      L[11] = m2l_fma(D[21], m, L[11]);
      L[12] = m2l_fma(D[22], m, L[12]);
      L[13] = m2l_fma(D[23], m, L[13]);
      L[14] = m2l_fma(D[25], m, L[14]);
      L[15] = m2l_fma(D[26], m, L[15]);
      L[16] = m2l_fma(D[31], m, L[16]);
      L[17] = m2l_fma(D[32], m, L[17]);
      L[18] = m2l_fma(D[33], m, L[18]);
      L[19] = m2l_fma(D[34], m, L[19]);
      L[20] = m2l_fma(D[35], m, L[20]);
      L[21] = m2l_fma(D[37], m, L[21]);
      L[22] = m2l_fma(D[38], m, L[22]);
      L[23] = m2l_fma(D[40], m, L[23]);
      L[24] = m2l_fma(D[41], m, L[24]);
      L[25] = m2l_fma(D[46], m, L[25]);
      L[26] = m2l_fma(D[47], m, L[26]);
      L[27] = m2l_fma(D[48], m, L[27]);
      L[28] = m2l_fma(D[49], m, L[28]);
      L[29] = m2l_fma(D[50], m, L[29]);
      L[30] = m2l_fma(D[52], m, L[30]);
      L[31] = m2l_fma(D[53], m, L[31]);
      L[32] = m2l_fma(D[55], m, L[32]);
      L[33] = m2l_fma(D[56], m, L[33]);
      L[34] = m2l_fma(D[58], m, L[34]);
      L[35] = m2l_fma(D[59], m, L[35]);
    }
    { const T m = -__ldg(Mr + 2) * rp;
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[20], m, L[9]);
      L[10] = m2l_fma(D[22], m, L[10]);
      L[11] = m2l_fma(D[23], m, L[11]);
      L[12] = m2l_fma(D[25], m, L[12]);
      L[13] = m2l_fma(D[26], m, L[13]);
      L[14] = m2l_fma(D[28], m, L[14]);
      L[15] = m2l_fma(D[29], m, L[15]);
      L[16] = m2l_fma(D[32], m, L[16]);
      L[17] = m2l_fma(D[34], m, L[17]);
      L[18] = m2l_fma(D[35], m, L[18]);
      L[19] = m2l_fma(D[37], m, L[19]);
      L[20] = m2l_fma(D[38], m, L[20]);
      L[21] = m2l_fma(D[40], m, L[21]);
      L[22] = m2l_fma(D[41], m, L[22]);
      L[23] = m2l_fma(D[43], m, L[23]);
      L[24] = m2l_fma(D[44], m, L[24]);
      L[25] = m2l_fma(D[47], m, L[25]);
      L[26] = m2l_fma(D[49], m, L[26]);
      L[27] = m2l_fma(D[50], m, L[27]);
      L[28] = m2l_fma(D[52], m, L[28]);
      L[29] = m2l_fma(D[53], m, L[29]);
      L[30] = m2l_fma(D[55], m, L[30]);
      L[31] = m2l_fma(D[56], m, L[31]);
      L[32] = m2l_fma(D[58], m, L[32]);
      L[33] = m2l_fma(D[59], m, L[33]);
      L[34] = m2l_fma(D[61], m, L[34]);
      L[35] = m2l_fma(D[62], m, L[35]);
    }
    { const T m = -__ldg(Mr + 3) * rp;
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[21], m, L[9]);
      L[10] = m2l_fma(D[23], m, L[10]);
      L[11] = m2l_fma(D[24], m, L[11]);
      L[12] = m2l_fma(D[26], m, L[12]);
      L[13] = m2l_fma(D[27], m, L[13]);
      L[14] = m2l_fma(D[29], m, L[14]);
      L[15] = m2l_fma(D[30], m, L[15]);
      L[16] = m2l_fma(D[33], m, L[16]);
      L[17] = m2l_fma(D[35], m, L[17]);
      L[18] = m2l_fma(D[36], m, L[18]);
      L[19] = m2l_fma(D[38], m, L[19]);
      L[20] = m2l_fma(D[39], m, L[20]);
      L[21] = m2l_fma(D[41], m, L[21]);
      L[22] = m2l_fma(D[42], m, L[22]);
      L[23] = m2l_fma(D[44], m, L[23]);
      L[24] = m2l_fma(D[45], m, L[24]);
      L[25] = m2l_fma(D[48], m, L[25]);
      L[26] = m2l_fma(D[50], m, L[26]);
      L[27] = m2l_fma(D[51], m, L[27]);
      L[28] = m2l_fma(D[53], m, L[28]);
      L[29] = m2l_fma(D[54], m, L[29]);
      L[30] = m2l_fma(D[56], m, L[30]);
      L[31] = m2l_fma(D[57], m, L[31]);
      L[32] = m2l_fma(D[59], m, L[32]);
      L[33] = m2l_fma(D[60], m, L[33]);
      L[34] = m2l_fma(D[62], m, L[34]);
      L[35] = m2l_fma(D[63], m, L[35]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 4) * rp;
      L[0] = m2l_fma(D[4], m, L[0]);
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
      L[4] = m2l_fma(D[19], m, L[4]);
      L[5] = m2l_fma(D[20], m, L[5]);
      L[6] = m2l_fma(D[21], m, L[6]);
      L[7] = m2l_fma(D[22], m, L[7]);
      L[8] = m2l_fma(D[23], m, L[8]);
      L[9] = m2l_fma(D[31], m, L[9]);
      L[10] = m2l_fma(D[32], m, L[10]);
      L[11] = m2l_fma(D[33], m, L[11]);
      L[12] = m2l_fma(D[34], m, L[12]);
      L[13] = m2l_fma(D[35], m, L[13]);
      L[14] = m2l_fma(D[37], m, L[14]);
      L[15] = m2l_fma(D[38], m, L[15]);
      L[16] = m2l_fma(D[46], m, L[16]);
      L[17] = m2l_fma(D[47], m, L[17]);
      L[18] = m2l_fma(D[48], m, L[18]);
      L[19] = m2l_fma(D[49], m, L[19]);
      L[20] = m2l_fma(D[50], m, L[20]);
      L[21] = m2l_fma(D[52], m, L[21]);
      L[22] = m2l_fma(D[53], m, L[22]);
      L[23] = m2l_fma(D[55], m, L[23]);
      L[24] = m2l_fma(D[56], m, L[24]);
    }
    { const T m = __ldg(Mr + 5) * rp;
      L[0] = m2l_fma(D[5], m, L[0]);
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[22], m, L[5]);
      L[6] = m2l_fma(D[23], m, L[6]);
      L[7] = m2l_fma(D[25], m, L[7]);
      L[8] = m2l_fma(D[26], m, L[8]);
      L[9] = m2l_fma(D[32], m, L[9]);
      L[10] = m2l_fma(D[34], m, L[10]);
      L[11] = m2l_fma(D[35], m, L[11]);
      L[12] = m2l_fma(D[37], m, L[12]);
      L[13] = m2l_fma(D[38], m, L[13]);
      L[14] = m2l_fma(D[40], m, L[14]);
      L[15] = m2l_fma(D[41], m, L[15]);
      L[16] = m2l_fma(D[47], m, L[16]);
      L[17] = m2l_fma(D[49], m, L[17]);
      L[18] = m2l_fma(D[50], m, L[18]);
      L[19] = m2l_fma(D[52], m, L[19]);
      L[20] = m2l_fma(D[53], m, L[20]);
      L[21] = m2l_fma(D[55], m, L[21]);
      L[22] = m2l_fma(D[56], m, L[22]);
      L[23] = m2l_fma(D[58], m, L[23]);
      L[24] = m2l_fma(D[59], m, L[24]);
    }
    { const T m = __ldg(Mr + 6) * rp;
      L[0] = m2l_fma(D[6], m, L[0]);
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(D[33], m, L[9]);
      L[10] = m2l_fma(D[35], m, L[10]);
      L[11] = m2l_fma(D[36], m, L[11]);
      L[12] = m2l_fma(D[38], m, L[12]);
      L[13] = m2l_fma(D[39], m, L[13]);
      L[14] = m2l_fma(D[41], m, L[14]);
      L[15] = m2l_fma(D[42], m, L[15]);
      L[16] = m2l_fma(D[48], m, L[16]);
      L[17] = m2l_fma(D[50], m, L[17]);
      L[18] = m2l_fma(D[51], m, L[18]);
      L[19] = m2l_fma(D[53], m, L[19]);
      L[20] = m2l_fma(D[54], m, L[20]);
      L[21] = m2l_fma(D[56], m, L[21]);
      L[22] = m2l_fma(D[57], m, L[22]);
      L[23] = m2l_fma(D[59], m, L[23]);
      L[24] = m2l_fma(D[60], m, L[24]);
    }
    { const T m = __ldg(Mr + 7) * rp;
      L[0] = m2l_fma(D[7], m, L[0]);
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[25], m, L[5]);
      L[6] = m2l_fma(D[26], m, L[6]);
      L[7] = m2l_fma(D[28], m, L[7]);
      L[8] = m2l_fma(D[29], m, L[8]);
      L[9] = m2l_fma(D[34], m, L[9]);
      L[10] = m2l_fma(D[37], m, L[10]);
      L[11] = m2l_fma(D[38], m, L[11]);
      L[12] = m2l_fma(D[40], m, L[12]);
      L[13] = m2l_fma(D[41], m, L[13]);
      L[14] = m2l_fma(D[43], m, L[14]);
      L[15] = m2l_fma(D[44], m, L[15]);
      L[16] = m2l_fma(D[49], m, L[16]);
      L[17] = m2l_fma(D[52], m, L[17]);
      L[18] = m2l_fma(D[53], m, L[18]);
      L[19] = m2l_fma(D[55], m, L[19]);
      L[20] = m2l_fma(D[56], m, L[20]);
      L[21] = m2l_fma(D[58], m, L[21]);
      L[22] = m2l_fma(D[59], m, L[22]);
      L[23] = m2l_fma(D[61], m, L[23]);
      L[24] = m2l_fma(D[62], m, L[24]);
    }
    { const T m = __ldg(Mr + 8) * rp;
      L[0] = m2l_fma(D[8], m, L[0]);
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[29], m, L[7]);
      L[8] = m2l_fma(D[30], m, L[8]);
      L[9] = m2l_fma(D[35], m, L[9]);
      L[10] = m2l_fma(D[38], m, L[10]);
      L[11] = m2l_fma(D[39], m, L[11]);
      L[12] = m2l_fma(D[41], m, L[12]);
      L[13] = m2l_fma(D[42], m, L[13]);
      L[14] = m2l_fma(D[44], m, L[14]);
      L[15] = m2l_fma(D[45], m, L[15]);
      L[16] = m2l_fma(D[50], m, L[16]);
      L[17] = m2l_fma(D[53], m, L[17]);
      L[18] = m2l_fma(D[54], m, L[18]);
      L[19] = m2l_fma(D[56], m, L[19]);
      L[20] = m2l_fma(D[57], m, L[20]);
      L[21] = m2l_fma(D[59], m, L[21]);
      L[22] = m2l_fma(D[60], m, L[22]);
      L[23] = m2l_fma(D[62], m, L[23]);
      L[24] = m2l_fma(D[63], m, L[24]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 9) * rp;
      L[0] = m2l_fma(D[10], m, L[0]);
      L[1] = m2l_fma(D[19], m, L[1]);
      L[2] = m2l_fma(D[20], m, L[2]);
      L[3] = m2l_fma(D[21], m, L[3]);
      L[4] = m2l_fma(D[31], m, L[4]);
      L[5] = m2l_fma(D[32], m, L[5]);
      L[6] = m2l_fma(D[33], m, L[6]);
      L[7] = m2l_fma(D[34], m, L[7]);
      L[8] = m2l_fma(D[35], m, L[8]);
      L[9] = m2l_fma(D[46], m, L[9]);
      L[10] = m2l_fma(D[47], m, L[10]);
      L[11] = m2l_fma(D[48], m, L[11]);
      L[12] = m2l_fma(D[49], m, L[12]);
      L[13] = m2l_fma(D[50], m, L[13]);
      L[14] = m2l_fma(D[52], m, L[14]);
      L[15] = m2l_fma(D[53], m, L[15]);
    }
    { const T m = -__ldg(Mr + 10) * rp;
      L[0] = m2l_fma(D[11], m, L[0]);
      L[1] = m2l_fma(D[20], m, L[1]);
      L[2] = m2l_fma(D[22], m, L[2]);
      L[3] = m2l_fma(D[23], m, L[3]);
      L[4] = m2l_fma(D[32], m, L[4]);
      L[5] = m2l_fma(D[34], m, L[5]);
      L[6] = m2l_fma(D[35], m, L[6]);
      L[7] = m2l_fma(D[37], m, L[7]);
      L[8] = m2l_fma(D[38], m, L[8]);
      L[9] = m2l_fma(D[47], m, L[9]);
      L[10] = m2l_fma(D[49], m, L[10]);
      L[11] = m2l_fma(D[50], m, L[11]);
      L[12] = m2l_fma(D[52], m, L[12]);
      L[13] = m2l_fma(D[53], m, L[13]);
      L[14] = m2l_fma(D[55], m, L[14]);
      L[15] = m2l_fma(D[56], m, L[15]);
    }
    { const T m = -__ldg(Mr + 11) * rp;
      L[0] = m2l_fma(D[12], m, L[0]);
      L[1] = m2l_fma(D[21], m, L[1]);
      L[2] = m2l_fma(D[23], m, L[2]);
      L[3] = m2l_fma(D[24], m, L[3]);
      L[4] = m2l_fma(D[33], m, L[4]);
      L[5] = m2l_fma(D[35], m, L[5]);
      L[6] = m2l_fma(D[36], m, L[6]);
      L[7] = m2l_fma(D[38], m, L[7]);
      L[8] = m2l_fma(D[39], m, L[8]);
      L[9] = m2l_fma(D[48], m, L[9]);
      L[10] = m2l_fma(D[50], m, L[10]);
      L[11] = m2l_fma(D[51], m, L[11]);
      L[12] = m2l_fma(D[53], m, L[12]);
      L[13] = m2l_fma(D[54], m, L[13]);
      L[14] = m2l_fma(D[56], m, L[14]);
      L[15] = m2l_fma(D[57], m, L[15]);
    }
    { const T m = -__ldg(Mr + 12) * rp;
      L[0] = m2l_fma(D[13], m, L[0]);
      L[1] = m2l_fma(D[22], m, L[1]);
      L[2] = m2l_fma(D[25], m, L[2]);
      L[3] = m2l_fma(D[26], m, L[3]);
      L[4] = m2l_fma(D[34], m, L[4]);
      L[5] = m2l_fma(D[37], m, L[5]);
      L[6] = m2l_fma(D[38], m, L[6]);
      L[7] = m2l_fma(D[40], m, L[7]);
      L[8] = m2l_fma(D[41], m, L[8]);
      L[9] = m2l_fma(D[49], m, L[9]);
      L[10] = m2l_fma(D[52], m, L[10]);
      L[11] = m2l_fma(D[53], m, L[11]);
      L[12] = m2l_fma(D[55], m, L[12]);
      L[13] = m2l_fma(D[56], m, L[13]);
      L[14] = m2l_fma(D[58], m, L[14]);
      L[15] = m2l_fma(D[59], m, L[15]);
    }
    { const T m = -__ldg(Mr + 13) * rp;
      L[0] = m2l_fma(D[14], m, L[0]);
      L[1] = m2l_fma(D[23], m, L[1]);
      L[2] = m2l_fma(D[26], m, L[2]);
      L[3] = m2l_fma(D[27], m, L[3]);
      L[4] = m2l_fma(D[35], m, L[4]);
      L[5] = m2l_fma(D[38], m, L[5]);
      L[6] = m2l_fma(D[39], m, L[6]);
      L[7] = m2l_fma(D[41], m, L[7]);
      L[8] = m2l_fma(D[42], m, L[8]);
      L[9] = m2l_fma(D[50], m, L[9]);
      L[10] = m2l_fma(D[53], m, L[10]);
      L[11] = m2l_fma(D[54], m, L[11]);
      L[12] = m2l_fma(D[56], m, L[12]);
      L[13] = m2l_fma(D[57], m, L[13]);
      L[14] = m2l_fma(D[59], m, L[14]);
      L[15] = m2l_fma(D[60], m, L[15]);
    }
    { const T m = -__ldg(Mr + 14) * rp;
      L[0] = m2l_fma(D[16], m, L[0]);
      L[1] = m2l_fma(D[25], m, L[1]);
      L[2] = m2l_fma(D[28], m, L[2]);
      L[3] = m2l_fma(D[29], m, L[3]);
      L[4] = m2l_fma(D[37], m, L[4]);
      L[5] = m2l_fma(D[40], m, L[5]);
      L[6] = m2l_fma(D[41], m, L[6]);
      L[7] = m2l_fma(D[43], m, L[7]);
      L[8] = m2l_fma(D[44], m, L[8]);
      L[9] = m2l_fma(D[52], m, L[9]);
      L[10] = m2l_fma(D[55], m, L[10]);
      L[11] = m2l_fma(D[56], m, L[11]);
      L[12] = m2l_fma(D[58], m, L[12]);
      L[13] = m2l_fma(D[59], m, L[13]);
      L[14] = m2l_fma(D[61], m, L[14]);
      L[15] = m2l_fma(D[62], m, L[15]);
    }
    { const T m = -__ldg(Mr + 15) * rp;
      L[0] = m2l_fma(D[17], m, L[0]);
      L[1] = m2l_fma(D[26], m, L[1]);
      L[2] = m2l_fma(D[29], m, L[2]);
      L[3] = m2l_fma(D[30], m, L[3]);
      L[4] = m2l_fma(D[38], m, L[4]);
      L[5] = m2l_fma(D[41], m, L[5]);
      L[6] = m2l_fma(D[42], m, L[6]);
      L[7] = m2l_fma(D[44], m, L[7]);
      L[8] = m2l_fma(D[45], m, L[8]);
      L[9] = m2l_fma(D[53], m, L[9]);
      L[10] = m2l_fma(D[56], m, L[10]);
      L[11] = m2l_fma(D[57], m, L[11]);
      L[12] = m2l_fma(D[59], m, L[12]);
      L[13] = m2l_fma(D[60], m, L[13]);
      L[14] = m2l_fma(D[62], m, L[14]);
      L[15] = m2l_fma(D[63], m, L[15]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 16) * rp;
      L[0] = m2l_fma(D[19], m, L[0]);
      L[1] = m2l_fma(D[31], m, L[1]);
      L[2] = m2l_fma(D[32], m, L[2]);
      L[3] = m2l_fma(D[33], m, L[3]);
      L[4] = m2l_fma(D[46], m, L[4]);
      L[5] = m2l_fma(D[47], m, L[5]);
      L[6] = m2l_fma(D[48], m, L[6]);
      L[7] = m2l_fma(D[49], m, L[7]);
      L[8] = m2l_fma(D[50], m, L[8]);
    }
    { const T m = __ldg(Mr + 17) * rp;
      L[0] = m2l_fma(D[20], m, L[0]);
      L[1] = m2l_fma(D[32], m, L[1]);
      L[2] = m2l_fma(D[34], m, L[2]);
      L[3] = m2l_fma(D[35], m, L[3]);
      L[4] = m2l_fma(D[47], m, L[4]);
      L[5] = m2l_fma(D[49], m, L[5]);
      L[6] = m2l_fma(D[50], m, L[6]);
      L[7] = m2l_fma(D[52], m, L[7]);
      L[8] = m2l_fma(D[53], m, L[8]);
    }
    { const T m = __ldg(Mr + 18) * rp;
      L[0] = m2l_fma(D[21], m, L[0]);
      L[1] = m2l_fma(D[33], m, L[1]);
      L[2] = m2l_fma(D[35], m, L[2]);
      L[3] = m2l_fma(D[36], m, L[3]);
      L[4] = m2l_fma(D[48], m, L[4]);
      L[5] = m2l_fma(D[50], m, L[5]);
      L[6] = m2l_fma(D[51], m, L[6]);
      L[7] = m2l_fma(D[53], m, L[7]);
      L[8] = m2l_fma(D[54], m, L[8]);
    }
    { const T m = __ldg(Mr + 19) * rp;
      L[0] = m2l_fma(D[22], m, L[0]);
      L[1] = m2l_fma(D[34], m, L[1]);
      L[2] = m2l_fma(D[37], m, L[2]);
      L[3] = m2l_fma(D[38], m, L[3]);
      L[4] = m2l_fma(D[49], m, L[4]);
      L[5] = m2l_fma(D[52], m, L[5]);
      L[6] = m2l_fma(D[53], m, L[6]);
      L[7] = m2l_fma(D[55], m, L[7]);
      L[8] = m2l_fma(D[56], m, L[8]);
    }
    { const T m = __ldg(Mr + 20) * rp;
      L[0] = m2l_fma(D[23], m, L[0]);
      L[1] = m2l_fma(D[35], m, L[1]);
      L[2] = m2l_fma(D[38], m, L[2]);
      L[3] = m2l_fma(D[39], m, L[3]);
      L[4] = m2l_fma(D[50], m, L[4]);
      L[5] = m2l_fma(D[53], m, L[5]);
      L[6] = m2l_fma(D[54], m, L[6]);
      L[7] = m2l_fma(D[56], m, L[7]);
      L[8] = m2l_fma(D[57], m, L[8]);
    }
    { const T m = __ldg(Mr + 21) * rp;
      L[0] = m2l_fma(D[25], m, L[0]);
      L[1] = m2l_fma(D[37], m, L[1]);
      L[2] = m2l_fma(D[40], m, L[2]);
      L[3] = m2l_fma(D[41], m, L[3]);
      L[4] = m2l_fma(D[52], m, L[4]);
      L[5] = m2l_fma(D[55], m, L[5]);
      L[6] = m2l_fma(D[56], m, L[6]);
      L[7] = m2l_fma(D[58], m, L[7]);
      L[8] = m2l_fma(D[59], m, L[8]);
    }
    { const T m = __ldg(Mr + 22) * rp;
      L[0] = m2l_fma(D[26], m, L[0]);
      L[1] = m2l_fma(D[38], m, L[1]);
      L[2] = m2l_fma(D[41], m, L[2]);
      L[3] = m2l_fma(D[42], m, L[3]);
      L[4] = m2l_fma(D[53], m, L[4]);
      L[5] = m2l_fma(D[56], m, L[5]);
      L[6] = m2l_fma(D[57], m, L[6]);
      L[7] = m2l_fma(D[59], m, L[7]);
      L[8] = m2l_fma(D[60], m, L[8]);
    }
    { const T m = __ldg(Mr + 23) * rp;
      L[0] = m2l_fma(D[28], m, L[0]);
      L[1] = m2l_fma(D[40], m, L[1]);
      L[2] = m2l_fma(D[43], m, L[2]);
      L[3] = m2l_fma(D[44], m, L[3]);
      L[4] = m2l_fma(D[55], m, L[4]);
      L[5] = m2l_fma(D[58], m, L[5]);
      L[6] = m2l_fma(D[59], m, L[6]);
      L[7] = m2l_fma(D[61], m, L[7]);
      L[8] = m2l_fma(D[62], m, L[8]);
    }
    { const T m = __ldg(Mr + 24) * rp;
      L[0] = m2l_fma(D[29], m, L[0]);
      L[1] = m2l_fma(D[41], m, L[1]);
      L[2] = m2l_fma(D[44], m, L[2]);
      L[3] = m2l_fma(D[45], m, L[3]);
      L[4] = m2l_fma(D[56], m, L[4]);
      L[5] = m2l_fma(D[59], m, L[5]);
      L[6] = m2l_fma(D[60], m, L[6]);
      L[7] = m2l_fma(D[62], m, L[7]);
      L[8] = m2l_fma(D[63], m, L[8]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 25) * rp;
      L[0] = m2l_fma(D[31], m, L[0]);
      L[1] = m2l_fma(D[46], m, L[1]);
      L[2] = m2l_fma(D[47], m, L[2]);
      L[3] = m2l_fma(D[48], m, L[3]);
    }
    { const T m = -__ldg(Mr + 26) * rp;
      L[0] = m2l_fma(D[32], m, L[0]);
      L[1] = m2l_fma(D[47], m, L[1]);
      L[2] = m2l_fma(D[49], m, L[2]);
      L[3] = m2l_fma(D[50], m, L[3]);
    }
    { const T m = -__ldg(Mr + 27) * rp;
      L[0] = m2l_fma(D[33], m, L[0]);
      L[1] = m2l_fma(D[48], m, L[1]);
      L[2] = m2l_fma(D[50], m, L[2]);
      L[3] = m2l_fma(D[51], m, L[3]);
    }
    { const T m = -__ldg(Mr + 28) * rp;
      L[0] = m2l_fma(D[34], m, L[0]);
      L[1] = m2l_fma(D[49], m, L[1]);
      L[2] = m2l_fma(D[52], m, L[2]);
      L[3] = m2l_fma(D[53], m, L[3]);
    }
    { const T m = -__ldg(Mr + 29) * rp;
      L[0] = m2l_fma(D[35], m, L[0]);
      L[1] = m2l_fma(D[50], m, L[1]);
      L[2] = m2l_fma(D[53], m, L[2]);
      L[3] = m2l_fma(D[54], m, L[3]);
    }
    { const T m = -__ldg(Mr + 30) * rp;
      L[0] = m2l_fma(D[37], m, L[0]);
      L[1] = m2l_fma(D[52], m, L[1]);
      L[2] = m2l_fma(D[55], m, L[2]);
      L[3] = m2l_fma(D[56], m, L[3]);
    }
    { const T m = -__ldg(Mr + 31) * rp;
      L[0] = m2l_fma(D[38], m, L[0]);
      L[1] = m2l_fma(D[53], m, L[1]);
      L[2] = m2l_fma(D[56], m, L[2]);
      L[3] = m2l_fma(D[57], m, L[3]);
    }
    { const T m = -__ldg(Mr + 32) * rp;
      L[0] = m2l_fma(D[40], m, L[0]);
      L[1] = m2l_fma(D[55], m, L[1]);
      L[2] = m2l_fma(D[58], m, L[2]);
      L[3] = m2l_fma(D[59], m, L[3]);
    }
    { const T m = -__ldg(Mr + 33) * rp;
      L[0] = m2l_fma(D[41], m, L[0]);
      L[1] = m2l_fma(D[56], m, L[1]);
      L[2] = m2l_fma(D[59], m, L[2]);
      L[3] = m2l_fma(D[60], m, L[3]);
    }
    { const T m = -__ldg(Mr + 34) * rp;
      L[0] = m2l_fma(D[43], m, L[0]);
      L[1] = m2l_fma(D[58], m, L[1]);
      L[2] = m2l_fma(D[61], m, L[2]);
      L[3] = m2l_fma(D[62], m, L[3]);
    }
    { const T m = -__ldg(Mr + 35) * rp;
      L[0] = m2l_fma(D[44], m, L[0]);
      L[1] = m2l_fma(D[59], m, L[1]);
      L[2] = m2l_fma(D[62], m, L[2]);
      L[3] = m2l_fma(D[63], m, L[3]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 36) * rp;
      L[0] = m2l_fma(D[46], m, L[0]);
    }
    { const T m = __ldg(Mr + 37) * rp;
      L[0] = m2l_fma(D[47], m, L[0]);
    }
    { const T m = __ldg(Mr + 38) * rp;
      L[0] = m2l_fma(D[48], m, L[0]);
    }
    { const T m = __ldg(Mr + 39) * rp;
      L[0] = m2l_fma(D[49], m, L[0]);
    }
    { const T m = __ldg(Mr + 40) * rp;
      L[0] = m2l_fma(D[50], m, L[0]);
    }
    { const T m = __ldg(Mr + 41) * rp;
      L[0] = m2l_fma(D[52], m, L[0]);
    }
    { const T m = __ldg(Mr + 42) * rp;
      L[0] = m2l_fma(D[53], m, L[0]);
    }
    { const T m = __ldg(Mr + 43) * rp;
      L[0] = m2l_fma(D[55], m, L[0]);
    }
    { const T m = __ldg(Mr + 44) * rp;
      L[0] = m2l_fma(D[56], m, L[0]);
    }
    { const T m = __ldg(Mr + 45) * rp;
      L[0] = m2l_fma(D[58], m, L[0]);
    }
    { const T m = __ldg(Mr + 46) * rp;
      L[0] = m2l_fma(D[59], m, L[0]);
    }
    { const T m = __ldg(Mr + 47) * rp;
      L[0] = m2l_fma(D[61], m, L[0]);
    }
    { const T m = __ldg(Mr + 48) * rp;
      L[0] = m2l_fma(D[62], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_h_6(const T (&D)[64], const T *__restrict__ Mr, T (&L)[49])
{
    { const T m = __ldg(Mr + 0);
      L[0] = D[0] * m;
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = -D[10] * m;
      L[10] = -D[11] * m;
      L[11] = -D[12] * m;
      L[12] = -D[13] * m;
      L[13] = -D[14] * m;
      L[14] = -D[16] * m;
      L[15] = -D[17] * m;
      L[16] = D[19] * m;
      L[17] = D[20] * m;
      L[18] = D[21] * m;
      L[19] = D[22] * m;
      L[20] = D[23] * m;
      L[21] = D[25] * m;
      L[22] = D[26] * m;
      L[23] = D[28] * m;
      L[24] = D[29] * m;
      L[25] = -D[31] * m;
      L[26] = -D[32] * m;
      L[27] = -D[33] * m;
      L[28] = -D[34] * m;
      L[29] = -D[35] * m;
      L[30] = -D[37] * m;
      L[31] = -D[38] * m;
      L[32] = -D[40] * m;
      L[33] = -D[41] * m;
      L[34] = -D[43] * m;
      L[35] = -D[44] * m;
      L[36] = D[46] * m;
      L[37] = D[47] * m;
      L[38] = D[48] * m;
      L[39] = D[49] * m;
      L[40] = D[50] * m;
      L[41] = D[52] * m;
      L[42] = D[53] * m;
      L[43] = D[55] * m;
      L[44] = D[56] * m;
      L[45] = D[58] * m;
      L[46] = D[59] * m;
      L[47] = D[61] * m;
      L[48] = D[62] * m;
    }
    { const T m = __ldg(Mr + 1);
      L[0] = m2l_fma(D[1], m, L[0]);
      L[1] = m2l_fma(-D[4], m, L[1]);
      L[2] = m2l_fma(-D[5], m, L[2]);
      L[3] = m2l_fma(-D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(-D[19], m, L[9]);
      L[10] = m2l_fma(-D[20], m, L[10]);
      L[11] = m2l_fma(-D[21], m, L[11]);
      L[12] = m2l_fma(-D[22], m, L[12]);
      L[13] = m2l_fma(-D[23], m, L[13]);
      L[14] = m2l_fma(-D[25], m, L[14]);
      L[15] = m2l_fma(-D[26], m, L[15]);
      L[16] = m2l_fma(D[31], m, L[16]);
      L[17] = m2l_fma(D[32], m, L[17]);
      L[18] = m2l_fma(D[33], m, L[18]);
      L[19] = m2l_fma(D[34], m, L[19]);
      L[20] = m2l_fma(D[35], m, L[20]);
      L[21] = m2l_fma(D[37], m, L[21]);
      L[22] = m2l_fma(D[38], m, L[22]);
      L[23] = m2l_fma(D[40], m, L[23]);
      L[24] = m2l_fma(D[41], m, L[24]);
      L[25] = m2l_fma(-D[46], m, L[25]);
      L[26] = m2l_fma(-D[47], m, L[26]);
      L[27] = m2l_fma(-D[48], m, L[27]);
      L[28] = m2l_fma(-D[49], m, L[28]);
      L[29] = m2l_fma(-D[50], m, L[29]);
      L[30] = m2l_fma(-D[52], m, L[30]);
      L[31] = m2l_fma(-D[53], m, L[31]);
      L[32] = m2l_fma(-D[55], m, L[32]);
      L[33] = m2l_fma(-D[56], m, L[33]);
      L[34] = m2l_fma(-D[58], m, L[34]);
      L[35] = m2l_fma(-D[59], m, L[35]);
    }
    { const T m = __ldg(Mr + 2);
      L[0] = m2l_fma(D[2], m, L[0]);
      L[1] = m2l_fma(-D[5], m, L[1]);
      L[2] = m2l_fma(-D[7], m, L[2]);
      L[3] = m2l_fma(-D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(-D[20], m, L[9]);
      L[10] = m2l_fma(-D[22], m, L[10]);
      L[11] = m2l_fma(-D[23], m, L[11]);
      L[12] = m2l_fma(-D[25], m, L[12]);
      L[13] = m2l_fma(-D[26], m, L[13]);
      L[14] = m2l_fma(-D[28], m, L[14]);
      L[15] = m2l_fma(-D[29], m, L[15]);
      L[16] = m2l_fma(D[32], m, L[16]);
      L[17] = m2l_fma(D[34], m, L[17]);
      L[18] = m2l_fma(D[35], m, L[18]);
      L[19] = m2l_fma(D[37], m, L[19]);
      L[20] = m2l_fma(D[38], m, L[20]);
      L[21] = m2l_fma(D[40], m, L[21]);
      L[22] = m2l_fma(D[41], m, L[22]);
      L[23] = m2l_fma(D[43], m, L[23]);
      L[24] = m2l_fma(D[44], m, L[24]);
      L[25] = m2l_fma(-D[47], m, L[25]);
      L[26] = m2l_fma(-D[49], m, L[26]);
      L[27] = m2l_fma(-D[50], m, L[27]);
      L[28] = m2l_fma(-D[52], m, L[28]);
      L[29] = m2l_fma(-D[53], m, L[29]);
      L[30] = m2l_fma(-D[55], m, L[30]);
      L[31] = m2l_fma(-D[56], m, L[31]);
      L[32] = m2l_fma(-D[58], m, L[32]);
      L[33] = m2l_fma(-D[59], m, L[33]);
      L[34] = m2l_fma(-D[61], m, L[34]);
      L[35] = m2l_fma(-D[62], m, L[35]);
    }
    { const T m = __ldg(Mr + 3);
      L[0] = m2l_fma(D[3], m, L[0]);
      L[1] = m2l_fma(-D[6], m, L[1]);
      L[2] = m2l_fma(-D[8], m, L[2]);
      L[3] = m2l_fma(-D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(-D[21], m, L[9]);
      L[10] = m2l_fma(-D[23], m, L[10]);
      L[11] = m2l_fma(-D[24], m, L[11]);
      L[12] = m2l_fma(-D[26], m, L[12]);
      L[13] = m2l_fma(-D[27], m, L[13]);
      L[14] = m2l_fma(-D[29], m, L[14]);
      L[15] = m2l_fma(-D[30], m, L[15]);
      L[16] = m2l_fma(D[33], m, L[16]);
      L[17] = m2l_fma(D[35], m, L[17]);
      L[18] = m2l_fma(D[36], m, L[18]);
      L[19] = m2l_fma(D[38], m, L[19]);
      L[20] = m2l_fma(D[39], m, L[20]);
      L[21] = m2l_fma(D[41], m, L[21]);
      L[22] = m2l_fma(D[42], m, L[22]);
      L[23] = m2l_fma(D[44], m, L[23]);
      L[24] = m2l_fma(D[45], m, L[24]);
      L[25] = m2l_fma(-D[48], m, L[25]);
      L[26] = m2l_fma(-D[50], m, L[26]);
      L[27] = m2l_fma(-D[51], m, L[27]);
      L[28] = m2l_fma(-D[53], m, L[28]);
      L[29] = m2l_fma(-D[54], m, L[29]);
      L[30] = m2l_fma(-D[56], m, L[30]);
      L[31] = m2l_fma(-D[57], m, L[31]);
      L[32] = m2l_fma(-D[59], m, L[32]);
      L[33] = m2l_fma(-D[60], m, L[33]);
      L[34] = m2l_fma(-D[62], m, L[34]);
      L[35] = m2l_fma(-D[63], m, L[35]);
    }
    { const T m = __ldg(Mr + 4);
      L[0] = m2l_fma(D[4], m, L[0]);
      L[1] = m2l_fma(-D[10], m, L[1]);
      L[2] = m2l_fma(-D[11], m, L[2]);
      L[3] = m2l_fma(-D[12], m, L[3]);
      L[4] = m2l_fma(D[19], m, L[4]);
      L[5] = m2l_fma(D[20], m, L[5]);
      L[6] = m2l_fma(D[21], m, L[6]);
      L[7] = m2l_fma(D[22], m, L[7]);
      L[8] = m2l_fma(D[23], m, L[8]);
      L[9] = m2l_fma(-D[31], m, L[9]);
      L[10] = m2l_fma(-D[32], m, L[10]);
      L[11] = m2l_fma(-D[33], m, L[11]);
      L[12] = m2l_fma(-D[34], m, L[12]);
      L[13] = m2l_fma(-D[35], m, L[13]);
      L[14] = m2l_fma(-D[37], m, L[14]);
      L[15] = m2l_fma(-D[38], m, L[15]);
      L[16] = m2l_fma(D[46], m, L[16]);
      L[17] = m2l_fma(D[47], m, L[17]);
      L[18] = m2l_fma(D[48], m, L[18]);
      L[19] = m2l_fma(D[49], m, L[19]);
      L[20] = m2l_fma(D[50], m, L[20]);
      L[21] = m2l_fma(D[52], m, L[21]);
      L[22] = m2l_fma(D[53], m, L[22]);
      L[23] = m2l_fma(D[55], m, L[23]);
      L[24] = m2l_fma(D[56], m, L[24]);
    }
    { const T m = __ldg(Mr + 5);
      L[0] = m2l_fma(D[5], m, L[0]);
      L[1] = m2l_fma(-D[11], m, L[1]);
      L[2] = m2l_fma(-D[13], m, L[2]);
      L[3] = m2l_fma(-D[14], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[22], m, L[5]);
      L[6] = m2l_fma(D[23], m, L[6]);
      L[7] = m2l_fma(D[25], m, L[7]);
      L[8] = m2l_fma(D[26], m, L[8]);
      L[9] = m2l_fma(-D[32], m, L[9]);
      L[10] = m2l_fma(-D[34], m, L[10]);
      L[11] = m2l_fma(-D[35], m, L[11]);
      L[12] = m2l_fma(-D[37], m, L[12]);
      L[13] = m2l_fma(-D[38], m, L[13]);
      L[14] = m2l_fma(-D[40], m, L[14]);
      L[15] = m2l_fma(-D[41], m, L[15]);
      L[16] = m2l_fma(D[47], m, L[16]);
      L[17] = m2l_fma(D[49], m, L[17]);
      L[18] = m2l_fma(D[50], m, L[18]);
      L[19] = m2l_fma(D[52], m, L[19]);
      L[20] = m2l_fma(D[53], m, L[20]);
      L[21] = m2l_fma(D[55], m, L[21]);
      L[22] = m2l_fma(D[56], m, L[22]);
      L[23] = m2l_fma(D[58], m, L[23]);
      L[24] = m2l_fma(D[59], m, L[24]);
    }
    { const T m = __ldg(Mr + 6);
      L[0] = m2l_fma(D[6], m, L[0]);
      L[1] = m2l_fma(-D[12], m, L[1]);
      L[2] = m2l_fma(-D[14], m, L[2]);
      L[3] = m2l_fma(-D[15], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(-D[33], m, L[9]);
      L[10] = m2l_fma(-D[35], m, L[10]);
      L[11] = m2l_fma(-D[36], m, L[11]);
      L[12] = m2l_fma(-D[38], m, L[12]);
      L[13] = m2l_fma(-D[39], m, L[13]);
      L[14] = m2l_fma(-D[41], m, L[14]);
      L[15] = m2l_fma(-D[42], m, L[15]);
      L[16] = m2l_fma(D[48], m, L[16]);
      L[17] = m2l_fma(D[50], m, L[17]);
      L[18] = m2l_fma(D[51], m, L[18]);
      L[19] = m2l_fma(D[53], m, L[19]);
      L[20] = m2l_fma(D[54], m, L[20]);
      L[21] = m2l_fma(D[56], m, L[21]);
      L[22] = m2l_fma(D[57], m, L[22]);
      L[23] = m2l_fma(D[59], m, L[23]);
      L[24] = m2l_fma(D[60], m, L[24]);
    }
    { const T m = __ldg(Mr + 7);
      L[0] = m2l_fma(D[7], m, L[0]);
      L[1] = m2l_fma(-D[13], m, L[1]);
      L[2] = m2l_fma(-D[16], m, L[2]);
      L[3] = m2l_fma(-D[17], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[25], m, L[5]);
      L[6] = m2l_fma(D[26], m, L[6]);
      L[7] = m2l_fma(D[28], m, L[7]);
      L[8] = m2l_fma(D[29], m, L[8]);
      L[9] = m2l_fma(-D[34], m, L[9]);
      L[10] = m2l_fma(-D[37], m, L[10]);
      L[11] = m2l_fma(-D[38], m, L[11]);
      L[12] = m2l_fma(-D[40], m, L[12]);
      L[13] = m2l_fma(-D[41], m, L[13]);
      L[14] = m2l_fma(-D[43], m, L[14]);
      L[15] = m2l_fma(-D[44], m, L[15]);
      L[16] = m2l_fma(D[49], m, L[16]);
      L[17] = m2l_fma(D[52], m, L[17]);
      L[18] = m2l_fma(D[53], m, L[18]);
      L[19] = m2l_fma(D[55], m, L[19]);
      L[20] = m2l_fma(D[56], m, L[20]);
      L[21] = m2l_fma(D[58], m, L[21]);
      L[22] = m2l_fma(D[59], m, L[22]);
      L[23] = m2l_fma(D[61], m, L[23]);
      L[24] = m2l_fma(D[62], m, L[24]);
    }
    { const T m = __ldg(Mr + 8);
      L[0] = m2l_fma(D[8], m, L[0]);
      L[1] = m2l_fma(-D[14], m, L[1]);
      L[2] = m2l_fma(-D[17], m, L[2]);
      L[3] = m2l_fma(-D[18], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[29], m, L[7]);
      L[8] = m2l_fma(D[30], m, L[8]);
      L[9] = m2l_fma(-D[35], m, L[9]);
      L[10] = m2l_fma(-D[38], m, L[10]);
      L[11] = m2l_fma(-D[39], m, L[11]);
      L[12] = m2l_fma(-D[41], m, L[12]);
      L[13] = m2l_fma(-D[42], m, L[13]);
      L[14] = m2l_fma(-D[44], m, L[14]);
      L[15] = m2l_fma(-D[45], m, L[15]);
      L[16] = m2l_fma(D[50], m, L[16]);
      L[17] = m2l_fma(D[53], m, L[17]);
      L[18] = m2l_fma(D[54], m, L[18]);
      L[19] = m2l_fma(D[56], m, L[19]);
      L[20] = m2l_fma(D[57], m, L[20]);
      L[21] = m2l_fma(D[59], m, L[21]);
      L[22] = m2l_fma(D[60], m, L[22]);
      L[23] = m2l_fma(D[62], m, L[23]);
      L[24] = m2l_fma(D[63], m, L[24]);
    }
    { const T m = __ldg(Mr + 9);
      L[0] = m2l_fma(D[10], m, L[0]);
      L[1] = m2l_fma(-D[19], m, L[1]);
      L[2] = m2l_fma(-D[20], m, L[2]);
      L[3] = m2l_fma(-D[21], m, L[3]);
      L[4] = m2l_fma(D[31], m, L[4]);
      L[5] = m2l_fma(D[32], m, L[5]);
      L[6] = m2l_fma(D[33], m, L[6]);
      L[7] = m2l_fma(D[34], m, L[7]);
      L[8] = m2l_fma(D[35], m, L[8]);
      L[9] = m2l_fma(-D[46], m, L[9]);
      L[10] = m2l_fma(-D[47], m, L[10]);
      L[11] = m2l_fma(-D[48], m, L[11]);
      L[12] = m2l_fma(-D[49], m, L[12]);
      L[13] = m2l_fma(-D[50], m, L[13]);
      L[14] = m2l_fma(-D[52], m, L[14]);
      L[15] = m2l_fma(-D[53], m, L[15]);
    }
    { const T m = __ldg(Mr + 10);
      L[0] = m2l_fma(D[11], m, L[0]);
      L[1] = m2l_fma(-D[20], m, L[1]);
      L[2] = m2l_fma(-D[22], m, L[2]);
      L[3] = m2l_fma(-D[23], m, L[3]);
      L[4] = m2l_fma(D[32], m, L[4]);
      L[5] = m2l_fma(D[34], m, L[5]);
      L[6] = m2l_fma(D[35], m, L[6]);
      L[7] = m2l_fma(D[37], m, L[7]);
      L[8] = m2l_fma(D[38], m, L[8]);
      L[9] = m2l_fma(-D[47], m, L[9]);
      L[10] = m2l_fma(-D[49], m, L[10]);
      L[11] = m2l_fma(-D[50], m, L[11]);
      L[12] = m2l_fma(-D[52], m, L[12]);
      L[13] = m2l_fma(-D[53], m, L[13]);
      L[14] = m2l_fma(-D[55], m, L[14]);
      L[15] = m2l_fma(-D[56], m, L[15]);
    }
    { const T m = __ldg(Mr + 11);
      L[0] = m2l_fma(D[12], m, L[0]);
      L[1] = m2l_fma(-D[21], m, L[1]);
      L[2] = m2l_fma(-D[23], m, L[2]);
      L[3] = m2l_fma(-D[24], m, L[3]);
      L[4] = m2l_fma(D[33], m, L[4]);
      L[5] = m2l_fma(D[35], m, L[5]);
      L[6] = m2l_fma(D[36], m, L[6]);
      L[7] = m2l_fma(D[38], m, L[7]);
      L[8] = m2l_fma(D[39], m, L[8]);
      L[9] = m2l_fma(-D[48], m, L[9]);
      L[10] = m2l_fma(-D[50], m, L[10]);
      L[11] = m2l_fma(-D[51], m, L[11]);
      L[12] = m2l_fma(-D[53], m, L[12]);
      L[13] = m2l_fma(-D[54], m, L[13]);
      L[14] = m2l_fma(-D[56], m, L[14]);
      L[15] = m2l_fma(-D[57], m, L[15]);
    }
    { const T m = __ldg(Mr + 12);
      L[0] = m2l_fma(D[13], m, L[0]);
      L[1] = m2l_fma(-D[22], m, L[1]);
      L[2] = m2l_fma(-D[25], m, L[2]);
      L[3] = m2l_fma(-D[26], m, L[3]);
      L[4] = m2l_fma(D[34], m, L[4]);
      L[5] = m2l_fma(D[37], m, L[5]);
      L[6] = m2l_fma(D[38], m, L[6]);
      L[7] = m2l_fma(D[40], m, L[7]);
      L[8] = m2l_fma(D[41], m, L[8]);
      L[9] = m2l_fma(-D[49], m, L[9]);
      L[10] = m2l_fma(-D[52], m, L[10]);
      L[11] = m2l_fma(-D[53], m, L[11]);
      L[12] = m2l_fma(-D[55], m, L[12]);
      L[13] = m2l_fma(-D[56], m, L[13]);
      L[14] = m2l_fma(-D[58], m, L[14]);
      L[15] = m2l_fma(-D[59], m, L[15]);
    }
    { const T m = __ldg(Mr + 13);
      L[0] = m2l_fma(D[14], m, L[0]);
      L[1] = m2l_fma(-D[23], m, L[1]);
      L[2] = m2l_fma(-D[26], m, L[2]);
      L[3] = m2l_fma(-D[27], m, L[3]);
      L[4] = m2l_fma(D[35], m, L[4]);
      L[5] = m2l_fma(D[38], m, L[5]);
      L[6] = m2l_fma(D[39], m, L[6]);
      L[7] = m2l_fma(D[41], m, L[7]);
      L[8] = m2l_fma(D[42], m, L[8]);
      L[9] = m2l_fma(-D[50], m, L[9]);
      L[10] = m2l_fma(-D[53], m, L[10]);
      L[11] = m2l_fma(-D[54], m, L[11]);
      L[12] = m2l_fma(-D[56], m, L[12]);
      L[13] = m2l_fma(-D[57], m, L[13]);
      L[14] = m2l_fma(-D[59], m, L[14]);
      L[15] = m2l_fma(-D[60], m, L[15]);
    }
    { const T m = __ldg(Mr + 14);
      L[0] = m2l_fma(D[16], m, L[0]);
      L[1] = m2l_fma(-D[25], m, L[1]);
      L[2] = m2l_fma(-D[28], m, L[2]);
      L[3] = m2l_fma(-D[29], m, L[3]);
      L[4] = m2l_fma(D[37], m, L[4]);
      L[5] = m2l_fma(D[40], m, L[5]);
      L[6] = m2l_fma(D[41], m, L[6]);
      L[7] = m2l_fma(D[43], m, L[7]);
      L[8] = m2l_fma(D[44], m, L[8]);
      L[9] = m2l_fma(-D[52], m, L[9]);
      L[10] = m2l_fma(-D[55], m, L[10]);
      L[11] = m2l_fma(-D[56], m, L[11]);
      L[12] = m2l_fma(-D[58], m, L[12]);
      L[13] = m2l_fma(-D[59], m, L[13]);
      L[14] = m2l_fma(-D[61], m, L[14]);
      L[15] = m2l_fma(-D[62], m, L[15]);
    }
    { const T m = __ldg(Mr + 15);
      L[0] = m2l_fma(D[17], m, L[0]);
      L[1] = m2l_fma(-D[26], m, L[1]);
      L[2] = m2l_fma(-D[29], m, L[2]);
      L[3] = m2l_fma(-D[30], m, L[3]);
      L[4] = m2l_fma(D[38], m, L[4]);
      L[5] = m2l_fma(D[41], m, L[5]);
      L[6] = m2l_fma(D[42], m, L[6]);
      L[7] = m2l_fma(D[44], m, L[7]);
      L[8] = m2l_fma(D[45], m, L[8]);
      L[9] = m2l_fma(-D[53], m, L[9]);
      L[10] = m2l_fma(-D[56], m, L[10]);
      L[11] = m2l_fma(-D[57], m, L[11]);
      L[12] = m2l_fma(-D[59], m, L[12]);
      L[13] = m2l_fma(-D[60], m, L[13]);
      L[14] = m2l_fma(-D[62], m, L[14]);
      L[15] = m2l_fma(-D[63], m, L[15]);
    }
    { const T m = __ldg(Mr + 16);
      L[0] = m2l_fma(D[19], m, L[0]);
      L[1] = m2l_fma(-D[31], m, L[1]);
      L[2] = m2l_fma(-D[32], m, L[2]);
      L[3] = m2l_fma(-D[33], m, L[3]);
      L[4] = m2l_fma(D[46], m, L[4]);
      L[5] = m2l_fma(D[47], m, L[5]);
      L[6] = m2l_fma(D[48], m, L[6]);
      L[7] = m2l_fma(D[49], m, L[7]);
      L[8] = m2l_fma(D[50], m, L[8]);
    }
    { const T m = __ldg(Mr + 17);
      L[0] = m2l_fma(D[20], m, L[0]);
      L[1] = m2l_fma(-D[32], m, L[1]);
      L[2] = m2l_fma(-D[34], m, L[2]);
      L[3] = m2l_fma(-D[35], m, L[3]);
      L[4] = m2l_fma(D[47], m, L[4]);
      L[5] = m2l_fma(D[49], m, L[5]);
      L[6] = m2l_fma(D[50], m, L[6]);
      L[7] = m2l_fma(D[52], m, L[7]);
      L[8] = m2l_fma(D[53], m, L[8]);
    }
    { const T m = __ldg(Mr + 18);
      L[0] = m2l_fma(D[21], m, L[0]);
      L[1] = m2l_fma(-D[33], m, L[1]);
      L[2] = m2l_fma(-D[35], m, L[2]);
      L[3] = m2l_fma(-D[36], m, L[3]);
      L[4] = m2l_fma(D[48], m, L[4]);
      L[5] = m2l_fma(D[50], m, L[5]);
      L[6] = m2l_fma(D[51], m, L[6]);
      L[7] = m2l_fma(D[53], m, L[7]);
      L[8] = m2l_fma(D[54], m, L[8]);
    }
    { const T m = __ldg(Mr + 19);
      L[0] = m2l_fma(D[22], m, L[0]);
      L[1] = m2l_fma(-D[34], m, L[1]);
      L[2] = m2l_fma(-D[37], m, L[2]);
      L[3] = m2l_fma(-D[38], m, L[3]);
      L[4] = m2l_fma(D[49], m, L[4]);
      L[5] = m2l_fma(D[52], m, L[5]);
      L[6] = m2l_fma(D[53], m, L[6]);
      L[7] = m2l_fma(D[55], m, L[7]);
      L[8] = m2l_fma(D[56], m, L[8]);
    }
    { const T m = __ldg(Mr + 20);
      L[0] = m2l_fma(D[23], m, L[0]);
      L[1] = m2l_fma(-D[35], m, L[1]);
      L[2] = m2l_fma(-D[38], m, L[2]);
      L[3] = m2l_fma(-D[39], m, L[3]);
      L[4] = m2l_fma(D[50], m, L[4]);
      L[5] = m2l_fma(D[53], m, L[5]);
      L[6] = m2l_fma(D[54], m, L[6]);
      L[7] = m2l_fma(D[56], m, L[7]);
      L[8] = m2l_fma(D[57], m, L[8]);
    }
    { const T m = __ldg(Mr + 21);
      L[0] = m2l_fma(D[25], m, L[0]);
      L[1] = m2l_fma(-D[37], m, L[1]);
      L[2] = m2l_fma(-D[40], m, L[2]);
      L[3] = m2l_fma(-D[41], m, L[3]);
      L[4] = m2l_fma(D[52], m, L[4]);
      L[5] = m2l_fma(D[55], m, L[5]);
      L[6] = m2l_fma(D[56], m, L[6]);
      L[7] = m2l_fma(D[58], m, L[7]);
      L[8] = m2l_fma(D[59], m, L[8]);
    }
    { const T m = __ldg(Mr + 22);
      L[0] = m2l_fma(D[26], m, L[0]);
      L[1] = m2l_fma(-D[38], m, L[1]);
      L[2] = m2l_fma(-D[41], m, L[2]);
      L[3] = m2l_fma(-D[42], m, L[3]);
      L[4] = m2l_fma(D[53], m, L[4]);
      L[5] = m2l_fma(D[56], m, L[5]);
      L[6] = m2l_fma(D[57], m, L[6]);
      L[7] = m2l_fma(D[59], m, L[7]);
      L[8] = m2l_fma(D[60], m, L[8]);
    }
    { const T m = __ldg(Mr + 23);
      L[0] = m2l_fma(D[28], m, L[0]);
      L[1] = m2l_fma(-D[40], m, L[1]);
      L[2] = m2l_fma(-D[43], m, L[2]);
      L[3] = m2l_fma(-D[44], m, L[3]);
      L[4] = m2l_fma(D[55], m, L[4]);
      L[5] = m2l_fma(D[58], m, L[5]);
      L[6] = m2l_fma(D[59], m, L[6]);
      L[7] = m2l_fma(D[61], m, L[7]);
      L[8] = m2l_fma(D[62], m, L[8]);
    }
    { const T m = __ldg(Mr + 24);
      L[0] = m2l_fma(D[29], m, L[0]);
      L[1] = m2l_fma(-D[41], m, L[1]);
      L[2] = m2l_fma(-D[44], m, L[2]);
      L[3] = m2l_fma(-D[45], m, L[3]);
      L[4] = m2l_fma(D[56], m, L[4]);
      L[5] = m2l_fma(D[59], m, L[5]);
      L[6] = m2l_fma(D[60], m, L[6]);
      L[7] = m2l_fma(D[62], m, L[7]);
      L[8] = m2l_fma(D[63], m, L[8]);
    }
    { const T m = __ldg(Mr + 25);
      L[0] = m2l_fma(D[31], m, L[0]);
      L[1] = m2l_fma(-D[46], m, L[1]);
      L[2] = m2l_fma(-D[47], m, L[2]);
      L[3] = m2l_fma(-D[48], m, L[3]);
    }
    { const T m = __ldg(Mr + 26);
      L[0] = m2l_fma(D[32], m, L[0]);
      L[1] = m2l_fma(-D[47], m, L[1]);
      L[2] = m2l_fma(-D[49], m, L[2]);
      L[3] = m2l_fma(-D[50], m, L[3]);
    }
    { const T m = __ldg(Mr + 27);
      L[0] = m2l_fma(D[33], m, L[0]);
      L[1] = m2l_fma(-D[48], m, L[1]);
      L[2] = m2l_fma(-D[50], m, L[2]);
      L[3] = m2l_fma(-D[51], m, L[3]);
    }
    { const T m = __ldg(Mr + 28);
      L[0] = m2l_fma(D[34], m, L[0]);
      L[1] = m2l_fma(-D[49], m, L[1]);
      L[2] = m2l_fma(-D[52], m, L[2]);
      L[3] = m2l_fma(-D[53], m, L[3]);
    }
    { const T m = __ldg(Mr + 29);
      L[0] = m2l_fma(D[35], m, L[0]);
      L[1] = m2l_fma(-D[50], m, L[1]);
      L[2] = m2l_fma(-D[53], m, L[2]);
      L[3] = m2l_fma(-D[54], m, L[3]);
    }
    { const T m = __ldg(Mr + 30);
      L[0] = m2l_fma(D[37], m, L[0]);
      L[1] = m2l_fma(-D[52], m, L[1]);
      L[2] = m2l_fma(-D[55], m, L[2]);
      L[3] = m2l_fma(-D[56], m, L[3]);
    }
    { const T m = __ldg(Mr + 31);
      L[0] = m2l_fma(D[38], m, L[0]);
      L[1] = m2l_fma(-D[53], m, L[1]);
      L[2] = m2l_fma(-D[56], m, L[2]);
      L[3] = m2l_fma(-D[57], m, L[3]);
    }
    { const T m = __ldg(Mr + 32);
      L[0] = m2l_fma(D[40], m, L[0]);
      L[1] = m2l_fma(-D[55], m, L[1]);
      L[2] = m2l_fma(-D[58], m, L[2]);
      L[3] = m2l_fma(-D[59], m, L[3]);
    }
    { const T m = __ldg(Mr + 33);
      L[0] = m2l_fma(D[41], m, L[0]);
      L[1] = m2l_fma(-D[56], m, L[1]);
      L[2] = m2l_fma(-D[59], m, L[2]);
      L[3] = m2l_fma(-D[60], m, L[3]);
    }
    { const T m = __ldg(Mr + 34);
      L[0] = m2l_fma(D[43], m, L[0]);
      L[1] = m2l_fma(-D[58], m, L[1]);
      L[2] = m2l_fma(-D[61], m, L[2]);
      L[3] = m2l_fma(-D[62], m, L[3]);
    }
    { const T m = __ldg(Mr + 35);
      L[0] = m2l_fma(D[44], m, L[0]);
      L[1] = m2l_fma(-D[59], m, L[1]);
      L[2] = m2l_fma(-D[62], m, L[2]);
      L[3] = m2l_fma(-D[63], m, L[3]);
    }
    { const T m = __ldg(Mr + 36);
      L[0] = m2l_fma(D[46], m, L[0]);
    }
    { const T m = __ldg(Mr + 37);
      L[0] = m2l_fma(D[47], m, L[0]);
    }
    { const T m = __ldg(Mr + 38);
      L[0] = m2l_fma(D[48], m, L[0]);
    }
    { const T m = __ldg(Mr + 39);
      L[0] = m2l_fma(D[49], m, L[0]);
    }
    { const T m = __ldg(Mr + 40);
      L[0] = m2l_fma(D[50], m, L[0]);
    }
    { const T m = __ldg(Mr + 41);
      L[0] = m2l_fma(D[52], m, L[0]);
    }
    { const T m = __ldg(Mr + 42);
      L[0] = m2l_fma(D[53], m, L[0]);
    }
    { const T m = __ldg(Mr + 43);
      L[0] = m2l_fma(D[55], m, L[0]);
    }
    { const T m = __ldg(Mr + 44);
      L[0] = m2l_fma(D[56], m, L[0]);
    }
    { const T m = __ldg(Mr + 45);
      L[0] = m2l_fma(D[58], m, L[0]);
    }
    { const T m = __ldg(Mr + 46);
      L[0] = m2l_fma(D[59], m, L[0]);
    }
    { const T m = __ldg(Mr + 47);
      L[0] = m2l_fma(D[61], m, L[0]);
    }
    { const T m = __ldg(Mr + 48);
      L[0] = m2l_fma(D[62], m, L[0]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_a_h_forces_6(const T (&D)[64], const T *__restrict__ Mr, T rho, T (&L)[49])
{
    L[0] = T(0);
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[1] = D[1] * m;
      L[2] = D[2] * m;
      L[3] = D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = D[10] * m;
      L[10] = D[11] * m;
      L[11] = D[12] * m;
      L[12] = D[13] * m;
      L[13] = D[14] * m;
      L[14] = D[16] * m;
      L[15] = D[17] * m;
      L[16] = D[19] * m;
      L[17] = D[20] * m;
      L[18] = D[21] * m;
      L[19] = D[22] * m;
      L[20] = D[23] * m;
      L[21] = D[25] * m;
      L[22] = D[26] * m;
      L[23] = D[28] * m;
      L[24] = D[29] * m;
      L[25] = D[31] * m;
      L[26] = D[32] * m;
      L[27] = D[33] * m;
      L[28] = D[34] * m;
      L[29] = D[35] * m;
      L[30] = D[37] * m;
      L[31] = D[38] * m;
      L[32] = D[40] * m;
      L[33] = D[41] * m;
      L[34] = D[43] * m;
      L[35] = D[44] * m;
      L[36] = D[46] * m;
      L[37] = D[47] * m;
      L[38] = D[48] * m;
      L[39] = D[49] * m;
      L[40] = D[50] * m;
      L[41] = D[52] * m;
      L[42] = D[53] * m;
      L[43] = D[55] * m;
      L[44] = D[56] * m;
      L[45] = D[58] * m;
      L[46] = D[59] * m;
      L[47] = D[61] * m;
      L[48] = D[62] * m;
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 1) * rp;
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(D[20], m, L[10]);
      L[11] = m2l_fma(D[21], m, L[11]);
      L[12] = m2l_fma(D[22], m, L[12]);
      L[13] = m2l_fma(D[23], m, L[13]);
      L[14] = m2l_fma(D[25], m, L[14]);
      L[15] = m2l_fma(D[26], m, L[15]);
      L[16] = m2l_fma(D[31], m, L[16]);
      L[17] = m2l_fma(D[32], m, L[17]);
      L[18] = m2l_fma(D[33], m, L[18]);
      L[19] = m2l_fma(D[34], m, L[19]);
      L[20] = m2l_fma(D[35], m, L[20]);
      L[21] = m2l_fma(D[37], m, L[21]);
      L[22] = m2l_fma(D[38], m, L[22]);
      L[23] = m2l_fma(D[40], m, L[23]);
      L[24] = m2l_fma(D[41], m, L[24]);
      L[25] = m2l_fma(D[46], m, L[25]);
      L[26] = m2l_fma(D[47], m, L[26]);
      L[27] = m2l_fma(D[48], m, L[27]);
      L[28] = m2l_fma(D[49], m, L[28]);
      L[29] = m2l_fma(D[50], m, L[29]);
      L[30] = m2l_fma(D[52], m, L[30]);
      L[31] = m2l_fma(D[53], m, L[31]);
      L[32] = m2l_fma(D[55], m, L[32]);
      L[33] = m2l_fma(D[56], m, L[33]);
      L[34] = m2l_fma(D[58], m, L[34]);
      L[35] = m2l_fma(D[59], m, L[35]);
    }
    { const T m = -__ldg(Mr + 2) * rp;
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[20], m, L[9]);
      L[10] = m2l_fma(D[22], m, L[10]);
      L[11] = m2l_fma(D[23], m, L[11]);
      L[12] = m2l_fma(D[25], m, L[12]);
      L[13] = m2l_fma(D[26], m, L[13]);
      L[14] = m2l_fma(D[28], m, L[14]);
      L[15] = m2l_fma(D[29], m, L[15]);
      L[16] = m2l_fma(D[32], m, L[16]);
      L[17] = m2l_fma(D[34], m, L[17]);
      L[18] = m2l_fma(D[35], m, L[18]);
      L[19] = m2l_fma(D[37], m, L[19]);
      L[20] = m2l_fma(D[38], m, L[20]);
      L[21] = m2l_fma(D[40], m, L[21]);
      L[22] = m2l_fma(D[41], m, L[22]);
      L[23] = m2l_fma(D[43], m, L[23]);
      L[24] = m2l_fma(D[44], m, L[24]);
      L[25] = m2l_fma(D[47], m, L[25]);
      L[26] = m2l_fma(D[49], m, L[26]);
      L[27] = m2l_fma(D[50], m, L[27]);
      L[28] = m2l_fma(D[52], m, L[28]);
      L[29] = m2l_fma(D[53], m, L[29]);
      L[30] = m2l_fma(D[55], m, L[30]);
      L[31] = m2l_fma(D[56], m, L[31]);
      L[32] = m2l_fma(D[58], m, L[32]);
      L[33] = m2l_fma(D[59], m, L[33]);
      L[34] = m2l_fma(D[61], m, L[34]);
      L[35] = m2l_fma(D[62], m, L[35]);
    }
    { const T m = -__ldg(Mr + 3) * rp;
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[21], m, L[9]);
      L[10] = m2l_fma(D[23], m, L[10]);
      L[11] = m2l_fma(D[24], m, L[11]);
      L[12] = m2l_fma(D[26], m, L[12]);
      L[13] = m2l_fma(D[27], m, L[13]);
      L[14] = m2l_fma(D[29], m, L[14]);
      L[15] = m2l_fma(D[30], m, L[15]);
      L[16] = m2l_fma(D[33], m, L[16]);
      L[17] = m2l_fma(D[35], m, L[17]);
      L[18] = m2l_fma(D[36], m, L[18]);
      L[19] = m2l_fma(D[38], m, L[19]);
      L[20] = m2l_fma(D[39], m, L[20]);
      L[21] = m2l_fma(D[41], m, L[21]);
      L[22] = m2l_fma(D[42], m, L[22]);
      L[23] = m2l_fma(D[44], m, L[23]);
      L[24] = m2l_fma(D[45], m, L[24]);
      L[25] = m2l_fma(D[48], m, L[25]);
      L[26] = m2l_fma(D[50], m, L[26]);
      L[27] = m2l_fma(D[51], m, L[27]);
      L[28] = m2l_fma(D[53], m, L[28]);
      L[29] = m2l_fma(D[54], m, L[29]);
      L[30] = m2l_fma(D[56], m, L[30]);
      L[31] = m2l_fma(D[57], m, L[31]);
      L[32] = m2l_fma(D[59], m, L[32]);
      L[33] = m2l_fma(D[60], m, L[33]);
      L[34] = m2l_fma(D[62], m, L[34]);
      L[35] = m2l_fma(D[63], m, L[35]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 4) * rp;
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
      L[4] = m2l_fma(D[19], m, L[4]);
      L[5] = m2l_fma(D[20], m, L[5]);
      L[6] = m2l_fma(D[21], m, L[6]);
      L[7] = m2l_fma(D[22], m, L[7]);
      L[8] = m2l_fma(D[23], m, L[8]);
      L[9] = m2l_fma(D[31], m, L[9]);
      L[10] = m2l_fma(D[32], m, L[10]);
      L[11] = m2l_fma(D[33], m, L[11]);
      L[12] = m2l_fma(D[34], m, L[12]);
      L[13] = m2l_fma(D[35], m, L[13]);
      L[14] = m2l_fma(D[37], m, L[14]);
      L[15] = m2l_fma(D[38], m, L[15]);
      L[16] = m2l_fma(D[46], m, L[16]);
      L[17] = m2l_fma(D[47], m, L[17]);
      L[18] = m2l_fma(D[48], m, L[18]);
      L[19] = m2l_fma(D[49], m, L[19]);
      L[20] = m2l_fma(D[50], m, L[20]);
      L[21] = m2l_fma(D[52], m, L[21]);
      L[22] = m2l_fma(D[53], m, L[22]);
      L[23] = m2l_fma(D[55], m, L[23]);
      L[24] = m2l_fma(D[56], m, L[24]);
    }
    { const T m = __ldg(Mr + 5) * rp;
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[22], m, L[5]);
      L[6] = m2l_fma(D[23], m, L[6]);
      L[7] = m2l_fma(D[25], m, L[7]);
      L[8] = m2l_fma(D[26], m, L[8]);
      L[9] = m2l_fma(D[32], m, L[9]);
      L[10] = m2l_fma(D[34], m, L[10]);
      L[11] = m2l_fma(D[35], m, L[11]);
      L[12] = m2l_fma(D[37], m, L[12]);
      L[13] = m2l_fma(D[38], m, L[13]);
      L[14] = m2l_fma(D[40], m, L[14]);
      L[15] = m2l_fma(D[41], m, L[15]);
      L[16] = m2l_fma(D[47], m, L[16]);
      L[17] = m2l_fma(D[49], m, L[17]);
      L[18] = m2l_fma(D[50], m, L[18]);
      L[19] = m2l_fma(D[52], m, L[19]);
      L[20] = m2l_fma(D[53], m, L[20]);
      L[21] = m2l_fma(D[55], m, L[21]);
      L[22] = m2l_fma(D[56], m, L[22]);
      L[23] = m2l_fma(D[58], m, L[23]);
      L[24] = m2l_fma(D[59], m, L[24]);
    }
    { const T m = __ldg(Mr + 6) * rp;
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(D[33], m, L[9]);
      L[10] = m2l_fma(D[35], m, L[10]);
      L[11] = m2l_fma(D[36], m, L[11]);
      L[12] = m2l_fma(D[38], m, L[12]);
      L[13] = m2l_fma(D[39], m, L[13]);
      L[14] = m2l_fma(D[41], m, L[14]);
      L[15] = m2l_fma(D[42], m, L[15]);
      L[16] = m2l_fma(D[48], m, L[16]);
      L[17] = m2l_fma(D[50], m, L[17]);
      L[18] = m2l_fma(D[51], m, L[18]);
      L[19] = m2l_fma(D[53], m, L[19]);
      L[20] = m2l_fma(D[54], m, L[20]);
      L[21] = m2l_fma(D[56], m, L[21]);
      L[22] = m2l_fma(D[57], m, L[22]);
      L[23] = m2l_fma(D[59], m, L[23]);
      L[24] = m2l_fma(D[60], m, L[24]);
    }
    { const T m = __ldg(Mr + 7) * rp;
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[25], m, L[5]);
      L[6] = m2l_fma(D[26], m, L[6]);
      L[7] = m2l_fma(D[28], m, L[7]);
      L[8] = m2l_fma(D[29], m, L[8]);
      L[9] = m2l_fma(D[34], m, L[9]);
      L[10] = m2l_fma(D[37], m, L[10]);
      L[11] = m2l_fma(D[38], m, L[11]);
      L[12] = m2l_fma(D[40], m, L[12]);
      L[13] = m2l_fma(D[41], m, L[13]);
      L[14] = m2l_fma(D[43], m, L[14]);
      L[15] = m2l_fma(D[44], m, L[15]);
      L[16] = m2l_fma(D[49], m, L[16]);
      L[17] = m2l_fma(D[52], m, L[17]);
      L[18] = m2l_fma(D[53], m, L[18]);
      L[19] = m2l_fma(D[55], m, L[19]);
      L[20] = m2l_fma(D[56], m, L[20]);
      L[21] = m2l_fma(D[58], m, L[21]);
      L[22] = m2l_fma(D[59], m, L[22]);
      L[23] = m2l_fma(D[61], m, L[23]);
      L[24] = m2l_fma(D[62], m, L[24]);
    }
    { const T m = __ldg(Mr + 8) * rp;
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[29], m, L[7]);
      L[8] = m2l_fma(D[30], m, L[8]);
      L[9] = m2l_fma(D[35], m, L[9]);
      L[10] = m2l_fma(D[38], m, L[10]);
      L[11] = m2l_fma(D[39], m, L[11]);
      L[12] = m2l_fma(D[41], m, L[12]);
      L[13] = m2l_fma(D[42], m, L[13]);
      L[14] = m2l_fma(D[44], m, L[14]);
      L[15] = m2l_fma(D[45], m, L[15]);
      L[16] = m2l_fma(D[50], m, L[16]);
      L[17] = m2l_fma(D[53], m, L[17]);
      L[18] = m2l_fma(D[54], m, L[18]);
      L[19] = m2l_fma(D[56], m, L[19]);
      L[20] = m2l_fma(D[57], m, L[20]);
      L[21] = m2l_fma(D[59], m, L[21]);
      L[22] = m2l_fma(D[60], m, L[22]);
      L[23] = m2l_fma(D[62], m, L[23]);
      L[24] = m2l_fma(D[63], m, L[24]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 9) * rp;
      L[1] = m2l_fma(D[19], m, L[1]);
      L[2] = m2l_fma(D[20], m, L[2]);
      L[3] = m2l_fma(D[21], m, L[3]);
      L[4] = m2l_fma(D[31], m, L[4]);
      L[5] = m2l_fma(D[32], m, L[5]);
      L[6] = m2l_fma(D[33], m, L[6]);
      L[7] = m2l_fma(D[34], m, L[7]);
      L[8] = m2l_fma(D[35], m, L[8]);
      L[9] = m2l_fma(D[46], m, L[9]);
      L[10] = m2l_fma(D[47], m, L[10]);
      L[11] = m2l_fma(D[48], m, L[11]);
      L[12] = m2l_fma(D[49], m, L[12]);
      L[13] = m2l_fma(D[50], m, L[13]);
      L[14] = m2l_fma(D[52], m, L[14]);
      L[15] = m2l_fma(D[53], m, L[15]);
    }
    { const T m = -__ldg(Mr + 10) * rp;
      L[1] = m2l_fma(D[20], m, L[1]);
      L[2] = m2l_fma(D[22], m, L[2]);
      L[3] = m2l_fma(D[23], m, L[3]);
      L[4] = m2l_fma(D[32], m, L[4]);
      L[5] = m2l_fma(D[34], m, L[5]);
      L[6] = m2l_fma(D[35], m, L[6]);
      L[7] = m2l_fma(D[37], m, L[7]);
      L[8] = m2l_fma(D[38], m, L[8]);
      L[9] = m2l_fma(D[47], m, L[9]);
      L[10] = m2l_fma(D[49], m, L[10]);
      L[11] = m2l_fma(D[50], m, L[11]);
      L[12] = m2l_fma(D[52], m, L[12]);
      L[13] = m2l_fma(D[53], m, L[13]);
      L[14] = m2l_fma(D[55], m, L[14]);
      L[15] = m2l_fma(D[56], m, L[15]);
    }
    { const T m = -__ldg(Mr + 11) * rp;
      L[1] = m2l_fma(D[21], m, L[1]);
      L[2] = m2l_fma(D[23], m, L[2]);
      L[3] = m2l_fma(D[24], m, L[3]);
      L[4] = m2l_fma(D[33], m, L[4]);
      L[5] = m2l_fma(D[35], m, L[5]);
      L[6] = m2l_fma(D[36], m, L[6]);
      L[7] = m2l_fma(D[38], m, L[7]);
      L[8] = m2l_fma(D[39], m, L[8]);
      L[9] = m2l_fma(D[48], m, L[9]);
      L[10] = m2l_fma(D[50], m, L[10]);
      L[11] = m2l_fma(D[51], m, L[11]);
      L[12] = m2l_fma(D[53], m, L[12]);
      L[13] = m2l_fma(D[54], m, L[13]);
      L[14] = m2l_fma(D[56], m, L[14]);
      L[15] = m2l_fma(D[57], m, L[15]);
    }
    { const T m = -__ldg(Mr + 12) * rp;
      L[1] = m2l_fma(D[22], m, L[1]);
      L[2] = m2l_fma(D[25], m, L[2]);
      L[3] = m2l_fma(D[26], m, L[3]);
      L[4] = m2l_fma(D[34], m, L[4]);
      L[5] = m2l_fma(D[37], m, L[5]);
      L[6] = m2l_fma(D[38], m, L[6]);
      L[7] = m2l_fma(D[40], m, L[7]);
      L[8] = m2l_fma(D[41], m, L[8]);
      L[9] = m2l_fma(D[49], m, L[9]);
      L[10] = m2l_fma(D[52], m, L[10]);
      L[11] = m2l_fma(D[53], m, L[11]);
      L[12] = m2l_fma(D[55], m, L[12]);
      L[13] = m2l_fma(D[56], m, L[13]);
      L[14] = m2l_fma(D[58], m, L[14]);
      L[15] = m2l_fma(D[59], m, L[15]);
    }
    { const T m = -__ldg(Mr + 13) * rp;
      L[1] = m2l_fma(D[23], m, L[1]);
      L[2] = m2l_fma(D[26], m, L[2]);
      L[3] = m2l_fma(D[27], m, L[3]);
      L[4] = m2l_fma(D[35], m, L[4]);
      L[5] = m2l_fma(D[38], m, L[5]);
      L[6] = m2l_fma(D[39], m, L[6]);
      L[7] = m2l_fma(D[41], m, L[7]);
      L[8] = m2l_fma(D[42], m, L[8]);
      L[9] = m2l_fma(D[50], m, L[9]);
      L[10] = m2l_fma(D[53], m, L[10]);
      L[11] = m2l_fma(D[54], m, L[11]);
      L[12] = m2l_fma(D[56], m, L[12]);
      L[13] = m2l_fma(D[57], m, L[13]);
      L[14] = m2l_fma(D[59], m, L[14]);
      L[15] = m2l_fma(D[60], m, L[15]);
    }
    { const T m = -__ldg(Mr + 14) * rp;
      L[1] = m2l_fma(D[25], m, L[1]);
      L[2] = m2l_fma(D[28], m, L[2]);
      L[3] = m2l_fma(D[29], m, L[3]);
      L[4] = m2l_fma(D[37], m, L[4]);
      L[5] = m2l_fma(D[40], m, L[5]);
      L[6] = m2l_fma(D[41], m, L[6]);
      L[7] = m2l_fma(D[43], m, L[7]);
      L[8] = m2l_fma(D[44], m, L[8]);
      L[9] = m2l_fma(D[52], m, L[9]);
      L[10] = m2l_fma(D[55], m, L[10]);
      L[11] = m2l_fma(D[56], m, L[11]);
      L[12] = m2l_fma(D[58], m, L[12]);
      L[13] = m2l_fma(D[59], m, L[13]);
      L[14] = m2l_fma(D[61], m, L[14]);
      L[15] = m2l_fma(D[62], m, L[15]);
    }
    { const T m = -__ldg(Mr + 15) * rp;
      L[1] = m2l_fma(D[26], m, L[1]);
      L[2] = m2l_fma(D[29], m, L[2]);
      L[3] = m2l_fma(D[30], m, L[3]);
      L[4] = m2l_fma(D[38], m, L[4]);
      L[5] = m2l_fma(D[41], m, L[5]);
      L[6] = m2l_fma(D[42], m, L[6]);
      L[7] = m2l_fma(D[44], m, L[7]);
      L[8] = m2l_fma(D[45], m, L[8]);
      L[9] = m2l_fma(D[53], m, L[9]);
      L[10] = m2l_fma(D[56], m, L[10]);
      L[11] = m2l_fma(D[57], m, L[11]);
      L[12] = m2l_fma(D[59], m, L[12]);
      L[13] = m2l_fma(D[60], m, L[13]);
      L[14] = m2l_fma(D[62], m, L[14]);
      L[15] = m2l_fma(D[63], m, L[15]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 16) * rp;
      L[1] = m2l_fma(D[31], m, L[1]);
      L[2] = m2l_fma(D[32], m, L[2]);
      L[3] = m2l_fma(D[33], m, L[3]);
      L[4] = m2l_fma(D[46], m, L[4]);
      L[5] = m2l_fma(D[47], m, L[5]);
      L[6] = m2l_fma(D[48], m, L[6]);
      L[7] = m2l_fma(D[49], m, L[7]);
      L[8] = m2l_fma(D[50], m, L[8]);
    }
    { const T m = __ldg(Mr + 17) * rp;
      L[1] = m2l_fma(D[32], m, L[1]);
      L[2] = m2l_fma(D[34], m, L[2]);
      L[3] = m2l_fma(D[35], m, L[3]);
      L[4] = m2l_fma(D[47], m, L[4]);
      L[5] = m2l_fma(D[49], m, L[5]);
      L[6] = m2l_fma(D[50], m, L[6]);
      L[7] = m2l_fma(D[52], m, L[7]);
      L[8] = m2l_fma(D[53], m, L[8]);
    }
    { const T m = __ldg(Mr + 18) * rp;
      L[1] = m2l_fma(D[33], m, L[1]);
      L[2] = m2l_fma(D[35], m, L[2]);
      L[3] = m2l_fma(D[36], m, L[3]);
      L[4] = m2l_fma(D[48], m, L[4]);
      L[5] = m2l_fma(D[50], m, L[5]);
      L[6] = m2l_fma(D[51], m, L[6]);
      L[7] = m2l_fma(D[53], m, L[7]);
      L[8] = m2l_fma(D[54], m, L[8]);
    }
    { const T m = __ldg(Mr + 19) * rp;
      L[1] = m2l_fma(D[34], m, L[1]);
      L[2] = m2l_fma(D[37], m, L[2]);
      L[3] = m2l_fma(D[38], m, L[3]);
      L[4] = m2l_fma(D[49], m, L[4]);
      L[5] = m2l_fma(D[52], m, L[5]);
      L[6] = m2l_fma(D[53], m, L[6]);
      L[7] = m2l_fma(D[55], m, L[7]);
      L[8] = m2l_fma(D[56], m, L[8]);
    }
    { const T m = __ldg(Mr + 20) * rp;
      L[1] = m2l_fma(D[35], m, L[1]);
      L[2] = m2l_fma(D[38], m, L[2]);
      L[3] = m2l_fma(D[39], m, L[3]);
      L[4] = m2l_fma(D[50], m, L[4]);
      L[5] = m2l_fma(D[53], m, L[5]);
      L[6] = m2l_fma(D[54], m, L[6]);
      L[7] = m2l_fma(D[56], m, L[7]);
      L[8] = m2l_fma(D[57], m, L[8]);
    }
    { const T m = __ldg(Mr + 21) * rp;
      L[1] = m2l_fma(D[37], m, L[1]);
      L[2] = m2l_fma(D[40], m, L[2]);
      L[3] = m2l_fma(D[41], m, L[3]);
      L[4] = m2l_fma(D[52], m, L[4]);
      L[5] = m2l_fma(D[55], m, L[5]);
      L[6] = m2l_fma(D[56], m, L[6]);
      L[7] = m2l_fma(D[58], m, L[7]);
      L[8] = m2l_fma(D[59], m, L[8]);
    }
    { const T m = __ldg(Mr + 22) * rp;
      L[1] = m2l_fma(D[38], m, L[1]);
      L[2] = m2l_fma(D[41], m, L[2]);
      L[3] = m2l_fma(D[42], m, L[3]);
      L[4] = m2l_fma(D[53], m, L[4]);
      L[5] = m2l_fma(D[56], m, L[5]);
      L[6] = m2l_fma(D[57], m, L[6]);
      L[7] = m2l_fma(D[59], m, L[7]);
      L[8] = m2l_fma(D[60], m, L[8]);
    }
    { const T m = __ldg(Mr + 23) * rp;
      L[1] = m2l_fma(D[40], m, L[1]);
      L[2] = m2l_fma(D[43], m, L[2]);
      L[3] = m2l_fma(D[44], m, L[3]);
      L[4] = m2l_fma(D[55], m, L[4]);
      L[5] = m2l_fma(D[58], m, L[5]);
      L[6] = m2l_fma(D[59], m, L[6]);
      L[7] = m2l_fma(D[61], m, L[7]);
      L[8] = m2l_fma(D[62], m, L[8]);
    }
    { const T m = __ldg(Mr + 24) * rp;
      L[1] = m2l_fma(D[41], m, L[1]);
      L[2] = m2l_fma(D[44], m, L[2]);
      L[3] = m2l_fma(D[45], m, L[3]);
      L[4] = m2l_fma(D[56], m, L[4]);
      L[5] = m2l_fma(D[59], m, L[5]);
      L[6] = m2l_fma(D[60], m, L[6]);
      L[7] = m2l_fma(D[62], m, L[7]);
      L[8] = m2l_fma(D[63], m, L[8]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 25) * rp;
      L[1] = m2l_fma(D[46], m, L[1]);
      L[2] = m2l_fma(D[47], m, L[2]);
      L[3] = m2l_fma(D[48], m, L[3]);
    }
    { const T m = -__ldg(Mr + 26) * rp;
      L[1] = m2l_fma(D[47], m, L[1]);
      L[2] = m2l_fma(D[49], m, L[2]);
      L[3] = m2l_fma(D[50], m, L[3]);
    }
    { const T m = -__ldg(Mr + 27) * rp;
      L[1] = m2l_fma(D[48], m, L[1]);
      L[2] = m2l_fma(D[50], m, L[2]);
      L[3] = m2l_fma(D[51], m, L[3]);
    }
    { const T m = -__ldg(Mr + 28) * rp;
      L[1] = m2l_fma(D[49], m, L[1]);
      L[2] = m2l_fma(D[52], m, L[2]);
      L[3] = m2l_fma(D[53], m, L[3]);
    }
    { const T m = -__ldg(Mr + 29) * rp;
      L[1] = m2l_fma(D[50], m, L[1]);
      L[2] = m2l_fma(D[53], m, L[2]);
      L[3] = m2l_fma(D[54], m, L[3]);
    }
    { const T m = -__ldg(Mr + 30) * rp;
      L[1] = m2l_fma(D[52], m, L[1]);
      L[2] = m2l_fma(D[55], m, L[2]);
      L[3] = m2l_fma(D[56], m, L[3]);
    }
    { const T m = -__ldg(Mr + 31) * rp;
      L[1] = m2l_fma(D[53], m, L[1]);
      L[2] = m2l_fma(D[56], m, L[2]);
      L[3] = m2l_fma(D[57], m, L[3]);
    }
    { const T m = -__ldg(Mr + 32) * rp;
      L[1] = m2l_fma(D[55], m, L[1]);
      L[2] = m2l_fma(D[58], m, L[2]);
      L[3] = m2l_fma(D[59], m, L[3]);
    }
    { const T m = -__ldg(Mr + 33) * rp;
      L[1] = m2l_fma(D[56], m, L[1]);
      L[2] = m2l_fma(D[59], m, L[2]);
      L[3] = m2l_fma(D[60], m, L[3]);
    }
    { const T m = -__ldg(Mr + 34) * rp;
      L[1] = m2l_fma(D[58], m, L[1]);
      L[2] = m2l_fma(D[61], m, L[2]);
      L[3] = m2l_fma(D[62], m, L[3]);
    }
    { const T m = -__ldg(Mr + 35) * rp;
      L[1] = m2l_fma(D[59], m, L[1]);
      L[2] = m2l_fma(D[62], m, L[2]);
      L[3] = m2l_fma(D[63], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_acc_h_forces_6(const T (&D)[64], const T *__restrict__ Mr, T rho, T (&L)[49])
{
    T rp = T(1);
    { const T m = __ldg(Mr + 0) * rp;
      L[1] = m2l_fma(D[1], m, L[1]);
      L[2] = m2l_fma(D[2], m, L[2]);
      L[3] = m2l_fma(D[3], m, L[3]);
      L[4] = m2l_fma(D[4], m, L[4]);
      L[5] = m2l_fma(D[5], m, L[5]);
      L[6] = m2l_fma(D[6], m, L[6]);
      L[7] = m2l_fma(D[7], m, L[7]);
      L[8] = m2l_fma(D[8], m, L[8]);
      L[9] = m2l_fma(D[10], m, L[9]);
      L[10] = m2l_fma(D[11], m, L[10]);
      L[11] = m2l_fma(D[12], m, L[11]);
      L[12] = m2l_fma(D[13], m, L[12]);
      L[13] = m2l_fma(D[14], m, L[13]);
      L[14] = m2l_fma(D[16], m, L[14]);
      L[15] = m2l_fma(D[17], m, L[15]);
      L[16] = m2l_fma(D[19], m, L[16]);
      L[17] = m2l_fma(D[20], m, L[17]);
      L[18] = m2l_fma(D[21], m, L[18]);
      L[19] = m2l_fma(D[22], m, L[19]);
      L[20] = m2l_fma(D[23], m, L[20]);
      L[21] = m2l_fma(D[25], m, L[21]);
      L[22] = m2l_fma(D[26], m, L[22]);
      L[23] = m2l_fma(D[28], m, L[23]);
      L[24] = m2l_fma(D[29], m, L[24]);
      L[25] = m2l_fma(D[31], m, L[25]);
      L[26] = m2l_fma(D[32], m, L[26]);
      L[27] = m2l_fma(D[33], m, L[27]);
      L[28] = m2l_fma(D[34], m, L[28]);
      L[29] = m2l_fma(D[35], m, L[29]);
      L[30] = m2l_fma(D[37], m, L[30]);
      L[31] = m2l_fma(D[38], m, L[31]);
      L[32] = m2l_fma(D[40], m, L[32]);
      L[33] = m2l_fma(D[41], m, L[33]);
      L[34] = m2l_fma(D[43], m, L[34]);
      L[35] = m2l_fma(D[44], m, L[35]);
      L[36] = m2l_fma(D[46], m, L[36]);
      L[37] = m2l_fma(D[47], m, L[37]);
      L[38] = m2l_fma(D[48], m, L[38]);
      L[39] = m2l_fma(D[49], m, L[39]);
      L[40] = m2l_fma(D[50], m, L[40]);
      L[41] = m2l_fma(D[52], m, L[41]);
      L[42] = m2l_fma(D[53], m, L[42]);
      L[43] = m2l_fma(D[55], m, L[43]);
      L[44] = m2l_fma(D[56], m, L[44]);
      L[45] = m2l_fma(D[58], m, L[45]);
      L[46] = m2l_fma(D[59], m, L[46]);
      L[47] = m2l_fma(D[61], m, L[47]);
      L[48] = m2l_fma(D[62], m, L[48]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 1) * rp;
      L[1] = m2l_fma(D[4], m, L[1]);
      L[2] = m2l_fma(D[5], m, L[2]);
      L[3] = m2l_fma(D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(D[19], m, L[9]);
      L[10] = m2l_fma(D[20], m, L[10]);
      L[11] = m2l_fma(D[21], m, L[11]);
      L[12] = m2l_fma(D[22], m, L[12]);
      L[13] = m2l_fma(D[23], m, L[13]);
      L[14] = m2l_fma(D[25], m, L[14]);
      L[15] = m2l_fma(D[26], m, L[15]);
      L[16] = m2l_fma(D[31], m, L[16]);
      L[17] = m2l_fma(D[32], m, L[17]);
      L[18] = m2l_fma(D[33], m, L[18]);
      L[19] = m2l_fma(D[34], m, L[19]);
      L[20] = m2l_fma(D[35], m, L[20]);
      L[21] = m2l_fma(D[37], m, L[21]);
      L[22] = m2l_fma(D[38], m, L[22]);
      L[23] = m2l_fma(D[40], m, L[23]);
      L[24] = m2l_fma(D[41], m, L[24]);
      L[25] = m2l_fma(D[46], m, L[25]);
      L[26] = m2l_fma(D[47], m, L[26]);
      L[27] = m2l_fma(D[48], m, L[27]);
      L[28] = m2l_fma(D[49], m, L[28]);
      L[29] = m2l_fma(D[50], m, L[29]);
      L[30] = m2l_fma(D[52], m, L[30]);
      L[31] = m2l_fma(D[53], m, L[31]);
      L[32] = m2l_fma(D[55], m, L[32]);
      L[33] = m2l_fma(D[56], m, L[33]);
      L[34] = m2l_fma(D[58], m, L[34]);
      L[35] = m2l_fma(D[59], m, L[35]);
    }
    { const T m = -__ldg(Mr + 2) * rp;
      L[1] = m2l_fma(D[5], m, L[1]);
      L[2] = m2l_fma(D[7], m, L[2]);
      L[3] = m2l_fma(D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(D[20], m, L[9]);
      L[10] = m2l_fma(D[22], m, L[10]);
      L[11] = m2l_fma(D[23], m, L[11]);
      L[12] = m2l_fma(D[25], m, L[12]);
      L[13] = m2l_fma(D[26], m, L[13]);
      L[14] = m2l_fma(D[28], m, L[14]);
      L[15] = m2l_fma(D[29], m, L[15]);
      L[16] = m2l_fma(D[32], m, L[16]);
      L[17] = m2l_fma(D[34], m, L[17]);
      L[18] = m2l_fma(D[35], m, L[18]);
      L[19] = m2l_fma(D[37], m, L[19]);
      L[20] = m2l_fma(D[38], m, L[20]);
      L[21] = m2l_fma(D[40], m, L[21]);
      L[22] = m2l_fma(D[41], m, L[22]);
      L[23] = m2l_fma(D[43], m, L[23]);
      L[24] = m2l_fma(D[44], m, L[24]);
      L[25] = m2l_fma(D[47], m, L[25]);
      L[26] = m2l_fma(D[49], m, L[26]);
      L[27] = m2l_fma(D[50], m, L[27]);
      L[28] = m2l_fma(D[52], m, L[28]);
      L[29] = m2l_fma(D[53], m, L[29]);
      L[30] = m2l_fma(D[55], m, L[30]);
      L[31] = m2l_fma(D[56], m, L[31]);
      L[32] = m2l_fma(D[58], m, L[32]);
      L[33] = m2l_fma(D[59], m, L[33]);
      L[34] = m2l_fma(D[61], m, L[34]);
      L[35] = m2l_fma(D[62], m, L[35]);
    }
    { const T m = -__ldg(Mr + 3) * rp;
      L[1] = m2l_fma(D[6], m, L[1]);
      L[2] = m2l_fma(D[8], m, L[2]);
      L[3] = m2l_fma(D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(D[21], m, L[9]);
      L[10] = m2l_fma(D[23], m, L[10]);
      L[11] = m2l_fma(D[24], m, L[11]);
      L[12] = m2l_fma(D[26], m, L[12]);
      L[13] = m2l_fma(D[27], m, L[13]);
      L[14] = m2l_fma(D[29], m, L[14]);
      L[15] = m2l_fma(D[30], m, L[15]);
      L[16] = m2l_fma(D[33], m, L[16]);
      L[17] = m2l_fma(D[35], m, L[17]);
      L[18] = m2l_fma(D[36], m, L[18]);
      L[19] = m2l_fma(D[38], m, L[19]);
      L[20] = m2l_fma(D[39], m, L[20]);
      L[21] = m2l_fma(D[41], m, L[21]);
      L[22] = m2l_fma(D[42], m, L[22]);
      L[23] = m2l_fma(D[44], m, L[23]);
      L[24] = m2l_fma(D[45], m, L[24]);
      L[25] = m2l_fma(D[48], m, L[25]);
      L[26] = m2l_fma(D[50], m, L[26]);
      L[27] = m2l_fma(D[51], m, L[27]);
      L[28] = m2l_fma(D[53], m, L[28]);
      L[29] = m2l_fma(D[54], m, L[29]);
      L[30] = m2l_fma(D[56], m, L[30]);
      L[31] = m2l_fma(D[57], m, L[31]);
      L[32] = m2l_fma(D[59], m, L[32]);
      L[33] = m2l_fma(D[60], m, L[33]);
      L[34] = m2l_fma(D[62], m, L[34]);
      L[35] = m2l_fma(D[63], m, L[35]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 4) * rp;
      L[1] = m2l_fma(D[10], m, L[1]);
      L[2] = m2l_fma(D[11], m, L[2]);
      L[3] = m2l_fma(D[12], m, L[3]);
      L[4] = m2l_fma(D[19], m, L[4]);
      L[5] = m2l_fma(D[20], m, L[5]);
      L[6] = m2l_fma(D[21], m, L[6]);
      L[7] = m2l_fma(D[22], m, L[7]);
      L[8] = m2l_fma(D[23], m, L[8]);
      L[9] = m2l_fma(D[31], m, L[9]);
      L[10] = m2l_fma(D[32], m, L[10]);
      L[11] = m2l_fma(D[33], m, L[11]);
      L[12] = m2l_fma(D[34], m, L[12]);
      L[13] = m2l_fma(D[35], m, L[13]);
      L[14] = m2l_fma(D[37], m, L[14]);
      L[15] = m2l_fma(D[38], m, L[15]);
      L[16] = m2l_fma(D[46], m, L[16]);
      L[17] = m2l_fma(D[47], m, L[17]);
      L[18] = m2l_fma(D[48], m, L[18]);
      L[19] = m2l_fma(D[49], m, L[19]);
      L[20] = m2l_fma(D[50], m, L[20]);
      L[21] = m2l_fma(D[52], m, L[21]);
      L[22] = m2l_fma(D[53], m, L[22]);
      L[23] = m2l_fma(D[55], m, L[23]);
      L[24] = m2l_fma(D[56], m, L[24]);
    }
    { const T m = __ldg(Mr + 5) * rp;
      L[1] = m2l_fma(D[11], m, L[1]);
      L[2] = m2l_fma(D[13], m, L[2]);
      L[3] = m2l_fma(D[14], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[22], m, L[5]);
      L[6] = m2l_fma(D[23], m, L[6]);
      L[7] = m2l_fma(D[25], m, L[7]);
      L[8] = m2l_fma(D[26], m, L[8]);
      L[9] = m2l_fma(D[32], m, L[9]);
      L[10] = m2l_fma(D[34], m, L[10]);
      L[11] = m2l_fma(D[35], m, L[11]);
      L[12] = m2l_fma(D[37], m, L[12]);
      L[13] = m2l_fma(D[38], m, L[13]);
      L[14] = m2l_fma(D[40], m, L[14]);
      L[15] = m2l_fma(D[41], m, L[15]);
      L[16] = m2l_fma(D[47], m, L[16]);
      L[17] = m2l_fma(D[49], m, L[17]);
      L[18] = m2l_fma(D[50], m, L[18]);
      L[19] = m2l_fma(D[52], m, L[19]);
      L[20] = m2l_fma(D[53], m, L[20]);
      L[21] = m2l_fma(D[55], m, L[21]);
      L[22] = m2l_fma(D[56], m, L[22]);
      L[23] = m2l_fma(D[58], m, L[23]);
      L[24] = m2l_fma(D[59], m, L[24]);
    }
    { const T m = __ldg(Mr + 6) * rp;
      L[1] = m2l_fma(D[12], m, L[1]);
      L[2] = m2l_fma(D[14], m, L[2]);
      L[3] = m2l_fma(D[15], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(D[33], m, L[9]);
      L[10] = m2l_fma(D[35], m, L[10]);
      L[11] = m2l_fma(D[36], m, L[11]);
      L[12] = m2l_fma(D[38], m, L[12]);
      L[13] = m2l_fma(D[39], m, L[13]);
      L[14] = m2l_fma(D[41], m, L[14]);
      L[15] = m2l_fma(D[42], m, L[15]);
      L[16] = m2l_fma(D[48], m, L[16]);
      L[17] = m2l_fma(D[50], m, L[17]);
      L[18] = m2l_fma(D[51], m, L[18]);
      L[19] = m2l_fma(D[53], m, L[19]);
      L[20] = m2l_fma(D[54], m, L[20]);
      L[21] = m2l_fma(D[56], m, L[21]);
      L[22] = m2l_fma(D[57], m, L[22]);
      L[23] = m2l_fma(D[59], m, L[23]);
      L[24] = m2l_fma(D[60], m, L[24]);
    }
    { const T m = __ldg(Mr + 7) * rp;
      L[1] = m2l_fma(D[13], m, L[1]);
      L[2] = m2l_fma(D[16], m, L[2]);
      L[3] = m2l_fma(D[17], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[25], m, L[5]);
      L[6] = m2l_fma(D[26], m, L[6]);
      L[7] = m2l_fma(D[28], m, L[7]);
      L[8] = m2l_fma(D[29], m, L[8]);
      L[9] = m2l_fma(D[34], m, L[9]);
      L[10] = m2l_fma(D[37], m, L[10]);
      L[11] = m2l_fma(D[38], m, L[11]);
      L[12] = m2l_fma(D[40], m, L[12]);
      L[13] = m2l_fma(D[41], m, L[13]);
      L[14] = m2l_fma(D[43], m, L[14]);
      L[15] = m2l_fma(D[44], m, L[15]);
      L[16] = m2l_fma(D[49], m, L[16]);
      L[17] = m2l_fma(D[52], m, L[17]);
      L[18] = m2l_fma(D[53], m, L[18]);
      L[19] = m2l_fma(D[55], m, L[19]);
      L[20] = m2l_fma(D[56], m, L[20]);
      L[21] = m2l_fma(D[58], m, L[21]);
      L[22] = m2l_fma(D[59], m, L[22]);
      L[23] = m2l_fma(D[61], m, L[23]);
      L[24] = m2l_fma(D[62], m, L[24]);
    }
    { const T m = __ldg(Mr + 8) * rp;
      L[1] = m2l_fma(D[14], m, L[1]);
      L[2] = m2l_fma(D[17], m, L[2]);
      L[3] = m2l_fma(D[18], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[29], m, L[7]);
      L[8] = m2l_fma(D[30], m, L[8]);
      L[9] = m2l_fma(D[35], m, L[9]);
      L[10] = m2l_fma(D[38], m, L[10]);
      L[11] = m2l_fma(D[39], m, L[11]);
      L[12] = m2l_fma(D[41], m, L[12]);
      L[13] = m2l_fma(D[42], m, L[13]);
      L[14] = m2l_fma(D[44], m, L[14]);
      L[15] = m2l_fma(D[45], m, L[15]);
      L[16] = m2l_fma(D[50], m, L[16]);
      L[17] = m2l_fma(D[53], m, L[17]);
      L[18] = m2l_fma(D[54], m, L[18]);
      L[19] = m2l_fma(D[56], m, L[19]);
      L[20] = m2l_fma(D[57], m, L[20]);
      L[21] = m2l_fma(D[59], m, L[21]);
      L[22] = m2l_fma(D[60], m, L[22]);
      L[23] = m2l_fma(D[62], m, L[23]);
      L[24] = m2l_fma(D[63], m, L[24]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 9) * rp;
      L[1] = m2l_fma(D[19], m, L[1]);
      L[2] = m2l_fma(D[20], m, L[2]);
      L[3] = m2l_fma(D[21], m, L[3]);
      L[4] = m2l_fma(D[31], m, L[4]);
      L[5] = m2l_fma(D[32], m, L[5]);
      L[6] = m2l_fma(D[33], m, L[6]);
      L[7] = m2l_fma(D[34], m, L[7]);
      L[8] = m2l_fma(D[35], m, L[8]);
      L[9] = m2l_fma(D[46], m, L[9]);
      L[10] = m2l_fma(D[47], m, L[10]);
      L[11] = m2l_fma(D[48], m, L[11]);
      L[12] = m2l_fma(D[49], m, L[12]);
      L[13] = m2l_fma(D[50], m, L[13]);
      L[14] = m2l_fma(D[52], m, L[14]);
      L[15] = m2l_fma(D[53], m, L[15]);
    }
    { const T m = -__ldg(Mr + 10) * rp;
      L[1] = m2l_fma(D[20], m, L[1]);
      L[2] = m2l_fma(D[22], m, L[2]);
      L[3] = m2l_fma(D[23], m, L[3]);
      L[4] = m2l_fma(D[32], m, L[4]);
      L[5] = m2l_fma(D[34], m, L[5]);
      L[6] = m2l_fma(D[35], m, L[6]);
      L[7] = m2l_fma(D[37], m, L[7]);
      L[8] = m2l_fma(D[38], m, L[8]);
      L[9] = m2l_fma(D[47], m, L[9]);
      L[10] = m2l_fma(D[49], m, L[10]);
      L[11] = m2l_fma(D[50], m, L[11]);
      L[12] = m2l_fma(D[52], m, L[12]);
      L[13] = m2l_fma(D[53], m, L[13]);
      L[14] = m2l_fma(D[55], m, L[14]);
      L[15] = m2l_fma(D[56], m, L[15]);
    }
    { const T m = -__ldg(Mr + 11) * rp;
      L[1] = m2l_fma(D[21], m, L[1]);
      L[2] = m2l_fma(D[23], m, L[2]);
      L[3] = m2l_fma(D[24], m, L[3]);
      L[4] = m2l_fma(D[33], m, L[4]);
      L[5] = m2l_fma(D[35], m, L[5]);
      L[6] = m2l_fma(D[36], m, L[6]);
      L[7] = m2l_fma(D[38], m, L[7]);
      L[8] = m2l_fma(D[39], m, L[8]);
      L[9] = m2l_fma(D[48], m, L[9]);
      L[10] = m2l_fma(D[50], m, L[10]);
      L[11] = m2l_fma(D[51], m, L[11]);
      L[12] = m2l_fma(D[53], m, L[12]);
      L[13] = m2l_fma(D[54], m, L[13]);
      L[14] = m2l_fma(D[56], m, L[14]);
      L[15] = m2l_fma(D[57], m, L[15]);
    }
    { const T m = -__ldg(Mr + 12) * rp;
      L[1] = m2l_fma(D[22], m, L[1]);
      L[2] = m2l_fma(D[25], m, L[2]);
      L[3] = m2l_fma(D[26], m, L[3]);
      L[4] = m2l_fma(D[34], m, L[4]);
      L[5] = m2l_fma(D[37], m, L[5]);
      L[6] = m2l_fma(D[38], m, L[6]);
      L[7] = m2l_fma(D[40], m, L[7]);
      L[8] = m2l_fma(D[41], m, L[8]);
      L[9] = m2l_fma(D[49], m, L[9]);
      L[10] = m2l_fma(D[52], m, L[10]);
      L[11] = m2l_fma(D[53], m, L[11]);
      L[12] = m2l_fma(D[55], m, L[12]);
      L[13] = m2l_fma(D[56], m, L[13]);
      L[14] = m2l_fma(D[58], m, L[14]);
      L[15] = m2l_fma(D[59], m, L[15]);
    }
    { const T m = -__ldg(Mr + 13) * rp;
      L[1] = m2l_fma(D[23], m, L[1]);
      L[2] = m2l_fma(D[26], m, L[2]);
      L[3] = m2l_fma(D[27], m, L[3]);
      L[4] = m2l_fma(D[35], m, L[4]);
      L[5] = m2l_fma(D[38], m, L[5]);
      L[6] = m2l_fma(D[39], m, L[6]);
      L[7] = m2l_fma(D[41], m, L[7]);
      L[8] = m2l_fma(D[42], m, L[8]);
      L[9] = m2l_fma(D[50], m, L[9]);
      L[10] = m2l_fma(D[53], m, L[10]);
      L[11] = m2l_fma(D[54], m, L[11]);
      L[12] = m2l_fma(D[56], m, L[12]);
      L[13] = m2l_fma(D[57], m, L[13]);
      L[14] = m2l_fma(D[59], m, L[14]);
      L[15] = m2l_fma(D[60], m, L[15]);
    }
    { const T m = -__ldg(Mr + 14) * rp;
      L[1] = m2l_fma(D[25], m, L[1]);
      L[2] = m2l_fma(D[28], m, L[2]);
      L[3] = m2l_fma(D[29], m, L[3]);
      L[4] = m2l_fma(D[37], m, L[4]);
      L[5] = m2l_fma(D[40], m, L[5]);
      L[6] = m2l_fma(D[41], m, L[6]);
      L[7] = m2l_fma(D[43], m, L[7]);
      L[8] = m2l_fma(D[44], m, L[8]);
      L[9] = m2l_fma(D[52], m, L[9]);
      L[10] = m2l_fma(D[55], m, L[10]);
      L[11] = m2l_fma(D[56], m, L[11]);
      L[12] = m2l_fma(D[58], m, L[12]);
      L[13] = m2l_fma(D[59], m, L[13]);
      L[14] = m2l_fma(D[61], m, L[14]);
      L[15] = m2l_fma(D[62], m, L[15]);
    }
    { const T m = -__ldg(Mr + 15) * rp;
      L[1] = m2l_fma(D[26], m, L[1]);
      L[2] = m2l_fma(D[29], m, L[2]);
      L[3] = m2l_fma(D[30], m, L[3]);
      L[4] = m2l_fma(D[38], m, L[4]);
      L[5] = m2l_fma(D[41], m, L[5]);
      L[6] = m2l_fma(D[42], m, L[6]);
      L[7] = m2l_fma(D[44], m, L[7]);
      L[8] = m2l_fma(D[45], m, L[8]);
      L[9] = m2l_fma(D[53], m, L[9]);
      L[10] = m2l_fma(D[56], m, L[10]);
      L[11] = m2l_fma(D[57], m, L[11]);
      L[12] = m2l_fma(D[59], m, L[12]);
      L[13] = m2l_fma(D[60], m, L[13]);
      L[14] = m2l_fma(D[62], m, L[14]);
      L[15] = m2l_fma(D[63], m, L[15]);
    }
    rp *= rho;
    { const T m = __ldg(Mr + 16) * rp;
      L[1] = m2l_fma(D[31], m, L[1]);
      L[2] = m2l_fma(D[32], m, L[2]);
      L[3] = m2l_fma(D[33], m, L[3]);
      L[4] = m2l_fma(D[46], m, L[4]);
      L[5] = m2l_fma(D[47], m, L[5]);
      L[6] = m2l_fma(D[48], m, L[6]);
      L[7] = m2l_fma(D[49], m, L[7]);
      L[8] = m2l_fma(D[50], m, L[8]);
    }
    { const T m = __ldg(Mr + 17) * rp;
      L[1] = m2l_fma(D[32], m, L[1]);
      L[2] = m2l_fma(D[34], m, L[2]);
      L[3] = m2l_fma(D[35], m, L[3]);
      L[4] = m2l_fma(D[47], m, L[4]);
      L[5] = m2l_fma(D[49], m, L[5]);
      L[6] = m2l_fma(D[50], m, L[6]);
      L[7] = m2l_fma(D[52], m, L[7]);
      L[8] = m2l_fma(D[53], m, L[8]);
    }
    { const T m = __ldg(Mr + 18) * rp;
      L[1] = m2l_fma(D[33], m, L[1]);
      L[2] = m2l_fma(D[35], m, L[2]);
      L[3] = m2l_fma(D[36], m, L[3]);
      L[4] = m2l_fma(D[48], m, L[4]);
      L[5] = m2l_fma(D[50], m, L[5]);
      L[6] = m2l_fma(D[51], m, L[6]);
      L[7] = m2l_fma(D[53], m, L[7]);
      L[8] = m2l_fma(D[54], m, L[8]);
    }
    { const T m = __ldg(Mr + 19) * rp;
      L[1] = m2l_fma(D[34], m, L[1]);
      L[2] = m2l_fma(D[37], m, L[2]);
      L[3] = m2l_fma(D[38], m, L[3]);
      L[4] = m2l_fma(D[49], m, L[4]);
      L[5] = m2l_fma(D[52], m, L[5]);
      L[6] = m2l_fma(D[53], m, L[6]);
      L[7] = m2l_fma(D[55], m, L[7]);
      L[8] = m2l_fma(D[56], m, L[8]);
    }
    { const T m = __ldg(Mr + 20) * rp;
      L[1] = m2l_fma(D[35], m, L[1]);
      L[2] = m2l_fma(D[38], m, L[2]);
      L[3] = m2l_fma(D[39], m, L[3]);
      L[4] = m2l_fma(D[50], m, L[4]);
      L[5] = m2l_fma(D[53], m, L[5]);
      L[6] = m2l_fma(D[54], m, L[6]);
      L[7] = m2l_fma(D[56], m, L[7]);
      L[8] = m2l_fma(D[57], m, L[8]);
    }
    { const T m = __ldg(Mr + 21) * rp;
      L[1] = m2l_fma(D[37], m, L[1]);
      L[2] = m2l_fma(D[40], m, L[2]);
      L[3] = m2l_fma(D[41], m, L[3]);
      L[4] = m2l_fma(D[52], m, L[4]);
      L[5] = m2l_fma(D[55], m, L[5]);
      L[6] = m2l_fma(D[56], m, L[6]);
      L[7] = m2l_fma(D[58], m, L[7]);
      L[8] = m2l_fma(D[59], m, L[8]);
    }
    { const T m = __ldg(Mr + 22) * rp;
      L[1] = m2l_fma(D[38], m, L[1]);
      L[2] = m2l_fma(D[41], m, L[2]);
      L[3] = m2l_fma(D[42], m, L[3]);
      L[4] = m2l_fma(D[53], m, L[4]);
      L[5] = m2l_fma(D[56], m, L[5]);
      L[6] = m2l_fma(D[57], m, L[6]);
      L[7] = m2l_fma(D[59], m, L[7]);
      L[8] = m2l_fma(D[60], m, L[8]);
    }
    { const T m = __ldg(Mr + 23) * rp;
      L[1] = m2l_fma(D[40], m, L[1]);
      L[2] = m2l_fma(D[43], m, L[2]);
      L[3] = m2l_fma(D[44], m, L[3]);
      L[4] = m2l_fma(D[55], m, L[4]);
      L[5] = m2l_fma(D[58], m, L[5]);
      L[6] = m2l_fma(D[59], m, L[6]);
      L[7] = m2l_fma(D[61], m, L[7]);
      L[8] = m2l_fma(D[62], m, L[8]);
    }
    { const T m = __ldg(Mr + 24) * rp;
      L[1] = m2l_fma(D[41], m, L[1]);
      L[2] = m2l_fma(D[44], m, L[2]);
      L[3] = m2l_fma(D[45], m, L[3]);
      L[4] = m2l_fma(D[56], m, L[4]);
      L[5] = m2l_fma(D[59], m, L[5]);
      L[6] = m2l_fma(D[60], m, L[6]);
      L[7] = m2l_fma(D[62], m, L[7]);
      L[8] = m2l_fma(D[63], m, L[8]);
    }
    rp *= rho;
    { const T m = -__ldg(Mr + 25) * rp;
      L[1] = m2l_fma(D[46], m, L[1]);
      L[2] = m2l_fma(D[47], m, L[2]);
      L[3] = m2l_fma(D[48], m, L[3]);
    }
    { const T m = -__ldg(Mr + 26) * rp;
      L[1] = m2l_fma(D[47], m, L[1]);
      L[2] = m2l_fma(D[49], m, L[2]);
      L[3] = m2l_fma(D[50], m, L[3]);
    }
    { const T m = -__ldg(Mr + 27) * rp;
      L[1] = m2l_fma(D[48], m, L[1]);
      L[2] = m2l_fma(D[50], m, L[2]);
      L[3] = m2l_fma(D[51], m, L[3]);
    }
    { const T m = -__ldg(Mr + 28) * rp;
      L[1] = m2l_fma(D[49], m, L[1]);
      L[2] = m2l_fma(D[52], m, L[2]);
      L[3] = m2l_fma(D[53], m, L[3]);
    }
    { const T m = -__ldg(Mr + 29) * rp;
      L[1] = m2l_fma(D[50], m, L[1]);
      L[2] = m2l_fma(D[53], m, L[2]);
      L[3] = m2l_fma(D[54], m, L[3]);
    }
    { const T m = -__ldg(Mr + 30) * rp;
      L[1] = m2l_fma(D[52], m, L[1]);
      L[2] = m2l_fma(D[55], m, L[2]);
      L[3] = m2l_fma(D[56], m, L[3]);
    }
    { const T m = -__ldg(Mr + 31) * rp;
      L[1] = m2l_fma(D[53], m, L[1]);
      L[2] = m2l_fma(D[56], m, L[2]);
      L[3] = m2l_fma(D[57], m, L[3]);
    }
    { const T m = -__ldg(Mr + 32) * rp;
      L[1] = m2l_fma(D[55], m, L[1]);
      L[2] = m2l_fma(D[58], m, L[2]);
      L[3] = m2l_fma(D[59], m, L[3]);
    }
    { const T m = -__ldg(Mr + 33) * rp;
      L[1] = m2l_fma(D[56], m, L[1]);
      L[2] = m2l_fma(D[59], m, L[2]);
      L[3] = m2l_fma(D[60], m, L[3]);
    }
    { const T m = -__ldg(Mr + 34) * rp;
      L[1] = m2l_fma(D[58], m, L[1]);
      L[2] = m2l_fma(D[61], m, L[2]);
      L[3] = m2l_fma(D[62], m, L[3]);
    }
    { const T m = -__ldg(Mr + 35) * rp;
      L[1] = m2l_fma(D[59], m, L[1]);
      L[2] = m2l_fma(D[62], m, L[2]);
      L[3] = m2l_fma(D[63], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_side_b_h_forces_6(const T (&D)[64], const T *__restrict__ Mr, T (&L)[49])
{
    L[0] = T(0);
    { const T m = __ldg(Mr + 0);
      L[1] = -D[1] * m;
      L[2] = -D[2] * m;
      L[3] = -D[3] * m;
      L[4] = D[4] * m;
      L[5] = D[5] * m;
      L[6] = D[6] * m;
      L[7] = D[7] * m;
      L[8] = D[8] * m;
      L[9] = -D[10] * m;
      L[10] = -D[11] * m;
      L[11] = -D[12] * m;
      L[12] = -D[13] * m;
      L[13] = -D[14] * m;
      L[14] = -D[16] * m;
      L[15] = -D[17] * m;
      L[16] = D[19] * m;
      L[17] = D[20] * m;
      L[18] = D[21] * m;
      L[19] = D[22] * m;
      L[20] = D[23] * m;
      L[21] = D[25] * m;
      L[22] = D[26] * m;
      L[23] = D[28] * m;
      L[24] = D[29] * m;
      L[25] = -D[31] * m;
      L[26] = -D[32] * m;
      L[27] = -D[33] * m;
      L[28] = -D[34] * m;
      L[29] = -D[35] * m;
      L[30] = -D[37] * m;
      L[31] = -D[38] * m;
      L[32] = -D[40] * m;
      L[33] = -D[41] * m;
      L[34] = -D[43] * m;
      L[35] = -D[44] * m;
      L[36] = D[46] * m;
      L[37] = D[47] * m;
      L[38] = D[48] * m;
      L[39] = D[49] * m;
      L[40] = D[50] * m;
      L[41] = D[52] * m;
      L[42] = D[53] * m;
      L[43] = D[55] * m;
      L[44] = D[56] * m;
      L[45] = D[58] * m;
      L[46] = D[59] * m;
      L[47] = D[61] * m;
      L[48] = D[62] * m;
    }
    { const T m = __ldg(Mr + 1);
      L[1] = m2l_fma(-D[4], m, L[1]);
      L[2] = m2l_fma(-D[5], m, L[2]);
      L[3] = m2l_fma(-D[6], m, L[3]);
      L[4] = m2l_fma(D[10], m, L[4]);
      L[5] = m2l_fma(D[11], m, L[5]);
      L[6] = m2l_fma(D[12], m, L[6]);
      L[7] = m2l_fma(D[13], m, L[7]);
      L[8] = m2l_fma(D[14], m, L[8]);
      L[9] = m2l_fma(-D[19], m, L[9]);
      L[10] = m2l_fma(-D[20], m, L[10]);
      L[11] = m2l_fma(-D[21], m, L[11]);
      L[12] = m2l_fma(-D[22], m, L[12]);
      L[13] = m2l_fma(-D[23], m, L[13]);
      L[14] = m2l_fma(-D[25], m, L[14]);
      L[15] = m2l_fma(-D[26], m, L[15]);
      L[16] = m2l_fma(D[31], m, L[16]);
      L[17] = m2l_fma(D[32], m, L[17]);
      L[18] = m2l_fma(D[33], m, L[18]);
      L[19] = m2l_fma(D[34], m, L[19]);
      L[20] = m2l_fma(D[35], m, L[20]);
      L[21] = m2l_fma(D[37], m, L[21]);
      L[22] = m2l_fma(D[38], m, L[22]);
      L[23] = m2l_fma(D[40], m, L[23]);
      L[24] = m2l_fma(D[41], m, L[24]);
      L[25] = m2l_fma(-D[46], m, L[25]);
      L[26] = m2l_fma(-D[47], m, L[26]);
      L[27] = m2l_fma(-D[48], m, L[27]);
      L[28] = m2l_fma(-D[49], m, L[28]);
      L[29] = m2l_fma(-D[50], m, L[29]);
      L[30] = m2l_fma(-D[52], m, L[30]);
      L[31] = m2l_fma(-D[53], m, L[31]);
      L[32] = m2l_fma(-D[55], m, L[32]);
      L[33] = m2l_fma(-D[56], m, L[33]);
      L[34] = m2l_fma(-D[58], m, L[34]);
      L[35] = m2l_fma(-D[59], m, L[35]);
    }
    { const T m = __ldg(Mr + 2);
      L[1] = m2l_fma(-D[5], m, L[1]);
      L[2] = m2l_fma(-D[7], m, L[2]);
      L[3] = m2l_fma(-D[8], m, L[3]);
      L[4] = m2l_fma(D[11], m, L[4]);
      L[5] = m2l_fma(D[13], m, L[5]);
      L[6] = m2l_fma(D[14], m, L[6]);
      L[7] = m2l_fma(D[16], m, L[7]);
      L[8] = m2l_fma(D[17], m, L[8]);
      L[9] = m2l_fma(-D[20], m, L[9]);
      L[10] = m2l_fma(-D[22], m, L[10]);
      L[11] = m2l_fma(-D[23], m, L[11]);
      L[12] = m2l_fma(-D[25], m, L[12]);
      L[13] = m2l_fma(-D[26], m, L[13]);
      L[14] = m2l_fma(-D[28], m, L[14]);
      L[15] = m2l_fma(-D[29], m, L[15]);
      L[16] = m2l_fma(D[32], m, L[16]);
      L[17] = m2l_fma(D[34], m, L[17]);
      L[18] = m2l_fma(D[35], m, L[18]);
      L[19] = m2l_fma(D[37], m, L[19]);
      L[20] = m2l_fma(D[38], m, L[20]);
      L[21] = m2l_fma(D[40], m, L[21]);
      L[22] = m2l_fma(D[41], m, L[22]);
      L[23] = m2l_fma(D[43], m, L[23]);
      L[24] = m2l_fma(D[44], m, L[24]);
      L[25] = m2l_fma(-D[47], m, L[25]);
      L[26] = m2l_fma(-D[49], m, L[26]);
      L[27] = m2l_fma(-D[50], m, L[27]);
      L[28] = m2l_fma(-D[52], m, L[28]);
      L[29] = m2l_fma(-D[53], m, L[29]);
      L[30] = m2l_fma(-D[55], m, L[30]);
      L[31] = m2l_fma(-D[56], m, L[31]);
      L[32] = m2l_fma(-D[58], m, L[32]);
      L[33] = m2l_fma(-D[59], m, L[33]);
      L[34] = m2l_fma(-D[61], m, L[34]);
      L[35] = m2l_fma(-D[62], m, L[35]);
    }
    { const T m = __ldg(Mr + 3);
      L[1] = m2l_fma(-D[6], m, L[1]);
      L[2] = m2l_fma(-D[8], m, L[2]);
      L[3] = m2l_fma(-D[9], m, L[3]);
      L[4] = m2l_fma(D[12], m, L[4]);
      L[5] = m2l_fma(D[14], m, L[5]);
      L[6] = m2l_fma(D[15], m, L[6]);
      L[7] = m2l_fma(D[17], m, L[7]);
      L[8] = m2l_fma(D[18], m, L[8]);
      L[9] = m2l_fma(-D[21], m, L[9]);
      L[10] = m2l_fma(-D[23], m, L[10]);
      L[11] = m2l_fma(-D[24], m, L[11]);
      L[12] = m2l_fma(-D[26], m, L[12]);
      L[13] = m2l_fma(-D[27], m, L[13]);
      L[14] = m2l_fma(-D[29], m, L[14]);
      L[15] = m2l_fma(-D[30], m, L[15]);
      L[16] = m2l_fma(D[33], m, L[16]);
      L[17] = m2l_fma(D[35], m, L[17]);
      L[18] = m2l_fma(D[36], m, L[18]);
      L[19] = m2l_fma(D[38], m, L[19]);
      L[20] = m2l_fma(D[39], m, L[20]);
      L[21] = m2l_fma(D[41], m, L[21]);
      L[22] = m2l_fma(D[42], m, L[22]);
      L[23] = m2l_fma(D[44], m, L[23]);
      L[24] = m2l_fma(D[45], m, L[24]);
      L[25] = m2l_fma(-D[48], m, L[25]);
      L[26] = m2l_fma(-D[50], m, L[26]);
      L[27] = m2l_fma(-D[51], m, L[27]);
      L[28] = m2l_fma(-D[53], m, L[28]);
      L[29] = m2l_fma(-D[54], m, L[29]);
      L[30] = m2l_fma(-D[56], m, L[30]);
      L[31] = m2l_fma(-D[57], m, L[31]);
      L[32] = m2l_fma(-D[59], m, L[32]);
      L[33] = m2l_fma(-D[60], m, L[33]);
      L[34] = m2l_fma(-D[62], m, L[34]);
      L[35] = m2l_fma(-D[63], m, L[35]);
    }
    { const T m = __ldg(Mr + 4);
      L[1] = m2l_fma(-D[10], m, L[1]);
      L[2] = m2l_fma(-D[11], m, L[2]);
      L[3] = m2l_fma(-D[12], m, L[3]);
      L[4] = m2l_fma(D[19], m, L[4]);
      L[5] = m2l_fma(D[20], m, L[5]);
      L[6] = m2l_fma(D[21], m, L[6]);
      L[7] = m2l_fma(D[22], m, L[7]);
      L[8] = m2l_fma(D[23], m, L[8]);
      L[9] = m2l_fma(-D[31], m, L[9]);
      L[10] = m2l_fma(-D[32], m, L[10]);
      L[11] = m2l_fma(-D[33], m, L[11]);
      L[12] = m2l_fma(-D[34], m, L[12]);
      L[13] = m2l_fma(-D[35], m, L[13]);
      L[14] = m2l_fma(-D[37], m, L[14]);
      L[15] = m2l_fma(-D[38], m, L[15]);
      L[16] = m2l_fma(D[46], m, L[16]);
      L[17] = m2l_fma(D[47], m, L[17]);
      L[18] = m2l_fma(D[48], m, L[18]);
      L[19] = m2l_fma(D[49], m, L[19]);
      L[20] = m2l_fma(D[50], m, L[20]);
      L[21] = m2l_fma(D[52], m, L[21]);
      L[22] = m2l_fma(D[53], m, L[22]);
      L[23] = m2l_fma(D[55], m, L[23]);
      L[24] = m2l_fma(D[56], m, L[24]);
    }
    { const T m = __ldg(Mr + 5);
      L[1] = m2l_fma(-D[11], m, L[1]);
      L[2] = m2l_fma(-D[13], m, L[2]);
      L[3] = m2l_fma(-D[14], m, L[3]);
      L[4] = m2l_fma(D[20], m, L[4]);
      L[5] = m2l_fma(D[22], m, L[5]);
      L[6] = m2l_fma(D[23], m, L[6]);
      L[7] = m2l_fma(D[25], m, L[7]);
      L[8] = m2l_fma(D[26], m, L[8]);
      L[9] = m2l_fma(-D[32], m, L[9]);
      L[10] = m2l_fma(-D[34], m, L[10]);
      L[11] = m2l_fma(-D[35], m, L[11]);
      L[12] = m2l_fma(-D[37], m, L[12]);
      L[13] = m2l_fma(-D[38], m, L[13]);
      L[14] = m2l_fma(-D[40], m, L[14]);
      L[15] = m2l_fma(-D[41], m, L[15]);
      L[16] = m2l_fma(D[47], m, L[16]);
      L[17] = m2l_fma(D[49], m, L[17]);
      L[18] = m2l_fma(D[50], m, L[18]);
      L[19] = m2l_fma(D[52], m, L[19]);
      L[20] = m2l_fma(D[53], m, L[20]);
      L[21] = m2l_fma(D[55], m, L[21]);
      L[22] = m2l_fma(D[56], m, L[22]);
      L[23] = m2l_fma(D[58], m, L[23]);
      L[24] = m2l_fma(D[59], m, L[24]);
    }
    { const T m = __ldg(Mr + 6);
      L[1] = m2l_fma(-D[12], m, L[1]);
      L[2] = m2l_fma(-D[14], m, L[2]);
      L[3] = m2l_fma(-D[15], m, L[3]);
      L[4] = m2l_fma(D[21], m, L[4]);
      L[5] = m2l_fma(D[23], m, L[5]);
      L[6] = m2l_fma(D[24], m, L[6]);
      L[7] = m2l_fma(D[26], m, L[7]);
      L[8] = m2l_fma(D[27], m, L[8]);
      L[9] = m2l_fma(-D[33], m, L[9]);
      L[10] = m2l_fma(-D[35], m, L[10]);
      L[11] = m2l_fma(-D[36], m, L[11]);
      L[12] = m2l_fma(-D[38], m, L[12]);
      L[13] = m2l_fma(-D[39], m, L[13]);
      L[14] = m2l_fma(-D[41], m, L[14]);
      L[15] = m2l_fma(-D[42], m, L[15]);
      L[16] = m2l_fma(D[48], m, L[16]);
      L[17] = m2l_fma(D[50], m, L[17]);
      L[18] = m2l_fma(D[51], m, L[18]);
      L[19] = m2l_fma(D[53], m, L[19]);
      L[20] = m2l_fma(D[54], m, L[20]);
      L[21] = m2l_fma(D[56], m, L[21]);
      L[22] = m2l_fma(D[57], m, L[22]);
      L[23] = m2l_fma(D[59], m, L[23]);
      L[24] = m2l_fma(D[60], m, L[24]);
    }
    { const T m = __ldg(Mr + 7);
      L[1] = m2l_fma(-D[13], m, L[1]);
      L[2] = m2l_fma(-D[16], m, L[2]);
      L[3] = m2l_fma(-D[17], m, L[3]);
      L[4] = m2l_fma(D[22], m, L[4]);
      L[5] = m2l_fma(D[25], m, L[5]);
      L[6] = m2l_fma(D[26], m, L[6]);
      L[7] = m2l_fma(D[28], m, L[7]);
      L[8] = m2l_fma(D[29], m, L[8]);
      L[9] = m2l_fma(-D[34], m, L[9]);
      L[10] = m2l_fma(-D[37], m, L[10]);
      L[11] = m2l_fma(-D[38], m, L[11]);
      L[12] = m2l_fma(-D[40], m, L[12]);
      L[13] = m2l_fma(-D[41], m, L[13]);
      L[14] = m2l_fma(-D[43], m, L[14]);
      L[15] = m2l_fma(-D[44], m, L[15]);
      L[16] = m2l_fma(D[49], m, L[16]);
      L[17] = m2l_fma(D[52], m, L[17]);
      L[18] = m2l_fma(D[53], m, L[18]);
      L[19] = m2l_fma(D[55], m, L[19]);
      L[20] = m2l_fma(D[56], m, L[20]);
      L[21] = m2l_fma(D[58], m, L[21]);
      L[22] = m2l_fma(D[59], m, L[22]);
      L[23] = m2l_fma(D[61], m, L[23]);
      L[24] = m2l_fma(D[62], m, L[24]);
    }
    { const T m = __ldg(Mr + 8);
      L[1] = m2l_fma(-D[14], m, L[1]);
      L[2] = m2l_fma(-D[17], m, L[2]);
      L[3] = m2l_fma(-D[18], m, L[3]);
      L[4] = m2l_fma(D[23], m, L[4]);
      L[5] = m2l_fma(D[26], m, L[5]);
      L[6] = m2l_fma(D[27], m, L[6]);
      L[7] = m2l_fma(D[29], m, L[7]);
      L[8] = m2l_fma(D[30], m, L[8]);
      L[9] = m2l_fma(-D[35], m, L[9]);
      L[10] = m2l_fma(-D[38], m, L[10]);
      L[11] = m2l_fma(-D[39], m, L[11]);
      L[12] = m2l_fma(-D[41], m, L[12]);
      L[13] = m2l_fma(-D[42], m, L[13]);
      L[14] = m2l_fma(-D[44], m, L[14]);
      L[15] = m2l_fma(-D[45], m, L[15]);
      L[16] = m2l_fma(D[50], m, L[16]);
      L[17] = m2l_fma(D[53], m, L[17]);
      L[18] = m2l_fma(D[54], m, L[18]);
      L[19] = m2l_fma(D[56], m, L[19]);
      L[20] = m2l_fma(D[57], m, L[20]);
      L[21] = m2l_fma(D[59], m, L[21]);
      L[22] = m2l_fma(D[60], m, L[22]);
      L[23] = m2l_fma(D[62], m, L[23]);
      L[24] = m2l_fma(D[63], m, L[24]);
    }
    { const T m = __ldg(Mr + 9);
      L[1] = m2l_fma(-D[19], m, L[1]);
      L[2] = m2l_fma(-D[20], m, L[2]);
      L[3] = m2l_fma(-D[21], m, L[3]);
      L[4] = m2l_fma(D[31], m, L[4]);
      L[5] = m2l_fma(D[32], m, L[5]);
      L[6] = m2l_fma(D[33], m, L[6]);
      L[7] = m2l_fma(D[34], m, L[7]);
      L[8] = m2l_fma(D[35], m, L[8]);
      L[9] = m2l_fma(-D[46], m, L[9]);
      L[10] = m2l_fma(-D[47], m, L[10]);
      L[11] = m2l_fma(-D[48], m, L[11]);
      L[12] = m2l_fma(-D[49], m, L[12]);
      L[13] = m2l_fma(-D[50], m, L[13]);
      L[14] = m2l_fma(-D[52], m, L[14]);
      L[15] = m2l_fma(-D[53], m, L[15]);
    }
    { const T m = __ldg(Mr + 10);
      L[1] = m2l_fma(-D[20], m, L[1]);
      L[2] = m2l_fma(-D[22], m, L[2]);
      L[3] = m2l_fma(-D[23], m, L[3]);
      L[4] = m2l_fma(D[32], m, L[4]);
      L[5] = m2l_fma(D[34], m, L[5]);
      L[6] = m2l_fma(D[35], m, L[6]);
      L[7] = m2l_fma(D[37], m, L[7]);
      L[8] = m2l_fma(D[38], m, L[8]);
      L[9] = m2l_fma(-D[47], m, L[9]);
      L[10] = m2l_fma(-D[49], m, L[10]);
      L[11] = m2l_fma(-D[50], m, L[11]);
      L[12] = m2l_fma(-D[52], m, L[12]);
      L[13] = m2l_fma(-D[53], m, L[13]);
      L[14] = m2l_fma(-D[55], m, L[14]);
      L[15] = m2l_fma(-D[56], m, L[15]);
    }
    { const T m = __ldg(Mr + 11);
      L[1] = m2l_fma(-D[21], m, L[1]);
      L[2] = m2l_fma(-D[23], m, L[2]);
      L[3] = m2l_fma(-D[24], m, L[3]);
      L[4] = m2l_fma(D[33], m, L[4]);
      L[5] = m2l_fma(D[35], m, L[5]);
      L[6] = m2l_fma(D[36], m, L[6]);
      L[7] = m2l_fma(D[38], m, L[7]);
      L[8] = m2l_fma(D[39], m, L[8]);
      L[9] = m2l_fma(-D[48], m, L[9]);
      L[10] = m2l_fma(-D[50], m, L[10]);
      L[11] = m2l_fma(-D[51], m, L[11]);
      L[12] = m2l_fma(-D[53], m, L[12]);
      L[13] = m2l_fma(-D[54], m, L[13]);
      L[14] = m2l_fma(-D[56], m, L[14]);
      L[15] = m2l_fma(-D[57], m, L[15]);
    }
    { const T m = __ldg(Mr + 12);
      L[1] = m2l_fma(-D[22], m, L[1]);
      L[2] = m2l_fma(-D[25], m, L[2]);
      L[3] = m2l_fma(-D[26], m, L[3]);
      L[4] = m2l_fma(D[34], m, L[4]);
      L[5] = m2l_fma(D[37], m, L[5]);
      L[6] = m2l_fma(D[38], m, L[6]);
      L[7] = m2l_fma(D[40], m, L[7]);
      L[8] = m2l_fma(D[41], m, L[8]);
      L[9] = m2l_fma(-D[49], m, L[9]);
      L[10] = m2l_fma(-D[52], m, L[10]);
      L[11] = m2l_fma(-D[53], m, L[11]);
      L[12] = m2l_fma(-D[55], m, L[12]);
      L[13] = m2l_fma(-D[56], m, L[13]);
      L[14] = m2l_fma(-D[58], m, L[14]);
      L[15] = m2l_fma(-D[59], m, L[15]);
    }
    { const T m = __ldg(Mr + 13);
      L[1] = m2l_fma(-D[23], m, L[1]);
      L[2] = m2l_fma(-D[26], m, L[2]);
      L[3] = m2l_fma(-D[27], m, L[3]);
      L[4] = m2l_fma(D[35], m, L[4]);
      L[5] = m2l_fma(D[38], m, L[5]);
      L[6] = m2l_fma(D[39], m, L[6]);
      L[7] = m2l_fma(D[41], m, L[7]);
      L[8] = m2l_fma(D[42], m, L[8]);
      L[9] = m2l_fma(-D[50], m, L[9]);
      L[10] = m2l_fma(-D[53], m, L[10]);
      L[11] = m2l_fma(-D[54], m, L[11]);
      L[12] = m2l_fma(-D[56], m, L[12]);
      L[13] = m2l_fma(-D[57], m, L[13]);
      L[14] = m2l_fma(-D[59], m, L[14]);
      L[15] = m2l_fma(-D[60], m, L[15]);
    }
    { const T m = __ldg(Mr + 14);
      L[1] = m2l_fma(-D[25], m, L[1]);
      L[2] = m2l_fma(-D[28], m, L[2]);
      L[3] = m2l_fma(-D[29], m, L[3]);
      L[4] = m2l_fma(D[37], m, L[4]);
      L[5] = m2l_fma(D[40], m, L[5]);
      L[6] = m2l_fma(D[41], m, L[6]);
      L[7] = m2l_fma(D[43], m, L[7]);
      L[8] = m2l_fma(D[44], m, L[8]);
      L[9] = m2l_fma(-D[52], m, L[9]);
      L[10] = m2l_fma(-D[55], m, L[10]);
      L[11] = m2l_fma(-D[56], m, L[11]);
      L[12] = m2l_fma(-D[58], m, L[12]);
      L[13] = m2l_fma(-D[59], m, L[13]);
      L[14] = m2l_fma(-D[61], m, L[14]);
      L[15] = m2l_fma(-D[62], m, L[15]);
    }
    { const T m = __ldg(Mr + 15);
      L[1] = m2l_fma(-D[26], m, L[1]);
      L[2] = m2l_fma(-D[29], m, L[2]);
      L[3] = m2l_fma(-D[30], m, L[3]);
      L[4] = m2l_fma(D[38], m, L[4]);
      L[5] = m2l_fma(D[41], m, L[5]);
      L[6] = m2l_fma(D[42], m, L[6]);
      L[7] = m2l_fma(D[44], m, L[7]);
      L[8] = m2l_fma(D[45], m, L[8]);
      L[9] = m2l_fma(-D[53], m, L[9]);
      L[10] = m2l_fma(-D[56], m, L[10]);
      L[11] = m2l_fma(-D[57], m, L[11]);
      L[12] = m2l_fma(-D[59], m, L[12]);
      L[13] = m2l_fma(-D[60], m, L[13]);
      L[14] = m2l_fma(-D[62], m, L[14]);
      L[15] = m2l_fma(-D[63], m, L[15]);
    }
    { const T m = __ldg(Mr + 16);
      L[1] = m2l_fma(-D[31], m, L[1]);
      L[2] = m2l_fma(-D[32], m, L[2]);
      L[3] = m2l_fma(-D[33], m, L[3]);
      L[4] = m2l_fma(D[46], m, L[4]);
      L[5] = m2l_fma(D[47], m, L[5]);
      L[6] = m2l_fma(D[48], m, L[6]);
      L[7] = m2l_fma(D[49], m, L[7]);
      L[8] = m2l_fma(D[50], m, L[8]);
    }
    { const T m = __ldg(Mr + 17);
      L[1] = m2l_fma(-D[32], m, L[1]);
      L[2] = m2l_fma(-D[34], m, L[2]);
      L[3] = m2l_fma(-D[35], m, L[3]);
      L[4] = m2l_fma(D[47], m, L[4]);
      L[5] = m2l_fma(D[49], m, L[5]);
      L[6] = m2l_fma(D[50], m, L[6]);
      L[7] = m2l_fma(D[52], m, L[7]);
      L[8] = m2l_fma(D[53], m, L[8]);
    }
    { const T m = __ldg(Mr + 18);
      L[1] = m2l_fma(-D[33], m, L[1]);
      L[2] = m2l_fma(-D[35], m, L[2]);
      L[3] = m2l_fma(-D[36], m, L[3]);
      L[4] = m2l_fma(D[48], m, L[4]);
      L[5] = m2l_fma(D[50], m, L[5]);
      L[6] = m2l_fma(D[51], m, L[6]);
      L[7] = m2l_fma(D[53], m, L[7]);
      L[8] = m2l_fma(D[54], m, L[8]);
    }
    { const T m = __ldg(Mr + 19);
      L[1] = m2l_fma(-D[34], m, L[1]);
      L[2] = m2l_fma(-D[37], m, L[2]);
      L[3] = m2l_fma(-D[38], m, L[3]);
      L[4] = m2l_fma(D[49], m, L[4]);
      L[5] = m2l_fma(D[52], m, L[5]);
      L[6] = m2l_fma(D[53], m, L[6]);
      L[7] = m2l_fma(D[55], m, L[7]);
      L[8] = m2l_fma(D[56], m, L[8]);
    }
    { const T m = __ldg(Mr + 20);
      L[1] = m2l_fma(-D[35], m, L[1]);
      L[2] = m2l_fma(-D[38], m, L[2]);
      L[3] = m2l_fma(-D[39], m, L[3]);
      L[4] = m2l_fma(D[50], m, L[4]);
      L[5] = m2l_fma(D[53], m, L[5]);
      L[6] = m2l_fma(D[54], m, L[6]);
      L[7] = m2l_fma(D[56], m, L[7]);
      L[8] = m2l_fma(D[57], m, L[8]);
    }
    { const T m = __ldg(Mr + 21);
      L[1] = m2l_fma(-D[37], m, L[1]);
      L[2] = m2l_fma(-D[40], m, L[2]);
      L[3] = m2l_fma(-D[41], m, L[3]);
      L[4] = m2l_fma(D[52], m, L[4]);
      L[5] = m2l_fma(D[55], m, L[5]);
      L[6] = m2l_fma(D[56], m, L[6]);
      L[7] = m2l_fma(D[58], m, L[7]);
      L[8] = m2l_fma(D[59], m, L[8]);
    }
    { const T m = __ldg(Mr + 22);
      L[1] = m2l_fma(-D[38], m, L[1]);
      L[2] = m2l_fma(-D[41], m, L[2]);
      L[3] = m2l_fma(-D[42], m, L[3]);
      L[4] = m2l_fma(D[53], m, L[4]);
      L[5] = m2l_fma(D[56], m, L[5]);
      L[6] = m2l_fma(D[57], m, L[6]);
      L[7] = m2l_fma(D[59], m, L[7]);
      L[8] = m2l_fma(D[60], m, L[8]);
    }
    { const T m = __ldg(Mr + 23);
      L[1] = m2l_fma(-D[40], m, L[1]);
      L[2] = m2l_fma(-D[43], m, L[2]);
      L[3] = m2l_fma(-D[44], m, L[3]);
      L[4] = m2l_fma(D[55], m, L[4]);
      L[5] = m2l_fma(D[58], m, L[5]);
      L[6] = m2l_fma(D[59], m, L[6]);
      L[7] = m2l_fma(D[61], m, L[7]);
      L[8] = m2l_fma(D[62], m, L[8]);
    }
    { const T m = __ldg(Mr + 24);
      L[1] = m2l_fma(-D[41], m, L[1]);
      L[2] = m2l_fma(-D[44], m, L[2]);
      L[3] = m2l_fma(-D[45], m, L[3]);
      L[4] = m2l_fma(D[56], m, L[4]);
      L[5] = m2l_fma(D[59], m, L[5]);
      L[6] = m2l_fma(D[60], m, L[6]);
      L[7] = m2l_fma(D[62], m, L[7]);
      L[8] = m2l_fma(D[63], m, L[8]);
    }
    { const T m = __ldg(Mr + 25);
      L[1] = m2l_fma(-D[46], m, L[1]);
      L[2] = m2l_fma(-D[47], m, L[2]);
      L[3] = m2l_fma(-D[48], m, L[3]);
    }
    { const T m = __ldg(Mr + 26);
      L[1] = m2l_fma(-D[47], m, L[1]);
      L[2] = m2l_fma(-D[49], m, L[2]);
      L[3] = m2l_fma(-D[50], m, L[3]);
    }
    { const T m = __ldg(Mr + 27);
      L[1] = m2l_fma(-D[48], m, L[1]);
      L[2] = m2l_fma(-D[50], m, L[2]);
      L[3] = m2l_fma(-D[51], m, L[3]);
    }
    { const T m = __ldg(Mr + 28);
      L[1] = m2l_fma(-D[49], m, L[1]);
      L[2] = m2l_fma(-D[52], m, L[2]);
      L[3] = m2l_fma(-D[53], m, L[3]);
    }
    { const T m = __ldg(Mr + 29);
      L[1] = m2l_fma(-D[50], m, L[1]);
      L[2] = m2l_fma(-D[53], m, L[2]);
      L[3] = m2l_fma(-D[54], m, L[3]);
    }
    { const T m = __ldg(Mr + 30);
      L[1] = m2l_fma(-D[52], m, L[1]);
      L[2] = m2l_fma(-D[55], m, L[2]);
      L[3] = m2l_fma(-D[56], m, L[3]);
    }
    { const T m = __ldg(Mr + 31);
      L[1] = m2l_fma(-D[53], m, L[1]);
      L[2] = m2l_fma(-D[56], m, L[2]);
      L[3] = m2l_fma(-D[57], m, L[3]);
    }
    { const T m = __ldg(Mr + 32);
      L[1] = m2l_fma(-D[55], m, L[1]);
      L[2] = m2l_fma(-D[58], m, L[2]);
      L[3] = m2l_fma(-D[59], m, L[3]);
    }
    { const T m = __ldg(Mr + 33);
      L[1] = m2l_fma(-D[56], m, L[1]);
      L[2] = m2l_fma(-D[59], m, L[2]);
      L[3] = m2l_fma(-D[60], m, L[3]);
    }
    { const T m = __ldg(Mr + 34);
      L[1] = m2l_fma(-D[58], m, L[1]);
      L[2] = m2l_fma(-D[61], m, L[2]);
      L[3] = m2l_fma(-D[62], m, L[3]);
    }
    { const T m = __ldg(Mr + 35);
      L[1] = m2l_fma(-D[59], m, L[1]);
      L[2] = m2l_fma(-D[62], m, L[2]);
      L[3] = m2l_fma(-D[63], m, L[3]);
    }
}

template <class T> __device__ __forceinline__ void m2l_reduce_moments_h_6(const T *__restrict__ Ms, T *__restrict__ Mr)
{
    T v0 = Ms[0];
    T v1 = Ms[1];
    T v2 = Ms[2];
    T v3 = Ms[3];
    T v4 = Ms[4];
    T v5 = Ms[5];
    T v6 = Ms[6];
    T v7 = Ms[7];
    T v8 = Ms[8];
    T v9 = Ms[9];
    T v10 = Ms[10];
    T v11 = Ms[11];
    T v12 = Ms[12];
    T v13 = Ms[13];
    T v14 = Ms[14];
    T v15 = Ms[15];
    T v16 = Ms[16];
    T v17 = Ms[17];
    T v18 = Ms[18];
    T v19 = Ms[19];
    T v20 = Ms[20];
    T v21 = Ms[21];
    T v22 = Ms[22];
    T v23 = Ms[23];
    T v24 = Ms[24];
    T v25 = Ms[25];
    T v26 = Ms[26];
    T v27 = Ms[27];
    T v28 = Ms[28];
    T v29 = Ms[29];
    T v30 = Ms[30];
    T v31 = Ms[31];
    T v32 = Ms[32];
    T v33 = Ms[33];
    T v34 = Ms[34];
    T v35 = Ms[35];
    T v36 = Ms[36];
    T v37 = Ms[37];
    T v38 = Ms[38];
    T v39 = Ms[39];
    T v40 = Ms[40];
    T v41 = Ms[41];
    T v42 = Ms[42];
    T v43 = Ms[43];
    T v44 = Ms[44];
    T v45 = Ms[45];
    T v46 = Ms[46];
    T v47 = Ms[47];
    T v48 = Ms[48];
    T v49 = Ms[49];
    T v50 = Ms[50];
    T v51 = Ms[51];
    T v52 = Ms[52];
    T v53 = Ms[53];
    T v54 = Ms[54];
    T v55 = Ms[55];
    T v56 = Ms[56];
    T v57 = Ms[57];
    T v58 = Ms[58];
    T v59 = Ms[59];
    T v60 = Ms[60];
    T v61 = Ms[61];
    T v62 = Ms[62];
    T v63 = Ms[63];
    T v64 = Ms[64];
    T v65 = Ms[65];
    T v66 = Ms[66];
    T v67 = Ms[67];
    T v68 = Ms[68];
    T v69 = Ms[69];
    T v70 = Ms[70];
    T v71 = Ms[71];
    T v72 = Ms[72];
    T v73 = Ms[73];
    T v74 = Ms[74];
    T v75 = Ms[75];
    T v76 = Ms[76];
    T v77 = Ms[77];
    T v78 = Ms[78];
    T v79 = Ms[79];
    T v80 = Ms[80];
    T v81 = Ms[81];
    T v82 = Ms[82];
    T v83 = Ms[83];
    v70 -= v83;
    v81 -= v83;
    v44 -= v55;
    v53 -= v55;
    v65 -= v76;
    v74 -= v76;
    v69 -= v82;
    v80 -= v82;
    v25 -= v34;
    v32 -= v34;
    v40 -= v49;
    v47 -= v49;
    v43 -= v54;
    v52 -= v54;
    v61 -= v70;
    v68 -= v70;
    v64 -= v75;
    v73 -= v75;
    v68 -= v81;
    v79 -= v81;
    v12 -= v19;
    v17 -= v19;
    v22 -= v29;
    v27 -= v29;
    v24 -= v33;
    v31 -= v33;
    v37 -= v44;
    v42 -= v44;
    v39 -= v48;
    v46 -= v48;
    v42 -= v53;
    v51 -= v53;
    v58 -= v65;
    v63 -= v65;
    v60 -= v69;
    v67 -= v69;
    v63 -= v74;
    v72 -= v74;
    v67 -= v80;
    v78 -= v80;
    v4 -= v9;
    v7 -= v9;
    v10 -= v15;
    v13 -= v15;
    v11 -= v18;
    v16 -= v18;
    v20 -= v25;
    v23 -= v25;
    v21 -= v28;
    v26 -= v28;
    v23 -= v32;
    v30 -= v32;
    v35 -= v40;
    v38 -= v40;
    v36 -= v43;
    v41 -= v43;
    v38 -= v47;
    v45 -= v47;
    v41 -= v52;
    v50 -= v52;
    v56 -= v61;
    v59 -= v61;
    v57 -= v64;
    v62 -= v64;
    v59 -= v68;
    v66 -= v68;
    v62 -= v73;
    v71 -= v73;
    v66 -= v79;
    v77 -= v79;
    Mr[0] = v0;
    Mr[1] = v1;
    Mr[2] = v2;
    Mr[3] = v3;
    Mr[4] = v4;
    Mr[5] = v5;
    Mr[6] = v6;
    Mr[7] = v7;
    Mr[8] = v8;
    Mr[9] = v10;
    Mr[10] = v11;
    Mr[11] = v12;
    Mr[12] = v13;
    Mr[13] = v14;
    Mr[14] = v16;
    Mr[15] = v17;
    Mr[16] = v20;
    Mr[17] = v21;
    Mr[18] = v22;
    Mr[19] = v23;
    Mr[20] = v24;
    Mr[21] = v26;
    Mr[22] = v27;
    Mr[23] = v30;
    Mr[24] = v31;
    Mr[25] = v35;
    Mr[26] = v36;
    Mr[27] = v37;
    Mr[28] = v38;
    Mr[29] = v39;
    Mr[30] = v41;
    Mr[31] = v42;
    Mr[32] = v45;
    Mr[33] = v46;
    Mr[34] = v50;
    Mr[35] = v51;
    Mr[36] = v56;
    Mr[37] = v57;
    Mr[38] = v58;
    Mr[39] = v59;
    Mr[40] = v60;
    Mr[41] = v62;
    Mr[42] = v63;
    Mr[43] = v66;
    Mr[44] = v67;
    Mr[45] = v71;
    Mr[46] = v72;
    Mr[47] = v77;
    Mr[48] = v78;
}

template <class T> __device__ __forceinline__ void m2l_complete_locals_h_6(const T *__restrict__ Lr, T *__restrict__ L)
{
    const T v0 = Lr[0];
    L[0] = v0;
    const T v1 = Lr[1];
    L[1] = v1;
    const T v2 = Lr[2];
    L[2] = v2;
    const T v3 = Lr[3];
    L[3] = v3;
    const T v4 = Lr[4];
    L[4] = v4;
    const T v5 = Lr[5];
    L[5] = v5;
    const T v6 = Lr[6];
    L[6] = v6;
    const T v7 = Lr[7];
    L[7] = v7;
    const T v8 = Lr[8];
    L[8] = v8;
    const T v9 = -v4 - v7;
    L[9] = v9;
    const T v10 = Lr[9];
    L[10] = v10;
    const T v11 = Lr[10];
    L[11] = v11;
    const T v12 = Lr[11];
    L[12] = v12;
    const T v13 = Lr[12];
    L[13] = v13;
    const T v14 = Lr[13];
    L[14] = v14;
    const T v15 = -v10 - v13;
    L[15] = v15;
    const T v16 = Lr[14];
    L[16] = v16;
    const T v17 = Lr[15];
    L[17] = v17;
    const T v18 = -v11 - v16;
    L[18] = v18;
    const T v19 = -v12 - v17;
    L[19] = v19;
    const T v20 = Lr[16];
    L[20] = v20;
    const T v21 = Lr[17];
    L[21] = v21;
    const T v22 = Lr[18];
    L[22] = v22;
    const T v23 = Lr[19];
    L[23] = v23;
    const T v24 = Lr[20];
    L[24] = v24;
    const T v25 = -v20 - v23;
    L[25] = v25;
    const T v26 = Lr[21];
    L[26] = v26;
    const T v27 = Lr[22];
    L[27] = v27;
    const T v28 = -v21 - v26;
    L[28] = v28;
    const T v29 = -v22 - v27;
    L[29] = v29;
    const T v30 = Lr[23];
    L[30] = v30;
    const T v31 = Lr[24];
    L[31] = v31;
    const T v32 = -v23 - v30;
    L[32] = v32;
    const T v33 = -v24 - v31;
    L[33] = v33;
    const T v34 = -v25 - v32;
    L[34] = v34;
    const T v35 = Lr[25];
    L[35] = v35;
    const T v36 = Lr[26];
    L[36] = v36;
    const T v37 = Lr[27];
    L[37] = v37;
    const T v38 = Lr[28];
    L[38] = v38;
    const T v39 = Lr[29];
    L[39] = v39;
    const T v40 = -v35 - v38;
    L[40] = v40;
    const T v41 = Lr[30];
    L[41] = v41;
    const T v42 = Lr[31];
    L[42] = v42;
    const T v43 = -v36 - v41;
    L[43] = v43;
    const T v44 = -v37 - v42;
    L[44] = v44;
    const T v45 = Lr[32];
    L[45] = v45;
    const T v46 = Lr[33];
    L[46] = v46;
    const T v47 = -v38 - v45;
    L[47] = v47;
    const T v48 = -v39 - v46;
    L[48] = v48;
    const T v49 = -v40 - v47;
    L[49] = v49;
    const T v50 = Lr[34];
    L[50] = v50;
    const T v51 = Lr[35];
    L[51] = v51;
    const T v52 = -v41 - v50;
    L[52] = v52;
    const T v53 = -v42 - v51;
    L[53] = v53;
    const T v54 = -v43 - v52;
    L[54] = v54;
    const T v55 = -v44 - v53;
    L[55] = v55;
    const T v56 = Lr[36];
    L[56] = v56;
    const T v57 = Lr[37];
    L[57] = v57;
    const T v58 = Lr[38];
    L[58] = v58;
    const T v59 = Lr[39];
    L[59] = v59;
    const T v60 = Lr[40];
    L[60] = v60;
    const T v61 = -v56 - v59;
    L[61] = v61;
    const T v62 = Lr[41];
    L[62] = v62;
    const T v63 = Lr[42];
    L[63] = v63;
    const T v64 = -v57 - v62;
    L[64] = v64;
    const T v65 = -v58 - v63;
    L[65] = v65;
    const T v66 = Lr[43];
    L[66] = v66;
    const T v67 = Lr[44];
    L[67] = v67;
    const T v68 = -v59 - v66;
    L[68] = v68;
    const T v69 = -v60 - v67;
    L[69] = v69;
    const T v70 = -v61 - v68;
    L[70] = v70;
    const T v71 = Lr[45];
    L[71] = v71;
    const T v72 = Lr[46];
    L[72] = v72;
    const T v73 = -v62 - v71;
    L[73] = v73;
    const T v74 = -v63 - v72;
    L[74] = v74;
    const T v75 = -v64 - v73;
    L[75] = v75;
    const T v76 = -v65 - v74;
    L[76] = v76;
    const T v77 = Lr[47];
    L[77] = v77;
    const T v78 = Lr[48];
    L[78] = v78;
    const T v79 = -v66 - v77;
    L[79] = v79;
    const T v80 = -v67 - v78;
    L[80] = v80;
    const T v81 = -v68 - v79;
    L[81] = v81;
    const T v82 = -v69 - v80;
    L[82] = v82;
    const T v83 = -v70 - v81;
    L[83] = v83;
}

template <int P> struct M2LGenH;
template <> struct M2LGenH<1> {
    static constexpr int NC = 4;
    static constexpr int ND = 4;
    template <class T> static __device__ __forceinline__ void dtensor(T dx, T dy, T dz, T (&D)[4]) { m2l_dtensor_h_1(dx, dy, dz, D); }
    template <class T> static __device__ __forceinline__ void side_a(const T (&D)[4], const T *Mr, T rho, T (&L)[4]) { m2l_side_a_h_1(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b(const T (&D)[4], const T *Mr, T (&L)[4]) { m2l_side_b_h_1(D, Mr, L); }
    template <class T> static __device__ __forceinline__ void side_a_forces(const T (&D)[4], const T *Mr, T rho, T (&L)[4]) { m2l_side_a_h_forces_1(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b_forces(const T (&D)[4], const T *Mr, T (&L)[4]) { m2l_side_b_h_forces_1(D, Mr, L); }
    template <class T> static __device__ __forceinline__ void acc(const T (&D)[4], const T *Mr, T rho, T (&L)[4]) { m2l_acc_h_1(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void acc_forces(const T (&D)[4], const T *Mr, T rho, T (&L)[4]) { m2l_acc_h_forces_1(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void reduce_moments(const T *Ms, T *Mr) { m2l_reduce_moments_h_1(Ms, Mr); }
    template <class T> static __device__ __forceinline__ void complete_locals(const T *Lr, T *L) { m2l_complete_locals_h_1(Lr, L); }
};
template <> struct M2LGenH<2> {
    static constexpr int NC = 9;
    static constexpr int ND = 10;
    template <class T> static __device__ __forceinline__ void dtensor(T dx, T dy, T dz, T (&D)[10]) { m2l_dtensor_h_2(dx, dy, dz, D); }
    template <class T> static __device__ __forceinline__ void side_a(const T (&D)[10], const T *Mr, T rho, T (&L)[9]) { m2l_side_a_h_2(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b(const T (&D)[10], const T *Mr, T (&L)[9]) { m2l_side_b_h_2(D, Mr, L); }
    template <class T> static __device__ __forceinline__ void side_a_forces(const T (&D)[10], const T *Mr, T rho, T (&L)[9]) { m2l_side_a_h_forces_2(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b_forces(const T (&D)[10], const T *Mr, T (&L)[9]) { m2l_side_b_h_forces_2(D, Mr, L); }
    template <class T> static __device__ __forceinline__ void acc(const T (&D)[10], const T *Mr, T rho, T (&L)[9]) { m2l_acc_h_2(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void acc_forces(const T (&D)[10], const T *Mr, T rho, T (&L)[9]) { m2l_acc_h_forces_2(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void reduce_moments(const T *Ms, T *Mr) { m2l_reduce_moments_h_2(Ms, Mr); }
    template <class T> static __device__ __forceinline__ void complete_locals(const T *Lr, T *L) { m2l_complete_locals_h_2(Lr, L); }
};
template <> struct M2LGenH<3> {
    static constexpr int NC = 16;
    static constexpr int ND = 19;
    template <class T> static __device__ __forceinline__ void dtensor(T dx, T dy, T dz, T (&D)[19]) { m2l_dtensor_h_3(dx, dy, dz, D); }
    template <class T> static __device__ __forceinline__ void side_a(const T (&D)[19], const T *Mr, T rho, T (&L)[16]) { m2l_side_a_h_3(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b(const T (&D)[19], const T *Mr, T (&L)[16]) { m2l_side_b_h_3(D, Mr, L); }
    template <class T> static __device__ __forceinline__ void side_a_forces(const T (&D)[19], const T *Mr, T rho, T (&L)[16]) { m2l_side_a_h_forces_3(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b_forces(const T (&D)[19], const T *Mr, T (&L)[16]) { m2l_side_b_h_forces_3(D, Mr, L); }
    template <class T> static __device__ __forceinline__ void acc(const T (&D)[19], const T *Mr, T rho, T (&L)[16]) { m2l_acc_h_3(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void acc_forces(const T (&D)[19], const T *Mr, T rho, T (&L)[16]) { m2l_acc_h_forces_3(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void reduce_moments(const T *Ms, T *Mr) { m2l_reduce_moments_h_3(Ms, Mr); }
    template <class T> static __device__ __forceinline__ void complete_locals(const T *Lr, T *L) { m2l_complete_locals_h_3(Lr, L); }
};
template <> struct M2LGenH<4> {
    static constexpr int NC = 25;
    static constexpr int ND = 31;
    template <class T> static __device__ __forceinline__ void dtensor(T dx, T dy, T dz, T (&D)[31]) { m2l_dtensor_h_4(dx, dy, dz, D); }
    template <class T> static __device__ __forceinline__ void side_a(const T (&D)[31], const T *Mr, T rho, T (&L)[25]) { m2l_side_a_h_4(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b(const T (&D)[31], const T *Mr, T (&L)[25]) { m2l_side_b_h_4(D, Mr, L); }
    template <class T> static __device__ __forceinline__ void side_a_forces(const T (&D)[31], const T *Mr, T rho, T (&L)[25]) { m2l_side_a_h_forces_4(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b_forces(const T (&D)[31], const T *Mr, T (&L)[25]) { m2l_side_b_h_forces_4(D, Mr, L); }
    template <class T> static __device__ __forceinline__ void acc(const T (&D)[31], const T *Mr, T rho, T (&L)[25]) { m2l_acc_h_4(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void acc_forces(const T (&D)[31], const T *Mr, T rho, T (&L)[25]) { m2l_acc_h_forces_4(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void reduce_moments(const T *Ms, T *Mr) { m2l_reduce_moments_h_4(Ms, Mr); }
    template <class T> static __device__ __forceinline__ void complete_locals(const T *Lr, T *L) { m2l_complete_locals_h_4(Lr, L); }
};
template <> struct M2LGenH<5> {
    static constexpr int NC = 36;
    static constexpr int ND = 46;
    template <class T> static __device__ __forceinline__ void dtensor(T dx, T dy, T dz, T (&D)[46]) { m2l_dtensor_h_5(dx, dy, dz, D); }
    template <class T> static __device__ __forceinline__ void side_a(const T (&D)[46], const T *Mr, T rho, T (&L)[36]) { m2l_side_a_h_5(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b(const T (&D)[46], const T *Mr, T (&L)[36]) { m2l_side_b_h_5(D, Mr, L); }
    template <class T> static __device__ __forceinline__ void side_a_forces(const T (&D)[46], const T *Mr, T rho, T (&L)[36]) { m2l_side_a_h_forces_5(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b_forces(const T (&D)[46], const T *Mr, T (&L)[36]) { m2l_side_b_h_forces_5(D, Mr, L); }
    template <class T> static __device__ __forceinline__ void acc(const T (&D)[46], const T *Mr, T rho, T (&L)[36]) { m2l_acc_h_5(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void acc_forces(const T (&D)[46], const T *Mr, T rho, T (&L)[36]) { m2l_acc_h_forces_5(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void reduce_moments(const T *Ms, T *Mr) { m2l_reduce_moments_h_5(Ms, Mr); }
    template <class T> static __device__ __forceinline__ void complete_locals(const T *Lr, T *L) { m2l_complete_locals_h_5(Lr, L); }
};
template <> struct M2LGenH<6> {
    static constexpr int NC = 49;
    static constexpr int ND = 64;
    template <class T> static __device__ __forceinline__ void dtensor(T dx, T dy, T dz, T (&D)[64]) { m2l_dtensor_h_6(dx, dy, dz, D); }
    template <class T> static __device__ __forceinline__ void side_a(const T (&D)[64], const T *Mr, T rho, T (&L)[49]) { m2l_side_a_h_6(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b(const T (&D)[64], const T *Mr, T (&L)[49]) { m2l_side_b_h_6(D, Mr, L); }
    template <class T> static __device__ __forceinline__ void side_a_forces(const T (&D)[64], const T *Mr, T rho, T (&L)[49]) { m2l_side_a_h_forces_6(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void side_b_forces(const T (&D)[64], const T *Mr, T (&L)[49]) { m2l_side_b_h_forces_6(D, Mr, L); }
    template <class T> static __device__ __forceinline__ void acc(const T (&D)[64], const T *Mr, T rho, T (&L)[49]) { m2l_acc_h_6(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void acc_forces(const T (&D)[64], const T *Mr, T rho, T (&L)[49]) { m2l_acc_h_forces_6(D, Mr, rho, L); }
    template <class T> static __device__ __forceinline__ void reduce_moments(const T *Ms, T *Mr) { m2l_reduce_moments_h_6(Ms, Mr); }
    template <class T> static __device__ __forceinline__ void complete_locals(const T *Lr, T *L) { m2l_complete_locals_h_6(Lr, L); }
};
