// p2p_tile.cuh -- float32 P2P of the self pair (A, A) of a leaf (Sec. 2.1, Eq. 2; the distinct leaf pairs are
// p2p_owner.cuh's).  For every particle pair the kernel value is computed once and applied with opposite signs to both
// particles (a_i += m_j g d, a_j -= m_i g d).  Positions are relative to the leaf's centre.  F-F pairs are skipped when
// classes are given (kickS2F feels slow masses only): the rows are the slow particles, which come first.
#pragma once
#include "p2p_pair.cuh"
#include "tg_common.cuh"

namespace tg {

// float32 pair value: Newton by default, Wendland correction inside eps (rare, predicated).
template <int KERNEL>
__device__ __forceinline__ void pair_kernel_f32(float r2, float eps, float eps2, float inv_eps, float inv_eps3, float &g,
                                                float &phi)
{
    if (KERNEL == TG_KERNEL_PLUMMER) {
        const float si = tg_rsqrt<float>(r2 + eps2);
        phi = -si;
        g = si * si * si;
        return;
    }
    const float ri = rsqrtf(r2);
    phi = -ri;
    g = ri * ri * ri;
    if (r2 < eps2) pair_kernel<float, TG_KERNEL_WENDLAND_C2>(r2, eps, eps2, inv_eps, inv_eps3, g, phi);
}

// Rows = the ns slow particles of A, ROWS per lane (row i0 + lane + 32 r), chunks of 32*ROWS; columns = its na
// particles, staged once in the warp's shared-memory slice and read in batches of 8; a pair counts when its
// column index is above its row index, i.e. each slow-slow and slow-fast pair once.  A lane keeps its rows' sums in registers and its 8 x 4
// column partials.  Lane l visits the 8 columns of a batch in the order c ^ ((l >> 2) & 7), so its
// partial for logical entry e sits in register e ^ (l & 28); the first three stages of the warp
// reduce-scatter (partners l ^ 16, l ^ 8, l ^ 4) then need no selects, and lane l ends with column
// l/4, component l%4, which it adds to global memory.
template <int KERNEL, int ROWS>
__device__ __noinline__ void p2p_self_f32(const float4 *__restrict__ pf, int fa, int ns, int na, float eps, double *acc4,
                                          int n, int lane, float4 *sq)
{
    const float eps2 = eps * eps, inv_eps = 1.0f / eps, inv_eps3 = inv_eps * inv_eps * inv_eps;
    const int cperm = (lane >> 2) & 7;
    for (int jc = 0; jc < na; jc += kMaxNcrit) {
        const int nbc = min(kMaxNcrit, na - jc);
        __syncwarp();
        for (int j = lane; j < nbc; j += 32) sq[j] = pf[fa + jc + j];
        __syncwarp();
        for (int i0 = 0; i0 < ns; i0 += 32 * ROWS) {
            float4 p[ROWS];
            int ir[ROWS];
            float ra[ROWS][4];
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                ir[r] = i0 + lane + 32 * r;
                p[r] = ir[r] < ns ? pf[fa + ir[r]] : make_float4(1e8f, 1e8f, 1e8f, 0.f);   // far away, massless
                ra[r][0] = ra[r][1] = ra[r][2] = ra[r][3] = 0.f;
            }
            for (int j0 = 0; j0 < nbc; j0 += 8) {
                float col[32];
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const int j = j0 + (c ^ cperm);
                    float cx = 0.f, cy = 0.f, cz = 0.f, cp = 0.f;
                    if (j < nbc) {
                        const float4 q = sq[j];
#pragma unroll
                        for (int r = 0; r < ROWS; ++r) {
                            const float dx = q.x - p[r].x, dy = q.y - p[r].y, dz = q.z - p[r].z;
                            float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                            const bool use = jc + j > ir[r];
                            r2 = use ? r2 : 1.0f;
                            float gk, ph;
                            pair_kernel_f32<KERNEL>(r2, eps, eps2, inv_eps, inv_eps3, gk, ph);
                            gk = use ? gk : 0.f;
                            ph = use ? ph : 0.f;
                            const float mq = q.w * gk, mp = p[r].w * gk;
                            ra[r][0] = fmaf(mq, dx, ra[r][0]);
                            ra[r][1] = fmaf(mq, dy, ra[r][1]);
                            ra[r][2] = fmaf(mq, dz, ra[r][2]);
                            ra[r][3] = fmaf(q.w, ph, ra[r][3]);
                            cx = fmaf(-mp, dx, cx);
                            cy = fmaf(-mp, dy, cy);
                            cz = fmaf(-mp, dz, cz);
                            cp = fmaf(p[r].w, ph, cp);
                        }
                    }
                    col[4 * c + 0] = cx;
                    col[4 * c + 1] = cy;
                    col[4 * c + 2] = cz;
                    col[4 * c + 3] = cp;
                }
                // reduce-scatter: column bits (partners l^16, l^8, l^4) without selects ...
#pragma unroll
                for (int h = 16; h >= 4; h >>= 1)
#pragma unroll
                    for (int q = 0; q < h; ++q) col[q] += __shfl_xor_sync(0xffffffffu, col[q + h], h);
                // ... component bits (l^2, l^1) with selects
#pragma unroll
                for (int h = 2; h >= 1; h >>= 1) {
                    const bool hi = (lane & h) != 0;
#pragma unroll
                    for (int q = 0; q < h; ++q) {
                        const float send = hi ? col[q] : col[q + h];
                        const float keep = hi ? col[q + h] : col[q];
                        col[q] = keep + __shfl_xor_sync(0xffffffffu, send, h);
                    }
                }
                const int cj = lane >> 2, comp = lane & 3;
                if (j0 + cj < nbc) atomicAdd(&acc4[(size_t)comp * n + fa + jc + j0 + cj], f2d_exact(col[0]));
            }
#pragma unroll
            for (int r = 0; r < ROWS; ++r)
                if (ir[r] < ns)
#pragma unroll
                    for (int comp = 0; comp < 4; ++comp)
                        atomicAdd(&acc4[(size_t)comp * n + fa + ir[r]], f2d_exact(ra[r][comp]));
        }
    }
}

}  // namespace tg
