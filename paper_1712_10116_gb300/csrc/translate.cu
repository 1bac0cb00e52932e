// translate.cu -- M2M and L2L at fixed order P <= 6 (Sec. 2.1 of Zhu 2017), and the moments as the harmonic M2L
// reads them.
//
// A child's centre lies at (+-s/4)^3 from its parent's, so a translation is three one-dimensional shifts by
// a = +-1/4, one axis after another, in place: with moments divided by n! and locals as derivatives both read
//   v^n <- sum_d v^(n -+ d e) a^d / d!,
// 126 multiply-adds an axis at p = 6, 378 in all against 840 for the three axes at once, on one thread's registers
// with every index a compile-time constant.  M2M takes eight lanes per parent, one per child, and adds the
// children with a reduce-scatter; L2L takes a thread per cell and class.  Small levels are bound by the latency
// of this chain, large ones by the rows they read and write.  (translate_gen.cuh is written by gen_translate.py.)
// Before (a block per parent and a warp per cell reading term lists from memory; passes of their own to scale and fold
// the moments and to complete the locals): 54,321-particle kick pair at p = 5 1045 us, now 938; the disk galaxy's at
// p = 6 37.2 ms, now 36.4; its HOLD step 847 ms, now 793.
#include "m2l_gen.cuh"
#include "tg_common.cuh"
#include "translate_gen.cuh"

namespace tg {

template <class T>
struct alignas(16) Vec16 {
    static constexpr int N = 16 / sizeof(T);
    T v[N];
};

// the first NC entries of a row (16-byte aligned, padded to a multiple of 16 bytes)
template <int NC, class T>
__device__ __forceinline__ void load_row(const T *row, T (&v)[NC])
{
    constexpr int W = Vec16<T>::N;
#pragma unroll
    for (int k = 0; k < NC; k += W) {
        const Vec16<T> q = *reinterpret_cast<const Vec16<T> *>(row + k);
#pragma unroll
        for (int e = 0; e < W; ++e)
            if (k + e < NC) v[k + e] = q.v[e];
    }
}

// a^d / d! for a = +-1/4
template <int P, class T>
__device__ __forceinline__ void shift_coef(bool neg, T (&c)[P + 1])
{
    T v = T(1);
#pragma unroll
    for (int d = 0; d <= P; ++d) {
        c[d] = v;
        v *= (neg ? T(-0.25) : T(0.25)) / T(d + 1);
    }
}

// ------------------------------------------------------------------ M2M
// M~_P^n = sum_children sum_{k <= n} C(n,k) 2^-(2|n-k| + |k|) (+-1)^(n-k) M~_c^k for the parents of one level.  The
// monopole and dipole are summed in float64 (M01), every order also in T.  The fast class is left out when the
// evaluation has no classes; with classes the slow particles of the children are counted too (nslow).
template <int P, class T>
__global__ void __launch_bounds__(128) m2m_fixed(TreeView t, int lb, int le, int masked, int ncp, T *M, double *M01,
                                                 int32_t *nslow, const DevEval *de, int lvl)
{
    if (de) {   // level range and classes on the device (batched path); levels past the tree are empty
        if (lvl + 1 >= de->nlev) return;
        lb = de->level_begin[lvl];
        le = de->level_begin[lvl + 1];
        masked = de->masked;
    }
    constexpr int NC = (P + 1) * (P + 2) * (P + 3) / 6, RL = (NC + 31) / 32 * 4, NP = 8 * RL, W = Vec16<T>::N;
    const int lane = threadIdx.x & 31, q = lane & 7;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = (gridDim.x * blockDim.x) >> 5;
    const int ngroup = (le - lb + 3) / 4;
    // a warp takes four parents and one class
    for (int w = warp; w < ngroup * (masked ? 2 : 1); w += nwarps) {
        const int cls = w >= ngroup ? 1 : 0, c = lb + 4 * (w - cls * ngroup) + (lane >> 3);
        const int nch = c < le ? t.nchild[c] : 0;
        const bool child = q < nch;
        const int ch = child ? t.child_first[c] + q : 0;
        const bool sx = child && !(t.cx[ch] & 1u), sy = child && !(t.cy[ch] & 1u), sz = child && !(t.cz[ch] & 1u);
        double lo[4] = {0.0, 0.0, 0.0, 0.0};
        T v[NP];
#pragma unroll
        for (int k = 0; k < NP; ++k) v[k] = T(0);
        if (child) {
            const double *Mc = M01 + ((size_t)ch * 2 + cls) * 4;
            lo[0] = Mc[0];
            lo[1] = 0.5 * Mc[1] + (sx ? -0.25 : 0.25) * lo[0];
            lo[2] = 0.5 * Mc[2] + (sy ? -0.25 : 0.25) * lo[0];
            lo[3] = 0.5 * Mc[3] + (sz ? -0.25 : 0.25) * lo[0];
            T(&m)[NC] = reinterpret_cast<T(&)[NC]>(v);
            load_row<NC>(M + ((size_t)ch * 2 + cls) * ncp, m);
            XlGen<P>::moments_in(m);
            T ax[P + 1], ay[P + 1], az[P + 1];
            shift_coef<P>(sx, ax);
            shift_coef<P>(sy, ay);
            shift_coef<P>(sz, az);
            XlGen<P>::shift_moments(m, ax, ay, az);
            XlGen<P>::moments_out(m);
        }
#pragma unroll
        for (int o = 1; o < 8; o <<= 1)
#pragma unroll
            for (int k = 0; k < 4; ++k) lo[k] += __shfl_xor_sync(0xffffffffu, lo[k], o);
        // the children's sum, lane q keeping entries RL q .. RL q + RL - 1
#pragma unroll
        for (int h = 4; h >= 1; h >>= 1) {
            const bool hi = (q & h) != 0;
#pragma unroll
            for (int k = 0; k < NP / 2; ++k)
                if (k < h * RL) {
                    const T send = hi ? v[k] : v[k + h * RL], keep = hi ? v[k + h * RL] : v[k];
                    v[k] = keep + __shfl_xor_sync(0xffffffffu, send, h);
                }
        }
        int slow = nslow && child ? nslow[ch] : 0;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) slow += __shfl_xor_sync(0xffffffffu, slow, o);
        if (nch == 0) continue;
        if (nslow && cls == 0 && q == 0) nslow[c] = slow;
        T *row = M + ((size_t)c * 2 + cls) * ncp;
        if (q < 4) {
            const double mine = q == 0 ? lo[0] : (q == 1 ? lo[1] : (q == 2 ? lo[2] : lo[3]));
            M01[((size_t)c * 2 + cls) * 4 + q] = mine;
            row[q] = (T)mine;
        }
#pragma unroll
        for (int k = 0; k < RL; k += W)
            if (RL * q + k >= 4 && RL * q + k < ncp) {
                Vec16<T> w;
#pragma unroll
                for (int e = 0; e < W; ++e) w.v[e] = v[k + e];
                *reinterpret_cast<Vec16<T> *>(row + RL * q + k) = w;
            }
    }
}

// ------------------------------------------------------------------ L2L
// L~_c^n += 2^-(|n| + 1) sum_d L~_P^(n+d) (+-1)^d 4^-|d| / d! for the cells of one level.
// HARM: M2L left the cells' sums in Lr (the coefficients n_z <= 1 of a harmonic expansion); a shifted harmonic
// expansion is harmonic too, so the two are added on those coefficients and the rest follows from
// L^(n+2e_z) = -L^(n+2e_x) - L^(n+2e_y): no pass of its own completes the locals, and L is only written.
// Otherwise L holds the cells' M2L sums.  The root (no parent, no M2L) goes with level 1.
template <int P, class T, bool HARM>
__global__ void __launch_bounds__(128) l2l_fixed(TreeView t, int lb, int le, int ncls, int ncp, T *L,
                                                 const T *__restrict__ Lr, int ncpr, const DevEval *de, int lvl)
{
    if (de) {
        if (lvl > 1 && lvl >= de->nlev) return;
        lb = lvl > 1 ? de->level_begin[lvl] : 0;
        le = de->level_begin[min(lvl, de->nlev - 1) + 1];
        ncls = de->masked ? 2 : 1;
    }
    constexpr int NC = (P + 1) * (P + 2) * (P + 3) / 6, W = Vec16<T>::N;
    const int cnt = le - lb;
    for (int w = blockIdx.x * blockDim.x + threadIdx.x; w < cnt * ncls; w += gridDim.x * blockDim.x) {
        const int cls = w >= cnt ? 1 : 0, c = lb + w - cls * cnt;
        const int par = t.parent[c];
        T v[NC];
        if (par > 0) {   // the root's own local expansion is zero
            load_row<NC>(L + ((size_t)par * 2 + cls) * ncp, v);
            T ax[P + 1], ay[P + 1], az[P + 1];
            shift_coef<P>(!(t.cx[c] & 1u), ax);
            shift_coef<P>(!(t.cy[c] & 1u), ay);
            shift_coef<P>(!(t.cz[c] & 1u), az);
            XlGen<P>::shift_locals(v, ax, ay, az);
            XlGen<P>::locals_out(v);
        } else {
#pragma unroll
            for (int k = 0; k < NC; ++k) v[k] = T(0);
        }
        T *row = L + ((size_t)c * 2 + cls) * ncp;
        if (HARM) {
            T h[XlGen<P>::NH];
            load_row<XlGen<P>::NH>(Lr + ((size_t)c * 2 + cls) * ncpr, h);
            XlGen<P>::locals_harmonic(v, h);
        } else {
            T own[NC];
            load_row<NC>(row, own);
#pragma unroll
            for (int k = 0; k < NC; ++k) v[k] += own[k];
        }
#pragma unroll
        for (int k = 0; k < NC; k += W) {
            Vec16<T> o;
#pragma unroll
            for (int e = 0; e < W; ++e) o.v[e] = k + e < NC ? v[k + e] : T(0);
            *reinterpret_cast<Vec16<T> *>(row + k) = o;
        }
    }
}

// ------------------------------------------------------------------ moments for the harmonic M2L
// Per cell and class: (M~_S + M~_F)/j! or M~_S/j!, folded onto j_z <= 1 (the vector that ends the set is filled up with
// zeros, a row's further padding is left as it is: nothing reads it); the monopole and dipole from the
// float64 sums.  One pass from the moments to what M2L reads.
template <int P, class T>
__global__ void __launch_bounds__(128) m2l_moments_h(int ncell, int masked, const T *__restrict__ M,
                                                     const double *__restrict__ M01, int ncp, T *__restrict__ Mr, int ncpr,
                                                     const DevEval *de)
{
    if (de) {
        ncell = de->ncell;
        masked = de->masked;
    }
    constexpr int NC = (P + 1) * (P + 2) * (P + 3) / 6, NH = (P + 1) * (P + 1), W = Vec16<T>::N;
    const int64_t total = (int64_t)ncell * (masked ? 2 : 1);
    for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < total; w += (int64_t)gridDim.x * blockDim.x) {
        const int cls = w >= ncell ? 1 : 0;
        const int64_t c = w - (int64_t)cls * ncell;
        T v[NC], r[NH + W];
        load_row<NC>(M + c * 2 * ncp, v);
        if (masked && cls == 0) {
            T f[NC];
            load_row<NC>(M + (c * 2 + 1) * ncp, f);
#pragma unroll
            for (int k = 4; k < NC; ++k) v[k] += f[k];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const double s = M01[c * 8 + k];
            v[k] = (T)(masked && cls == 0 ? s + M01[c * 8 + 4 + k] : s);
        }
        XlGen<P>::moments_scale(v);
        M2LGenH<P>::reduce_moments(v, r);
#pragma unroll
        for (int k = NH; k < NH + W; ++k) r[k] = T(0);
        T *row = Mr + (c * 2 + cls) * ncpr;
#pragma unroll
        for (int k = 0; k < NH; k += W) {
            Vec16<T> o;
#pragma unroll
            for (int e = 0; e < W; ++e) o.v[e] = r[k + e];
            *reinterpret_cast<Vec16<T> *>(row + k) = o;
        }
    }
}

#define TG_BY_ORDER(CALL)        \
    switch (p) {                 \
    case 1: CALL(1); break;      \
    case 2: CALL(2); break;      \
    case 3: CALL(3); break;      \
    case 4: CALL(4); break;      \
    case 5: CALL(5); break;      \
    default: CALL(6);            \
    }

template <class T>
void launch_m2m_fixed(tg_ctx *c, const TreeView &t, int lb, int le, int p, int ncp, bool masked, T *M, double *M01,
                      int32_t *nslow, const DevEval *de, int lvl)
{
    const int grid = de ? c->num_sms * 4 : grid_for((int64_t)(le - lb) * 8 * (masked ? 2 : 1), 128, c->num_sms * 8);
    ProfScope ps_(c, TG_K_UP);
#define TG_CALL(PP) m2m_fixed<PP, T><<<grid, 128, 0, c->stream>>>(t, lb, le, masked, ncp, M, M01, nslow, de, lvl)
    TG_BY_ORDER(TG_CALL)
#undef TG_CALL
}

template <class T>
void launch_l2l_fixed(tg_ctx *c, const TreeView &t, int lb, int le, int p, int ncp, int ncls, T *L, const T *Lr, int ncpr,
                      const DevEval *de, int lvl)
{
    const int grid = de ? c->num_sms * 4 : grid_for((int64_t)(le - lb) * ncls, 128, c->num_sms * 8);
    ProfScope ps_(c, TG_K_DOWN);
#define TG_CALL(PP)                                                                                            \
    if (Lr) l2l_fixed<PP, T, true><<<grid, 128, 0, c->stream>>>(t, lb, le, ncls, ncp, L, Lr, ncpr, de, lvl);     \
    else l2l_fixed<PP, T, false><<<grid, 128, 0, c->stream>>>(t, lb, le, ncls, ncp, L, nullptr, 0, de, lvl)
    TG_BY_ORDER(TG_CALL)
#undef TG_CALL
}

template <class T>
void launch_m2l_moments(tg_ctx *c, int ncell, int p, int ncp, bool masked, const T *M, const double *M01, T *Mr, int ncpr,
                        const DevEval *de)
{
    const int grid = grid_for((int64_t)ncell * 2, 128, c->num_sms * 16);
    ProfScope ps_(c, TG_K_UP);
#define TG_CALL(PP) m2l_moments_h<PP, T><<<grid, 128, 0, c->stream>>>(ncell, masked, M, M01, ncp, Mr, ncpr, de)
    TG_BY_ORDER(TG_CALL)
#undef TG_CALL
}

#define TG_INST(T)                                                                                                      \
    template void launch_m2m_fixed<T>(tg_ctx *, const TreeView &, int, int, int, int, bool, T *, double *, int32_t *, const DevEval *, int); \
    template void launch_l2l_fixed<T>(tg_ctx *, const TreeView &, int, int, int, int, int, T *, const T *, int,          \
                                      const DevEval *, int);                                                            \
    template void launch_m2l_moments<T>(tg_ctx *, int, int, int, bool, const T *, const double *, T *, int, const DevEval *);
TG_INST(float)
TG_INST(double)
#undef TG_INST

}  // namespace tg
