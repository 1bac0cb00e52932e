// p2p_owner_f64.cuh -- mutual P2P in float64, by owner leaf (the work units of p2p_owner.cuh).
//
// GB300's float64 pipe takes under 2 lanes per clock and SM (5.27e11 operations/s from a loop of independent
// operations on registers, 1.7 per clock and SM), so the kernel is bound by its float64 operations: what counts is
// the operations per pair and that every lane of an issued warp holds a pair; loads, shuffles and integer work are
// nearly free beside them.  A warp holds an owner's particles as columns in shared
// memory and packs its partners' particles densely into rows, 64 at a time (less for the rest of a unit).  A pair
// takes 18 operations (21 with the potential, see pair_f64.cuh).  The columns' reaction sums go through a
// reduce-scatter of four columns at a time, 14 more operations for the 8 pairs of a lane's batch.
// One block per leaf pair, with a full warp sum for every column and row slots padded to 64 per leaf,
// took 66.8 ms for the 4.21e8 pairs of a 100,003-particle sphere's kick pair; this form takes 16.6 ms.  Its 8.3e9
// operations take 15.7 ms at the rate above.
#pragma once
#include "p2p_owner.cuh"
#include "pair_f64.cuh"

namespace tg {

constexpr int kOwn64Warps = 4;   // warps per block
constexpr int kOwn64Cols = kMaxNcrit + 4;

// The partners of one work unit, in slot order.
struct Own64Batch {
    int first[32];    // first particle of the partner
    int nslow[32];    // slow particles of the partner (all of them without classes)
    int inc[2][32];   // inclusive row counts over slots: [0] slow rows, [1] fast rows
};

// The sorted particles as the caller gave them.  Differences of the original coordinates are exact for close pairs;
// coordinates relative to leaf centres would have to be shifted into the owner's frame, a rounding per
// coordinate.  (With that rounding the chaotic 2^14-particle disk left the oracle's trajectory ten times faster.)
struct Bodies {
    const double *x, *y, *z, *m;
    __device__ __forceinline__ dbl4 get(int i) const
    {
        dbl4 v;
        v.x = x[i];
        v.y = y[i];
        v.z = z[i];
        v.w = m[i];
        return v;
    }
};

struct Own64Shared {
    dbl4 q[kOwn64Warps][kOwn64Cols];           // owner's particles (columns), per warp
    double acc[kOwn64Warps][kOwn64Cols][4];    // owner's reaction sums (ax, ay, az, phi), per warp
    Own64Batch b[kOwn64Warps];
};

// Rows i0 .. i0 + 32*ROWS of one phase (0: slow rows, 1: fast rows) against the first ncol staged columns
// (a multiple of 4).  Columns at or past nkeep are massless and their reaction sums are not kept; pairs with
// one, or with a slot that holds no row, are evaluated at r = 1, where the value is finite whatever the softening and
// the coordinates are (the two selects run on the integer pipe).  Lane l visits column
// c ^ ((l >> 3) & 3) of a batch at step c, so that the column stages of the reduce-scatter (partners l^16,
// l^8) need no selects.
//
// S > 1 (ROWS = 1): a rest of at most 32 / S rows.  Lanes l, l^16 (and l^8) share a row and split the columns of
// a batch: each computes the 4 / S columns that it would keep after the first stages of the reduce-scatter, which
// fall away.
template <int KERNEL, int ROWS, int S, bool POT>
__device__ __noinline__ void owner_rows_f64(const Bodies &pf, const Own64Batch *ob, int phase, int i0,
                                            int nrows, const dbl4 *sq, double (*sacc)[4], int ncol, int nkeep,
                                            const PairF64 &k, double *acc4, int n, int lane)
{
    constexpr int NC = POT ? 4 : 3;
    const int *inc = ob->inc[phase];
    dbl4 p[ROWS];
    int gi[ROWS];
    double ra[ROWS][NC];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        const int i = i0 + (lane & (32 / S - 1)) + 32 * r;
        gi[r] = -1;
        p[r].x = p[r].y = p[r].z = p[r].w = 0.0;   // massless
        if (i < nrows) {
            int s = 0;   // slot: the first with inc[s] > i
#pragma unroll
            for (int b = 16; b >= 1; b >>= 1)
                if (inc[s + b - 1] <= i) s += b;
            gi[r] = ob->first[s] + (phase ? ob->nslow[s] : 0) + i - (s ? inc[s - 1] : 0);
            p[r] = pf.get(gi[r]);
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) ra[r][c] = 0.0;
    }
    const int cperm = (lane >> 3) & 3;
    for (int j0 = 0; j0 < ncol; j0 += 4) {
        double col[4 / S][NC];
#pragma unroll
        for (int c = 0; c < 4 / S; ++c) {
            const dbl4 q = sq[j0 + (c ^ cperm)];
            const bool column = j0 + (c ^ cperm) < nkeep;
#pragma unroll
            for (int e = 0; e < NC; ++e) col[c][e] = 0.0;
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                const double dx = q.x - p[r].x, dy = q.y - p[r].y, dz = q.z - p[r].z;
                double g, ri;
                const double s = pair_s2<KERNEL>(dx, dy, dz, k);
                pair_f64<KERNEL, POT>(column && gi[r] >= 0 ? s : 1.0, k, g, ri);
                const double mq = q.w * g, mp = p[r].w * g;
                ra[r][0] = fma(mq, dx, ra[r][0]);
                ra[r][1] = fma(mq, dy, ra[r][1]);
                ra[r][2] = fma(mq, dz, ra[r][2]);
                if (r == 0) {
                    col[c][0] = mp * dx;
                    col[c][1] = mp * dy;
                    col[c][2] = mp * dz;
                } else {
                    col[c][0] = fma(mp, dx, col[c][0]);
                    col[c][1] = fma(mp, dy, col[c][1]);
                    col[c][2] = fma(mp, dz, col[c][2]);
                }
                if (POT) {   // potentials negated here, turned at the flushes
                    ra[r][NC - 1] = fma(q.w, ri, ra[r][NC - 1]);
                    col[c][NC - 1] = fma(p[r].w, ri, col[c][NC - 1]);
                }
            }
        }
#pragma unroll
        for (int h = 2 / S; h >= 1; h >>= 1)
#pragma unroll
            for (int c = 0; c < h; ++c)
#pragma unroll
                for (int e = 0; e < NC; ++e) col[c][e] += __shfl_xor_sync(0xffffffffu, col[c + h][e], 8 * h);
        // the eight lanes of a column: component bits (l^2, l^1) with selects, then l^4; lane l ends with
        // column l/8, component l%4
        const bool hi2 = (lane & 2) != 0, hi1 = (lane & 1) != 0;
        const double c3 = POT ? col[0][NC - 1] : 0.0;
        const double v0 = (hi2 ? col[0][2] : col[0][0]) + __shfl_xor_sync(0xffffffffu, hi2 ? col[0][0] : col[0][2], 2);
        const double v1 = (hi2 ? c3 : col[0][1]) + __shfl_xor_sync(0xffffffffu, hi2 ? col[0][1] : c3, 2);
        double v = (hi1 ? v1 : v0) + __shfl_xor_sync(0xffffffffu, hi1 ? v0 : v1, 1);
        v += __shfl_xor_sync(0xffffffffu, v, 4);
        if (!(lane & 4) && j0 + (lane >> 3) < nkeep) sacc[j0 + (lane >> 3)][lane & 3] += v;
    }
#pragma unroll
    for (int o = 32 / S; o < 32; o <<= 1)
#pragma unroll
        for (int c = 0; c < NC; ++c) ra[0][c] += __shfl_xor_sync(0xffffffffu, ra[0][c], o);
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
        if (gi[r] >= 0 && lane < 32 / S)
#pragma unroll
            for (int c = 0; c < NC; ++c) atomicAdd(&acc4[(size_t)c * n + gi[r]], c == 3 ? -ra[r][c] : ra[r][c]);
}

// All rows of a phase: 64 at a time, the rest in chunks that fit (a float64 slot without a row costs as much as one
// with a row).
template <int KERNEL, bool POT>
__device__ __forceinline__ void owner_phase_f64(const Bodies &pf, const Own64Batch *ob, int phase, int nrows,
                                                const dbl4 *sq, double (*sacc)[4], int ncol, int nkeep,
                                                const PairF64 &k, double *acc4, int n, int lane)
{
#define TG_ROWS64(R, S) owner_rows_f64<KERNEL, R, S, POT>(pf, ob, phase, i0, nrows, sq, sacc, ncol, nkeep, k, acc4, n, lane)
    for (int i0 = 0; i0 < nrows;) {
        const int rest = nrows - i0;
        if (rest > 48) {
            TG_ROWS64(2, 1);
            i0 += 64;
        } else if (rest > 16) {
            TG_ROWS64(1, 1);
            i0 += 32;
        } else if (rest > 8) {
            TG_ROWS64(1, 2);
            break;
        } else {
            TG_ROWS64(1, 4);
            break;
        }
    }
#undef TG_ROWS64
}

// Rows 8g .. 8g + 7 of a self pair (A, A), g = group, group + kSelf64Groups, ...: every particle sums over the
// others (both directions computed: a self pair is one of a leaf's hundred or more, and no column sums are
// needed).  A lane takes one of 8 rows and every fourth column, so that a deep rung's few leaves spread over
// several warps.  Fast rows feel the slow particles only.
constexpr int kSelf64Groups = 8;

template <int KERNEL, bool POT>
__device__ __noinline__ void self_pair_f64(const Bodies &pf, int fa, int na, int sa, int group, dbl4 *sq,
                                           const PairF64 &k, double *acc4, int n, int lane)
{
    const int slice = lane >> 3;
    for (int jc = 0; jc < na; jc += kMaxNcrit) {
        const int nbc = min(kMaxNcrit, na - jc);
        __syncwarp();
        for (int j = lane; j < nbc; j += 32) sq[j] = pf.get(fa + jc + j);
        __syncwarp();
        for (int i0 = 8 * group; i0 < na; i0 += 8 * kSelf64Groups) {
            const int i = i0 + (lane & 7);
            const bool row = i < na, slow = i < sa;
            const int jend = i0 < sa ? nbc : min(nbc, sa - jc);   // fast rows stop at the slow columns
            dbl4 p;
            p.x = p.y = p.z = p.w = 0.0;
            if (row) p = pf.get(fa + i);
            double ax = 0, ay = 0, az = 0, ph = 0;
            for (int j = slice; j < jend; j += 4) {
                const dbl4 q = sq[j];
                const bool use = jc + j != i && (slow || jc + j < sa);
                const double m = use ? q.w : 0.0;
                const double dx = q.x - p.x, dy = q.y - p.y, dz = q.z - p.z;
                double g, ri;
                const double s = pair_s2<KERNEL>(dx, dy, dz, k);
                pair_f64<KERNEL, POT>(use ? s : 1.0, k, g, ri);   // excluded: r = 1, finite at any softening
                const double mg = m * g;
                ax = fma(mg, dx, ax);
                ay = fma(mg, dy, ay);
                az = fma(mg, dz, az);
                if (POT) ph = fma(-m, ri, ph);
            }
#pragma unroll
            for (int o = 8; o <= 16; o <<= 1) {
                ax += __shfl_xor_sync(0xffffffffu, ax, o);
                ay += __shfl_xor_sync(0xffffffffu, ay, o);
                az += __shfl_xor_sync(0xffffffffu, az, o);
                if (POT) ph += __shfl_xor_sync(0xffffffffu, ph, o);
            }
            // lane slice c adds component c of its row
            const double v = slice == 0 ? ax : (slice == 1 ? ay : (slice == 2 ? az : ph));
            if (row && jend > 0 && slice < (POT ? 4 : 3)) atomicAdd(&acc4[(size_t)slice * n + fa + i], v);
        }
    }
}

// One warp per work unit of `unit` partners (own_unit), then the self pairs in row groups, all handed out by one counter
// as in p2p_owner_f32.
template <int KERNEL, bool POT>
__global__ void __launch_bounds__(32 * kOwn64Warps)
    p2p_owner_f64(TreeView t, const uint2 *__restrict__ units, uint32_t *ctr, const uint32_t *__restrict__ own_off,
                  const uint32_t *__restrict__ own_cnt, const int32_t *__restrict__ partners, int64_t npairs,
                  const uint2 *__restrict__ self_pairs, uint32_t nself, const Bodies pf,
                  const int32_t *__restrict__ nslow, double eps, double *acc4, int n,
                  unsigned long long *pair_counter, const unsigned long long *walk_ctr, const uint2 *p2p_base,
                  unsigned long long cap_p2p)
{
    if (walk_ctr) {
        npairs = (int64_t)walk_ctr[2];
        nself = (uint32_t)walk_ctr[4];
        self_pairs = p2p_base + (cap_p2p - nself);
    }
    extern __shared__ __align__(32) unsigned char own64_smem[];
    Own64Shared &sh = *reinterpret_cast<Own64Shared *>(own64_smem);
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    dbl4 *sq = sh.q[wib];
    double(*sacc)[4] = sh.acc[wib];
    Own64Batch *ob = &sh.b[wib];
    PairF64 k;
    k.init(eps, KERNEL == TG_KERNEL_PLUMMER);
    const int unit = own_unit(npairs, true);
    const uint32_t nunits = ctr[0];
    unsigned long long my_pairs = 0;
    for (;;) {
        uint32_t w = 0;
        if (lane == 0) w = atomicAdd(&ctr[1], 1u);
        w = __shfl_sync(0xffffffffu, w, 0);
        if (w >= nunits) {
            const uint32_t si = (w - nunits) / kSelf64Groups, group = (w - nunits) % kSelf64Groups;
            if (si >= nself) break;
            const int A = (int)self_pairs[si].x;
            const int fa = t.first[A], na = t.count[A], sa = nslow ? nslow[A] : na;
            if (sa == 0 || 8 * (int)group >= na) continue;   // no slow particle: every pair of the leaf is fast-fast
            self_pair_f64<KERNEL, POT>(pf, fa, na, sa, (int)group, sq, k, acc4, n, lane);
            if (lane == 0 && group == 0) {
                const unsigned long long nf = na - sa;
                my_pairs += (unsigned long long)na * (na - 1) / 2 - nf * (nf - (nf > 0 ? 1 : 0)) / 2;
            }
            continue;
        }
        const uint2 u = units[w];
        const int B = (int)u.x, pb = (int)u.y;
        const int np = min(unit, (int)own_cnt[B] - pb);
        const int fb = t.first[B], nb = t.count[B], sB = nslow ? nslow[B] : nb;
        __syncwarp();
        int cS = 0, cF = 0;
        if (lane < np) {
            const int A = partners[own_off[B] + pb + lane];
            const int na = t.count[A];
            cS = nslow ? nslow[A] : na;
            cF = na - cS;
            ob->first[lane] = t.first[A];
            ob->nslow[lane] = cS;
            my_pairs += (unsigned long long)na * nb - (unsigned long long)cF * (nb - sB);   // all minus fast-fast
        }
        const int incS = warp_incl_scan(cS, lane), incF = warp_incl_scan(cF, lane);
        ob->inc[0][lane] = incS;
        ob->inc[1][lane] = incF;
        const int Ts = __shfl_sync(0xffffffffu, incS, 31), Tf = __shfl_sync(0xffffffffu, incF, 31);
        if (Ts == 0 && (Tf == 0 || sB == 0)) continue;   // nothing but fast-fast pairs
        for (int jc = 0; jc < nb; jc += kMaxNcrit) {
            // columns in leaf order (slow first), padded to a multiple of 4 with massless ones; without
            // slow rows only the slow columns are staged
            const int nbc = min(kMaxNcrit, nb - jc), nsc = max(0, min(sB - jc, nbc));
            const int ns4 = (nsc + 3) & ~3, nt4 = (nbc + 3) & ~3;
            const int nstage = Ts > 0 ? nt4 : ns4, nflush = Ts > 0 ? nbc : nsc;
            if (nstage == 0) continue;
            __syncwarp();
            for (int j = lane; j < nstage; j += 32) {
                dbl4 q;
                q.x = q.y = q.z = q.w = 0.0;
                if (j < nbc) q = pf.get(fb + jc + j);
                sq[j] = q;
                sacc[j][0] = sacc[j][1] = sacc[j][2] = sacc[j][3] = 0.0;
            }
            __syncwarp();
            owner_phase_f64<KERNEL, POT>(pf, ob, 0, Ts, sq, sacc, nt4, nbc, k, acc4, n, lane);
            if (nsc > 0 && Tf > 0) {
                // fast rows meet the slow columns only: the fast columns of the last batch are made massless and
                // their reaction sums dropped
                __syncwarp();
                for (int j = nsc + lane; j < ns4; j += 32) sq[j].w = 0.0;
                __syncwarp();
                owner_phase_f64<KERNEL, POT>(pf, ob, 1, Tf, sq, sacc, ns4, nsc, k, acc4, n, lane);
            }
            __syncwarp();
            // a row's force is m_col g d, a column's -m_row g d
            for (int j = lane; j < nflush; j += 32)
#pragma unroll
                for (int c = 0; c < (POT ? 4 : 3); ++c) atomicAdd(&acc4[(size_t)c * n + fb + jc + j], -sacc[j][c]);
        }
    }
    my_pairs = warp_sum(my_pairs);
    if (lane == 0 && my_pairs) atomicAdd(pair_counter, my_pairs);
}

// Every float64 P2P pair, one launch.  Sizes from the host (npairs, self pairs) or, with walk_ctr, from the
// device (batched HOLD step), as for float32.
static tg_status launch_owner_f64(tg_ctx *c, const TreeView &t, const OwnerLists &o, int64_t npairs,
                                  const uint2 *self_pairs, int64_t nself, const Bodies &pf, const int32_t *nslow, bool pot,
                                  double *acc4, int stride, const unsigned long long *walk_ctr,
                                  const uint2 *p2p, size_t cap_p2p)
{
    const int smem = (int)sizeof(Own64Shared);
    ProfScope ps_(c, TG_K_P2P);
#define TG_OWNER64(K, PT)                                                                                          \
    do {                                                                                                           \
        cudaFuncSetAttribute(p2p_owner_f64<K, PT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);             \
        p2p_owner_f64<K, PT><<<c->num_sms * 3, 32 * kOwn64Warps, smem, c->stream>>>(                               \
            t, o.units, o.ctr, o.off, o.cnt, o.partners, npairs, self_pairs, (uint32_t)nself, pf, nslow, c->prm.eps, \
            acc4, stride, c->d_counters, walk_ctr, p2p, (unsigned long long)cap_p2p);                           \
    } while (0)
    if (c->prm.kernel == TG_KERNEL_PLUMMER) {
        if (pot) TG_OWNER64(TG_KERNEL_PLUMMER, true);
        else TG_OWNER64(TG_KERNEL_PLUMMER, false);
    } else {
        if (pot) TG_OWNER64(TG_KERNEL_WENDLAND_C2, true);
        else TG_OWNER64(TG_KERNEL_WENDLAND_C2, false);
    }
#undef TG_OWNER64
    return cuda_check(c, cudaGetLastError(), "p2p owner launch (float64)");
}

tg_status launch_p2p_f64(tg_ctx *c, const TreeView &t, const uint2 *pairs, int64_t npairs, const uint2 *self_pairs,
                         int64_t nself, const double *const xyzm[4], const int32_t *nslow, bool pot, double *acc4)
{
    if (npairs + nself == 0) return TG_OK;
    OwnerLists o;
    tg_status st = owner_lists(c, t, pairs, npairs, true, &o);
    if (st) return st;
    const Bodies pf{xyzm[0], xyzm[1], xyzm[2], xyzm[3]};
    return launch_owner_f64(c, t, o, npairs, self_pairs, nself, pf, nslow, pot, acc4, t.n, nullptr, nullptr, 0);
}

tg_status launch_p2p_f64_dev(tg_ctx *c, const TreeView &t, const DevEval *de, const unsigned long long *walk_ctr,
                             const uint2 *p2p, size_t cap_p2p, int cap_cells, const double *const xyzm[4],
                             const int32_t *nslow, double *acc4, int stride)
{
    OwnerLists o;
    tg_status st = owner_lists_dev(c, t, de, walk_ctr, p2p, cap_p2p, cap_cells, true, acc4, stride, &o);
    if (st) return st;
    const Bodies pf{xyzm[0], xyzm[1], xyzm[2], xyzm[3]};
    return launch_owner_f64(c, t, o, 0, nullptr, 0, pf, nslow, false, acc4, stride, walk_ctr, p2p, cap_p2p);
}

}  // namespace tg
