// octree.cu -- the octree of sorted Morton keys (Sec. 2.3 of Zhu 2017), built without a loop over its levels.
//
// A cell splits iff it holds more than n_crit particles.  With L(i, j) the number of levels at which the sorted
// keys i and j share their cell, the cell of level l around particle s splits iff some window of n_crit + 1
// consecutive keys around s lies inside it, i.e. iff l <= D(s) = max over a in [s - n_crit, s] of L(a, a + n_crit).
// So particle s lies in a leaf of level min(D(s) + 1, max_level) (level 0 if no window fits), and cells of the
// levels L(s - 1, s) + 1 .. leaf(s) begin at s.  One kernel finds both numbers for every particle and counts
// the cells per level and tile; a scan of these counts in level-major order gives every cell its place (cells of
// a level in Morton order, levels one after another); a second kernel writes the cells, and a third turns the
// ends into counts.  Four launches and no host wait, whatever the depth: bound by launch latency on small
// systems and by one and a half reads of the keys on large ones.
// (Splitting level by level took a count, a scan, a host read or a finishing launch, and an emit for each of
// up to 22 levels, and 130 of the 239 launches of a batched evaluation.  An evaluation of 1021 particles went from
// 745 to 537 us, a kick pair of 54,321 from 1389 to 1160 us, the disk galaxy's HOLD step from 883 to 846 ms.)
#include "tg_common.cuh"

namespace tg {

constexpr int kOctThreads = 256, kOctItems = 4, kOctTile = kOctThreads * kOctItems;
constexpr int kOctHalo = 2 * kMaxNcrit;            // largest n_crit
constexpr int kOctLevels = kMaxLevel + 1;
constexpr int kOctSlots = kOctTile / 32;           // warp-sized runs of a tile, in particle order
static_assert(kOctSlots == 32, "a warp scans one value per run");

// levels (1 .. 21) at which two keys share their cell
__device__ __forceinline__ int common_levels(uint64_t a, uint64_t b)
{
    const uint64_t x = a ^ b;
    return x == 0 ? kMaxLevel : kMaxLevel - 1 - (63 - __clzll((long long)x)) / 3;
}

__device__ __forceinline__ uint32_t compact3_21(uint64_t v)
{
    v &= 0x1249249249249249ull;
    v = (v | (v >> 2)) & 0x10c30c30c30c30c3ull;
    v = (v | (v >> 4)) & 0x100f00f00f00f00full;
    v = (v | (v >> 8)) & 0x1f0000ff0000ffull;
    v = (v | (v >> 16)) & 0x1f00000000ffffull;
    v = (v | (v >> 32)) & 0x1fffffull;
    return (uint32_t)v;
}

// lvl[s] = leaf(s) | (L(s - 1, s) + 1) << 8, and the cells of each level that begin in each tile:
// cnt[level * ntile + tile], ntile tiles over the positions 0 .. n (the last one closes the cells).
__global__ void __launch_bounds__(kOctThreads) oct_levels(const uint64_t *__restrict__ keys, int n, const int *dn,
                                                          int n_crit, int max_level, uint16_t *lvl, uint32_t *cnt)
{
    n = dev_or(dn, n);
    const int ntile = n / kOctTile + 1;
    __shared__ uint64_t sk[kOctTile + 2 * kOctHalo + 1];
    __shared__ int8_t win[2][kOctTile + kOctHalo];
    __shared__ uint32_t sc[kOctLevels];
    const int lane = threadIdx.x & 31;
    for (int tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
        const int s0 = tile * kOctTile, k0 = s0 - n_crit - 1;   // sk[i] = keys[k0 + i]
        __syncthreads();
        for (int i = threadIdx.x; i < kOctTile + 2 * n_crit + 1; i += kOctThreads)
            sk[i] = (k0 + i >= 0 && k0 + i < n) ? keys[k0 + i] : 0ull;
        if (threadIdx.x < kOctLevels) sc[threadIdx.x] = 0u;
        __syncthreads();
        // win[i]: the window starting at a = s0 - n_crit + i, -1 if it does not fit
        const int nw = kOctTile + n_crit;
        for (int i = threadIdx.x; i < nw; i += kOctThreads) {
            const int a = s0 - n_crit + i;
            win[0][i] = (a >= 0 && a + n_crit < n) ? (int8_t)common_levels(sk[i + 1], sk[i + 1 + n_crit]) : (int8_t)-1;
        }
        // maxima over runs of 2^k windows ending at i, up to the largest power of two in n_crit + 1
        int buf = 0, run = 1;
        for (; 2 * run <= n_crit + 1; run *= 2, buf ^= 1) {
            __syncthreads();
            for (int i = threadIdx.x; i < nw; i += kOctThreads) {
                const int8_t a = win[buf][i], b = i >= run ? win[buf][i - run] : (int8_t)-1;
                win[buf ^ 1][i] = a > b ? a : b;
            }
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kOctItems; ++j) {
            const int q = j * kOctThreads + threadIdx.x, s = s0 + q;
            int leaf = -1, from = 0;
            if (s < n) {
                // windows a in [s - n_crit, s] are entries q .. q + n_crit
                const int8_t a = win[buf][q + n_crit], b = win[buf][q + run - 1];
                const int split = a > b ? a : b;
                leaf = min(split + 1, max_level);
                from = s > 0 ? common_levels(sk[q + n_crit], sk[q + n_crit + 1]) + 1 : 0;
                lvl[s] = (uint16_t)(leaf | (from << 8));
            }
            for (int l = 0; l <= max_level; ++l) {
                const unsigned m = __ballot_sync(0xffffffffu, from <= l && l <= leaf);
                if (m && lane == 0) atomicAdd(&sc[l], (uint32_t)__popc(m));
            }
        }
        __syncthreads();
        if (threadIdx.x <= max_level) cnt[(size_t)threadIdx.x * ntile + tile] = sc[threadIdx.x];
    }
}

// Exclusive scan of cnt (levels 0 .. max_level, ntile entries each), and the sizes of the tree.  One block: the
// array holds (max_level + 1) entries per 1024 particles.  Levels beyond `levels` or cells beyond `cap` (batched
// path) are cut off: the tree then ends at the last level that fits, and the step is redone.  After a sort that gave
// up the keys are in no order: the evaluation then goes on without cells and without particles, so that nothing behind it
// reads a cell or an index.
__global__ void __launch_bounds__(1024) oct_scan(int n, const int *dn, int max_level, uint32_t *cnt, DevEval *de, int cap,
                                                 int levels, const uint32_t *flag)
{
    n = dev_or(dn, n);
    const int ntile = n / kOctTile + 1, m = (max_level + 1) * ntile;
    __shared__ uint32_t wtot[32], s_carry;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_carry = 0u;
    __syncthreads();
    for (int b = 0; b < m; b += 4096) {
        const int i0 = b + 4 * threadIdx.x;
        uint32_t v[4], sum = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            v[q] = i0 + q < m ? cnt[i0 + q] : 0u;
            sum += v[q];
        }
        uint32_t x = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wtot[warp] = x;
        __syncthreads();
        if (warp == 0) {
            uint32_t t = wtot[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, t, o);
                if (lane >= o) t += y;
            }
            wtot[lane] = t;
        }
        __syncthreads();
        uint32_t pre = s_carry + (warp ? wtot[warp - 1] : 0u) + x - sum;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (i0 + q < m) cnt[i0 + q] = pre;
            pre += v[q];
        }
        __syncthreads();
        if (threadIdx.x == 0) s_carry += wtot[31];
        __syncthreads();
    }
    if (threadIdx.x != 0) return;
    const int total = (int)s_carry;
    uint32_t over = 0u;
    int nlev = 0;
    de->level_begin[0] = 0;
    const bool unsorted = ((flag ? *flag : de->overflow) & kSortGaveUp) != 0;
    if (unsorted) de->n = 0;
    for (int l = 0; l <= max_level && !unsorted; ++l) {
        const int begin = (int)cnt[(size_t)l * ntile], end = l < max_level ? (int)cnt[(size_t)(l + 1) * ntile] : total;
        if (end == begin) break;
        if (end > cap) {
            over |= 1u;
            break;
        }
        if (l > levels) break;
        if (l == levels && levels < max_level) over |= 2u;   // deeper than the levels the later passes are issued for
        de->level_begin[l] = begin;
        de->level_begin[l + 1] = end;
        nlev = l + 1;
    }
    const int ncell = de->level_begin[nlev];
    de->nlev = nlev;
    de->ncell = ncell;
    de->rows = 2 * ncell;
    if (flag) de->overflow = *flag | over;   // host path: the sort's flag travels with the sizes
    else if (over) de->overflow |= over;
}

struct OctCells {
    uint8_t *level, *nchild;
    uint32_t *cx, *cy, *cz, *cend;   // cend: one past the last child (scratch)
    int32_t *first, *count, *child_first, *parent;
};

// The cells: rank of a cell among those of its level = cells of the level that begin at earlier positions.  A position
// also ends the cells of its predecessor at the levels where their keys differ (count holds the end until
// oct_finish).
__global__ void __launch_bounds__(kOctThreads) oct_cells(const uint64_t *__restrict__ keys, int n, const int *dn,
                                                         const uint16_t *__restrict__ lvl, int max_level,
                                                         const uint32_t *__restrict__ cnt, const DevEval *de, OctCells o)
{
    n = dev_or(dn, n);
    const int ntile = n / kOctTile + 1, last = de->nlev - 1;
    __shared__ uint32_t wc[kOctLevels][kOctSlots];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    for (int tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
        const int s0 = tile * kOctTile;
        int leaf[kOctItems], from[kOctItems], prev[kOctItems];
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kOctItems; ++j) {
            const int s = s0 + j * kOctThreads + threadIdx.x;
            leaf[j] = -1;
            from[j] = s <= n ? 0 : kOctLevels;
            prev[j] = -1;
            if (s < n) {
                const int v = lvl[s];
                leaf[j] = min(v & 0xff, last);
                from[j] = v >> 8;
            }
            if (s > 0 && s <= n) prev[j] = min((int)(lvl[s - 1] & 0xff), last);
            for (int l = 0; l <= last; ++l) {
                const unsigned m = __ballot_sync(0xffffffffu, from[j] <= l && l <= leaf[j]);
                if (lane == 0) wc[l][j * (kOctThreads / 32) + warp] = (uint32_t)__popc(m);
            }
        }
        __syncthreads();
        // place of the first cell of each run of 32 positions
        for (int l = warp; l <= last; l += kOctThreads / 32) {
            const uint32_t v = wc[l][lane];
            uint32_t x = v;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
                if (lane >= d) x += y;
            }
            wc[l][lane] = cnt[(size_t)l * ntile + tile] + x - v;
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kOctItems; ++j) {
            const int s = s0 + j * kOctThreads + threadIdx.x;
            const uint64_t key = s < n ? keys[s] : 0ull;
            const uint32_t x21 = compact3_21(key >> 2), y21 = compact3_21(key >> 1), z21 = compact3_21(key);
            int e_up = 0;        // cells of the level above that begin before s
            bool up = false;     // one of them begins at s
            for (int l = 0; l <= last; ++l) {
                const bool start = from[j] <= l && l <= leaf[j];
                const unsigned m = __ballot_sync(0xffffffffu, start);
                const int e = (int)(wc[l][j * (kOctThreads / 32) + warp] + __popc(m & lt));
                if (start) {
                    o.level[e] = (uint8_t)l;
                    o.cx[e] = x21 >> (kMaxLevel - l);
                    o.cy[e] = y21 >> (kMaxLevel - l);
                    o.cz[e] = z21 >> (kMaxLevel - l);
                    o.first[e] = s;
                    o.parent[e] = l > 0 ? e_up + (up ? 1 : 0) - 1 : -1;
                    if (l == leaf[j]) o.child_first[e] = -1;
                    if (up) o.child_first[e_up] = e;   // the first child begins where its parent does
                }
                if (from[j] <= l && l <= prev[j]) o.count[e - 1] = s;
                // the children of the cell that ends here were all placed before e
                if (from[j] < l && l <= prev[j]) o.cend[e_up - 1] = (uint32_t)e;
                e_up = e;
                up = start;
            }
        }
    }
}

__global__ void oct_finish(const DevEval *de, OctCells o)
{
    const int ncell = de->ncell;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < ncell; c += gridDim.x * blockDim.x) {
        o.count[c] -= o.first[c];
        o.nchild[c] = o.child_first[c] < 0 ? (uint8_t)0 : (uint8_t)((int)o.cend[c] - o.child_first[c]);
    }
}

static tg_status oct_buffers(tg_ctx *c, int cells, OctCells *o)
{
    tg_status st;
    if ((st = ensure_t(c, B_C_LEVEL, cells, &o->level)) || (st = ensure_t(c, B_C_X, cells, &o->cx)) ||
        (st = ensure_t(c, B_C_Y, cells, &o->cy)) || (st = ensure_t(c, B_C_Z, cells, &o->cz)) ||
        (st = ensure_t(c, B_C_FIRST, cells, &o->first)) || (st = ensure_t(c, B_C_COUNT, cells, &o->count)) ||
        (st = ensure_t(c, B_C_CHILD, cells, &o->child_first)) || (st = ensure_t(c, B_C_PARENT, cells, &o->parent)) ||
        (st = ensure_t(c, B_C_NCHILD, cells, &o->nchild)) || (st = ensure_t(c, B_C_CEND, cells, &o->cend)))
        return st;
    return TG_OK;
}

size_t oct_count_words(int n) { return (size_t)kOctLevels * (size_t)(n / kOctTile + 1); }

tg_status build_octree(tg_ctx *c, int n, int *ncell_out)
{
    tg_status st;
    const uint64_t *keys = static_cast<const uint64_t *>(c->buf[B_KEYS0].p);
    const Geom *geom = static_cast<const Geom *>(c->buf[B_GEOM].p);
    uint16_t *lvl;
    uint32_t *cnt;
    DevEval *de;
    if ((st = ensure_t(c, B_C_LVL, n, &lvl)) || (st = ensure_t(c, B_C_CNT, oct_count_words(n), &cnt)) ||
        (st = ensure_t(c, B_OCT, 1, &de)))
        return st;
    const int grid = std::min(n / kOctTile + 1, c->num_sms * 8);
    {
        ProfScope ps_(c, TG_K_TREE);
        oct_levels<<<grid, kOctThreads, 0, c->stream>>>(keys, n, nullptr, c->prm.n_crit, c->prm.max_level, lvl, cnt);
    }
    {
        ProfScope ps_(c, TG_K_TREE);
        oct_scan<<<1, 1024, 0, c->stream>>>(n, nullptr, c->prm.max_level, cnt, de, INT32_MAX, kMaxLevel + 1,
                                            sort_scratch(c->buf[B_SORT].p, n).flag);
    }
    // the sizes of the tree, and the root cube's side for the walk, with one wait
    DevEval *h = reinterpret_cast<DevEval *>(c->h_pinned);
    static_assert(sizeof(DevEval) <= 32 * sizeof(int64_t), "read into the first half of the staging area");
    cudaMemcpyAsync(h, de, sizeof(DevEval), cudaMemcpyDeviceToHost, c->stream);
    cudaMemcpyAsync(c->h_pinned + 32, &geom->log2L, sizeof(int), cudaMemcpyDeviceToHost, c->stream);
    cudaError_t e = stream_sync(c);
    if (e != cudaSuccess) return cuda_check(c, e, "octree");
    c->walk_log2L = *reinterpret_cast<int *>(c->h_pinned + 32);
    if (h->overflow & kSortGaveUp) {
        cudaMemsetAsync(c->buf[B_SORT].p, 0, 256, c->stream);
        return set_err(c, TG_ERR_TIMEOUT, "a bounded wait of the particle sort ran out");
    }
    const int ncell = h->ncell;
    c->level_begin.assign(h->level_begin, h->level_begin + h->nlev + 1);
    OctCells o;
    if ((st = oct_buffers(c, ncell, &o))) return st;
    {
        ProfScope ps_(c, TG_K_TREE);
        oct_cells<<<grid, kOctThreads, 0, c->stream>>>(keys, n, nullptr, lvl, c->prm.max_level, cnt, de, o);
    }
    {
        ProfScope ps_(c, TG_K_TREE);
        oct_finish<<<grid_for(ncell, 256), 256, 0, c->stream>>>(de, o);
    }
    *ncell_out = ncell;
    return cuda_check(c, cudaGetLastError(), "octree");
}

// The same with every size on the device (batched path): at most `cap` cells, and levels up to `levels`; a tree that
// needs more sets an overflow bit and is cut off at the last level that fits.
tg_status build_octree_dev(tg_ctx *c, DevEval *de, int cap_n, int cap, int levels)
{
    tg_status st;
    const uint64_t *keys = static_cast<const uint64_t *>(c->buf[B_KEYS0].p);
    uint16_t *lvl;
    uint32_t *cnt;
    OctCells o;
    if ((st = ensure_t(c, B_C_LVL, cap_n, &lvl)) || (st = ensure_t(c, B_C_CNT, oct_count_words(cap_n), &cnt)) ||
        (st = oct_buffers(c, cap, &o)))
        return st;
    const int grid = std::min(cap_n / kOctTile + 1, c->num_sms * 8);
    ProfScope ps0_(c, TG_K_TREE), ps1_(c, TG_K_TREE), ps2_(c, TG_K_TREE), ps3_(c, TG_K_TREE);
    oct_levels<<<grid, kOctThreads, 0, c->stream>>>(keys, 0, &de->n, c->prm.n_crit, c->prm.max_level, lvl, cnt);
    oct_scan<<<1, 1024, 0, c->stream>>>(0, &de->n, c->prm.max_level, cnt, de, cap, levels, nullptr);
    oct_cells<<<grid, kOctThreads, 0, c->stream>>>(keys, 0, &de->n, lvl, c->prm.max_level, cnt, de, o);
    oct_finish<<<grid_for(cap, 256, c->num_sms * 8), 256, 0, c->stream>>>(de, o);
    return cuda_check(c, cudaGetLastError(), "octree (device sizes)");
}

}  // namespace tg
