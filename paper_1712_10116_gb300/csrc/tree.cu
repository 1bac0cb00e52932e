// tree.cu -- root cube, Morton keys, stable LSD radix sort and gather (Sec. 2.3 of Zhu 2017: octree with leaf
// size n_crit, built for every call; the octree itself is octree.cu).
//
// Keys: 21 bits per axis, x the most significant bit of each 3-bit group, so a cell at level l
// is the run of sorted keys sharing the top 3l bits.  The sort orders (key, input index), so ties
// keep input order.  Cells are emitted level by level in Morton order of their key prefix.
#include <cstdarg>
#include <cstring>

#include "tg_common.cuh"

namespace tg {

// ------------------------------------------------------------------ errors and buffers
tg_status set_err(tg_ctx *c, tg_status code, const char *fmt, ...)
{
    if (c->err.code == TG_OK) {
        char msg[512];
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(msg, sizeof msg, fmt, ap);
        va_end(ap);
        c->err.code = code;
        c->err.msg = msg;
    }
    return code;
}

cudaError_t stream_sync(tg_ctx *c)
{
    c->stats.host_syncs += 1;
    return cudaStreamSynchronize(c->stream);
}

tg_status cuda_check(tg_ctx *c, cudaError_t e, const char *what)
{
    if (e == cudaSuccess) return TG_OK;
    return set_err(c, e == cudaErrorMemoryAllocation ? TG_ERR_OOM : TG_ERR_CUDA, "%s: %s", what,
                   cudaGetErrorString(e));
}

tg_status injected_alloc_failure(tg_ctx *c, size_t bytes, int slot)
{
    if (c->debug_fail_alloc_after < 0) return TG_OK;
    if (c->debug_fail_alloc_after == 0)
        return set_err(c, TG_ERR_OOM, "allocation of %zu bytes for scratch slot %d failed (injected)", bytes, slot);
    c->debug_fail_alloc_after -= 1;
    return TG_OK;
}

tg_status ensure(tg_ctx *c, int slot, size_t bytes, void **out)
{
    Buf &b = c->buf[slot];
    if (b.bytes < bytes) {
        size_t nb = bytes + bytes / 4 + 256;
        if (c->capturing)
            return set_err(c, TG_ERR_CAPACITY, "scratch slot %d would grow to %zu bytes inside a graph capture", slot, nb);
        if (tg_status inj = injected_alloc_failure(c, nb, slot)) return inj;
        c->alloc_epoch += 1;
        if (b.p) {
            cudaError_t e = stream_sync(c);
            if (e != cudaSuccess) return cuda_check(c, e, "sync before regrow");
            cudaFree(b.p);
            b.p = nullptr;
            b.bytes = 0;
        }
        cudaError_t e = cudaMalloc(&b.p, nb);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return set_err(c, TG_ERR_OOM, "cudaMalloc(%zu) for scratch slot %d failed", nb, slot);
        }
        b.bytes = nb;
    }
    *out = b.p;
    return TG_OK;
}

// ------------------------------------------------------------------ live kernel timing
ProfScope::ProfScope(tg_ctx *ctx, int k) : c(ctx), cls(k), timed(false)
{
    c->prof_launches[k] += 1;
    if (c->prof_level >= 2 || (c->prof_level == 1 && (k == TG_K_M2L || k == TG_K_P2P))) {
        if (c->prof_used >= 2048) prof_collect(c);
        while (c->prof_events.size() < 2 * (c->prof_used + 1)) {
            cudaEvent_t e;
            if (cudaEventCreate(&e) != cudaSuccess) {
                cudaGetLastError();
                return;
            }
            c->prof_events.push_back(e);
        }
        if (c->prof_class.size() < c->prof_used + 1) c->prof_class.resize(c->prof_used + 1);
        c->prof_class[c->prof_used] = k;
        cudaEventRecord(c->prof_events[2 * c->prof_used], c->stream);
        timed = true;
    }
}

ProfScope::~ProfScope()
{
    if (!timed) return;
    cudaEventRecord(c->prof_events[2 * c->prof_used + 1], c->stream);
    c->prof_used += 1;
}

tg_status prof_collect(tg_ctx *c)
{
    if (c->prof_used == 0) return TG_OK;
    cudaError_t e = stream_sync(c);
    if (e != cudaSuccess) return cuda_check(c, e, "profile collect");
    for (size_t i = 0; i < c->prof_used; ++i) {
        float ms = 0.f;
        if (cudaEventElapsedTime(&ms, c->prof_events[2 * i], c->prof_events[2 * i + 1]) == cudaSuccess)
            c->prof_ms[c->prof_class[i]] += ms;
        else
            cudaGetLastError();
    }
    c->prof_used = 0;
    return TG_OK;
}

// ------------------------------------------------------------------ exclusive scan (uint32)
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t *total)
{
    __shared__ uint32_t warp_tot[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[warp] = x;
    __syncthreads();
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
        uint32_t t = lane < nw ? warp_tot[lane] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        warp_tot[lane] = t;   // inclusive
    }
    __syncthreads();
    uint32_t base = warp > 0 ? warp_tot[warp - 1] : 0u;
    *total = warp_tot[(blockDim.x >> 5) - 1];
    __syncthreads();
    return base + x - v;
}

__global__ void scan_tiles(const uint32_t *in, uint32_t *out, uint32_t *tile_sums, int n, const int *dn)
{
    n = dev_or(dn, n);
    const int64_t base = (int64_t)blockIdx.x * kScanTile + threadIdx.x * kScanItems;
    uint32_t v[kScanItems];
    uint32_t s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        v[i] = (base + i < n) ? in[base + i] : 0u;
        s += v[i];
    }
    uint32_t tot;
    uint32_t pre = block_exclusive_scan(s, &tot);
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        if (base + i < n) out[base + i] = pre;
        pre += v[i];
    }
    if (threadIdx.x == 0) tile_sums[blockIdx.x] = tot;
}

__global__ void scan_add(uint32_t *out, const uint32_t *tile_pre, int n, const int *dn)
{
    n = dev_or(dn, n);
    const int64_t base = (int64_t)blockIdx.x * kScanTile + threadIdx.x * kScanItems;
    const uint32_t add = tile_pre[blockIdx.x];
#pragma unroll
    for (int i = 0; i < kScanItems; ++i)
        if (base + i < n) out[base + i] += add;
}

size_t scan_scratch_words(int n)
{
    size_t need = 4;
    for (int m = n;;) {
        const int nt = (m + kScanTile - 1) / kScanTile;
        need += 2 * (size_t)nt + 2;
        if (nt == 1) break;
        m = nt;
    }
    return need;
}

// Exclusive scan of n uint32 values (out may alias in).  The total is written to d_total (device word)
// when it is not null.  Recursive over tile sums.  With dn (a device count) the first
// level scans dn[0] <= n values; the launches are sized for n, and the tiles past dn[0] hand up
// zero sums, so the upper levels need no device count.
tg_status exclusive_scan_u32(tg_ctx *c, const uint32_t *in, uint32_t *out, int n, uint32_t *d_total, const int *dn)
{
    if (n <= 0) {
        if (d_total) cudaMemsetAsync(d_total, 0, sizeof(uint32_t), c->stream);
        return cuda_check(c, cudaGetLastError(), "exclusive scan");
    }
    uint32_t *tmp = nullptr;
    tg_status st = ensure_t(c, B_SCAN_TMP, scan_scratch_words(n), &tmp);
    if (st) return st;
    struct Level { uint32_t *out; int n, ntiles; uint32_t *sums, *pre; };
    Level lv[8];
    int depth = 0;
    const uint32_t *cin = in;
    uint32_t *cout = out;
    int cn = n;
    uint32_t *cursor = tmp;
    while (true) {
        int nt = (cn + kScanTile - 1) / kScanTile;
        lv[depth] = {cout, cn, nt, cursor, cursor + nt};
        {
            ProfScope ps_(c, TG_K_OTHER);
            scan_tiles<<<nt, kScanThreads, 0, c->stream>>>(cin, cout, cursor, cn, depth == 0 ? dn : nullptr);
        }
        ++depth;
        if (nt == 1) break;
        cin = cursor;
        cout = cursor + nt;
        cn = nt;
        cursor += 2 * nt + 2;
    }
    for (int d = depth - 2; d >= 0; --d)
        {
            ProfScope ps_(c, TG_K_OTHER);
            scan_add<<<lv[d].ntiles, kScanThreads, 0, c->stream>>>(lv[d].out, lv[d].pre, lv[d].n, d == 0 ? dn : nullptr);
        }
    if (d_total)
        cudaMemcpyAsync(d_total, lv[depth - 1].sums, sizeof(uint32_t), cudaMemcpyDeviceToDevice, c->stream);
    return cuda_check(c, cudaGetLastError(), "exclusive scan");
}

// ------------------------------------------------------------------ root cube
__device__ __forceinline__ double pos_at(const double *pos, int64_t stride, const int64_t *sub, int64_t q, int axis)
{
    int64_t i = sub ? sub[q] : q;
    return pos[axis * stride + i];
}

// The box over the block's threads: mn, mx per thread in, r[0..2] = minimum, r[3..5] = maximum out (shared memory,
// six values per warp in s).  The whole block calls it.
__device__ __forceinline__ void block_box(double (&mn)[3], double (&mx)[3], double (*s)[32], double *r)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        double lo = mn[a], hi = mx[a];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
            hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        }
        if (lane == 0) {
            s[a][warp] = lo;
            s[3 + a][warp] = hi;
        }
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        double v = s[threadIdx.x][0];
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w)
            v = threadIdx.x < 3 ? fmin(v, s[threadIdx.x][w]) : fmax(v, s[threadIdx.x][w]);
        r[threadIdx.x] = v;
    }
    __syncthreads();
}

// Root cube from the bounding box r: L = smallest power of two >= extent * (1 + 2^-20) (1 if the extent is 0),
// lo = floor(min / h) * h with h = L / 2^21.
__device__ __forceinline__ void root_of_box(const double *r, int n, Geom *g)
{
    if (n <= 0) {
        for (int a = 0; a < 3; ++a) g->lo[a] = 0.0;
        g->L = 1.0;
        g->log2L = 0;
        g->inv_h = ldexp(1.0, kMaxLevel);
        return;
    }
    double ext = 0.0;
    for (int a = 0; a < 3; ++a) {
        double e = __dsub_rn(r[3 + a], r[a]);
        if (e > ext) ext = e;
    }
    double L = 1.0;
    int log2L = 0;
    if (ext > 0.0) {
        double t = __dmul_rn(ext, 1.0 + ldexp(1.0, -20));
        int e;
        double f = frexp(t, &e);
        if (f == 0.5) {
            L = t;
            log2L = e - 1;
        } else {
            L = ldexp(1.0, e);
            log2L = e;
        }
    }
    double h = ldexp(L, -kMaxLevel);
    for (int a = 0; a < 3; ++a) g->lo[a] = __dmul_rn(floor(__ddiv_rn(r[a], h)), h);
    g->L = L;
    g->log2L = log2L;
    g->inv_h = ldexp(1.0, kMaxLevel - log2L);
}

// Bounding box and root cube in one launch: the block that finishes last reduces the blocks' boxes (s.done counts
// them and is back at zero afterwards).  The blocks also clear the sort's counters.
__global__ void __launch_bounds__(kBoxThreads) root_cube(const double *pos, int64_t stride, const int64_t *sub, int n,
                                                         const int *dn, SortScratch s, Geom *g)
{
    n = dev_or(dn, n);
    if (dn && n <= kSmallSort) return;   // batched path: sort_small does it
    __shared__ double part[6][32], r[6];
    __shared__ bool s_last;
    double mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY};
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, nt = (int64_t)gridDim.x * blockDim.x;
    for (int64_t q = tid; q < n; q += nt) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            double v = pos_at(pos, stride, sub, q, a);
            mn[a] = fmin(mn[a], v);
            mx[a] = fmax(mx[a], v);
        }
    }
    for (int64_t i = tid; i < kSortPasses * (kSortBins + 1); i += nt) s.hist[i] = 0u;   // and the tickets behind them
    block_box(mn, mx, part, r);
    if (threadIdx.x < 6) s.boxes[blockIdx.x * 6 + threadIdx.x] = r[threadIdx.x];
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(s.done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        mn[a] = INFINITY;
        mx[a] = -INFINITY;
    }
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x)
        for (int a = 0; a < 3; ++a) {
            mn[a] = fmin(mn[a], __ldcg(&s.boxes[b * 6 + a]));
            mx[a] = fmax(mx[a], __ldcg(&s.boxes[b * 6 + 3 + a]));
        }
    block_box(mn, mx, part, r);
    if (threadIdx.x == 0) {
        root_of_box(r, n, g);
        *s.done = 0u;
    }
}

// ------------------------------------------------------------------ input check
__global__ void count_nonfinite(const double *pos, int64_t stride, const int64_t *sub, int64_t n, const double *mass,
                                unsigned long long *bad)
{
    unsigned long long cnt = 0;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = sub ? sub[q] : q;
        const bool ok = isfinite(pos[i]) && isfinite(pos[stride + i]) && isfinite(pos[2 * stride + i]) &&
                        (mass == nullptr || isfinite(mass[i]));
        cnt += ok ? 0ull : 1ull;
    }
    cnt = warp_sum(cnt);
    if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(bad, cnt);
}

tg_status check_finite(tg_ctx *c, int64_t n, const double *pos, int64_t stride, const int64_t *sub, const double *mass)
{
    if (n <= 0) return TG_OK;
    unsigned long long *bad = c->d_counters + 10;
    cudaMemsetAsync(bad, 0, sizeof(unsigned long long), c->stream);
    {
        ProfScope ps_(c, TG_K_OTHER);
        count_nonfinite<<<grid_for(n, 256, 2 * c->num_sms), 256, 0, c->stream>>>(pos, stride, sub, n, mass, bad);
    }
    unsigned long long *h = reinterpret_cast<unsigned long long *>(c->h_pinned + 56);
    cudaMemcpyAsync(h, bad, sizeof(unsigned long long), cudaMemcpyDeviceToHost, c->stream);
    cudaError_t e = stream_sync(c);
    if (e != cudaSuccess) return cuda_check(c, e, "finiteness check");
    if (*h) return set_err(c, TG_ERR_NONFINITE, "%llu particles have a non-finite position or mass", *h);
    return TG_OK;
}

// ------------------------------------------------------------------ keys
__device__ __forceinline__ uint64_t cell_coord(double x, double lo, double inv_h)
{
    double t = floor(__dmul_rn(__dsub_rn(x, lo), inv_h));
    if (t < 0.0) t = 0.0;
    const double top = (double)((1 << kMaxLevel) - 1);
    if (t > top) t = top;
    return (uint64_t)t;
}

__device__ __forceinline__ uint64_t morton_key(const double *pos, int64_t stride, const int64_t *sub, int64_t q, const Geom &g)
{
    const uint64_t cx = cell_coord(pos_at(pos, stride, sub, q, 0), g.lo[0], g.inv_h);
    const uint64_t cy = cell_coord(pos_at(pos, stride, sub, q, 1), g.lo[1], g.inv_h);
    const uint64_t cz = cell_coord(pos_at(pos, stride, sub, q, 2), g.lo[2], g.inv_h);
    return (spread3_21(cx) << 2) | (spread3_21(cy) << 1) | spread3_21(cz);
}

// Keys and indices in input order, the digit counts of all seven passes of the sort, and the cleared tile states of
// the first.
__global__ void __launch_bounds__(256) morton_keys(const double *pos, int64_t stride, const int64_t *sub, int n,
                                                   const int *dn, const Geom *gp, uint64_t *keys, uint32_t *vals,
                                                   SortScratch s)
{
    n = dev_or(dn, n);
    if (dn && n <= kSmallSort) return;
    __shared__ uint32_t h[kSortPasses * kSortBins];
    for (int d = threadIdx.x; d < kSortPasses * kSortBins; d += blockDim.x) h[d] = 0u;
    __syncthreads();
    const Geom g = *gp;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, nt = (int64_t)gridDim.x * blockDim.x;
    for (int64_t q = tid; q < n; q += nt) {
        const uint64_t key = morton_key(pos, stride, sub, q, g);
        keys[q] = key;
        vals[q] = (uint32_t)q;
#pragma unroll
        for (int p = 0; p < kSortPasses; ++p)
            atomicAdd(&h[p * kSortBins + (int)((key >> (p * kSortBits)) & (kSortBins - 1u))], 1u);
    }
    const int64_t words = (int64_t)((n + kSortTileItems - 1) / kSortTileItems) * kSortBins;
    for (int64_t i = tid; i < words; i += nt) s.state[0][i] = 0u;
    __syncthreads();
    for (int d = threadIdx.x; d < kSortPasses * kSortBins; d += blockDim.x)
        if (h[d]) atomicAdd(&s.hist[d], h[d]);
}

// ------------------------------------------------------------------ radix sort
// Stable LSD over the 63 key bits in 9-bit digits, one launch per pass.  Tiles of 2048 items: 8 warps x 8 rounds x
// 32 lanes, item index = warp*256 + round*32 + lane, so a warp's rounds run in input order and ranks are stable.
// A tile's digit counts are published in s.state as soon as they are known, (count << 2) | 1, and the sum over
// this and all earlier tiles, (sum << 2) | 2, once it is; a tile adds up its predecessors' words backwards until
// it meets a sum (decoupled look-back, Merrill and Garland 2016).  Tiles are handed out by a ticket, so a tile
// only waits for blocks that already run and wait for nothing before they publish; the wait is bounded all the
// same and raises s.flag when it runs out.  A pass that gave up leaves part of its output unwritten, so nothing
// reads the sorted indices while the flag is up: the gather returns, the octree comes out empty, and the host
// reports TG_ERR_TIMEOUT.  Each pass clears the other pass's states.
// Bound by latency up to a million items (10 us a pass at 54,321, where a histogram launch, one to three scan
// launches and a scatter launch took 28; the whole allocation-free sort of 200,001 went from 231 to 116 us) and at
// 1.7 TB/s beyond (4,194,304 items: 61 us a pass, about 85 before).  Reading 4 / 8 / 16 predecessors at a time: 123 / 116 /
// 118 us for 200,001.
constexpr int kSortThreads = 256;
constexpr int kSortItems = 8;
constexpr unsigned kSortSpin = 1u << 18;   // some 0.2 s; a wait lasts microseconds
constexpr unsigned kSortSpinHeld = 1u << 10;   // with a held tile, which every wait runs into
static_assert(kSortBins == 2 * kSortThreads, "two digits to each thread");
static_assert(kSortThreads * kSortItems == kSortTileItems, "tile size");

// Sums over the tiles before `tile` of a thread's two digit counts (one 64-bit word per tile and thread, so both
// flags change at once).  Eight predecessors are read at a time: their loads overlap.
constexpr int kSortAhead = 8;
template <unsigned LIMIT>
__device__ __forceinline__ uint2 look_back(const volatile unsigned long long *state, int tile, uint32_t *flag)
{
    uint2 sum = make_uint2(0u, 0u);
    unsigned spins = 0;
    for (int t = tile - 1; t >= 0;) {
        unsigned long long w[kSortAhead];
#pragma unroll
        for (int k = 0; k < kSortAhead; ++k) w[k] = state[(size_t)max(t - k, 0) * kSortThreads];
#pragma unroll
        for (int k = 0; k < kSortAhead; ++k) {
            const uint32_t lo = (uint32_t)w[k], hi = (uint32_t)(w[k] >> 32);
            if ((lo & 3u) == 0u) break;   // not published yet: read it again
            sum.x += lo >> 2;
            sum.y += hi >> 2;
            --t;
            if (lo & 2u) return sum;   // tile 0 always holds a sum
            spins = 0;
        }
        if (++spins > LIMIT) {
            atomicOr(flag, kSortGaveUp);
            return sum;
        }
    }
    return sum;
}

// HELD: the test hook, a variant of its own (the tile and the limit as arguments of the one kernel made a sort of
// 200,001 particles 123 us instead of 116).
template <bool HELD>
__global__ void __launch_bounds__(kSortThreads) radix_pass(const uint64_t *__restrict__ keys_in,
                                                           const uint32_t *__restrict__ vals_in, uint64_t *keys_out,
                                                           uint32_t *vals_out, int n, const int *dn, int pass,
                                                           SortScratch s, int hold)
{
    n = dev_or(dn, n);
    if (dn && n <= kSmallSort) return;
    const int ntile = (n + kSortTileItems - 1) / kSortTileItems, shift = pass * kSortBits;
    if ((int)blockIdx.x >= ntile) return;
    __shared__ uint32_t wcount[8][kSortBins];
    __shared__ uint32_t dstart[kSortBins], place[kSortBins];
    __shared__ uint32_t wsum[8], hsum[8];
    __shared__ uint64_t sk[kSortTileItems];
    __shared__ uint32_t sv[kSortTileItems];
    __shared__ int s_tile;
    if (threadIdx.x == 0) s_tile = (int)atomicAdd(&s.hist[kSortPasses * kSortBins + pass], 1u);
    for (int i = threadIdx.x; i < 8 * kSortBins; i += kSortThreads) (&wcount[0][0])[i] = 0;
    __syncthreads();
    const int tile = s_tile;
    if (tile >= ntile) return;   // calls that overlap on one scratch array (allocation-free sort) only
    uint32_t *state = s.state[pass & 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t lt_mask = (1u << lane) - 1u;
    const int64_t base = (int64_t)tile * kSortTileItems + warp * 256 + lane;
    uint64_t k[kSortItems];
    uint32_t v[kSortItems], rank[kSortItems], dig[kSortItems];
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const int64_t idx = base + r * 32;
        const bool valid = idx < n;
        k[r] = valid ? keys_in[idx] : ~0ull;   // past the end: the largest digit, after every valid item
        v[r] = valid ? vals_in[idx] : 0u;
    }
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const uint32_t d = (uint32_t)((k[r] >> shift) & (kSortBins - 1u));
        dig[r] = d;
        const uint32_t peers = __match_any_sync(0xffffffffu, d);
        const uint32_t lower = peers & lt_mask;
        const uint32_t pre = wcount[warp][d];
        rank[r] = pre + __popc(lower);
        __syncwarp();
        if (lower == 0) wcount[warp][d] = pre + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    // thread t owns digits 2t, 2t + 1: prefix over the warps, tile totals (less the padding), published at once
    const int tile0 = tile * kSortTileItems, cnt = min(n - tile0, kSortTileItems);
    uint32_t tot[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int d = 2 * threadIdx.x + q;
        uint32_t run = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            const uint32_t t = wcount[w][d];
            wcount[w][d] = run;
            run += t;
        }
        tot[q] = run - (d == (int)kSortBins - 1 ? (uint32_t)(kSortTileItems - cnt) : 0u);
    }
    volatile unsigned long long *mine =
        reinterpret_cast<volatile unsigned long long *>(state) + (size_t)tile * kSortThreads + threadIdx.x;
    {
        const uint32_t f = tile == 0 ? 2u : 1u;
        if (!HELD || tile != hold) *mine = (unsigned long long)((tot[0] << 2) | f) | ((unsigned long long)((tot[1] << 2) | f) << 32);
        reinterpret_cast<uint2 *>(s.state[(pass + 1) & 1] + (size_t)tile * kSortBins)[threadIdx.x] = make_uint2(0u, 0u);
    }
    // exclusive scans over the digits: of the tile's totals (with the padding, which sits at the end) and of the
    // whole input's digit counts
    const uint2 all = reinterpret_cast<const uint2 *>(s.hist + pass * kSortBins)[threadIdx.x];
    uint32_t incl = tot[0] + tot[1], hincl = all.x + all.y;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o), z = __shfl_up_sync(0xffffffffu, hincl, o);
        if (lane >= o) {
            incl += y;
            hincl += z;
        }
    }
    if (lane == 31) {
        wsum[warp] = incl;
        hsum[warp] = hincl;
    }
    __syncthreads();
    uint32_t before = 0, hbefore = 0;
    for (int w = 0; w < warp; ++w) {
        before += wsum[w];
        hbefore += hsum[w];
    }
    const uint32_t excl = before + incl - (tot[0] + tot[1]), hexcl = hbefore + hincl - (all.x + all.y);
    dstart[2 * threadIdx.x] = excl;
    dstart[2 * threadIdx.x + 1] = excl + tot[0];
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const uint32_t lp = dstart[dig[r]] + wcount[warp][dig[r]] + rank[r];
        sk[lp] = k[r];
        sv[lp] = v[r];
    }
    // where the tile's run of each digit goes, less its place in the tile
    uint2 pre = make_uint2(0u, 0u);
    if (tile > 0) {
        pre = look_back<HELD ? kSortSpinHeld : kSortSpin>(
            reinterpret_cast<const volatile unsigned long long *>(state) + threadIdx.x, tile, s.flag);
        if (!HELD || tile != hold)
            *mine = (unsigned long long)(((pre.x + tot[0]) << 2) | 2u) | ((unsigned long long)(((pre.y + tot[1]) << 2) | 2u) << 32);
    }
    place[2 * threadIdx.x] = hexcl + pre.x - excl;
    place[2 * threadIdx.x + 1] = hexcl + all.x + pre.y - (excl + tot[0]);
    __syncthreads();
    for (int i = threadIdx.x; i < cnt; i += kSortThreads) {
        const uint64_t key = sk[i];
        const uint32_t at = place[(uint32_t)((key >> shift) & (kSortBins - 1u))] + (uint32_t)i;
        if (at < (uint32_t)n) {
            keys_out[at] = key;
            vals_out[at] = sv[i];
        }
    }
}

__device__ __forceinline__ void gather_one(int64_t s, uint32_t q, const double *pos, int64_t stride, const int64_t *sub,
                                           const double *mass, const uint8_t *fast, const SortedOut &o)
{
    const int64_t i = sub ? sub[q] : (int64_t)q;
    o.x[s] = pos[i];
    o.y[s] = pos[stride + i];
    o.z[s] = pos[2 * stride + i];
    o.m[s] = mass[i];
    o.f[s] = fast ? (fast[q] != 0) : 0;
}

__global__ void gather_sorted(const uint32_t *perm, const double *pos, int64_t stride, const int64_t *sub,
                              const double *mass, const uint8_t *fast, int n, const int *dn, const uint32_t *flag,
                              SortedOut o)
{
    n = dev_or(dn, n);
    if (dn && n <= kSmallSort) return;
    if (*flag & kSortGaveUp) return;   // perm is incomplete: indices of an earlier call or none at all
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x)
        gather_one(s, perm[s], pos, stride, sub, mass, fast, o);
}

// Up to kSmallSort particles: root cube, keys, the seven passes and the gather in one launch of one block, the items
// in shared memory between the passes (a launch costs as much as a pass on so few items).  Warp w holds the
// items [w R 32, (w + 1) R 32), R = ceil(n / 1024), in rounds of 32.
struct SmallSort {
    uint64_t k[kSmallSort];
    uint16_t v[kSmallSort];
    uint16_t wcount[32][kSortBins];
    uint32_t dstart[kSortBins], wsum[32];
    double part[6][32], box[6];
    Geom g;
};

__global__ void __launch_bounds__(1024) sort_small(const double *pos, int64_t stride, const int64_t *sub, int n,
                                                   const int *dn, const double *mass, const uint8_t *fast, Geom *g,
                                                   uint64_t *keys, uint32_t *vals, SortedOut o)
{
    n = dev_or(dn, n);
    if (n > kSmallSort) return;
    extern __shared__ __align__(16) unsigned char small_smem[];
    SmallSort &sh = *reinterpret_cast<SmallSort *>(small_smem);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t lt_mask = (1u << lane) - 1u;
    const int rounds = (n + 1023) / 1024, i0 = warp * rounds * 32 + lane;
    double mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int q = threadIdx.x; q < n; q += 1024)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double v = pos_at(pos, stride, sub, q, a);
            mn[a] = fmin(mn[a], v);
            mx[a] = fmax(mx[a], v);
        }
    block_box(mn, mx, sh.part, sh.box);
    if (threadIdx.x == 0) {
        root_of_box(sh.box, n, &sh.g);
        *g = sh.g;
    }
    __syncthreads();
    constexpr int R = kSmallSort / 1024;
    uint64_t k[R];
    uint16_t v[R], rank[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = i0 + r * 32;
        const bool valid = r < rounds && i < n;
        k[r] = valid ? morton_key(pos, stride, sub, i, sh.g) : ~0ull;   // padding: after every valid item
        v[r] = (uint16_t)i;
    }
    for (int pass = 0; pass < kSortPasses; ++pass) {
        const int shift = pass * kSortBits;
        for (int i = threadIdx.x; i < 32 * kSortBins / 2; i += 1024) reinterpret_cast<uint32_t *>(&sh.wcount[0][0])[i] = 0u;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (r >= rounds) break;
            const uint32_t d = (uint32_t)((k[r] >> shift) & (kSortBins - 1u));
            const uint32_t peers = __match_any_sync(0xffffffffu, d), lower = peers & lt_mask;
            const uint16_t pre = sh.wcount[warp][d];
            rank[r] = (uint16_t)(pre + __popc(lower));
            __syncwarp();
            if (lower == 0) sh.wcount[warp][d] = (uint16_t)(pre + __popc(peers));
            __syncwarp();
        }
        __syncthreads();
        // digit totals and their exclusive scan (the padding counts too: it takes the last places)
        uint32_t run = 0, x = 0;
        if (threadIdx.x < kSortBins) {
#pragma unroll 8
            for (int w = 0; w < 32; ++w) {
                const uint16_t t = sh.wcount[w][threadIdx.x];
                sh.wcount[w][threadIdx.x] = (uint16_t)run;
                run += t;
            }
            x = run;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
                if (lane >= d) x += y;
            }
            if (lane == 31) sh.wsum[warp] = x;
        }
        __syncthreads();
        if (threadIdx.x < kSortBins) {
            uint32_t before = 0;
            for (int w = 0; w < warp; ++w) before += sh.wsum[w];
            sh.dstart[threadIdx.x] = before + x - run;
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (r >= rounds) break;
            const uint32_t d = (uint32_t)((k[r] >> shift) & (kSortBins - 1u));
            const uint32_t at = sh.dstart[d] + sh.wcount[warp][d] + rank[r];
            sh.k[at] = k[r];
            sh.v[at] = v[r];
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (r >= rounds) break;
            k[r] = sh.k[i0 + r * 32];
            v[r] = sh.v[i0 + r * 32];
        }
    }
    for (int i = threadIdx.x; i < n; i += 1024) {
        const uint32_t q = sh.v[i];
        keys[i] = sh.k[i];
        vals[i] = q;
        if (o.x) gather_one(i, q, pos, stride, sub, mass, fast, o);
    }
}

// Bytes of the sort's scratch for n particles, and its parts (the first block of it must be zero before the first use).
size_t sort_scratch_bytes(int64_t n)
{
    const size_t tiles = (size_t)((n + kSortTileItems - 1) / kSortTileItems);
    return 256 + sizeof(double) * 6 * kBoxBlocks + sizeof(uint32_t) * (kSortPasses * (kSortBins + 1) + 1) +
           2 * sizeof(uint32_t) * kSortBins * tiles;
}

tg_status ensure_sort_scratch(tg_ctx *c, int64_t n, void **out)
{
    const uint64_t epoch = c->alloc_epoch;
    tg_status st = ensure(c, B_SORT, sort_scratch_bytes(n), out);
    if (st) return st;
    if (epoch == c->alloc_epoch) return TG_OK;
    return cuda_check(c, cudaMemsetAsync(*out, 0, 256, c->stream), "sort scratch");   // a new allocation
}

SortScratch sort_scratch(void *base, int64_t n)
{
    const size_t tiles = (size_t)((n + kSortTileItems - 1) / kSortTileItems);
    char *p = static_cast<char *>(base);
    SortScratch s;
    s.done = reinterpret_cast<uint32_t *>(p);
    s.flag = s.done + 1;
    s.boxes = reinterpret_cast<double *>(p + 256);
    s.state[0] = reinterpret_cast<uint32_t *>(p + 256 + sizeof(double) * 6 * kBoxBlocks);
    s.state[1] = s.state[0] + kSortBins * tiles;
    s.hist = s.state[1] + kSortBins * tiles;
    return s;
}

// Root cube, keys and sort on a stream: the sorted keys and indices end in k0 / v0 when *swapped is false, in k1 / v1
// when it is true.  With o the small sort also gathers (*gathered).  dn: device count (n is then the capacity,
// and the launches of both sizes are issued).  hold: test hook, the tile that publishes nothing (< 0: none).
cudaError_t launch_sort(cudaStream_t st, int n, const int *dn, const double *pos, int64_t stride, const int64_t *sub,
                        const double *mass, const uint8_t *fast, Geom *g, uint64_t *k0, uint64_t *k1, uint32_t *v0,
                        uint32_t *v1, const SortScratch &s, const SortedOut &o, int hold, bool *swapped, bool *gathered, int *launches)
{
    static_assert(kSortPasses % 2 == 1, "an odd number of passes ends in the second pair of buffers");
    *swapped = *gathered = false;
    *launches = 0;
    if (n <= kSmallSort || dn) {
        const int smem = (int)sizeof(SmallSort);
        cudaError_t e = cudaFuncSetAttribute(sort_small, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        const bool swap = n > kSmallSort;   // batched: the same buffers as the passes end in
        sort_small<<<1, 1024, smem, st>>>(pos, stride, sub, n, dn, mass, fast, g, swap ? k1 : k0, swap ? v1 : v0, o);
        *launches = 1;
        if (n <= kSmallSort) {
            *gathered = o.x != nullptr;
            return cudaGetLastError();
        }
    }
    const int nt = (n + kSortTileItems - 1) / kSortTileItems;
    root_cube<<<grid_for(n, kBoxThreads, kBoxBlocks), kBoxThreads, 0, st>>>(pos, stride, sub, n, dn, s, g);
    morton_keys<<<grid_for(n, 256, 152 * 8), 256, 0, st>>>(pos, stride, sub, n, dn, g, k0, v0, s);
    for (int pass = 0; pass < kSortPasses; ++pass) {
        const bool odd = pass & 1;
        (hold < 0 ? radix_pass<false> : radix_pass<true>)<<<nt, kSortThreads, 0, st>>>(
            odd ? k1 : k0, odd ? v1 : v0, odd ? k0 : k1, odd ? v0 : v1, n, dn, pass, s, hold);
    }
    *swapped = true;
    *launches += 2 + kSortPasses;
    return cudaGetLastError();
}

tg_status sort_particles(tg_ctx *c, int n, const double *pos, int64_t stride, const int64_t *sub, const double *mass,
                         const uint8_t *fast, Geom *d_geom, const DevEval *de)
{
    // with de the size lives on the device; n is then the capacity the launches are sized for
    const int *dn = de ? &de->n : nullptr;
    uint64_t *k0, *k1;
    uint32_t *v0, *v1;
    SortedOut o;
    tg_status st;
    void *scratch;
    if ((st = ensure_t(c, B_KEYS0, n, &k0)) || (st = ensure_t(c, B_KEYS1, n, &k1)) ||
        (st = ensure_t(c, B_VALS0, n, &v0)) || (st = ensure_t(c, B_VALS1, n, &v1)) ||
        (st = ensure_sort_scratch(c, n, &scratch)) ||
        (st = ensure_t(c, B_XS, n, &o.x)) || (st = ensure_t(c, B_YS, n, &o.y)) || (st = ensure_t(c, B_ZS, n, &o.z)) ||
        (st = ensure_t(c, B_MS, n, &o.m)) || (st = ensure_t(c, B_FS, n, &o.f)))
        return st;
    bool swapped, gathered;
    int launches = 0;
    cudaError_t e;
    SortScratch s = sort_scratch(scratch, n);
    if (de) s.flag = const_cast<uint32_t *>(&de->overflow);
    {
        ProfScope ps_(c, TG_K_TREE);
        e = launch_sort(c->stream, n, dn, pos, stride, sub, mass, fast, d_geom, k0, k1, v0, v1, s, o,
                        c->debug_sort_hold, &swapped, &gathered, &launches);
        c->prof_launches[TG_K_TREE] += launches - 1;
    }
    if (e != cudaSuccess) return cuda_check(c, e, "keys and sort");
    // the sorted keys and permutation live in the B_KEYS0 / B_VALS0 slots from here on
    if (swapped) {
        std::swap(c->buf[B_KEYS0], c->buf[B_KEYS1]);
        std::swap(c->buf[B_VALS0], c->buf[B_VALS1]);
    }
    if (!gathered) {
        ProfScope ps_(c, TG_K_TREE);
        gather_sorted<<<grid_for(n, 256), 256, 0, c->stream>>>(swapped ? v1 : v0, pos, stride, sub, mass, fast, n, dn,
                                                               s.flag, o);
    }
    return cuda_check(c, cudaGetLastError(), "keys/sort/gather");
}

TreeView tree_view(tg_ctx *c, int n, int ncell)
{
    TreeView t;
    t.n = n;
    t.ncell = ncell;
    t.level = static_cast<const uint8_t *>(c->buf[B_C_LEVEL].p);
    t.cx = static_cast<const uint32_t *>(c->buf[B_C_X].p);
    t.cy = static_cast<const uint32_t *>(c->buf[B_C_Y].p);
    t.cz = static_cast<const uint32_t *>(c->buf[B_C_Z].p);
    t.first = static_cast<const int32_t *>(c->buf[B_C_FIRST].p);
    t.count = static_cast<const int32_t *>(c->buf[B_C_COUNT].p);
    t.child_first = static_cast<const int32_t *>(c->buf[B_C_CHILD].p);
    t.parent = static_cast<const int32_t *>(c->buf[B_C_PARENT].p);
    t.nchild = static_cast<const uint8_t *>(c->buf[B_C_NCHILD].p);
    return t;
}

}  // namespace tg
