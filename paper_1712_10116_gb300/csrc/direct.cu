// direct.cu -- float64 direct summation for a sample of sinks (tg_direct_forces): the sum that force errors
// are measured against.
//
// Bound by the float64 pipe: 14 operations per pair (16 with the potential).  The sinks are few (thousands)
// and the sources many, so the sources are split: a cluster of eight blocks takes a tile of up to 32
// sinks, each block an eighth of the sources, and inside a block 256 / tile groups of threads take every
// (256 / tile)-th source.  The partial sums are added in a fixed order, first in the block and then over the
// cluster's shared memory, so no scratch memory is needed and two runs agree bit for bit.
// 4096 sinks, 100,003 sources, with the potential: 193.3 ms with one thread per sink walking all sources (16 of
// 152 SMs busy, 1/sqrt by the library), 13.7 ms in this form: 4.8e11 float64 operations per second, of the
// 5.27e11 that a loop of independent operations on registers reaches.
#include <cooperative_groups.h>

#include "pair_f64.cuh"
#include "tg_common.cuh"

namespace cg = cooperative_groups;

namespace tg {

constexpr int kDirThreads = 256, kDirCluster = 8;

struct __align__(16) Src4 {
    double x, y, z, w;
};

template <int KERNEL, bool POT>
__global__ void __cluster_dims__(kDirCluster, 1, 1) __launch_bounds__(kDirThreads)
    direct_sum(int64_t n, const double *__restrict__ pos, const double *__restrict__ mass,
               const uint8_t *__restrict__ fast, int64_t n_sink, const int64_t *__restrict__ sink_idx, double eps,
               double *acc, double *pot, int log2_tile)
{
    __shared__ Src4 src[kDirThreads];
    __shared__ uint8_t sf[kDirThreads];
    __shared__ double part[4][kDirThreads];
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int tile = 1 << log2_tile, nslice = kDirThreads >> log2_tile;
    const int slot = threadIdx.x & (tile - 1), slice = threadIdx.x >> log2_tile;
    const int64_t t = ((int64_t)(blockIdx.x / kDirCluster) << log2_tile) + slot;
    const bool active = t < n_sink;
    const int64_t i = active ? (sink_idx ? sink_idx[t] : t) : 0;
    const double xi = active ? pos[i] : 0.0, yi = active ? pos[n + i] : 0.0, zi = active ? pos[2 * n + i] : 0.0;
    const bool fi = active && fast && fast[i];
    PairF64 k;
    k.init(eps, KERNEL == TG_KERNEL_PLUMMER);
    double ax = 0, ay = 0, az = 0, ph = 0;
    const int64_t jb = n * rank / kDirCluster, je = n * (rank + 1) / kDirCluster;
    for (int64_t j0 = jb; j0 < je; j0 += kDirThreads) {
        const int64_t j = j0 + threadIdx.x;
        __syncthreads();
        if (j < je) {
            src[threadIdx.x] = Src4{pos[j], pos[n + j], pos[2 * n + j], mass[j]};
            sf[threadIdx.x] = fast ? fast[j] : 0;
        }
        __syncthreads();
        const int cnt = (int)(je - j0 < kDirThreads ? je - j0 : kDirThreads);
        if (active) {
            for (int q = slice; q < cnt; q += nslice) {
                const Src4 s = src[q];
                // the sink itself and fast-fast pairs are left out
                if (j0 + q == i || (fi && sf[q])) continue;
                const double dx = s.x - xi, dy = s.y - yi, dz = s.z - zi;
                double g, ri;
                pair_f64<KERNEL, POT>(pair_s2<KERNEL>(dx, dy, dz, k), k, g, ri);
                const double mg = s.w * g;
                ax = fma(mg, dx, ax);
                ay = fma(mg, dy, ay);
                az = fma(mg, dz, az);
                if (POT) ph = fma(-s.w, ri, ph);
            }
        }
    }
    part[0][threadIdx.x] = ax;
    part[1][threadIdx.x] = ay;
    part[2][threadIdx.x] = az;
    part[3][threadIdx.x] = ph;
    __syncthreads();
    // the block's sums: thread (component, sink) adds the slices in order
    constexpr int NC = POT ? 4 : 3;
    double mine = 0.0;
    const int comp = threadIdx.x >> log2_tile;   // for the first NC * tile threads
    if (threadIdx.x < NC * tile)
        for (int s = 0; s < nslice; ++s) mine += part[comp][(s << log2_tile) + slot];
    __syncthreads();
    if (threadIdx.x < NC * tile) part[comp][slot] = mine;
    cluster.sync();
    if (rank == 0 && threadIdx.x < NC * tile && active) {
        double sum = 0.0;
        for (int r = 0; r < kDirCluster; ++r) sum += cluster.map_shared_rank(&part[comp][slot], r)[0];
        if (comp < 3) acc[comp * n_sink + t] = sum;
        else pot[t] = sum;
    }
    cluster.sync();   // the other blocks' shared memory stays until it has been read
}

tg_status direct_eval(tg_ctx *c, int64_t n, const double *pos, const double *mass, const uint8_t *fast,
                      int64_t n_sink, const int64_t *sink_idx, double *acc, double *pot)
{
    if (n_sink <= 0) return TG_OK;
    // the widest tile that still gives every SM a few blocks: fewer sinks per tile re-read the sources more
    // often, which the float64 pipe hides
    int log2_tile = 5;
    while (log2_tile > 2 && ((n_sink + (1 << log2_tile) - 1) >> log2_tile) * kDirCluster < 4 * c->num_sms) --log2_tile;
    const int64_t tiles = (n_sink + (1 << log2_tile) - 1) >> log2_tile;
    if (tiles > INT32_MAX / kDirCluster) return set_err(c, TG_ERR_ARG, "direct summation: too many sinks");
    const int grid = (int)tiles * kDirCluster;
    {
        ProfScope ps_(c, TG_K_OTHER);
#define TG_DIRECT(K, PT) \
    direct_sum<K, PT><<<grid, kDirThreads, 0, c->stream>>>(n, pos, mass, fast, n_sink, sink_idx, c->prm.eps, acc, pot, log2_tile)
        if (c->prm.kernel == TG_KERNEL_PLUMMER) {
            if (pot) TG_DIRECT(TG_KERNEL_PLUMMER, true);
            else TG_DIRECT(TG_KERNEL_PLUMMER, false);
        } else {
            if (pot) TG_DIRECT(TG_KERNEL_WENDLAND_C2, true);
            else TG_DIRECT(TG_KERNEL_WENDLAND_C2, false);
        }
#undef TG_DIRECT
    }
    return cuda_check(c, cudaGetLastError(), "direct summation");
}

}  // namespace tg
