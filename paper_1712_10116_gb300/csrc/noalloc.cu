// noalloc.cu -- tg_morton_sort_noalloc: root cube, Morton keys and the stable radix sort for
// callers that cannot allocate device memory.
//
// Some callers must not call cudaMalloc: applications whose device memory is owned by another
// allocator (a framework's pool, a fixed memory budget that raw allocations would break) and
// loops that cannot afford the device-wide synchronisation an allocation can cause.  This entry
// point takes the caller's input and output buffers and keeps all of its scratch in one
// file-scope device array of fixed size, so it never allocates.
//
// The array lives in every GPU that loads the library until the process exits.  Host code must
// not use the array's name as a pointer: on the host it is only a stand-in for the device
// symbol.  Every call looks the device address up with cudaGetSymbolAddress, with the caller's
// device current (a cheap query that allocates nothing), so no address outlives a device reset.
#include "tg_common.cuh"

namespace {

using namespace tg;

constexpr int64_t kMaxN = TG_NOALLOC_MAX_N;
constexpr size_t kMaxSortTiles = (size_t)((kMaxN + kSortTileItems - 1) / kSortTileItems);

// byte layout of the scratch array (every part 256-byte aligned)
constexpr size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }
constexpr size_t kOffGeom = 0;
constexpr size_t kOffKeys0 = align256(kOffGeom + sizeof(Geom));
constexpr size_t kOffKeys1 = align256(kOffKeys0 + sizeof(uint64_t) * kMaxN);
constexpr size_t kOffVals0 = align256(kOffKeys1 + sizeof(uint64_t) * kMaxN);
constexpr size_t kOffVals1 = align256(kOffVals0 + sizeof(uint32_t) * kMaxN);
constexpr size_t kOffSort = align256(kOffVals1 + sizeof(uint32_t) * kMaxN);
// the parts that sort_scratch lays out (its size is checked against this on every call)
constexpr size_t kSortBytes = 256 + sizeof(double) * 6 * kBoxBlocks + sizeof(uint32_t) * (kSortPasses * (kSortBins + 1) + 1) +
                              2 * sizeof(uint32_t) * kSortBins * kMaxSortTiles;
constexpr size_t kScratchBytes = align256(kOffSort + kSortBytes);
static_assert(kScratchBytes < (8u << 20), "the allocation-free scratch must stay modest (< 8 MB)");

// The scratch.  Device code could name it directly; host code uses the looked-up address.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

// Address of the scratch on the current device.  Looked up on every call: the query is cheap,
// allocates nothing, and stays right after a device reset reloads the module.
tg_status scratch_for_current_device(unsigned char **out)
{
    void *p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || p == nullptr) {
        cudaGetLastError();
        return TG_ERR_CUDA;
    }
    *out = static_cast<unsigned char *>(p);
    return TG_OK;
}

// The call returns before the sort has run, so a sort whose bounded wait gave up cannot become a status: its
// permutation is all -1 instead.
__global__ void noalloc_export(int n, const uint64_t *keys, const uint32_t *vals, const uint32_t *flag, uint64_t *keys_out,
                               int64_t *perm_out)
{
    const bool bad = *flag != 0;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
        keys_out[s] = keys[s];
        perm_out[s] = bad ? -1 : (int64_t)vals[s];
    }
}

// device memory of the current device (managed memory is reachable from any device)
int check_dev(const void *p)
{
    cudaPointerAttributes a;
    int dev = -1;
    if (!p || cudaPointerGetAttributes(&a, p) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    if (a.type == cudaMemoryTypeManaged) return 1;
    return a.type == cudaMemoryTypeDevice && a.device == dev;
}

}  // namespace

static tg_status morton_sort(int64_t n, const double *pos, uint64_t *keys_out, int64_t *perm_out, void *cuda_stream, int hold)
{
    if (n < 0 || n > kMaxN) return TG_ERR_ARG;
    if (n == 0) return TG_OK;
    if (!check_dev(pos) || !check_dev(keys_out) || !check_dev(perm_out)) return TG_ERR_ARG;
    unsigned char *base = nullptr;
    tg_status st = scratch_for_current_device(&base);
    if (st) return st;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    Geom *geom = reinterpret_cast<Geom *>(base + kOffGeom);
    uint64_t *k0 = reinterpret_cast<uint64_t *>(base + kOffKeys0), *k1 = reinterpret_cast<uint64_t *>(base + kOffKeys1);
    uint32_t *v0 = reinterpret_cast<uint32_t *>(base + kOffVals0), *v1 = reinterpret_cast<uint32_t *>(base + kOffVals1);
    const int ni = (int)n;
    if (sort_scratch_bytes(n) > kSortBytes) return TG_ERR_ARG;
    // the sort's first block starts out zero (calls that overlapped may have left it otherwise); every other word is
    // written before it is read
    if (cudaMemsetAsync(base + kOffSort, 0, 256, s) != cudaSuccess) return TG_ERR_CUDA;
    bool swapped, gathered;
    int launches;
    const SortScratch ss = sort_scratch(base + kOffSort, n);
    if (launch_sort(s, ni, nullptr, pos, n, nullptr, nullptr, nullptr, geom, k0, k1, v0, v1, ss, SortedOut{},
                    hold, &swapped, &gathered, &launches) != cudaSuccess)
        return TG_ERR_CUDA;
    noalloc_export<<<grid_for(n, 256), 256, 0, s>>>(ni, swapped ? k1 : k0, swapped ? v1 : v0, ss.flag, keys_out, perm_out);
    if (cudaGetLastError() != cudaSuccess) return TG_ERR_CUDA;
    return TG_OK;
}

extern "C" tg_status tg_morton_sort_noalloc(int64_t n, const double *pos, uint64_t *keys_out, int64_t *perm_out,
                                            void *cuda_stream)
{
    return morton_sort(n, pos, keys_out, perm_out, cuda_stream, -1);
}

extern "C" tg_status tg_debug_morton_sort_noalloc(int64_t n, const double *pos, uint64_t *keys_out, int64_t *perm_out,
                                                  void *cuda_stream, int hold_tile)
{
    return morton_sort(n, pos, keys_out, perm_out, cuda_stream, hold_tile < 0 ? -1 : hold_tile);
}
