// sbh_noalloc.cu -- sbh_morton_sort_noalloc: the Morton ordering step of the tree build for
// callers that cannot allocate device memory.
//
// Some callers cannot call cudaMalloc or any allocating routine: real-time loops where the
// implicit synchronisation of an allocation is not acceptable, and host applications that hand a
// library a fixed device-memory budget up front and own every allocation themselves. For them
// this entry point orders points exactly as sbh_build does (same codes, same stable order) using
// only the caller's input and output buffers plus one scratch array of fixed size that lives in
// this library's static device memory.
//
// The scratch array is a file-scope __device__ array; every GPU that loads the library holds it
// until the process exits. Host code cannot use the array's name as a device address, so every
// call looks up its address with cudaGetSymbolAddress in the current device's context (a lookup,
// no allocation). The address is not cached: it belongs to the context it was taken in, and a
// cudaDeviceReset or another context on the same device would leave a cached one stale. The first
// call on a device also loads this module's device code there.
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>

#include "sbh.h"
#include "sbh_build.cuh"
#include "sbh_sort.cuh"

namespace sbh {

namespace {

constexpr int64_t kNoAllocMaxPoints = SBH_NOALLOC_MAX_POINTS;
constexpr int kNoAllocMaxTiles = (int)((kNoAllocMaxPoints + kSortTile - 1) / kSortTile);

constexpr size_t round256(size_t x) { return (x + 255) & ~(size_t)255; }

// layout of the scratch array
constexpr size_t kOffKeys = 0;                                                          // u64 [max]
constexpr size_t kOffVals = kOffKeys + round256(sizeof(uint64_t) * kNoAllocMaxPoints);  // i32 [max]
constexpr size_t kOffStatus = kOffVals + round256(sizeof(int32_t) * kNoAllocMaxPoints); // u32 [2][tiles][256]
constexpr size_t kOffHead = kOffStatus + round256(2 * 256 * sizeof(uint32_t) * kNoAllocMaxTiles);
constexpr size_t kOffCtrl = kOffHead + round256(sizeof(SortHead));                      // TreeCtrl [2]
constexpr size_t kScratchBytes = kOffCtrl + round256(2 * sizeof(TreeCtrl));

static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

}  // namespace

}  // namespace sbh

extern "C" {

sbh_status sbh_morton_sort_noalloc(const float* points, int64_t n, uint64_t* codes, int32_t* perm, void* stream)
{
    using namespace sbh;
    set_error_message("");
    if (n < 1 || n > kNoAllocMaxPoints) {
        set_error_message("sbh_morton_sort_noalloc: n = %lld outside [1, %lld] (SBH_NOALLOC_MAX_POINTS)", (long long)n,
                          (long long)kNoAllocMaxPoints);
        return SBH_EINVAL;
    }
    if (!points || !codes || !perm) {
        set_error_message("sbh_morton_sort_noalloc: points, codes and perm must be non-NULL");
        return SBH_EINVAL;
    }
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) {
        set_error_message("sbh_morton_sort_noalloc: cudaGetSymbolAddress failed: %s", cudaGetErrorString(e));
        return SBH_ECUDA;
    }
    unsigned char* base = (unsigned char*)p;
    cudaStream_t s = (cudaStream_t)stream;
    TreeCtrl* ctrl = (TreeCtrl*)(base + kOffCtrl);
    // the sort goes back and forth between the caller's outputs and the scratch copy and ends in the
    // outputs. The count of bad weights is not used here; the points array stands in for the weights
    // (it has 3n floats, so the n reads stay inside it). There is no status to return later: a sort whose
    // bounded wait gave up says so in perm[0].
    uint64_t* const k[2] = {codes, (uint64_t*)(base + kOffKeys)};
    int32_t* const v[2] = {perm, (int32_t*)(base + kOffVals)};
    e = sort_codes(points, points, n, k, v, (SortHead*)(base + kOffHead), (uint32_t*)(base + kOffStatus), ctrl,
                   ctrl + 1, perm, s);
    if (e != cudaSuccess) {
        set_error_message("sbh_morton_sort_noalloc: kernel launch failed: %s", cudaGetErrorString(e));
        return SBH_ECUDA;
    }
    return SBH_OK;
}

}  // extern "C"
