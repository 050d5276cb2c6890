// sbh_build.cu -- GPU construction of the octree-like tree of Sec. 3.1 (Madan et al. 2025).
//
// The paper builds its tree on the CPU (Sec. 4.1); here every stage is a CUDA kernel:
//   1. bounds + validation   per-axis min/max of the points (the root cube), counts of NaN/Inf
//                            coordinates and of non-positive weights
//   2. Morton codes          20-bit FP32 quantisation per axis, interleaved to 60 bits
//   3. stable LSD radix sort (code, index), 8 passes of 8 bits, one kernel each (one for all up to a tile)
//   4. gather                points, weights and normals into Morton order
//   5. topology              a node whose points span several cells one level down has those runs
//                            as children; a run that stays inside one cell collapses into its
//                            deepest split; a run of <= leaf_size points (or at the deepest level)
//                            is a leaf whose children are its points
//   6. aggregates            FP64 bottom-up sums of m, m p, m n per node, FP32 records, the children's
//                            prefix mass fractions and the child pick's guide table
//
// Node ids are generation-major (breadth-first): every node's children are contiguous, in
// Morton order, and the top generations that every query reads sit at the front of each array.
#include <cuda_runtime.h>

#include <mutex>
#include <unordered_map>
#include <stdint.h>

#include "sbh_build.cuh"
#include "sbh_sort.cuh"

namespace sbh {

namespace {
constexpr int kThreads = 256;
constexpr int kMortonThreads = 1024;
// blocks for n items, at most 16 per SM of the current device (grid-stride loops do the rest)
inline unsigned grid_for(int64_t n, int per_block = kThreads, unsigned cap = 0)
{
    if (cap == 0) cap = 16u * (unsigned)device_sm_count();
    int64_t g = (n + per_block - 1) / per_block;
    if (g < 1) g = 1;
    return (unsigned)(g > cap ? cap : g);
}
}  // namespace

// ----------------------------------------------------------------------------------------------
// device memory: the library's stream-ordered pool, or the caller's allocator; an optional cap on
// the bytes the library holds at once (allocations beyond it fail as out of memory)
// ----------------------------------------------------------------------------------------------
namespace {
struct Block {
    size_t bytes;
    sbh_free_fn free_fn;  // nullptr: the library's pool
    void* ctx;
};
std::mutex g_mem_mutex;
cudaMemPool_t g_pool[64];
bool g_pool_ready[64];
sbh_alloc_fn g_alloc_fn = nullptr;
sbh_free_fn g_free_fn = nullptr;
void* g_alloc_ctx = nullptr;
uint64_t g_limit = 0;
uint64_t g_in_use = 0;
std::unordered_map<void*, Block> g_blocks;
}  // namespace

cudaError_t dalloc(void** p, size_t bytes, cudaStream_t s)
{
    *p = nullptr;
    if (bytes == 0) bytes = 16;
    std::lock_guard<std::mutex> lock(g_mem_mutex);
    if (g_limit && g_in_use + bytes > g_limit) return cudaErrorMemoryAllocation;
    if (g_alloc_fn) {
        void* q = g_alloc_fn(bytes, (void*)s, g_alloc_ctx);
        if (!q) return cudaErrorMemoryAllocation;
        if (((uintptr_t)q & 255u) != 0) {  // misaligned: hand it back and fail
            g_free_fn(q, (void*)s, g_alloc_ctx);
            return cudaErrorMisalignedAddress;
        }
        *p = q;
        g_blocks[q] = Block{bytes, g_free_fn, g_alloc_ctx};
        g_in_use += bytes;
        return cudaSuccess;
    }
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!g_pool_ready[dev]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        e = cudaMemPoolCreate(&g_pool[dev], &props);
        if (e != cudaSuccess) return e;
        uint64_t keep = UINT64_MAX;  // keep freed blocks for reuse by later builds
        cudaMemPoolSetAttribute(g_pool[dev], cudaMemPoolAttrReleaseThreshold, &keep);
        g_pool_ready[dev] = true;
    }
    e = cudaMallocFromPoolAsync(p, bytes, g_pool[dev], s);
    if (e != cudaSuccess) return e;
    g_blocks[*p] = Block{bytes, nullptr, nullptr};
    g_in_use += bytes;
    return cudaSuccess;
}

void dfree(void* p, cudaStream_t s)
{
    if (!p) return;
    Block b{0, nullptr, nullptr};
    {
        std::lock_guard<std::mutex> lock(g_mem_mutex);
        auto it = g_blocks.find(p);
        if (it != g_blocks.end()) {
            b = it->second;
            g_in_use -= b.bytes;
            g_blocks.erase(it);
        }
    }
    if (b.free_fn) b.free_fn(p, (void*)s, b.ctx);
    else cudaFreeAsync(p, s);
}

void set_allocator(sbh_alloc_fn a, sbh_free_fn f, void* ctx)
{
    std::lock_guard<std::mutex> lock(g_mem_mutex);
    g_alloc_fn = a;
    g_free_fn = f;
    g_alloc_ctx = ctx;
}

void set_memory_limit(uint64_t bytes)
{
    std::lock_guard<std::mutex> lock(g_mem_mutex);
    g_limit = bytes;
}

uint64_t memory_in_use()
{
    std::lock_guard<std::mutex> lock(g_mem_mutex);
    return g_in_use;
}

// ----------------------------------------------------------------------------------------------
// 1. bounds and validation
// ----------------------------------------------------------------------------------------------
__device__ __forceinline__ int ordered_int(float f)
{
    const int i = __float_as_int(f);
    return i >= 0 ? i : (i ^ 0x7FFFFFFF);
}
__device__ __forceinline__ float from_ordered(int i) { return __int_as_float(i >= 0 ? i : (i ^ 0x7FFFFFFF)); }

// The float order as unsigned integers, so that a maximum taken by atomicMax can start from zero
__device__ __forceinline__ uint32_t ordered_uint(float f) { return (uint32_t)ordered_int(f) ^ 0x80000000u; }
__device__ __forceinline__ float from_ordered_uint(uint32_t u) { return from_ordered((int)(u ^ 0x80000000u)); }

// Whether the calling block is the last of the grid to come here (every thread gets the answer):
// what the other blocks wrote before is then visible to it. *done starts at zero.
__device__ __forceinline__ bool last_block(unsigned* done)
{
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// Per-axis extremes and the counts of bad inputs, then (the last block) the root cube: lo = per-axis
// min, side = largest extent (1 if every point coincides), and the cell diagonal table |B|(level) =
// sqrt(3) * side * 2^-(shift * level) for each branching
__global__ void __launch_bounds__(kThreads) k_bounds(const float* __restrict__ pts, const float* __restrict__ w,
                                                     int64_t n, SortHead* __restrict__ H, TreeCtrl* c4, TreeCtrl* c2)
{
    uint32_t mx[6] = {0, 0, 0, 0, 0, 0};  // of the negated order (the minima), of the order
    int bad_p = 0, bad_w = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float v = pts[3 * i + a];
            if (!isfinite(v)) { ++bad_p; continue; }
            const uint32_t o = ordered_uint(v);
            mx[a] = max(mx[a], ~o);
            mx[3 + a] = max(mx[3 + a], o);
        }
        const float m = w[i];
        if (!(m > 0.0f) || !isfinite(m)) ++bad_w;
    }
    // across the warp, then across the block's warps, so that each block adds one set of atomics
    __shared__ uint32_t s_red[kThreads / 32][8];
    const int warp = threadIdx.x >> 5;
    uint32_t r[8];
#pragma unroll
    for (int a = 0; a < 6; ++a) r[a] = __reduce_max_sync(0xFFFFFFFFu, mx[a]);
    r[6] = __reduce_add_sync(0xFFFFFFFFu, (unsigned)bad_p);
    r[7] = __reduce_add_sync(0xFFFFFFFFu, (unsigned)bad_w);
    if ((threadIdx.x & 31) < 8) {
#pragma unroll
        for (int a = 0; a < 8; ++a)
            if ((int)(threadIdx.x & 31) == a) s_red[warp][a] = r[a];
    }
    __syncthreads();
    if (threadIdx.x < 8) {
        uint32_t t = s_red[0][threadIdx.x];
        for (int k = 1; k < (int)(blockDim.x >> 5); ++k)
            t = threadIdx.x < 6 ? max(t, s_red[k][threadIdx.x]) : t + s_red[k][threadIdx.x];
        if (threadIdx.x < 6) atomicMax(&H->bounds[threadIdx.x], t);
        else if (t) atomicAdd(&H->bounds[threadIdx.x], t);
    }
    if (!last_block(&H->done[0])) return;
    float lo[3], side = 0.0f;
    for (int a = 0; a < 3; ++a) {
        lo[a] = from_ordered_uint(~__ldcg(&H->bounds[a]));
        const float ext = __fsub_rn(from_ordered_uint(__ldcg(&H->bounds[3 + a])), lo[a]);
        side = ext > side ? ext : side;
    }
    if (side == 0.0f) side = 1.0f;
    const float diam0 = __fmul_rn(1.7320508075688772f, side);
    if (threadIdx.x < kDiamLevels) {
        c4->diam[threadIdx.x] = ldexpf(diam0, -2 * (int)threadIdx.x);
        c2->diam[threadIdx.x] = ldexpf(diam0, -(int)threadIdx.x);
    }
    if (threadIdx.x == 0) {
        for (int a = 0; a < 3; ++a) { c4->lo[a] = lo[a]; c2->lo[a] = lo[a]; }
        c4->side = side;
        c2->side = side;
        c4->bad_points = (int32_t)__ldcg(&H->bounds[6]);
        c4->bad_weights = (int32_t)__ldcg(&H->bounds[7]);
        c4->error = c4->bad_points || c4->bad_weights ? kErrorInput : 0;
        c2->error = 0;
    }
}

// ----------------------------------------------------------------------------------------------
// 2. Morton codes: c = min(2^20 - 1, floor((x - lo) * (2^20 / side))), FP32 with one rounding
//    per operation; bits interleaved x, y, z from the most significant bit down.
// ----------------------------------------------------------------------------------------------
__device__ __forceinline__ uint64_t spread3(uint32_t v)
{
    uint64_t x = v & 0x1FFFFFu;
    x = (x | (x << 32)) & 0x001F00000000FFFFull;
    x = (x | (x << 16)) & 0x001F0000FF0000FFull;
    x = (x | (x << 8)) & 0x100F00F00F00F00Full;
    x = (x | (x << 4)) & 0x10C30C30C30C30C3ull;
    x = (x | (x << 2)) & 0x1249249249249249ull;
    return x;
}

__device__ __forceinline__ uint32_t quantise(float x, float lo, float scale)
{
    const float t = __fmul_rn(__fsub_rn(x, lo), scale);
    const float f = floorf(t);
    const uint32_t c = f <= 0.0f ? 0u : (uint32_t)f;
    return c > 1048575u ? 1048575u : c;
}

// The codes, and the histogram of each of their eight digits: counted per block in shared memory, added
// up, and made exclusive sums (where each digit's run starts in its pass) by the last block. Lanes
// that share a digit add once together in the top one, which has 16 values. PASSES = kQueryPasses: the
// codes of queries, eight bits an axis over the cube of twice the side around the root cube (queries
// further out are taken as on its border).
template <int PASSES>
__global__ void __launch_bounds__(kMortonThreads) k_morton(const float* __restrict__ pts, int64_t n,
                                                           const TreeCtrl* __restrict__ c4, uint64_t* __restrict__ code,
                                                           SortHead* __restrict__ H)
{
    __shared__ int s_hist[PASSES][256];
    for (int k = threadIdx.x; k < PASSES * 256; k += blockDim.x) (&s_hist[0][0])[k] = 0;
    __syncthreads();
    constexpr bool kQuery = PASSES == kQueryPasses;
    const float out = kQuery ? 0.5f * c4->side : 0.0f;
    const float lx = c4->lo[0] - out, ly = c4->lo[1] - out, lz = c4->lo[2] - out;
    const float scale = __fdiv_rn(kQuery ? 128.0f : 1048576.0f, c4->side);
    constexpr uint32_t kTop = kQuery ? 255u : 1048575u;
    for (int64_t b = blockIdx.x * (int64_t)blockDim.x; b < n; b += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = b + threadIdx.x;
        const unsigned live = __ballot_sync(0xFFFFFFFFu, i < n);
        if (i >= n) continue;
        const uint32_t cx = min(quantise(pts[3 * i], lx, scale), kTop);
        const uint32_t cy = min(quantise(pts[3 * i + 1], ly, scale), kTop);
        const uint32_t cz = min(quantise(pts[3 * i + 2], lz, scale), kTop);
        const uint64_t c = (spread3(cx) << 2) | (spread3(cy) << 1) | spread3(cz);
        code[i] = c;
#pragma unroll
        for (int p = 0; p < PASSES; ++p) {
            const int d = (int)(c >> (8 * p)) & 0xFF;
            if (p < PASSES - 1) {
                atomicAdd(&s_hist[p][d], 1);
            } else {
                const unsigned peers = __match_any_sync(live, d);
                if ((threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&s_hist[p][d], __popc(peers));
            }
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < PASSES * 256; k += blockDim.x) {
        const int v = (&s_hist[0][0])[k];
        if (v) atomicAdd(&H->hist[0][0] + k, v);
    }
    if (!last_block(&H->done[1])) return;
    const int p = threadIdx.x >> 5, lane = threadIdx.x & 31;  // a warp to a digit, eight values to a lane
    if (p >= PASSES) return;
    int v[8], sum = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) { v[k] = __ldcg(&H->hist[p][8 * lane + k]); sum += v[k]; }
    int x = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xFFFFFFFFu, x, off);
        if (lane >= off) x += y;
    }
    x -= sum;
#pragma unroll
    for (int k = 0; k < 8; ++k) { H->hist[p][8 * lane + k] = x; x += v[k]; }
}

// ----------------------------------------------------------------------------------------------
// 3. stable LSD radix sort of (code, index) pairs, 8-bit digits, one kernel per pass: each tile
//    ranks its keys by digit (warp by warp, lanes of equal digit found by a match, so the order is
//    kept), learns from the tiles before it how many keys of each digit they hold, and writes its keys
//    in runs. The tiles' counts pass along by decoupled look-back (Merrill and Garland, "Single-pass
//    Parallel Prefix Scan with Decoupled Look-back", 2016; as a sort: Adinets and Merrill,
//    "Onesweep", 2022): a status word per (tile, digit) says nothing yet, the tile's own count, or
//    the count of it and all before it. A tile number is drawn when a block starts, so every tile
//    waited for is already running; each wait is bounded all the same. One that runs out sets H->error
//    and hands on what it has: keys may then be missing from the sorted arrays and their places hold
//    what was in memory before, which nothing may use as an index. k_gather leaves the points in the
//    caller's order and sets the tree's error, no records are made, and sbh_build returns SBH_ETIMEOUT;
//    the walk drops the order of its queries; sbh_morton_sort_noalloc marks its output (`report`).
//    What bounds it: the latency of a tile's steps (load, rank, look back, write) with two blocks of
//    512 threads to an SM; the 24 bytes a key moves take a quarter of the time. It replaces a count, a
//    scan of up to three kernels and a scatter that sorted its tile by nine one-bit splits: 40 kernels
//    and 650 us for 2^22 keys, now 8 and 307 us (2^20: 230 -> 106 us), and the histograms of all
//    digits come with the codes.
// ----------------------------------------------------------------------------------------------
constexpr uint32_t kStatusOwn = 1u << 30, kStatusAll = 2u << 30, kStatusMask = (1u << 30) - 1;
#ifndef SBH_SPIN_LIMIT
#define SBH_SPIN_LIMIT (1 << 22)
#endif
constexpr int kSpinLimit = SBH_SPIN_LIMIT;  // polls before a wait gives up (seconds); below 0: all do, at once (for tests)
constexpr int kLook = 4;             // status words a digit's thread has in flight

// The lanes of the warp whose 8-bit digit equals the caller's, by one ballot per bit: about 40 cycles
// whatever the digits are. (A match instruction takes 9 cycles where few digits occur, but grows with
// their number: a pass over 2^22 keys took 60 us with it where the digits are random.)
__device__ __forceinline__ unsigned same_digit(int d)
{
    unsigned peers = 0xFFFFFFFFu;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const bool on = (d >> b) & 1;
        const unsigned m = __ballot_sync(0xFFFFFFFFu, on);
        peers &= on ? m : ~m;
    }
    return peers;
}

// REPORT (of the last pass): *report = -1 if a wait of any pass gave up
template <bool REPORT>
__global__ void __launch_bounds__(kSortThreads, REPORT ? 1 : 2) k_radix_pass(const uint64_t* __restrict__ kin,
                                                             const int32_t* __restrict__ vin, int64_t n, int pass,
                                                             SortHead* __restrict__ H, uint32_t* status,
                                                             uint32_t* __restrict__ next_status,
                                                             uint64_t* __restrict__ kout, int32_t* __restrict__ vout,
                                                             int32_t* report)
{
    constexpr int ITEMS = kSortItems, kTile = kSortTile, kWarps = kSortThreads / 32;
    extern __shared__ __align__(16) unsigned char s_sort[];
    uint64_t* s_key = reinterpret_cast<uint64_t*>(s_sort);
    int32_t* s_val = reinterpret_cast<int32_t*>(s_key + kTile);
    uint16_t(*s_cnt)[256] = reinterpret_cast<uint16_t(*)[256]>(s_val + kTile);  // per warp and digit
    __shared__ int s_start[256];   // first place of a digit in the sorted tile
    __shared__ int s_out[256];     // where that place goes, minus it
    __shared__ int s_warp[kWarps];
    __shared__ int s_tile;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (t == 0) s_tile = (int)atomicAdd(&H->next_tile[pass], 1u);
    for (int k = t; k < kWarps * 128; k += kSortThreads) reinterpret_cast<uint32_t*>(s_cnt)[k] = 0u;
    __syncthreads();
    const int tile = s_tile;
    const int64_t base = (int64_t)tile * kTile;
    const int count = (n - base) < kTile ? (int)(n - base) : kTile;
    const int shift = 8 * pass;
    // a warp takes consecutive keys; what lies past the end ranks behind every key (digit 255, last)
    uint64_t key[ITEMS];
    const int w0 = warp * 32 * ITEMS + lane;
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) key[k] = w0 + 32 * k < count ? kin[base + w0 + 32 * k] : ~0ull;
    if (t < 256) next_status[(int64_t)tile * 256 + t] = 0u;  // the next pass's words (read last in the pass before)
    // a key's rank among the warp's keys of its digit; keys of equal digit in a row of 32 find each other
    uint32_t rank[ITEMS / 2];  // two 16-bit ranks to a word
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const int d = (int)(key[k] >> shift) & 0xFF;
        const unsigned peers = same_digit(d);
        const uint32_t r = s_cnt[warp][d] + __popc(peers & ((1u << lane) - 1u));
        __syncwarp();
        if (lane == 31 - __clz(peers)) s_cnt[warp][d] = (uint16_t)(r + 1u);
        __syncwarp();
        if (k & 1) rank[k / 2] |= r << 16;
        else rank[k / 2] = r;
    }
    __syncthreads();
    // thread t < 256: digit t
    volatile uint32_t* st = status;
    int own = 0, real = 0;
    if (t < 256) {
#pragma unroll
        for (int k = 0; k < kWarps; ++k) { const int c = s_cnt[k][t]; s_cnt[k][t] = (uint16_t)own; own += c; }
        real = t == 255 ? own - (kTile - count) : own;
        st[(int64_t)tile * 256 + t] = (tile == 0 ? kStatusAll : kStatusOwn) | (uint32_t)real;
    }
    int x = own;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xFFFFFFFFu, x, off);
        if (lane >= off) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    if (t < 256) {
        int add = x - own;
#pragma unroll
        for (int k = 0; k < 7; ++k) add += k < warp ? s_warp[k] : 0;
        s_start[t] = add;
    }
    __syncthreads();
    // into digit order in shared memory, while the first status words come in
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const int i = w0 + 32 * k;
        const int d = (int)(key[k] >> shift) & 0xFF;
        const int at = s_start[d] + s_cnt[warp][d] + (int)((rank[k / 2] >> (16 * (k & 1))) & 0xFFFFu);
        s_key[at] = key[k];
        s_val[at] = i < count ? (vin ? vin[base + i] : (int32_t)(base + i)) : 0;
    }
    // look back, kLook tiles at a time
    uint32_t before = 0;
    if (tile > 0 && t < 256) {
        int spin = 0;
        for (int p = tile - 1; p >= 0;) {
            if (kSpinLimit < 0) { H->error = 1; break; }
            uint32_t v[kLook];
#pragma unroll
            for (int k = 0; k < kLook; ++k) v[k] = p - k >= 0 ? st[(int64_t)(p - k) * 256 + t] : (uint32_t)kStatusAll;
            bool wait = false;
#pragma unroll
            for (int k = 0; k < kLook; ++k) {
                if (p < 0 || wait) continue;
                if (v[k] == 0u) { wait = true; continue; }
                before += v[k] & kStatusMask;
                p = (v[k] & kStatusAll) ? -1 : p;
            }
            if (p >= 0) {
                // how many of the words were there: step over them
                int got = 0;
#pragma unroll
                for (int k = 0; k < kLook; ++k) got += (got == k && v[k] != 0u) ? 1 : 0;
                p -= got;
                if (got == 0 && ++spin > kSpinLimit) { H->error = 1; break; }
            }
        }
        st[(int64_t)tile * 256 + t] = kStatusAll | ((before + (uint32_t)real) & kStatusMask);
    }
    if (t < 256) s_out[t] = H->hist[pass][t] + (int)before - s_start[t];
    __syncthreads();
    for (int i = t; i < count; i += kSortThreads) {
        const uint64_t k = s_key[i];
        const uint32_t dst = (uint32_t)(s_out[(int)(k >> shift) & 0xFF] + i);
        if (dst < (uint32_t)n) {  // always, unless a wait gave up
            kout[dst] = k;
            vout[dst] = s_val[i];
        }
    }
    if constexpr (REPORT) {
        if (last_block(&H->done[2]) && t == 0 && *(volatile int32_t*)&H->error) *report = -1;
    }
}

// All passes of a sort that is one tile, in shared memory: k_radix_pass's ranking, without the other
// tiles, the histograms and the way through global memory. 4,096 keys: 8 kernels and 53 us -> 30 us.
constexpr size_t kSortTileSmem = kSortTile * (sizeof(uint64_t) + sizeof(uint16_t)) + (kSortThreads / 32) * 256 * sizeof(uint16_t);

__global__ void __launch_bounds__(kSortThreads) k_sort_tile(uint64_t* __restrict__ keys, int32_t* __restrict__ vals, int n)
{
    constexpr int kWarps = kSortThreads / 32;
    extern __shared__ __align__(16) unsigned char s_sort[];
    uint64_t* s_key = reinterpret_cast<uint64_t*>(s_sort);
    uint16_t* s_val = reinterpret_cast<uint16_t*>(s_key + kSortTile);
    uint16_t(*s_cnt)[256] = reinterpret_cast<uint16_t(*)[256]>(s_val + kSortTile);
    __shared__ int s_start[256];
    __shared__ int s_warp[kWarps];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int w0 = warp * 32 * kSortItems + lane;
    uint64_t key[kSortItems];
    uint32_t val[kSortItems];
#pragma unroll
    for (int k = 0; k < kSortItems; ++k) {  // what lies past the end stays behind every key
        const int i = w0 + 32 * k;
        key[k] = i < n ? keys[i] : ~0ull;
        val[k] = (uint32_t)i;
    }
    for (int pass = 0; pass < kPasses; ++pass) {
        const int shift = 8 * pass;
        for (int k = t; k < kWarps * 128; k += kSortThreads) reinterpret_cast<uint32_t*>(s_cnt)[k] = 0u;
        __syncthreads();
        uint32_t rank[kSortItems];
#pragma unroll
        for (int k = 0; k < kSortItems; ++k) {
            const int d = (int)(key[k] >> shift) & 0xFF;
            const unsigned peers = same_digit(d);
            rank[k] = s_cnt[warp][d] + __popc(peers & ((1u << lane) - 1u));
            __syncwarp();
            if (lane == 31 - __clz(peers)) s_cnt[warp][d] = (uint16_t)(rank[k] + 1u);
            __syncwarp();
        }
        __syncthreads();
        int own = 0;
        if (t < 256) {
#pragma unroll
            for (int k = 0; k < kWarps; ++k) { const int c = s_cnt[k][t]; s_cnt[k][t] = (uint16_t)own; own += c; }
        }
        int x = own;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, x, off);
            if (lane >= off) x += y;
        }
        if (lane == 31) s_warp[warp] = x;
        __syncthreads();
        if (t < 256) {
            int add = x - own;
#pragma unroll
            for (int k = 0; k < 7; ++k) add += k < warp ? s_warp[k] : 0;
            s_start[t] = add;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kSortItems; ++k) {
            const int d = (int)(key[k] >> shift) & 0xFF;
            const int at = s_start[d] + s_cnt[warp][d] + (int)rank[k];
            s_key[at] = key[k];
            s_val[at] = (uint16_t)val[k];
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kSortItems; ++k) {
            key[k] = s_key[w0 + 32 * k];
            val[k] = s_val[w0 + 32 * k];
        }
    }
#pragma unroll
    for (int k = 0; k < kSortItems; ++k) {
        const int i = w0 + 32 * k;
        if (i < n) {
            keys[i] = key[k];
            vals[i] = (int32_t)val[k];
        }
    }
}
static_assert(kSortTile <= 65536, "places of a tile fit 16 bits");

int64_t sort_tiles(int64_t n) { return (n + kSortTile - 1) / kSortTile; }

size_t sort_status_bytes(int64_t n) { return (size_t)sort_tiles(n) * 256 * sizeof(uint32_t); }

constexpr size_t kPassSmem = kSortTile * (sizeof(uint64_t) + sizeof(int32_t)) + (kSortThreads / 32) * 256 * sizeof(uint16_t);

static cudaError_t radix_passes(uint64_t* const k[2], int32_t* const v[2], int64_t n, int passes, SortHead* H,
                                uint32_t* status, int32_t* report, cudaStream_t s)
{
    const unsigned tiles = (unsigned)sort_tiles(n);
    const size_t words = (size_t)tiles * 256;
    for (int pass = 0; pass < passes; ++pass) {
        const int a = pass & 1;
        const auto kernel = report && pass == passes - 1 ? k_radix_pass<true> : k_radix_pass<false>;
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPassSmem);
        if (e != cudaSuccess) return e;
        kernel<<<tiles, kSortThreads, kPassSmem, s>>>(k[a], pass ? v[a] : nullptr, n, pass, H, status + a * words,
                                                      status + (a ^ 1) * words, k[a ^ 1], v[a ^ 1], report);
        note_launch();
    }
    return cudaGetLastError();
}

cudaError_t sort_codes(const float* pts, const float* w, int64_t n, uint64_t* const k[2], int32_t* const v[2],
                       SortHead* H, uint32_t* status, TreeCtrl* c4, TreeCtrl* c2, int32_t* report, cudaStream_t s)
{
    const bool one_tile = n <= kSortTile;
    cudaError_t e = cudaMemsetAsync(H, 0, sizeof(SortHead), s);
    if (e == cudaSuccess && !one_tile) e = cudaMemsetAsync(status, 0, sort_status_bytes(n), s);  // the first pass's half
    if (e != cudaSuccess) return e;
    k_bounds<<<grid_for(n, kThreads, 4u * (unsigned)device_sm_count()), kThreads, 0, s>>>(pts, w, n, H, c4, c2);
    note_launch();
    k_morton<kPasses><<<grid_for(n, kMortonThreads, 2u * (unsigned)device_sm_count()), kMortonThreads, 0, s>>>(pts, n, c4, k[0], H);
    note_launch();
    if (one_tile) {
        e = cudaFuncSetAttribute(k_sort_tile, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSortTileSmem);
        if (e != cudaSuccess) return e;
        k_sort_tile<<<1, kSortThreads, kSortTileSmem, s>>>(k[0], v[0], (int)n);
        note_launch();
        return cudaGetLastError();
    }
    return radix_passes(k, v, n, kPasses, H, status, report, s);
}

cudaError_t sort_queries(const float* q, int64_t n, const TreeCtrl* ctrl, void** scratch, const int32_t** order,
                         const int32_t** error, cudaStream_t s)
{
    if (n < 1 || n >= (1 << 28)) return cudaSuccess;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(s, &cap);
    if (e != cudaSuccess) return e;
    if (cap != cudaStreamCaptureStatusNone) return cudaSuccess;
    const auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const size_t kb = up(n * sizeof(uint64_t)), vb = up(n * sizeof(int32_t)), hb = up(sizeof(SortHead));
    if (dalloc(scratch, 2 * kb + 2 * vb + hb + 2 * sort_status_bytes(n), s) != cudaSuccess) {
        cudaGetLastError();  // no memory: the caller's order
        *scratch = nullptr;
        return cudaSuccess;
    }
    unsigned char* at = static_cast<unsigned char*>(*scratch);
    SortHead* H = reinterpret_cast<SortHead*>(at);
    uint64_t* const k[2] = {reinterpret_cast<uint64_t*>(at + hb), reinterpret_cast<uint64_t*>(at + hb + kb)};
    int32_t* const v[2] = {reinterpret_cast<int32_t*>(at + hb + 2 * kb), reinterpret_cast<int32_t*>(at + hb + 2 * kb + vb)};
    uint32_t* status = reinterpret_cast<uint32_t*>(at + hb + 2 * kb + 2 * vb);
    e = cudaMemsetAsync(H, 0, sizeof(SortHead), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(status, 0, sort_status_bytes(n), s);
    if (e == cudaSuccess) {
        k_morton<kQueryPasses><<<grid_for(n, kMortonThreads, 2u * (unsigned)device_sm_count()), kMortonThreads, 0, s>>>(q, n, ctrl, k[0], H);
        note_launch();
        e = radix_passes(k, v, n, kQueryPasses, H, status, nullptr, s);
    }
    if (e != cudaSuccess) {
        dfree(*scratch, s);
        *scratch = nullptr;
        return e;
    }
    *order = v[kQueryPasses & 1];
    *error = &H->error;
    return cudaSuccess;
}

// ----------------------------------------------------------------------------------------------
// 4. gather into Morton order; shared code digits of neighbouring codes
//    lcp[i] = leading code digits (6 bits for d = 4, 3 bits for d = 2) shared by sorted codes i-1 and
//    i, capped at the deepest level; lcp[0] is not used
// ----------------------------------------------------------------------------------------------
constexpr int kTopoThreads = 512;
constexpr int kTopoWarps = kTopoThreads / 32;
constexpr int kTopoTile = 8 * kTopoThreads;  // positions to a block, eight to a thread
inline int64_t topo_tiles(int64_t n) { return (n + kTopoTile - 1) / kTopoTile; }

// What a run of boundaries tells a scan from one side: bit L (L < 24) says whether the last boundary
// with lcp <= L had lcp = L; bits 24..28 hold the smallest lcp. No boundary at all: kNoRun.
constexpr uint32_t kNoRun = 31u << 24;
__device__ __forceinline__ uint32_t run_one(int l) { return (1u << l) | ((uint32_t)l << 24); }
// the run `far` followed by the run `near`: a boundary of near with lcp l settles every level >= l
__device__ __forceinline__ uint32_t run_join(uint32_t far, uint32_t near)
{
    const uint32_t mf = far >> 24, mn = near >> 24;
    const uint32_t keep = mn < 24u ? (1u << mn) - 1u : 0xFFFFFFu;
    return (far & keep) | (near & 0xFFFFFFu) | (min(mf, mn) << 24);
}

// A thread's eight boundaries (bytes of l8; b of them exist, the first is position 0's if `first`) as
// runs from the left and from the right, joined over the block: the tile's runs for both sides
__device__ __forceinline__ void tile_runs(uint64_t l8, int b, bool first, uint32_t* __restrict__ from_left,
                                          uint32_t* __restrict__ from_right, uint32_t (*s_run)[kTopoWarps])
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t f = kNoRun, r = kNoRun;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        if (k >= b || (k == 0 && first)) continue;
        const uint32_t o = run_one((int)(l8 >> (8 * k)) & 0xFF);
        f = run_join(f, o);
        r = run_join(o, r);
    }
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t g = __shfl_down_sync(0xFFFFFFFFu, f, off), q = __shfl_down_sync(0xFFFFFFFFu, r, off);
        f = run_join(f, g);  // lane 0 ends with the whole warp, in order
        r = run_join(q, r);
    }
    if (lane == 0) { s_run[0][warp] = f; s_run[1][warp] = r; }
    __syncthreads();
    if (threadIdx.x == 0) {
        f = r = kNoRun;
        for (int k = 0; k < kTopoWarps; ++k) f = run_join(f, s_run[0][k]);
        for (int k = kTopoWarps - 1; k >= 0; --k) r = run_join(r, s_run[1][k]);
        from_left[blockIdx.x] = f;
        from_right[blockIdx.x] = r;
    }
}

// the runs from the right are joined far to near too: the boundaries further right are `far`
__global__ void __launch_bounds__(kTopoThreads) k_gather(const float* __restrict__ pts, const float* __restrict__ w,
                                                         const float* __restrict__ nrm,
                                                         const int32_t* __restrict__ perm,
                                                         const uint64_t* __restrict__ code, int64_t n,
                                                         float4* __restrict__ spw, float4* __restrict__ snrm,
                                                         uint8_t* __restrict__ lcp4, uint8_t* __restrict__ lcp2,
                                                         const SortHead* __restrict__ H, TreeCtrl* ctrl)
{
    // Where a wait of the sort gave up, perm and code hold anything: the points stay where they are, and
    // the shared digits are kept in range, for which any values make a tree
    const bool sorted = H->error == 0;
    if (blockIdx.x == 0 && threadIdx.x == 0 && !sorted) ctrl->error = kErrorTimeout;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = sorted ? perm[i] : i;
        spw[i] = make_float4(pts[3 * j], pts[3 * j + 1], pts[3 * j + 2], w[j]);
        if (nrm) snrm[i] = make_float4(nrm[3 * j], nrm[3 * j + 1], nrm[3 * j + 2], 0.0f);
        const int same = i ? max(__clzll((long long)(code[i] ^ code[i - 1])) - 4, 0) : 0;  // codes use 60 bits
        lcp4[i] = (uint8_t)min(same / 6, kMaxLevel4);
        lcp2[i] = (uint8_t)min(same / 3, kMaxLevel2);
        // equal codes are the points of one cell of the deepest level
        if (sorted && i >= (int64_t)kMaxChildren && code[i] == code[i - kMaxChildren]) ctrl->error = kErrorChildren;
    }
}

// ----------------------------------------------------------------------------------------------
// 5. topology, all generations at once
//    The levels at which the nodes above point i split are a set A_i: level L is in it when the
//    L-digit cell of i holds a boundary with lcp = L, that is when the nearest boundary with lcp <= L
//    to the left of i, or to the right, has lcp = L. Both sides are scans of the boundaries (run_join).
//    The generation of the node that splits at L is the number of smaller levels in A_i, the point's own
//    is |A_i|, and the nodes whose first point is i are those that split below the boundary on its
//    left, L > lcp[i], and the point: consecutive generations g0 .. g1. A node's id is its generation's
//    base plus the number of nodes of that generation that start before it, so one scan of counts per
//    (generation, tile) gives every id, and a node's first child, parent, last child and end are
//    ids at the same position. With leaf_size > 1 the levels below the first ancestor with at most that
//    many points are dropped from A_i (kSmallLeaf marks that ancestor).
//    What bounds it: a few passes over the positions, one for each generation in the last kernel. It
//    replaces seven kernels over all positions for every generation: 84 kernels and 1,180 us for 2^22
//    points, now four and 155 us (2^20: 470 -> 54 us)
// ----------------------------------------------------------------------------------------------
constexpr uint32_t kSmallLeaf = 1u << 31;  // in a mask: its last level is a leaf for its size

struct BuildArrays {
    int32_t* nb;
    int32_t* ne;
    int32_t* fc;
    int32_t* parent;
    uint32_t* meta;
    int32_t* skip;        // depth-first successors, or nullptr
    int32_t* last_child;  // scratch, per node
    uint32_t* mask;       // scratch, per position: A_i
    int32_t* count;       // scratch, [generation][tile]
    uint32_t* from_left;  // scratch, per tile
    uint32_t* from_right;
    const uint8_t* lcp;
    TreeCtrl* ctrl;
    int64_t n;
    int leaf_size;
    int max_level;
    int tiles;
};

// eight lcp bytes from position i on (i a multiple of eight), and how many of them exist
__device__ __forceinline__ uint64_t lcp8(const BuildArrays& B, int64_t i, int& have)
{
    have = B.n - i >= 8 ? 8 : (B.n > i ? (int)(B.n - i) : 0);
    if (have == 8) return *reinterpret_cast<const uint64_t*>(B.lcp + i);
    uint64_t x = 0;
    for (int k = 0; k < have; ++k) x |= (uint64_t)B.lcp[i + k] << (8 * k);
    return x;
}

__global__ void __launch_bounds__(kTopoThreads) k_topo_runs(BuildArrays B)
{
    __shared__ uint32_t s_run[2][kTopoWarps];
    const int64_t i = (int64_t)blockIdx.x * kTopoTile + 8 * threadIdx.x;
    int have;
    const uint64_t l8 = lcp8(B, i, have);
    if (i == 0) B.from_right[B.tiles] = B.from_right[B.tiles + 1] = 0u;  // k_aggregate's barrier
    tile_runs(l8, have, i == 0, B.from_left, B.from_right, s_run);
}

// The run of all tiles before tile t (dir = -1) or after it (+1), by one warp, nearest tiles first:
// it stops where level 0 is settled, which settles every level
__device__ __forceinline__ uint32_t carry_run(const uint32_t* __restrict__ runs, int t, int dir, int tiles)
{
    const int lane = threadIdx.x & 31;
    uint32_t carry = kNoRun;
    for (int p = t + dir; p >= 0 && p < tiles; p += 32 * dir) {
        const int k = p + lane * dir;
        uint32_t x = k >= 0 && k < tiles ? runs[k] : kNoRun;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_down_sync(0xFFFFFFFFu, x, off);  // higher lanes are further away
            x = run_join(lane + off < 32 ? y : kNoRun, x);
        }
        carry = run_join(__shfl_sync(0xFFFFFFFFu, x, 0), carry);
        if ((carry >> 24) == 0u) break;
    }
    return carry;
}

// the levels of mask A that split at or above the boundary with lcp l on a node's left: g0 of them
__device__ __forceinline__ int first_gen(uint32_t A, int l) { return __popc(A & ((2u << l) - 1u) & ~kSmallLeaf); }
__device__ __forceinline__ int point_gen(uint32_t A) { return __popc(A & ~kSmallLeaf); }

// A_i of every position, and the nodes of each generation that start in the tile
__global__ void __launch_bounds__(kTopoThreads) k_topo_masks(BuildArrays B)
{
    __shared__ uint32_t s_run[2][kTopoWarps];
    __shared__ uint32_t s_carry[2];
    __shared__ int s_count[kMaxDepth + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i0 = (int64_t)blockIdx.x * kTopoTile + 8 * threadIdx.x;
    int have;
    const uint64_t l8 = lcp8(B, i0, have);
    if (threadIdx.x <= kMaxDepth) s_count[threadIdx.x] = 0;
    // runs of the thread, then inclusive over the lanes before (after) it
    uint32_t f = kNoRun, r = kNoRun;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        if (k >= have || (k == 0 && i0 == 0)) continue;
        const uint32_t o = run_one((int)(l8 >> (8 * k)) & 0xFF);
        f = run_join(f, o);
        r = run_join(o, r);
    }
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t g = __shfl_up_sync(0xFFFFFFFFu, f, off), q = __shfl_down_sync(0xFFFFFFFFu, r, off);
        if (lane >= off) f = run_join(g, f);
        if (lane + off < 32) r = run_join(q, r);
    }
    if (lane == 31) s_run[0][warp] = f;
    if (lane == 0) s_run[1][warp] = r;
    if (warp == 0) {
        const uint32_t c = carry_run(B.from_left, (int)blockIdx.x, -1, B.tiles);
        if (lane == 0) s_carry[0] = c;
    }
    if (warp == 1) {
        const uint32_t c = carry_run(B.from_right, (int)blockIdx.x, 1, B.tiles);
        if (lane == 0) s_carry[1] = c;
    }
    f = __shfl_up_sync(0xFFFFFFFFu, f, 1);
    r = __shfl_down_sync(0xFFFFFFFFu, r, 1);
    if (lane == 0) f = kNoRun;
    if (lane == 31) r = kNoRun;
    __syncthreads();
    uint32_t left = s_carry[0], right = s_carry[1];
    for (int k = 0; k < warp; ++k) left = run_join(left, s_run[0][k]);
    for (int k = kTopoWarps - 1; k > warp; --k) right = run_join(right, s_run[1][k]);
    left = run_join(left, f);
    right = run_join(right, r);
    // each position: the boundaries up to its own from the left, those after it from the right
    uint32_t A[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        if (k < have && !(k == 0 && i0 == 0)) left = run_join(left, run_one((int)(l8 >> (8 * k)) & 0xFF));
        A[k] = left & 0xFFFFFFu;
    }
#pragma unroll
    for (int k = 7; k >= 0; --k) {
        A[k] |= right & 0xFFFFFFu;
        if (k < have && !(k == 0 && i0 == 0)) right = run_join(right, run_one((int)(l8 >> (8 * k)) & 0xFF));
    }
    if (B.leaf_size > 1) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (k >= have) continue;
            // widen the point's run level by level, deepest first, while it is small enough for a leaf
            int64_t a = i0 + k, b = a + 1;
            uint32_t rest = A[k], keep = A[k];
            while (rest) {
                const int L = 31 - __clz(rest);
                while (a > 0 && b - a <= B.leaf_size && (int)B.lcp[a] >= L) --a;
                while (b < B.n && b - a <= B.leaf_size && (int)B.lcp[b] >= L) ++b;
                if (b - a > B.leaf_size) break;
                keep = (A[k] & ((2u << L) - 1u)) | kSmallLeaf;
                rest &= ~(1u << L);
            }
            A[k] = keep;
        }
    }
    if (have == 8) {
        uint4* d = reinterpret_cast<uint4*>(B.mask + i0);
        d[0] = make_uint4(A[0], A[1], A[2], A[3]);
        d[1] = make_uint4(A[4], A[5], A[6], A[7]);
    } else {
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (k < have) B.mask[i0 + k] = A[k];
    }
    // bit g of gens: a node of generation g starts here
    uint32_t gens[8], any = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int l = i0 + k == 0 ? -1 : (int)(l8 >> (8 * k)) & 0xFF;
        gens[k] = k < have ? (2u << point_gen(A[k])) - (1u << (l < 0 ? 0 : first_gen(A[k], l))) : 0u;
        any |= gens[k];
    }
    any = __reduce_or_sync(0xFFFFFFFFu, any);
    for (int g = 0; any >> g; ++g) {
        int c = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) c += (int)(gens[k] >> g) & 1;
        c = __reduce_add_sync(0xFFFFFFFFu, c);
        if (lane == 0) atomicAdd(&s_count[g], c);
    }
    __syncthreads();
    if (threadIdx.x <= kMaxDepth) B.count[(int64_t)threadIdx.x * B.tiles + blockIdx.x] = s_count[threadIdx.x];
}

// Exclusive sums of the counts along the tiles, a warp to a generation, and the control block
__global__ void __launch_bounds__(1024) k_topo_scan(BuildArrays B)
{
    __shared__ int s_total[32];
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
    int run = 0;
    if (g <= kMaxDepth) {
        int32_t* c = B.count + (int64_t)g * B.tiles;
        for (int b = 0; b < B.tiles; b += 128) {
            int v[4], sum = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int i = b + 4 * lane + k;
                v[k] = i < B.tiles ? c[i] : 0;
                sum += v[k];
            }
            int x = sum;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int y = __shfl_up_sync(0xFFFFFFFFu, x, off);
                if (lane >= off) x += y;
            }
            int at = run + x - sum;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int i = b + 4 * lane + k;
                if (i < B.tiles) c[i] = at;
                at += v[k];
            }
            run += __shfl_sync(0xFFFFFFFFu, x, 31);
        }
    }
    if (lane == 0) s_total[g] = run;
    __syncthreads();
    if (threadIdx.x != 0) return;
    int base = 0, deepest = 0;
    for (int k = 0; k <= kMaxDepth; ++k) {
        B.ctrl->depth_base[k] = base;
        base += s_total[k];
        if (s_total[k]) deepest = k;
    }
    B.ctrl->depth_base[kMaxDepth + 1] = base;
    B.ctrl->max_depth = deepest;
    B.ctrl->n_nodes = base;
    B.ctrl->first_sub = deepest > 0 ? 1 : 0;  // the root's children, or a lone point
    B.ctrl->n_sub = s_total[deepest > 0 ? 1 : 0];
}

// The nodes' ranges, links, levels and kinds. A warp takes 256 positions, 32 at a time; for each
// generation a ballot says at which of them a node starts.
__global__ void __launch_bounds__(kTopoThreads) k_topo_emit(BuildArrays B)
{
    __shared__ int32_t s_base[kTopoWarps][kMaxDepth + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned below = (1u << lane) - 1u;
    const int64_t i0 = (int64_t)blockIdx.x * kTopoTile + warp * 256;
    const int top = B.ctrl->max_depth;
    {
        uint32_t gens[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int64_t i = i0 + 32 * k + lane;
            gens[k] = 0u;
            if (i < B.n) {
                const uint32_t A = B.mask[i];
                gens[k] = (2u << point_gen(A)) - (1u << (i ? first_gen(A, B.lcp[i]) : 0));
            }
        }
        for (int g = 0; g <= top; ++g) {
            int c = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) c += (int)(gens[k] >> g) & 1;
            c = __reduce_add_sync(0xFFFFFFFFu, c);
            if (lane == 0) s_base[warp][g] = c;
        }
    }
    __syncthreads();
    if ((int)threadIdx.x <= top) {  // where each warp's nodes of a generation begin
        int at = B.ctrl->depth_base[threadIdx.x] + B.count[(int64_t)threadIdx.x * B.tiles + blockIdx.x];
        for (int k = 0; k < kTopoWarps; ++k) {
            const int c = s_base[k][threadIdx.x];
            s_base[k][threadIdx.x] = at;
            at += c;
        }
    }
    __syncthreads();
    for (int k = 0; k < 8; ++k) {
        const int64_t i = i0 + 32 * k + lane;
        const bool live = i < B.n;
        if (!__any_sync(0xFFFFFFFFu, live)) break;
        const uint32_t A = live ? B.mask[i] : 0u;
        const int l = live && i ? (int)B.lcp[i] : -1;
        const int g1 = live ? point_gen(A) : -1;
        const int g0 = live ? (l < 0 ? 0 : first_gen(A, l)) : kMaxDepth + 1;
        int gp = __shfl_up_sync(0xFFFFFFFFu, g1, 1);  // the generation of the point before
        if (lane == 0) gp = i0 + 32 * k > 0 ? point_gen(B.mask[i0 + 32 * k - 1]) : -1;
        const bool end = live && i == B.n - 1;
        const bool small = (A & kSmallLeaf) != 0u;
        uint32_t rest = A & ~kSmallLeaf;
        int level = -1;       // of the generation before
        int32_t before = 0;   // nodes of the generation before that start before this position (as ids)
        int32_t first = -1;   // the first node that starts here
        int started = 0;      // whether one of the generation before starts here
        for (int g = 0; g <= top; ++g) {
            const int starts = g >= g0 && g <= g1 ? 1 : 0;
            const unsigned bal = __ballot_sync(0xFFFFFFFFu, starts);
            const int32_t id = s_base[warp][g] + __popc(bal & below);
            __syncwarp();
            if (lane == 0) s_base[warp][g] += __popc(bal);
            __syncwarp();
            if (g <= g1) {
                uint32_t kind = kPoint;
                const int split = __ffs(rest) - 1;
                rest &= rest - 1u;
                if (g == g1) level = level + 1;
                else if (small && g == g1 - 1) { kind = kMultiLeaf; level = level + 1; }
                else { kind = split >= B.max_level ? kMultiLeaf : kInternal; level = split; }
                if (starts) {
                    if (g == g0) first = id;
                    B.nb[id] = (int32_t)i;
                    B.parent[id] = g ? before + started - 1 : -1;
                    B.meta[id] = meta_pack(0, (uint32_t)level, kind);
                    if (kind == kPoint) B.fc[id] = -1;
                    if (started) B.fc[before] = id;
                }
            }
            if (live && i > 0 && g >= g0 && g <= gp) {  // the node before this position ends here
                B.ne[id - 1] = (int32_t)i;
                if (B.skip) B.skip[id - 1] = first;
            }
            if (live && i > 0 && g > g0 && g <= gp) B.last_child[before - 1] = id - 1;
            if (end && g <= g1) {
                B.ne[id + starts - 1] = (int32_t)B.n;
                if (B.skip) B.skip[id + starts - 1] = -1;
                if (g) B.last_child[before + started - 1] = id + starts - 1;
            }
            before = id;
            started = starts;
        }
    }
}

// ----------------------------------------------------------------------------------------------
// 6. aggregates and records, children before parents: one kernel over the generations from the deepest
//    up, with a barrier of the grid between them. A node gets the FP64 sums of m, m p, m n of its
//    children in their order, its FP32 record (quotients rounded once to FP32) and its child count;
//    its children get their prefix mass fractions and the slots of the child pick's guide table.
//    What bounds it is the FP64 unit, two lanes to an SM: a warp's FP64 instruction holds it for 16
//    clocks, however few lanes take part. So
//      - a lane works on one sum of a node, eight lanes to a node with normals (one is padding) and four
//        without (a thread to a node issued seven additions a child, for the widest of 32 nodes);
//      - the prefix sums are the running sum of m (each child summed them anew);
//      - quotients are FP32 pairs (quotient_rn), and conversions integer operations;
//      - points, three nodes of four, take a lane each and only the products m p, m n.
//    2^22 points: 1,090 us in 16 kernels -> 389 us; 4,096 points: 137 -> 39 us; the 8-ary and 64-ary
//    trees of 2^18: 434 us in 42 kernels -> 168 us (without normals).
// ----------------------------------------------------------------------------------------------
struct Split {
    float h, l;
    bool ok;  // h + l is the value to 2^-47 of it, and far from FP32's limits
};
__device__ __forceinline__ Split split(double x)
{
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const uint32_t e = (hi >> 20) & 0x7FFu, sign = hi & 0x80000000u;
    Split r;
    r.ok = e - 963u <= 120u;  // 2^-60 .. 2^60
    r.h = __uint_as_float(sign | ((((hi & 0x7FFFFFFFu) - 0x38000000u) << 3) | lo >> 29));
    r.l = (float)(lo & 0x1FFFFFFFu) * __uint_as_float(sign | ((e - 948u) << 23));  // 2^(e - 1023 - 52)
    return r;
}

// __double2float_rn(a / b), B = split(b), y = 1 / B.h to a few roundings. The quotient to 2^-44 of it as
// an FP32 pair decides the rounding unless it is that near to the middle of two floats: there, a
// remainder of zero says that the quotient is the middle (the centre of two equal masses often is),
// and anything else takes the division.
__device__ __forceinline__ float quotient_rn(double a, double b, const Split& B, float y)
{
    const uint32_t ah = (uint32_t)__double2hiint(a);
    if (((ah << 1) | (uint32_t)__double2loint(a)) == 0u) return __uint_as_float(ah);
    const Split A = split(a);
    if (!A.ok || !B.ok) return __double2float_rn(a / b);
    const float q1 = __fmul_rn(A.h, y);
    const float r = __fadd_rn(__fmaf_rn(-q1, B.l, __fmaf_rn(-q1, B.h, A.h)), A.l);
    const float q2 = __fmul_rn(r, y);
    const float s = __fadd_rn(q1, q2);
    const float err = __fsub_rn(q2, __fsub_rn(s, q1)), ae = fabsf(err);
    const float half = __uint_as_float((__float_as_uint(s) & 0x7F800000u) - (24u << 23));  // of the gap to the next float
    const bool power = (__float_as_uint(s) & 0x7FFFFFu) == 0u;  // the gap below is half of it
    if (ae <= half * (power ? 0.49999237f : 0.99999237f)) return s;
    const float gap = power && ae < 0.75f * half && (err < 0.0f) != (s < 0.0f) ? 0.5f * half : half;
    const double mid = (double)s + (double)copysignf(gap, err);
    if (fma(-mid, b, a) == 0.0) return __double2float_rn(mid);
    return __double2float_rn(a / b);
}

// __double2float_rn(x) by integer operations
__device__ __forceinline__ float narrow(double x)
{
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    if (((hi >> 20) & 0x7FFu) - 898u > 250u) return ((hi << 1) | lo) == 0u ? __uint_as_float(hi) : __double2float_rn(x);
    const uint32_t t = (((hi & 0x7FFFFFFFu) - 0x38000000u) << 3) | lo >> 29, rest = lo << 3;  // 24 bits, and the 29 below
    const uint32_t up = rest > 0x80000000u || (rest == 0x80000000u && (t & 1u)) ? 1u : 0u;
    return __uint_as_float((hi & 0x80000000u) | (t + up));
}

constexpr int kAggThreads = 256, kAggWarps = kAggThreads / 32, kAggBlocks = 4;  // blocks resident on an SM
constexpr int kAggChildren = 64;  // prefix sums kept per node (a leaf of duplicates may have more children)

template <bool NORMALS>
struct AggShape {
    static constexpr int kLanes = NORMALS ? 8 : 4;  // of a node, and doubles of its sums
    static constexpr int kSums = NORMALS ? 7 : 4;
    static constexpr int kNodes = 32 / kLanes;      // of a warp at a time
};

template <bool NORMALS>
struct AggScratch {
    double pre[AggShape<NORMALS>::kNodes][kAggChildren];
    float cdf[AggShape<NORMALS>::kNodes][kAggChildren];
};

struct AggArrays {
    BuildArrays B;
    const float4* spw;
    const float4* snrm;
    double* agg;
    float4* pm;
    float4* dip;
    float4* pmd;
    float* cdf;
    uint8_t* gd;
    unsigned* barrier;  // [0] blocks that are through with a generation, over all of them; [1] signs of life
};

// A leaf of many coincident points is one warp's work for 0.5 us a point, while every other block waits
// for it: the warp gives a sign of life after at most so many children, and a wait gives up only where
// there was none for its whole limit. (By the count of polls alone, some three million points in one
// cell, of 2^24 - 1 that are allowed, ended the build with SBH_ETIMEOUT.)
constexpr int kBeat = 4096;
__device__ __forceinline__ void beat(const AggArrays& A) { atomicAdd(A.barrier + 1, 1u); }

// Every block's writes of the generations so far are visible to every block. The grid is a cooperative
// launch, so all its blocks are running; the wait is bounded all the same, by kSpinLimit polls without a
// sign of life.
__device__ __forceinline__ void grid_barrier(const AggArrays& A, unsigned target)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(A.barrier, 1u);
        volatile unsigned* at = A.barrier;
        int spin = 0;
        unsigned seen = 0;
        while (*at < target || kSpinLimit < 0) {
            if (++spin <= kSpinLimit) continue;
            const unsigned beats = at[1];
            if (kSpinLimit < 0 || beats == seen) {
                atomicCAS(&A.B.ctrl->error, 0, kErrorTimeout);
                break;
            }
            seen = beats;
            spin = 0;
        }
        __threadfence();
    }
    __syncthreads();
}

// The child pick's guide table (Chen and Asau's method), one entry per child slot: for slot j of
// a node with nc children, the number of prefix fractions cdf_c <= u_j among the first nc - 1
// children, where u_j = ceil(j 2^24 / nc) 2^-24 is the smallest 24-bit draw whose slot
// floor(u nc) is j. It is stored at the child's own id (first child + j): every node but the root
// fills one slot of its parent. That count never decreases with u, so a pick with draw u in slot
// j that scans up from the entry finds the same child as counting all prefix fractions. The fractions
// never decrease, so the count is a bisection.
__device__ __forceinline__ uint8_t guide_entry(const float* cdf, uint32_t nc, uint32_t j)
{
    const uint32_t mj = (uint32_t)((((uint64_t)j << 24) + nc - 1u) / nc);  // < 2^24: exact in FP32
    const float uj = (float)mj * 5.9604644775390625e-8f;
    uint32_t lo = 0, hi = nc - 1u;
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (cdf[mid] <= uj) lo = mid + 1u;
        else hi = mid;
    }
    return (uint8_t)lo;
}

// The records of the node of one group of lanes (v < 0: none): its sums in order, then what follows from
// them. Every lane of the warp comes here.
template <bool NORMALS>
__device__ __forceinline__ void aggregate_node(const AggArrays& A, AggScratch<NORMALS>& S, int32_t v)
{
    constexpr int kLanes = AggShape<NORMALS>::kLanes, kSums = AggShape<NORMALS>::kSums;
    const int lane = threadIdx.x & 31, sub = lane % kLanes, group = lane / kLanes, first = lane - sub;
    int32_t f = 0;
    int nc = 0;
    if (v >= 0) {
        f = A.B.fc[v];
        nc = A.B.last_child[v] - f + 1;
    }
    const int wide = __reduce_max_sync(0xFFFFFFFFu, nc);
    double sum = 0.0;
    constexpr int kAhead = 8;
    double next[kAhead];
#pragma unroll
    for (int k = 0; k < kAhead; ++k) next[k] = k < nc ? __ldcg(&A.agg[kLanes * (int64_t)(f + k) + sub]) : 0.0;
    for (int c0 = 0; c0 < wide; c0 += kAhead) {
        if (c0 && c0 % kBeat == 0 && lane == 0) beat(A);
        double x[kAhead];
#pragma unroll
        for (int k = 0; k < kAhead; ++k) {
            x[k] = next[k];
            const int c = c0 + kAhead + k;
            next[k] = c < nc ? __ldcg(&A.agg[kLanes * (int64_t)(f + c) + sub]) : 0.0;
        }
#pragma unroll
        for (int k = 0; k < kAhead; ++k) {
            if (c0 + k >= nc) continue;
            // 0 + x of the first child is x, but for the sign of a zero
            if (c0 + k == 0) sum = __double_as_longlong(x[0]) == (long long)0x8000000000000000ull ? 0.0 : x[0];
            else sum += x[k];
            if (sub == 0 && c0 + k < kAggChildren) S.pre[group][c0 + k] = sum;
        }
    }
    __syncwarp();
    const double m = __shfl_sync(0xFFFFFFFFu, sum, first);
    const Split M = split(m);
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(M.h));
    const float r = v >= 0 && sub >= 1 && sub <= 3 ? quotient_rn(sum, m, M, y) : narrow(sum);
    float out[kSums];  // m, centre, dipole
#pragma unroll
    for (int k = 0; k < kSums; ++k) out[k] = __shfl_sync(0xFFFFFFFFu, r, first + k);
    if (v >= 0) {
        A.agg[kLanes * (int64_t)v + sub] = sub == kSums ? 0.0 : sum;
        const float4 pm = make_float4(out[1], out[2], out[3], out[0]);
        if (sub == 0) A.pm[v] = pm;
        if constexpr (NORMALS) {
            const float4 dp = make_float4(out[4], out[5], out[6], 0.0f);
            if (sub == 1) A.dip[v] = dp;
            if (sub == 4 && A.pmd) A.pmd[2 * (int64_t)v] = pm;
            if (sub == 5 && A.pmd) A.pmd[2 * (int64_t)v + 1] = dp;
        }
        if (sub == 2) A.B.meta[v] |= (uint32_t)nc & kMaxChildren;
        if (nc <= kAggChildren) {
            for (int c = sub; c < nc; c += kLanes) {
                const float q = c == nc - 1 ? 1.0f : quotient_rn(S.pre[group][c], m, M, y);
                S.cdf[group][c] = q;
                A.cdf[f + c] = q;
            }
        }
    }
    __syncwarp();
    if (v >= 0 && nc <= kAggChildren)
        for (int j = sub; j < nc; j += kLanes) A.gd[f + j] = guide_entry(S.cdf[group], (uint32_t)nc, (uint32_t)j);
    // a leaf of many duplicates: the prefix sums once more, 64 children at a time
    if (wide > kAggChildren) {
        const bool mine = v >= 0 && nc > kAggChildren;
        double pre = 0.0;
        for (int c0 = 0; c0 < wide; c0 += kAggChildren) {
            __syncwarp();
            if (c0 % kBeat == 0 && lane == 0) beat(A);
            if (mine && sub == 0)
                for (int c = c0; c < nc && c < c0 + kAggChildren; ++c) {
                    pre += __ldcg(&A.agg[kLanes * (int64_t)(f + c)]);
                    S.pre[group][c - c0] = pre;
                }
            __syncwarp();
            if (mine)
                for (int c = c0 + sub; c < nc && c < c0 + kAggChildren; c += kLanes)
                    A.cdf[f + c] = c == nc - 1 ? 1.0f : quotient_rn(S.pre[group][c - c0], m, M, y);
        }
        __threadfence_block();
        __syncwarp();
        if (mine)
            for (int j = sub; j < nc; j += kLanes) {
                if (j && j % kBeat == 0) beat(A);
                A.gd[f + j] = guide_entry(A.cdf + f, (uint32_t)nc, (uint32_t)j);
            }
    }
    __syncwarp();
}

template <bool NORMALS>
__global__ void __launch_bounds__(kAggThreads, kAggBlocks) k_aggregate(AggArrays A)
{
    __shared__ AggScratch<NORMALS> s_scratch[kAggWarps];
    constexpr int kLanes = AggShape<NORMALS>::kLanes, kNodes = AggShape<NORMALS>::kNodes;
    AggScratch<NORMALS>& S = s_scratch[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const TreeCtrl* ctrl = A.B.ctrl;
    const int deepest = ctrl->max_depth;
    // Input that is refused has no records made: points that are not numbers, say, are one leaf of all of
    // them, a single warp's work (2^18: the refusal took 128 ms). Errors of this kernel itself end it too.
    if (ctrl->error) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) {  // the root is nobody's child
        A.cdf[0] = 1.0f;
        A.gd[0] = 0;
    }
    for (int gen = deepest; gen >= 0; --gen) {
        const int32_t lo = ctrl->depth_base[gen], hi = ctrl->depth_base[gen + 1];
        // up to 32 ids to a warp, fewer where the generation has fewer than 32 to each warp of the grid:
        // a warp takes kNodes of them at a time
        const int warps = (int)gridDim.x * kAggWarps;
        int span = 32;
        while (span > kNodes && (int64_t)(hi - lo) * 2 <= (int64_t)span * warps) span >>= 1;
        for (int64_t b = lo + (int64_t)span * (blockIdx.x * kAggWarps + (threadIdx.x >> 5)); b < hi; b += (int64_t)span * warps) {
            const int32_t v = (int32_t)b + lane;
            const bool live = lane < span && b + lane < hi;
            const bool point = live && meta_kind(A.B.meta[v]) == kPoint;
            unsigned nodes = __ballot_sync(0xFFFFFFFFu, live && !point);
            if (point) {
                const int32_t i = A.B.nb[v];
                const float4 p = A.spw[i];
                const double w = widen(p.w);
                double2* d = reinterpret_cast<double2*>(A.agg + kLanes * (int64_t)v);
                d[0] = make_double2(w, w * widen(p.x));
                d[1] = make_double2(w * widen(p.y), w * widen(p.z));
                A.pm[v] = p;
                if constexpr (NORMALS) {
                    const float4 q = A.snrm[i];
                    d[2] = make_double2(w * widen(q.x), w * widen(q.y));
                    d[3] = make_double2(w * widen(q.z), 0.0);
                    // m n: one FP32 rounding of the exact product, as the FP64 sum rounded to FP32
                    const float4 dp = make_float4(__fmul_rn(p.w, q.x), __fmul_rn(p.w, q.y), __fmul_rn(p.w, q.z), 0.0f);
                    A.dip[v] = dp;
                    if (A.pmd) {  // the same two records side by side, for one 32-byte load
                        A.pmd[2 * (int64_t)v] = p;
                        A.pmd[2 * (int64_t)v + 1] = dp;
                    }
                }
            }
            while (nodes) {
                int32_t mine = -1;
#pragma unroll
                for (int k = 0; k < kNodes; ++k) {
                    if (nodes && lane / kLanes == k) mine = (int32_t)b + __ffs(nodes) - 1;
                    nodes &= nodes - 1u;
                }
                aggregate_node<NORMALS>(A, S, mine);
            }
        }
        if (gen) grid_barrier(A, (unsigned)(deepest - gen + 1) * gridDim.x);
    }
}

// ----------------------------------------------------------------------------------------------
// host orchestration
// ----------------------------------------------------------------------------------------------
#define SBH_TRY(x)                               \
    do {                                         \
        cudaError_t e_ = (x);                    \
        if (e_ != cudaSuccess) return e_;        \
    } while (0)

// Scratch buffers of one build step: whatever is still held when the step returns (on success or
// on an error part way) goes back in stream order; keep() hands a buffer over to the tree.
struct ScratchSet {
    cudaStream_t s;
    void* p[8] = {};
    int n = 0;
    explicit ScratchSet(cudaStream_t st) : s(st) {}
    ScratchSet(const ScratchSet&) = delete;
    ScratchSet& operator=(const ScratchSet&) = delete;
    template <class T>
    cudaError_t alloc(T** q, size_t bytes)
    {
        if (n == 8) return cudaErrorInvalidValue;
        const cudaError_t e = dalloc((void**)q, bytes, s);
        if (e == cudaSuccess) p[n++] = (void*)*q;
        return e;
    }
    void keep(const void* q)
    {
        for (int i = 0; i < n; ++i)
            if (p[i] == q) p[i] = nullptr;
    }
    ~ScratchSet()
    {
        for (int i = 0; i < n; ++i) dfree(p[i], s);
    }
};

cudaError_t alloc_tree(DeviceTree& D, int64_t n, bool with_dip, bool with_skip, bool with_rec, cudaStream_t s)
{
    const int64_t cap = 2 * n + 1;
    D.cap = cap;  // D.ctrl is kept if the caller allocated it already
    SBH_TRY(dalloc((void**)&D.pm, cap * sizeof(float4), s));
    if (with_dip) SBH_TRY(dalloc((void**)&D.dip, cap * sizeof(float4), s));
    if (with_dip && with_rec) SBH_TRY(dalloc((void**)&D.pmd, 2 * cap * sizeof(float4), s));
    SBH_TRY(dalloc((void**)&D.cdf, cap * sizeof(float), s));
    SBH_TRY(dalloc((void**)&D.gd, cap * sizeof(uint8_t), s));
    SBH_TRY(dalloc((void**)&D.fc, cap * sizeof(int32_t), s));
    SBH_TRY(dalloc((void**)&D.meta, cap * sizeof(uint32_t), s));
    SBH_TRY(dalloc((void**)&D.nb, cap * sizeof(int32_t), s));
    SBH_TRY(dalloc((void**)&D.ne, cap * sizeof(int32_t), s));
    SBH_TRY(dalloc((void**)&D.parent, cap * sizeof(int32_t), s));
    if (with_skip) SBH_TRY(dalloc((void**)&D.skip, cap * sizeof(int32_t), s));
    SBH_TRY(dalloc((void**)&D.agg, cap * D.agg_stride() * sizeof(double), s));
    if (!D.ctrl) SBH_TRY(dalloc((void**)&D.ctrl, sizeof(TreeCtrl), s));
    return cudaSuccess;
}

void free_tree(DeviceTree& D, cudaStream_t s)
{
    dfree(D.pm, s); dfree(D.dip, s); dfree(D.pmd, s); dfree(D.cdf, s); dfree(D.gd, s); dfree(D.fc, s); dfree(D.meta, s); dfree(D.nb, s);
    dfree(D.ne, s); dfree(D.parent, s); dfree(D.skip, s); dfree(D.rec, s); dfree(D.agg, s); dfree(D.ctrl, s);
    D = DeviceTree();
}

cudaError_t build_sorted(sbh_tree* T, const float* pts, const float* w, const float* nrm, cudaStream_t s)
{
    const int64_t n = T->n;
    ScratchSet guard(s);
    uint64_t* k[2] = {nullptr, nullptr};
    int32_t* v[2] = {nullptr, nullptr};
    SortHead* head = nullptr;
    uint32_t* status = nullptr;
    SBH_TRY(guard.alloc(&head, sizeof(SortHead)));
    SBH_TRY(guard.alloc(&status, 2 * sort_status_bytes(n)));
    for (int a = 0; a < 2; ++a) {
        SBH_TRY(guard.alloc(&k[a], n * sizeof(uint64_t)));
        SBH_TRY(guard.alloc(&v[a], n * sizeof(int32_t)));
    }
    SBH_TRY(sort_codes(pts, w, n, k, v, head, status, T->t4.ctrl, T->t2.ctrl, nullptr, s));
    T->code = k[0];  // an even number of passes ends where it began
    T->perm = v[0];
    guard.keep(k[0]);
    guard.keep(v[0]);
    SBH_TRY(dalloc((void**)&T->spw, n * sizeof(float4), s));
    if (nrm) SBH_TRY(dalloc((void**)&T->snrm, n * sizeof(float4), s));
    SBH_TRY(dalloc((void**)&T->lcp4, n, s));
    SBH_TRY(dalloc((void**)&T->lcp2, n, s));
    k_gather<<<grid_for(n, kTopoThreads, 8u * (unsigned)device_sm_count()), kTopoThreads, 0, s>>>(
        pts, w, nrm, T->perm, T->code, n, T->spw, T->snrm, T->lcp4, T->lcp2, head, T->t4.ctrl);
    note_launch();
    return cudaGetLastError();
}

cudaError_t build_tree(sbh_tree* T, DeviceTree& D, const uint8_t* lcp, int max_level, int level_shift,
                       bool with_skip, cudaStream_t s)
{
    const int64_t n = T->n;
    D.max_level = max_level;
    D.level_shift = level_shift;
    ScratchSet guard(s);
    const int64_t tiles = topo_tiles(n);
    BuildArrays B;
    B.nb = D.nb; B.ne = D.ne; B.fc = D.fc; B.parent = D.parent; B.meta = D.meta;
    B.skip = with_skip ? D.skip : nullptr;
    B.lcp = lcp; B.ctrl = D.ctrl; B.n = n; B.leaf_size = T->leaf_size; B.max_level = max_level; B.tiles = (int)tiles;
    SBH_TRY(guard.alloc(&B.mask, n * sizeof(uint32_t)));
    SBH_TRY(guard.alloc(&B.last_child, D.cap * sizeof(int32_t)));
    SBH_TRY(guard.alloc(&B.count, (kMaxDepth + 1) * tiles * sizeof(int32_t)));
    SBH_TRY(guard.alloc(&B.from_left, (2 * tiles + 2) * sizeof(uint32_t)));
    B.from_right = B.from_left + tiles;

    k_topo_runs<<<(unsigned)tiles, kTopoThreads, 0, s>>>(B);
    note_launch();
    k_topo_masks<<<(unsigned)tiles, kTopoThreads, 0, s>>>(B);
    note_launch();
    k_topo_scan<<<1, 1024, 0, s>>>(B);
    note_launch();
    k_topo_emit<<<(unsigned)tiles, kTopoThreads, 0, s>>>(B);
    note_launch();
    SBH_TRY(cudaGetLastError());
    AggArrays A = {B, T->spw, T->snrm, D.agg, D.pm, D.dip, D.pmd, D.cdf, D.gd, reinterpret_cast<unsigned*>(B.from_right + tiles)};
    void* args[] = {&A};
    const void* kernel = T->snrm ? reinterpret_cast<const void*>(k_aggregate<true>) : reinterpret_cast<const void*>(k_aggregate<false>);
    int per_sm = 0;  // blocks of a cooperative launch must all be resident: as many as fit, at most kAggBlocks
    SBH_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kAggThreads, 0));
    int64_t blocks = (2 * n + kAggThreads - 1) / kAggThreads;
    const int64_t resident = (int64_t)(per_sm < kAggBlocks ? per_sm : kAggBlocks) * device_sm_count();
    if (blocks > resident) blocks = resident;
    SBH_TRY(cudaLaunchCooperativeKernel(kernel, dim3((unsigned)blocks),
                                        dim3(kAggThreads), args, 0, s));
    note_launch();
    SBH_TRY(cudaGetLastError());
    D.built = true;
    return cudaSuccess;
}

// Node v's walk record: centre of mass and mass; first child (-1: a point), skip, level times 4, nothing. In
// trees with normals: centre of mass and level times 4 (kWalkPoint: a point); dipole sum and skip.
__global__ void __launch_bounds__(kThreads) k_walk_records(TreeView T, float4* __restrict__ rec)
{
    const int32_t N = T.ctrl->n_nodes;
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < N; v += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t m = T.meta[v];
        const bool point = meta_kind(m) == kPoint;
        const int lvl = 4 * (int)meta_level(m);
        float4 p = T.pm[v];
        float4 r;
        if (T.dip) {
            r = T.dip[v];
            r.w = __int_as_float(T.skip[v]);
            p.w = __int_as_float(point ? kWalkPoint : lvl);
        } else {
            r = make_float4(__int_as_float(point ? -1 : T.fc[v]), __int_as_float(T.skip[v]), __int_as_float(lvl), 0.0f);
        }
        rec[2 * v] = p;
        rec[2 * v + 1] = r;
    }
}

cudaError_t add_walk_records(DeviceTree& D, cudaStream_t s)
{
    if (dalloc((void**)&D.rec, 2 * D.cap * sizeof(float4), s) != cudaSuccess) {
        cudaGetLastError();
        D.rec = nullptr;
        return cudaSuccess;
    }
    k_walk_records<<<grid_for(D.cap), kThreads, 0, s>>>(D.view(), D.rec);
    note_launch();
    return cudaGetLastError();
}

}  // namespace sbh
