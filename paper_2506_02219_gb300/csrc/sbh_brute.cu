// sbh_brute.cu -- the exact kernel sum F(q) = sum_i m_i f(p_i, q) (Madan et al. 2025, Eq. 1) and its
// query gradient by tiled brute force (the paper's ground truth, Sec. 4.3).
//
// Where queries are few for the chip, a block of eight warps works on one group of 32 x QPT queries, QPT to
// a lane, and every warp of it on another eighth of each source tile; a cluster of up to eight blocks
// splits the sources further. So a few thousand queries fill the chip (5,001 queries: 79 groups of 64
// make 632 blocks instead of the 20 that one query per thread makes), and a source read from shared
// memory serves QPT queries. Partial sums meet in shared memory, then across the cluster's
// distributed shared memory, always in the same order: no scratch memory, no atomics, results
// reproducible. Where queries are many or sources few, each warp has queries of its own and goes
// through all sources, and there is nothing to join (launch_kind).
//
// Sources are staged two by two, so that the packed FP32 instructions take both of a pair at once.
// What bounds it: the FP32 pipe's register reads. A winding term is 12 FMA-pipe operations, most of them on
// three different registers, which this chip runs at 1.6 cycles per warp and scheduler (1.1 with a
// repeated operand; measured, packed or scalar alike): 19 cycles a term, of which the reciprocal root's 8.4
// run beside. The Coulomb term takes 9.7 cycles, near the root's own rate.
// 65,536 queries against 2^20 sources, winding: 49.1 -> 32.2 ms; smooth distance and gradient, 5,001
// queries against 2^19 sources: 47.3 -> 2.3 ms (one query per thread ran on 20 of 152 SMs, and the FP64
// sums were rescaled with every new smallest distance).
//
// With fp64_accum every FP32 partial sum of at most 256 terms is added into an FP64 accumulator, which
// keeps the rounding error of million-term sums at the level of one such partial.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "sbh_eval.cuh"
#include "sbh_f32x2.cuh"

namespace sbh {

namespace {

namespace cg = cooperative_groups;

constexpr int kBruteWarps = 8;
constexpr int kBruteThreads = 32 * kBruteWarps;
constexpr int kWarpTile = 128;                       // sources of a tile that one warp takes
constexpr int kBruteTile = kWarpTile * kBruteWarps;  // sources staged at a time
constexpr int kOwnTile = 256;                        // the same where each warp takes all of them
constexpr int kMaxCluster = 8;

__device__ __forceinline__ float ex2_ftz(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// A pair of staged sources: (x0 x1 y0 y1)(z0 z1 s0 s1) with s the mass, or for the winding kernel
// z of the dipole m n, whose x and y follow: (nx0 nx1 ny0 ny1)
template <int KIND>
struct Pair {
    static constexpr int kQuads = KIND == SBH_WINDING ? 3 : 2;
    f2 x, y, z, s, nx, ny;
    __device__ __forceinline__ void load(const float4* t)
    {
        const float4 a = t[0], b = t[1];
        x = f2_make(a.x, a.y); y = f2_make(a.z, a.w);
        z = f2_make(b.x, b.y); s = f2_make(b.z, b.w);
        if constexpr (KIND == SBH_WINDING) {
            const float4 c = t[2];
            nx = f2_make(c.x, c.y); ny = f2_make(c.z, c.w);
        }
    }
};

// Running sums of one query: FP32 partials by pair half, and what they are flushed into. The smooth
// distance keeps the partials in the frame exp(-alpha ref), ref the smallest distance so far, and what
// they are flushed into in the frame of aref, the ref of the last flush (an FP64 product costs 20
// cycles of the SM, so the frame of the FP64 sums moves once a flush and not with every new ref).
// The winding sums leave out 1 / (4 pi), the smooth distance's gradient alpha.
template <int KIND, bool FP64, bool GRAD>
struct Sums {
    using Acc = typename std::conditional<FP64, double, float>::type;
    f2 nqx, nqy, nqz;  // minus the query, in both halves
    f2 v, g[GRAD ? 3 : 1];
    Acc av, ag[GRAD ? 3 : 1];
    float ref, aref;

    __device__ __forceinline__ void init(float3 q)
    {
        nqx = f2_dup(-q.x); nqy = f2_dup(-q.y); nqz = f2_dup(-q.z);
        v = f2_dup(0.0f);
        av = 0;
        if constexpr (GRAD)
            for (int c = 0; c < 3; ++c) { g[c] = f2_dup(0.0f); ag[c] = 0; }
        ref = aref = 3.0e38f;
    }
    // SPLIT as in k_brute; where a query has few terms the conversions count, and integer operations do them
    template <bool SPLIT>
    __device__ __forceinline__ void flush(float c2)
    {
        const auto acc = [](float x) -> Acc {
            if constexpr (FP64 && !SPLIT) return widen(x);
            else return (Acc)x;
        };
        if constexpr (KIND == SBH_SMOOTHDIST) {
            if (ref < aref) {
                const Acc f = (Acc)ex2_ftz(c2 * (aref - ref));
                av *= f;
                if constexpr (GRAD)
                    for (int c = 0; c < 3; ++c) ag[c] *= f;
                aref = ref;
            }
        }
        av += acc(f2_lo(v) + f2_hi(v));
        v = f2_dup(0.0f);
        if constexpr (GRAD)
            for (int c = 0; c < 3; ++c) { ag[c] += acc(f2_lo(g[c]) + f2_hi(g[c])); g[c] = f2_dup(0.0f); }
    }
    // the frame moves down to distance d (rare: about ln n times a query)
    __device__ __forceinline__ void lower(float d, float c2)
    {
        const float f = ex2_ftz(c2 * (ref - d));
        const f2 f22 = f2_dup(f);
        v = v * f22;
        if constexpr (GRAD)
            for (int c = 0; c < 3; ++c) g[c] = g[c] * f22;
        ref = d;
    }
    // add a pair's terms (BOTH false: the second source is padding)
    template <bool BOTH>
    __device__ __forceinline__ void add(const Pair<KIND>& p, const KernelParams& kp, float c2)
    {
        const f2 dx = p.x + nqx, dy = p.y + nqy, dz = p.z + nqz;
        if constexpr (KIND == SBH_COULOMB) {
            const f2 e = f2_fma(dx, dx, f2_fma(dy, dy, f2_fma(dz, dz, f2_dup(kp.eps2))));
            const f2 ir = f2_make(rsqrt_ftz(f2_lo(e)), rsqrt_ftz(f2_hi(e)));
            if constexpr (GRAD) {
                f2 t = p.s * ir, c = t * (ir * ir);
                if (!BOTH) { t = f2_make(f2_lo(t), 0.0f); c = f2_make(f2_lo(c), 0.0f); }
                v = v + t;
                add_grad<BOTH>(c, dx, dy, dz);
            } else if (BOTH) {
                v = f2_fma(p.s, ir, v);
            } else {
                v = v + f2_make(f2_lo(p.s) * f2_lo(ir), 0.0f);
            }
        } else if constexpr (KIND == SBH_WINDING) {
            // 4 pi times the term, ((p - q).N) / r^3; 0 where r^2 is below the smallest normal float. The
            // root's argument is clamped there, so that its powers stay finite and the select can sit
            // before the last FMA (a select of the product cost an addition, 8% of the FMA pipe's work)
            const f2 r2 = f2_fma(dx, dx, f2_fma(dy, dy, dz * dz));
            const f2 dn = f2_fma(dx, p.nx, f2_fma(dy, p.ny, dz * p.s));
            const float r2l = f2_lo(r2), r2h = f2_hi(r2);
            const f2 ir = f2_make(rsqrt_ftz(fmaxf(r2l, kMinNormal)), rsqrt_ftz(fmaxf(r2h, kMinNormal)));
            const f2 ir2 = ir * ir, u = dn * ir;
            const bool l = r2l >= kMinNormal, h = BOTH && r2h >= kMinNormal;
            const f2 us = f2_make(l ? f2_lo(u) : 0.0f, h ? f2_hi(u) : 0.0f);
            v = f2_fma(us, ir2, v);
            if constexpr (GRAD) {  // 3 ((p - q).N) (p - q) / r^5 - N / r^3
                f2 x = dx, y = dy, z = dz, mx = p.nx, my = p.ny, mz = p.s;
                f2 c = (us * ir2) * (ir2 * f2_dup(3.0f));
                f2 b = ir * ir2 * f2_dup(-1.0f);
                if (!(l && h)) {  // coincident, NaN or padding: the half adds nothing (0 times NaN is not 0)
                    const auto mask = [&](f2 a) { return f2_make(l ? f2_lo(a) : 0.0f, h ? f2_hi(a) : 0.0f); };
                    x = mask(x); y = mask(y); z = mask(z); mx = mask(mx); my = mask(my); mz = mask(mz);
                    c = mask(c); b = mask(b);
                }
                g[0] = f2_fma(c, x, f2_fma(b, mx, g[0]));
                g[1] = f2_fma(c, y, f2_fma(b, my, g[1]));
                g[2] = f2_fma(c, z, f2_fma(b, mz, g[2]));
            }
        } else if constexpr (KIND == SBH_SMOOTHDIST) {
            const f2 r2 = f2_fma(dx, dx, f2_fma(dy, dy, dz * dz));
            const float r2l = f2_lo(r2), r2h = f2_hi(r2);
            const f2 ir = f2_make(rsqrt_ftz(fmaxf(r2l, 1e-37f)), rsqrt_ftz(fmaxf(r2h, 1e-37f)));
            const f2 d = r2 * ir;
            const float dm = BOTH ? fminf(f2_lo(d), f2_hi(d)) : f2_lo(d);
            if (dm < ref) lower(dm, c2);
            const f2 x = (d + f2_dup(-ref)) * f2_dup(c2);
            f2 t = p.s * f2_make(ex2_ftz(f2_lo(x)), ex2_ftz(f2_hi(x)));
            if (!BOTH) t = f2_make(f2_lo(t), 0.0f);
            v = v + t;
            if constexpr (GRAD) {
                const f2 c0 = t * ir;
                add_grad<BOTH>(f2_make(r2l > 0.0f ? f2_lo(c0) : 0.0f, BOTH && r2h > 0.0f ? f2_hi(c0) : 0.0f), dx, dy,
                               dz);
            }
        } else {
            const f2 h = f2_fma(f2_dup(kp.g[0]), dx, f2_fma(f2_dup(kp.g[1]), dy, f2_dup(kp.g[2]) * dz));
            f2 t = p.s * (f2_dup(1.0f) + h);
            if (!BOTH) t = f2_make(f2_lo(t), 0.0f);
            v = v + t;
            if constexpr (GRAD) {
                const f2 m = BOTH ? p.s : f2_make(f2_lo(p.s), 0.0f);
                for (int c = 0; c < 3; ++c) g[c] = f2_fma(m, f2_dup(-kp.g[c]), g[c]);
            }
        }
    }
    template <bool BOTH>
    __device__ __forceinline__ void add_grad(f2 c, f2 dx, f2 dy, f2 dz)
    {
        if constexpr (!BOTH) {  // the padding's difference is not used (0 times it could be NaN)
            dx = f2_make(f2_lo(dx), 0.0f); dy = f2_make(f2_lo(dy), 0.0f); dz = f2_make(f2_lo(dz), 0.0f);
        }
        g[0] = f2_fma(c, dx, g[0]); g[1] = f2_fma(c, dy, g[1]); g[2] = f2_fma(c, dz, g[2]);
    }
};

// what a warp, a block and then the cluster hand on about one query
template <bool FP64, bool GRAD>
struct Part {
    typename std::conditional<FP64, double, float>::type v, g[GRAD ? 3 : 1];
    float ref;
};

// sum of parts 0 .. count - 1 (get(k)), in that order; smooth distance: in the frame of the smallest
template <int KIND, bool FP64, bool GRAD, class Get>
__device__ __forceinline__ Part<FP64, GRAD> sum_parts(int count, float alpha, Get get)
{
    using P = Part<FP64, GRAD>;
    P s = get(0);
    if constexpr (KIND == SBH_SMOOTHDIST) {
        for (int k = 1; k < count; ++k) s.ref = fminf(s.ref, get(k).ref);
        s.v = 0;
        if (GRAD) for (int c = 0; c < 3; ++c) s.g[c] = 0;
    }
    for (int k = KIND == SBH_SMOOTHDIST ? 0 : 1; k < count; ++k) {
        const P p = get(k);
        if constexpr (KIND == SBH_SMOOTHDIST) {
            using A = decltype(s.v);
            A f;
            if constexpr (FP64) f = exp(-(double)alpha * ((double)p.ref - (double)s.ref));
            else f = __expf(-alpha * (p.ref - s.ref));
            s.v += p.v * f;
            if (GRAD) for (int c = 0; c < 3; ++c) s.g[c] += p.g[c] * f;
        } else {
            s.v += p.v;
            if (GRAD) for (int c = 0; c < 3; ++c) s.g[c] += p.g[c];
        }
    }
    return s;
}

// The results of query j from its sums over all sources
template <int KIND, bool GRAD, class Acc>
__device__ __forceinline__ void write_query(int64_t j, Acc sum, const Acc* g, float ref, const KernelParams& kp,
                                            float* __restrict__ out, float* __restrict__ grad)
{
    const double v = (double)sum;
    if constexpr (KIND == SBH_SMOOTHDIST) {
        const bool pos = v > 0.0;
        out[j] = pos ? (float)((double)ref - log(v) / (double)kp.alpha) : __int_as_float(0x7F800000);
        if constexpr (GRAD)  // d = ref - log(acc) / alpha: grad d = -grad acc / (alpha acc); alpha cancels
            for (int c = 0; c < 3; ++c)
                grad[3 * j + c] = pos ? (float)(-(double)g[c] / v) : __int_as_float(0x7FC00000);
    } else {
        const double f = KIND == SBH_WINDING ? 0.07957747154594766788 : 1.0;  // 1 / (4 pi)
        out[j] = (float)(v * f);
        if constexpr (GRAD)
            for (int c = 0; c < 3; ++c) grad[3 * j + c] = (float)((double)g[c] * f);
    }
}

// Blocks to an SM that a split kernel is compiled for (0: as it comes). Left alone, some get a few registers
// more than a block more would allow, others fewer than they could use. With these, against without:
// the smooth distance 0.92 of the time (28 sizes), its gradient 2.52 -> 2.29 ms (5,001 queries, 2^19 sources),
// winding gradients 0.93 to 1.00 (two blocks either way, at 90 registers without).
template <int KIND, bool FP64, bool GRAD, bool SPLIT>
constexpr int brute_blocks()
{
    if (!SPLIT) return 0;
    if (GRAD) return KIND == SBH_WINDING ? 2 : 3;
    return KIND == SBH_SMOOTHDIST && FP64 ? 4 : 0;
}

// SPLIT: the warps of a block work on the same queries, else each on its own
template <int KIND, bool FP64, bool GRAD, int QPT, bool SPLIT>
__global__ void __launch_bounds__(kBruteThreads, brute_blocks<KIND, FP64, GRAD, SPLIT>()) k_brute(
    const float* __restrict__ P, const float* __restrict__ W, const float* __restrict__ N, int64_t n,
    const float* __restrict__ Q, int64_t nq, KernelParams kp, float c2, float* __restrict__ out, float* __restrict__ grad)
{
    constexpr int kQuads = Pair<KIND>::kQuads;
    constexpr int kGroup = 32 * QPT;
    constexpr int kTile = SPLIT ? kBruteTile : kOwnTile, kShare = SPLIT ? kBruteWarps : 1;
    using PartT = Part<FP64, GRAD>;
    constexpr size_t kTileBytes = (size_t)(kTile / 2) * kQuads * sizeof(float4);
    constexpr size_t kPartBytes = SPLIT ? sizeof(PartT) * kGroup * kBruteWarps : 0;
    __shared__ __align__(16) unsigned char s_buf[kTileBytes > kPartBytes ? kTileBytes : kPartBytes];
    float4* tile = reinterpret_cast<float4*>(s_buf);
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = SPLIT ? (int)cluster.block_rank() : 0, ranks = SPLIT ? (int)cluster.num_blocks() : 1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t q0 = (SPLIT ? (int64_t)(blockIdx.x / ranks) : (int64_t)blockIdx.x * kBruteWarps + warp) * kGroup;
    // this block's sources: as even shares as whole 128s go, so that loads start on a line
    const int64_t s_lo = (n * rank / ranks) & ~(int64_t)127;
    const int64_t s_hi = rank == ranks - 1 ? n : (n * (rank + 1) / ranks) & ~(int64_t)127;

    Sums<KIND, FP64, GRAD> S[QPT];
#pragma unroll
    for (int k = 0; k < QPT; ++k) {
        const int64_t j = q0 + 32 * k + lane;
        S[k].init(j < nq ? make_float3(Q[3 * j], Q[3 * j + 1], Q[3 * j + 2]) : make_float3(0.f, 0.f, 0.f));
    }
    const int tiles = (int)((s_hi - s_lo + kTile - 1) / kTile);
    for (int t = 0; t < tiles; ++t) {
        const int64_t base = s_lo + (int64_t)t * kTile;
        const int cnt = (s_hi - base) < kTile ? (int)(s_hi - base) : kTile;
        __syncthreads();
        for (int k = threadIdx.x; k < (cnt + 1) / 2; k += kBruteThreads) {
            const int64_t i = base + 2 * k, i1 = i + 1 < s_hi ? i + 1 : i;
            float4* d = tile + kQuads * k;
            const float w0 = W[i], w1 = W[i1];
            d[0] = make_float4(P[3 * i], P[3 * i1], P[3 * i + 1], P[3 * i1 + 1]);
            if constexpr (KIND == SBH_WINDING) {
                d[1] = make_float4(P[3 * i + 2], P[3 * i1 + 2], w0 * N[3 * i + 2], w1 * N[3 * i1 + 2]);
                d[2] = make_float4(w0 * N[3 * i], w1 * N[3 * i1], w0 * N[3 * i + 1], w1 * N[3 * i1 + 1]);
            } else {
                d[1] = make_float4(P[3 * i + 2], P[3 * i1 + 2], w0, w1);
            }
        }
        __syncthreads();
        // the warp's part of the tile, in whole pairs; only the last pair of all may hold padding
        const int per = cnt == kTile ? kTile / 2 / kShare : ((cnt + 1) / 2 + kShare - 1) / kShare;
        const int lo = SPLIT ? warp * per : 0, full = cnt / 2;
        const int hi = lo + per < full ? lo + per : full;
        // measured per kernel: 20.3 / 18.9 cycles a winding term at 2 / 4, 21.7 / 21.0 / 23.7 a smooth-distance
        // one at 2 / 1 / 4, its gradient 2.51 / 2.58 ms (5,001 queries, 2^19 sources) at 2 / 1
        constexpr int kUnroll = GRAD ? 2 : (KIND == SBH_SMOOTHDIST ? 1 : 4);
#pragma unroll kUnroll
        for (int k = lo; k < hi; ++k) {
            Pair<KIND> p;
            p.load(tile + kQuads * k);
#pragma unroll
            for (int u = 0; u < QPT; ++u) S[u].template add<true>(p, kp, c2);
        }
        if ((cnt & 1) && full >= lo && full < lo + per) {
            Pair<KIND> p;
            p.load(tile + kQuads * full);
#pragma unroll
            for (int u = 0; u < QPT; ++u) S[u].template add<false>(p, kp, c2);
        }
        if (!SPLIT || (t & 1)) {  // 256 terms at most
#pragma unroll
            for (int u = 0; u < QPT; ++u) S[u].template flush<SPLIT>(c2);
        }
    }
    if constexpr (!SPLIT) {
#pragma unroll
        for (int u = 0; u < QPT; ++u) {
            const int64_t j = q0 + 32 * u + lane;
            if (j < nq) write_query<KIND, GRAD>(j, S[u].av, S[u].ag, S[u].ref, kp, out, grad);
        }
    } else {
        __shared__ PartT s_block[kGroup];
        __syncthreads();  // the tile's memory becomes the warps' parts
        PartT* parts = reinterpret_cast<PartT*>(s_buf);
#pragma unroll
        for (int u = 0; u < QPT; ++u) {
            S[u].template flush<SPLIT>(c2);
            PartT p;
            p.v = S[u].av;
            if (GRAD) for (int c = 0; c < 3; ++c) p.g[c] = S[u].ag[c];
            p.ref = S[u].ref;
            parts[warp * kGroup + 32 * u + lane] = p;
        }
        __syncthreads();
        if (threadIdx.x < kGroup)
            s_block[threadIdx.x] = sum_parts<KIND, FP64, GRAD>(kBruteWarps, kp.alpha,
                                                               [&](int k) { return parts[k * kGroup + threadIdx.x]; });
        cluster.sync();
        const int64_t j = q0 + threadIdx.x;
        if (rank == 0 && threadIdx.x < kGroup && j < nq) {
            const PartT s = sum_parts<KIND, FP64, GRAD>(
                ranks, kp.alpha, [&](int k) { return *cluster.map_shared_rank(&s_block[threadIdx.x], k); });
            write_query<KIND, GRAD>(j, s.v, s.g, s.ref, kp, out, grad);
        }
        cluster.sync();  // no block leaves while its sums are being read
    }
}

struct BruteCall {
    const float *P, *W, *N;
    int64_t n;
    const float* Q;
    int64_t nq;
    KernelParams kp;
    float *out, *grad;
    cudaStream_t s;
};

template <int KIND, bool FP64, bool GRAD, int QPT, bool SPLIT>
cudaError_t launch_group(const BruteCall& B)
{
    const int64_t per_block = 32 * QPT * (SPLIT ? 1 : kBruteWarps);
    const int64_t groups = (B.nq + per_block - 1) / per_block;
    // as many blocks to a cluster as fill the chip several times over, a tile to each at least, eight at most
    int ranks = 1;
    while (SPLIT && ranks < kMaxCluster && groups * ranks < 16 * (int64_t)device_sm_count() &&
           2 * (int64_t)ranks * kBruteTile <= B.n)
        ranks *= 2;
    // exp(-alpha x) = 2^(c2 x), with c2 finite for every alpha: the nearest source's x is 0
    const float c2 = fmaxf(-B.kp.alpha * 1.44269504088896341f, -3.0e38f);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(groups * ranks));
    cfg.blockDim = dim3(kBruteThreads);
    cfg.stream = B.s;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)ranks;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_brute<KIND, FP64, GRAD, QPT, SPLIT>, B.P, B.W, B.N, B.n, B.Q, B.nq,
                                             B.kp, c2, B.out, B.grad);
    if (e == cudaSuccess) note_launch();
    return e;
}

// Which way a call goes. Joining the parts of a query that was split costs about as much as 200 to 800 of
// its terms (FP64 additions, and for the smooth distance an FP64 exponential for each part), so
// queries are split over warps only where that is what fills the chip, and over blocks only as
// far. 10^6 queries, us: one query a thread and no packed pairs (the kernel before this one) / every call
// split over eight warps and up to eight blocks / as now:
//   sources             10                100               1000                 10^4
//   Coulomb             29 / 85 / 26      53 / 85 / 48      304 / 264 / 247      2,800 / 3,615 / 2,250
//   smooth distance    141 / 499 / 109   306 / 482 / 115    775 / 596 / 548      6,440 / 8,398 / 5,106
//   its gradient       240 / 783 / 186   660 / 818 / 187  1,430 / 1,224 / 711    8,840 / 18,081 / 6,410
// Queries to a lane: four split (a shared-memory read of a source then costs each a quarter) where that
// still leaves several blocks to every SM, else two; two unsplit, one where two would leave too few
// blocks. The gradient's sums have registers for two, the smooth distance's are faster with one (5,270 / 5,459 us for
// 2 10^6 queries against 4,096 sources). Sums kept in FP32 stay split over the warps where sources are many:
// it is as fast, and their chains of additions are shorter.
template <int KIND, bool FP64, bool GRAD>
cudaError_t launch_kind(const BruteCall& B)
{
    constexpr bool kSmoothGrad = GRAD && KIND == SBH_SMOOTHDIST;
    const bool many = B.nq >= (kSmoothGrad ? 1 << 18 : 5 << 17) && (FP64 || B.n <= 4096);
    if (many || B.n < (B.nq >= 1 << 16 ? 1024 : 128)) {
        if constexpr (!kSmoothGrad) {
            if (many) return launch_group<KIND, FP64, GRAD, 2, false>(B);
        }
        return launch_group<KIND, FP64, GRAD, 1, false>(B);
    }
    if constexpr (!GRAD) {
        if (B.nq >= (int64_t)128 * device_sm_count()) return launch_group<KIND, FP64, GRAD, 4, true>(B);
    }
    return launch_group<KIND, FP64, GRAD, 2, true>(B);
}

template <bool FP64, bool GRAD>
cudaError_t launch_any(const BruteCall& B)
{
    if (B.nq <= 0) return cudaSuccess;
    cudaError_t e;
    switch (B.kp.kind) {
    case SBH_COULOMB: e = launch_kind<SBH_COULOMB, FP64, GRAD>(B); break;
    case SBH_WINDING: e = launch_kind<SBH_WINDING, FP64, GRAD>(B); break;
    case SBH_SMOOTHDIST: e = launch_kind<SBH_SMOOTHDIST, FP64, GRAD>(B); break;
    case SBH_AFFINE: e = launch_kind<SBH_AFFINE, FP64, GRAD>(B); break;
    default: return cudaErrorInvalidValue;
    }
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

cudaError_t launch_brute(const float* P, const float* W, const float* N, int64_t n, const float* Q, int64_t nq,
                         const KernelParams& kp, int fp64_accum, float* out, cudaStream_t s)
{
    const BruteCall B = {P, W, N, n, Q, nq, kp, out, nullptr, s};
    return fp64_accum ? launch_any<true, false>(B) : launch_any<false, false>(B);
}

cudaError_t launch_brute_grad(const float* P, const float* W, const float* N, int64_t n, const float* Q, int64_t nq,
                              const KernelParams& kp, float* out, float* grad, cudaStream_t s)
{
    return launch_any<true, true>({P, W, N, n, Q, nq, kp, out, grad, s});
}

}  // namespace sbh
