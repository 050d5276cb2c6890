// sbh_bh.cu -- deterministic Barnes-Hut (Madan et al. 2025, Sec. 3.1, Eq. 2, Algorithm 1) on
// the 8-ary tree, the GPU baseline the estimator is compared with.
//
// A node is used whole -- m_a f(p_a, q) added -- when it is a source point or its far-field ratio
// ||q - p_a|| / |B_a| >= beta; otherwise the walk enters its first child. The walk is stackless:
// after a node is used it continues at skip[node], the next node of a depth-first order after
// that node's subtree (its next sibling, else its parent's skip). With warp voting the 32 queries
// of a warp walk together: a node is opened when any of them needs it, so every lane reads the
// same node (one broadcast load) and no lane diverges; the sum only gets more accurate.
//
// What bounds the walk is the instructions of a step and the chain from one node's record to the
// next one's address, so a step is kept short:
//   - one 32-byte record per node (k_walk_records) holds its centre, mass, first child, skip and level, where
//     position, meta word and link were three loads, the last of them behind the test. All lanes of a
//     warp read one node, and each word delivered to 32 lanes is a wavefront of the L1 data path, which ran
//     at 83% with that record and the dipole: in trees with normals the record is the winding walk's,
//     with the dipole sum for the mass, and the first child is read when a node is opened, one in
//     eight (5.06 -> 4.85 ms; without normals, where the record is one load, that was slower). The
//     other kernels walk a tree with normals by its arrays;
//   - the far-field ratio is a correctly rounded root and quotient, and monotone in the squared
//     distance, so the test is one comparison with the smallest squared distance that passes it at
//     the node's level (open_limit): the same decisions without either operation.
// Without voting a warp takes as long as its lanes' paths differ, and each lane reads its own record. Calls
// of kSortFrom queries or more are walked in the order of the queries' Morton codes (sort_queries), a
// warp going through the nodes that any of its queries visits (kTogether): neither changes a query's
// walk or its sum.
//   2^20 winding sources, 2^21 grid queries, voting, theta 0.5: 8.04 -> 6.04 ms with the record and the
// comparison, 5.06 ms with the term taken from the test's differences. 2^18 Coulomb sources, 10^6 random
// queries, theta 0.8, no voting: 1.68 -> 0.67 ms sorted, lanes alone, 0.58 ms together (0.60 with the
// fused sum of the Coulomb term; the call with its sort 0.69 ms).
#include <cuda_runtime.h>
#include <stdint.h>

#include "sbh_build.cuh"
#include "sbh_eval.cuh"
#include "sbh_sort.cuh"

namespace sbh {

// The node's term from d = p - q, its squared length a fused sum: the test's own, whose every operation is
// rounded, would save the Coulomb term two instructions, but a fifth of its accuracy (mean error 2.9e-8 -> 3.2e-8).
template <int KIND>
__device__ __forceinline__ void bh_add(float4 p, float4 dp, float3 d, const KernelParams& kp, float& acc,
                                       ExpAcc& ex)
{
    if constexpr (KIND == SBH_COULOMB) {
        acc = fmaf(p.w, rsqrt_ftz(fmaf(d.x, d.x, fmaf(d.y, d.y, fmaf(d.z, d.z, kp.eps2)))), acc);
    } else if constexpr (KIND == SBH_WINDING) {
        const float f2 = fmaf(d.x, d.x, fmaf(d.y, d.y, d.z * d.z));
        const float ir = rsqrt_ftz(f2);
        const float t = fmaf(d.x, dp.x, fmaf(d.y, dp.y, d.z * dp.z)) * (ir * ir * ir) * kInv4Pi;
        acc += f2 >= kMinNormal ? t : 0.0f;
    } else if constexpr (KIND == SBH_AFFINE) {
        acc = fmaf(p.w, 1.0f + fmaf(kp.g[0], d.x, fmaf(kp.g[1], d.y, kp.g[2] * d.z)), acc);
    } else {
        const float f2 = fmaf(d.x, d.x, fmaf(d.y, d.y, d.z * d.z));
        const float r = f2 * rsqrt_ftz(fmaxf(f2, 1e-37f));
        ex.lower(r, kp.alpha);
        ex.acc = fmaf(p.w, ex.scale(r, kp.alpha), ex.acc);
    }
}

// The smallest squared distance s with sqrt(s) / B >= beta, both operations rounded to nearest: they
// never decrease with s, so a bisection over the floats finds it, near (beta B)^2 when that is a
// normal number. NaN (no s passes) when even infinity does not.
__device__ __forceinline__ bool far_enough(uint32_t s, float B, float beta)
{
    return __fdiv_rn(__fsqrt_rn(__uint_as_float(s)), B) >= beta;
}
__device__ float open_limit(float B, float beta)
{
    const uint32_t inf = 0x7F800000u;
    const float t = beta * B;
    const uint32_t g = min(__float_as_uint(t * t) & 0x7FFFFFFFu, inf);
    uint32_t lo = g > 8u ? g - 8u : 0u, hi = min(g + 8u, inf);
    if (far_enough(lo, B, beta)) {
        if (far_enough(0u, B, beta)) return 0.0f;
        hi = lo;
        lo = 0u;
    }
    if (!far_enough(hi, B, beta)) {
        if (!far_enough(inf, B, beta)) return __uint_as_float(0x7FC00000u);
        lo = hi;
        hi = inf;
    }
    while (hi - lo > 1u) {  // lo does not pass, hi does
        const uint32_t mid = lo + (hi - lo) / 2u;
        if (far_enough(mid, B, beta)) hi = mid;
        else lo = mid;
    }
    return __uint_as_float(hi);
}

// How the lanes of a warp walk:
//   kAlone     each for itself;
//   kVote      together, a node opened for all when one needs it;
//   kTogether  each query's own walk, the warp going through the nodes that any lane visits: a lane that
//              is through with a subtree the others enter waits at its skip. All lanes read one record
//              where lanes walking alone read one each, as soon as their paths differ. For queries near
//              each other (sorted), whose nodes are mostly the same.
enum { kAlone = 0, kVote = 1, kTogether = 2 };

// What a step of the walk reads of node v, from the kernel's walk records (REC) or the tree's arrays
template <int KIND, bool REC>
struct Node {
    float4 p, dp;         // (dp: the winding kernel's dipole)
    int32_t skip, first;  // (first: where the record has it; skip: there, or asked for ahead)
    int lvl;              // level times 4
    bool point;
};
template <int KIND, bool REC, bool AHEAD>
__device__ __forceinline__ Node<KIND, REC> load_node(const TreeView& T, const float4* __restrict__ rec, int32_t v)
{
    Node<KIND, REC> n;
    n.first = 0;
    if constexpr (REC && KIND == SBH_WINDING) {
        n.p = __ldg(rec + 2 * (int64_t)v);
        n.dp = __ldg(rec + 2 * (int64_t)v + 1);
        n.lvl = __float_as_int(n.p.w);
        n.skip = __float_as_int(n.dp.w);
        n.point = n.lvl == kWalkPoint;
    } else if constexpr (REC) {
        float4 r;
        ld_pmd(rec, v, n.p, r);
        n.first = __float_as_int(r.x);
        n.skip = __float_as_int(r.y);
        n.lvl = __float_as_int(r.z);
        n.point = n.first < 0;
    } else {
        n.p = __ldg(&T.pm[v]);
        if constexpr (KIND == SBH_WINDING) n.dp = __ldg(&T.dip[v]);
        const uint32_t m = __ldg(&T.meta[v]);
        n.skip = AHEAD ? __ldg(&T.skip[v]) : 0;
        n.lvl = 4 * (int)meta_level(m);
        n.point = meta_kind(m) == kPoint;
    }
    return n;
}

// AHEAD: the next node is asked for before the node's term is formed (kAheadTo)
template <int KIND, int MODE, bool REC, bool AHEAD>
__global__ void __launch_bounds__(256) k_bh_eval(TreeView T, const float4* __restrict__ rec,
                                                 const float* __restrict__ Q, int64_t nq, KernelParams kp, float beta,
                                                 const int32_t* __restrict__ order, const int32_t* sort_error,
                                                 float* __restrict__ out)
{
    __shared__ float s_limit[kDiamLevels];
    if (threadIdx.x < kDiamLevels) s_limit[threadIdx.x] = open_limit(T.ctrl->diam[threadIdx.x], beta);
    __syncthreads();
    if (order && *sort_error) order = nullptr;  // a bounded wait of the sort gave up: the caller's order
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int32_t n_nodes = T.ctrl->error ? -1 : T.ctrl->n_nodes;
    // the loop bound is warp-uniform so that voting warps stay converged
    const int64_t warp_base = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31);
    for (int64_t jb = warp_base; jb < nq; jb += stride) {
        const int64_t i = jb + (threadIdx.x & 31);
        const bool active = i < nq;
        const int64_t j = active && order ? (int64_t)order[i] : i;
        const float3 q = active ? make_float3(Q[3 * j], Q[3 * j + 1], Q[3 * j + 2]) : make_float3(0.f, 0.f, 0.f);
        float acc = 0.0f;
        ExpAcc ex;
        ex.init(3.0e38f);
        int32_t v = 0;
        int32_t own = active ? 0 : -1;  // kTogether: the node the lane's own walk is at
        // a depth-first walk enters every node at most once; the bound only guards a damaged tree
        int32_t budget = n_nodes + 1;
        if (MODE != kAlone || active) {
            Node<KIND, REC> node;
            if constexpr (AHEAD) node = load_node<KIND, REC, AHEAD>(T, rec, 0);
            while (v >= 0 && budget-- > 0) {
                if constexpr (!AHEAD) node = load_node<KIND, REC, AHEAD>(T, rec, v);
                const Node<KIND, REC> at = node;
                const float4 p = at.p;
                const float limit = *reinterpret_cast<const float*>(reinterpret_cast<const char*>(s_limit) + at.lvl);
                // dist2_rn, its differences kept
                const float3 d = make_float3(__fsub_rn(p.x, q.x), __fsub_rn(p.y, q.y), __fsub_rn(p.z, q.z));
                const float r2 = __fadd_rn(__fadd_rn(__fmul_rn(d.x, d.x), __fmul_rn(d.y, d.y)), __fmul_rn(d.z, d.z));
                bool use = at.point || r2 >= limit;
                if (MODE == kVote) use = __all_sync(0xFFFFFFFFu, use || !active);
                const bool mine = MODE == kTogether ? own == v : active;
                if (!AHEAD && use && mine) bh_add<KIND>(p, KIND == SBH_WINDING ? at.dp : p, d, kp, acc, ex);
                int32_t skip = at.skip;
                if constexpr (!REC && !AHEAD) skip = use ? __ldg(&T.skip[v]) : 0;
                const bool open = MODE == kTogether ? __any_sync(0xFFFFFFFFu, mine && !use) : !use;
                int32_t first = at.first;
                if (!REC || KIND == SBH_WINDING) first = open ? __ldg(&T.fc[v]) : 0;
                if (MODE == kTogether && mine) own = use ? skip : first;
                v = open ? first : skip;
                if constexpr (AHEAD) node = load_node<KIND, REC, AHEAD>(T, rec, v < 0 ? 0 : v);
                if (AHEAD && use && mine) bh_add<KIND>(p, KIND == SBH_WINDING ? at.dp : p, d, kp, acc, ex);
            }
        }
        if (v >= 0) acc = ex.acc = __int_as_float(0x7FC00000);  // walk did not finish: NaN
        if (active) {
            if constexpr (KIND == SBH_SMOOTHDIST)
                out[j] = ex.acc > 0.0f ? ex.ref - __logf(ex.acc) / kp.alpha : __int_as_float(0x7F800000);
            else out[j] = acc;
        }
    }
}

namespace {
// Queries from which a walk without voting is sorted and walked together. The sort takes 30 us and 20 us per
// million queries, and the fewer the queries, the further apart a warp's 32 are and the more nodes they
// visit between them; the larger theta, the less there is to gain. us sorted / not, at theta 0.5, 0.8, 1.2:
//                                              2^18 queries                        2^19                                2^20
//   Coulomb, 2^12 sources, grid         489/645   257/261   161/119     794/1211   387/466   221/206    1335/2277   622/840   331/342
//   Coulomb, 2^18 sources, random      2268/3185  853/987   389/363    3316/6787  1226/2072  523/791   5029/12472 1870/3852  768/1365
//   winding, 2^20 sources, grid        4508/5896 1722/1679  743/551    6889/11982 2526/3365 1033/1132 10471/22698 3779/6053 1539/1873
//   smooth distance, 2^14, random      1170/1496  523/533   263/219    1766/2910   788/1010  378/400   3021/5830  1245/1982  576/785
//   smooth distance, 2^20, grid        4666/3940 1736/1138  777/380    6983/8161  2491/2281 1044/783  10253/14920 3762/4064 1550/1303
// At 2^19 the smooth distance, whose terms cost most beside the reads, is the one that can lose, on a
// grid at large theta; below, all of them do.
constexpr int64_t kSortFrom = 1 << 19;

// Queries up to which a walk asks for the next node before it forms a node's term, to an SM: the wait for a
// node is then all that a step takes, where few warps share an SM, but it takes 5 to 13 registers more,
// and warps where there are many. 16 warps to an SM; times with / without, over three kernels, 5,000 to 2^20
// sources, theta 0.5 and 0.9: 20,000 queries 0.76 to 0.95, 78,000 0.77 to 1.04, 155,000 0.88 to 1.16, 310,000
// 0.98 to 1.29. (Without it a walk that opens every node, at theta 0, took up to a quarter longer from
// the records, a 32-byte sector each, than from the arrays, which hold neighbours in one sector.)
constexpr int64_t kAheadTo = 512;

struct BhLaunch {
    TreeView T;
    const float4* rec;
    const float* Q;
    int64_t nq;
    KernelParams kp;
    float beta;
    const int32_t* order;
    const int32_t* sort_error;
    float* out;
    cudaStream_t s;
    unsigned blocks;
};

template <int KIND, int MODE, bool REC, bool AHEAD>
void launch_bh(const BhLaunch& L)
{
    k_bh_eval<KIND, MODE, REC, AHEAD><<<L.blocks, 256, 0, L.s>>>(L.T, L.rec, L.Q, L.nq, L.kp, L.beta, L.order, L.sort_error, L.out);
    note_launch();
}

template <int KIND, int MODE>
void launch_bh_mode(const BhLaunch& L)
{
    if (L.nq <= kAheadTo * device_sm_count()) L.rec ? launch_bh<KIND, MODE, true, true>(L) : launch_bh<KIND, MODE, false, true>(L);
    else L.rec ? launch_bh<KIND, MODE, true, false>(L) : launch_bh<KIND, MODE, false, false>(L);
}

template <int KIND>
void launch_bh_kind(const BhLaunch& L, bool vote)
{
    if (vote) launch_bh_mode<KIND, kVote>(L);
    else if (L.order) launch_bh<KIND, kTogether, true, false>(L);
    else launch_bh_mode<KIND, kAlone>(L);
}
}  // namespace

cudaError_t launch_bh_eval(const DeviceTree& D, const float* Q, int64_t nq, const KernelParams& kp, float beta,
                           int warp_vote, float* out, cudaStream_t s)
{
    if (nq <= 0) return cudaSuccess;
    int64_t blocks = (nq + 255) / 256;
    const int64_t cap = (int64_t)device_sm_count() * 64;
    if (blocks > cap) blocks = cap;
    // the walk records of a tree with normals are the winding walk's
    const float4* rec = (kp.kind == SBH_WINDING) == (D.dip != nullptr) ? D.rec : nullptr;
    BhLaunch L = {D.view(), rec, Q, nq, kp, beta, nullptr, nullptr, out, s, (unsigned)blocks};
    void* scratch = nullptr;
    if (!warp_vote && rec && nq >= kSortFrom) {
        const cudaError_t e = sort_queries(Q, nq, D.ctrl, &scratch, &L.order, &L.sort_error, s);
        if (e != cudaSuccess) return e;
    }
    cudaError_t e = cudaSuccess;
    switch (kp.kind) {
    case SBH_COULOMB: launch_bh_kind<SBH_COULOMB>(L, warp_vote); break;
    case SBH_WINDING: launch_bh_kind<SBH_WINDING>(L, warp_vote); break;
    case SBH_SMOOTHDIST: launch_bh_kind<SBH_SMOOTHDIST>(L, warp_vote); break;
    case SBH_AFFINE: launch_bh_kind<SBH_AFFINE>(L, warp_vote); break;
    default: e = cudaErrorInvalidValue;
    }
    if (e == cudaSuccess) e = cudaGetLastError();
    dfree(scratch, s);
    return e;
}

}  // namespace sbh
