// sbh_learned.cu -- the learned child proposal: a 6-32-32-1 ReLU network that scores each child
// of a node from query-relative geometry, trained on the residuals met by the estimator's own
// traversals, and used in place of the mass-proportional pick of Algorithm 2.
//
// The paper samples the path index in proportion to mass and names importance sampling as future
// work (Sec. 3.3); this is the project's extension. At a node T with 2..64 children whose centre
// is nearer to the query than `near` cell diagonals, the proposal is
//   pi_c = (1 - eps) softmax(clamp(s))_c + eps m_c / m_T,   eps = 0.1, scores clamped to [-40, 40];
// elsewhere pi_c = m_c / m_T. Every child keeps a probability > 0, so the estimator stays unbiased
// with p(I in T) the product of the pi's along the path. Training: every training query walks
// Algorithm 2's own paths, each decision node within reach becomes a set, and its children's
// targets are |R_c(q)|, the exact residual of the child's subtree (its exact sum minus its
// centre-of-mass term), the per-level proposal that minimises the variance of the child's
// contribution; cross-entropy to the normalised targets, Adam on FP32 master weights, an FP16
// copy for inference. The estimator scores on the tensor cores (sbh_eval_batched.cu).
//
// Parameter layout (1313 values): W1[32][6], b1[32], W2[32][32], b2[32], w3[32], b3.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "sbh_build.cuh"
#include "sbh_learned.cuh"

namespace sbh {

namespace {

// Scores of feature rows with the estimator's tensor-core scorer: one warp per chunk of 32 rows.
constexpr int kScoreWarps = 8;

__global__ void __launch_bounds__(32 * kScoreWarps) k_scores(const __half* __restrict__ wg,
                                                            const float* __restrict__ feats, int64_t n,
                                                            float* __restrict__ out)
{
    __shared__ MlpFrag F;
    __shared__ __align__(16) uint32_t A[kScoreWarps][32 * kChunkWords];
    __shared__ float sc[kScoreWarps][32];
    mlp_frag_fill(wg, F);
    __syncthreads();
    MlpRegs R;
    load_mlp_regs(F, R);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t chunks = (n + 31) / 32;
    for (int64_t c = (int64_t)blockIdx.x * kScoreWarps + warp; c < chunks; c += (int64_t)gridDim.x * kScoreWarps) {
        const int64_t r = c * 32 + lane;
        const bool live = r < n;
        float x[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        if (live)
            for (int k = 0; k < 6; ++k) x[k] = feats[6 * r + k];
        store_feature_row(&A[warp][lane * kChunkWords], x, live);
        __syncwarp();
        const float s = score_chunk(R, A[warp], sc[warp]);
        if (live) out[r] = s;
        __syncwarp();
    }
}

// ------------------------------------------------------------------------------------------------
// training sets from the estimator's own traversals: every training query walks the paths of
// Algorithm 2 (mass-proportional picks, Eq. 5 roulette; its own random stream) and records each
// node it takes a decision at where the network would be used. Pass 0 counts per query, pass 1
// writes (query, node) at the query's offset. At most max_per_query sets per query, the first in
// the order (subdomain, sample, depth).
//   A block is a query and a thread one of its paths: a path is a chain of dependent reads of a few
// levels, and paths are all there is to run side by side. One thread to a query walked a few hundred
// such chains one after the other: 650 us a pass for 256 queries, now 8.
// ------------------------------------------------------------------------------------------------
constexpr int kVisitThreads = 256;

template <int PASS>
__global__ void __launch_bounds__(kVisitThreads) k_visit(TreeView T, const float* __restrict__ Q, int samples, uint2 key,
                                                         float near, int max_per_query, int32_t* __restrict__ count,
                                                         const int64_t* __restrict__ base, int32_t* __restrict__ set_q,
                                                         int32_t* __restrict__ set_node)
{
    __shared__ float diam[kDiamLevels];
    __shared__ int s_warp[kVisitThreads / 32];
    if (threadIdx.x < kDiamLevels) diam[threadIdx.x] = T.ctrl->diam[threadIdx.x];
    __syncthreads();
    const int j = (int)blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float3 q = make_float3(Q[3 * (int64_t)j], Q[3 * (int64_t)j + 1], Q[3 * (int64_t)j + 2]);
    const int32_t first_sub = T.ctrl->first_sub;
    const int64_t n_paths = (int64_t)T.ctrl->n_sub * samples;
    int n = 0;
    for (int64_t p0 = 0; p0 < n_paths && n < max_per_query; p0 += kVisitThreads) {
        const int64_t path = p0 + threadIdx.x;
        int32_t found[kMaxDepth];  // the path's decision nodes within reach (PASS 1)
        int c = 0;
        if (path < n_paths) {
            const int ai = (int)(path / samples), s = (int)(path % samples);
            int32_t node = first_sub + ai;
            const float4 pa = __ldg(&T.pm[node]);
            uint32_t mT = __ldg(&T.meta[node]);
            float dT = dist_rn(pa.x, pa.y, pa.z, q);
            uint4 blk = make_uint4(0u, 0u, 0u, 0u);
            for (uint32_t depth = 0; meta_kind(mT) != kPoint && depth < (uint32_t)kMaxDepth; ++depth) {
                const int nc = (int)meta_nchild(mT);
                if (learned_gate(nc, dT, near, diam[meta_level(mT)])) {
                    if (PASS == 1) found[c] = node;
                    ++c;
                }
                // the estimator's stream layout: one block serves depths 2i and 2i + 1
                if ((depth & 1u) == 0u) blk = philox4x32_10(make_uint4((uint32_t)j, (uint32_t)ai, (uint32_t)s, depth), key);
                const uint2 x = (depth & 1u) ? make_uint2(blk.z, blk.w) : make_uint2(blk.x, blk.y);
                const int32_t f = __ldg(&T.fc[node]);
                const float u = unit24(x.x);
                int lo = 0, hi = nc - 1;
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (__ldg(&T.cdf[f + mid]) <= u) lo = mid + 1;
                    else hi = mid;
                }
                const int32_t ch = f + lo;
                const float4 pc = __ldg(&T.pm[ch]);
                const uint32_t mc = __ldg(&T.meta[ch]);
                const float dc = dist_rn(pc.x, pc.y, pc.z, q);
                float p;
                if (!rr_continue(0, unit24(x.y), dT, diam[meta_level(mT)], meta_level(mT), dc, meta_level(mc), p)) break;
                node = ch;
                mT = mc;
                dT = dc;
            }
        }
        // where the path's sets go among those of the paths before it
        int x = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_warp[warp] = x;
        __syncthreads();
        int before = 0, total = 0;
        for (int k = 0; k < kVisitThreads / 32; ++k) {
            before += k < warp ? s_warp[k] : 0;
            total += s_warp[k];
        }
        __syncthreads();
        if (PASS == 1) {
            const int at = n + before + x - c;
            for (int i = 0; i < c && at + i < max_per_query; ++i) {
                set_q[base[j] + at + i] = j;
                set_node[base[j] + at + i] = found[i];
            }
        }
        n = min(n + total, max_per_query);
    }
    if (PASS == 0 && threadIdx.x == 0) count[j] = n;
}

__global__ void k_set_rows(TreeView T, const int32_t* __restrict__ set_node, int64_t n_sets, int64_t* __restrict__ rows)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n_sets) rows[i] = (int64_t)meta_nchild(__ldg(&T.meta[set_node[i]]));
}

// ------------------------------------------------------------------------------------------------
// training set: for every training query and every subdomain a with 2..64 children, one decision
// set = the children of a, features and |exact residual| targets (FP64 sums over the child's
// points, in Morton order)
// ------------------------------------------------------------------------------------------------
// m f(p, q) in FP64 (p: position and mass, N: m n of a node or a unit normal, whose m is then scale), by
// correctly rounded roots and quotients: a child that is one point has the residual zero exactly, and a
// set of such children uniform targets. (A reciprocal root refined from FP32's takes a third off the
// kernel, but leaves such sets the noise of its last places as targets.)
struct Query64 {
    double x, y, z;
};
template <int KIND>
__device__ __forceinline__ double value64(float4 p, float4 N, double scale, const Query64& q, const KernelParams& kp)
{
    const double dx = widen(p.x) - q.x, dy = widen(p.y) - q.y, dz = widen(p.z) - q.z;
    const double r2 = dx * dx + dy * dy + dz * dz;
    if constexpr (KIND == SBH_COULOMB) return widen(p.w) / sqrt(r2 + (double)kp.eps2);
    else if constexpr (KIND == SBH_WINDING) {
        if (r2 == 0.0) return 0.0;
        return scale * (dx * widen(N.x) + dy * widen(N.y) + dz * widen(N.z)) / (4.0 * 3.141592653589793 * r2 * sqrt(r2));
    } else if constexpr (KIND == SBH_SMOOTHDIST) {
        return widen(p.w) * exp(-(double)kp.alpha * sqrt(r2));
    } else {
        return widen(p.w) * (1.0 + kp.g[0] * dx + kp.g[1] * dy + kp.g[2] * dz);
    }
}
// A block to a decision set s = (query set_q[s], node set_node[s]), a warp to each of its children in
// turn: rows set_off[s] .. (sets near the root hold thousands of points a child, so a warp to a whole
// set left most of the chip waiting for the last of them). With widen for the conversions: 1,183 -> 616 us for the 256
// training queries of 2^17 winding sources.
constexpr int kDatasetWarps = 4;

template <int KIND>
__global__ void __launch_bounds__(32 * kDatasetWarps) k_dataset(TreeView T, const float4* __restrict__ spw,
                                                                const float4* __restrict__ snrm,
                                                                const float* __restrict__ Q,
                                                                const int32_t* __restrict__ set_q,
                                                                const int32_t* __restrict__ set_node, int64_t n_sets,
                                                                const int64_t* __restrict__ set_off, KernelParams kp,
                                                                float* __restrict__ feats, float* __restrict__ targets)
{
    __shared__ float diam[kDiamLevels];
    if (threadIdx.x < kDiamLevels) diam[threadIdx.x] = T.ctrl->diam[threadIdx.x];
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t s = blockIdx.x; s < n_sets; s += gridDim.x) {
        const int64_t j = set_q[s];
        const int32_t a = set_node[s];
        const float3 q = make_float3(Q[3 * j], Q[3 * j + 1], Q[3 * j + 2]);
        const uint32_t ma = __ldg(&T.meta[a]);
        const float4 pa = __ldg(&T.pm[a]);
        const int32_t f = __ldg(&T.fc[a]);
        const int nc = (int)meta_nchild(ma);
        const int64_t r0 = set_off[s];
        const float4 none = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        const Query64 q64 = {(double)q.x, (double)q.y, (double)q.z};
        for (int c = warp; c < nc; c += kDatasetWarps) {
            const int32_t ch = f + c;
            const int32_t b = __ldg(&T.nb[ch]), e = __ldg(&T.ne[ch]);
            double sum = 0.0;
            for (int32_t i = b + lane; i < e; i += 32) {
                const float4 p = spw[i];
                sum += value64<KIND>(p, KIND == SBH_WINDING ? snrm[i] : none, KIND == SBH_WINDING ? widen(p.w) : 1.0, q64, kp);
            }
            for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, off);
            if (lane == 0) {
                const float4 pc = __ldg(&T.pm[ch]);
                const double r = sum - value64<KIND>(pc, KIND == SBH_WINDING ? __ldg(&T.dip[ch]) : none, 1.0, q64, kp);
                targets[r0 + c] = (float)fabs(r);
                float x[6];
                child_features(T, diam, ma, pa, ch, pc, __ldg(&T.meta[ch]), q, KIND == SBH_WINDING, x);
                for (int k = 0; k < 6; ++k) feats[6 * (r0 + c) + k] = x[k];
            }
        }
    }
}

// ------------------------------------------------------------------------------------------------
// loss and gradient: mean over sets of the cross-entropy between softmax(scores) and the set's
// normalised targets. One warp per set, lane i = hidden unit i of both layers: its row and its column
// of W2 and its row of the W2 gradient are in registers (168 of them; 80 bytes are spilled), and the activations of the set's rows in
// shared memory, where a row's 32 values are read four at a time by all lanes at once. Four rows are
// worked on together, as each value is a chain of 32 dependent multiply-adds. The scores and the
// softmax have a row to a lane. Each warp keeps its partial gradient, the block adds its warps'
// partials in warp order and writes one row per block; k_sum_blocks adds the rows in block order.
// No atomics, and every sum in a fixed order: the training is the same bit for bit on every run.
//   It takes 96 multiply-adds per row and lane and half as many other instructions: bound by the latency
// of their chains, with 12 warps to an SM (registers and shared memory) that issue 37% of the time. Reading W2 from shared memory with a
// row to a lane (every lane in the same bank) and passing activations by shuffles took 534 us a step
// for 2,219 sets, now 40: 555 blocks are 1.2 waves, so a part of it is the second wave's.
// ------------------------------------------------------------------------------------------------
constexpr int kTrainWarps = 4;
constexpr int kTrainRows = 4;                // rows worked on together
constexpr int kPartStride = kMlpParams + 1;  // a block's row: the gradient, then its loss
constexpr int kActFloats = kMaxLearnedChildren * kH;  // a set's activations of one layer
constexpr size_t kLossSmem = (size_t)kTrainWarps * 2 * kActFloats * sizeof(float);
static_assert(kTrainWarps * kPartStride <= kTrainWarps * 2 * kActFloats, "the warps' partial gradients reuse the activations");
static_assert(kMaxLearnedChildren % kTrainRows == 0 && kH == 32, "a lane to a unit, whole groups of rows");

// Where units 4 k .. 4 k + 3 of row r are (in groups of four floats): spread over the banks so that a
// row to a lane reads without conflicts too
__device__ __forceinline__ int act4(int r, int k) { return r * (kH / 4) + (k ^ (r & 7)); }

__global__ void __launch_bounds__(32 * kTrainWarps, 3) k_loss_grad(const float* __restrict__ wg,
                                                                  const float* __restrict__ feats,
                                                                  const float* __restrict__ targets,
                                                                  const int64_t* __restrict__ off, int64_t n_sets,
                                                                  float inv_sets, float* __restrict__ part)
{
    extern __shared__ float4 s_act[];
    __shared__ __align__(16) float s_w3[kH];
    __shared__ float s_sc[kTrainWarps][kMaxLearnedChildren];  // scores, then their log-probabilities
    __shared__ float s_t[kTrainWarps][kMaxLearnedChildren];   // targets
    __shared__ float s_d[kTrainWarps][kMaxLearnedChildren];   // exp(score), then d loss / d score
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x < kH) s_w3[threadIdx.x] = wg[ow3 + threadIdx.x];
    // W2 through shared memory (rows of 33: a row to a lane without bank conflicts), where the activations
    // go later
    float* s_w2 = reinterpret_cast<float*>(s_act);
    for (int i = threadIdx.x; i < kH * kH; i += blockDim.x) s_w2[(i / kH) * (kH + 1) + i % kH] = wg[oW2 + i];
    __syncthreads();
    float4* h1s = s_act + (size_t)warp * 2 * (kActFloats / 4);
    float4* h2s = h1s + kActFloats / 4;  // of the second layer, then its gradient
    float* sc = s_sc[warp];
    float* st = s_t[warp];
    float* sd = s_d[warp];
    float gW1[kIn] = {0, 0, 0, 0, 0, 0}, gW2[kH], gb1 = 0, gb2 = 0, gw3 = 0, gb3 = 0, lsum = 0;
    float w1[kIn], w2row[kH], w2col[kH];
#pragma unroll
    for (int k = 0; k < kIn; ++k) w1[k] = wg[oW1 + lane * kIn + k];
#pragma unroll
    for (int k = 0; k < kH; ++k) {
        gW2[k] = 0.0f;
        w2row[k] = s_w2[lane * (kH + 1) + k];
        w2col[k] = s_w2[k * (kH + 1) + lane];
    }
    __syncthreads();
    const float b1 = wg[ob1 + lane], b2 = wg[ob2 + lane], w3 = wg[ow3 + lane], b3 = wg[ob3];
    const int mine = lane & 3;  // this lane's unit within its group of four

    for (int64_t s = (int64_t)blockIdx.x * kTrainWarps + warp; s < n_sets; s += (int64_t)gridDim.x * kTrainWarps) {
        const int64_t r0 = off[s];
        const int nc = (int)(off[s + 1] - r0);
        if (nc < 2 || nc > kMaxLearnedChildren) continue;
        // forward (rows past the set's last repeat it and count for nothing)
        for (int r = 0; r < nc; r += kTrainRows) {
#pragma unroll
            for (int j = 0; j < kTrainRows; ++j) {
                const float* x = feats + 6 * (r0 + min(r + j, nc - 1));
                float z = b1;
#pragma unroll
                for (int k = 0; k < kIn; ++k) z = fmaf(w1[k], x[k], z);
                reinterpret_cast<float*>(h1s + act4(r + j, lane >> 2))[mine] = fmaxf(z, 0.0f);
            }
            __syncwarp();
            float z2[kTrainRows];
#pragma unroll
            for (int j = 0; j < kTrainRows; ++j) z2[j] = b2;
#pragma unroll
            for (int k = 0; k < kH / 4; ++k) {
#pragma unroll
                for (int j = 0; j < kTrainRows; ++j) {
                    const float4 h = h1s[act4(r + j, k)];
                    z2[j] = fmaf(w2row[4 * k], h.x, z2[j]);
                    z2[j] = fmaf(w2row[4 * k + 1], h.y, z2[j]);
                    z2[j] = fmaf(w2row[4 * k + 2], h.z, z2[j]);
                    z2[j] = fmaf(w2row[4 * k + 3], h.w, z2[j]);
                }
            }
#pragma unroll
            for (int j = 0; j < kTrainRows; ++j)
                reinterpret_cast<float*>(h2s + act4(r + j, lane >> 2))[mine] = fmaxf(z2[j], 0.0f);
        }
        __syncwarp();
        // scores, a row to a lane: the products summed in halves (16, 8, 4, 2, 1)
        float tmax = 0.0f, mx = -3.0e38f;
        for (int c = lane; c < nc; c += 32) {
            float u[kH / 2];
#pragma unroll
            for (int k = 0; k < kH / 8; ++k) {
                const float4 a = h2s[act4(c, k)], b = h2s[act4(c, k + kH / 8)];
                const float4 wa = reinterpret_cast<const float4*>(s_w3)[k];
                const float4 wb = reinterpret_cast<const float4*>(s_w3)[k + kH / 8];
                u[4 * k] = __fadd_rn(__fmul_rn(wa.x, a.x), __fmul_rn(wb.x, b.x));
                u[4 * k + 1] = __fadd_rn(__fmul_rn(wa.y, a.y), __fmul_rn(wb.y, b.y));
                u[4 * k + 2] = __fadd_rn(__fmul_rn(wa.z, a.z), __fmul_rn(wb.z, b.z));
                u[4 * k + 3] = __fadd_rn(__fmul_rn(wa.w, a.w), __fmul_rn(wb.w, b.w));
            }
#pragma unroll
            for (int o = kH / 4; o > 0; o >>= 1) {
#pragma unroll
                for (int k = 0; k < o; ++k) u[k] = __fadd_rn(u[k], u[k + o]);
            }
            const float v = u[0] + b3, t = targets[r0 + c];
            sc[c] = v;
            st[c] = t;
            mx = fmaxf(mx, v);
            tmax = fmaxf(tmax, t);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
            tmax = fmaxf(tmax, __shfl_xor_sync(0xFFFFFFFFu, tmax, o));
        }
        // normalised targets t_c / sum_c' t_c', formed as (t_c / t_max) / sum_c' (t_c' / t_max): the
        // smooth distance's residuals exp(-alpha r) can be FP32 denormals, whose sum has no finite
        // reciprocal
        for (int c = lane; c < nc; c += 32) {
            sd[c] = __expf(sc[c] - mx);
            st[c] = tmax > 0.0f ? st[c] / tmax : 0.0f;
        }
        __syncwarp();
        float tsum = 0.0f, Z = 0.0f;
#pragma unroll 4
        for (int c = 0; c < nc; ++c) {
            tsum += st[c];
            Z += sd[c];
        }
        __syncwarp();
        const float logZ = __logf(Z);
        const float tnorm = tsum > 0.0f ? 1.0f / tsum : 0.0f;
        for (int c = lane; c < nc; c += 32) {
            const float t = tsum > 0.0f ? st[c] * tnorm : 1.0f / nc;
            const float lp = sc[c] - mx - logZ;
            st[c] = t;
            sc[c] = lp;
            sd[c] = (__expf(lp) - t) * inv_sets;
        }
        __syncwarp();
        // backward
        for (int r = 0; r < nc; r += kTrainRows) {
            float dh1[kTrainRows], dh2[kTrainRows];
#pragma unroll
            for (int j = 0; j < kTrainRows; ++j) {
                float* at = reinterpret_cast<float*>(h2s + act4(r + j, lane >> 2)) + mine;
                const float h2 = *at;
                float ds = 0.0f;
                if (r + j < nc) {
                    ds = sd[r + j];
                    lsum -= st[r + j] * sc[r + j];
                    gb3 += ds;
                    gw3 = fmaf(ds, h2, gw3);
                }
                dh2[j] = h2 > 0.0f ? ds * w3 : 0.0f;
                gb2 += dh2[j];
                *at = dh2[j];
                dh1[j] = 0.0f;
            }
            __syncwarp();
#pragma unroll
            for (int k = 0; k < kH / 4; ++k) {
#pragma unroll
                for (int j = 0; j < kTrainRows; ++j) {
                    const float4 h = h1s[act4(r + j, k)], d = h2s[act4(r + j, k)];
                    gW2[4 * k] = fmaf(dh2[j], h.x, gW2[4 * k]);
                    gW2[4 * k + 1] = fmaf(dh2[j], h.y, gW2[4 * k + 1]);
                    gW2[4 * k + 2] = fmaf(dh2[j], h.z, gW2[4 * k + 2]);
                    gW2[4 * k + 3] = fmaf(dh2[j], h.w, gW2[4 * k + 3]);
                    // dh1 of unit `lane`: sum_i W2[i][lane] dh2_i
                    dh1[j] = fmaf(w2col[4 * k], d.x, dh1[j]);
                    dh1[j] = fmaf(w2col[4 * k + 1], d.y, dh1[j]);
                    dh1[j] = fmaf(w2col[4 * k + 2], d.z, dh1[j]);
                    dh1[j] = fmaf(w2col[4 * k + 3], d.w, dh1[j]);
                }
            }
#pragma unroll
            for (int j = 0; j < kTrainRows; ++j) {
                const float* x = feats + 6 * (r0 + min(r + j, nc - 1));
                const float h1 = reinterpret_cast<const float*>(h1s + act4(r + j, lane >> 2))[mine];
                const float d = h1 > 0.0f && r + j < nc ? dh1[j] : 0.0f;
                gb1 += d;
                if (r + j < nc) {
#pragma unroll
                    for (int k = 0; k < kIn; ++k) gW1[k] = fmaf(d, x[k], gW1[k]);
                }
            }
        }
        __syncwarp();
    }
    __syncthreads();  // every warp is through with its activations
    float* wp = reinterpret_cast<float*>(s_act) + warp * kPartStride;
#pragma unroll
    for (int k = 0; k < kIn; ++k) wp[oW1 + lane * kIn + k] = gW1[k];
    wp[ob1 + lane] = gb1;
#pragma unroll
    for (int k = 0; k < kH; ++k) wp[oW2 + lane * kH + k] = gW2[k];
    wp[ob2 + lane] = gb2;
    wp[ow3 + lane] = gw3;
    if (lane == 0) {
        wp[ob3] = gb3;
        wp[kMlpParams] = lsum * inv_sets;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kPartStride; i += blockDim.x) {
        float t = 0.0f;
        for (int v = 0; v < kTrainWarps; ++v) t += reinterpret_cast<const float*>(s_act)[v * kPartStride + i];
        part[(int64_t)blockIdx.x * kPartStride + i] = t;
    }
}

// grad[i] = sum over blocks b (in order) of part[b][i]; loss likewise from the last column. ADAM: and
// the Adam step with that gradient. One warp to a block, and kSumAhead rows asked for before the first
// is added: the chain of additions is kept, the waits for the rows are not (25 -> 11 us for 555 rows, with the Adam step).
constexpr int kSumThreads = 32, kSumAhead = 64;

template <bool ADAM>
__global__ void __launch_bounds__(kSumThreads) k_sum_blocks(const float* __restrict__ part, int blocks,
                                                            float* __restrict__ grad, float* __restrict__ loss,
                                                            float* __restrict__ w, float* __restrict__ m,
                                                            float* __restrict__ v, __half* __restrict__ wh, float lr,
                                                            float c1, float c2)
{
    const int i = blockIdx.x * kSumThreads + threadIdx.x;
    if (i >= kPartStride) return;
    float t = 0.0f;
    for (int b = 0; b < blocks; b += kSumAhead) {
        float a[kSumAhead];
#pragma unroll
        for (int k = 0; k < kSumAhead; ++k) a[k] = b + k < blocks ? part[(int64_t)(b + k) * kPartStride + i] : 0.0f;
#pragma unroll
        for (int k = 0; k < kSumAhead; ++k)
            if (b + k < blocks) t += a[k];
    }
    if (i >= kMlpParams) {
        *loss = t;
        return;
    }
    grad[i] = t;
    if constexpr (ADAM) {
        const float mi = 0.9f * m[i] + 0.1f * t;
        const float vi = 0.999f * v[i] + 0.001f * t * t;
        m[i] = mi;
        v[i] = vi;
        const float wi = w[i] - lr * (mi * c1) / (sqrtf(vi * c2) + 1e-8f);
        w[i] = wi;
        wh[i] = __float2half_rn(wi);
    }
}

__global__ void k_to_half(const float* __restrict__ w, __half* __restrict__ wh)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < kMlpParams) wh[i] = __float2half_rn(w[i]);
}

}  // namespace

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
cudaError_t mlp_alloc(MlpState& M, cudaStream_t s)
{
    cudaError_t e = dalloc((void**)&M.w, kMlpParams * sizeof(float), s);
    if (e == cudaSuccess) e = dalloc((void**)&M.wh, kMlpParams * sizeof(__half), s);
    if (e == cudaSuccess) e = dalloc((void**)&M.m, kMlpParams * sizeof(float), s);
    if (e == cudaSuccess) e = dalloc((void**)&M.v, kMlpParams * sizeof(float), s);
    if (e == cudaSuccess) e = dalloc((void**)&M.grad, kMlpParams * sizeof(float), s);
    if (e == cudaSuccess) e = dalloc((void**)&M.loss, sizeof(float), s);
    M.part_blocks = 8 * device_sm_count();
    if (e == cudaSuccess) e = dalloc((void**)&M.part, (size_t)M.part_blocks * kPartStride * sizeof(float), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(M.m, 0, kMlpParams * sizeof(float), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(M.v, 0, kMlpParams * sizeof(float), s);
    return e;
}

void mlp_release(MlpState& M, cudaStream_t s)
{
    dfree(M.w, s); dfree(M.wh, s); dfree(M.m, s); dfree(M.v, s); dfree(M.grad, s); dfree(M.loss, s);
    dfree(M.part, s);
    M = MlpState();
}

cudaError_t mlp_sync_half(MlpState& M, cudaStream_t s)
{
    k_to_half<<<(kMlpParams + 255) / 256, 256, 0, s>>>(M.w, M.wh);
    note_launch();
    return cudaGetLastError();
}

cudaError_t mlp_scores(const MlpState& M, const float* feats, int64_t n, float* out, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    int64_t blocks = ((n + 31) / 32 + kScoreWarps - 1) / kScoreWarps;
    const int64_t cap = 8 * (int64_t)device_sm_count();
    if (blocks > cap) blocks = cap;
    k_scores<<<(unsigned)blocks, 32 * kScoreWarps, 0, s>>>(M.wh, feats, n, out);
    note_launch();
    return cudaGetLastError();
}

namespace {
// the blocks' partial gradients; *blocks: how many there are
cudaError_t partial_gradients(MlpState& M, const float* feats, const float* targets, const int64_t* off, int64_t n_sets,
                              int* blocks, cudaStream_t s)
{
    int64_t b = (n_sets + kTrainWarps - 1) / kTrainWarps;
    if (b > M.part_blocks) b = M.part_blocks;  // the partial sums are then added in a fixed order
    *blocks = (int)b;
    const cudaError_t e = cudaFuncSetAttribute(k_loss_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLossSmem);
    if (e != cudaSuccess) return e;
    k_loss_grad<<<(unsigned)b, 32 * kTrainWarps, kLossSmem, s>>>(M.w, feats, targets, off, n_sets,
                                                                1.0f / (float)n_sets, M.part);
    note_launch();
    return cudaGetLastError();
}
constexpr unsigned kSumGrid = (kPartStride + kSumThreads - 1) / kSumThreads;
}  // namespace

cudaError_t mlp_loss_grad(MlpState& M, const float* feats, const float* targets, const int64_t* off, int64_t n_sets,
                          cudaStream_t s)
{
    if (n_sets <= 0) {
        cudaError_t e = cudaMemsetAsync(M.grad, 0, kMlpParams * sizeof(float), s);
        if (e == cudaSuccess) e = cudaMemsetAsync(M.loss, 0, sizeof(float), s);
        return e;
    }
    int blocks;
    const cudaError_t e = partial_gradients(M, feats, targets, off, n_sets, &blocks, s);
    if (e != cudaSuccess) return e;
    k_sum_blocks<false><<<kSumGrid, kSumThreads, 0, s>>>(M.part, blocks, M.grad, M.loss, nullptr, nullptr, nullptr,
                                                         nullptr, 0.0f, 0.0f, 0.0f);
    note_launch();
    return cudaGetLastError();
}

cudaError_t mlp_train_step(MlpState& M, const float* feats, const float* targets, const int64_t* off, int64_t n_sets,
                           float lr, float* loss, cudaStream_t s)
{
    int blocks;
    const cudaError_t e = partial_gradients(M, feats, targets, off, n_sets, &blocks, s);
    if (e != cudaSuccess) return e;
    M.step += 1;
    const float c1 = 1.0f / (1.0f - powf(0.9f, (float)M.step));
    const float c2 = 1.0f / (1.0f - powf(0.999f, (float)M.step));
    k_sum_blocks<true><<<kSumGrid, kSumThreads, 0, s>>>(M.part, blocks, M.grad, loss, M.w, M.m, M.v, M.wh, lr, c1, c2);
    note_launch();
    return cudaGetLastError();
}

cudaError_t mlp_visit(const TreeView& T, const float* Q, int nq, int samples, uint64_t seed, float near,
                      int max_per_query, int32_t* count, const int64_t* base, int32_t* set_q, int32_t* set_node,
                      cudaStream_t s)
{
    if (nq <= 0) return cudaSuccess;
    const uint2 key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
    if (base == nullptr) k_visit<0><<<(unsigned)nq, kVisitThreads, 0, s>>>(T, Q, samples, key, near, max_per_query, count, nullptr, nullptr, nullptr);
    else k_visit<1><<<(unsigned)nq, kVisitThreads, 0, s>>>(T, Q, samples, key, near, max_per_query, nullptr, base, set_q, set_node);
    note_launch();
    return cudaGetLastError();
}

cudaError_t mlp_set_rows(const TreeView& T, const int32_t* set_node, int64_t n_sets, int64_t* rows, cudaStream_t s)
{
    if (n_sets <= 0) return cudaSuccess;
    k_set_rows<<<(unsigned)((n_sets + 255) / 256), 256, 0, s>>>(T, set_node, n_sets, rows);
    note_launch();
    return cudaGetLastError();
}

cudaError_t mlp_dataset(const sbh_tree* tree, const float* Q, const int32_t* set_q, const int32_t* set_node,
                        int64_t n_sets, const int64_t* set_off, const KernelParams& kp, float* feats, float* targets,
                        cudaStream_t s)
{
    if (n_sets <= 0) return cudaSuccess;
    const TreeView T = tree->t4.view();
    const int64_t cap = 1 << 20;
    const int64_t blocks = n_sets < cap ? n_sets : cap;
    const unsigned b = (unsigned)blocks;
    switch (kp.kind) {
    case SBH_COULOMB: k_dataset<SBH_COULOMB><<<b, 32 * kDatasetWarps, 0, s>>>(T, tree->spw, tree->snrm, Q, set_q, set_node, n_sets, set_off, kp, feats, targets); break;
    case SBH_WINDING: k_dataset<SBH_WINDING><<<b, 32 * kDatasetWarps, 0, s>>>(T, tree->spw, tree->snrm, Q, set_q, set_node, n_sets, set_off, kp, feats, targets); break;
    case SBH_SMOOTHDIST: k_dataset<SBH_SMOOTHDIST><<<b, 32 * kDatasetWarps, 0, s>>>(T, tree->spw, tree->snrm, Q, set_q, set_node, n_sets, set_off, kp, feats, targets); break;
    case SBH_AFFINE: k_dataset<SBH_AFFINE><<<b, 32 * kDatasetWarps, 0, s>>>(T, tree->spw, tree->snrm, Q, set_q, set_node, n_sets, set_off, kp, feats, targets); break;
    default: return cudaErrorInvalidValue;
    }
    note_launch();
    return cudaGetLastError();
}

}  // namespace sbh
