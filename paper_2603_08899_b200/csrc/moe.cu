// Contemplate-token embedding as a mixture of expert embeddings: router linear layer on the hidden
// state of the most recently accepted token, softmax over the experts, the k largest scores, sum of
// the chosen experts' embeddings weighted by their gating scores.
//
// A cluster of 8 CTAs per 1, 2 or 4 sequences (the more sequences in the call, the more share a cluster and
// with it a pass over the router matrix).  The router is n_expert dot products of length H_in: each CTA takes an eighth
// of the experts, a warp a dot product or a part of one (16-byte loads, fp32 accumulation, parts added in a
// fixed order); the scores are written into all eight CTAs' shared memory, every CTA does softmax and selection
// (k rounds of a warp argmax, the lower index on equal scores; a warp per sequence), and writes an eighth of the
// output columns.  Bound by latency: a few hundred KB per CTA from L2.  One CTA per sequence read the whole router
// by itself: B 8, 12288 -> 4096, 64 experts, bf16: 51 us, now 7.9 us (B 64: 17 us).
//
// A non-finite router score (a NaN or an infinity in the hidden state or the router) makes the
// scores of the sequence meaningless: the sequence's output row is written as zeros, its selection
// as experts 0..k-1 with gate 0, and status[b] (optional) gets CONFU_ST_NONFINITE.  The selected
// indices are clamped to the table whatever the scores are, so no input value can send a load or a
// store out of bounds.
#include <cooperative_groups.h>

#include "common.cuh"

namespace confu {

namespace cg = cooperative_groups;

constexpr int kMoeThreads = 512;
constexpr int kMoeMaxExperts = 1024;
constexpr int kMoeMaxK = 32;
constexpr int kMoeCluster = 8;

template <typename T> struct Vec16;
template <> struct Vec16<__nv_bfloat16> { static constexpr int n = 8; };
template <> struct Vec16<float> { static constexpr int n = 4; };

template <typename T>
__device__ __forceinline__ void load_vec(const T* p, float (&x)[Vec16<T>::n])
{
    if constexpr (sizeof(T) == 2) {
        const uint4 v = *reinterpret_cast<const uint4*>(p);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            x[2 * j] = __uint_as_float(w[j] << 16);
            x[2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u);
        }
    } else {
        const float4 v = *reinterpret_cast<const float4*>(p);
        x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
    }
}

__device__ __forceinline__ void store_vec(float* p, const float (&x)[4]) { *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]); }
__device__ __forceinline__ void store_vec(__nv_bfloat16* p, const float (&x)[8])
{
    __nv_bfloat162 h[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) h[j] = __floats2bfloat162_rn(x[2 * j], x[2 * j + 1]);
    *reinterpret_cast<uint4*>(p) = *reinterpret_cast<const uint4*>(h);
}

template <typename T, int NS>
__global__ void __launch_bounds__(kMoeThreads) con_embedding_kernel(
    int B, int H_in, int H_out, int n_expert, int k_expert, const T* __restrict__ hidden, const T* __restrict__ router_w,
    const T* __restrict__ router_b, const T* __restrict__ experts, int renormalize, T* __restrict__ out,
    int32_t* __restrict__ sel, float* __restrict__ gate, int32_t* __restrict__ status)
{
    constexpr int kVec = Vec16<T>::n, kWarps = kMoeThreads / 32;
    __shared__ float s_score[NS][kMoeMaxExperts];
    __shared__ float s_part[NS][kWarps];             // parts of dot products that several warps share
    __shared__ int s_sel[NS][kMoeMaxK];
    __shared__ float s_w[NS][kMoeMaxK];
    __shared__ int s_bad[NS];
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int b0 = (int)(blockIdx.x / kMoeCluster) * NS, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool vec_in = H_in % kVec == 0, vec_out = H_out % kVec == 0;

    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");      // the others' shared memory exists: waited for below
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // ---- router logits: experts e0 .. e1 - 1 are this CTA's; with fewer of them than warps each is cut into parts ----
    const int e0 = rank * n_expert / kMoeCluster, n_own = (rank + 1) * n_expert / kMoeCluster - e0;
    int parts = 1;
    while (n_own > 0 && 2 * parts * n_own <= kWarps) parts *= 2;
    const T* h[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) h[s] = hidden + (size_t)min(b0 + s, B - 1) * H_in;
    bool first_round = true;
    for (int i0 = 0; i0 < n_own * parts; i0 += kWarps) {
        const int item = i0 + warp, e = e0 + item / parts, part = item % parts;
        float acc[NS];
#pragma unroll
        for (int s = 0; s < NS; ++s) acc[s] = 0.f;
        if (item < n_own * parts) {
            const T* w = router_w + (size_t)e * H_in;
            if (vec_in) {
                const int n_vec = H_in / kVec, v1 = (int)((int64_t)(part + 1) * n_vec / parts);
#pragma unroll 8
                for (int v = (int)((int64_t)part * n_vec / parts) + lane; v < v1; v += 32) {
                    float y[kVec];
                    load_vec(w + (size_t)v * kVec, y);
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        float x[kVec];
                        load_vec(h[s] + (size_t)v * kVec, x);
#pragma unroll
                        for (int j = 0; j < kVec; ++j) acc[s] = fmaf(x[j], y[j], acc[s]);
                    }
                }
            } else {
                const int i1 = (int)((int64_t)(part + 1) * H_in / parts);
                for (int i = (int)((int64_t)part * H_in / parts) + lane; i < i1; i += 32)
#pragma unroll
                    for (int s = 0; s < NS; ++s) acc[s] = fmaf(to_f32(h[s][i]), to_f32(w[i]), acc[s]);
            }
        }
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            acc[s] = warp_sum(acc[s]);
            if (lane == 0) s_part[s][warp] = acc[s];
        }
        if (first_round) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
        first_round = false;
        __syncthreads();
        // the items of this round, one thread each per sequence and receiving CTA: the score goes to all eight
        for (int i = tid; i < kWarps / parts * NS * kMoeCluster; i += kMoeThreads) {
            const int peer = i % kMoeCluster, s = i / kMoeCluster % NS, first = i / (kMoeCluster * NS) * parts;
            if (i0 + first < n_own * parts) {
                const int expert = e0 + (i0 + first) / parts;
                float sc = 0.f;
                for (int q = 0; q < parts; ++q) sc += s_part[s][first + q];
                if (router_b) sc += to_f32(router_b[expert]);
                *cluster.map_shared_rank(&s_score[s][expert], peer) = sc;
            }
        }
        __syncthreads();
    }
    if (first_round) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");       // no expert of its own
    cluster.sync();

    // ---- softmax and the k largest scores (warp s: sequence s) ----
    if (warp < NS && b0 + warp < B) {
        float* score = s_score[warp];
        const int b = b0 + warp;
        const bool writer = rank == 0;
        float m = -INFINITY;
        bool bad = false;
        for (int e = lane; e < n_expert; e += 32) {
            m = fmaxf(m, score[e]);
            bad = bad || !(fabsf(score[e]) <= 3.0e38f);
        }
        bad = __any_sync(0xffffffffu, bad);
        if (lane == 0) s_bad[warp] = bad;
        if (bad) {
            if (writer && lane < k_expert) {
                if (sel) sel[(size_t)b * k_expert + lane] = lane;
                if (gate) gate[(size_t)b * k_expert + lane] = 0.f;
            }
            if (writer && lane == 0 && status) status[b] = CONFU_ST_NONFINITE;
        } else {
            m = warp_max(m);
            float z = 0.f;
            for (int e = lane; e < n_expert; e += 32) {
                const float p = __expf(score[e] - m);
                score[e] = p;
                z += p;
            }
            z = warp_sum(z);
            const float inv_z = 1.f / z;
            __syncwarp();
            float wsum = 0.f;
            for (int k = 0; k < k_expert; ++k) {
                float bv = -1.f;                     // scores are >= 0; a taken expert is marked -1
                int be = INT_MAX;
                for (int e = lane; e < n_expert; e += 32) {
                    const float p = score[e];
                    if (p > bv) { bv = p; be = e; }              // ascending e: the lower index wins a tie
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
                    const int oe = __shfl_xor_sync(0xffffffffu, be, o);
                    if (ov > bv || (ov == bv && oe < be)) { bv = ov; be = oe; }
                }
                be = min(max(be, 0), n_expert - 1);   // finite scores always give an index; never trust that for an address
                if (lane == 0) {
                    s_sel[warp][k] = be;
                    s_w[warp][k] = bv * inv_z;
                    score[be] = -1.f;
                }
                wsum += bv * inv_z;
                __syncwarp();
            }
            if (renormalize && lane < k_expert) s_w[warp][lane] = s_w[warp][lane] / wsum;
            __syncwarp();
            if (writer && lane < k_expert) {
                if (sel) sel[(size_t)b * k_expert + lane] = s_sel[warp][lane];
                if (gate) gate[(size_t)b * k_expert + lane] = s_w[warp][lane];
            }
        }
    }
    __syncthreads();

    // ---- weighted sum of the chosen embeddings: this CTA's eighth of the columns (all zero for a bad sequence) ----
    const int unit = vec_out ? kVec : 1, n_unit = H_out / unit;
    const int u0 = (int)((int64_t)rank * n_unit / kMoeCluster), n_cols = (int)((int64_t)(rank + 1) * n_unit / kMoeCluster) - u0;
    for (int i = tid; i < NS * n_cols; i += kMoeThreads) {
        const int s = i / n_cols, j = (u0 + i % n_cols) * unit;
        if (b0 + s >= B) break;
        T* o = out + (size_t)(b0 + s) * H_out + j;
        const int n_k = s_bad[s] ? 0 : k_expert;
        if (vec_out) {
            float acc[kVec];
#pragma unroll
            for (int v = 0; v < kVec; ++v) acc[v] = 0.f;
            for (int k = 0; k < n_k; ++k) {
                float x[kVec];
                load_vec(experts + (size_t)s_sel[s][k] * H_out + j, x);
                const float w = s_w[s][k];
#pragma unroll
                for (int v = 0; v < kVec; ++v) acc[v] = fmaf(w, x[v], acc[v]);
            }
            store_vec(o, acc);
        } else {
            float acc = 0.f;
            for (int k = 0; k < n_k; ++k) acc = fmaf(s_w[s][k], to_f32(experts[(size_t)s_sel[s][k] * H_out + j]), acc);
            o[0] = from_f32<T>(acc);
        }
    }
}

template <typename T, int NS>
static cudaError_t launch_ns(int B, int H_in, int H_out, int n_expert, int k_expert, const void* hidden, const void* router_w,
                             const void* router_b, const void* experts, int renormalize, void* out, int32_t* sel, float* gate,
                             int32_t* status, cudaStream_t st)
{
    cudaLaunchAttribute attrs[2];
    attrs[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attrs[0].val.programmaticStreamSerializationAllowed = 1;
    attrs[1].id = cudaLaunchAttributeClusterDimension;
    attrs[1].val.clusterDim.x = kMoeCluster;
    attrs[1].val.clusterDim.y = attrs[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((B + NS - 1) / NS) * kMoeCluster);
    cfg.blockDim = dim3(kMoeThreads);
    cfg.stream = st;
    cfg.attrs = attrs;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, con_embedding_kernel<T, NS>, B, H_in, H_out, n_expert, k_expert, (const T*)hidden,
                              (const T*)router_w, (const T*)router_b, (const T*)experts, renormalize, (T*)out, sel, gate, status);
}

cudaError_t launch_con_embedding(int B, int H_in, int H_out, int n_expert, int k_expert, int dtype, const void* hidden,
                                 const void* router_w, const void* router_b, const void* experts, int renormalize,
                                 void* out, int32_t* sel, float* gate, int32_t* status, cudaStream_t st)
{
    if (B == 0) return cudaSuccess;
    // one sequence per cluster while that leaves SMs free, then two, then four: the router is read once per cluster
    // (B 16: 9.2 us, B 17: 10.2, B 32: 11.7, B 33: 12.7, B 64: 17.1)
    const bool f32 = dtype == CONFU_F32;
    auto launch = B <= 16   ? (f32 ? launch_ns<float, 1> : launch_ns<__nv_bfloat16, 1>)
                  : B <= 32 ? (f32 ? launch_ns<float, 2> : launch_ns<__nv_bfloat16, 2>)
                            : (f32 ? launch_ns<float, 4> : launch_ns<__nv_bfloat16, 4>);
    return launch(B, H_in, H_out, n_expert, k_expert, hidden, router_w, router_b, experts, renormalize, out, sel, gate, status, st);
}

}  // namespace confu
