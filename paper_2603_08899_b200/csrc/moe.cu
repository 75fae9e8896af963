// Contemplate-token embedding as a mixture of expert embeddings: router linear layer on the hidden
// state of the most recently accepted token, softmax over the experts, the k largest scores, sum of
// the chosen experts' embeddings weighted by their gating scores.
//
// Two forms.  Where the router is small for the batch, one CTA per sequence (or four): see con_embedding_row_kernel.  Else a
// cluster of 8 CTAs per 1, 2 or 4 sequences (the more sequences in the call, the more share a cluster and
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

template <typename T> __device__ __forceinline__ uint4 raw_vec(const T* p) { return *reinterpret_cast<const uint4*>(p); }
template <typename T> __device__ __forceinline__ void unpack(const uint4& v, float (&x)[Vec16<T>::n]) { load_vec(reinterpret_cast<const T*>(&v), x); }

__device__ __forceinline__ void store_vec(float* p, const float (&x)[4]) { *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]); }
__device__ __forceinline__ void store_vec(__nv_bfloat16* p, const float (&x)[8])
{
    __nv_bfloat162 h[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) h[j] = __floats2bfloat162_rn(x[2 * j], x[2 * j + 1]);
    *reinterpret_cast<uint4*>(p) = *reinterpret_cast<const uint4*>(h);
}

// Scores of NS sequences (from b0 on) as they lie in a CTA's shared memory, and what is made of them.
template <int NS>
struct Scores {
    float score[NS][kMoeMaxExperts];
    int sel[NS][kMoeMaxK];
    float w[NS][kMoeMaxK];
    int bad[NS];
};

// Softmax, selection, and the weighted sum of the chosen embeddings: this CTA's share, the rank-th of n, of the columns.
template <typename T, int NS, int NT>
__device__ __forceinline__ void mix(Scores<NS>& sh, int rank, int n, int b0, int B, int H_out, int n_expert, int k_expert, const T* __restrict__ experts,
                                    int renormalize, T* __restrict__ out, int32_t* __restrict__ sel, float* __restrict__ gate,
                                    int32_t* __restrict__ status)
{
    constexpr int kVec = Vec16<T>::n;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool vec_out = H_out % kVec == 0;
    // ---- softmax and the k largest scores (warp s: sequence s) ----
    if (warp < NS && b0 + warp < B) {
        float* score = sh.score[warp];
        const int b = b0 + warp;
        const bool writer = rank == 0;
        float m = -INFINITY;
        bool bad = false;
        for (int e = lane; e < n_expert; e += 32) {
            m = fmaxf(m, score[e]);
            bad = bad || !(fabsf(score[e]) <= 3.0e38f);
        }
        bad = __any_sync(0xffffffffu, bad);
        if (lane == 0) sh.bad[warp] = bad;
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
                    sh.sel[warp][k] = be;
                    sh.w[warp][k] = bv * inv_z;
                    score[be] = -1.f;
                }
                wsum += bv * inv_z;
                __syncwarp();
            }
            if (renormalize && lane < k_expert) sh.w[warp][lane] = sh.w[warp][lane] / wsum;
            __syncwarp();
            if (writer && lane < k_expert) {
                if (sel) sel[(size_t)b * k_expert + lane] = sh.sel[warp][lane];
                if (gate) gate[(size_t)b * k_expert + lane] = sh.w[warp][lane];
            }
        }
    }
    __syncthreads();

    // ---- weighted sum of the chosen embeddings: this CTA's share of the columns (all zero for a bad sequence) ----
    const int unit = vec_out ? kVec : 1, n_unit = H_out / unit;
    const int u0 = (int)((int64_t)rank * n_unit / n), n_cols = (int)((int64_t)(rank + 1) * n_unit / n) - u0;
    for (int i = tid; i < NS * n_cols; i += NT) {
        const int s = i / n_cols, j = (u0 + i % n_cols) * unit;
        if (b0 + s >= B) break;
        T* o = out + (size_t)(b0 + s) * H_out + j;
        const int n_k = sh.bad[s] ? 0 : k_expert;
        if (vec_out) {
            float acc[kVec];
#pragma unroll
            for (int v = 0; v < kVec; ++v) acc[v] = 0.f;
            for (int k = 0; k < n_k; ++k) {
                float x[kVec];
                load_vec(experts + (size_t)sh.sel[s][k] * H_out + j, x);
                const float w = sh.w[s][k];
#pragma unroll
                for (int v = 0; v < kVec; ++v) acc[v] = fmaf(w, x[v], acc[v]);
            }
            store_vec(o, acc);
        } else {
            float acc = 0.f;
            for (int k = 0; k < n_k; ++k) acc = fmaf(sh.w[s][k], to_f32(experts[(size_t)sh.sel[s][k] * H_out + j]), acc);
            o[0] = from_f32<T>(acc);
        }
    }
}

template <typename T, int NS>
__global__ void __launch_bounds__(kMoeThreads) con_embedding_kernel(
    int B, int H_in, int H_out, int n_expert, int k_expert, const T* __restrict__ hidden, const T* __restrict__ router_w,
    const T* __restrict__ router_b, const T* __restrict__ experts, int renormalize, T* __restrict__ out,
    int32_t* __restrict__ sel, float* __restrict__ gate, int32_t* __restrict__ status)
{
    constexpr int kVec = Vec16<T>::n, kWarps = kMoeThreads / 32;
    __shared__ Scores<NS> sh;
    __shared__ float s_part[NS][kWarps];             // parts of dot products that several warps share
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int b0 = (int)(blockIdx.x / kMoeCluster) * NS, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool vec_in = H_in % kVec == 0;

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
                *cluster.map_shared_rank(&sh.score[s][expert], peer) = sc;
            }
        }
        __syncthreads();
    }
    if (first_round) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");       // no expert of its own
    cluster.sync();

    mix<T, NS, kMoeThreads>(sh, rank, kMoeCluster, b0, B, H_out, n_expert, k_expert, experts, renormalize, out, sel, gate, status);
}

// The same by one CTA of NT threads per NS sequences: no cluster to set up and wait for.  A warp takes a dot product, or, where
// there are fewer of them than warps, a part of one of at least 32 vectors.
template <typename T, int NS, int NT>
__global__ void __launch_bounds__(NT) con_embedding_row_kernel(
    int B, int H_in, int H_out, int n_expert, int k_expert, const T* __restrict__ hidden, const T* __restrict__ router_w,
    const T* __restrict__ router_b, const T* __restrict__ experts, int renormalize, T* __restrict__ out,
    int32_t* __restrict__ sel, float* __restrict__ gate, int32_t* __restrict__ status)
{
    constexpr int kVec = Vec16<T>::n, kWarps = NT / 32;
    __shared__ Scores<NS> sh;
    __shared__ float s_part[NS][kWarps];
    const int b0 = (int)blockIdx.x * NS, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool vec_in = H_in % kVec == 0;

    asm volatile("griddepcontrol.wait;" ::: "memory");
    int lp = 0;                                      // parts per dot product: 2^lp
    while ((2 * n_expert << lp) <= kWarps && H_in / kVec >= 64 << lp) ++lp;
    const T* h[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) h[s] = hidden + (size_t)min(b0 + s, B - 1) * H_in;
    for (int item = warp; item < n_expert << lp; item += kWarps) {
        const int e = item >> lp, part = item & ((1 << lp) - 1);
        const T* w = router_w + (size_t)e * H_in;
        float acc[NS];
#pragma unroll
        for (int s = 0; s < NS; ++s) acc[s] = 0.f;
        if (vec_in) {
            auto add = [&](const uint4& wv, const uint4 (&hv)[NS]) {
                float y[kVec], x[kVec];
                unpack<T>(wv, y);
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    unpack<T>(hv[s], x);
#pragma unroll
                    for (int j = 0; j < kVec; ++j) acc[s] = fmaf(x[j], y[j], acc[s]);
                }
            };
            // (four vectors of each in flight per lane: left to itself the compiler keeps two or three)
            constexpr int kFly = NS == 1 ? 4 : 2;
            const int n_vec = H_in / kVec, v1 = (int)((int64_t)(part + 1) * n_vec >> lp);
            int v = (int)((int64_t)part * n_vec >> lp) + lane;
            for (; v + 32 * (kFly - 1) < v1; v += 32 * kFly) {
                uint4 wv[kFly], hv[kFly][NS];
#pragma unroll
                for (int u = 0; u < kFly; ++u) {
                    wv[u] = raw_vec(w + (size_t)(v + 32 * u) * kVec);
#pragma unroll
                    for (int s = 0; s < NS; ++s) hv[u][s] = raw_vec(h[s] + (size_t)(v + 32 * u) * kVec);
                }
#pragma unroll
                for (int u = 0; u < kFly; ++u) add(wv[u], hv[u]);
            }
            for (; v < v1; v += 32) {
                uint4 hv[NS];
#pragma unroll
                for (int s = 0; s < NS; ++s) hv[s] = raw_vec(h[s] + (size_t)v * kVec);
                add(raw_vec(w + (size_t)v * kVec), hv);
            }
        } else {
            const int i1 = (int)((int64_t)(part + 1) * H_in >> lp);
            for (int i = (int)((int64_t)part * H_in >> lp) + lane; i < i1; i += 32)
#pragma unroll
                for (int s = 0; s < NS; ++s) acc[s] = fmaf(to_f32(h[s][i]), to_f32(w[i]), acc[s]);
        }
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            acc[s] = warp_sum(acc[s]);
            if (lane == 0) {
                if (lp == 0) sh.score[s][e] = acc[s] + (router_b ? to_f32(router_b[e]) : 0.f);
                else s_part[s][warp] = acc[s];       // (then there is one round: an item per warp)
            }
        }
    }
    __syncthreads();
    if (lp > 0) {
        if (tid < NS * n_expert) {
            const int s = tid % NS, e = tid / NS;
            float sc = 0.f;
            for (int q = 0; q < 1 << lp; ++q) sc += s_part[s][(e << lp) + q];
            sh.score[s][e] = sc + (router_b ? to_f32(router_b[e]) : 0.f);
        }
        __syncthreads();
    }
    mix<T, NS, NT>(sh, 0, 1, b0, B, H_out, n_expert, k_expert, experts, renormalize, out, sel, gate, status);
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

template <typename T, int NS, int NT>
static cudaError_t launch_row(int B, int H_in, int H_out, int n_expert, int k_expert, const void* hidden, const void* router_w,
                              const void* router_b, const void* experts, int renormalize, void* out, int32_t* sel, float* gate,
                              int32_t* status, cudaStream_t st)
{
    return launch_pdl(con_embedding_row_kernel<T, NS, NT>, dim3((unsigned)((B + NS - 1) / NS)), dim3(NT), st, B, H_in, H_out, n_expert,
                      k_expert, (const T*)hidden, (const T*)router_w, (const T*)router_b, (const T*)experts, renormalize, (T*)out, sel,
                      gate, status);
}

// Which form is the faster one, by a line fitted to either side (us; n experts, H: size of a row in units of two bytes; measured
// for H 64..12288, n 1..256, B 1..1024.  Cluster against row form: B 1, n 4, H 64 4.4 / 3.0, n 64, H 12288 7.1 / 24.7; B 128, n 16,
// H 2400 6.5 / 5.0, n 64, H 4096 9.7 / 12.2; B 1024, n 16, H 768 42 / 6.6).  32 clusters run side by side, so with one
// per four sequences a batch of 1024 goes in eight turns; of the row form three CTAs of 512 threads or six of 256 share an SM.
static constexpr int kWideRows = 3 * 148, kNarrowRows = 6 * 148;
static bool row_form(int B, double n, double H)
{
    const double cluster = B <= 16   ? 4.3 + n * (0.0125 + 3.2e-6 * H)
                           : B <= 32 ? 4.6 + n * (0.0145 + 7.2e-6 * H)
                                     : (double)((B + 127) / 128) * (5.3 + n * (0.019 + 1.32e-5 * H));
    const double row = B <= kWideRows     ? 3.2 + 6e-5 * H + n * (0.045 + 2.2e-5 * H) * (B <= 148 ? 1. : B <= 296 ? 1.7 : 2.5)
                       : B <= kNarrowRows ? 3.2 + 1.5e-4 * H + n * (0.12 + 7.5e-5 * H) * (B <= 512 ? 1. : B / 512.)
                                          : (double)((B + 2367) / 2368) * (3.4 + 4e-4 * H + n * (0.1 + 1.67e-4 * H));
    return row < 0.92 * cluster;
}

cudaError_t launch_con_embedding(int B, int H_in, int H_out, int n_expert, int k_expert, int dtype, const void* hidden,
                                 const void* router_w, const void* router_b, const void* experts, int renormalize,
                                 void* out, int32_t* sel, float* gate, int32_t* status, cudaStream_t st)
{
    if (B == 0) return cudaSuccess;
    const bool f32 = dtype == CONFU_F32;
    auto launch = f32 ? launch_ns<float, 1> : launch_ns<__nv_bfloat16, 1>;
    if (row_form(B, n_expert, f32 ? 2. * H_in : H_in))
        launch = B <= kWideRows     ? (f32 ? launch_row<float, 1, 512> : launch_row<__nv_bfloat16, 1, 512>)
                 : B <= kNarrowRows ? (f32 ? launch_row<float, 1, 256> : launch_row<__nv_bfloat16, 1, 256>)
                                    : (f32 ? launch_row<float, 4, 256> : launch_row<__nv_bfloat16, 4, 256>);
    // one sequence per cluster while that leaves SMs free, then two, then four: the router is read once per cluster
    // (B 16: 9.2 us, B 17: 10.2, B 32: 11.7, B 33: 12.7, B 64: 17.1)
    else if (B > 16)
        launch = B <= 32 ? (f32 ? launch_ns<float, 2> : launch_ns<__nv_bfloat16, 2>)
                         : (f32 ? launch_ns<float, 4> : launch_ns<__nv_bfloat16, 4>);
    return launch(B, H_in, H_out, n_expert, k_expert, hidden, router_w, router_b, experts, renormalize, out, sel, gate, status, st);
}

}  // namespace confu
