// Tree attention on CUDA cores in fp32 arithmetic, for what the tensor-core kernels do not take: fp32
// tensors, soft prompts longer than one key tile, more than 32 query heads per kv head.
//
// The R x G query rows that share a kv head are cut into blocks of M rows; a thread-block cluster of up
// to 8 CTAs works on one block, each CTA on a contiguous range of 64-key tiles, and the CTAs' partial
// results (O, m, l) meet in distributed shared memory at the end, merged in rank order.  Per tile:
//     S = Q K^T     4 rows x 64 / X keys per thread, operands read from shared memory 16 bytes at a time
//     P = exp(S - m) with the running maximum of each row (X threads share 4 rows)
//     O += P V      4 rows x D / X columns per thread
// with X = 16 threads in blocks of 64 rows, 32 in smaller ones (an SM holds one block: a block of 32 rows with
// 16 threads per row group had one warp per scheduler and a quarter of the issue slots used).
// The next tile's K and V travel (cp.async, fp32 only) while this one is worked on.
//
// fp32, one layer: B 4, 32 / 8 heads of 128, R 64, prefixes 500..4000: 323 us (20.7 TFLOP/s); B 6, 64 / 8 heads, R 120,
// prefixes 700..6000: 2.4 ms (28 TFLOP/s).  Bound by fp32 FMA issue once a machine full of blocks has several tiles each, by latency below that.
// A row of K is padded by 16 bytes so that the threads of a row group read different bank groups.
//
// Key order: [soft-prompt entries (contemplate rows only)] [prefix slots] [slots of the query rows].
#include <cooperative_groups.h>

#include <type_traits>

#include "common.cuh"

namespace confu {
namespace {

namespace cg = cooperative_groups;

constexpr int kKeys = 64;                            // keys per tile
constexpr int kMaxCluster = 8;

template <int D, int M>
struct Smem {
    float q[M][D + 4];                               // scaled
    float k[2][kKeys][D + 4];
    float v[2][kKeys][D];
    float p[M][kKeys + 4];
    float m[M], l[M];
};
template <int D, int M> __device__ __forceinline__ float (*o_tile(Smem<D, M>& sh))[D + 4]
{
    return reinterpret_cast<float (*)[D + 4]>(&sh.k[0][0][0]);       // M <= 64 rows over the K buffer once the keys are done
}

template <typename T> __device__ __forceinline__ void copy4(float* dst, const T* src);
template <> __device__ __forceinline__ void copy4<float>(float* dst, const float* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
template <> __device__ __forceinline__ void copy4<__nv_bfloat16>(float* dst, const __nv_bfloat16* src)
{
    const uint2 w = *reinterpret_cast<const uint2*>(src);
    *reinterpret_cast<float4*>(dst) = make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u),
                                                  __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xffff0000u));
}
template <typename T> __device__ __forceinline__ void store4(T* dst, float4 v);
template <> __device__ __forceinline__ void store4<float>(float* dst, float4 v) { *reinterpret_cast<float4*>(dst) = v; }
template <> __device__ __forceinline__ void store4<__nv_bfloat16>(__nv_bfloat16* dst, float4 v)
{
    __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
    *reinterpret_cast<uint2*>(dst) = make_uint2(*reinterpret_cast<uint32_t*>(&a), *reinterpret_cast<uint32_t*>(&b));
}

// max / sum over the X threads of a row group (a warp or half of one)
template <int X> __device__ __forceinline__ float group_max(float v)
{
#pragma unroll
    for (int o = X / 2; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
template <int X> __device__ __forceinline__ float group_sum(float v)
{
#pragma unroll
    for (int o = X / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// threads per row group of four rows, by rows per block
template <int M> constexpr int kGroupThreads = M == 64 ? 16 : 32;

template <typename T, int D, int M>
__global__ void __launch_bounds__(M / 4 * kGroupThreads<M>, 1) attention_generic_kernel(
    confu_dims dm, const T* __restrict__ q, const T* __restrict__ kc, const T* __restrict__ vc, const SlotMap map,
    const int32_t* __restrict__ prefix_len, const T* __restrict__ ks, const T* __restrict__ vs, const void* plan_raw,
    T* __restrict__ out, float* __restrict__ lse)
{
    constexpr int X = kGroupThreads<M>, NT = M / 4 * X;
    constexpr int kPer = kKeys / X;                  // keys of a tile per thread: tx, tx + X, ...
    constexpr int W = D / X < 4 ? D / X : 4;         // columns of O per thread: pieces of W, tx * W + i * X * W
    constexpr int kCols = D / X / W;
    using Vec = typename std::conditional<W == 4, float4, float2>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem<D, M>& sh = *reinterpret_cast<Smem<D, M>*>(smem_raw);
    cg::cluster_group cluster = cg::this_cluster();
    const int n_ranks = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int unit = (int)blockIdx.x / n_ranks, g = unit % dm.Hkv, block = unit / dm.Hkv, b = blockIdx.y;
    const int R = dm.T + dm.C, Hq = dm.Hq, Hkv = dm.Hkv, G = Hq / Hkv;
    const int tid = threadIdx.x, tx = tid % X, ty = tid / X, row0 = 4 * ty;
    // row i of the block is query row (block * M + i) / G, head (block * M + i) % G of the group
    const int n_rows = min(M, R * G - block * M);
    auto out_at = [&](int i) { const int f = block * M + i; return ((size_t)b * R + f / G) * Hq + g * G + f % G; };

    asm volatile("griddepcontrol.wait;" ::: "memory");
    PlanView pv = plan_view(const_cast<void*>(plan_raw), dm.B, dm.Hkv);
    if (pv.bad[b]) {                                 // malformed tree: zero rows (the whole cluster leaves)
        if (rank == 0) {
            for (int i = tid; i < n_rows * (D / 4); i += NT) store4(out + out_at(i / (D / 4)) * D + 4 * (i % (D / 4)), make_float4(0.f, 0.f, 0.f, 0.f));
            if (lse && tid < n_rows) lse[out_at(tid)] = 0.f;
        }
        return;
    }
    const int64_t P = prefix_len[b], n = dm.S + P + R;
    const float scale = dm.sm_scale != 0.f ? dm.sm_scale : rsqrtf((float)D);
    const int n_tiles = (int)((n + kKeys - 1) / kKeys);
    const int t0 = (int)((int64_t)rank * n_tiles / n_ranks), t1 = (int)((int64_t)(rank + 1) * n_tiles / n_ranks);

    auto load_tile = [&](int tile, int buf) {
        for (int i = tid; i < kKeys * (D / 4); i += NT) {
            const int kk = i / (D / 4), c = 4 * (i % (D / 4));
            const int64_t j = (int64_t)tile * kKeys + kk;
            if (j < n) {
                const T* kp = j < dm.S ? ks + ((size_t)j * Hkv + g) * D : kc + ((size_t)pool_slot(map, b, j - dm.S) * Hkv + g) * D;
                const T* vp = j < dm.S ? vs + ((size_t)j * Hkv + g) * D : vc + ((size_t)pool_slot(map, b, j - dm.S) * Hkv + g) * D;
                copy4(&sh.k[buf][kk][c], kp + c);
                copy4(&sh.v[buf][kk][c], vp + c);
            } else {                                 // past the last slot: never interpreted
                *reinterpret_cast<float4*>(&sh.k[buf][kk][c]) = make_float4(0.f, 0.f, 0.f, 0.f);
                *reinterpret_cast<float4*>(&sh.v[buf][kk][c]) = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (t0 < t1) load_tile(t0, 0);
    for (int i = tid; i < M * D; i += NT) sh.q[i / D][i % D] = i / D < n_rows ? to_f32(q[out_at(i / D) * D + i % D]) * scale : 0.f;

    uint64_t mask[4];
    int r_of[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        r_of[i] = min((block * M + row0 + i) / G, R - 1);
        mask[i] = pv.mask[(size_t)b * kMaxRows + r_of[i]];
    }
    float m_run[4], l_run[4], acc[4][W * kCols];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        m_run[i] = -INFINITY;
        l_run[i] = 0.f;
#pragma unroll
        for (int c = 0; c < W * kCols; ++c) acc[i][c] = 0.f;
    }
    for (int tile = t0; tile < t1; ++tile) {
        const int buf = (tile - t0) & 1;
        if (tile + 1 < t1) {
            load_tile(tile + 1, buf ^ 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        // ---- S ----
        float s[4][kPer];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < kPer; ++j) s[i][j] = 0.f;
#pragma unroll 4
        for (int d = 0; d < D; d += 4) {
            float4 a[4], k4[kPer];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4*>(&sh.q[row0 + i][d]);
#pragma unroll
            for (int j = 0; j < kPer; ++j) k4[j] = *reinterpret_cast<const float4*>(&sh.k[buf][tx + X * j][d]);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < kPer; ++j)
                    s[i][j] = fmaf(a[i].x, k4[j].x, fmaf(a[i].y, k4[j].y, fmaf(a[i].z, k4[j].z, fmaf(a[i].w, k4[j].w, s[i][j]))));
        }
        // ---- visibility: only the tiles with soft-prompt entries or with slots of the query rows need it ----
        const int64_t j0 = (int64_t)tile * kKeys;
        const bool masked = j0 < dm.S || j0 + kKeys > dm.S + P;
        if (masked) {
#pragma unroll
            for (int j = 0; j < kPer; ++j) {
                const int64_t key = j0 + tx + X * j, own = key - dm.S - P;      // own >= 0: the slot of query row `own`
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const bool vis = key < dm.S ? r_of[i] >= dm.T
                                   : own < 0    ? true
                                   : own < dm.T ? (bool)((mask[i] >> own) & 1ull)
                                                : own == r_of[i];
                    if (!vis || key >= n) s[i][j] = -INFINITY;
                }
            }
        }
        // ---- weights ----
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float top = s[i][0];
#pragma unroll
            for (int j = 1; j < kPer; ++j) top = fmaxf(top, s[i][j]);
            const float m_new = fmaxf(m_run[i], group_max<X>(top));
            const float base = m_new == -INFINITY ? 0.f : m_new;                 // nothing visible yet: weights 0
            const float alpha = expf(m_run[i] - base);
            m_run[i] = m_new;
            float sum = 0.f;
#pragma unroll
            for (int j = 0; j < kPer; ++j) {
                const float w = expf(s[i][j] - base);
                sum += w;
                sh.p[row0 + i][tx + X * j] = w;
            }
            l_run[i] = l_run[i] * alpha + group_sum<X>(sum);
#pragma unroll
            for (int c = 0; c < W * kCols; ++c) acc[i][c] *= alpha;
        }
        __syncwarp();                                // a row's weights are written and read by the same warp
        // ---- O += P V ----
        auto pv_tile = [&](auto skip_zero) {
#pragma unroll 4
            for (int kk = 0; kk < kKeys; kk += 4) {
                float4 w4[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) w4[i] = *reinterpret_cast<const float4*>(&sh.p[row0 + i][kk]);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
#pragma unroll
                    for (int c = 0; c < kCols; ++c) {
                        const Vec x = *reinterpret_cast<const Vec*>(&sh.v[buf][kk + e][W * (X * c + tx)]);
                        const float* xe = reinterpret_cast<const float*>(&x);
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const float w = e == 0 ? w4[i].x : e == 1 ? w4[i].y : e == 2 ? w4[i].z : w4[i].w;
                            if (decltype(skip_zero)::value && w == 0.f) continue;     // a slot the row does not see: whatever it holds
#pragma unroll
                            for (int z = 0; z < W; ++z) acc[i][W * c + z] = fmaf(w, xe[z], acc[i][W * c + z]);
                        }
                    }
                }
            }
        };
        if (masked) pv_tile(std::true_type());
        else pv_tile(std::false_type());
        __syncthreads();                             // the buffers may be refilled
    }
    // ---- the cluster's partial results, merged in rank order: rank c takes rows c, c + n_ranks, ... ----
    float (*o)[D + 4] = o_tile(sh);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
#pragma unroll
        for (int c = 0; c < kCols; ++c)
#pragma unroll
            for (int z = 0; z < W; ++z) o[row0 + i][W * (X * c + tx) + z] = acc[i][W * c + z];
        if (tx == 0) { sh.m[row0 + i] = m_run[i]; sh.l[row0 + i] = l_run[i]; }
    }
    cluster.sync();
    const int mx = tid & 15;                         // 16 threads to a row, 16-byte pieces
    constexpr int kPieces = D / 64;
    for (int i = rank * (NT / 16) + (tid >> 4); i < n_rows; i += n_ranks * (NT / 16)) {
        float mm = -INFINITY;
        for (int c = 0; c < n_ranks; ++c) mm = fmaxf(mm, *cluster.map_shared_rank(&sh.m[i], c));
        float4 sum[kPieces];
        float l = 0.f;
#pragma unroll
        for (int c = 0; c < kPieces; ++c) sum[c] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int c = 0; c < n_ranks; ++c) {
            const float m_c = *cluster.map_shared_rank(&sh.m[i], c);
            const float w = expf(m_c - mm);          // a rank that saw no key of the row: 0 (and 0 times its sums; NaN if it saw only NaN)
            l = fmaf(w, *cluster.map_shared_rank(&sh.l[i], c), l);
#pragma unroll
            for (int cc = 0; cc < kPieces; ++cc) {
                const float4 x = *reinterpret_cast<const float4*>(cluster.map_shared_rank(&o[i][64 * cc + 4 * mx], c));
                sum[cc].x = fmaf(w, x.x, sum[cc].x); sum[cc].y = fmaf(w, x.y, sum[cc].y);
                sum[cc].z = fmaf(w, x.z, sum[cc].z); sum[cc].w = fmaf(w, x.w, sum[cc].w);
            }
        }
#pragma unroll
        for (int cc = 0; cc < kPieces; ++cc)
            store4(out + out_at(i) * D + 64 * cc + 4 * mx, make_float4(sum[cc].x / l, sum[cc].y / l, sum[cc].z / l, sum[cc].w / l));
        if (lse && mx == 0) lse[out_at(i)] = mm + logf(l);
    }
    cluster.sync();                                  // no CTA leaves while another reads its shared memory
}

template <typename T, int D, int M>
cudaError_t launch_m(int ranks, const confu_dims& d, const void* q, const void* kc, const void* vc, const SlotMap& map,
                     const int32_t* prefix_len, const void* ks, const void* vs, const void* plan, void* out, float* lse,
                     cudaStream_t st)
{
    const size_t smem = sizeof(Smem<D, M>);
    static OncePerDevice attr_done;
    cudaError_t e = attr_done.run([&] {
        return cudaFuncSetAttribute(attention_generic_kernel<T, D, M>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    });
    if (e != cudaSuccess) return e;
    const int blocks = ((d.T + d.C) * (d.Hq / d.Hkv) + M - 1) / M * d.Hkv;
    cudaLaunchAttribute attrs[2];
    attrs[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attrs[0].val.programmaticStreamSerializationAllowed = 1;
    attrs[1].id = cudaLaunchAttributeClusterDimension;
    attrs[1].val.clusterDim.x = (unsigned)ranks;
    attrs[1].val.clusterDim.y = attrs[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(ranks * blocks), (unsigned)d.B);     // (x holds 2^31 of them, y 65535)
    cfg.blockDim = dim3(M / 4 * kGroupThreads<M>);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attrs;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, attention_generic_kernel<T, D, M>, d, (const T*)q, (const T*)kc, (const T*)vc, map, prefix_len,
                              (const T*)ks, (const T*)vs, plan, (T*)out, lse);
}

// Rows per block and CTAs per cluster: the pair with the shortest estimated launch.  A CTA's work is rows x
// keys, that is M / ranks, at a cost per row of 4 : 5 : 8 (a block of 64 rows uses each byte it reads for 64 rows,
// one of 16 has a warp per scheduler).  An SM holds one CTA, and because a cluster stays inside a group of
// neighbouring SMs only 15 clusters of 8, or 33 of 4, run at once on 148 SMs: a sixteenth cluster of 8 would wait
// for a second wave (fp32, B 1, 8 heads of 128, R 64, prefix 2000: 16 clusters of 8 with 32 rows 94 us, this choice 61 us).
template <typename T, int D>
cudaError_t launch_d(int sm_count, const confu_dims& d, const void* q, const void* kc, const void* vc, const SlotMap& map,
                     const int32_t* prefix_len, const void* ks, const void* vs, const void* plan, void* out, float* lse,
                     cudaStream_t st)
{
    if (d.B == 0) return cudaSuccess;
    const int rows = (d.T + d.C) * (d.Hq / d.Hkv);
    int best_m = 16, best_ranks = 1;
    double best = 0.;
    for (int m = 64; m >= 16; m /= 2) {
        if (m > 16 && rows <= m / 2) continue;
        const int64_t blocks = (int64_t)((rows + m - 1) / m) * d.Hkv * d.B;
        for (int ranks = kMaxCluster; ranks >= 1; ranks /= 2) {
            const int64_t cap = ranks == 8 ? sm_count * 13 / 16 : ranks == 4 ? sm_count * 8 / 9 : sm_count;
            const double waves = (double)((blocks * ranks + cap - 1) / cap);
            const double cost = waves * m / ranks * (m == 64 ? 4 : m == 32 ? 5 : 8);
            if (best == 0. || cost < best) { best = cost; best_m = m; best_ranks = ranks; }
        }
    }
    auto launch = best_m == 64 ? launch_m<T, D, 64> : best_m == 32 ? launch_m<T, D, 32> : launch_m<T, D, 16>;
    return launch(best_ranks, d, q, kc, vc, map, prefix_len, ks, vs, plan, out, lse, st);
}

}  // namespace

cudaError_t launch_attention_generic(const Ctx* ctx, const confu_dims& d, const void* q, const void* k_cache,
                                     const void* v_cache, const SlotMap& map, const int32_t* prefix_len,
                                     const void* k_soft, const void* v_soft, const void* plan, void* out,
                                     float* lse, cudaStream_t st)
{
    auto launch = d.kv_dtype == CONFU_F32 ? (d.D == 64 ? launch_d<float, 64> : launch_d<float, 128>)
                                          : (d.D == 64 ? launch_d<__nv_bfloat16, 64> : launch_d<__nv_bfloat16, 128>);
    return launch(ctx->sm_count, d, q, k_cache, v_cache, map, prefix_len, k_soft, v_soft, plan, out, lse, st);
}

}  // namespace confu
