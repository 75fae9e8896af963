// Row statistics over the vocabulary and the host side of the acceptance call.
//
//   row_stats_kernel   one streaming pass over every logit row of the target and draft matrices:
//                      per row chunk the running max, the sum of exp((x - max)/temperature) (online
//                      softmax), the lowest index of the max, and a non-finite flag.  HBM bound.
// The walks that use them (or compute their own on demand) are in accept_walk.cu.
#include <limits.h>

#include "accept.cuh"

namespace confu {

constexpr int kEpt = 8;                                   // consecutive vocabulary entries per thread and load

size_t accept_workspace_bytes(int B, int T, int /*V*/)
{
    return (size_t)2 * B * T * kStatChunksMax * sizeof(RowStat);
}

template <typename T>
__device__ __forceinline__ void load8(const T* __restrict__ row, int i0, int V, float (&x)[kEpt])
{
    if (i0 + kEpt <= V) {
        if constexpr (sizeof(T) == 2) {
            const uint4 v = *reinterpret_cast<const uint4*>(row + i0);
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                x[2 * j] = __uint_as_float(w[j] << 16);
                x[2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u);
            }
        } else {
            const float4 a = *reinterpret_cast<const float4*>(row + i0);
            const float4 c = *reinterpret_cast<const float4*>(row + i0 + 4);
            x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
            x[4] = c.x; x[5] = c.y; x[6] = c.z; x[7] = c.w;
        }
    } else {
#pragma unroll
        for (int j = 0; j < kEpt; ++j) x[j] = (i0 + j < V) ? to_f32(row[i0 + j]) : -INFINITY;
    }
}

// ---------------------------------------------------------------------------------------------
// K3: row statistics
// ---------------------------------------------------------------------------------------------
// A lane's running sum, with what its additions have lost so far (Kahan's summation).  A warp that has a row or a chunk of one to itself
// makes hundreds of them, and beside a weight of 1 each can drop half a unit in the last place: fp32, V 151936, 16 sequences
// of 60 rows, one logit 18.75 above all others: 1.1e-5 of a row's sum (256 threads to a chunk: 4.5e-6), so 1.2e-7; deviation 5: root mean
// square 3.3e-7 (1.7e-7), so 4.8e-8; bf16 3.0e-6 (1.2e-6) and 9.8e-8 (3.3e-7), so 1.1e-7 and 5.2e-8.  (That ex2 flushes weights below
// 2^-126 of the lane's largest changes no sum: exp2f gave the same bits.)
struct Sum {
    float s = 0.f, over = 0.f;                       // over: by how much s is above the exact sum
    __device__ __forceinline__ void add(float a)
    {
        const float y = a - over, t = s + y;
        over = (t - s) - y;
        s = t;
    }
    __device__ __forceinline__ void scale(float f) { s *= f; over *= f; }
};

// N vectors of eight bf16 logits (16 bytes, starting at index ib and kStep apart) folded into a thread's running
// statistics: maximum m, non-finite flag, and what the walk behind it reads: sampling the sum of exp2((x - m) * k2), greedy the lowest
// index arg of the maximum.  (A search for the index is long, and with 32 lanes and a chunk of a few batches some lane finds a
// new maximum in nearly every one.)  Maximum and minimum are taken on packed bf16 pairs with NaN propagation, so one
// comparison of each against the finite range finds NaN and both infinities.  The exponent is (x - m) * k2, the difference first: as one
// fused operation with m * k2 it is wrong where that product leaves fp32 (a row mostly masked with -2.5e38) or is rounded by
// more than the exponents (temperature 1e-9), and no faster (B 32, T 60, V 128256: 217.4 us with the walk, 214.7 so).
template <int N, bool kGreedy>
__device__ __forceinline__ void stats_bf16(const uint4 (&v)[N], int ib, int step, float k2, float& m, Sum& sum, int& arg, int& flag)
{
    uint32_t w[4 * N];
#pragma unroll
    for (int u = 0; u < N; ++u) { w[4 * u] = v[u].x; w[4 * u + 1] = v[u].y; w[4 * u + 2] = v[u].z; w[4 * u + 3] = v[u].w; }
    auto h = [&](int j) { return *reinterpret_cast<const __nv_bfloat162*>(&w[j]); };
    __nv_bfloat162 mx2 = h(0), mn2 = h(0);
#pragma unroll
    for (int j = 1; j < 4 * N; ++j) { mx2 = __hmax2_nan(mx2, h(j)); mn2 = __hmin2_nan(mn2, h(j)); }
    const float hi0 = __low2float(mx2), hi1 = __high2float(mx2), lo0 = __low2float(mn2), lo1 = __high2float(mn2);
    if (!(hi0 <= 3.0e38f && hi1 <= 3.0e38f && lo0 >= -3.0e38f && lo1 >= -3.0e38f)) flag = 1;
    const float cm = fmaxf(hi0, hi1);
    if (cm > m) {
        if (!kGreedy) sum.scale(exp2f((m - cm) * k2));   // (with ex2 the kernel spills registers)
        m = cm;
        if (kGreedy) {                                   // the first element equal to it
#pragma unroll
            for (int j = 8 * N - 1; j >= 0; --j) {
                const float x = __uint_as_float((j & 1) ? (w[j >> 1] & 0xffff0000u) : (w[j >> 1] << 16));
                if (x == cm) arg = ib + (j >> 3) * step + (j & 7);
            }
        }
    }
    if (kGreedy) return;
    uint64_t acc[2] = {f2_pack(0.f, 0.f), f2_pack(0.f, 0.f)};
    const uint64_t k22 = f2_pack(k2, k2), nm2 = f2_pack(-m, -m);
#pragma unroll
    for (int j = 0; j < 4 * N; ++j) {
        float x0, x1;
        f2_unpack(f2_mul(f2_add(f2_pack(__uint_as_float(w[j] << 16), __uint_as_float(w[j] & 0xffff0000u)), nm2), k22), x0, x1);
        acc[j & 1] = f2_add(acc[j & 1], f2_pack(ex2(x0), ex2(x1)));
    }
    float a0, a1;
    f2_unpack(f2_add(acc[0], acc[1]), a0, a1);
    sum.add(a0 + a1);
}

// A warp's statistics in every lane: the maximum (as an integer of the same order: one reduction instruction), the sums
// brought to it once, the lowest index that has it.  Values that are not there are (-inf, 0, INT_MAX).
template <bool kGreedy>
__device__ __forceinline__ void warp_stats(float k2, float& m, float& s, int& arg, int& flag)
{
    auto order = [](int i) { return i ^ ((i >> 31) & 0x7fffffff); };
    const float M = __int_as_float(order(__reduce_max_sync(0xffffffffu, order(__float_as_int(m)))));
    if (kGreedy) arg = __reduce_min_sync(0xffffffffu, m == M ? arg : INT_MAX);
    else s = warp_sum(m == M ? s : s * ex2((m - M) * k2));
    flag = __any_sync(0xffffffffu, flag);
    m = M;
}

// W warps work on an item, a chunk of a row, then on the next; the launch is as many warps as the GPU holds at once.  HBM bound: what
// counts is that enough loads are in flight (four vectors a lane) and that nothing else takes time: rounds of equal items that come
// out even (see the launch) and a handful of reductions at the end of an item.
constexpr int kStatWarps = 8;
constexpr int kStatBlocks = 5;                            // per SM
template <typename T, int W, bool kGreedy>
__global__ void __launch_bounds__(32 * kStatWarps, kStatBlocks) row_stats_kernel(const T* __restrict__ tl, const T* __restrict__ dl, int V, int n_rows,
                                                                       int items, int nch, int chunk_elems, float k2,
                                                                       RowStat* __restrict__ stats)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int leader = warp / W * W;
    __shared__ float sm[2][kStatWarps], ss[2][kStatWarps];
    __shared__ int sa[2][kStatWarps], sf[2][kStatWarps];
    int turn = 0;
    for (int item = blockIdx.x * (kStatWarps / W) + warp / W; item < items; item += gridDim.x * (kStatWarps / W)) {
        const int both = item / nch, chunk = item - both * nch, mat = both >= n_rows, row = both - (mat ? n_rows : 0);
        // counted from the 16-byte boundary at or before the row's first entry, which has place `shift` (a chunk that is left without
        // entries of its row writes the statistics of none)
        const T* first = (mat == 0 ? tl : dl) + (size_t)row * V;
        const int shift = (int)((reinterpret_cast<uintptr_t>(first) & 15u) / sizeof(T));
        const T* base = first - shift;
        const int lo = chunk * chunk_elems, hi = min(V + shift, lo + chunk_elems);
        const int tid = (warp % W) * 32 + lane;
        constexpr int kStep = W * 32 * kEpt;

        float m = -INFINITY;
        Sum sum;
        int arg = INT_MAX, flag = 0;

        int i0 = lo + tid * kEpt;
        if (i0 < shift) {                                    // the vector that holds the row's first entries
            for (int i = shift; i < min(kEpt, hi); ++i) {
                const float v = to_f32(base[i]);
                if (!(fabsf(v) <= 3.0e38f)) flag = 1;
                if (v > m) { if (!kGreedy) sum.scale(ex2((m - v) * k2)); m = v; arg = i; }
                if (!kGreedy) sum.add(ex2((v - m) * k2));
            }
            i0 += kStep;
        }
        if constexpr (sizeof(T) == 2) {
            for (; i0 + 3 * kStep + kEpt <= hi; i0 += 4 * kStep) {
                uint4 v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = *reinterpret_cast<const uint4*>(base + i0 + u * kStep);
                stats_bf16<4, kGreedy>(v, i0, kStep, k2, m, sum, arg, flag);
            }
        }
        for (; i0 < hi; i0 += 2 * kStep) {
            float x[2][kEpt];
            const int i1 = i0 + kStep;
            if constexpr (sizeof(T) == 2) {
                // bf16 rows, both 8-element vectors whole: packed path (about 4 instructions per logit)
                if (i1 + kEpt <= hi) {
                    const uint4 v[2] = {*reinterpret_cast<const uint4*>(base + i0), *reinterpret_cast<const uint4*>(base + i1)};
                    stats_bf16<2, kGreedy>(v, i0, kStep, k2, m, sum, arg, flag);
                    continue;
                }
            }
            load8(base, i0, hi, x[0]);
            if (i1 < hi) load8(base, i1, hi, x[1]);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int ib = u == 0 ? i0 : i1;
                if (ib >= hi) break;
                float lm = x[u][0];
#pragma unroll
                for (int j = 1; j < kEpt; ++j) lm = fmaxf(lm, x[u][j]);
                if (lm > m) {
                    if (!kGreedy) sum.scale(ex2((m - lm) * k2));
                    m = lm;
                    if (kGreedy) {
#pragma unroll
                        for (int j = kEpt - 1; j >= 0; --j)
                            if (x[u][j] == lm) arg = ib + j;
                    }
                }
                float acc = 0.f;
#pragma unroll
                for (int j = 0; j < kEpt; ++j) {
                    const float v = x[u][j];
                    if (ib + j < hi && !(fabsf(v) <= 3.0e38f)) flag = 1;
                    if (!kGreedy) acc += ex2((v - m) * k2);                          // out-of-range entries are -inf -> 0
                }
                if (!kGreedy) sum.add(acc);
            }
        }
        float s = sum.s - sum.over;
        warp_stats<kGreedy>(k2, m, s, arg, flag);
        if constexpr (W > 1) {
            if (lane == 0) { sm[turn][warp] = m; ss[turn][warp] = s; sa[turn][warp] = arg; sf[turn][warp] = flag; }
            asm volatile("bar.sync %0, %1;" ::"r"(1 + warp / W), "r"(32 * W) : "memory");
            m = -INFINITY; s = 0.f; arg = INT_MAX; flag = 0;
            if (lane < W) { m = sm[turn][leader + lane]; s = ss[turn][leader + lane]; arg = sa[turn][leader + lane]; flag = sf[turn][leader + lane]; }
            if (warp == leader) warp_stats<kGreedy>(k2, m, s, arg, flag);
            turn ^= 1;                               // (the next item's are written elsewhere: one barrier an item)
        }
        if (lane == 0 && warp == leader) {
            RowStat r;
            r.m = m; r.s = s; r.arg = arg == INT_MAX ? arg : arg - shift; r.flag = flag;
            stats[(size_t)both * kStatChunksMax + chunk] = r;
        }
    }
}

// The statistics of all rows.  Chunks per row and warps per chunk: so that the rounds that a warp makes come out even, by what a round
// takes it: its share of the entries, the end of an item (some 256 entries' time), and a last batch that is not whole: its vectors
// come a few at a time, each after the one before, half a batch's time, or a whole one's where other items wait.  So chunks of
// whole batches are on offer too; several warps to a chunk keep less in flight (5/4).  With the walk behind it, us, chunks of any length ->
// so: bf16, T 64, V 128256, B 31 240 -> 217, T 45, V 90000, B 40 177 -> 162, T 60, V 128256, B 3 39.4 -> 35.7, 8 73.0 -> 67.9, 16 117 -> 113;
// V 32000, B 32 81.3 -> 78.7; greedy, T 64, V 12000, B 32 13.6 -> 10.2; fp32, greedy, T 64, V 151936, B 5 44.3 -> 35.7.  Against a block
// of 8 warps per row or chunk, maximum's index and sum both, parts merged as a tree: 217, 164, 40.2, 78.0, 123, 84.3, 16.9, 42.3.
// Blocks per SM (registers against warps) 3, 4, 5, 6, 8 at B 16: 132, 132, 119, 126, 134; the next four vectors loaded ahead: 120 -> 132.
template <typename T, bool kGreedy>
static cudaError_t launch_stats(int sm_count, int n_rows, int nmat, int V, const T* tl, const T* dl, float k2, RowStat* stats, int& nch, cudaStream_t st)
{
    const int all = ((size_t)V * sizeof(T)) % 16 == 0 ? V : V + 16 / (int)sizeof(T) - 1;      // places of a row, whatever its shift
    const int64_t rows = (int64_t)n_rows * nmat, room = (int64_t)sm_count * kStatBlocks * kStatWarps;
    constexpr int kBatch = 32 * kEpt * (sizeof(T) == 2 ? 4 : 2);                             // entries that a warp loads at a time
    int W = 1, chunk_elems = 0;
    int64_t least = INT64_MAX;
    auto offer = [&](int share, int w, bool whole) {
        const int unit = whole ? kBatch : 16, n = (share + unit - 1) / unit * unit;
        const int64_t parts = (all + n - 1) / n, groups = room / w, rounds = (rows * parts + groups - 1) / groups;
        const int tail = (rounds > 1 ? 2 : n < kBatch ? 0 : 1) * kBatch / 2;
        const int64_t cost = rounds * (w > 1 ? n / w * 5 / 4 + 512 : whole ? n + 512 : n + 256 + tail);
        if (cost < least && (parts == 1 || rows * parts < (1 << 30))) { least = cost; nch = (int)parts; W = w; chunk_elems = n; }
    };
    for (int c = 1; c <= kStatChunksMax; ++c) {
        const int share = (all + c - 1) / c;
        for (int w = 1; w <= kStatWarps; w *= 2) offer(share, w, false);
        offer(share, 1, true);
    }
    const int64_t items = rows * nch, per = kStatWarps / W, want = (items + per - 1) / per, most = (int64_t)sm_count * kStatBlocks;
    const int64_t blocks = want < most ? want : most;
    auto kernel = W == 1 ? row_stats_kernel<T, 1, kGreedy> : W == 2 ? row_stats_kernel<T, 2, kGreedy> : W == 4 ? row_stats_kernel<T, 4, kGreedy> : row_stats_kernel<T, 8, kGreedy>;
    return launch_pdl(kernel, dim3((unsigned)blocks), dim3(32 * kStatWarps), st, tl, dl, V, n_rows, (int)items, nch, chunk_elems, k2, stats);
}

template <typename T>
static cudaError_t launch_accept_t(int sm_count, int B, int Tn, int C, int V, const void* tl, const void* dl, const int32_t* tokens,
                                   const int32_t* parent, const int32_t* con_owner, const float* uniforms,
                                   float temperature, int mode_flags, int32_t* accept_len, int32_t* path,
                                   int32_t* next_token, int32_t* future_row, int32_t* counters, void* workspace,
                                   int32_t* status, cudaStream_t st)
{
    if (B == 0) return cudaSuccess;
    const int mode = mode_flags & 0xff, lazy = (mode_flags & CONFU_ACCEPT_LAZY) ? 1 : 0;
    const bool greedy = !(temperature > 0.f);
    const int n_rows = B * Tn;
    const int nmat = greedy ? 1 : 2;
    int nch = 0;
    const float k2 = (greedy ? 1.f : 1.f / temperature) * kLog2e;
    RowStat* stats = (RowStat*)workspace;
    if (!lazy) {
        const cudaError_t e = greedy ? launch_stats<T, true>(sm_count, n_rows, nmat, V, (const T*)tl, (const T*)dl, k2, stats, nch, st)
                                     : launch_stats<T, false>(sm_count, n_rows, nmat, V, (const T*)tl, (const T*)dl, k2, stats, nch, st);
        if (e != cudaSuccess) return e;
    }
    return launch_walk(sizeof(T) == 4 ? CONFU_F32 : CONFU_BF16, B, Tn, C, V, tl, dl, tokens, parent, con_owner, uniforms, temperature,
                       mode, nch, lazy ? nullptr : stats, accept_len, path, next_token, future_row, counters, status, st);
}

// SM count of the current device, asked once per device (for callers without a context).
static cudaError_t current_sm_count(int& n)
{
    static int cached[OncePerDevice::kMaxDevices] = {};
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= OncePerDevice::kMaxDevices) return cudaErrorInvalidDevice;
    if (!cached[dev]) {
        int v = 0;
        e = cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        cached[dev] = v;
    }
    n = cached[dev];
    return cudaSuccess;
}

cudaError_t launch_accept(const Ctx* ctx, int B, int T, int C, int V, int logit_dtype, const void* tl, const void* dl,
                          const int32_t* tokens, const int32_t* parent, const int32_t* con_owner,
                          const float* uniforms, float temperature, int sibling_mode, int32_t* accept_len,
                          int32_t* path, int32_t* next_token, int32_t* future_row, int32_t* counters,
                          void* workspace, int32_t* status, cudaStream_t st)
{
    int sm_count = ctx ? ctx->sm_count : 0;
    if (!ctx) {
        cudaError_t e = current_sm_count(sm_count);
        if (e != cudaSuccess) return e;
    }
    if (logit_dtype == CONFU_F32)
        return launch_accept_t<float>(sm_count, B, T, C, V, tl, dl, tokens, parent, con_owner, uniforms, temperature,
                                      sibling_mode, accept_len, path, next_token, future_row, counters, workspace,
                                      status, st);
    return launch_accept_t<__nv_bfloat16>(sm_count, B, T, C, V, tl, dl, tokens, parent, con_owner, uniforms, temperature,
                                          sibling_mode, accept_len, path, next_token, future_row, counters, workspace,
                                          status, st);
}

}  // namespace confu
