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
// N vectors of eight bf16 logits (16 bytes, starting at index ib and kStep apart) folded into a thread's running
// statistics: maximum m, sum s of exp2((x - m) * k2), lowest index arg of the largest value bestv,
// non-finite flag.  Maximum and minimum are taken on packed bf16 pairs with NaN propagation, so one
// comparison of each against the finite range finds NaN and both infinities.
template <int N>
__device__ __forceinline__ void stats_bf16(const uint4 (&v)[N], int ib, int step, float k2, float& m, float& s, float& bestv, int& arg,
                                           int& flag)
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
    if (cm > bestv) {                                    // rare after the first vectors: find the first element equal to it
        bestv = cm;
#pragma unroll
        for (int j = 8 * N - 1; j >= 0; --j) {
            const float x = __uint_as_float((j & 1) ? (w[j >> 1] & 0xffff0000u) : (w[j >> 1] << 16));
            if (x == cm) arg = ib + (j >> 3) * step + (j & 7);
        }
    }
    if (cm > m) { s *= ex2((m - cm) * k2); m = cm; }
    const float nmk = -m * k2;
    uint64_t acc[2] = {f2_pack(0.f, 0.f), f2_pack(0.f, 0.f)};
    const uint64_t k22 = f2_pack(k2, k2), nmk2 = f2_pack(nmk, nmk);
#pragma unroll
    for (int j = 0; j < 4 * N; ++j) {
        float x0, x1;
        f2_unpack(f2_fma(f2_pack(__uint_as_float(w[j] << 16), __uint_as_float(w[j] & 0xffff0000u)), k22, nmk2), x0, x1);
        acc[j & 1] = f2_add(acc[j & 1], f2_pack(ex2(x0), ex2(x1)));
    }
    float a0, a1;
    f2_unpack(f2_add(acc[0], acc[1]), a0, a1);
    s += a0 + a1;
}

template <typename T>
__global__ void __launch_bounds__(256) row_stats_kernel(const T* __restrict__ tl, const T* __restrict__ dl, int V,
                                                        int n_rows, int nch, int chunk_elems, float k2,
                                                        RowStat* __restrict__ stats)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int row = blockIdx.x, chunk = blockIdx.y, mat = blockIdx.z;
    // counted from the 16-byte boundary at or before the row's first entry, which has place `shift` (a chunk that is left without
    // entries of its row writes the statistics of none)
    const T* first = (mat == 0 ? tl : dl) + (size_t)row * V;
    const int shift = (int)((reinterpret_cast<uintptr_t>(first) & 15u) / sizeof(T));
    const T* base = first - shift;
    const int lo = chunk * chunk_elems, hi = min(V + shift, lo + chunk_elems);
    const int tid = threadIdx.x;

    float m = -INFINITY, s = 0.f, bestv = -INFINITY;
    int arg = INT_MAX, flag = 0;

    int i0 = lo + tid * kEpt;
    if (i0 < shift) {                                    // the vector that holds the row's first entries
        for (int i = shift; i < min(kEpt, hi); ++i) {
            const float v = to_f32(base[i]);
            if (!(fabsf(v) <= 3.0e38f)) flag = 1;
            if (v > bestv) { bestv = v; arg = i; }
            if (v > m) { s *= ex2((m - v) * k2); m = v; }
            s += ex2((v - m) * k2);
        }
        i0 += 256 * kEpt;
    }
    if constexpr (sizeof(T) == 2) {
        // four vectors in flight per thread and folded in together (two, one after the other: 195 us for the 985 MB of 32
        // sequences of 60 nodes, V 128256; now 172 us, 5.7 TB/s)
        constexpr int kStep = 256 * kEpt;
        for (; i0 + 3 * kStep + kEpt <= hi; i0 += 4 * kStep) {
            uint4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = *reinterpret_cast<const uint4*>(base + i0 + u * kStep);
            stats_bf16(v, i0, kStep, k2, m, s, bestv, arg, flag);
        }
    }
    for (; i0 < hi; i0 += 256 * kEpt * 2) {
        float x[2][kEpt];
        const int i1 = i0 + 256 * kEpt;
        if constexpr (sizeof(T) == 2) {
            // bf16 rows, both 8-element vectors whole: packed path (about 4 instructions per logit)
            if (i1 + kEpt <= hi) {
                const uint4 v[2] = {*reinterpret_cast<const uint4*>(base + i0), *reinterpret_cast<const uint4*>(base + i1)};
                stats_bf16(v, i0, 256 * kEpt, k2, m, s, bestv, arg, flag);
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
            if (lm > m) { s *= exp2f((m - lm) * k2); m = lm; }
            float acc = 0.f;
#pragma unroll
            for (int j = 0; j < kEpt; ++j) {
                const float v = x[u][j];
                const bool in = ib + j < hi;
                if (in && !(fabsf(v) <= 3.0e38f)) flag = 1;
                acc += exp2f((v - m) * k2);                      // out-of-range entries are -inf -> 0
                if (v > bestv) { bestv = v; arg = ib + j; }
            }
            s += acc;
        }
    }
    // block reduction of (m, s), (bestv, arg), flag
    auto merge = [&](float m2, float s2, float v2, int a2, int f2) {
        const float mm = fmaxf(m, m2);
        const float c1 = (m == mm) ? 1.f : exp2f((m - mm) * k2);
        const float c2 = (m2 == mm) ? 1.f : exp2f((m2 - mm) * k2);
        s = s * c1 + s2 * c2;
        m = mm;
        if (v2 > bestv || (v2 == bestv && a2 < arg)) { bestv = v2; arg = a2; }
        flag |= f2;
    };
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float m2 = __shfl_xor_sync(0xffffffffu, m, o);
        const float s2 = __shfl_xor_sync(0xffffffffu, s, o);
        const float v2 = __shfl_xor_sync(0xffffffffu, bestv, o);
        const int a2 = __shfl_xor_sync(0xffffffffu, arg, o);
        const int f2 = __shfl_xor_sync(0xffffffffu, flag, o);
        merge(m2, s2, v2, a2, f2);
    }
    __shared__ float sm[8], ss[8], sv[8];
    __shared__ int sa[8], sf[8];
    if ((tid & 31) == 0) { sm[tid >> 5] = m; ss[tid >> 5] = s; sv[tid >> 5] = bestv; sa[tid >> 5] = arg; sf[tid >> 5] = flag; }
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < 8; ++w) merge(sm[w], ss[w], sv[w], sa[w], sf[w]);
        RowStat r;
        r.m = m; r.s = s; r.arg = arg == INT_MAX ? arg : arg - shift; r.flag = flag;
        stats[((size_t)mat * n_rows + row) * kStatChunksMax + chunk] = r;
    }
    (void)nch;
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
    // enough CTAs to fill the machine a few times over, chunks a multiple of the vector width
    int nch = (sm_count * 8 + n_rows * nmat - 1) / (n_rows * nmat);
    nch = nch < 1 ? 1 : (nch > kStatChunksMax ? kStatChunksMax : nch);
    const int all = ((size_t)V * sizeof(T)) % 16 == 0 ? V : V + 16 / (int)sizeof(T) - 1;      // places of a row, whatever its shift
    int chunk_elems = (all + nch - 1) / nch;
    chunk_elems = (chunk_elems + 15) / 16 * 16;
    nch = (all + chunk_elems - 1) / chunk_elems;
    const float k2 = (greedy ? 1.f : 1.f / temperature) * kLog2e;
    RowStat* stats = (RowStat*)workspace;
    if (!lazy) {
        const cudaError_t e = launch_pdl(row_stats_kernel<T>, dim3(n_rows, nch, nmat), dim3(256), st, (const T*)tl, (const T*)dl, V,
                                         n_rows, nch, chunk_elems, k2, stats);
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
