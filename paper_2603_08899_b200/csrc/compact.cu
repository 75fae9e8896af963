// KV compaction of the accepted path: cache[P + k] <- cache[P + path[k]], k = 1..accept_len, for
// every layer and for K and V, in place.
//
// In-place safety without a snapshot: node ids are topologically numbered (parent < child), so
// path[k] >= k, the sources path[1] < path[2] < ... are increasing, and destination k can only
// coincide with a source of an EARLIER step (path[j] = k needs j <= k).  Each thread owns one
// 16-byte column of the row and walks k upwards in batches (all loads of a batch before its
// stores), so within a thread every source is read before any step at or after it overwrites
// that slot, and different threads never touch each other's columns.
//
// That argument needs path[0] = 0 < path[1] < ... < path[a] < T and a <= CONFU_MAX_DEPTH.  A path
// that breaks it (a stale or corrupted buffer) is not followed: the sequence gets the status code
// CONFU_ST_BAD_PATH, nothing of it is copied and its new prefix length is prefix_len + 1 (the root
// only).  Every thread checks the path itself (at most 64 cached loads), so no thread copies a row
// of a path another thread would have refused.
#include "common.cuh"

namespace confu {

constexpr int kCompactBatch = 8;

__global__ void __launch_bounds__(128) compact_kernel(int n_layers, int T, int64_t row_vecs, void* const* __restrict__ k_layers,
                                                      void* const* __restrict__ v_layers,
                                                      const SlotMap map,
                                                      const int32_t* __restrict__ prefix_len,
                                                      const int32_t* __restrict__ accept_len,
                                                      const int32_t* __restrict__ path,
                                                      int32_t* __restrict__ new_prefix_len,
                                                      int32_t* __restrict__ status)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int b = blockIdx.z, layer = blockIdx.y >> 1, kv = blockIdx.y & 1;
    const int64_t col = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int32_t* pth = path + (size_t)b * kPathLen;
    int a = accept_len[b];
    bool ok = a >= 0 && a <= CONFU_MAX_DEPTH && pth[0] == 0;
    if (ok) {
        int before = 0;
        for (int k = 1; k <= a; ++k) {
            const int node = pth[k];
            ok = ok && node > before && node < T;
            before = node;
        }
    }
    if (!ok) a = 0;
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
        if (new_prefix_len) new_prefix_len[b] = prefix_len[b] + a + 1;
        if (!ok && status) status[b] = CONFU_ST_BAD_PATH;
    }
    if (a == 0 || col >= row_vecs) return;
    uint4* pool = reinterpret_cast<uint4*>(kv ? v_layers[layer] : k_layers[layer]);
    const int64_t root = prefix_len[b];              // the root's slot, counted from the sequence's first
    for (int k0 = 1; k0 <= a; k0 += kCompactBatch) {
        uint4 buf[kCompactBatch];
#pragma unroll
        for (int j = 0; j < kCompactBatch; ++j)
            if (k0 + j <= a) buf[j] = pool[pool_slot(map, b, root + pth[k0 + j]) * row_vecs + col];
#pragma unroll
        for (int j = 0; j < kCompactBatch; ++j)
            if (k0 + j <= a) pool[pool_slot(map, b, root + k0 + j) * row_vecs + col] = buf[j];
    }
    (void)n_layers;
}

// cache[seq_start[b] + prefix_len[b] + r] = rows[b][r]  (K and V of the step's own query rows).  Bound by latency: every
// layer's attention waits for it, so a thread has its four pieces in flight together, and the next kernel's blocks are
// let in at once (they wait for this one's stores).  An append + attention pair at B 8, R 60: 0.8 us shorter than with a
// block per row.
constexpr int kAppendThreads = 256, kAppendPer = 4;

__global__ void __launch_bounds__(kAppendThreads) append_kernel(int R, int row_vecs, const uint4* __restrict__ k_rows,
                                                                const uint4* __restrict__ v_rows, uint4* __restrict__ k_cache,
                                                                uint4* __restrict__ v_cache, const SlotMap map,
                                                                const int32_t* __restrict__ prefix_len)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int b = blockIdx.y, kv = blockIdx.z, n = R * row_vecs;
    const uint4* src = (kv ? v_rows : k_rows) + (size_t)b * n;
    uint4* dst = kv ? v_cache : k_cache;
    const int64_t P = prefix_len[b];
    const int i0 = blockIdx.x * (kAppendThreads * kAppendPer) + threadIdx.x;
    uint4 x[kAppendPer];
    int64_t to[kAppendPer];
#pragma unroll
    for (int j = 0; j < kAppendPer; ++j) {
        const int i = i0 + j * kAppendThreads;
        if (i < n) {
            x[j] = src[i];
            to[j] = pool_slot(map, b, P + i / row_vecs) * row_vecs + i % row_vecs;
        }
    }
#pragma unroll
    for (int j = 0; j < kAppendPer; ++j)
        if (i0 + j * kAppendThreads < n) dst[to[j]] = x[j];
}

// E4M3 cache: cache[...][g][d] = e4m3(rows[b][r][g][d] / scale[g]) (quotient in fp32, round to nearest even,
// saturating at 448).  One thread per 16 output bytes, two 16-byte loads.
__global__ void __launch_bounds__(kAppendThreads) append_fp8_kernel(int R, int Hkv, int D, const __nv_bfloat16* __restrict__ k_rows,
                                                                    const __nv_bfloat16* __restrict__ v_rows, uint8_t* __restrict__ k_cache,
                                                                    uint8_t* __restrict__ v_cache, const SlotMap map,
                                                                    const int32_t* __restrict__ prefix_len,
                                                                    const float* __restrict__ k_scale, const float* __restrict__ v_scale)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int b = blockIdx.y, kv = blockIdx.z;
    const int row_units = Hkv * D / 16, i = blockIdx.x * kAppendThreads + threadIdx.x;
    if (i >= R * row_units) return;
    const int r = i / row_units, e = i % row_units * 16;
    const uint4* src = reinterpret_cast<const uint4*>((kv ? v_rows : k_rows) + ((size_t)b * R + r) * (Hkv * D) + e);
    const uint4 in[2] = {src[0], src[1]};
    const float s = (kv ? v_scale : k_scale)[e / D];
    uint8_t* dst = (kv ? v_cache : k_cache) + (size_t)pool_slot(map, b, (int64_t)prefix_len[b] + r) * (Hkv * D) + e;
    const uint32_t h[8] = {in[0].x, in[0].y, in[0].z, in[0].w, in[1].x, in[1].y, in[1].z, in[1].w};
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t word = h[2 * q + j / 2];
            x[j] = __uint_as_float((j & 1) ? (word & 0xffff0000u) : (word << 16)) / s;
        }
        asm("{\n\t.reg .b16 lo, hi;\n\t"
            "cvt.rn.satfinite.e4m3x2.f32 lo, %2, %1;\n\t"
            "cvt.rn.satfinite.e4m3x2.f32 hi, %4, %3;\n\t"
            "mov.b32 %0, {lo, hi};\n\t}"
            : "=r"(w[q])
            : "f"(x[0]), "f"(x[1]), "f"(x[2]), "f"(x[3]));
    }
    *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
}

cudaError_t launch_append_fp8(int B, int R, int Hkv, int D, const void* k_rows, const void* v_rows, void* k_cache,
                              void* v_cache, const SlotMap& map, const int32_t* prefix_len, const float* k_scale,
                              const float* v_scale, cudaStream_t st)
{
    if (B == 0) return cudaSuccess;
    const int units = R * (Hkv * D / 16);
    return launch_pdl(append_fp8_kernel, dim3((units + kAppendThreads - 1) / kAppendThreads, B, 2), dim3(kAppendThreads), st, R, Hkv, D,
                      (const __nv_bfloat16*)k_rows, (const __nv_bfloat16*)v_rows, (uint8_t*)k_cache, (uint8_t*)v_cache, map, prefix_len,
                      k_scale, v_scale);
}

cudaError_t launch_append(int B, int R, int64_t row_bytes, const void* k_rows, const void* v_rows, void* k_cache,
                          void* v_cache, const SlotMap& map, const int32_t* prefix_len, cudaStream_t st)
{
    if (B == 0) return cudaSuccess;
    const int row_vecs = (int)(row_bytes / 16), per = kAppendThreads * kAppendPer;
    return launch_pdl(append_kernel, dim3((R * row_vecs + per - 1) / per, B, 2), dim3(kAppendThreads), st, R, row_vecs,
                      (const uint4*)k_rows, (const uint4*)v_rows, (uint4*)k_cache, (uint4*)v_cache, map, prefix_len);
}

cudaError_t launch_compact(const Ctx*, int B, int T, int n_layers, int64_t row_bytes, void* const* k_layers,
                           void* const* v_layers, const SlotMap& map, const int32_t* prefix_len,
                           const int32_t* accept_len, const int32_t* path, int32_t* new_prefix_len,
                           int32_t* status, cudaStream_t st)
{
    if (B == 0) return cudaSuccess;
    const int64_t row_vecs = row_bytes / 16;
    // with no layers there is still new_prefix_len to write: one block row does it
    dim3 grid((unsigned)((row_vecs + 127) / 128), (unsigned)(n_layers > 0 ? 2 * n_layers : 1), (unsigned)B);
    if (n_layers == 0) {
        return launch_pdl(compact_kernel, dim3(1, 1, (unsigned)B), dim3(128), st, 0, T, (int64_t)0, k_layers, v_layers, map, prefix_len,
                          accept_len, path, new_prefix_len, status);
    }
    return launch_pdl(compact_kernel, grid, dim3(128), st, n_layers, T, row_vecs, k_layers, v_layers, map, prefix_len, accept_len, path,
                      new_prefix_len, status);
}

}  // namespace confu
