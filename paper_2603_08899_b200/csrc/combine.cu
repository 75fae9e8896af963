// Merge of the split-KV partial results of the tensor-core attention kernels: a pair (sequence, kv
// head, row group) whose key tiles were walked by several work units has one unnormalised partial (O, m,
// l) per unit; merge_kernel combines them into the output rows.
//
// Bound by latency: the partials are in L2 (a few MB per layer at batch 1), and the next layer waits.  The plan says who
// walked a pair, so a warp has one read to make before it knows what to fetch (working that out from the cost line took
// three reads and two 64-bit divisions); it then has eight pieces of partial rows in flight -- four rows of two parts,
// two rows of up to four, or one row eight parts at a time -- together with the parts' maxima and sums (sixteen
// pieces at half as many warps per SM: up to 2 us slower).  The order of every sum is fixed by the part index
// alone, so the result does not depend on the run.  A layer (attention + merge) before -> now: B 1, prefix 4096, R 64
// 17.9 -> 17.5 us, R 120 24.8 -> 21.8; B 8, prefixes 101..3001, R 60: 33.4 -> 28.5; B 16, 512..8000: 85 -> 77.
#include "attn_tc.cuh"

namespace confu {
namespace tc {
namespace {

// A lane's share of a row of D fp32 columns: D / 32 of them, columns lane * D / 32 onwards.
template <int D>
struct Piece {
    static constexpr int n = D / 32;
    float x[n];
    __device__ __forceinline__ static Piece zero()
    {
        Piece p;
#pragma unroll
        for (int i = 0; i < n; ++i) p.x[i] = 0.f;
        return p;
    }
    // partial results are read past L1: they were written by other SMs
    __device__ __forceinline__ static Piece load(const float* row, int lane)
    {
        Piece p;
        if constexpr (n == 4) {
            const float4 v = __ldcg(reinterpret_cast<const float4*>(row) + lane);
            p.x[0] = v.x; p.x[1] = v.y; p.x[2] = v.z; p.x[3] = v.w;
        } else {
            const float2 v = __ldcg(reinterpret_cast<const float2*>(row) + lane);
            p.x[0] = v.x; p.x[1] = v.y;
        }
        return p;
    }
    __device__ __forceinline__ void add(float w, const Piece& o)
    {
#pragma unroll
        for (int i = 0; i < n; ++i) x[i] = fmaf(w, o.x[i], x[i]);
    }
    // times s, rounded to bf16, into the output row
    __device__ __forceinline__ void store(__nv_bfloat16* row, int lane, float s) const
    {
        if constexpr (n == 4)
            reinterpret_cast<uint2*>(row)[lane] = make_uint2(pack_bf16(x[0] * s, x[1] * s), pack_bf16(x[2] * s, x[3] * s));
        else
            reinterpret_cast<uint32_t*>(row)[lane] = pack_bf16(x[0] * s, x[1] * s);
    }
};

constexpr int kMergeThreads = 256, kMergeWarps = kMergeThreads / 32;

struct Pair {
    int b, g, rg;
    int c0, n;                 // first work unit and number of units that walked the pair (every n_rg-th from c0)
};
__device__ __forceinline__ const float* part_of(const Params& prm, const Pair& u, int p)
{
    return prm.partials + (size_t)(2 * (u.c0 + p * prm.n_rg) + (p < u.n - 1 ? 1 : 0)) * (partial_slot_bytes() / sizeof(float));
}
// query row of row `lane_row` of M tile t (may be past the last)
__device__ __forceinline__ int query_row(const Params& prm, const Pair& u, int t, int lane_row) { return prm.rpt * (prm.tpg * u.rg + t) + lane_row / prm.G; }

template <int D>
__device__ __forceinline__ void finish(const Params& prm, const Pair& u, int r, int lane_row, const Piece<D>& acc, float M, float L, int lane)
{
    const size_t row = ((size_t)u.b * (prm.d.T + prm.d.C) + r) * prm.d.Hq + u.g * prm.G + lane_row % prm.G;
    acc.store(prm.out + row * D, lane, 1.f / L);
    if (prm.lse && lane == 0) prm.lse[row] = natural_lse(M, L);
}

// NR rows (row0, row0 + 1, ... below `rows`) of up to NP parts each, all loads in flight at once
template <int D, int NP, int NR>
__device__ __forceinline__ void merge_rows(const Params& prm, const Pair& u, int t, int row0, int rows, int lane)
{
    float m = -INFINITY, l = 0.f;                    // lane k * NP + p: part p of row k
    if (lane < NP * NR && lane % NP < u.n) {
        const float* ml = part_of(prm, u, lane % NP) + (size_t)kPartRows * kPartD + t * 128 + min(row0 + lane / NP, rows - 1);
        m = __ldcg(ml);
        l = __ldcg(ml + kPartRows);
    }
    Piece<D> v[NR][NP];
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        const float* part = part_of(prm, u, p) + (size_t)(t * 128) * kPartD;
#pragma unroll
        for (int k = 0; k < NR; ++k)
            v[k][p] = p < u.n ? Piece<D>::load(part + (size_t)min(row0 + k, rows - 1) * kPartD, lane) : Piece<D>::zero();
    }
    float M = m;
#pragma unroll
    for (int o = NP / 2; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
    const float w = m == -INFINITY ? 0.f : ex2(m - M);
    float L = w * l;
#pragma unroll
    for (int o = NP / 2; o > 0; o >>= 1) L += __shfl_xor_sync(0xffffffffu, L, o);
#pragma unroll
    for (int k = 0; k < NR; ++k) {
        Piece<D> acc = Piece<D>::zero();
#pragma unroll
        for (int p = 0; p < NP; ++p) acc.add(__shfl_sync(0xffffffffu, w, k * NP + p), v[k][p]);
        const float Mk = __shfl_sync(0xffffffffu, M, k * NP), Lk = __shfl_sync(0xffffffffu, L, k * NP);
        const int r = query_row(prm, u, t, row0 + k);
        if (row0 + k < rows && r < prm.d.T + prm.d.C) finish<D>(prm, u, r, row0 + k, acc, Mk, Lk, lane);
    }
}

// one row of any number of parts, eight at a time
template <int D>
__device__ __forceinline__ void merge_long(const Params& prm, const Pair& u, int t, int row0, int lane)
{
    constexpr int K = 8;
    const int row = t * 128 + row0;
    auto load = [&](Piece<D> (&v)[K], int p0) {
#pragma unroll
        for (int k = 0; k < K; ++k) v[k] = p0 + k < u.n ? Piece<D>::load(part_of(prm, u, p0 + k) + (size_t)row * kPartD, lane) : Piece<D>::zero();
    };
    auto stat = [&](int p, int which) { return __ldcg(part_of(prm, u, p) + (size_t)kPartRows * kPartD + which * kPartRows + row); };
    float m = lane < u.n ? stat(lane, 0) : -INFINITY, l = lane < u.n ? stat(lane, 1) : 0.f;
    Piece<D> v[K];
    load(v, 0);
    float M = m;
    for (int p = 32 + lane; p < u.n; p += 32) M = fmaxf(M, stat(p, 0));
    M = warp_max(M);
    Piece<D> acc = Piece<D>::zero();
    float L = 0.f;
    for (int p0 = 0; p0 < u.n; p0 += 32) {
        if (p0 > 0) {
            m = p0 + lane < u.n ? stat(p0 + lane, 0) : -INFINITY;
            l = p0 + lane < u.n ? stat(p0 + lane, 1) : 0.f;
        }
        const float w = m == -INFINITY ? 0.f : ex2(m - M);
        L += warp_sum(w * l);
        for (int q0 = 0; q0 < 32 && p0 + q0 < u.n; q0 += K) {
            if (p0 + q0 > 0) load(v, p0 + q0);
#pragma unroll
            for (int k = 0; k < K; ++k) acc.add(__shfl_sync(0xffffffffu, w, q0 + k), v[k]);      // 0 past the last part
        }
    }
    const int r = query_row(prm, u, t, row0);
    if (r < prm.d.T + prm.d.C) finish<D>(prm, u, r, row0, acc, M, L, lane);
}

// Block (pair, M tile, group of 8 * per_warp rows): a warp takes per_warp rows.
template <int D>
__global__ void __launch_bounds__(kMergeThreads, 4) merge_kernel(const Params prm, int per_warp)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the next kernel may start its prologue
    asm volatile("griddepcontrol.wait;" ::: "memory");      // the attention kernel has completed
    const PlanView pv = plan_view(const_cast<void*>(prm.plan), prm.d.B, prm.d.Hkv);
    // pairs: sequence major, then kv head, then row group
    const int bg = blockIdx.x / prm.n_rg, t = blockIdx.y, lane = threadIdx.x & 31;
    Pair u;
    u.b = bg / prm.d.Hkv;
    u.g = bg % prm.d.Hkv;
    u.rg = blockIdx.x % prm.n_rg;
    // A plan for another kind of work unit has been refused by the attention kernel.  Its share numbers must not be followed:
    // they belong to another number of row groups, and the partial slots they lead to may lie past the workspace.
    const Parts parts = {__ldg(&pv.parts[bg].word)};
    if (parts.kind() != prm.kind) {
        if (prm.status && threadIdx.x == 0 && u.g == 0 && u.rg == 0 && blockIdx.y == 0 && blockIdx.z == 0) prm.status[u.b] = CONFU_ST_BAD_PLAN;
        return;
    }
    u.c0 = parts.first() * prm.n_rg + u.rg;
    u.n = parts.n();
    if (u.n == 1) return;                                   // one unit covered the pair and wrote the output itself
    const int rows = prm.rpt * prm.G;                       // of an M tile
    const int row0 = (blockIdx.z * kMergeWarps + (threadIdx.x >> 5)) * per_warp, end = min(row0 + per_warp, rows);
    if (u.n == 0) {                                         // malformed tree: nobody worked on the pair; its rows read 0
        for (int i = row0; i < end; ++i) {
            const int r = query_row(prm, u, t, i);
            if (r >= prm.d.T + prm.d.C) break;
            const size_t row = ((size_t)u.b * (prm.d.T + prm.d.C) + r) * prm.d.Hq + u.g * prm.G + i % prm.G;
            Piece<D>::zero().store(prm.out + row * D, lane, 0.f);
            if (prm.lse && lane == 0) prm.lse[row] = 0.f;
        }
        return;
    }
    if (row0 >= rows || query_row(prm, u, t, row0) >= prm.d.T + prm.d.C) return;
    if (u.n <= 4 && per_warp == 1) merge_rows<D, 4, 1>(prm, u, t, row0, end, lane);
    else if (u.n == 2 && per_warp == 4) merge_rows<D, 2, 4>(prm, u, t, row0, end, lane);
    else if (u.n == 2) merge_rows<D, 2, 2>(prm, u, t, row0, end, lane);
    else if (u.n <= 4)
        for (int i = row0; i < end; i += 2) merge_rows<D, 4, 2>(prm, u, t, i, end, lane);
    else
        for (int i = row0; i < end; ++i) merge_long<D>(prm, u, t, i, lane);
}

}  // namespace

cudaError_t launch_combine(const Params& prm, int units, cudaStream_t st)
{
    // Rows per warp: one where that leaves every warp's rows in flight together, more where there are many pairs (a
    // quarter of the blocks, two to four parts each).  B 8, prefixes 101..3001, per layer: 2 rows 27.2 us, 4 rows 27.9; B 4,
    // 500..4000: 1 row 20.7 us, and 22.7 with the loads of rows that the warp does not have repeated instead of left out.
    const int n_pairs = prm.d.B * prm.d.Hkv * prm.n_rg, tiles = n_pairs * prm.n_mt;
    const int per_warp = tiles <= units ? 1 : tiles <= 2 * units ? 2 : 4;
    const dim3 grid((unsigned)n_pairs, (unsigned)prm.n_mt, (unsigned)(128 / (kMergeWarps * per_warp)));
    return prm.d.D == 64 ? launch_pdl(merge_kernel<64>, grid, dim3(kMergeThreads), st, prm, per_warp)
                         : launch_pdl(merge_kernel<kD>, grid, dim3(kMergeThreads), st, prm, per_warp);
}

}  // namespace tc
}  // namespace confu
