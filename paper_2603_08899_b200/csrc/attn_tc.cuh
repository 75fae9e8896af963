// Declarations shared by the tensor-core attention kernel (attn_tc.cu) and the kernels that merge
// its split-KV partial results (combine.cu).
#pragma once

#include "common.cuh"

namespace confu {
namespace tc {

constexpr int kD = 128;         // largest head dim of the tensor-core kernels

struct Params {
    confu_dims d;
    SlotMap map;         // packed pool (seq_start) or paged pool (block table, pages of 128 slots = one key tile)
    const int32_t* prefix_len;
    const void* plan;
    float* partials;
    __nv_bfloat16* out;
    float* lse;
    int32_t* status;
    int kind;            // PlanKind of the launch's work units: a plan for another kind is refused
    int n_mt;            // M tiles in use (2 unless one holds all rows)
    int n_rg;            // groups of query rows; a pair = (sequence, kv head, row group)
    int G;               // query heads per kv head
    int rpt;             // query rows per M tile (128 / G)
    int tpg;             // M tiles per row group
    float c;             // sm_scale * log2(e)
    unsigned long long wait_ns;   // limit of every wait on an mbarrier (wall clock)
    const float* k_scale;         // E4M3 cache: value = code * scale[kv head] (device, [Hkv]); unused otherwise
    const float* v_scale;
};

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// The kind of a launch's work units and its row packing (see rows_per_tile).
inline void set_rows(Params& p, const confu_dims& d, int kind)
{
    const int tpg = tiles_per_group(kind);
    p.kind = kind;
    p.tpg = tpg;
    p.G = d.Hq / d.Hkv;
    p.rpt = rows_per_tile(p.G);
    p.n_mt = d.T + d.C > p.rpt ? tpg : 1;
    p.n_rg = row_groups(d.T + d.C, p.G, tpg);
}

// Enqueues the merge of the partial results that the attention launch with the same parameters
// left in prm.partials (pairs whose key tiles were split over several CTAs).
cudaError_t launch_combine(const Params& prm, int units, cudaStream_t st);

}  // namespace tc
}  // namespace confu
