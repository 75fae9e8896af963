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
    int prefetch;                 // 1: the plan was made by an earlier call, what it says can be fetched ahead of time
};

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// Natural logarithm of a row's softmax denominator l 2^m.  In 64 bits but for the logarithm: with fp32 products and sums the result
// carries three roundings instead of one (head dim 64, scores of size 4: 7e-8 of it, now 4e-8).
__device__ __forceinline__ float natural_lse(float m, float l) { return (float)((double)m * 0.6931471805599453 + (double)logf(l)); }

// Whether softmax weights are handed to the tensor pipe as the sum of two bf16 numbers instead of one.  Head dim 64 and more than
// four query heads per kv head: on CUDA cores these dims have fp32 weights, and 16 bits of a weight keep that precision: the
// error against 64 bits is 1.000001 times that of rounding the output to bf16 (prefixes 100..6000, every G; with weights of 8 bits
// 1.25-1.4 times).  It costs twice the instructions of P V and four more per pair of weights: one layer with its own
// plan, B 4, 64 / 8 heads of 128, prefixes 500..4000: 36.0 -> 39.8 us; B 2, 32 / 8 heads of 64, 1500..2500: 17.7 -> 18.7; where
// the tensor pipe is busy more: B 32, 64 / 8 heads of 128, 500..4000 174 -> 248; B 48, 32 / 8 heads of 64 112 -> 145.
inline bool split_weights(const confu_dims& d) { return d.D == 64 || d.Hq / d.Hkv > 4; }

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
