// Row statistics: what row_stats_kernel leaves for the acceptance walks.
#pragma once

#include "common.cuh"

namespace confu {

constexpr int kStatChunksMax = 16;
constexpr float kLog2e = 1.4426950408889634f;

struct alignas(16) RowStat {
    float m;        // max raw logit of the chunk
    float s;        // sampling: sum over the chunk of exp((x - m) / temperature)
    int32_t arg;    // greedy: lowest index of the max
    int32_t flag;   // 1: a non-finite logit was met
};

// The walks of the ratio rule (sampling and greedy; stats == nullptr: statistics on demand).
cudaError_t launch_walk(int logit_dtype, int B, int T, int C, int V, const void* tl, const void* dl, const int32_t* tokens,
                        const int32_t* parent, const int32_t* con_owner, const float* uniforms, float temperature, int mode,
                        int nch, const RowStat* stats, int32_t* accept_len, int32_t* path, int32_t* next_token,
                        int32_t* future_row, int32_t* counters, int32_t* status, cudaStream_t st);

}  // namespace confu
