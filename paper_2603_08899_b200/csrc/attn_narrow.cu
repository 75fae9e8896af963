// Tensor-core tree attention for small batches: one M tile per CTA.
//
// With few (sequence, kv head) pairs every pair is spread over many CTAs, each with a handful of key tiles: what
// counts is how long a CTA takes from its start to its last store.  A CTA here works on one M tile (128 / G query
// rows x G heads) of a pair; the CTAs of a pair's tiles walk the same keys side by side (the second read of a K/V tile is
// served by L2).  Against a pair of CTAs on one M = 256 operand (attn_tc2.cu) there is no cluster handshake at either end
// and no relay between the loads and the issuing thread; against the one-CTA kernel with two M tiles (attn_tc.cu) half as
// much to load into registers, exponentiate and store per key tile.
//
// Per 128-key tile, in tensor memory S of two tiles (P over S, as bf16) and two accumulators:
//     S = Q K^T           tcgen05.mma, M 128 N 128, issued one tile ahead
//     P_h = exp2(S_h c - m_h), O_h += P_h V_h     for the two halves h of the tile's keys: warps 0-3 work on keys 0-63,
//                         warps 4-7 on keys 64-127 of the same rows, each with a reference maximum, sum and accumulator
//                         of its own; the two meet once, at the end of a run
// so two warps per scheduler keep the exponential unit busy on every tile, and a tile's weights are ready in half the
// time that one warp would take.  A quarter of the exponentials goes to the FMA pipe (batch 1, a layer: prefix 8192 19.1 ->
// 18.7 us, 16000 26.7 -> 25.7; three eighths: no better than none.  In the kernels with two M tiles, where each scheduler
// has two chains to choose from, it costs 2-8 %).
//
// A layer (this kernel and the merge) against CTA pairs: batch 1, 32/8 heads, R 64, prefix 512: 12.0 -> 9.8 us, 4096: 16.9
// -> 14.7, 8192: 21.0 -> 19.0; R 120, 4096: 20.4 -> 18.9; 8 sequences of 101..3001, R 60: 26.9 -> 23.8.  Of the 14.7 us
// about 2 go to the two changes of kernel, 2 to storing 64 KB per CTA (the SM writes 35 bytes per clock), 2.7 to the merge.
//
// Roles (384 threads): warps 0-7 softmax, warp 8 TMA producer, warp 9 tensor memory and MMA (one lane issues), warp 10
// zeroes the rows of a V tile past the sequence's last slot.  K and V tiles travel in a ring of 32 KB slots in the order
// K0 K1 V0 K2 V1 ... V(n-1).  Every wait is bounded, as in the other kernels.
#include "tc_walk.cuh"

namespace confu {
namespace tc {
namespace narrow {

constexpr int kThreads = 384;
constexpr int kSlots = 5;
constexpr uint32_t kTmemCols = 512, kColO = 256;     // S0 S1 | O of half 0, O of half 1 (128 columns each)
constexpr float kRescaleThreshold = 8.f;
template <int D> constexpr int kTile = kTileKeys * D * 2;

template <int D>
struct SharedStorage {
    alignas(1024) uint8_t q[kTile<D>];
    alignas(1024) uint8_t kv[kSlots][kTile<D>];
    // per softmax warp: first its rows' {reference maximum, sum of weights} for the warp with the other half of the keys, then
    // a 32 x 32 fp32 transpose tile for output rows
    alignas(16) float4 xpose[8][32 * 8];
    alignas(8) uint64_t q_full, q_empty;
    uint64_t full[kSlots], empty[kSlots];
    uint64_t s_full[2], p_full[2][2], o_done;        // [S buffer], [S buffer][half]
    uint64_t v_fixed[kSlots];                        // per slot: the warp that zeroes ragged rows may be a run ahead of the MMA warp
    uint64_t x_bar[4], y_bar[4], r_bar[4];           // per pair of warps with the same rows: written / read the exchange, read O
    uint32_t tmem_base;
    int abort;
};

template <int D>
__device__ __forceinline__ bool wait_warp(SharedStorage<D>& sh, uint64_t* bar, uint32_t parity, unsigned long long limit_ns)
{
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, &sh.abort, limit_ns));
}

template <int D>
__device__ void producer_role(SharedStorage<D>& sh, const Params& prm, const PlanView& pv, const CUtensorMap* q_map,
                              const CUtensorMap* k_map, const CUtensorMap* v_map, const CUtensorMap* ks_map,
                              const CUtensorMap* vs_map)
{
    Walker w;
    Segment s;
    uint32_t i = 0, seg = 0;
    const int R = prm.d.T + prm.d.C;
    auto fill = [&](const CUtensorMap* m, int g, int z) -> bool {
        const uint32_t st = i % kSlots;
        if (!mbar_wait(&sh.empty[st], ((i / kSlots) & 1) ^ 1, &sh.abort, prm.wait_ns)) return false;
        mbar_arrive_expect_tx(&sh.full[st], kTile<D>);
#pragma unroll
        for (int kb = 0; kb < D / 64; ++kb) tma_load_3d(sh.kv[st] + kb * kHalfTile, m, &sh.full[st], kb * 64, g, z);
        ++i;
        return true;
    };
    const CUtensorMap* prev_map = nullptr;           // V of the tile before
    int prev_g = 0, prev_z = 0;
    for (bool run = w.begin(pv, prm, blockIdx.x, kPlanNarrow, s); run; run = w.next(s)) {
        for (int t = s.t0; t < s.t1; ++t) {
            const bool soft = t >= s.nkt;
            const int z = soft ? 0
                        : prm.map.block_table ? prm.map.block_table[(size_t)s.b * prm.map.max_pages + t] * kTileKeys
                                              : (int)(s.slot0 + (int64_t)t * kTileKeys);
            if (!fill(soft ? ks_map : k_map, s.g, z)) return;
            if (prev_map && !fill(prev_map, prev_g, prev_z)) return;
            prev_map = soft ? vs_map : v_map;
            prev_g = s.g;
            prev_z = z;
            if (t == s.t0) {
                if (!mbar_wait(&sh.q_empty, (seg & 1) ^ 1, &sh.abort, prm.wait_ns)) return;
                mbar_arrive_expect_tx(&sh.q_full, (D / 64) * (uint32_t)(prm.rpt * prm.G) * 128u);
#pragma unroll
                for (int kb = 0; kb < D / 64; ++kb)
                    tma_load_3d(sh.q + kb * kHalfTile, q_map, &sh.q_full, kb * 64, s.g * prm.G, s.b * R + prm.rpt * s.rg);
            }
        }
        ++seg;
    }
    if (prev_map) fill(prev_map, prev_g, prev_z);
}

// Slot order: Q K^T of tile g before P V of tile g - 1 (whose weights are being worked on meanwhile); where tile g starts a
// run, after it: the new Q lands while the old run's last weights are worked on.  Instructions of one thread reach the
// pipe in order, so Q K^T of tile g may overwrite the buffer that P V of tile g - 2 read.
template <int D, bool kSplit>
__device__ void mma_role(SharedStorage<D>& sh, const Params& prm, const PlanView& pv, uint32_t tmem)
{
    Walker w;
    Segment s;
    const bool issuer = elect_lane();
    uint32_t i = 0, g = 0, seg = 0, fix_phase = 0;   // slots, tiles, runs so far; phase of every slot's v_fixed
    const uint32_t q_lo = desc_lo(smem_u32(sh.q), 16), k_lo0 = desc_lo(smem_u32(sh.kv[0]), 16);
    const uint32_t v_lo0 = desc_lo(smem_u32(sh.kv[0]), kHalfTile);
    constexpr uint32_t kStep = kTile<D> >> 4;
    auto issue_qk = [&](uint32_t slot, bool last) -> bool {
        if (!mbar_wait(&sh.full[slot % kSlots], (slot / kSlots) & 1, &sh.abort, prm.wait_ns)) return false;
        tc_fence_after();
        if (!issuer) return true;
        const uint32_t kl = k_lo0 + (slot % kSlots) * kStep, d = tmem + (g & 1) * 128;
#pragma unroll
        for (int j = 0; j < D / 16; ++j) {
            const uint32_t off = ((uint32_t)(j >> 2) * kHalfTile + (uint32_t)(j & 3) * 32u) >> 4;
            mma_ss(d, q_lo + off, kl + off, kIdescQK, j > 0 ? 1u : 0u);
        }
        tc_commit(&sh.s_full[g & 1]);
        tc_commit(&sh.empty[slot % kSlots]);
        if (last) tc_commit(&sh.q_empty);
        return true;
    };
    auto issue_pv = [&](uint32_t slot, bool first, bool last, bool ragged) -> bool {     // of tile g - 1
        if (!mbar_wait(&sh.full[slot % kSlots], (slot / kSlots) & 1, &sh.abort, prm.wait_ns)) return false;
        if (ragged) {
            const uint32_t st = slot % kSlots;
            if (!mbar_wait(&sh.v_fixed[st], (fix_phase >> st) & 1, &sh.abort, prm.wait_ns)) return false;
            fix_phase ^= 1u << st;
        }
        const uint32_t buf = (g - 1) & 1, vl = v_lo0 + (slot % kSlots) * kStep;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (!mbar_wait(&sh.p_full[buf][h], ((g - 1) >> 1) & 1, &sh.abort, prm.wait_ns)) return false;
            tc_fence_after();
            if (!issuer) continue;
#pragma unroll
            for (int j = 0; j < (kSplit ? 8 : 4); ++j)           // (4..7: what bf16 leaves of the weights, 32 columns on)
                mma_ts(tmem + kColO + h * 128, tmem + buf * 128 + h * 64 + j * 8, vl + (4 * h + j % 4) * (2048u >> 4),
                       D == 128 ? kIdescPV : kIdescPV64, (first && j == 0) ? 0u : 1u);
        }
        if (issuer) {
            if (last) tc_commit(&sh.o_done);
            tc_commit(&sh.empty[slot % kSlots]);
        }
        return true;
    };
    const int R = prm.d.T + prm.d.C;
    bool have_prev = false, prev_first = false, prev_ragged = false;
    for (bool run = w.begin(pv, prm, blockIdx.x, kPlanNarrow, s); run; run = w.next(s)) {
        for (int t = s.t0; t < s.t1; ++t) {
            const uint32_t ks = i++, vs = have_prev ? i++ : 0;
            const bool cur_last = t + 1 == s.t1;
            if (t > s.t0) {
                if (!issue_qk(ks, cur_last)) return;
                if (!issue_pv(vs, prev_first, false, prev_ragged)) return;
            } else {
                if (have_prev && !issue_pv(vs, prev_first, true, prev_ragged)) return;
                if (!mbar_wait(&sh.q_full, seg & 1, &sh.abort, prm.wait_ns)) return;
                if (!issue_qk(ks, cur_last)) return;
            }
            have_prev = true;
            prev_first = t == s.t0;
            prev_ragged = ragged_rows(s, t, R) > 0;
            ++g;
        }
        ++seg;
    }
    if (have_prev) issue_pv(i, prev_first, true, prev_ragged);
}

// Sees every slot before it is filled again (it arrives on the slot's empty barrier) and, where it holds the V tile of a
// sequence's last key tile, zeroes the rows past the last slot.  It does not wait for the MMA warp: while that waits for the
// weights of a run's last tiles, the whole of a next run of one tile may be here and be repaired too.  So a slot
// has a barrier of its own, which cannot complete twice before the MMA warp has used the slot.
template <int D>
__device__ void tail_role(SharedStorage<D>& sh, const Params& prm, const PlanView& pv)
{
    Walker w;
    Segment s;
    const int R = prm.d.T + prm.d.C, lane = threadIdx.x & 31;
    uint32_t i = 0;
    auto see = [&](int valid) -> bool {
        const uint32_t st = i % kSlots;
        if (!wait_warp(sh, &sh.full[st], (i / kSlots) & 1, prm.wait_ns)) return false;
        if (valid > 0) {
            const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
            for (int kb = 0; kb < D / 64; ++kb)
                for (int off = valid * 128 + lane * 16; off < kHalfTile; off += 32 * 16)
                    *reinterpret_cast<uint4*>(sh.kv[st] + kb * kHalfTile + off) = zero;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.v_fixed[st]);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh.empty[st]);
        ++i;
        return true;
    };
    int prev = -1;                                   // ragged rows of the tile before (0: whole), -1: none
    for (bool run = w.begin(pv, prm, blockIdx.x, kPlanNarrow, s); run; run = w.next(s)) {
        for (int t = s.t0; t < s.t1; ++t) {
            if (!see(0)) return;
            if (prev >= 0 && !see(prev)) return;
            prev = ragged_rows(s, t, R);
        }
    }
    if (prev >= 0) see(prev);
}

template <int D, bool kSplit>
__device__ void softmax_role(SharedStorage<D>& sh, const Params& prm, const PlanView& pv, uint32_t tmem)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int half = warp >> 2, wq = warp & 3;               // half of every key tile, quarter of the rows
    const int lane_row = wq * 32 + lane;                     // row of the M tile = tensor-memory lane
    const uint32_t lane_base = (uint32_t)(wq * 32) << 16;
    const int G = prm.G, T = prm.d.T, R = prm.d.T + prm.d.C, S = prm.d.S, Hq = prm.d.Hq;
    const int hl = lane_row % G;
    const float c = prm.c;
    const uint32_t s_addr = tmem + lane_base + 64 * half, o_addr = tmem + lane_base + kColO + 128 * half;

    Walker w;
    Segment s;
    uint32_t g = 0, seg = 0;
    for (bool run = w.begin(pv, prm, blockIdx.x, kPlanNarrow, s); run; run = w.next(s)) {
        const int r = prm.rpt * s.rg + lane_row / G;         // query row of this thread in this run
        const bool row_valid = lane_row < prm.rpt * G && r < R;
        const uint64_t mask = row_valid ? pv.mask[(size_t)s.b * kMaxRows + r] : 0ull;
        float m_ref = -INFINITY, l = 0.f;                    // of this half's keys
        for (int tile = s.t0; tile < s.t1; ++tile, ++g) {
            const uint32_t buf = g & 1;
            if (!wait_warp(sh, &sh.s_full[buf], (g >> 1) & 1, prm.wait_ns)) return;
            tc_fence_after();
            uint32_t sv[64];
            tmem_ld32(s_addr + buf * 128, *reinterpret_cast<uint32_t(*)[32]>(&sv[0]));
            tmem_ld32(s_addr + buf * 128 + 32, *reinterpret_cast<uint32_t(*)[32]>(&sv[32]));
            tc_wait_ld();
            if (tile >= s.masked) {
                uint64_t lo, hi;
                visible_bits(s, tile, R, T, S, r, row_valid, mask, lo, hi);
                const uint64_t vis = half ? hi : lo;
#pragma unroll
                for (int j = 0; j < 64; ++j)
                    if (!((vis >> j) & 1ull)) sv[j] = 0xff800000u;           // -inf
            }
            const float m_new = fmaxf(m_ref, max64(sv) * c);
            if (tile == s.t0) {
                m_ref = m_new;
            } else {
                const bool move = m_new - m_ref > kRescaleThreshold;         // false when both are -inf (NaN)
                if (__any_sync(0xffffffffu, move)) {
                    // P V of the tile before has completed when its V tile's slot (number 2 g of the walk) is free
                    if (!wait_warp(sh, &sh.empty[2 * g % kSlots], (2 * g / kSlots) & 1, prm.wait_ns)) return;
                    tc_fence_after();
                    const float alpha = move ? ex2(m_ref - m_new) : 1.f;
                    if (move) { m_ref = m_new; l *= alpha; }
#pragma unroll 1
                    for (int q4 = 0; q4 < D / 16; ++q4) {
                        uint32_t ov[16];
                        tmem_ld16(o_addr + q4 * 16, ov);
                        tc_wait_ld();
#pragma unroll
                        for (int j = 0; j < 16; ++j) ov[j] = __float_as_uint(__uint_as_float(ov[j]) * alpha);
                        tmem_st16(o_addr + q4 * 16, ov);
                    }
                }
            }
            const float neg_m = (m_ref == -INFINITY) ? 0.f : -m_ref;
            // P over this half's columns of S (which sit in registers by now)
            l += store_weights64<kSplit, true>(sv, c, neg_m, s_addr + buf * 128);
            tc_wait_st();
            // P V of a run's first tile overwrites both accumulators: both warps of these rows have read the old ones
            if (tile == s.t0 && seg > 0 && !wait_warp(sh, &sh.r_bar[wq], (seg - 1) & 1, prm.wait_ns)) return;
            tc_fence_before();
            // (Every thread for itself: 22 cycles; a __syncwarp and one arrival for the warp 116, of some 1750 a tile.  Batch 1, R 120: 600
            // -> 596 us a step of 32 layers, prefix 8192 681 -> 676; 8 sequences 820 -> 812.)
            mbar_arrive(&sh.p_full[buf][half]);
        }
        // ---- end of the run, while the last P V goes on: the halves' sums, at the larger (= the row's) reference maximum ----
        float4* xp = sh.xpose[warp];
        reinterpret_cast<float2*>(xp)[lane] = make_float2(m_ref, l);
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh.x_bar[wq]);
        if (!wait_warp(sh, &sh.x_bar[wq], seg & 1, prm.wait_ns)) return;
        const float2 other = reinterpret_cast<const float2*>(sh.xpose[warp ^ 4])[lane];
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh.y_bar[wq]);
        const float m_row = fmaxf(m_ref, other.x);
        const float a_me = m_ref == -INFINITY ? 0.f : ex2(m_ref - m_row), a_ot = other.x == -INFINITY ? 0.f : ex2(other.x - m_row);
        const float l_row = l * a_me + other.y * a_ot;
        const int h = s.g * G + hl;
        const bool whole = s.part_slot < 0;
        const float inv_l = whole ? 1.f / l_row : 1.f;
        const float f0 = (half ? a_ot : a_me) * inv_l, f1 = (half ? a_me : a_ot) * inv_l;
        // Each 32-column chunk goes through the warp's transpose tile and leaves as whole rows in 16-byte
        // pieces: eight rows per instruction for the bf16 output, four for an fp32 partial.
        __nv_bfloat16* o_ptr[4];
        float* p_ptr = nullptr;
        if (whole) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                const int lr = wq * 32 + 8 * kk + (lane >> 2);
                const int rk = prm.rpt * s.rg + lr / G;
                o_ptr[kk] = (lr < prm.rpt * G && rk < R)
                                ? prm.out + (((size_t)s.b * R + rk) * Hq + s.g * G + lr % G) * D + 8 * (lane & 3)
                                : nullptr;
            }
        } else {
            p_ptr = prm.partials + (size_t)s.part_slot * (partial_slot_bytes() / sizeof(float)) +
                    (size_t)(wq * 32 + (lane >> 3)) * kPartD + 4 * (lane & 7);
            if (half == 0) {
                float* ml = prm.partials + (size_t)s.part_slot * (partial_slot_bytes() / sizeof(float)) + (size_t)kPartRows * kPartD;
                ml[lane_row] = m_row;
                ml[kPartRows + lane_row] = l_row;
            }
        }
        if (whole && half == 0 && row_valid && prm.lse)
            prm.lse[((size_t)s.b * R + r) * Hq + h] = natural_lse(m_row, l_row);
        if (!wait_warp(sh, &sh.y_bar[wq], seg & 1, prm.wait_ns)) return;     // the exchange has been read: its place is free
        if (!wait_warp(sh, &sh.o_done, seg & 1, prm.wait_ns)) return;
        tc_fence_after();
        constexpr int kChunks = D / 64;                      // of 32 columns; this half's warps write D / 2 columns
#pragma unroll 1
        for (int q4 = kChunks * half; q4 < kChunks * half + kChunks; ++q4) {
            uint32_t u0[32], u1[32];
            tmem_ld32(tmem + lane_base + kColO + q4 * 32, u0);
            tmem_ld32(tmem + lane_base + kColO + 128 + q4 * 32, u1);
            tc_wait_ld();
            auto sum = [&](int i) { return fmaf(__uint_as_float(u0[i]), f0, __uint_as_float(u1[i]) * f1); };
#pragma unroll
            for (int q = 0; q < 8; ++q)
                xp[lane * 8 + (q ^ (lane & 7))] = make_float4(sum(4 * q), sum(4 * q + 1), sum(4 * q + 2), sum(4 * q + 3));
            __syncwarp();
            if (q4 == kChunks * half + kChunks - 1) {
                tc_fence_before();
                if (lane == 0) mbar_arrive(&sh.r_bar[wq]);
            }
            if (whole) {
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const int k = 8 * kk + (lane >> 2), q = 2 * (lane & 3);
                    const float4 a = xp[k * 8 + (q ^ (k & 7))], b2 = xp[k * 8 + ((q + 1) ^ (k & 7))];
                    if (o_ptr[kk])
                        *reinterpret_cast<uint4*>(o_ptr[kk] + q4 * 32) =
                            make_uint4(pack_bf16(a.x, a.y), pack_bf16(a.z, a.w), pack_bf16(b2.x, b2.y), pack_bf16(b2.z, b2.w));
                }
            } else {
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) {
                    const int k = 4 * kk + (lane >> 3);
                    *reinterpret_cast<float4*>(p_ptr + (size_t)(4 * kk) * kPartD + q4 * 32) = xp[k * 8 + ((lane & 7) ^ (k & 7))];
                }
            }
            __syncwarp();
        }
        ++seg;
    }
}

template <int D, bool kSplit>
__global__ void __launch_bounds__(kThreads, 1)
attention_narrow_kernel(const __grid_constant__ CUtensorMap q_map, const __grid_constant__ CUtensorMap k_map,
                        const __grid_constant__ CUtensorMap v_map, const __grid_constant__ CUtensorMap ks_map,
                        const __grid_constant__ CUtensorMap vs_map, const Params prm)
{
    extern __shared__ uint8_t smem_raw[];
    SharedStorage<D>& sh = *reinterpret_cast<SharedStorage<D>*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5;

    if (threadIdx.x == 0) {
        mbar_init(&sh.q_full, 1);
        mbar_init(&sh.q_empty, 1);
        // a slot is free again when its MMAs have completed and the tail warp has seen it
        for (int i = 0; i < kSlots; ++i) { mbar_init(&sh.full[i], 1); mbar_init(&sh.empty[i], 2); mbar_init(&sh.v_fixed[i], 1); }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sh.s_full[i], 1);
            for (int h = 0; h < 2; ++h) mbar_init(&sh.p_full[i][h], 128);
        }
        mbar_init(&sh.o_done, 1);
        for (int i = 0; i < 4; ++i) { mbar_init(&sh.x_bar[i], 2); mbar_init(&sh.y_bar[i], 2); mbar_init(&sh.r_bar[i], 2); }
        sh.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 9) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh.tmem_base)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh.tmem_base;
    const PlanView pv = plan_view(const_cast<void*>(prm.plan), prm.d.B, prm.d.Hkv);
    prefetch_first<D, 64>(prm, pv, &q_map, &k_map);
    // global memory is read and written from here on: the kernels before this one have completed
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (warp < 8) softmax_role<D, kSplit>(sh, prm, pv, tmem);
    else if (warp == 8) {
        if ((threadIdx.x & 31) == 0) producer_role(sh, prm, pv, &q_map, &k_map, &v_map, &ks_map, &vs_map);
    } else if (warp == 9)
        mma_role<D, kSplit>(sh, prm, pv, tmem);
    else if (warp == 10)
        tail_role(sh, prm, pv);
    else if (blockIdx.x == 0 && prm.status && pv.hdr->kind != kPlanNarrow)
        for (int b = threadIdx.x & 31; b < prm.d.B; b += 32) prm.status[b] = CONFU_ST_BAD_PLAN;
    __syncwarp();
    // ---- teardown ----
    tc_fence_before();
    __syncthreads();
    if (sh.abort) {
        // give copies that may still be in flight time to land before the CTA's shared memory goes away
        const unsigned long long t0 = global_ns();
        while (global_ns() - t0 < 200000ull) __nanosleep(1000);
        if (threadIdx.x == 0 && prm.status)
            for (int b = 0; b < prm.d.B; ++b) prm.status[b] = CONFU_ST_TIMEOUT;
        __syncthreads();
    }
    if (warp == 9) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
}

}  // namespace narrow

bool make_tile_map(CUtensorMap* map, const void* base, uint64_t rows, uint64_t heads, uint32_t box_rows, uint32_t box_heads, uint32_t head_dim);

}  // namespace tc

template <int D, bool kSplit>
static cudaError_t launch_d(const Ctx* ctx, const confu_dims& d, const void* q, const void* k_cache, const void* v_cache,
                            int64_t n_slots, const SlotMap& map, const int32_t* prefix_len, const void* k_soft,
                            const void* v_soft, const void* plan, void* partials, void* out, float* lse, int32_t* status,
                            cudaStream_t st)
{
    using namespace tc;
    using namespace tc::narrow;
    const int R = d.T + d.C, G = d.Hq / d.Hkv;
    CUtensorMap q_map, k_map, v_map, ks_map, vs_map;
    bool ok = make_tile_map(&q_map, q, (uint64_t)d.B * R, d.Hq, rows_per_tile(G), G, D) && make_tile_map(&k_map, k_cache, n_slots, d.Hkv, kTileKeys, 1, D) &&
              make_tile_map(&v_map, v_cache, n_slots, d.Hkv, kTileKeys, 1, D);
    if (d.S > 0) ok = ok && make_tile_map(&ks_map, k_soft, d.S, d.Hkv, kTileKeys, 1, D) && make_tile_map(&vs_map, v_soft, d.S, d.Hkv, kTileKeys, 1, D);
    else { ks_map = k_map; vs_map = v_map; }
    if (!ok) return cudaErrorInvalidValue;
    Params prm;
    prm.d = d;
    prm.map = map;
    prm.prefix_len = prefix_len;
    prm.plan = plan;
    prm.prefetch = plan != ctx->workspace;           // (where a call's own plan lies)
    prm.partials = (float*)partials;
    prm.out = (__nv_bfloat16*)out;
    prm.lse = lse;
    prm.status = status;
    set_rows(prm, d, kPlanNarrow);
    prm.c = (d.sm_scale != 0.f ? d.sm_scale : 1.f / sqrtf((float)d.D)) * 1.4426950408889634f;
    prm.wait_ns = ctx->wait_ns;
    prm.k_scale = prm.v_scale = nullptr;
    const size_t smem = sizeof(SharedStorage<D>) + 1024;
    static OncePerDevice attr_done;
    cudaError_t e = attr_done.run([&] {
        return cudaFuncSetAttribute(attention_narrow_kernel<D, kSplit>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    });
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute pdl[1];
    pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctx->sm_count);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = pdl;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, attention_narrow_kernel<D, kSplit>, q_map, k_map, v_map, ks_map, vs_map, prm);
    if (e != cudaSuccess) return e;
    return launch_combine(prm, ctx->sm_count / 2, st);
}

cudaError_t launch_attention_narrow(const Ctx* ctx, const confu_dims& d, const void* q, const void* k_cache,
                                    const void* v_cache, int64_t n_slots, const SlotMap& map,
                                    const int32_t* prefix_len, const void* k_soft, const void* v_soft, const void* plan,
                                    void* partials, void* out, float* lse, int32_t* status, cudaStream_t st)
{
    auto launch = d.D == 64 ? launch_d<64, true> : tc::split_weights(d) ? launch_d<128, true> : launch_d<128, false>;
    return launch(ctx, d, q, k_cache, v_cache, n_slots, map, prefix_len, k_soft, v_soft, plan,
                                                      partials, out, lse, status, st);
}

}  // namespace confu
