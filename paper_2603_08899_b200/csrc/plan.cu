// Step-level planning kernel: tree validation, ancestor bitmasks, split-KV tile counts.
//
// Mask rule (tree attention over a token tree, with one contemplate token hung on a node's
// branch): a tree row sees itself and its ancestors; a contemplate row sees itself, its owner
// and the owner's ancestors.  Bit j < T of mask[b][r] says "row r sees the slot of tree row j";
// that a contemplate row sees its own slot (and no other contemplate row's) is implied.
//
// One CTA, a chain of short phases: what it costs is latency (global loads that depend on one another, barriers,
// 64-bit divisions), and every step waits for it.  A warp takes a sequence: parents go through shared memory, so that
// walking to the root is a few shared loads; the cost line is a warp scan; each CTA's share is found by bisection in
// shared memory.  B 32: 35 -> 10 us, B 8: 12 -> 7 us; at B 1 the step is 5 us shorter: the attention kernel of the first
// layer sets itself up meanwhile.  The search for shares of their own starts at the smallest that can fit, sums are one
// reduction instruction, the step's constants and first slots go through shared memory, and the line is left out where no
// tensor-core kernel takes the dims.  Plan and one layer, 8 kv heads: B 1 prefix 4096 20.6 -> 19.1 us, B 8 of 300..4000
// 55.2 -> 47.3, B 32 of 300..2000 81.5 -> 78.0; the fp32 layer of 256 keys 13.7 -> 10.7.  The search has one copy of the test in a
// loop that is not unrolled: code that is fetched once is paid for in full (B 2: three copies and 4 KB more of shared memory
// +1.4 us).
#include "common.cuh"

namespace confu {

constexpr int kPlanThreads = 1024, kPlanWarps = kPlanThreads / 32;      // at most; at least kPlanMaxCtas threads
constexpr int kPlanCached = 1024;                    // sequences whose tile counts, positions and first slots fit shared memory

// Shares of their own, none longer than `own` where a run weighs its tiles + kRunOverheadTiles: a sequence's (sequence, kv head)
// stretches are cut into equal pieces, one to a share, or, where they are short, several whole ones make up a share.  (A change of run
// takes 3000 to 4800 cycles, a key tile 1750 with one M tile and 3600 with two.  Slack of 1, 2, 4 tiles against the line: 1 is 2-6 %
// slower at 6 to 12 sequences, 4 is the same or 2 % slower.)
constexpr int kRunOverheadTiles = 2;
struct Shares {
    int pieces;                                      // shares of a stretch
    int whole;                                       // stretches of a share (1 where they are cut)
    int total;                                       // shares of the sequence
};
__device__ __forceinline__ Shares shares_of(int tiles, int own, int Hkv)
{
    if (tiles == 0) return {0, 1, 0};
    if (tiles + kRunOverheadTiles > own) {
        const int pieces = (int)((uint32_t)(tiles + own - kRunOverheadTiles - 1) / (uint32_t)(own - kRunOverheadTiles));
        return {pieces, 1, (int)min((int64_t)pieces * Hkv, (int64_t)kPlanMaxCtas + 1)};
    }
    const int whole = min((int)((uint32_t)own / (uint32_t)(tiles + kRunOverheadTiles)), min(Hkv, 1 << 14));
    if (whole == 1) return {1, 1, min(Hkv, kPlanMaxCtas + 1)};
    return {1, whole, (int)min((uint32_t)(Hkv + whole - 1) / (uint32_t)whole, (uint32_t)kPlanMaxCtas + 1)};
}

__global__ void __launch_bounds__(kPlanThreads) plan_kernel(confu_dims d, int units, int kind, const int64_t* __restrict__ seq_start,
                                                            const int32_t* __restrict__ prefix_len,
                                                            const int32_t* __restrict__ parent,
                                                            const int32_t* __restrict__ con_owner, void* plan_raw,
                                                            int32_t* status)
{
    const int B = d.B, T = d.T, C = d.C, R = d.T + d.C;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    __shared__ int8_t s_par[kPlanWarps][kMaxTree];
    __shared__ uint64_t s_mask[kPlanWarps][kMaxTree];
    __shared__ int32_t s_tiles[kPlanCached];
    __shared__ int64_t s_base[kPlanCached + 1], s_slot[kPlanCached];
    __shared__ int64_t s_line;
    __shared__ int s_warp[kPlanMaxCtas / 32], s_own, s_ctas;
    // shares of their own: pieces of a stretch, whole stretches of a share (in the place of the masks, which are done by then)
    short2* s_cut = reinterpret_cast<short2*>(s_mask);
    static_assert(sizeof(s_mask) >= kPlanCached * sizeof(short2), "s_cut");
    PlanView pv = plan_view(plan_raw, B, d.Hkv);
    const bool cached = B <= kPlanCached;

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // ---- validation, masks, tile counts: a warp per sequence ----
    for (int b = warp; b < B; b += (int)(blockDim.x >> 5)) {
        int p[2], o[2];
        bool bad_parent = false, bad_owner = false;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = lane + 32 * h;
            p[h] = r < T ? parent[(size_t)b * T + r] : 0;
            o[h] = r < C ? con_owner[(size_t)b * C + r] : 0;
        }
        const int P = prefix_len[b];
        const int64_t slot = seq_start ? seq_start[b] : 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = lane + 32 * h;
            if (r < T) {
                bad_parent = bad_parent || (r == 0 ? p[h] != -1 : (p[h] < 0 || p[h] >= r));
                s_par[warp][r] = (int8_t)p[h];
            }
            bad_owner = bad_owner || (r < C && (o[h] < 0 || o[h] >= T));
        }
        bad_parent = __any_sync(0xffffffffu, bad_parent);
        bad_owner = __any_sync(0xffffffffu, bad_owner);
        const int code = bad_parent ? CONFU_ST_BAD_PARENT : bad_owner ? CONFU_ST_BAD_OWNER : 0;
        __syncwarp();
#pragma unroll
        for (int h = 0; h < 2; ++h) {                // a tree row sees itself and its ancestors
            const int r = lane + 32 * h;
            if (r < T) {
                uint64_t m = 1ull << r;
                if (!code)
                    for (int a = s_par[warp][r]; a >= 0; a = s_par[warp][a]) m |= 1ull << a;
                s_mask[warp][r] = m;
            }
        }
        __syncwarp();
        // tree rows, then contemplate rows (owner and its ancestors; its own slot is implied), then nothing
        uint64_t* mask = pv.mask + (size_t)b * kMaxRows;
        for (int r = lane; r < T; r += 32) mask[r] = s_mask[warp][r];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = lane + 32 * h;
            if (k < C) mask[T + k] = code ? 0 : s_mask[warp][o[h]];
        }
        for (int r = R + lane; r < kMaxRows; r += 32) mask[r] = 0;
        if (lane == 0) {
            pv.bad[b] = code;
            if (code && status) status[b] = code;
            const int64_t keys = (int64_t)P + R;
            const int tiles = code ? 0 : (int32_t)((keys + kTileKeys - 1) / kTileKeys) + (d.S > 0 ? 1 : 0);
            (cached ? s_tiles : pv.tiles)[b] = tiles;
            if (cached) s_slot[b] = slot;
        }
        __syncwarp();
    }
    __syncthreads();
    if (kind == kPlanMasks) return;
    // ---- shares of their own, or the cost line: one stretch per (sequence, kv head); its groups of query rows are walked
    // side by side ----
    const int n_rg = row_groups(R, d.Hq / d.Hkv, tiles_per_group(kind));
    if (warp == 0) {
        // The work is cut into `lanes` shares; CTA lane * n_rg + rg walks the lane's share for row group rg,
        // so the CTAs of a lane read the same K/V tiles at about the same time (the second read hits L2).
        int lanes = (units < kPlanMaxCtas ? units : kPlanMaxCtas) / n_rg;
        // Every run costs its CTA a load of Q, a drain and output rows, or partial rows that the merge reads again: shares of
        // their own (above) have one run or whole ones, where the line's have the end of one stretch and the beginning of another.
        // They are taken where the longest is not over the line's share by more than what a run weighs.  (A layer with its append
        // and merge, 8 kv heads, paged, 8 sequences of 101..3001, R 60: 27.7 -> 25.4 us, 72 instead of 144 CTAs with partial rows;
        // 4 sequences of 500..4000, 64 / 8 heads, own plan: 40.0 -> 39.1; batch 1, prefix 4096: 34 tiles in 9 shares of 4
        // instead of a line cut into shares of 4.1: 17.5 -> 16.9.  32 sequences of 512..16384: no such shares, the line.)
        int own = 0;
        if (cached && lanes > 0) {
            bool huge = false;
            uint32_t tiles = 0, line = 0;
            for (int b = lane; b < B; b += 32) {
                huge = huge || s_tiles[b] >= (1 << 20);
                tiles += (uint32_t)s_tiles[b];
                line += s_tiles[b] ? (uint32_t)(s_tiles[b] + kPairOverheadTiles) : 0;
            }
            tiles = __reduce_add_sync(0xffffffffu, tiles);
            line = __reduce_add_sync(0xffffffffu, line);
            // (32 bits hold these sums, and the products with the heads but for absurd numbers of them)
            if (!__any_sync(0xffffffffu, huge) && tiles && (uint64_t)line * d.Hkv < (1u << 30)) {
                const uint32_t L = (uint32_t)lanes, H = (uint32_t)d.Hkv;
                int lo = (int)((tiles * H + L - 1) / L) + kRunOverheadTiles;         // no share is shorter than the mean
                const int longest = (int)((line * H + L - 1) / L) + kRunOverheadTiles;
// The shortest that fits.  Larger batches seldom have one, so the longest is tried first there: a search that goes all the way
                // up for nothing costs more (plan alone, 8 kv heads, B 12 8.0 -> 7.3 us, 16 8.0 -> 7.2, 32 of 512..16384 11.7 -> 10.8, 128 24.7 ->
                // 21.3) than one more trial (B 8 5.7, the same; B 4 4.5 -> 4.8, 1 4.0 -> 4.2).
#pragma unroll 1
                for (int hi = longest + 1, at = B > 8 ? longest : lo; ; at = (lo + hi) / 2) {
                    if (lo >= hi) {
                        own = hi <= longest ? hi : 0;
                        break;
                    }
                    uint32_t n = 0;
#pragma unroll 1
                    for (int b = lane; b < B; b += 32) n += (uint32_t)shares_of(s_tiles[b], at, d.Hkv).total;
                    if ((int)__reduce_add_sync(0xffffffffu, n) <= lanes) hi = at;
                    else lo = at + 1;
                }
            }
        }
        // positions on the line, or share numbers
        int64_t acc = 0;
        for (int b0 = 0; b0 < B; b0 += 32) {
            const int b = b0 + lane;
            const int tiles = b < B ? (cached ? s_tiles[b] : pv.tiles[b]) : 0;
            int64_t mine = tiles > 0 ? (int64_t)(tiles + kPairOverheadTiles) * d.Hkv : 0;
            if (own) {
                const Shares sh = shares_of(tiles, own, d.Hkv);
                mine = sh.total;
                if (b < B) s_cut[b] = make_short2((short)sh.pieces, (short)sh.whole);
            }
            int64_t incl = mine;
#pragma unroll 1
            for (int k = 1; k < 32 && k < B; k <<= 1) {
                const int64_t t = __shfl_up_sync(0xffffffffu, incl, k);
                if (lane >= k) incl += t;
            }
            if (b < B) (cached ? s_base : pv.tile_base)[b] = acc + incl - mine;
            acc += __shfl_sync(0xffffffffu, incl, B - b0 < 32 ? B - b0 - 1 : 31);
        }
        if ((int64_t)lanes > acc) lanes = (int)acc;
        if (lane == 0) {
            s_own = own;
            s_ctas = lanes * n_rg;
            s_line = acc;
            (cached ? s_base : pv.tile_base)[B] = acc;
            PlanHeader h;
            h.B = B; h.Hkv = d.Hkv; h.T = T; h.C = C; h.S = d.S; h.R = R;
            h.n_tiles = acc;
            h.n_ctas = lanes * n_rg;
            h.kind = kind;
            *pv.hdr = h;
        }
    }
    __syncthreads();
    // The runs of key tiles of every CTA of the tensor-core attention kernel, worked out once per step
    // instead of by every role of every CTA of every layer: thread c walks CTA c's share of the cost
    // line, first to count its runs, then (behind a prefix sum) to write them down.
    const int64_t N = s_line;
    const int n_ctas = s_ctas, n_lanes = n_ctas / n_rg;
    auto base_of = [&](int b) { return cached ? s_base[b] : pv.tile_base[b]; };
    const int c = tid;
    int64_t f0 = 0, f1 = 0;
    int seq0 = 0;
    if (c < n_ctas) {
        f0 = c / n_rg;
        if (!s_own) {
            f1 = (f0 + 1) * N / n_lanes;
            f0 = f0 * N / n_lanes;
        }
        for (int hi = B; seq0 + 1 < hi;) {           // the last sequence whose stretch starts at or before f0
            const int mid = (seq0 + hi) / 2;
            if (base_of(mid) <= f0) seq0 = mid;
            else hi = mid;
        }
    }
    if (s_own) {
        for (int u = tid; u < B * d.Hkv; u += (int)blockDim.x) {
            const int b = u / d.Hkv, h = u % d.Hkv, pieces = s_cut[b].x, whole = s_cut[b].y;
            pv.parts[u] = Parts::make(pieces ? (int)s_base[b] + (whole > 1 ? h / whole : h * pieces) : 0, pieces, kind);
        }
        int n_runs = 0, begin = 0;
        if (c < n_ctas) {
            const int nt = s_tiles[seq0], local = c / n_rg - (int)s_base[seq0], pieces = s_cut[seq0].x, whole = s_cut[seq0].y;
            const int head = pieces > 1 ? local / pieces : local, p = local - head * pieces, head0 = head * whole;
            n_runs = min(whole, d.Hkv - head0);
            begin = (seq0 * d.Hkv + head0) * n_rg + c % n_rg * n_runs;       // (a share's runs have its stretches' places)
            SegDesc s;
            s.b = seq0;
            s.t0 = pieces > 1 ? p * nt / pieces : 0;             // (256 pieces of 2^20 tiles at most)
            s.t1 = pieces > 1 ? (p + 1) * nt / pieces : nt;
            s.nt = nt;
            s.P = prefix_len[seq0];
            s.part_slot = pieces == 1 ? -1 : 2 * c + (p + 1 < pieces ? 1 : 0);
            s.pad0 = 0;
            s.slot0 = s_slot[seq0];
            s.pad1 = 0;
            for (int i = 0; i < n_runs; ++i) {
                s.g_rg = (head0 + i) | ((c % n_rg) << 16);
                if (i == 0) pv.cta[c].first = s;
                else pv.segs[begin + i] = s;
            }
        }
        if (c < kPlanMaxCtas) {
            pv.cta[c].n_runs = n_runs;
            pv.cta[c].begin = begin;
            pv.cta[c].kind = kind;
        }
        return;
    }
    // Key tile q of (sequence, kv head) sits at position F + q of the line; position x belongs to share
    // floor(((x + 1) * n - 1) / N) of n.
    for (int u = tid; u < B * d.Hkv; u += (int)blockDim.x) {
        const int b = u / d.Hkv, nt = cached ? s_tiles[b] : pv.tiles[b];
        Parts parts = Parts::make(0, 0, kind);
        if (nt > 0) {
            const int64_t F = base_of(b) + (int64_t)(u % d.Hkv) * (nt + kPairOverheadTiles) + kPairOverheadTiles;
            const int lo = (int)(((F + 1) * n_lanes - 1) / N), hi = (int)(((F + nt) * n_lanes - 1) / N);
            parts = Parts::make(lo, hi - lo + 1, kind);
        }
        pv.parts[u] = parts;
    }
    int first = 0;
    for (int pass = 0; pass < 2; ++pass) {
        int n = 0;
        if (c < n_ctas) {
            SegDesc* out = pv.segs + first;
            int seq = seq0;
            int64_t base = base_of(seq), next = base_of(seq + 1);
            for (int64_t f = f0; f < f1;) {
                while (next <= f) {                  // (f < f1 <= N: ends at the last sequence with tiles at the latest)
                    base = next;
                    next = base_of(++seq + 1);
                }
                const int nt = cached ? s_tiles[seq] : pv.tiles[seq];
                const uint32_t cost = (uint32_t)(nt + kPairOverheadTiles), local = (uint32_t)(f - base);
                const int head = (int)(local / cost), pos = (int)(local - head * cost);
                const int64_t room = f1 - f;
                const int take = (int64_t)(cost - pos) <= room ? (int)cost - pos : (int)room;
                f += take;
                const int t0 = pos > kPairOverheadTiles ? pos - kPairOverheadTiles : 0;
                const int t1 = pos + take > kPairOverheadTiles ? pos + take - kPairOverheadTiles : 0;
                if (t1 <= t0) continue;              // the share ended inside this pair's overhead zone
                if (pass) {
                    SegDesc s;
                    s.b = seq;
                    s.g_rg = head | ((c % n_rg) << 16);          // the stretches of a sequence are in kv-head order
                    s.t0 = t0;
                    s.t1 = t1;
                    s.nt = nt;
                    s.P = prefix_len[seq];
                    s.part_slot = (t0 == 0 && t1 == nt) ? -1 : 2 * c + (t1 < nt ? 1 : 0);
                    s.pad0 = 0;
                    s.slot0 = cached ? s_slot[seq] : seq_start ? seq_start[seq] : 0;
                    s.pad1 = 0;
                    out[n] = s;
                    if (n == 0) pv.cta[c].first = s;
                }
                ++n;
            }
        }
        if (!pass) {                                 // exclusive scan of the counts over the first kPlanMaxCtas threads
            int incl = n;
#pragma unroll
            for (int k = 1; k < 32; k <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, incl, k);
                if (lane >= k) incl += t;
            }
            if (warp < kPlanMaxCtas / 32 && lane == 31) s_warp[warp] = incl;
            __syncthreads();
            if (c < kPlanMaxCtas) {
                int before = 0;
                for (int w = 0; w < warp; ++w) before += s_warp[w];
                first = before + incl - n;
                pv.cta[c].n_runs = n;                // (0 past the last unit)
                pv.cta[c].begin = first;
                pv.cta[c].kind = kind;
            }
        }
    }
}

cudaError_t launch_plan(const Ctx* ctx, const confu_dims& d, const int64_t* seq_start, const int32_t* prefix_len,
                        const int32_t* parent, const int32_t* con_owner, void* plan, int32_t* status, int kind,
                        cudaStream_t st)
{
    // work units of the attention launch the plan is for: one CTA per SM, or one CTA pair per two SMs
    const int units = kind == kPlanPair ? ctx->sm_count / 2 : ctx->sm_count;
    // a warp per sequence, no more threads than that needs (a CTA of 1024 starts 0.5 us later than one of 256)
    const int threads = d.B <= 8 ? 256 : d.B <= 16 ? 512 : kPlanThreads;
    return launch_pdl(plan_kernel, dim3(1), dim3((unsigned)threads), st, d, units, kind, seq_start, prefix_len, parent, con_owner,
                      plan, status);
}

}  // namespace confu
