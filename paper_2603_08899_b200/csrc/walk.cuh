// What the acceptance walks share: a thread-block cluster per sequence, each CTA holding its slice of the
// current node's rows in registers, sums exchanged through distributed shared memory.
//
// The walk is a serial chain of decisions, each behind a reduction over the vocabulary: what it costs is
// latency.  So a node's rows are read once, the weights stay in registers from one rejection to the next
// (re-reading both rows and redoing the k-level recursion per pass was 8-10 us per rejection), a
// reduction is warp sums -> one store per warp and peer -> one cluster barrier, everything about the tree
// (tokens, parents, uniforms, each token's two logits, the row statistics of all nodes) is fetched before the walk
// starts, and each rule is a kernel of its own (one kernel with every branch was 160 KB of code, and fetching
// it was most of a cold walk).  B 1, V 128256: 67 -> 15-20 us; B 8 with statistics on demand: 140 -> 45 us; B 32: 124 -> 61 us;
// sample-and-match, B 16, V 151936: 38 -> 26 us.
#pragma once

#include <cooperative_groups.h>
#include <limits.h>

#include "common.cuh"

namespace confu {
namespace walk {

namespace cg = cooperative_groups;

constexpr int kThreads = 512, kWarps = kThreads / 32;
constexpr int kRun = 8;                              // consecutive entries of a thread
constexpr int kStrip = kThreads * kRun;              // entries a CTA holds per kRun registers
constexpr int kMaxRanks = 16;
constexpr double kBorderline = 1e-5;

struct Tree {
    int tok[kMaxTree], par[kMaxTree], own[kMaxTree];
    float uni[kMaxTree];
    float lt[kMaxTree], ld[kMaxTree];                // logits of node i's token in its parent's target and draft row
    int path[kPathLen];
    int code, cur, len, tests, hits, border_tests;
};

struct Exchange {
    uint4 slot[2][kMaxRanks][kWarps];                // [parity][rank][warp]
    int pick[2][2];                                  // [parity]: entry found by its owner, 1: borderline
};

// search inside the owner CTA
struct Search {
    double tot[8 * kWarps];                          // [strip][warp]
    double off, target;
    int at, found, last;
};

// ---------------------------------------------------------------------------------------------
// slices
// ---------------------------------------------------------------------------------------------
// A row is counted from the 16-byte boundary at or before its first entry, `shift` places earlier, so that vectors can be loaded
// whatever the vocabulary size is (rows that start anywhere, entry by entry: B 3, V 77777, ratio rule with statistics 49 us, now 31).
// kRagged: a row's bytes are no multiple of 16, so shifts differ from row to row.  Without it the code for ends of rows, which aligned rows
// never run, is left out: it costs registers (ratio rule, bf16, 32 entries a thread: spill loads 196 bytes with it, 132 without).
// CTA `rank` of n owns places [rank * chunk, (rank + 1) * chunk), chunk a multiple of 8; run s of thread t starts at place
// rank * chunk + s * kStrip + 8 t.
struct Span {
    int base, lim;                                   // the CTA's places
    int shift, end;                                  // of the present row: place of its first entry, first place past its last one or past lim
};
// places that a row of V entries takes, whatever its shift
template <typename T> __host__ __device__ constexpr int places(int V) { return ((size_t)V * sizeof(T)) % 16 == 0 ? V : V + 16 / (int)sizeof(T) - 1; }
template <typename T>
__device__ __forceinline__ Span span_of(int V, int rank, int n)
{
    const int all = places<T>(V), chunk = ((all + n - 1) / n + kRun - 1) / kRun * kRun;
    Span s;
    s.base = min(rank * chunk, all);
    s.lim = min(s.base + chunk, all);
    s.shift = 0;
    s.end = s.lim;
    return s;
}
template <bool kRagged, typename T>
__device__ __forceinline__ void to_row(Span& s, const T* row, int V)
{
    if (!kRagged) return;
    s.shift = (int)((reinterpret_cast<uintptr_t>(row) & 15u) / sizeof(T));
    s.end = min(s.lim, V + s.shift);
}

// E entries of a row as they lie in memory (bf16: two to a word); places outside the slice or the row are -inf.
template <typename T, int E, bool kRagged> struct Raw;
template <int E, bool kRagged> struct Raw<__nv_bfloat16, E, kRagged> {
    uint32_t w[E / 2];
    __device__ __forceinline__ void load(const __nv_bfloat16* row, const Span& sp)
    {
        const uint16_t* r = reinterpret_cast<const uint16_t*>(row) - sp.shift;
        const int i = sp.base + (int)threadIdx.x * kRun;
#pragma unroll
        for (int s = 0; s < E / kRun; ++s) {
            uint4 v = make_uint4(0xff80ff80u, 0xff80ff80u, 0xff80ff80u, 0xff80ff80u);
            if ((!kRagged || s > 0 || i >= sp.shift) && i + s * kStrip + kRun <= sp.end) v = *reinterpret_cast<const uint4*>(r + i + s * kStrip);
            w[4 * s] = v.x; w[4 * s + 1] = v.y; w[4 * s + 2] = v.z; w[4 * s + 3] = v.w;
        }
        if (!kRagged || (sp.shift | sp.end % kRun) == 0) return;
        // the vectors that hold the row's first and last entries
        auto piece = [&](int k, int j) {
            const int a = k + 2 * j;
            const uint32_t lo = a >= sp.shift && a < sp.end ? r[a] : 0xff80u, hi = a + 1 >= sp.shift && a + 1 < sp.end ? r[a + 1] : 0xff80u;
            return lo | (hi << 16);
        };
        if (i < sp.shift) {
#pragma unroll
            for (int j = 0; j < kRun / 2; ++j) w[j] = piece(i, j);
        }
        const int k = sp.end / kRun * kRun, at = (k - i) / kStrip;
        if (k < sp.end && k >= sp.base && (k - sp.base) % kStrip == (int)threadIdx.x * kRun && k >= sp.shift) {
#pragma unroll
            for (int j = 0; j < kRun / 2; ++j) {
                const uint32_t v = piece(k, j);
#pragma unroll
                for (int s = 0; s < E / kRun; ++s) w[4 * s + j] = s == at ? v : w[4 * s + j];
            }
        }
    }
    __device__ __forceinline__ float at(int e) const { return __uint_as_float((e & 1) ? (w[e >> 1] & 0xffff0000u) : (w[e >> 1] << 16)); }
};
template <int E, bool kRagged> struct Raw<float, E, kRagged> {
    float x[E];
    __device__ __forceinline__ void load(const float* row, const Span& sp)
    {
        const float* r = row - sp.shift;
        const int i = sp.base + (int)threadIdx.x * kRun;
#pragma unroll
        for (int h = 0; h < E / 4; ++h) {
            const int k = i + h / 2 * kStrip + h % 2 * 4;
            float4 v = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
            if ((!kRagged || h > 0 || i >= sp.shift) && k + 4 <= sp.end) v = *reinterpret_cast<const float4*>(r + k);
            x[4 * h] = v.x; x[4 * h + 1] = v.y; x[4 * h + 2] = v.z; x[4 * h + 3] = v.w;
        }
        if (!kRagged || (sp.shift | sp.end % 4) == 0) return;
        auto piece = [&](int k) { return k >= sp.shift && k < sp.end ? r[k] : -INFINITY; };
        if (i < sp.shift) {
#pragma unroll
            for (int j = 0; j < 4; ++j) x[j] = piece(i + j);
        }
        const int k = sp.end / 4 * 4, at = (k - i) / kStrip * 2 + (k - sp.base) % kRun / 4;
        if (k < sp.end && k >= sp.base && (k - sp.base) % kStrip / kRun == (int)threadIdx.x && k >= sp.shift) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float v = piece(k + j);
#pragma unroll
                for (int h = 0; h < E / 4; ++h) x[4 * h + j] = h == at ? v : x[4 * h + j];
            }
        }
    }
    __device__ __forceinline__ float at(int e) const { return x[e]; }
};
// asks for a row's slice to be brought into L2 (a hint: the loads come later)
template <typename T, int E>
__device__ __forceinline__ void prefetch_slice(const T* row, const Span& sp)
{
#pragma unroll
    for (int s = 0; s < E / kRun; ++s) {
        const int i = sp.base + s * kStrip + (int)threadIdx.x * kRun - sp.shift;
        if (i >= 0 && i + sp.shift < sp.end) asm volatile("prefetch.global.L2 [%0];" ::"l"(row + i));
    }
}
// vocabulary index of a thread's entry e (negative: before the row)
__device__ __forceinline__ int entry(const Span& sp, int e) { return sp.base - sp.shift + (e / kRun) * kStrip + (int)threadIdx.x * kRun + e % kRun; }

// an entry that belongs to the slice and is not a finite number (padding is -inf and does not count)
template <typename T, int E, bool kRagged>
__device__ __forceinline__ bool nonfinite(const Raw<T, E, kRagged>& r, const Span& sp)
{
    bool bad = false;
#pragma unroll
    for (int e = 0; e < E; ++e) bad = bad || (!(fabsf(r.at(e)) <= 3.0e38f) && (unsigned)entry(sp, e) < (unsigned)(sp.end - sp.shift));
    return bad;
}

// ---------------------------------------------------------------------------------------------
// exchange
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// This warp's 16 bytes (the same in every lane) go to every CTA of the cluster; on return everybody's are there.
// A slot is used again two exchanges later: by then every CTA has passed a barrier behind its last read of it.
__device__ __forceinline__ void exchange(Exchange& ex, int parity, int rank, int n, uint4 v)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane < n) *cg::this_cluster().map_shared_rank(&ex.slot[parity][rank][warp], lane) = v;
    __syncwarp();
    cluster_arrive();
    cluster_wait();
}
__device__ __forceinline__ uint4 as_quad(double d)
{
    const long long b = __double_as_longlong(d);
    return make_uint4((uint32_t)b, (uint32_t)(b >> 32), 0u, 0u);
}
__device__ __forceinline__ double quad_double(const uint4& q) { return __longlong_as_double((long long)(((uint64_t)q.y << 32) | q.x)); }

// 2^(d k) for d <= 0 (0 for -infinity): the factor between two parts of a row whose weights are relative to maxima d apart.  A
// second exponential of the exponential unit's precision on top of the entry's own would double a weight's error, so the
// sums of a row's parts are joined in fp64.  The power series of 2^f = e^(f ln 2) to the 9th power (|f| <= 1/2: within 7e-12), by
// hand so that several go side by side (statistics and ratio rule at batch 1: 27.3 us with ex2, 28.4 with calls
// of exp2, 27.8 so).
__device__ __forceinline__ double joint(float d, double k)
{
    const double a = fmax((double)d * k, -1100.0), t = a + 6755399441055744.0;      // 1.5 * 2^52: a, rounded, in the low word
    const int n = __double2loint(t);
    const double f = (a - (t - 6755399441055744.0)) * 0.69314718055994531;
    double p = fma(f, 1.0 / 362880.0, 1.0 / 40320.0);
    p = fma(p, f, 1.0 / 5040.0);
    p = fma(p, f, 1.0 / 720.0);
    p = fma(p, f, 1.0 / 120.0);
    p = fma(p, f, 1.0 / 24.0);
    p = fma(p, f, 1.0 / 6.0);
    p = fma(p, f, 0.5);
    p = fma(p, f, 1.0);
    p = fma(p, f, 1.0);
    return n < -1000 ? 0.0 : __hiloint2double(__double2hiint(p) + (n << 20), __double2loint(p));
}

// The same rounded to fp32 (error at most 1.3 * 2^-24), for where a lane has eight of them on the critical path (sample-and-match, B 16,
// V 151936: 25.3 us with ex2, 25.9 so, 26.6 and more in fp64): the argument and its product with ln 2 as sums of two fp32
// numbers, then the power series of e^t to the 7th power (|t| <= ln 2 / 2: within 5e-9).
__device__ __forceinline__ float joint_f32(float d, float k2)
{
    const float ah = d * k2, al = fmaf(d, k2, -ah), n = rintf(ah), r = ah - n;
    constexpr float kLn2 = 0.69314718f, kLn2Lo = -1.9046543e-9f;                 // their sum is ln 2 to 2^-50
    const float t = r * kLn2, tl = fmaf(r, kLn2, -t) + fmaf(al, kLn2, r * kLn2Lo);
    float p = fmaf(t, 1.f / 5040.f, 1.f / 720.f);
    p = fmaf(p, t, 1.f / 120.f);
    p = fmaf(p, t, 1.f / 24.f);
    p = fmaf(p, t, 1.f / 6.f);
    p = fmaf(p, t, 0.5f);
    const float pt = p * t, u = fmaf(fmaf(pt, t, t), tl, tl);                      // e^t tl
    p = 1.f + (t + fmaf(pt, t, u));
    return n < -126.f ? 0.f : p * __int_as_float(((int)n + 127) << 23);
}

// One warp: the CTAs' totals, rank c's in lanes 2 c and 2 c + 1 (0 past the last rank); f turns a slot into its
// share.  The order of every sum is fixed.
template <typename F>
__device__ __forceinline__ double rank_totals(const Exchange& ex, int parity, int n, F f)
{
    const int lane = threadIdx.x & 31, r = lane >> 1;
    double a = 0.0;
    if (r < n) {
#pragma unroll
        for (int w = 0; w < kWarps / 2; ++w) a += f(ex.slot[parity][r][(lane & 1) * (kWarps / 2) + w]);
    }
    return a + __shfl_xor_sync(0xffffffffu, a, 1);
}
// sum over the ranks of what rank_totals returned
__device__ __forceinline__ double sum_ranks(double a)
{
#pragma unroll
    for (int o = 2; o < 32; o <<= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    return a;
}
// One warp: which rank's share holds `target` (running sums in rank order), and the sum of all shares before it.
// When rounding leaves none: the last rank with a positive share.
__device__ __forceinline__ int owner_of(double a, double target, double& before)
{
    const int lane = threadIdx.x & 31;
    double incl = a;                                 // inclusive sums over ranks (pairs of lanes hold the same rank)
#pragma unroll
    for (int o = 2; o < 32; o <<= 1) {
        const double t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    const unsigned hit = __ballot_sync(0xffffffffu, a > 0.0 && incl > target), mass = __ballot_sync(0xffffffffu, a > 0.0);
    const int src = hit ? __ffs(hit) - 1 : mass ? (31 - __clz(mass)) : 0;
    before = __shfl_sync(0xffffffffu, incl - a, src);
    return src >> 1;
}

// ---------------------------------------------------------------------------------------------
// inverse CDF inside the owner CTA (all its threads): the first entry whose running sum, starting at `off`,
// exceeds `target`; when rounding leaves none, the last entry with a positive weight.  w(e): weight of entry e.
// Returns the vocabulary index to every thread; lo, hi: running sums before and behind it (found: not by the
// fallback), in the thread that found it only.
// ---------------------------------------------------------------------------------------------
template <int E, typename W>
__device__ __forceinline__ int locate(Search& sr, const Span& sp, double off, double target, W w, bool& mine, double& lo, double& hi)
{
    constexpr int S = E / kRun;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) { sr.at = -1; sr.found = INT_MAX; sr.last = -1; }
    double incl[S], own[S];
#pragma unroll
    for (int s = 0; s < S; ++s) {
        float a = 0.f;
#pragma unroll
        for (int j = 0; j < kRun; ++j) a += w(s * kRun + j);
        own[s] = incl[s] = (double)a;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double t = __shfl_up_sync(0xffffffffu, incl[s], o);
            if (lane >= o) incl[s] += t;
        }
        if (lane == 31) sr.tot[s * kWarps + warp] = incl[s];
    }
    __syncthreads();
    if (warp == 0) {                                 // running sums over [strip][warp]: 4 consecutive ones per lane
        constexpr int n = S * kWarps, per = (n + 31) / 32;
        double part[per], a = 0.0;
#pragma unroll
        for (int i = 0; i < per; ++i) {
            part[i] = lane * per + i < n ? sr.tot[lane * per + i] : 0.0;
            a += part[i];
        }
        double inc = a;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        double run = off + (inc - a);
        int at = -1;
        double at_off = 0.0;
#pragma unroll
        for (int i = 0; i < per; ++i) {
            if (at < 0 && lane * per + i < n && run + part[i] > target) { at = lane * per + i; at_off = run; }
            run += part[i];
        }
        const unsigned hit = __ballot_sync(0xffffffffu, at >= 0);
        if (hit && lane == __ffs(hit) - 1) { sr.at = at; sr.off = at_off; }
    }
    __syncthreads();
    mine = false;
    if (sr.at >= 0 && (sr.at % kWarps) == warp) {
        const int strip = sr.at / kWarps;
        float wt[kRun];
        double run = 0.0;
#pragma unroll
        for (int s = 0; s < S; ++s) {                // (selects, so that the arrays stay in registers)
            run = s == strip ? sr.off + (incl[s] - own[s]) : run;
#pragma unroll
            for (int j = 0; j < kRun; ++j) wt[j] = s == strip ? w(s * kRun + j) : s == 0 ? 0.f : wt[j];
        }
        int got = -1;
#pragma unroll
        for (int j = 0; j < kRun; ++j) {
            const double before = run;
            run += (double)wt[j];
            if (got < 0 && run > target) { got = sp.base - sp.shift + strip * kStrip + tid * kRun + j; lo = before; hi = run; }
        }
        const unsigned hit = __ballot_sync(0xffffffffu, got >= 0);
        if (hit && lane == __ffs(hit) - 1) { sr.found = got; mine = true; }
    }
    __syncthreads();
    if (sr.found == INT_MAX) {                       // rounding pushed the target past the last running sum
        int last = -1;
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (w(e) > 0.f) last = max(last, entry(sp, e));
        if (last >= 0) atomicMax(&sr.last, last);
        __syncthreads();
        return max(sr.last, 0);
    }
    return sr.found;
}
// a draw u is borderline when it lies within 1e-5 of an edge of the cell [lo, hi) / total
__device__ __forceinline__ bool near_edge(double u, double lo, double hi, double total)
{
    return fmin(fabs(u * total - lo), fabs(hi - u * total)) < kBorderline * total;
}

// ---------------------------------------------------------------------------------------------
// tree data, validation, outputs
// ---------------------------------------------------------------------------------------------
struct Args {
    int T, C, V;
    const int32_t *tokens, *parent, *con_owner;
    const float* uniforms;
    float temperature;
    int mode;
    int32_t *accept_len, *path, *next_token, *future_row, *counters, *status;
};

// Fetches tokens, parents, owners and uniforms of sequence b and checks them; on return (after a
// barrier) tr.code is the lowest code met, INT_MAX if none.  siblings: also refuse equal tokens among siblings.
__device__ __forceinline__ void load_tree(Tree& tr, const Args& a, int b, bool siblings)
{
    const int tid = threadIdx.x;
    if (tid < a.T) {
        tr.tok[tid] = a.tokens[(size_t)b * a.T + tid];
        tr.par[tid] = a.parent[(size_t)b * a.T + tid];
        tr.uni[tid] = a.uniforms ? a.uniforms[(size_t)b * a.T + tid] : 0.f;
    } else if (tid >= kMaxTree && tid < kMaxTree + a.C)
        tr.own[tid - kMaxTree] = a.con_owner[(size_t)b * a.C + tid - kMaxTree];
    if (tid == 0) {
        tr.code = INT_MAX;
        tr.cur = tr.len = tr.tests = tr.hits = tr.border_tests = 0;
        tr.path[0] = 0;
    }
    __syncthreads();
    if (tid < a.T) {
        const int p = tr.par[tid], x = tr.tok[tid];
        int code = INT_MAX;
        if (tid == 0 ? p != -1 : (p < 0 || p >= tid)) code = CONFU_ST_BAD_PARENT;
        else if (x < 0 || x >= a.V) code = CONFU_ST_BAD_TOKEN;
        if (code != INT_MAX) atomicMin(&tr.code, code);
    } else if (tid >= kMaxTree && tid < kMaxTree + a.C) {
        const int o = tr.own[tid - kMaxTree];
        if (o < 0 || o >= a.T) atomicMin(&tr.code, (int)CONFU_ST_BAD_OWNER);
    }
    if (siblings) {
        for (int k = tid; k < kMaxTree * a.T; k += (int)blockDim.x) {
            const int i = k % kMaxTree, j = k / kMaxTree;
            if (i > 0 && i < j && tr.par[i] == tr.par[j] && tr.tok[i] == tr.tok[j]) atomicMin(&tr.code, (int)CONFU_ST_DUP_SIBLING);
        }
    }
    __syncthreads();
}

// what a sequence gets whose walk could not be made (one CTA writes)
__device__ __forceinline__ void write_failure(const Args& a, int b, int code, bool counters)
{
    const int tid = threadIdx.x;
    if (tid < kPathLen) a.path[(size_t)b * kPathLen + tid] = tid == 0 ? 0 : -1;
    if (tid == 0) {
        a.accept_len[b] = 0;
        a.next_token[b] = -1;
        if (a.future_row) a.future_row[b] = -1;
        if (a.status) a.status[b] = code;
    }
    if (counters && a.counters && tid < 4) a.counters[4 * b + tid] = 0;
}

// accepted path, its length, and the contemplate row of the last accepted node or of its nearest ancestor that
// owns one (one CTA writes, after a barrier behind the last change of tr)
__device__ __forceinline__ void write_path(const Tree& tr, const Args& a, int b)
{
    const int tid = threadIdx.x;
    if (tid >= 32 && tid - 32 < kPathLen) a.path[(size_t)b * kPathLen + tid - 32] = tid - 32 <= tr.len ? tr.path[tid - 32] : -1;
    if (tid < 32) {
        if (tid == 0) a.accept_len[b] = tr.len;
        int fr = -1;
        for (int n = tr.cur; n >= 0 && fr < 0; n = tr.par[n]) {
            const unsigned lo = __ballot_sync(0xffffffffu, tid < a.C && tr.own[tid] == n);
            const unsigned hi = __ballot_sync(0xffffffffu, tid + 32 < a.C && tr.own[tid + 32] == n);
            if (lo) fr = a.T + __ffs(lo) - 1;
            else if (hi) fr = a.T + 32 + __ffs(hi) - 1;
        }
        if (tid == 0 && a.future_row) a.future_row[b] = fr;
    }
}

}  // namespace walk
}  // namespace confu
