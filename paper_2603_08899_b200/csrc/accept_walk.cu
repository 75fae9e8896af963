// The acceptance walks, one kernel per rule (see walk.cuh for what they share):
//
//   ratio_walk_kernel        rejection sampling along the tree: ratio tests in fp64 by one warp (a lane per node holds
//                            its token's p and q and updates them with every rejection), residual weights of all
//                            entries in registers; statistics of the rows from row_stats_kernel, or on demand
//   match_walk_kernel        sample-and-match rule (and its greedy form), statistics on demand
//   greedy_walk_kernel       temperature 0 with row statistics: no vocabulary pass at all
//   greedy_lazy_walk_kernel  temperature 0, argmax of a row when the first child of a kept node comes up
#include <type_traits>

#include "walk.cuh"

#include "accept.cuh"

namespace confu {
namespace walk {

__device__ __forceinline__ float warp_max_nan(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max_nan(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// exp((x - M) / temperature) / Z in fp64 of a token's two logits (one call for both: an fp64 exponential is a
// microsecond of latency, and the two overlap)
__device__ __noinline__ double2 probs(float xt, float Mt, float iZt, float xd, float Md, float iZd, double inv_temp)
{
    const double p = exp(((double)xt - (double)Mt) * inv_temp) * (double)iZt;
    const double q = exp(((double)xd - (double)Md) * inv_temp) * (double)iZd;
    return make_double2(p, q);
}

enum { kAccept = 0, kReject = 1, kDraw = 2 };

struct RatioShared {
    Tree tr;
    Exchange ex;
    Search sr;
    float M[2][kMaxTree], iZ_row[2][kMaxTree];       // maximum and inverse normaliser of every row (statistics on demand: of the current node)
    double p[kMaxTree], q[kMaxTree];                 // of every node's token in its parent's rows
    int act, x, nonfinite, degenerate, owner;
    float cs, iZ;
    double iZ64[2];                                  // statistics on demand: inverse normalisers of the current node's rows
    double off, target, total;
};

template <typename T, int E, bool kRagged, bool kLazy>
__global__ void __launch_bounds__(kThreads, 1) ratio_walk_kernel(const Args a, const T* __restrict__ tl, const T* __restrict__ dl, int nch,
                                                              int n_rows, const RowStat* __restrict__ stats)
{
    __shared__ RatioShared sh;
    Tree& tr = sh.tr;
    const cg::cluster_group cluster = cg::this_cluster();
    const int n = (int)cluster.num_blocks(), rank = (int)cluster.block_rank(), b = blockIdx.x / n;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    Span sp = span_of<T>(a.V, rank, n);
    const double inv_temp = 1.0 / (double)a.temperature;
    const float k2 = (float)inv_temp * kLog2e;
    const double k64 = inv_temp * 1.4426950408889634;
    const T* tl_b = tl + (size_t)b * a.T * a.V;
    const T* dl_b = dl + (size_t)b * a.T * a.V;

    cluster_arrive();                                // the peers' shared memory exists: waited for before the first exchange
    asm volatile("griddepcontrol.wait;" ::: "memory");
    to_row<kRagged>(sp, tl_b, a.V);
    prefetch_slice<T, E>(tl_b, sp);                  // the root's rows travel while the tree is fetched and checked
    prefetch_slice<T, E>(dl_b, sp);
    int flag = 0;
    if (!kLazy) {
        // chunk statistics of all rows, half a warp to a row, joined in fp64
        constexpr int kRounds = 2 * kMaxTree / (2 * kWarps);
        const int c = lane & 15, half = 2 * warp + (lane >> 4);
        uint4 v[kRounds];
#pragma unroll
        for (int k = 0; k < kRounds; ++k) {
            const int row = k * 2 * kWarps + half;       // target rows, then draft rows
            v[k] = make_uint4(0xff800000u, 0u, 0u, 0u);
            if (row < 2 * a.T && c < nch)
                v[k] = *reinterpret_cast<const uint4*>(stats + ((size_t)(row / a.T) * n_rows + (size_t)b * a.T + row % a.T) * kStatChunksMax + c);
            flag |= (int)v[k].w;
        }
#pragma unroll
        for (int k = 0; k < kRounds; ++k) {
            const int row = k * 2 * kWarps + half;
            const float m = __uint_as_float(v[k].x);
            float mm = m;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) mm = fmaxf(mm, __shfl_xor_sync(0xffffffffu, mm, o));
            double z = m > -INFINITY ? (double)__uint_as_float(v[k].y) : 0.0;
            z *= joint(m - mm, k64);
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
            if (c == 0 && row < 2 * a.T) { sh.M[row / a.T][row % a.T] = mm; sh.iZ_row[row / a.T][row % a.T] = (float)(1.0 / z); }
        }
    }
    if (tid == 0) { sh.nonfinite = 0; sh.degenerate = 0; }
    load_tree(tr, a, b, a.mode == 1);
    if (flag) atomicMin(&tr.code, (int)CONFU_ST_NONFINITE);
    if (tid > 0 && tid < a.T && tr.code == INT_MAX) {
        const size_t at = (size_t)tr.par[tid] * a.V + tr.tok[tid];
        tr.lt[tid] = to_f32(tl_b[at]);
        tr.ld[tid] = to_f32(dl_b[at]);
        if (!kLazy) {
            const int r = tr.par[tid];
            const double2 pq = probs(tr.lt[tid], sh.M[0][r], sh.iZ_row[0][r], tr.ld[tid], sh.M[1][r], sh.iZ_row[1][r], inv_temp);
            sh.p[tid] = pq.x;
            sh.q[tid] = pq.y;
        }
    }
    __syncthreads();
    cluster_wait();
    if (tr.code != INT_MAX) {
        if (rank == 0) write_failure(a, b, tr.code, true);
        return;
    }

    int parity = 0, cur = 0;
    bool again = false;                              // a node whose residual had no mass: drawn from its target row after all
    for (;;) {
        Raw<T, E, kRagged> xt, xd;
        float p[E], q[E];
        to_row<kRagged>(sp, tl_b + (size_t)cur * a.V, a.V);   // (both matrices are aligned alike)
        xt.load(tl_b + (size_t)cur * a.V, sp);
        xd.load(dl_b + (size_t)cur * a.V, sp);
        // ---- maxima and normalisers of the node's two rows ----
        float wt = 0.f, wd = 0.f;                    // kLazy: this warp's maxima, which p and q are relative to until the first rejection
        if (kLazy) {
            wt = wd = -INFINITY;
#pragma unroll
            for (int e = 0; e < E; ++e) { wt = fmaxf(wt, xt.at(e)); wd = fmaxf(wd, xd.at(e)); }
            const bool bad = nonfinite(xt, sp) || nonfinite(xd, sp);
            wt = warp_max(wt);
            wd = warp_max(wd);
            const float bt = wt == -INFINITY ? 0.f : wt, bd = wd == -INFINITY ? 0.f : wd;
            float st = 0.f, sd = 0.f;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                p[e] = ex2((xt.at(e) - bt) * k2);
                q[e] = ex2((xd.at(e) - bd) * k2);
                st += p[e];
                sd += q[e];
            }
            st = warp_sum(st);
            sd = warp_sum(sd);
            const bool any_bad = __any_sync(0xffffffffu, bad);
            exchange(sh.ex, parity, rank, n, make_uint4(__float_as_uint(any_bad ? NAN : wt), __float_as_uint(st), __float_as_uint(wd), __float_as_uint(sd)));
            if (warp == 0) {
                // eight warps' parts per lane, relative to the lane's own maxima first
                const int r = lane >> 1;
                const uint4* slot = &sh.ex.slot[parity][r < n ? r : 0][(lane & 1) * (kWarps / 2)];
                float lt = -INFINITY, ld = -INFINITY;
                double zt = 0.0, zd = 0.0;
                if (r < n) {
                    for (int w = 0; w < kWarps / 2; ++w) {
                        lt = max_nan(lt, __uint_as_float(slot[w].x));
                        ld = fmaxf(ld, __uint_as_float(slot[w].z));
                    }
                    const float bt2 = lt == -INFINITY ? 0.f : lt, bd2 = ld == -INFINITY ? 0.f : ld;
                    for (int w = 0; w < kWarps / 2; ++w) {
                        zt += (double)(__uint_as_float(slot[w].y) * ex2((__uint_as_float(slot[w].x) - bt2) * k2));
                        zd += (double)(__uint_as_float(slot[w].w) * ex2((__uint_as_float(slot[w].z) - bd2) * k2));
                    }
                }
                const float mt = warp_max_nan(lt), md = warp_max(ld);
                zt = warp_sum(zt * joint(lt - mt, k2));
                zd = warp_sum(zd * joint(ld - md, k2));
                if (lane == 0) {
                    sh.M[0][cur] = mt; sh.M[1][cur] = md;
                    sh.iZ64[0] = 1.0 / zt; sh.iZ64[1] = 1.0 / zd;
                    sh.iZ_row[0][cur] = (float)sh.iZ64[0]; sh.iZ_row[1][cur] = (float)sh.iZ64[1];
                    sh.nonfinite = !(mt == mt);
                }
            }
            parity ^= 1;
        }
        // ---- warp 0: lane i holds the p and q of nodes i and i + 32 where they are children of this one ----
        unsigned long long kids = 0;
        double p0 = 0.0, q0 = 0.0, p1 = 0.0, q1 = 0.0;
        bool no_mass = false;                        // the draft row has no mass left: no further tests
        if (warp == 0) {
            __syncwarp();
            const bool c0 = lane > cur && lane < a.T && tr.par[lane] == cur;
            const bool c1 = lane + 32 > cur && lane + 32 < a.T && tr.par[lane + 32] == cur;
            kids = (unsigned long long)__ballot_sync(0xffffffffu, c0) | ((unsigned long long)__ballot_sync(0xffffffffu, c1) << 32);
            if (again) kids = 0;
            if (kLazy) {
                for (int h = 0; h < 2; ++h) {
                    const int i = lane + 32 * h;
                    if (h ? c1 : c0) {
                        const double2 pq = probs(tr.lt[i], sh.M[0][cur], sh.iZ_row[0][cur], tr.ld[i], sh.M[1][cur], sh.iZ_row[1][cur], inv_temp);
                        sh.p[i] = pq.x;
                        sh.q[i] = pq.y;
                    }
                }
            }
            if (c0) { p0 = sh.p[lane]; q0 = sh.q[lane]; }
            if (c1) { p1 = sh.p[lane + 32]; q1 = sh.q[lane + 32]; }
        }
        const auto Mt = [&] { return sh.M[0][cur]; };
        const auto iZt = [&] { return sh.iZ_row[0][cur]; };
        // weights of the row itself (no rejection): p, with q = 0
        auto target_weights = [&]() {
            if (kLazy) {
                const float f = (float)(joint(wt - Mt(), k2) * sh.iZ64[0]);
#pragma unroll
                for (int e = 0; e < E; ++e) p[e] *= f;
            } else {
#pragma unroll
                for (int e = 0; e < E; ++e) p[e] = ex2((xt.at(e) - Mt()) * k2) * iZt();
            }
        };
        auto send_sums = [&]() {
            double acc = 0.0;
#pragma unroll
            for (int s = 0; s < E / kRun; ++s) {
                float r = 0.f;
#pragma unroll
                for (int j = 0; j < kRun; ++j) r += fmaxf(p[s * kRun + j] - q[s * kRun + j], 0.f);
                acc += (double)r;
            }
            exchange(sh.ex, parity, rank, n, as_quad(warp_sum(acc)));
            parity ^= 1;
        };
        // the next test of this node (warp 0), made known to all threads
        auto decide = [&]() {
            if (warp == 0) {
                int what = kDraw;
                if (kids && !no_mass) {
                    const int c = __ffsll((long long)kids) - 1;
                    kids &= kids - 1;
                    const double pc = __shfl_sync(0xffffffffu, c < 32 ? p0 : p1, c & 31), qc = __shfl_sync(0xffffffffu, c < 32 ? q0 : q1, c & 31);
                    const double u = (double)tr.uni[c];
                    // u < p / q without the division (q = 0: accepted iff p > 0); borderline: |p / q - u| < 1e-5
                    what = u * qc < pc ? kAccept : kReject;
                    const double rem = 1.0 - qc;
                    if (what == kReject && a.mode == 1 && !(rem > 0.0)) no_mass = true;
                    if (lane == 0) {
                        ++tr.tests;
                        if (qc > 0.0 ? fabs(pc - u * qc) < kBorderline * qc : pc == 0.0 && u < kBorderline) ++tr.border_tests;
                        if (what == kAccept) {
                            tr.path[++tr.len] = c;                       // at most T - 1 <= CONFU_MAX_DEPTH of them
                            tr.cur = c;
                        } else {
                            ++tr.hits;
                            sh.x = tr.tok[c];
                            sh.cs = rem > 0.0 ? (float)(1.0 / rem) : 0.f;
                        }
                    }
                }
                if (lane == 0) sh.act = what;
            }
            __syncthreads();
            return sh.act;
        };
        int act = decide();
        bool rejected = false;
        if (act == kReject && !(kLazy && sh.nonfinite)) {
            // residual weights after k rejections: max(p - q, 0), p and q kept in registers from one to the next
            rejected = true;
            target_weights();
            if (kLazy) {
                const float f = (float)(joint(wd - sh.M[1][cur], k2) * sh.iZ64[1]);
#pragma unroll
                for (int e = 0; e < E; ++e) q[e] *= f;
            } else {
#pragma unroll
                for (int e = 0; e < E; ++e) q[e] = ex2((xd.at(e) - sh.M[1][cur]) * k2) * sh.iZ_row[1][cur];
            }
            for (;;) {
                const int x = sh.x;
                const float cs = sh.cs;
                send_sums();
                if (warp == 0) {
                    const double Z = sum_ranks(rank_totals(sh.ex, parity ^ 1, n, [](const uint4& v) { return quad_double(v); }));
                    if (Z > 0.0) {
                        const float iz = (float)(1.0 / Z);
                        if (lane == 0) sh.iZ = iz;
                        p0 = fmax(p0 - q0, 0.0) * (double)iz;
                        p1 = fmax(p1 - q1, 0.0) * (double)iz;
                        if (a.mode == 1) {
                            q0 = tr.tok[lane] == x ? 0.0 : q0 * (double)cs;
                            q1 = tr.tok[lane + 32] == x ? 0.0 : q1 * (double)cs;
                        }
                    } else {
                        if (lane == 0) sh.degenerate = 1;
                        kids = 0;
                    }
                    __syncwarp();
                }
                act = decide();
                if (act != kReject) break;
                const float iz = sh.iZ;
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    p[e] = fmaxf(p[e] - q[e], 0.f) * iz;
                    if (a.mode == 1) q[e] = entry(sp, e) == x ? 0.f : q[e] * cs;
                }
            }
        }
        if (kLazy && sh.nonfinite) {
            if (rank == 0) write_failure(a, b, CONFU_ST_NONFINITE, true);
            return;
        }
        if (act == kAccept) {
            cur = tr.cur;
            __syncthreads();                         // everybody has read it and sh.act before warp 0 writes the next ones
            continue;
        }
        if (rejected && sh.degenerate) {             // no residual mass: the target row is used instead
            __syncthreads();
            again = true;
            continue;
        }
        // ---- the next token: inverse CDF over the residual weights, or over the target row itself ----
        if (!rejected) {
            target_weights();
#pragma unroll
            for (int e = 0; e < E; ++e) q[e] = 0.f;
            send_sums();
        }
        const double u = (double)tr.uni[0];
        if (warp == 0) {
            const double mine = rank_totals(sh.ex, parity ^ 1, n, [](const uint4& v) { return quad_double(v); });
            const double total = sum_ranks(mine);
            double before;
            const int owner = owner_of(mine, u * total, before);
            if (lane == 0) { sh.owner = owner; sh.off = before; sh.target = u * total; sh.total = total; }
        }
        __syncthreads();
        if (sh.owner == rank) {
            bool found;
            double lo = 0.0, hi = 0.0;
            const int pick = locate<E>(sh.sr, sp, sh.off, sh.target, [&](int e) { return fmaxf(p[e] - q[e], 0.f); }, found, lo, hi);
            if (found || (tid == 0 && sh.sr.found == INT_MAX)) {
                a.next_token[b] = pick;
                if (a.counters) a.counters[4 * b + 3] = !found || near_edge(u, lo, hi, sh.total) ? 1 : 0;
            }
        }
        break;
    }
    if (rank == 0) {
        write_path(tr, a, b);
        if (tid == 0 && a.counters) {
            a.counters[4 * b] = tr.tests;
            a.counters[4 * b + 1] = tr.hits;
            a.counters[4 * b + 2] = tr.border_tests;
        }
        if (tid == 0 && sh.degenerate && a.status) a.status[b] = CONFU_ST_DEGENERATE;
    }
}

struct MatchShared {
    Tree tr;
    Exchange ex;
    Search sr;
    int owner, x, done, code;
    float M;
    double off, target, total;
};

// One warp: largest value of the cluster's (value, index) slots in .x and .y, lowest index among equals; NaN if any is.
__device__ __forceinline__ void best_slot(const Exchange& ex, int parity, int n, float& m, int& arg)
{
    const int lane = threadIdx.x & 31, r = lane >> 1;
    m = -INFINITY;
    arg = INT_MAX;
    bool bad = false;
    if (r < n)
        for (int w = 0; w < kWarps / 2; ++w) {
            const uint4 v = ex.slot[parity][r][(lane & 1) * (kWarps / 2) + w];
            const float x = __uint_as_float(v.x);
            bad = bad || !(x == x);
            if (x > m || (x == m && (int)v.y < arg)) { m = x; arg = (int)v.y; }
        }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float om = __shfl_xor_sync(0xffffffffu, m, o);
        const int oa = __shfl_xor_sync(0xffffffffu, arg, o);
        if (om > m || (om == m && oa < arg)) { m = om; arg = oa; }
    }
    if (__any_sync(0xffffffffu, bad)) m = NAN;
}
// A warp's largest entry and its lowest index (INT_MAX: no entry); every lane gets both.
template <typename T, int E, bool kRagged>
__device__ __forceinline__ void warp_best(const Raw<T, E, kRagged>& x, const Span& sp, float& m, int& arg)
{
    m = -INFINITY;
#pragma unroll
    for (int e = 0; e < E; ++e) m = fmaxf(m, x.at(e));
    arg = INT_MAX;
    if (m > -INFINITY) {
#pragma unroll
        for (int e = E - 1; e >= 0; --e)
            if (x.at(e) == m) arg = entry(sp, e);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float om = __shfl_xor_sync(0xffffffffu, m, o);
        const int oa = __shfl_xor_sync(0xffffffffu, arg, o);
        if (om > m || (om == m && oa < arg)) { m = om; arg = oa; }
    }
}

template <typename T, int E, bool kRagged>
__global__ void __launch_bounds__(kThreads, 1) match_walk_kernel(const Args a, const T* __restrict__ tl)
{
    __shared__ MatchShared sh;
    Tree& tr = sh.tr;
    const cg::cluster_group cluster = cg::this_cluster();
    const int n = (int)cluster.num_blocks(), rank = (int)cluster.block_rank(), b = blockIdx.x / n;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    Span sp = span_of<T>(a.V, rank, n);
    const bool greedy = !(a.temperature > 0.f);
    const float k2 = (greedy ? 1.f : 1.f / a.temperature) * kLog2e;
    const T* tl_b = tl + (size_t)b * a.T * a.V;

    cluster_arrive();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    to_row<kRagged>(sp, tl_b, a.V);
    prefetch_slice<T, E>(tl_b, sp);                  // the root's row travels while the tree is fetched and checked
    load_tree(tr, a, b, false);
    if (tid == 0) { sh.code = tr.code == INT_MAX ? 0 : tr.code; sh.done = 0; }
    __syncthreads();
    cluster_wait();
    int parity = 0, cur = 0, next = -1;
    while (!sh.code) {
        Raw<T, E, kRagged> x;
        to_row<kRagged>(sp, tl_b + (size_t)cur * a.V, a.V);
        x.load(tl_b + (size_t)cur * a.V, sp);
        // ---- the row's maximum and, when sampling, the sum of its weights 2^((x - maximum) k2) ----
        const bool bad = __any_sync(0xffffffffu, nonfinite(x, sp));
        float m, w[E];
        int arg = 0;
        if (greedy) {
            warp_best(x, sp, m, arg);
            exchange(sh.ex, parity, rank, n, make_uint4(__float_as_uint(bad ? NAN : m), (uint32_t)arg, 0u, 0u));
        } else {
            m = -INFINITY;
#pragma unroll
            for (int e = 0; e < E; ++e) m = fmaxf(m, x.at(e));
            m = warp_max(m);
            const float base = m == -INFINITY ? 0.f : m;
            double acc = 0.0;
#pragma unroll
            for (int s = 0; s < E / kRun; ++s) {
                float r = 0.f;
#pragma unroll
                for (int j = 0; j < kRun; ++j) {
                    w[s * kRun + j] = ex2((x.at(s * kRun + j) - base) * k2);
                    r += w[s * kRun + j];
                }
                acc += (double)r;
            }
            const uint4 sum = as_quad(warp_sum(acc));
            exchange(sh.ex, parity, rank, n, make_uint4(__float_as_uint(bad ? NAN : m), 0u, sum.x, sum.y));
        }
        const double u = (double)tr.uni[cur];
        if (warp == 0) {
            float M;
            int best;
            best_slot(sh.ex, parity, n, M, best);
            if (!(M == M)) {
                if (lane == 0) sh.code = CONFU_ST_NONFINITE;
            } else if (greedy) {
                if (lane == 0) sh.x = best;
            } else {
                const double mine = rank_totals(sh.ex, parity, n, [&](const uint4& v) {
                    return quad_double(make_uint4(v.z, v.w, 0u, 0u)) * (double)joint_f32(__uint_as_float(v.x) - M, k2);
                });
                const double total = sum_ranks(mine);
                double before;
                const int owner = owner_of(mine, u * total, before);
                if (lane == 0) { sh.owner = owner; sh.off = before; sh.target = u * total; sh.total = total; sh.M = M; }
            }
        }
        __syncthreads();
        if (sh.code) break;
        if (!greedy) {
            if (sh.owner == rank) {
                const float f = joint_f32(m - sh.M, k2);
                bool found;
                double lo = 0.0, hi = 0.0;
                const int pick = locate<E>(sh.sr, sp, sh.off, sh.target, [&](int e) { return w[e] * f; }, found, lo, hi);
                if (found || (tid == 0 && sh.sr.found == INT_MAX)) {
                    const int border = !found || near_edge(u, lo, hi, sh.total) ? 1 : 0;
                    for (int c = 0; c < n; ++c) {
                        int* to = cluster.map_shared_rank(&sh.ex.pick[parity][0], c);
                        to[0] = pick;
                        to[1] = border;
                    }
                }
            }
            __syncwarp();
            cluster_arrive();
            cluster_wait();
        }
        // ---- the child that carries the drawn token ----
        if (warp == 0) {
            const int tok = greedy ? sh.x : sh.ex.pick[parity][0];
            const unsigned c0 = __ballot_sync(0xffffffffu, lane > cur && lane < a.T && tr.par[lane] == cur && tr.tok[lane] == tok);
            const unsigned c1 = __ballot_sync(0xffffffffu, lane + 32 > cur && lane + 32 < a.T && tr.par[lane + 32] == cur && tr.tok[lane + 32] == tok);
            if (lane == 0) {
                ++tr.tests;
                if (!greedy) tr.border_tests += sh.ex.pick[parity][1];
                if (c0 | c1) {
                    tr.cur = c0 ? __ffs(c0) - 1 : __ffs(c1) + 31;
                    tr.path[++tr.len] = tr.cur;
                    ++tr.hits;
                } else {
                    sh.done = 1;
                    sh.x = tok;
                }
            }
        }
        parity ^= 1;
        __syncthreads();
        cur = tr.cur;
        next = sh.x;
        if (sh.done) break;
        __syncthreads();                             // everybody has read them before warp 0 writes the next ones
    }
    if (rank != 0) return;
    if (sh.code) {
        write_failure(a, b, sh.code, true);
        return;
    }
    write_path(tr, a, b);
    if (tid == 0) {
        a.next_token[b] = next;
        if (a.counters) {
            a.counters[4 * b] = tr.tests;
            a.counters[4 * b + 1] = tr.hits;
            a.counters[4 * b + 2] = tr.border_tests;
            a.counters[4 * b + 3] = 0;
        }
    }
}

// ---------------------------------------------------------------------------------------------
// greedy (temperature 0)
// ---------------------------------------------------------------------------------------------
// The deepest kept node, the lowest index among equally deep ones, becomes the end of the path: of the nodes whose
// token is the argmax of their parent's row (`hit`), those with all ancestors in it too.  One warp.
__device__ __forceinline__ void deepest_path(Tree& tr, int T, unsigned long long hit)
{
    const int lane = threadIdx.x & 31;
    int best = 0;                                    // depth << 8 | 255 - node
    for (int i = lane; i < T; i += 32) {
        int d = 0, k = i;
        while (k > 0 && ((hit >> k) & 1ull)) { ++d; k = tr.par[k]; }
        if (k == 0) best = max(best, (d << 8) | (255 - i));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, o));
    if (lane == 0) {
        const int node = 255 - (best & 255);
        tr.len = best >> 8;
        for (int k = node, d = tr.len; k >= 0; k = tr.par[k], --d) tr.path[d] = k;
        tr.cur = node;
    }
    __syncwarp();
}

constexpr int kGreedyThreads = 128;

__global__ void __launch_bounds__(kGreedyThreads) greedy_walk_kernel(const Args a, int nch, const RowStat* __restrict__ stats)
{
    __shared__ Tree tr;
    __shared__ int s_best[kMaxTree];
    const int b = blockIdx.x, tid = threadIdx.x;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    load_tree(tr, a, b, false);
    if (tid < a.T) {
        const RowStat* s = stats + ((size_t)b * a.T + tid) * kStatChunksMax;
        float m = -INFINITY;
        int arg = INT_MAX, flag = 0;
        uint4 st[kStatChunksMax];
#pragma unroll
        for (int c = 0; c < kStatChunksMax; ++c)
            if (c < nch) st[c] = *reinterpret_cast<const uint4*>(s + c);
#pragma unroll
        for (int c = 0; c < kStatChunksMax; ++c) {
            if (c >= nch) break;
            const uint4 v = st[c];
            if (__uint_as_float(v.x) > m) { m = __uint_as_float(v.x); arg = (int)v.z; }
            flag |= (int)v.w;
        }
        s_best[tid] = arg;
        if (flag) atomicMin(&tr.code, (int)CONFU_ST_NONFINITE);
    }
    __syncthreads();
    if (tr.code != INT_MAX) {
        write_failure(a, b, tr.code, true);
        return;
    }
    if (tid < 32) {
        const bool h0 = tid > 0 && tid < a.T && tr.tok[tid] == s_best[tr.par[tid]];
        const bool h1 = tid + 32 < a.T && tr.tok[tid + 32] == s_best[tr.par[tid + 32]];
        const unsigned long long lo = __ballot_sync(0xffffffffu, h0), hi = __ballot_sync(0xffffffffu, h1);
        deepest_path(tr, a.T, lo | (hi << 32));
        if (tid == 0) a.next_token[b] = s_best[tr.cur];
    }
    if (a.counters && tid < 4) a.counters[4 * b + tid] = 0;
    __syncthreads();
    write_path(tr, a, b);
}

struct GreedyShared {
    Tree tr;
    Exchange ex;
    int best[kMaxTree];
    int code;
};

template <typename T, int E, bool kRagged>
__global__ void __launch_bounds__(kThreads, 1) greedy_lazy_walk_kernel(const Args a, const T* __restrict__ tl)
{
    __shared__ GreedyShared sh;
    Tree& tr = sh.tr;
    const cg::cluster_group cluster = cg::this_cluster();
    const int n = (int)cluster.num_blocks(), rank = (int)cluster.block_rank(), b = blockIdx.x / n;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    Span sp = span_of<T>(a.V, rank, n);

    cluster_arrive();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    load_tree(tr, a, b, false);
    if (tid < kMaxTree) sh.best[tid] = -2;
    if (tid == 0) sh.code = tr.code == INT_MAX ? 0 : tr.code;
    __syncthreads();
    cluster_wait();
    int parity = 0;
    // argmax of a node's target row, into sh.best (all CTAs of the cluster take the same branches)
    auto need = [&](int node) {
        Raw<T, E, kRagged> x;
        to_row<kRagged>(sp, tl + ((size_t)b * a.T + node) * a.V, a.V);
        x.load(tl + ((size_t)b * a.T + node) * a.V, sp);
        const bool bad = __any_sync(0xffffffffu, nonfinite(x, sp));
        float m;
        int arg;
        warp_best(x, sp, m, arg);
        exchange(sh.ex, parity, rank, n, make_uint4(__float_as_uint(bad ? NAN : m), (uint32_t)arg, 0u, 0u));
        if (warp == 0) {
            best_slot(sh.ex, parity, n, m, arg);
            if (lane == 0) {
                if (m == m) sh.best[node] = arg;
                else sh.code = CONFU_ST_NONFINITE;
            }
        }
        parity ^= 1;
        __syncthreads();
    };
    if (!sh.code) {
        unsigned long long keep = 1ull;
        for (int i = 1; i < a.T; ++i) {
            const int p = tr.par[i];
            if (!((keep >> p) & 1ull)) continue;
            if (sh.best[p] == -2) {
                need(p);
                if (sh.code) break;
            }
            if (tr.tok[i] == sh.best[p]) keep |= 1ull << i;
        }
        __syncthreads();
        if (!sh.code) {
            if (warp == 0) deepest_path(tr, a.T, keep);
            __syncthreads();
            if (sh.best[tr.cur] == -2) need(tr.cur);
        }
    }
    if (rank != 0) return;
    if (sh.code) {
        write_failure(a, b, sh.code, true);
        return;
    }
    write_path(tr, a, b);
    if (tid == 0) a.next_token[b] = sh.best[tr.cur];
    if (a.counters && tid < 4) a.counters[4 * b + tid] = 0;
}

// ---------------------------------------------------------------------------------------------
// launches
// ---------------------------------------------------------------------------------------------
template <typename... P, typename... A>
static cudaError_t launch_cluster(void (*kernel)(P...), OncePerDevice& attr_done, int B, int n, cudaStream_t st, A... args)
{
    cudaError_t e = attr_done.run([&] { return cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1); });
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attrs[2];
    attrs[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attrs[0].val.programmaticStreamSerializationAllowed = 1;
    attrs[1].id = cudaLaunchAttributeClusterDimension;
    attrs[1].val.clusterDim.x = (unsigned)n;
    attrs[1].val.clusterDim.y = attrs[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(B * n));
    cfg.blockDim = dim3(kThreads);
    cfg.stream = st;
    cfg.attrs = attrs;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Where all rows are aligned a walk without the code for ends of rows (kRagged) is taken if it is the faster one, us with it -> without: ratio
// rule, bf16, statistics given, 16 sequences of V 4096 (8 entries a thread) 18.9 -> 18.6, of 128256 (32) 60.0 -> 57.0, on demand 23.1 ->
// 22.4, 38.7 -> 38.4; fp32, 5 of 151936 (24) 91.8 -> 89.8, but 9 of them (40) 71.0 -> 72.7; argmax on demand up to 16 entries, fp32, V
// 4096 12.0 -> 11.8, but bf16, 16 of 128256 17.9 -> 18.5; sample-and-match from 24 on, bf16, 9 of 151936 14.2 -> 13.8, but 4 of 32000 (8)
// 13.1 -> 14.0.
template <bool kTight, typename F>
static cudaError_t by_alignment(bool aligned, F f)
{
    if constexpr (kTight) {
        if (aligned) return f(std::false_type());
    }
    return f(std::true_type());
}
template <typename T, int E>
static cudaError_t walk_e(int n, int B, const Args& a, const T* tl, const T* dl, int nch, const RowStat* stats, cudaStream_t st)
{
    const bool aligned = places<T>(a.V) == a.V;
    if (!(a.temperature > 0.f))
        return by_alignment<E <= 16>(aligned, [&](auto ragged) {
            static OncePerDevice once;
            return launch_cluster(greedy_lazy_walk_kernel<T, E, decltype(ragged)::value>, once, B, n, st, a, tl);
        });
    if (!stats)
        return by_alignment<true>(aligned, [&](auto ragged) {
            static OncePerDevice once;
            return launch_cluster(ratio_walk_kernel<T, E, decltype(ragged)::value, true>, once, B, n, st, a, tl, dl, nch, B * a.T, stats);
        });
    return by_alignment<(sizeof(T) * E < 160)>(aligned, [&](auto ragged) {
        static OncePerDevice once;
        return launch_cluster(ratio_walk_kernel<T, E, decltype(ragged)::value, false>, once, B, n, st, a, tl, dl, nch, B * a.T, stats);
    });
}
template <typename T, int E>
static cudaError_t match_e(int n, int B, const Args& a, const T* tl, cudaStream_t st)
{
    return by_alignment<E >= 24>(places<T>(a.V) == a.V, [&](auto ragged) {
        static OncePerDevice once;
        return launch_cluster(match_walk_kernel<T, E, decltype(ragged)::value>, once, B, n, st, a, tl);
    });
}

// CTAs per sequence and entries per thread.  A walk is as fast as its slices are small, so a small batch with a large
// vocabulary takes 16 CTAs a sequence (B 1, V 128256, ratio rule: 15-20 us against 24-28 us with 8; sample-and-match 6.7
// against 8.1 us): up to 7 sequences, because 7 clusters of 16 run at once on 148 SMs (32 sequences: 78 against 61 us).
// A small vocabulary gains nothing (V 1000: 13.9 against 12.1 us), and one above 163840 entries needs the 16 CTAs to
// fit the registers.  Two CTAs share an SM: more sequences than that holds at 8 take fewer CTAs each, as long as a thread keeps 16
// entries or less (greedy sample-and-match, 256 sequences of V 1000: 8 CTAs 98.8 us, one 14.3; of V 32000: 8 102.9, 4 56.2;
// ratio rule 154 / 33 and 377 / 276).
template <typename F>
static cudaError_t by_vocabulary(int B, int V, F f)
{
    const bool wide = (V > 8 * kStrip && B <= 7) || V > 8 * 5 * kStrip;
    int n = wide ? 16 : 8;
    while (n > 1 && B * n > 2 * 148 && V <= n / 2 * 2 * kStrip) n /= 2;
    const int strips = (V + n * kStrip - 1) / (n * kStrip);
    switch (strips) {
        case 0: case 1: return f(std::integral_constant<int, 8>(), n);
        case 2: return f(std::integral_constant<int, 16>(), n);
        case 3: return f(std::integral_constant<int, 24>(), n);
        case 4: return f(std::integral_constant<int, 32>(), n);
        default: return f(std::integral_constant<int, 40>(), n);
    }
}

template <typename T>
static cudaError_t walk_t(int B, const Args& a, const void* tl, const void* dl, int nch, const RowStat* stats, cudaStream_t st)
{
    return by_vocabulary(B, places<T>(a.V), [&](auto e, int n) {
        return walk_e<T, decltype(e)::value>(n, B, a, (const T*)tl, (const T*)dl, nch, stats, st);
    });
}
template <typename T>
static cudaError_t match_t(int B, const Args& a, const void* tl, cudaStream_t st)
{
    return by_vocabulary(B, places<T>(a.V), [&](auto e, int n) { return match_e<T, decltype(e)::value>(n, B, a, (const T*)tl, st); });
}

}  // namespace walk

cudaError_t launch_walk(int logit_dtype, int B, int T, int C, int V, const void* tl, const void* dl, const int32_t* tokens,
                        const int32_t* parent, const int32_t* con_owner, const float* uniforms, float temperature, int mode,
                        int nch, const RowStat* stats, int32_t* accept_len, int32_t* path, int32_t* next_token,
                        int32_t* future_row, int32_t* counters, int32_t* status, cudaStream_t st)
{
    const bool greedy = !(temperature > 0.f);
    const walk::Args a = {T, C, V, tokens, parent, con_owner, greedy ? nullptr : uniforms, temperature, mode,
                          accept_len, path, next_token, future_row, counters, status};
    if (greedy && stats) {
        cudaLaunchAttribute pdl[1];
        pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        pdl[0].val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)B);
        cfg.blockDim = dim3(walk::kGreedyThreads);
        cfg.stream = st;
        cfg.attrs = pdl;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, walk::greedy_walk_kernel, a, nch, stats);
    }
    if (logit_dtype == CONFU_F32) return walk::walk_t<float>(B, a, tl, dl, nch, stats, st);
    return walk::walk_t<__nv_bfloat16>(B, a, tl, dl, nch, stats, st);
}

cudaError_t launch_accept_match(int B, int T, int C, int V, int logit_dtype, const void* tl, const int32_t* tokens,
                                const int32_t* parent, const int32_t* con_owner, const float* uniforms,
                                float temperature, int32_t* accept_len, int32_t* path, int32_t* next_token,
                                int32_t* future_row, int32_t* counters, int32_t* status, cudaStream_t st)
{
    if (B == 0) return cudaSuccess;
    const walk::Args a = {T, C, V, tokens, parent, con_owner, temperature > 0.f ? uniforms : nullptr, temperature, 0,
                          accept_len, path, next_token, future_row, counters, status};
    if (logit_dtype == CONFU_F32) return walk::match_t<float>(B, a, tl, st);
    return walk::match_t<__nv_bfloat16>(B, a, tl, st);
}

}  // namespace confu
