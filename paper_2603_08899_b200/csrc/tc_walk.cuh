// What the tensor-core attention kernels share about walking a CTA's share of the work: the runs of
// key tiles the plan lists per CTA (or per CTA pair), and which keys of a tile a query row may see.
#pragma once

#include "tc_ptx.cuh"

namespace confu {
namespace tc {

constexpr int kTileBytes = kTileKeys * kD * 2;      // one 128-key tile of K or V of one kv head: 32 KB
constexpr int kHalfTile = kTileBytes / 2;           // one 64-wide half of the head dim: [128 rows][128 B]

struct Segment {
    int b, g, rg;      // sequence, kv head, group of query rows
    int t0, t1;        // tiles [t0, t1) of this pair
    int nt, nkt;       // tiles of the pair; key tiles (the soft-prompt tile, if any, is tile nkt)
    // first tile with keys that not every row sees, the first that reaches past the prefix: worked out once a run.  (As a comparison of
    // the tile's end, in 64 bits, with the prefix in front of every tile's or half tile's maximum: 32 sequences of 512..16384, E4M3 4950
    // us a step of 16 layers, now 4741, bf16 6200 -> 6114; batch 1, R 120, 32 layers 615 -> 602; 8 sequences 837 -> 823.)
    int masked;
    int64_t P;         // prefix length
    int64_t slot0;     // packed pool: the sequence's first slot
    int part_slot;     // -1: the range covers the whole pair, write the output directly
};

// The runs of key tiles of a work unit (CTA or CTA pair), in walking order: the first from the unit's own record in
// the plan (one read tells a role what to start with), the others from 48-byte descriptors.
struct Walker {
    const SegDesc* cur;
    int left;
    bool soft;
    // The unit's first run; false when it has nothing to do, or when the plan is for another kind of unit.
    __device__ bool begin(const PlanView& v, const Params& p, int unit, int kind, Segment& s)
    {
        const uint4* q = reinterpret_cast<const uint4*>(v.cta + unit);
        const uint4 w0 = __ldg(q), w1 = __ldg(q + 1), w2 = __ldg(q + 2), w3 = __ldg(q + 3);
        soft = p.d.S > 0;
        cur = v.segs + (int)w3.y;
        left = (int)w3.z == kind ? (int)w3.x : 0;
        take(s, w0, w1, w2);
        return left > 0;
    }
    // The next run; false when the share is used up.
    __device__ bool next(Segment& s)
    {
        if (--left <= 0) return false;
        const uint4* q = reinterpret_cast<const uint4*>(++cur);
        take(s, __ldg(q), __ldg(q + 1), __ldg(q + 2));
        return true;
    }

private:
    __device__ void take(Segment& s, const uint4& w0, const uint4& w1, const uint4& w2) const
    {
        s.b = (int)w0.x;
        s.g = (int)(w0.y & 0xffffu);
        s.rg = (int)(w0.y >> 16);
        s.t0 = (int)w0.z;
        s.t1 = (int)w0.w;
        s.nt = (int)w1.x;
        s.nkt = s.nt - (soft ? 1 : 0);
        s.P = (int)w1.y;
        s.masked = (int)w1.y / kTileKeys;
        s.part_slot = (int)w1.z;
        s.slot0 = (int64_t)(((uint64_t)w2.y << 32) | w2.x);
    }
};

// What the CTA reads first, its first K tile and Q, into L2 while the kernels before this one still run (kXStep: columns of a K box).
// A hint: the plan may not be there yet, K and Q may still be written.  So nothing that is read here is used for anything else,
// it is read past L1, and a box that lies outside its tensor is not fetched.  One lane of a warp that has nothing else to do, before
// griddepcontrol.wait (the producer's own lane would start its loads late: prefix 8192 +0.7 %).  A step of 28 layers at batch 1,
// prefix 2048: 395 -> 388 us; 32 layers, prefix 4096: 505 -> 501; 8 sequences of 101..3001, 32 layers with their appends: 855 -> 837;
// 27 of 39..794, 9 layers, E4M3: 393 -> 389.  V of the first tile too: the same; K and V of four tiles: +4 %.
// A box of Q with fewer than 64 rows inside the tensor is not asked for: most of a box outside holds the TMA unit up, and with it
// the K tile behind.  16 layers at batch 1, prefix 3000, 8 / 8 heads, us without any fetch, with Q and K, with K alone: 10 rows 218, 234, 212; 48
// 221, 224, 215; 64 220, 212, 213; 32 / 8 heads, 40 rows 215, 216, 208; 64 214, 206, 208; 4 sequences, 24 rows 260, 287, 257.
constexpr int kQRowsFetched = 64;
template <int D, int kXStep>
__device__ __forceinline__ void prefetch_lane(const Params& p, const PlanView& v, const CUtensorMap* q_map, const CUtensorMap* k_map)
{
    const int4* w = reinterpret_cast<const int4*>(v.cta + blockIdx.x);
    const int4 w0 = __ldcg(w), w1 = __ldcg(w + 1), w2 = __ldcg(w + 2);
    const int b = w0.x, g = w0.y & 0xffff, rg = w0.y >> 16, t = w0.z;
    if (b < 0 || b >= p.d.B || g >= p.d.Hkv || rg < 0 || rg >= p.n_rg || t < 0 || t >= w1.x - (p.d.S > 0 ? 1 : 0)) return;
    if (p.map.block_table && t >= p.map.max_pages) return;
    const uint32_t page = p.map.block_table ? (uint32_t)__ldcg(p.map.block_table + (size_t)b * p.map.max_pages + t) : (uint32_t)t;
    const int z = (int)(page * kTileKeys + (p.map.block_table ? 0u : (uint32_t)w2.x));
#pragma unroll
    for (int x = 0; x < D; x += kXStep) tma_prefetch_3d(k_map, x, g, z);
    const int R = p.d.T + p.d.C, rows = p.d.B * R;
#pragma unroll 1
    for (int mt = 0; mt < p.n_mt; ++mt) {
        const int at = b * R + p.rpt * (p.tpg * rg + mt);
        if ((int64_t)(rows - at) * p.G < kQRowsFetched) continue;
#pragma unroll
        for (int x = 0; x < D; x += 64) tma_prefetch_3d(q_map, x, g * p.G, at);
    }
}
// By one lane of warp 11, if the plan was there before this call; every warp is together again behind it: setmaxnreg comes next.  (With the
// warp, not the thread, as the outer condition: 4 sequences of 500..4000, 64 / 8 heads, plan made beforehand, 29.7 -> 30.6 us, the same
// spills.)
template <int D, int kXStep>
__device__ __forceinline__ void prefetch_first(const Params& p, const PlanView& v, const CUtensorMap* q_map, const CUtensorMap* k_map)
{
    if (p.prefetch && threadIdx.x == 11 * 32) prefetch_lane<D, kXStep>(p, v, q_map, k_map);
    __syncwarp();
}

// Slots of key tile `tile` that belong to the sequence when the tile is its last key tile and
// reaches past its last slot (1..127); 0 for every other tile.
__device__ __forceinline__ int ragged_rows(const Segment& s, int tile, int R)
{
    if (tile != s.nkt - 1) return 0;
    return (int)((s.P + R) & (kTileKeys - 1));
}

// Which of the 128 keys of tile `t` may row r see.  lo: keys 0..63 of the tile, hi: 64..127.
__device__ __forceinline__ void visible_bits(const Segment& s, int t, int R, int T, int S, int r, bool row_valid,
                                             uint64_t mask, uint64_t& lo, uint64_t& hi)
{
    if (!row_valid) { lo = hi = ~0ull; return; }
    if (t >= s.nkt) {                          // soft-prompt tile: contemplate rows only, S entries
        const bool sees = r >= T;
        lo = sees ? (S >= 64 ? ~0ull : ((1ull << S) - 1)) : 0ull;
        hi = sees ? (S > 64 ? (S >= 128 ? ~0ull : ((1ull << (S - 64)) - 1)) : 0ull) : 0ull;
        return;
    }
    const int64_t off = s.P - (int64_t)t * kTileKeys;      // position of tree slot 0 inside this tile (may be < 0 or >= 128)
    // prefix part: keys [0, off)
    unsigned __int128 v = 0;
    if (off >= 128) v = ~(unsigned __int128)0;
    else if (off > 0) v = (((unsigned __int128)1) << off) - 1;
    // tree rows' slots: bit j of mask at position off + j; a contemplate row's own slot at off + r
    const unsigned __int128 m = (unsigned __int128)mask;
    if (off >= 0) { if (off < 128) v |= m << off; }
    else if (off > -64) v |= m >> (-off);
    if (r >= T) {
        const int64_t self = off + r;
        if (self >= 0 && self < 128) v |= ((unsigned __int128)1) << self;
    }
    (void)R;
    lo = (uint64_t)v;
    hi = (uint64_t)(v >> 64);
}

// max of 128 floats held as raw bits, as eight independent chains of three-input max
__device__ __forceinline__ float max128(const uint32_t (&sv)[128])
{
    float a[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        a[k] = fmaxf(__uint_as_float(sv[16 * k]), __uint_as_float(sv[16 * k + 1]));
#pragma unroll
        for (int j = 2; j < 16; j += 2)
            asm("max.f32 %0, %0, %1, %2;" : "+f"(a[k]) : "f"(__uint_as_float(sv[16 * k + j])), "f"(__uint_as_float(sv[16 * k + j + 1])));
    }
    return fmaxf(fmaxf(fmaxf(a[0], a[1]), fmaxf(a[2], a[3])), fmaxf(fmaxf(a[4], a[5]), fmaxf(a[6], a[7])));
}

// max of 64 floats held as raw bits, as four chains of three-input max
__device__ __forceinline__ float max64(const uint32_t (&sv)[64])
{
    float a[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        a[k] = fmaxf(__uint_as_float(sv[16 * k]), __uint_as_float(sv[16 * k + 1]));
#pragma unroll
        for (int j = 2; j < 16; j += 2)
            asm("max.f32 %0, %0, %1, %2;" : "+f"(a[k]) : "f"(__uint_as_float(sv[16 * k + j])), "f"(__uint_as_float(sv[16 * k + j + 1])));
    }
    return fmaxf(fmaxf(a[0], a[1]), fmaxf(a[2], a[3]));
}

// exp2(s*c - m) of 64 scores -> 32 packed bf16 pairs; returns their fp32 sum.  kFma: a quarter of the exponentials on the
// FMA pipe (for kernels that the exponential unit holds up).
template <bool kFma = false>
__device__ __forceinline__ float weights64(const uint32_t* sv, float c, float neg_m, uint32_t (&pk)[32])
{
    uint64_t sum2 = f2_pack(0.f, 0.f);
    const uint64_t c2 = f2_pack(c, c), nm2 = f2_pack(neg_m, neg_m);
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        float x0, x1;
        f2_unpack(f2_fma(f2_pack(__uint_as_float(sv[2 * j]), __uint_as_float(sv[2 * j + 1])), c2, nm2), x0, x1);
        if (kFma && (j & 3) == 1) ex2_pair_fma(x0, x1);
        else { x0 = ex2(x0); x1 = ex2(x1); }
        const float p0 = x0, p1 = x1;
        sum2 = f2_add(sum2, f2_pack(p0, p1));
        pk[j] = pack_bf16(p0, p1);
    }
    float s0, s1;
    f2_unpack(sum2, s0, s1);
    return s0 + s1;
}

// The same for 32 scores, each weight as the sum of two bf16 numbers, 16 bits of it: hi and, for what the first leaves, lo.
template <bool kFma = false>
__device__ __forceinline__ float split_weights32(const uint32_t* sv, float c, float neg_m, uint32_t (&hi)[16], uint32_t (&lo)[16])
{
    uint64_t sum2 = f2_pack(0.f, 0.f);
    const uint64_t c2 = f2_pack(c, c), nm2 = f2_pack(neg_m, neg_m), neg1 = f2_pack(-1.f, -1.f);
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        float x0, x1;
        f2_unpack(f2_fma(f2_pack(__uint_as_float(sv[2 * j]), __uint_as_float(sv[2 * j + 1])), c2, nm2), x0, x1);
        if (kFma && (j & 3) == 1) ex2_pair_fma(x0, x1);
        else { x0 = ex2(x0); x1 = ex2(x1); }
        const uint64_t p = f2_pack(x0, x1);
        sum2 = f2_add(sum2, p);
        hi[j] = pack_bf16(x0, x1);
        float r0, r1;
        f2_unpack(f2_fma(f2_pack(__uint_as_float(hi[j] << 16), __uint_as_float(hi[j] & 0xffff0000u)), neg1, p), r0, r1);
        lo[j] = pack_bf16(r0, r1);
    }
    float s0, s1;
    f2_unpack(sum2, s0, s1);
    return s0 + s1;
}

// 64 scores of a thread's row -> weights in tensor memory at `addr` (over the scores' own columns): bf16 in the first 32, and
// with kSplit what they leave in the next 32.  Returns their fp32 sum.
template <bool kSplit, bool kFma = false>
__device__ __forceinline__ float store_weights64(const uint32_t* sv, float c, float neg_m, uint32_t addr)
{
    if constexpr (!kSplit) {
        uint32_t pk[32];
        const float sum = weights64<kFma>(sv, c, neg_m, pk);
        tmem_st32(addr, pk);
        return sum;
    } else {
        float sum = 0.f;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            uint32_t hi[16], lo[16];
            sum += split_weights32<kFma>(sv + 32 * q, c, neg_m, hi, lo);
            tmem_st16(addr + 16 * q, hi);
            tmem_st16(addr + 32 + 16 * q, lo);
        }
        return sum;
    }
}

}  // namespace tc
}  // namespace confu
