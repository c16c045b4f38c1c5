// Predicted composite fields (Sec. 6 composition, Sec. 8 sequence of fields)
// on sm_103a: device code shared by the stand-alone kernel and the batched
// persistent kernel.
//
// The field of the humans at time t is the exact signed EDT of the voxels
// inside their capsules; its sites all lie in the z-slab [zlo, zlo + S) that
// the capsules touch.  Two kernels build the composite of every t:
//
//  k_dyn_xy      one CTA per (slab slice, 64 columns, t): the exact x-interval
//                of each capsule on every row of the slice, then the y pass
//                of the static EDT (capsule_xy_block in edt_full.cuh).
//                Output: the 2-D partial field of the slice (signed int32),
//                with no row-pass intermediate in memory.
//  k_composite_z one CTA per (64 columns, up to kMaxSteps time steps): the z
//                pass over the slab fused with the min against the static
//                field and the float epilogue.
//
// The CTA keeps the slab's partials of its columns and steps in shared memory
// as the tiles of blockmin.cuh (clamped to 16 bits, with the bounds of their
// blocks of 8 slices).  A warp then takes blocks of 8 slices of the grid: it
// loads the static block once and, for each t, starts from the static values
// and lowers them by the slab elements that can matter: those whose block's
// least partial plus squared gap lies below the block's largest value.  For
// most blocks there is none, and no voxel inside a human: the static block is
// stored as it is; no bounds of the static field are needed beforehand.  Where
// the humans are nearer the float field is the root of the new value, elsewhere
// the static float field itself.  Voxels inside a human take the distance to
// the free voxels (set F), from the same tile, whatever the static map holds
// there: it is the lower one where a human reaches deeper into a wall or floor
// than the wall's own depth.  A block left with a value past the 16-bit range
// is done in 32 bits from the partials: far_block().
//
// Bound by the stores: T fields of 8 bytes per voxel.
#pragma once

#include "blockmin.cuh"
#include "edt_full.cuh"

namespace pcdf {
namespace comp {

using namespace blockmin;

constexpr int kMaxSteps = 4;   // time steps per CTA: the static block is read once for all of them
constexpr int kThreadsZ = 256;     // of k_composite_z; any whole number of warps from 4 on
static_assert(kMaxSteps * (kMaxBlocks / 4) <= 64, "a warp's blocks and steps in one mask");

// The z blocks [first, first + count) that a slab's tile covers: its slices
// and one on either side (free voxels next to an occupied one).
struct SlabBlocks {
    int first, count;
};
__host__ __device__ inline SlabBlocks slab_blocks(int zlo, int S, int nz)
{
    if (S <= 0)
        return SlabBlocks{0, 0};
    const int lo = zlo > 0 ? zlo - 1 : 0, hi = zlo + S < nz ? zlo + S : nz - 1;
    return SlabBlocks{lo / kBlk, hi / kBlk - lo / kBlk + 1};
}
// Shared words of one step's tile.
__host__ __device__ inline size_t slab_words(int zlo, int S, int nz)
{
    const size_t nb = (size_t)slab_blocks(zlo, S, nz).count;
    return (nb * (2 + kPitch * kBlk + 32) + 3) / 4 * 4;
}
// Time steps that a CTA takes together within `limit` shared bytes.
__host__ inline int steps_per_cta(int zlo, int S, int nz, int T, size_t limit)
{
    const size_t w = slab_words(zlo, S, nz) * 4;
    int most = kMaxSteps;
    while (most > 1 && most * w > limit)
        --most;
    const int groups = (T + most - 1) / most;
    return (T + groups - 1) / groups;
}

// (d - j)^2 in both halves, 8 words for each offset d from kSqMin on: read
// through L1, so that a CTA need not build it.
struct alignas(16) SquareTable {
    uint32_t w[kSqWords];
};
constexpr SquareTable square_table()
{
    SquareTable t{};
    for (int d = kSqMin; d <= kSqMax; ++d)
        for (int j = 0; j < kBlk; ++j)
            t.w[kBlk * (d - kSqMin) + j] = both((d - j) * (d - j));
    return t;
}
static __device__ const SquareTable g_squares = square_table();

template <bool kSq, bool kSdfOut, bool kStaticSdf>
struct Composite {
    const int32_t *static_sq;
    const float *static_sdf;
    const int32_t *dyn_mid;  // [T][S][V2] slab partials
    const uint8_t *rep;      // [T][S]: slab element e is stored in slice rep[t][e] (NULL: e)
    int32_t *comp_sq;
    float *comp_sdf;
    int V2, nz, zlo, S;
    float vox;
    bool vec;  // two adjacent columns per lane, moved in 8 bytes (else two 32 apart)

    // Slab element of slice z (-1: outside the slab, no human there).
    __device__ __forceinline__ int element(int z) const { return z >= zlo && z < zlo + S ? z - zlo : -1; }
    __device__ __forceinline__ int stored(int t, int e) const { return rep ? rep[t * S + e] : e; }

    // Partials of slab element e at time t in the lane's columns (dead: none).
    template <bool kVec>
    __device__ __forceinline__ void partial(int t, int e, int o, const bool (&live)[2], int &v0, int &v1) const
    {
        v0 = v1 = kInf32;
        if (e < 0 || !live[0])
            return;
        const int slice = stored(t, e);
        const int32_t *p = dyn_mid + ((long long)t * S + slice) * V2 + o;
        if (!PCDF_IN(slice, S) || !PCDF_IN(o, V2))
            return;
        if (kVec) {
            const int2 v = __ldcg(reinterpret_cast<const int2 *>(p));
            v0 = v.x;
            v1 = v.y;
        } else {
            v0 = __ldcg(p);
            if (live[1] && PCDF_IN(o + 32, V2))
                v1 = __ldcg(p + 32);
        }
    }

    // The static block of 8 slices at offset i0: the first r0 rows of the
    // lane's first column and the first r1 of its second (others: 0).
    template <bool kVec>
    __device__ __forceinline__ void load(int i0, int r0, int r1, int2 (&s)[kBlk], float2 (&f)[kBlk]) const
    {
        const int32_t *p = static_sq + i0;
        const float *g = static_sdf + (kStaticSdf ? i0 : 0);
#pragma unroll
        for (int k = 0; k < kBlk; ++k, p += V2, g += kStaticSdf ? V2 : 0) {
            s[k] = make_int2(0, 0);
            f[k] = make_float2(0.f, 0.f);
            if (kVec) {
                if (k < r0 && PCDF_IN(i0 + k * V2 + 1, V2 * nz)) {
                    s[k] = __ldcg(reinterpret_cast<const int2 *>(p));
                    if (kStaticSdf)
                        f[k] = __ldcg(reinterpret_cast<const float2 *>(g));
                }
            } else {
                if (k < r0 && PCDF_IN(i0 + k * V2, V2 * nz)) {
                    s[k].x = __ldcg(p);
                    if (kStaticSdf)
                        f[k].x = __ldcg(g);
                }
                if (k < r1 && PCDF_IN(i0 + k * V2 + 32, V2 * nz)) {
                    s[k].y = __ldcg(p + 32);
                    if (kStaticSdf)
                        f[k].y = __ldcg(g + 32);
                }
            }
        }
        if (kSdfOut && !kStaticSdf) {
#pragma unroll
            for (int k = 0; k < kBlk; ++k)
                f[k] = make_float2(sq_to_sdf_fast(s[k].x, vox), sq_to_sdf_fast(s[k].y, vox));
        }
    }

    // A row of the static field at offset i (in0, in1: whether the lane's
    // columns take part; others: 0), and of its float field.
    template <bool kVec>
    __device__ __forceinline__ int2 row_sq(int i, bool in0, bool in1) const
    {
        int2 s = make_int2(0, 0);
        if (kVec) {
            if (in0 && PCDF_IN(i + 1, V2 * nz))
                s = __ldcg(reinterpret_cast<const int2 *>(static_sq + i));
        } else {
            if (in0 && PCDF_IN(i, V2 * nz))
                s.x = __ldcg(static_sq + i);
            if (in1 && PCDF_IN(i + 32, V2 * nz))
                s.y = __ldcg(static_sq + i + 32);
        }
        return s;
    }
    template <bool kVec>
    __device__ __forceinline__ float2 row_sdf(int i, bool in0, bool in1) const
    {
        float2 f = make_float2(0.f, 0.f);
        if (kVec) {
            if ((in0 || in1) && PCDF_IN(i + 1, V2 * nz))
                f = __ldcg(reinterpret_cast<const float2 *>(static_sdf + i));
        } else {
            if (in0 && PCDF_IN(i, V2 * nz))
                f.x = __ldcg(static_sdf + i);
            if (in1 && PCDF_IN(i + 32, V2 * nz))
                f.y = __ldcg(static_sdf + i + 32);
        }
        return f;
    }

    // A row of the output at offset i (in0, in1: whether the lane's columns take part).
    template <bool kVec>
    __device__ __forceinline__ void store(int32_t *q, float *g, int i, bool in0, bool in1, int2 s, float2 f) const
    {
        if (kVec) {
            if (in0 && PCDF_IN(i + 1, V2 * nz)) {
                if (kSq)
                    __stcs(reinterpret_cast<int2 *>(q), s);
                if (kSdfOut)
                    __stcs(reinterpret_cast<float2 *>(g), f);
            }
        } else {
            if (in0 && PCDF_IN(i, V2 * nz)) {
                if (kSq)
                    __stcs(q, s.x);
                if (kSdfOut)
                    __stcs(g, f.x);
            }
            if (in1 && PCDF_IN(i + 32, V2 * nz)) {
                if (kSq)
                    __stcs(q + 32, s.y);
                if (kSdfOut)
                    __stcs(g + 32, f.y);
            }
        }
    }

    __device__ __forceinline__ Tile tile(uint32_t *smem, int step, const SlabBlocks &sb) const
    {
        uint32_t *w = smem + step * slab_words(zlo, S, nz);
        uint32_t *v = w + (2 * sb.count + 3) / 4 * 4;
        return Tile(reinterpret_cast<uint2 *>(w), nullptr, v, v + sb.count * kPitch * kBlk, nz, sb.count);
    }

    // Bound of slab block q for block c (both counted from the tile's first).
    template <bool kF>
    __device__ __forceinline__ int bound(const Tile &t, int q, int c) const
    {
        const int m = abs(q - c);
        const Info i = t.about(q);
        return !kF && m == 0 ? (int)(i.w.y & 0xffffu) : i.template least16<kF>(q > c) + (m ? gap2(m) : 0);
    }

    // Can an element of the slab lie below um in block b?
    __device__ __forceinline__ bool reached(const Tile &t, int first, int b, int lane, int um) const
    {
        bool any = false;
        for (int q = lane; q < t.nb; q += 32)
            any |= bound<false>(t, q, b - first) < um;
        return __any_sync(0xffffffffu, any);
    }

    // Lowers best (the lane's packed values of block b) by the slab's O or F;
    // u, um: their largest in the lane and the warp, kept up to date.
    template <bool kF>
    __device__ __forceinline__ void lower(uint32_t (&best)[kBlk], uint32_t &u, int &um, uint32_t alive, const Tile &t,
                                          int first, int b, int lane) const
    {
        const int c = b - first;  // the block itself, maybe outside the tile
        const uint32_t *src = t.v + kBlk * c * kPitch + lane;
        for (int q0 = 0; q0 < t.nb; q0 += 32) {
            const int key = q0 + lane < t.nb ? bound<kF>(t, q0 + lane, c) : INT32_MAX;
            const uint32_t upto = 0xffffffffu >> (31 - min(max(c - q0, 0), 31));
            uint32_t rest = 0xffffffffu;
            for (;;) {
                const uint32_t a = __ballot_sync(0xffffffffu, key < um) & rest;
                if (!a)
                    break;
                const int below = 31 - __clz(a & upto), above = __ffs(a & ~upto) - 1;  // -1: none
                const int i = above < 0 || (below >= 0 && c - q0 - below <= above - (c - q0)) ? below : above;
                rest &= ~(1u << i);
                const int Q = q0 + i, s = Q - c;
                if (!kF && s != 0) {
                    const int gap = gap2(abs(s));
                    if (!__any_sync(0xffffffffu, __viaddmin_u16x2(t.lo[Q * 32 + lane], both(gap), u) != u))
                        continue;
                }
                uint32_t rows;
                if (kF && t.about(Q).flat()) {  // the nearest slice stands for all
                    rows = s ? (s > 0 ? 0x01u : 0x80u) : 0u;
                    if (s == 0) {
#pragma unroll
                        for (int k = 0; k < kBlk; ++k)
                            best[k] = __vminu2(best[k], part<true>(src[k * kPitch]));
                    }
                } else if (kF) {
                    rows = (1u << min(nz - kBlk * (first + Q), kBlk)) - 1u;
                } else if (s) {
                    rows = t.about(Q).use(s > 0);
                } else {  // each slice for itself, then those that count for others of the block
#pragma unroll
                    for (int k = 0; k < kBlk; ++k)
                        best[k] = __vminu2(best[k], part<false>(src[k * kPitch]));
                    rows = t.about(Q).own();
                }
                visit<kF>(best, g_squares.w, src, s, rows);
                u = largest(best) & alive;
                um = warp_largest(u);
            }
        }
    }

    // The value and its float at a voxel: static s (float f), the humans' d
    // (positive: least of the static value and the distance, or anything
    // larger; negative: inside a human).
    __device__ __forceinline__ void pick(int s, float f, int d, int &cs, float &cf) const
    {
        cs = min(s, d);
        cf = s <= d ? f : sq_to_sdf_fast(d, vox);
    }

    // Block b in the lane's columns: offset of its first row, rows of each column.
    template <bool kVec>
    struct Block {
        int at, r0, r1;
        __device__ __forceinline__ Block(const Composite &c, int b, int o, const bool (&live)[2])
            : at(o + kBlk * b * c.V2), r0(live[0] ? min(c.nz - kBlk * b, kBlk) : 0), r1(live[1] ? min(c.nz - kBlk * b, kBlk) : 0)
        {
        }
        __device__ __forceinline__ int32_t *sq_of(const Composite &c, int t) const
        {
            return kSq ? c.comp_sq + ((long long)t * c.V2 * c.nz + at) : nullptr;
        }
        __device__ __forceinline__ float *sdf_of(const Composite &c, int t) const
        {
            return kSdfOut ? c.comp_sdf + ((long long)t * c.V2 * c.nz + at) : nullptr;
        }
    };

    // best: the least of the static values s (negative ones as 0) and the
    // distance to the humans; returns the warp's largest.
    __device__ __forceinline__ int least_of(const Tile &tl, int first, int b, int lane, uint32_t alive, const int2 (&s)[kBlk],
                                            uint32_t (&best)[kBlk]) const
    {
#pragma unroll
        for (int k = 0; k < kBlk; ++k)
            best[k] = part<false>(clamp16(s[k].x, s[k].y));
        uint32_t u = largest(best) & alive;
        int um = warp_largest(u);
        lower<false>(best, u, um, alive, tl, first, b, lane);
        return um;
    }

    // The CTA (4 warps or more) computes columns col0 .. col0 + 63 of time
    // steps t0 .. t0 + nt - 1; smem: nt * slab_words().
    __device__ __forceinline__ void run(int t0, int nt, long long col0, uint32_t *smem) const
    {
        if (vec)
            run_as<true>(t0, nt, (int)col0, smem);
        else
            run_as<false>(t0, nt, (int)col0, smem);
    }

    // The tiles of the steps: values, bounds, links.
    template <bool kVec>
    __device__ __forceinline__ void fill(int t0, int nt, int o, const bool (&live)[2], const SlabBlocks &sb,
                                         uint32_t *smem) const
    {
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
        for (int Q = wid; Q < sb.count; Q += nw) {
            const int e0 = kBlk * (sb.first + Q) - zlo;  // slab element of the block's first slice
#pragma unroll 1
            for (int step = 0; step < nt; ++step) {
                const int t = t0 + step;
                const Tile tl = tile(smem, step, sb);
                uint32_t *dst = tl.v + Q * kBlk * kPitch + lane;
                const int32_t *src = dyn_mid + ((long long)t * S * V2 + o);
                // lane k: where slice k of the block is stored (-1: outside the slab)
                const int e = e0 + (lane & 7);
                int slot = -1;
                if (e >= 0 && e < S)
                    slot = rep && PCDF_IN(e, S) ? rep[t * S + e] : e;
                const int first = __shfl_sync(0xffffffffu, slot, 0);
                auto get = [&](int at, int &v0, int &v1) {
                    v0 = v1 = kInf32;
                    if (at < 0 || !live[0] || !PCDF_IN(at, S) || !PCDF_IN(o, V2))
                        return;
                    const int32_t *p = src + at * V2;  // a slab holds less than 2^31 values
                    if (kVec) {
                        const int2 v = __ldcg(reinterpret_cast<const int2 *>(p));
                        v0 = v.x;
                        v1 = v.y;
                    } else {
                        v0 = __ldcg(p);
                        if (live[1] && PCDF_IN(o + 32, V2))
                            v1 = __ldcg(p + 32);
                    }
                };
                // slices of equal cross-sections throughout (an upright human
                // between its ends): one load, and all is known
                if (__all_sync(0xffffffffu, slot == first) && first >= 0) {
                    int a0, a1;
                    get(first, a0, a1);
                    const uint32_t v = clamp16(a0, a1);
#pragma unroll
                    for (int k = 0; k < kBlk; ++k)
                        dst[k * kPitch] = v;
                    tl.record_flat(Q, lane, v);
                    continue;
                }
                int a0[kBlk], a1[kBlk];
#pragma unroll
                for (int k = 0; k < kBlk; ++k)
                    get(__shfl_sync(0xffffffffu, slot, k), a0[k], a1[k]);
                uint32_t v[kBlk], sign = 0;
#pragma unroll
                for (int k = 0; k < kBlk; ++k) {
                    v[k] = clamp16(a0[k], a1[k]);
                    sign |= v[k];
                    dst[k * kPitch] = v[k];
                }
                tl.record(Q, lane, v, __any_sync(0xffffffffu, (sign & 0x80008000u) != 0));
            }
        }
        __syncthreads();
        for (int Q = wid; Q + 1 < sb.count; Q += nw)
#pragma unroll 1
            for (int step = 0; step < nt; ++step)
                link(tile(smem, step, sb), Q, lane);
        __syncthreads();
    }

    template <bool kVec>
    __device__ __forceinline__ void run_as(int t0, int nt, int col0, uint32_t *smem) const
    {
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
        const SlabBlocks sb = slab_blocks(zlo, S, nz);
        const int o = col0 + (kVec ? 2 * lane : lane);
        const bool live[2] = {o < V2, o + (kVec ? 1 : 32) < V2};
        const uint32_t alive = (live[0] ? 0x0000ffffu : 0u) | (live[1] ? 0xffff0000u : 0u);
        fill<kVec>(t0, nt, o, live, sb, smem);

        // Three loops over the warp's blocks and steps, from the lean to the
        // rare: copies of the static block, blocks that a human can change,
        // blocks with voxels inside a human.  In one loop the compiler's code
        // for the rare paths slowed the others (366 M instead of 214 M
        // instructions at 256^3, T = 20).
        unsigned long long near = 0, inside = 0, far = 0, deep = 0;  // bit kMaxSteps * block + step
        for (int b = wid, i = 0; kBlk * b < nz; b += nw, i += kMaxSteps) {
            const Block<kVec> B(*this, b, o, live);
            int2 s[kBlk];
            float2 f[kBlk];
            load<kVec>(B.at, B.r0, B.r1, s, f);
            uint32_t u = 0;
#pragma unroll
            for (int k = 0; k < kBlk; ++k)
                u = __vmaxu2(u, part<false>(clamp16(s[k].x, s[k].y)));
            const int um = warp_largest(u & alive);
#pragma unroll 1
            for (int step = 0; step < nt; ++step) {
                const Tile tl = tile(smem, step, sb);
                const int c = b - sb.first;
                // voxels inside a human come first: the humans' field is
                // negative there, below any bound and any solid static block
                if (c >= 0 && c < sb.count && tl.about(c).occupied()) {
                    inside |= 1ull << (i + step);
                } else if (reached(tl, sb.first, b, lane, um)) {
                    near |= 1ull << (i + step);
                } else if (um >= kFar16 && sb.count) {
                    far |= 1ull << (i + step);
                } else {
                    int32_t *q = B.sq_of(*this, t0 + step);
                    float *g = B.sdf_of(*this, t0 + step);
#pragma unroll
                    for (int k = 0; k < kBlk; ++k, q += kSq ? V2 : 0, g += kSdfOut ? V2 : 0)
                        store<kVec>(q, g, B.at + k * V2, k < B.r0, k < B.r1, s[k], f[k]);
                }
            }
        }
        unsigned long long todo = near;
        for (int b = wid, i = 0; todo; b += nw, i += kMaxSteps, todo >>= kMaxSteps) {
            if (!(todo & ((1u << kMaxSteps) - 1u)))
                continue;
            const Block<kVec> B(*this, b, o, live);
            int2 s[kBlk];
            float2 f[kBlk];
            load<kVec>(B.at, B.r0, B.r1, s, f);
#pragma unroll 1
            for (int step = 0; step < nt; ++step) {
                if (!((todo >> step) & 1u))
                    continue;
                uint32_t best[kBlk];
                if (least_of(tile(smem, step, sb), sb.first, b, lane, alive, s, best) >= kFar16) {
                    far |= 1ull << (i + step);
                    continue;
                }
                int32_t *q = B.sq_of(*this, t0 + step);
                float *g = B.sdf_of(*this, t0 + step);
#pragma unroll
                for (int k = 0; k < kBlk; ++k, q += kSq ? V2 : 0, g += kSdfOut ? V2 : 0) {
                    // the static value where it is the least (or negative)
                    const int b0 = (int)(best[k] & 0xffffu), b1 = (int)(best[k] >> 16);
                    int2 cs = s[k];
                    float2 cf = f[k];
                    if (b0 < s[k].x) {
                        cs.x = b0;
                        cf.x = kSdfOut ? full::root_near(b0, vox) : 0.f;
                    }
                    if (b1 < s[k].y) {
                        cs.y = b1;
                        cf.y = kSdfOut ? full::root_near(b1, vox) : 0.f;
                    }
                    store<kVec>(q, g, B.at + k * V2, k < B.r0, k < B.r1, cs, cf);
                }
            }
        }
        todo = inside;
        for (int b = wid, i = 0; todo; b += nw, i += kMaxSteps, todo >>= kMaxSteps) {
            if (!(todo & ((1u << kMaxSteps) - 1u)))
                continue;
            const Block<kVec> B(*this, b, o, live);
            int2 s[kBlk];
            float2 f[kBlk];
            load<kVec>(B.at, B.r0, B.r1, s, f);
#pragma unroll 1
            for (int step = 0; step < nt; ++step) {
                if (!((todo >> step) & 1u))
                    continue;
                const Tile tl = tile(smem, step, sb);
                uint32_t best[kBlk], fr[kBlk], uf = both(kFar16);
                const int um = least_of(tl, sb.first, b, lane, alive, s, best);
                int umf = kFar16;
#pragma unroll
                for (int k = 0; k < kBlk; ++k)
                    fr[k] = kBlk * b + k < nz ? both(kFar16) : 0u;
                lower<true>(fr, uf, umf, alive, tl, sb.first, b, lane);
                if (um >= kFar16 || umf >= kFar16) {
                    deep |= 1ull << (i + step);
                    continue;
                }
                int32_t *q = B.sq_of(*this, t0 + step);
                float *g = B.sdf_of(*this, t0 + step);
#pragma unroll
                for (int k = 0; k < kBlk; ++k, q += kSq ? V2 : 0, g += kSdfOut ? V2 : 0) {
                    const int f0 = (int)(fr[k] & 0xffffu), f1 = (int)(fr[k] >> 16);
                    int2 cs;
                    float2 cf;
                    pick(s[k].x, f[k].x, f0 ? -f0 : (s[k].x < 0 ? kInf32 : (int)(best[k] & 0xffffu)), cs.x, cf.x);
                    pick(s[k].y, f[k].y, f1 ? -f1 : (s[k].y < 0 ? kInf32 : (int)(best[k] >> 16)), cs.y, cf.y);
                    store<kVec>(q, g, B.at + k * V2, k < B.r0, k < B.r1, cs, cf);
                }
            }
        }

        // voxels inside a human in a block that reaches out of the 16-bit
        // range: rare, and written for few registers (a search with arrays here
        // slowed the loops above: 356 M instead of 254 M instructions at 256^3,
        // T = 20)
        for (int b = wid; deep; b += nw, deep >>= kMaxSteps)
#pragma unroll 1
            for (int step = 0; step < nt; ++step)
                if ((deep >> step) & 1u)
#pragma unroll 1
                    for (int k = 0; k < kBlk && kBlk * b + k < nz; ++k)
                        whole_column<kVec>(t0 + step, kBlk * b + k, o, live);
        // blocks 177 voxels or more from the humans and the map: an empty map, or one with few obstacles
        for (int b = wid; far; b += nw, far >>= kMaxSteps)
#pragma unroll 1
            for (int step = 0; step < nt; ++step)
                if ((far >> step) & 1u)
                    far_block<kVec>(t0 + step, b, o, live);
    }

    // Block b of time t, none of whose voxels is inside a human, in 32 bits and
    // without the tile: the slab's runs of slices of equal cross-sections (an
    // upright human between its ends is one) one by one, those that can lower a
    // column.  An empty map of 256^3, T = 8 and one human (most of the field is
    // 177 voxels or more from the human): 0.58 ms, where the whole slab for
    // every voxel took 5.6; on a map of five boxes 0.23 ms.  Issue and latency
    // of about 1,200 instructions per block and step.
    template <bool kVec>
    __device__ __forceinline__ void far_block(int t, int b, int o, const bool (&live)[2]) const
    {
        const int lane = threadIdx.x & 31;
        const Block<kVec> B(*this, b, o, live);
        int p[kBlk], q[kBlk];  // the least of the static values (negative ones as 0) and the distance to the humans
#pragma unroll
        for (int k = 0; k < kBlk; ++k) {
            const int2 s = row_sq<kVec>(B.at + k * V2, k < B.r0, k < B.r1);
            p[k] = min(max(s.x, 0), kCap32);
            q[k] = min(max(s.y, 0), kCap32);
        }
        int u0 = largest32(p), u1 = largest32(q);
        bool lower = false;  // some run lies below in some column
        const int32_t *src = dyn_mid + ((long long)t * S * V2 + o);
        // 32 slices at a time, from the middle one's run (the humans' trunks: the least in most columns)
        const int words = (S + 31) / 32, mid = S / 2, z0 = kBlk * b;
        for (int n = 0; n < words; ++n) {
            const int w = mid / 32 + n, e0 = 32 * (w < words ? w : w - words), count = min(S - e0, 32);
            const int slot = lane < count ? stored(t, e0 + lane) : -1, before = __shfl_up_sync(0xffffffffu, slot, 1);
            const uint32_t starts = __ballot_sync(0xffffffffu, lane < count && (lane == 0 || slot != before));
            auto get = [&](int i, int &v0, int &v1) {
                v0 = v1 = kInf32;
                const int at = __shfl_sync(0xffffffffu, slot, i);
                if (!live[0] || !PCDF_IN(at, S) || !PCDF_IN(o, V2))
                    return;
                const int32_t *from = src + at * V2;  // a slab holds less than 2^31 values
                if (kVec) {
                    const int2 v = __ldcg(reinterpret_cast<const int2 *>(from));
                    v0 = v.x;
                    v1 = v.y;
                } else {
                    v0 = __ldcg(from);
                    if (live[1] && PCDF_IN(o + 32, V2))
                        v1 = __ldcg(from + 32);
                }
            };
            int i = n == 0 ? 31 - __clz(starts & ((2u << (mid & 31)) - 1u)) : 0, a0, a1;
            uint32_t todo = starts & ~(1u << i);
            get(i, a0, a1);
#pragma unroll 1
            for (;;) {  // warp-uniform; the next run's load in flight (two of them cost the batch kernel spills)
                const int next = __ffs(todo) - 1;
                int v0 = 0, v1 = 0;
                if (next >= 0)
                    get(next, v0, v1);
                todo &= todo - 1;
                const uint32_t above = starts & (0xfffffffeu << i);
                const int za = zlo + e0 + i, zb = zlo + e0 + (above ? __ffs(above) - 2 : count - 1);
                const int g0 = min(max(a0, 0), kCap32), g1 = min(max(a1, 0), kCap32);
                const int gap = max(max(za - (z0 + kBlk - 1), z0 - zb), 0);
                if (__any_sync(0xffffffffu, g0 + gap * gap < u0 || g1 + gap * gap < u1)) {
                    lower = true;
#pragma unroll
                    for (int k = 0; k < kBlk; ++k) {
                        const int d = max(max(za - (z0 + k), z0 + k - zb), 0);
                        p[k] = __viaddmin_s32(g0, d * d, p[k]);
                        q[k] = __viaddmin_s32(g1, d * d, q[k]);
                    }
                    u0 = largest32(p);
                    u1 = largest32(q);
                }
                if (next < 0)
                    break;
                i = next;
                a0 = v0;
                a1 = v1;
            }
        }
        int32_t *g = B.sq_of(*this, t);
        float *h = B.sdf_of(*this, t);
#pragma unroll
        for (int k = 0; k < kBlk; ++k, g += kSq ? V2 : 0, h += kSdfOut ? V2 : 0) {
            const int i = B.at + k * V2;
            const bool in0 = k < B.r0, in1 = k < B.r1;
            int2 s = row_sq<kVec>(i, in0, in1);
            float2 f = make_float2(0.f, 0.f);
            if (kStaticSdf)
                f = row_sdf<kVec>(i, in0, in1);
            else if (kSdfOut)
                f = make_float2(sq_to_sdf_fast(s.x, vox), sq_to_sdf_fast(s.y, vox));
            if (lower) {  // warp-uniform
                const bool n0 = p[k] < s.x && p[k] < kCap32, n1 = q[k] < s.y && q[k] < kCap32;
                s = make_int2(n0 ? p[k] : s.x, n1 ? q[k] : s.y);
                if (kSdfOut)
                    f = make_float2(n0 ? full::root_near(p[k], vox) : f.x, n1 ? full::root_near(q[k], vox) : f.y);
            }
            store<kVec>(g, h, i, in0, in1, s, f);
        }
    }

    // Slice z of time t in 32 bits: both sets over the whole slab.
    template <bool kVec>
    __device__ __forceinline__ void whole_column(int t, int z, int o, const bool (&live)[2]) const
    {
        int o0 = kCap32, o1 = kCap32, f0 = kCap32, f1 = kCap32;
        const int zend = min(zlo + S, nz - 1);  // a slice beyond the slab holds free voxels only
#pragma unroll 1
        for (int w = max(zlo - 1, 0); w <= zend; ++w) {
            int v0, v1;
            partial<kVec>(t, element(w), o, live, v0, v1);
            const int d = (z - w) * (z - w);
            o0 = min(o0, d + min(max(v0, 0), kCap32));
            o1 = min(o1, d + min(max(v1, 0), kCap32));
            f0 = min(f0, d + min(max(-v0, 0), kCap32));
            f1 = min(f1, d + min(max(-v1, 0), kCap32));
        }
        int v0, v1;
        partial<kVec>(t, element(z), o, live, v0, v1);
        const int d0 = v0 < 0 ? (f0 >= kCap32 ? -kInf32 : -f0) : (o0 >= kCap32 ? kInf32 : o0);
        const int d1 = v1 < 0 ? (f1 >= kCap32 ? -kInf32 : -f1) : (o1 >= kCap32 ? kInf32 : o1);
        const int i = o + z * V2;
        const long long w = t * (long long)V2 * nz + i;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = h * (kVec ? 1 : 32), d = h ? d1 : d0;
            if (!live[h] || !PCDF_IN(i + j, V2 * nz))
                continue;
            const int s = static_sq[i + j];
            const float f = kStaticSdf ? static_sdf[i + j] : (kSdfOut ? sq_to_sdf_fast(s, vox) : 0.f);
            int cs;
            float cf;
            pick(s, f, d, cs, cf);
            if (kSq)
                comp_sq[w + j] = cs;
            if (kSdfOut)
                comp_sdf[w + j] = cf;
        }
    }
};

}  // namespace comp
}  // namespace pcdf
