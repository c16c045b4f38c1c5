// The y and z passes of the exact EDT (Sec. 6: the environment's exact
// distance field; the full per-field recompute): per column, the least
// (e - s)^2 + G(s) over the sites s of the other state.
//
// Input: signed values v(e) of the axes already done: v >= 0 a free voxel whose
// partial squared distance to the nearest occupied voxel is v, v < 0 an
// occupied voxel whose partial squared distance to the nearest free voxel is
// -v; magnitude kInf32: none.  Output per element, the squared distance with
// this axis added, same convention.  With O(s) = max(v(s), 0) and
// F(s) = max(-v(s), 0) the output is
//     min_s (e - s)^2 + O(s)  -  min_s (e - s)^2 + F(s):
// the first term is zero at occupied voxels (O = 0 there) and the second at
// free ones.
//
// A CTA holds 64 columns of n elements in shared memory, two columns per lane
// as packed 16-bit values, clamped at kFar16 = 177^2.  One warp computes a
// block of 8 elements of the 64 columns from the elements that can matter, one
// candidate element at a time: 8 packed add-and-minimum instructions
// (__viaddmin_u16x2, two columns each) against squares that depend only on the
// difference of the positions.
//  * Candidate blocks are visited outwards from the block itself.  One is
//    skipped when its least O (or F) over the 64 columns plus the squared gap
//    between the blocks reaches the block's largest value so far (32
//    candidates either side in one ballot), or when that holds in every column
//    by itself.
//  * Of a candidate block only the elements are taken that the next one
//    towards the output block does not beat in every column (a slice that
//    repeats its neighbour's distances, as along the sides of a box, never
//    counts): a byte per block and side, found when the tile is filled, the
//    neighbouring block's nearest element included.  A block without such
//    elements is no candidate.  The same holds inside the block itself.
// On the 256^3 map of 60 boxes that leaves 3 to 7 elements per block of 8, on
// one with 0.2 % of speckle 9 to 16.  Sums stay below 2^16 within 22 blocks;
// beyond them the squared gap alone is kFar16, so a block whose results are
// all below kFar16 is exact.  A block with a larger result (a voxel 177 or more
// voxels from the nearest site, or with no site) is computed again in 32 bits.
//
// Bound by instruction issue, the 64 lane-instructions per clock and SM of
// the add-and-minimum among it.  It replaced a lower envelope of parabolas
// built by 8 threads per column (stack pops, seam merges and a second sweep,
// 120 to 190 thread instructions per voxel).
#pragma once

#include "edt_common.cuh"

namespace pcdf {
namespace blockmin {

constexpr int kTileCols = 64;  // columns per CTA, two per lane
constexpr int kBlk = 8;        // elements per block
constexpr int kPitch = 36;       // shared words per element: 32 lanes, and 4 so that the 16-byte stores of edt_xy_block
                               // (two words of a row to a thread pair) fall into different banks
constexpr int kFarDist = 177;
constexpr int kFar16 = kFarDist * kFarDist;   // clamp of the 16-bit values
constexpr int kReach = 22;                    // blocks either side that 16-bit sums can take
constexpr int kSqMin = -kBlk * kReach;        // squares for elements kSqMin .. kSqMax from a block's first
constexpr int kSqMax = kBlk * kReach + kBlk - 1;
constexpr int kSqWords = kBlk * (kSqMax - kSqMin + 1);
constexpr int kMaxBlocks = 512 / kBlk;        // PCDF_MAX_DIM
constexpr int kNoCandidate = 1 << 29;         // bound of a block that cannot matter
constexpr int kCap32 = 1 << 28;               // "no site" in the 32-bit search: sums stay below 2^31
static_assert(kBlk * (kReach + 1) - (kBlk - 1) >= kFarDist, "blocks beyond the reach cannot improve a value below kFar16");
static_assert(kFar16 + (kBlk * kReach + kBlk - 1) * (kBlk * kReach + kBlk - 1) < 65536 && kFar16 < 32768, "16-bit sums");

constexpr uint32_t both(int v) { return (uint32_t)v * 0x10001u; }

__host__ __device__ constexpr int blocks_of(int n) { return (n + kBlk - 1) / kBlk; }

// Shared words of a tile of n elements.
__host__ __device__ constexpr size_t tile_words(int n)
{
    return kSqWords + 4 * kMaxBlocks + (size_t)blocks_of(n) * (kPitch * kBlk + 32);
}

// two signed values as 16 bits each, clamped at +-kFar16 (low half: a)
__device__ __forceinline__ uint32_t clamp16(int a, int b)
{
    uint32_t p;
    asm("cvt.pack.sat.s16.s32 %0, %1, %2;" : "=r"(p) : "r"(b), "r"(a));
    return __vmaxs2(__vmins2(p, both(kFar16)), both(65536 - kFar16));
}

// O or F of packed signed values
template <bool kF>
__device__ __forceinline__ uint32_t part(uint32_t v)
{
    return kF ? __viaddmax_s16x2_relu(~v, both(1), 0u) : __vmaxs2(v, 0u);
}

// What is known of a block: .x the elements that count for blocks after it
// (byte 0), before it (byte 1), for others of the block (byte 2), each for O,
// and flags (byte 3); .y its least O (low half) and F.
struct Info {
    uint2 w;
    __device__ __forceinline__ uint32_t use(bool before) const { return (before ? w.x >> 8 : w.x) & 0xffu; }
    __device__ __forceinline__ uint32_t own() const { return (w.x >> 16) & 0xffu; }
    // the least O or F of a block that counts, after or before another one
    template <bool kF>
    __device__ __forceinline__ int least16(bool after) const
    {
        return kF ? (int)(w.y >> 16) : (use(after) ? (int)(w.y & 0xffffu) : kNoCandidate);
    }
    __device__ __forceinline__ bool occupied() const { return (w.x >> 24) & 1u; }
    __device__ __forceinline__ bool flat() const { return (w.x >> 27) & 1u; }  // recorded as flat
    // the least O or F is at the clamp: the whole block is far from its sites, or has none
    template <bool kF>
    __device__ __forceinline__ bool far() const
    {
        return (kF ? w.y >> 16 : w.y & 0xffffu) >= (uint32_t)kFar16;
    }
};

// The squares at the start of a tile (a barrier before they are used).
__device__ __forceinline__ void fill_squares(uint32_t *sq)
{
    for (int i = threadIdx.x; i < kSqWords / 4; i += blockDim.x) {
        const int d = i / 2 + kSqMin - 4 * (i & 1);
        reinterpret_cast<uint4 *>(sq)[i] =
            make_uint4(both(d * d), both((d - 1) * (d - 1)), both((d - 2) * (d - 2)), both((d - 3) * (d - 3)));
    }
}

struct Tile {
    uint32_t *sq;      // sq[8 (d - kSqMin) + j] = (d - j)^2 in both halves
    uint2 *info;       // [nb]
    int2 *far;         // [nb] least O and F in 32 bits (kCap32: none), where the one in info is at the clamp
    uint32_t *v;       // [8 nb][kPitch] packed values (lane l: word l), the largest value past the end
    uint32_t *lo;      // [nb][32] least O of each block in the lane's columns
    int n, nb;
    __device__ __forceinline__ Tile(uint32_t *smem, int n_) : n(n_), nb(blocks_of(n_))
    {
        sq = smem;
        info = reinterpret_cast<uint2 *>(sq + kSqWords);
        far = reinterpret_cast<int2 *>(info + kMaxBlocks);
        v = reinterpret_cast<uint32_t *>(far + kMaxBlocks);
        lo = v + nb * kPitch * kBlk;
    }
    // a tile without squares, its parts anywhere
    __device__ __forceinline__ Tile(uint2 *info_, int2 *far_, uint32_t *v_, uint32_t *lo_, int n_, int nb_)
        : sq(nullptr), info(info_), far(far_), v(v_), lo(lo_), n(n_), nb(nb_)
    {
    }
    __device__ __forceinline__ Info about(int b) const { return Info{info[b]}; }
    // One warp records block b, whose values are x; returns its least O and F
    // as clamped (warp-uniform; the caller notes `far` where one is at the clamp).
    __device__ __forceinline__ uint2 record(int b, int lane, const uint32_t (&x)[kBlk], bool occ) const
    {
        uint32_t prev = part<false>(x[0]), mn = prev;
        uint32_t bits = 0;  // bit k: o[k] >= o[k + 1]; bit 8 + k + 1: o[k + 1] >= o[k], in both columns
#pragma unroll
        for (int k = 0; k + 1 < kBlk; ++k) {
            const uint32_t next = part<false>(x[k + 1]);
            const uint32_t m = __vmaxu2(prev, next);
            if (m == prev)
                bits |= 1u << k;
            if (m == next)
                bits |= 0x200u << k;
            mn = __vminu2(mn, next);
            prev = next;
        }
        lo[b * 32 + lane] = mn;
        bits = ~__reduce_and_sync(0xffffffffu, bits);
        const uint32_t wo = __reduce_min_sync(0xffffffffu, min(mn & 0xffffu, mn >> 16));
        uint32_t wf = 0, flags = 0;  // with a free voxel (or an element past the end) F is 0 there
        if (occ) {
            uint32_t mx = x[0];
#pragma unroll
            for (int k = 1; k < kBlk; ++k)
                mx = __vmaxs2(mx, x[k]);
            const uint32_t f = part<true>(mx);
            wf = __reduce_min_sync(0xffffffffu, min(f & 0xffffu, f >> 16));
            flags = 1u << 24;
        }
        if (lane == 0 && PCDF_IN(b, kMaxBlocks))
            info[b] = make_uint2((bits & 0xffffu) | (((bits & 0x7fu) | ((bits >> 8) & 0xfeu)) << 16) | flags, wo | (wf << 16));
        return make_uint2(wo, wf);
    }

    // One warp notes block b, whose O or F is at the clamp in every column, in
    // 32 bits: the least O and F and, where it is O, by column the least O
    // rounded down to eighths in 16 bits (no 16-bit search asks for the lanes'
    // least O there).  l0, l1: the least O of the lane's columns, below 2^19 or
    // none; f: the least F.
    __device__ __forceinline__ void note_far(int b, int lane, int l0, int l1, int f) const
    {
        const int o = min(__reduce_min_sync(0xffffffffu, min(l0, l1)), kCap32);
        if (o >= kFar16)
            lo[b * 32 + lane] = (uint32_t)min(l0 >> 3, 0xffff) | ((uint32_t)min(l1 >> 3, 0xffff) << 16);
        if (lane == 0 && PCDF_IN(b, kMaxBlocks))
            far[b] = make_int2(o, f);
    }
    // Can O of block b, a squared gap away, lie below u0 or u1 in some lane's column?
    __device__ __forceinline__ bool matters32(int b, int lane, int gap, int u0, int u1) const
    {
        const uint32_t l = lo[b * 32 + lane];
        const int unit = about(b).far<false>() ? 3 : 0;
        return __any_sync(0xffffffffu, (int)((l & 0xffffu) << unit) + gap < u0 || (int)((l >> 16) << unit) + gap < u1);
    }

    // record() for a block of 8 elements that all are x, none of them past the end.
    __device__ __forceinline__ void record_flat(int b, int lane, uint32_t x) const
    {
        const uint32_t o = part<false>(x), f = part<true>(x);
        lo[b * 32 + lane] = o;
        const bool occ = __any_sync(0xffffffffu, (x & 0x80008000u) != 0);
        const uint32_t wo = __reduce_min_sync(0xffffffffu, min(o & 0xffffu, o >> 16));
        const uint32_t wf = occ ? __reduce_min_sync(0xffffffffu, min(f & 0xffffu, f >> 16)) : 0u;
        if (lane == 0 && PCDF_IN(b, kMaxBlocks))
            info[b] = make_uint2(0x08000180u | (occ ? 1u << 24 : 0u), wo | (wf << 16));  // before: element 0, after: element 7
    }
};

// One warp compares the last element of block b with the first of block b + 1
// (after the barrier that ends the records; another one before the tile is
// used): the one that the other beats in every column no longer counts beyond it.
__device__ __forceinline__ void link(const Tile &t, int b, int lane)
{
    if (b + 1 >= t.nb)
        return;
    const uint32_t *p = t.v + (kBlk * (b + 1) - 1) * kPitch + lane;
    const uint32_t here = part<false>(p[0]), there = part<false>(p[kPitch]), m = __vmaxu2(here, there);
    const bool ge = __all_sync(0xffffffffu, m == here), le = __all_sync(0xffffffffu, m == there);
    if (lane == 0) {  // bytes 0 and 1 of two blocks: no other warp writes them
        uint8_t *q = reinterpret_cast<uint8_t *>(t.info + b);
        if (ge)
            q[0] &= 0x7fu;
        if (le)
            q[sizeof(uint2) + 1] &= 0xfeu;
    }
}

// The elements of block b inside the column.
__device__ __forceinline__ uint32_t in_column(const Tile &t, int b) { return (1u << min(t.n - kBlk * b, kBlk)) - 1u; }

// Squared gap between blocks m >= 1 apart.
__device__ __forceinline__ int gap2(int m) { return (kBlk * m - kBlk + 1) * (kBlk * m - kBlk + 1); }

// Calls go(s) for the candidate blocks b + s, |s| from c0 + 1 to c0 + 32
// and at most kMost, in order of distance: lane i holds the bounds key(block) +
// gap2 of the two blocks c0 + 1 + i away, and only those below um, which go may
// lower, are called for.
template <bool kF, int kMost, class Key, class Go>
__device__ __forceinline__ void outwards(const Tile &t, int b, int c0, int lane, int &um, const Key &key, const Go &go)
{
    const int m = c0 + 1 + lane, g = gap2(m);
    int kl = INT32_MAX, kr = INT32_MAX;
    if (m <= kMost) {
        if (b - m >= 0)
            kl = key(b - m) + g;
        if (b + m < t.nb)
            kr = key(b + m) + g;
    }
    uint32_t rest = 0xffffffffu;
    for (;;) {
        const uint32_t L = __ballot_sync(0xffffffffu, kl < um), R = __ballot_sync(0xffffffffu, kr < um);
        const uint32_t a = (L | R) & rest;
        if (!a)
            break;
        const int i = __ffs(a) - 1, d = c0 + 1 + i;
        rest = 0xfffffffeu << i;
        if ((L >> i) & 1u)
            go(-d);
        if ((R >> i) & 1u)
            go(d);
    }
}

__device__ __forceinline__ uint32_t largest(const uint32_t (&best)[kBlk])
{
    return __vimax3_u16x2(__vimax3_u16x2(best[0], best[1], best[2]), __vimax3_u16x2(best[3], best[4], best[5]),
                          __vmaxu2(best[6], best[7]));
}
__device__ __forceinline__ int warp_largest(uint32_t u)
{
    return (int)__reduce_max_sync(0xffffffffu, max(u & 0xffffu, u >> 16));
}

// best[j] = min(best[j], part of element 8 s + k of the block, plus its
// squared distance to element j), over the k in `rows`; src: element 0.
template <bool kF>
__device__ __forceinline__ void visit(uint32_t (&best)[kBlk], const uint32_t *sq, const uint32_t *src, int s, uint32_t rows)
{
#pragma unroll 1
    for (; rows; rows &= rows - 1) {  // warp-uniform
        const int d = kBlk * s + __ffs(rows) - 1;
        const uint4 *q = reinterpret_cast<const uint4 *>(sq + kBlk * (d - kSqMin));
        const uint4 q0 = q[0], q1 = q[1];  // (d - j)^2
        const uint32_t g = part<kF>(src[d * kPitch]);
        best[0] = __viaddmin_u16x2(g, q0.x, best[0]);
        best[1] = __viaddmin_u16x2(g, q0.y, best[1]);
        best[2] = __viaddmin_u16x2(g, q0.z, best[2]);
        best[3] = __viaddmin_u16x2(g, q0.w, best[3]);
        best[4] = __viaddmin_u16x2(g, q1.x, best[4]);
        best[5] = __viaddmin_u16x2(g, q1.y, best[5]);
        best[6] = __viaddmin_u16x2(g, q1.z, best[6]);
        best[7] = __viaddmin_u16x2(g, q1.w, best[7]);
    }
}

// The packed minima of block b over O or F and, in u, their maxima; returns
// the largest of them in the warp.  Elements past the end count as 0, columns
// outside the grid (alive: the lane's columns inside) not at all.
template <bool kF>
__device__ __forceinline__ int search16(uint32_t (&best)[kBlk], uint32_t &u, const Tile &t, int b, int lane, uint32_t own,
                                        uint32_t alive)
{
    const uint32_t *src = t.v + kBlk * b * kPitch + lane;
#pragma unroll
    for (int k = 0; k < kBlk; ++k)
        best[k] = part<kF>(src[k * kPitch]);
    if (kF) {  // next to a free voxel everywhere (single occupied voxels, thin walls): nothing can be nearer
        const int most = warp_largest(largest(best) & alive);
        if (most <= 1 && kBlk * (b + 1) <= t.n) {
            u = 0;
            return most;
        }
    }
    if (!kF && __popc(own) < 5) {
        visit<kF>(best, t.sq, src, 0, own);
    } else {  // most elements count: constant squares
        uint32_t g[kBlk];
#pragma unroll
        for (int k = 0; k < kBlk; ++k)
            g[k] = kF && kBlk * b + k >= t.n ? both(kFar16) : best[k];  // past the end: no site
        if (!kF || !t.about(b).template far<true>()) {  // else its own elements cannot matter
#pragma unroll
            for (int k = 0; k < kBlk; ++k)
#pragma unroll
                for (int j = 0; j < kBlk; ++j)
                    if (j != k)
                        best[j] = __viaddmin_u16x2(g[k], both((k - j) * (k - j)), best[j]);
        }
    }
    if (kBlk * (b + 1) > t.n) {
#pragma unroll
        for (int j = 0; j < kBlk; ++j)
            best[j] = kBlk * b + j < t.n ? best[j] : 0u;
    }
    u = largest(best) & alive;
    int um = warp_largest(u);
    outwards<kF, kReach>(
        t, b, 0, lane, um, [&](int q) { return t.about(q).least16<kF>(q > b); },
        [&](int s) {
            const int q = b + s;
            if (!kF) {
                const int gap = gap2(abs(s));
                if (!__any_sync(0xffffffffu, __viaddmin_u16x2(t.lo[q * 32 + lane], both(gap), u) != u))
                    return;
            }
            if (!PCDF_IN(q, t.nb))
                return;
            visit<kF>(best, t.sq, src, s, kF ? in_column(t, q) : t.about(q).use(s > 0));
            u = largest(best) & alive;
            um = warp_largest(u);
        });
    return um;
}

// One warp computes block b: out.near(row, best) takes the lane's packed values
// of a block of free voxels whose results are below kFar16, out.any(row, r0, r1) any value.  False (warp-uniform, nothing written): some
// result is out of the 16-bit range.
template <class Out>
__device__ __forceinline__ bool block16(const Tile &t, int b, int lane, uint32_t alive, Out &out)
{
    uint32_t best[kBlk], u;
    const Info info = t.about(b);
    if (search16<false>(best, u, t, b, lane, info.own(), alive) >= kFar16)
        return false;
    const int r0 = kBlk * b;
    if (info.occupied()) {
        uint32_t f[kBlk], uf;
        if (search16<true>(f, uf, t, b, lane, 0, alive) >= kFar16)
            return false;
#pragma unroll
        for (int j = 0; j < kBlk; ++j)
            best[j] = __vsub2(best[j], f[j]);
    }
    if (info.occupied() || r0 + kBlk > t.n) {
#pragma unroll
        for (int j = 0; j < kBlk; ++j)
            if (r0 + j < t.n)
                out.any(r0 + j, (int)(int16_t)(best[j] & 0xffffu), (int)best[j] >> 16);
    } else {
        out.near(r0, best);
    }
    return true;
}

// --- 32 bits -------------------------------------------------------------

// p[j], q[j] = min(.., g + (d - j)^2) for the lane's two columns
__device__ __forceinline__ void lower32(int (&p)[kBlk], int (&q)[kBlk], int g0, int g1, int d)
{
#pragma unroll
    for (int j = 0; j < kBlk; ++j) {
        p[j] = __viaddmin_s32(g0, (d - j) * (d - j), p[j]);
        q[j] = __viaddmin_s32(g1, (d - j) * (d - j), q[j]);
    }
}
__device__ __forceinline__ int largest32(const int (&p)[kBlk])
{
    return __vimax3_s32(__vimax3_s32(p[0], p[1], p[2]), __vimax3_s32(p[3], p[4], p[5]), max(p[6], p[7]));
}
__device__ __forceinline__ int warp_largest32(const int (&p)[kBlk], const int (&q)[kBlk])
{
    return (int)__reduce_max_sync(0xffffffffu, max(largest32(p), largest32(q)));
}

// A tile that holds signed distances (none: 1 << 14, whose square is kCap32)
// and was recorded as such: the same search on their squares.
struct DistTile {
    const Tile &t;
    uint32_t alive;  // the lane's columns inside the grid
    template <bool kF>
    __device__ __forceinline__ void search(int (&p)[kBlk], int (&q)[kBlk], int b, int lane) const
    {
        const uint32_t *src = t.v + kBlk * b * kPitch + lane;
        auto visit = [&](int s, uint32_t rows) {
#pragma unroll 1
            for (; rows; rows &= rows - 1) {
                const int d = kBlk * s + __ffs(rows) - 1;
                const uint32_t e = part<kF>(src[d * kPitch]);
                const int d0 = (int)(e & 0xffffu), d1 = (int)(e >> 16);
                lower32(p, q, d0 * d0, d1 * d1, d);
            }
        };
#pragma unroll
        for (int j = 0; j < kBlk; ++j) {
            p[j] = kBlk * b + j < t.n && (alive & 0xffffu) ? kCap32 : 0;
            q[j] = kBlk * b + j < t.n && (alive >> 16) ? kCap32 : 0;
        }
        const uint32_t in = in_column(t, b);
        uint32_t rows = kF ? in : t.about(b).own() & in;
        if (!kF) {  // each element is a candidate for itself
#pragma unroll
            for (int j = 0; j < kBlk; ++j) {
                const uint32_t e = part<kF>(src[j * kPitch]);
                const int d0 = (int)(e & 0xffffu), d1 = (int)(e >> 16);
                p[j] = min(p[j], d0 * d0);
                q[j] = min(q[j], d1 * d1);
            }
        }
        visit(0, rows);
        int um = warp_largest32(p, q);
        for (int c0 = 0; c0 < t.nb; c0 += 32)
            outwards<kF, kMaxBlocks>(
                t, b, c0, lane, um,
                [&](int q) {
                    const int d = t.about(q).least16<kF>(q > b);
                    return d == kNoCandidate ? d : d * d;
                },
                [&](int s) {
                    visit(s, kF ? in_column(t, b + s) : t.about(b + s).use(s > 0) & in_column(t, b + s));
                    um = warp_largest32(p, q);
                });
    }
};

// A source of unclamped values src(row, v0, v1) next to the clamped tile.
// Blocks whose least value is at the clamp have it in 32 bits in t.far and the
// elements that count recorded from the unclamped values; of the others every
// element is a candidate.  On maps with few obstacles nearly every block is
// searched here: k_edt_z 87 us on 256^3 with one box and 670 us on 512^3 with
// three, 111 and 1180 us with the clamp itself for a bound.
template <class Src>
struct RawTile {
    const Tile &t;
    const Src &src;
    uint32_t alive;  // the lane's columns inside the grid
    template <bool kF>
    __device__ __forceinline__ void search(int (&p)[kBlk], int (&q)[kBlk], int b, int lane) const
    {
#pragma unroll
        for (int j = 0; j < kBlk; ++j) {
            p[j] = kBlk * b + j < t.n && (alive & 0xffffu) ? kCap32 : 0;
            q[j] = kBlk * b + j < t.n && (alive >> 16) ? kCap32 : 0;
        }
        auto least = [&](int q) {
            const Info i = t.about(q);
            return i.far<kF>() ? (kF ? t.far[q].y : t.far[q].x) : (int)(kF ? i.w.y >> 16 : i.w.y & 0xffffu);
        };
        int u0 = kCap32, u1 = kCap32, um = kCap32;
        auto go = [&](int s) {
            const Info i = t.about(b + s);
            uint32_t rows = in_column(t, b + s);
            if (s != 0) {
                if (i.far<kF>())  // the nearest element always counts: link() compares clamped values
                    rows &= i.use(s > 0) | (s > 0 ? 0x01u : 0x80u);
                if (!kF && !t.matters32(b + s, lane, gap2(abs(s)), u0, u1))  // in every column by itself
                    return;
            }
#pragma unroll 1
            for (; rows; rows &= rows - 1) {  // warp-uniform
                const int d = kBlk * s + __ffs(rows) - 1;
                const uint32_t e = part<kF>(t.v[(kBlk * b + d) * kPitch + lane]);
                int v0 = (int)(e & 0xffffu), v1 = (int)(e >> 16);
                if (__any_sync(0xffffffffu, max(v0, v1) >= kFar16)) {  // clamped in some column
                    src(kBlk * b + d, v0, v1);
                    v0 = min(max(kF ? -v0 : v0, 0), kCap32);
                    v1 = min(max(kF ? -v1 : v1, 0), kCap32);
                }
                const int near = d < 0 ? d : max(d - (kBlk - 1), 0);  // to the block's nearest element
                if (__any_sync(0xffffffffu, v0 + near * near < u0 || v1 + near * near < u1))
                    lower32(p, q, v0, v1, d);
            }
            u0 = largest32(p);
            u1 = largest32(q);
            um = (int)__reduce_max_sync(0xffffffffu, max(u0, u1));
        };
        if (least(b) < kCap32)
            go(0);
        for (int c0 = 0; c0 < t.nb; c0 += 32)
            outwards<kF, kMaxBlocks>(t, b, c0, lane, um, least, go);
    }
};

// Block b in 32 bits: rare, in a loop of its own after the 16-bit blocks (a
// call inside their loop, or out of line, made the compiler spill around it:
// the z pass of a 256^3 map took 58 us instead of 50).
template <bool kRaw, class S>
__device__ __forceinline__ void block32(const S &from, const Tile &t, int b, int lane, int2 *res)
{
    int p[kBlk], q[kBlk];
    if (kRaw && t.about(b).template far<true>()) {  // solid throughout
#pragma unroll
        for (int j = 0; j < kBlk; ++j)
            p[j] = q[j] = 0;
    } else {
        from.template search<false>(p, q, b, lane);
    }
#pragma unroll
    for (int j = 0; j < kBlk; ++j)
        res[j] = make_int2(p[j] >= kCap32 ? kInf32 : p[j], q[j] >= kCap32 ? kInf32 : q[j]);
    if (t.about(b).occupied()) {
        from.template search<true>(p, q, b, lane);
#pragma unroll
        for (int j = 0; j < kBlk; ++j) {
            if (p[j])
                res[j].x = p[j] >= kCap32 ? -kInf32 : -p[j];
            if (q[j])
                res[j].y = q[j] >= kCap32 ? -kInf32 : -q[j];
        }
    }
}

}  // namespace blockmin
}  // namespace pcdf
