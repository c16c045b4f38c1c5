// Static-map utilities of the mapping pipeline (Sec. 8) on sm_103a.
//
//  k_voxel_filter  clears every occupied voxel with fewer than a given number
//                  of occupied voxels among its 26 in-grid neighbours (the
//                  paper clears voxels with fewer than five connected voxels).
//                  A CTA owns a 32 x 8 tile of columns and 32 slices, staged
//                  with their one-voxel halo in shared memory at once; each
//                  thread then sweeps its column with the 3 x 3 sums of the
//                  previous, current and next slice in registers.
//  k_voxel_filter_bits the same filter on 32 voxels per word when rows are
//                  whole 16-byte pieces: the bytes become bits as they are
//                  staged, and the 3 x 3 x 3 counts are taken in bit planes
//                  (one three-input sum and one majority per carry-save step),
//                  so that a word's 32 counts cost about 60 logical
//                  instructions.
//  k_voxel_filter4 the same filter on four voxels per thread when rows are
//                  whole 32-bit words (nx % 4 == 0, 4-byte aligned maps): a
//                  word holds the four voxels' bytes, the 3 x 3 x 3 count is
//                  taken byte-wise in the word (x by shifts with the
//                  neighbouring words' end bytes, from the lanes beside it,
//                  then y and z by word additions: a count is at most 27, so
//                  no byte carries into the next), and the four results are
//                  stored as one word.  A CTA stages a tile of words with
//                  its halo in shared memory (all loads in flight at once)
//                  and forms the x, then y, then z sums there, each once.
//  k_collapse      the 2-D map for the prediction module: a column is
//                  occupied if any of its voxels in a slice range is.  Its EDT
//                  is the static EDT of a grid one slice thick.
#include <cuda_runtime.h>

#include "host.h"

using namespace pcdf::host;

namespace pcdf {
namespace {

constexpr int kFX = 32, kFY = 8, kFZ = 32;  // tile of a CTA: columns x, y; slices per CTA
constexpr int kHX = kFX + 2, kHY = kFY + 2;

// The CTA stages its slices and their one-voxel halo (kFZ + 2 slices of
// kHY x kHX bytes) with every load in flight at once, then each thread sweeps
// its column keeping the 3 x 3 sums of three consecutive slices.
__global__ void __launch_bounds__(kFX *kFY)
    k_voxel_filter(const uint8_t *__restrict__ occ, int nx, int ny, int nz, int min_n, uint8_t *__restrict__ out)
{
    __shared__ uint8_t tile[kFZ + 2][kHY][kHX];
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * kFX + tx;
    const int x = blockIdx.x * kFX + tx, y = blockIdx.y * kFY + ty;
    const int z0 = blockIdx.z * kFZ, z1 = min(z0 + kFZ, nz);
    const long long V2 = (long long)nx * ny;
    const int x0 = blockIdx.x * kFX - 1, y0 = blockIdx.y * kFY - 1;
    const int n = (z1 - z0 + 2) * kHY * kHX;
    for (int v = tid; v < n; v += kFX * kFY) {
        const int zz = v / (kHY * kHX), rem = v - zz * (kHY * kHX);
        const int hy = rem / kHX, hx = rem - hy * kHX;
        const int gx = x0 + hx, gy = y0 + hy, gz = z0 - 1 + zz;
        uint8_t o = 0;
        if (gz >= 0 && gz < nz && gx >= 0 && gx < nx && gy >= 0 && gy < ny)
            o = __ldg(occ + gz * V2 + (long long)gy * nx + gx) != 0;
        tile[zz][hy][hx] = o;
    }
    __syncthreads();
    auto sum3 = [&](int zz) {
        int s = 0;
#pragma unroll
        for (int dy = 0; dy < 3; ++dy)
#pragma unroll
            for (int dx = 0; dx < 3; ++dx)
                s += tile[zz][ty + dy][tx + dx];
        return s;
    };
    if (x >= nx || y >= ny)
        return;  // no block-level synchronisation below
    int s_prev = sum3(0), s_cur = sum3(1);
    for (int z = z0; z < z1; ++z) {
        const int zz = z - z0 + 1;
        const int s_next = sum3(zz + 1);
        const int o = tile[zz][ty + 1][tx + 1];
        out[z * V2 + (long long)y * nx + x] = (uint8_t)(o && s_prev + s_cur + s_next - 1 >= min_n);
        s_prev = s_cur;
        s_cur = s_next;
    }
}

// 0x01 in every byte of w that is non-zero, 0x00 elsewhere
__device__ __forceinline__ uint32_t bytes_nonzero(uint32_t w)
{
    uint32_t t = w | (w >> 4);
    t |= t >> 2;
    t |= t >> 1;
    return t & 0x01010101u;
}

// k_voxel_filter4 tile: 32 words (lanes; words 1..30 are outputs, 0 and 31
// the x halo) x 8 rows x 8 slices of outputs, staged with a one-row and
// one-slice halo
constexpr int kF4Out = 30, kF4Y = 8, kF4Z = 8;
constexpr int kF4HY = kF4Y + 2, kF4HZ = kF4Z + 2;

// Lane l holds word wi = blockIdx.x * kF4Out + l - 1 of every staged row (0
// outside the grid), so the lanes 1..30 find both x neighbours of their four
// voxels in the lanes beside them.  Warp w (of 8) works on staged rows
// w, w + 8, ... in each pass:
//  0. stage the kF4HZ x kF4HY rows of words (slices z0 - 1 .., rows y0 - 1 ..),
//     every load in flight at once;
//  1. per staged row: bytes normalised to 0/1 and summed over x, the
//     normalised words of the output rows kept aside;
//  2. per slice and output row: the x sums of the row and its two y
//     neighbours added;
//  3. per output slice and row: the x+y sums of the slice and its two z
//     neighbours added, compared with min_neighbours + 1 (the count includes
//     the voxel) and masked by the voxel's own occupancy.
__global__ void __launch_bounds__(32 * kF4Y)
    k_voxel_filter4(const uint32_t *__restrict__ occ4, int nw, int ny, int nz, uint32_t thresh4,
                    uint32_t *__restrict__ out4)
{
    __shared__ uint32_t sx[kF4HZ][kF4HY][32];   // x sums of the staged rows
    __shared__ uint32_t sxy[kF4HZ][kF4Y][32];   // x+y sums of the output rows
    __shared__ uint32_t cen[kF4Z][kF4Y][32];    // normalised words of the outputs
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int wi = blockIdx.x * kF4Out + lane - 1;
    const int y0 = blockIdx.y * kF4Y, z0 = blockIdx.z * kF4Z;
    const bool xin = wi >= 0 && wi < nw;
    const long long nwords = (long long)nz * ny * nw;
    constexpr int kRows = kF4HZ * kF4HY;
    constexpr int kPer = (kRows + kF4Y - 1) / kF4Y;
    uint32_t v[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int r = warp + k * kF4Y;
        const int zz = r / kF4HY, yy = r - zz * kF4HY;
        const int z = z0 - 1 + zz, y = y0 - 1 + yy;
        const bool in = r < kRows && xin && z >= 0 && z < nz && y >= 0 && y < ny;
        const long long o = ((long long)(in ? z : 0) * ny + (in ? y : 0)) * nw + (in ? wi : 0);
        v[k] = in && PCDF_IN(o, nwords) ? __ldg(occ4 + o) : 0u;
    }
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int r = warp + k * kF4Y;
        if (r >= kRows)
            break;  // warp-uniform
        const int zz = r / kF4HY, yy = r - zz * kF4HY;
        const uint32_t n = bytes_nonzero(v[k]);
        const uint32_t l = __shfl_up_sync(0xffffffffu, n, 1), rr = __shfl_down_sync(0xffffffffu, n, 1);
        sx[zz][yy][lane] = n + ((n << 8) | (l >> 24)) + ((n >> 8) | (rr << 24));
        if (zz >= 1 && zz <= kF4Z && yy >= 1 && yy <= kF4Y)
            cen[zz - 1][yy - 1][lane] = n;
    }
    __syncthreads();
    for (int r = warp; r < kF4HZ * kF4Y; r += kF4Y) {
        const int zz = r / kF4Y, yy = r - zz * kF4Y;
        sxy[zz][yy][lane] = sx[zz][yy][lane] + sx[zz][yy + 1][lane] + sx[zz][yy + 2][lane];
    }
    __syncthreads();
    if (!xin || lane == 0 || lane == 31)
        return;  // no block-level synchronisation below
    for (int r = warp; r < kF4Z * kF4Y; r += kF4Y) {
        const int zz = r / kF4Y, yy = r - zz * kF4Y;
        const int z = z0 + zz, y = y0 + yy;
        if (z >= nz || y >= ny)
            continue;
        const uint32_t total = sxy[zz][yy][lane] + sxy[zz + 1][yy][lane] + sxy[zz + 2][yy][lane];
        const uint32_t keep = __vcmpgeu4(total, thresh4) & (cen[zz][yy][lane] * 0xFFu);
        const long long o = ((long long)z * ny + y) * nw + wi;
        if (PCDF_IN(o, nwords))
            out4[o] = keep & 0x01010101u;
    }
}

// the same as four bits
__device__ __forceinline__ uint32_t byte_bits(uint32_t w) { return (bytes_nonzero(w) * 0x01020408u) >> 24; }
// four bits as four bytes
__device__ __forceinline__ uint32_t bit_bytes(uint32_t n) { return (n * 0x00204081u) & 0x01010101u; }
__device__ __forceinline__ uint32_t majority(uint32_t a, uint32_t b, uint32_t c) { return (a & b) | (a & c) | (b & c); }

// Tile of a CTA: kBW words of a row, 64 / kBW rows, kBZ slices of outputs,
// staged as bits with one row, slice and voxel around them.
constexpr int kBZ = 8, kBHZ = kBZ + 2, kBThreads = 256;

// nx a multiple of 16, both maps aligned to 16 bytes.
// thresh: least count, the voxel itself among it, that keeps an occupied voxel.
// Bound by the loads of its tiles (1.6 times the map, the halo from L2): 12 us
// at 256^3 (31.5 us with byte-wise counts in shared memory; 2 bytes per voxel
// take 5).
template <int kBW>
__global__ void __launch_bounds__(kBThreads)
    k_voxel_filter_bits(const uint8_t *__restrict__ occ, int nx, int ny, int nz, int thresh, uint8_t *__restrict__ out)
{
    constexpr int kBY = 64 / kBW, kBHY = kBY + 2, kBPitch = kBW + 2;
    __shared__ uint32_t bits[kBHZ * kBHY * kBPitch];  // word 0 of a row: the voxel before the tile in bit 31; word kBW + 1: the one after it
    const int tid = threadIdx.x;
    const int x0 = 32 * kBW * blockIdx.x, y0 = kBY * blockIdx.y, z0 = kBZ * blockIdx.z;
    const long long V = (long long)nx * ny * nz;
    // the staged row r (z0 - 1 + r / kBHY, y0 - 1 + r % kBHY): its first voxel's index, or -1 outside the grid
    auto row_at = [&](int r) -> long long {
        const int z = z0 - 1 + r / kBHY, y = y0 - 1 + r % kBHY;
        return z >= 0 && z < nz && y >= 0 && y < ny ? ((long long)z * ny + y) * nx : -1;
    };
    constexpr int kRows = kBHZ * kBHY;
    constexpr int kItems = kRows * 2 * kBW, kPer = (kItems + kBThreads - 1) / kBThreads;
    uint4 v[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int i = tid + k * kBThreads, x = x0 + 16 * (i % (2 * kBW));
        const long long at = i < kItems ? row_at(i / (2 * kBW)) : -1;
        v[k] = make_uint4(0, 0, 0, 0);
        if (at >= 0 && x < nx && PCDF_IN(at + x + 15, V))
            v[k] = __ldg(reinterpret_cast<const uint4 *>(occ + at + x));
    }
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int i = tid + k * kBThreads, r = i / (2 * kBW), half = i % (2 * kBW);
        if (i < kItems)
            reinterpret_cast<uint16_t *>(bits)[2 * (r * kBPitch + 1) + half] =
                (uint16_t)(byte_bits(v[k].x) | (byte_bits(v[k].y) << 4) | (byte_bits(v[k].z) << 8) | (byte_bits(v[k].w) << 12));
    }
    for (int i = tid; i < 2 * kRows; i += kBThreads) {
        const int r = i >> 1, after = i & 1, x = after ? x0 + 32 * kBW : x0 - 1;
        const long long at = row_at(r);
        const bool o = at >= 0 && x >= 0 && x < nx && PCDF_IN(at + x, V) && __ldg(occ + at + x) != 0;
        bits[r * kBPitch + (after ? kBW + 1 : 0)] = o ? (after ? 1u : 0x80000000u) : 0u;
    }
    __syncthreads();

    // thread: word w of row y of two output slices; per staged slice the 3 x 3 count in four planes
    const int w = tid % kBW, yy = tid / kBW % kBY, zz = 2 * (tid / (kBW * kBY));
    static_assert(kBThreads == kBW * kBY * kBZ / 2, "two slices per thread");
    const int x = x0 + 32 * w, y = y0 + yy;
    uint32_t c[4][4], mid[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        uint32_t a[3], b[3];  // sum and carry planes of the three rows
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const uint32_t *p = bits + ((zz + s) * kBHY + yy + d) * kBPitch + w;
            const uint32_t l = __funnelshift_l(p[0], p[1], 1), m = p[1], r = __funnelshift_r(p[1], p[2], 1);
            a[d] = l ^ m ^ r;
            b[d] = majority(l, m, r);
            if (d == 1)
                mid[s] = m;
        }
        const uint32_t k = majority(a[0], a[1], a[2]), t = b[0] ^ b[1] ^ b[2], m = majority(b[0], b[1], b[2]);
        c[s][0] = a[0] ^ a[1] ^ a[2];
        c[s][1] = t ^ k;
        c[s][2] = m ^ (t & k);
        c[s][3] = m & (t & k);
    }
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const int z = z0 + zz + s;
        if (z >= nz || y >= ny || x >= nx)
            continue;
        const uint32_t *A = c[s], *B = c[s + 1], *C = c[s + 2];
        uint32_t v[5];
        v[0] = A[0] ^ B[0] ^ C[0];
        const uint32_t k1 = majority(A[0], B[0], C[0]), t1 = A[1] ^ B[1] ^ C[1], m1 = majority(A[1], B[1], C[1]);
        v[1] = t1 ^ k1;
        const uint32_t n1 = t1 & k1, t2 = A[2] ^ B[2] ^ C[2], m2 = majority(A[2], B[2], C[2]);
        v[2] = t2 ^ m1 ^ n1;
        const uint32_t n2 = majority(t2, m1, n1), t3 = A[3] ^ B[3] ^ C[3], m3 = majority(A[3], B[3], C[3]);
        v[3] = t3 ^ m2 ^ n2;
        v[4] = m3 | majority(t3, m2, n2);  // at most 27 in all
        uint32_t ge = 0xffffffffu;         // count >= thresh, from the lowest plane up
#pragma unroll
        for (int i = 0; i < 5; ++i)
            ge = (thresh >> i) & 1 ? v[i] & ge : v[i] | ge;
        const uint32_t keep = mid[s + 1] & ge;
        const long long o = ((long long)z * ny + y) * nx + x;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t k = keep >> (16 * h);
            if (x + 16 * h < nx && PCDF_IN(o + 16 * h + 15, V))
                *reinterpret_cast<uint4 *>(out + o + 16 * h) =
                    make_uint4(bit_bytes(k & 15u), bit_bytes((k >> 4) & 15u), bit_bytes((k >> 8) & 15u), bit_bytes((k >> 12) & 15u));
        }
    }
}

// A CTA takes 32 pieces of kPiece columns; its 8 warps share the slices.
template <int kPiece>
__global__ void __launch_bounds__(256)
    k_collapse(const uint8_t *__restrict__ occ, int nx, int ny, int z0, int z1, uint8_t *__restrict__ out2d)
{
    __shared__ uint32_t part[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long V2 = (long long)nx * ny, c = ((long long)blockIdx.x * 32 + lane) * kPiece;
    uint32_t o = 0;
    if (c < V2) {
#pragma unroll 8
        for (int z = z0 + w; z < z1; z += 8) {
            const uint8_t *p = occ + z * V2 + c;
            o |= kPiece == 4 ? __ldg(reinterpret_cast<const uint32_t *>(p)) : __ldg(p);
        }
    }
    part[w][lane] = o;
    __syncthreads();
    if (w == 0 && c < V2) {
#pragma unroll
        for (int k = 1; k < 8; ++k)
            o |= part[k][lane];
        if (kPiece == 4)
            *reinterpret_cast<uint32_t *>(out2d + c) = bit_bytes(byte_bits(o));
        else
            out2d[c] = o != 0;
    }
}

template <int kBW>
void filter_bits(const uint8_t *occ, const pcdf_grid &g, int thresh, uint8_t *out, cudaStream_t st)
{
    constexpr int kBY = 64 / kBW;
    const dim3 tiles((unsigned)((g.nx + 32 * kBW - 1) / (32 * kBW)), (unsigned)((g.ny + kBY - 1) / kBY),
                     (unsigned)((g.nz + kBZ - 1) / kBZ));
    k_voxel_filter_bits<kBW><<<tiles, kBThreads, 0, st>>>(occ, g.nx, g.ny, g.nz, thresh, out);
}

}  // namespace
}  // namespace pcdf

extern "C" {

int pcdf_filter_voxels(const pcdf_grid *grid, const uint8_t *occ, int32_t min_neighbours, uint8_t *out, void *stream)
{
    if (int rc = check_grid(grid))
        return rc;
    if (!occ || !out || occ == out)
        return fail(PCDF_EINVAL, "occ and out must be non-NULL and distinct");
    if (min_neighbours < 0 || min_neighbours > 27)
        return fail(PCDF_EINVAL, "min_neighbours %d outside [0, 27]", min_neighbours);
    const uintptr_t at = (uintptr_t)occ | (uintptr_t)out;
    if (grid->nx % 16 == 0 && (at & 15u) == 0) {
        // words beyond the grid's rows cost as much as others, so two words per
        // row up to 64 voxels (64 x 300 x 300: 7.4 us; 14.6 by words of four
        // voxels), four up to 128 (128 x 300 x 300: 9.1 us; 23.8), else eight
        const auto run = grid->nx <= 64 ? pcdf::filter_bits<2> : grid->nx <= 128 ? pcdf::filter_bits<4> : pcdf::filter_bits<8>;
        run(occ, *grid, min_neighbours + 1, out, (cudaStream_t)stream);
    } else if (grid->nx % 4 == 0 && (at & 3u) == 0) {
        // staged as bits from 4-byte pieces, with a load and three shuffles per
        // four voxels, these rows were slower: 132 x 300 x 300 34 us instead of
        // 24, 196 x 300 x 300 38 instead of 24
        const int nw = grid->nx / 4;
        const dim3 grd((unsigned)((nw + pcdf::kF4Out - 1) / pcdf::kF4Out),
                       (unsigned)((grid->ny + pcdf::kF4Y - 1) / pcdf::kF4Y),
                       (unsigned)((grid->nz + pcdf::kF4Z - 1) / pcdf::kF4Z));
        const uint32_t thresh4 = (uint32_t)(min_neighbours + 1) * 0x01010101u;  // <= 28 per byte
        pcdf::k_voxel_filter4<<<grd, 32 * pcdf::kF4Y, 0, (cudaStream_t)stream>>>(
            (const uint32_t *)occ, nw, grid->ny, grid->nz, thresh4, (uint32_t *)out);
    } else {
        const dim3 blk(pcdf::kFX, pcdf::kFY);
        const dim3 grd((grid->nx + pcdf::kFX - 1) / pcdf::kFX, (grid->ny + pcdf::kFY - 1) / pcdf::kFY,
                       (grid->nz + pcdf::kFZ - 1) / pcdf::kFZ);
        pcdf::k_voxel_filter<<<grd, blk, 0, (cudaStream_t)stream>>>(occ, grid->nx, grid->ny, grid->nz,
                                                                    min_neighbours, out);
    }
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PCDF_OK : cuda_fail(e, "voxel filter");
}

int pcdf_collapse_2d(const pcdf_grid *grid, const uint8_t *occ, int32_t z0, int32_t z1, uint8_t *out2d, void *stream)
{
    if (int rc = check_grid(grid))
        return rc;
    if (!occ || !out2d)
        return fail(PCDF_EINVAL, "occ and out2d must be non-NULL");
    const int a = z0 < 0 ? 0 : z0, b = z1 > grid->nz ? grid->nz : z1;
    const long long V2 = (long long)grid->nx * grid->ny;
    const int end = b < a ? a : b;
    if (V2 % 4 == 0 && (((uintptr_t)occ | (uintptr_t)out2d) & 3u) == 0)  // four columns per access
        pcdf::k_collapse<4><<<(unsigned)((V2 + 127) / 128), 256, 0, (cudaStream_t)stream>>>(occ, grid->nx, grid->ny, a, end,
                                                                                            out2d);
    else
        pcdf::k_collapse<1><<<(unsigned)((V2 + 31) / 32), 256, 0, (cudaStream_t)stream>>>(occ, grid->nx, grid->ny, a, end,
                                                                                          out2d);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PCDF_OK : cuda_fail(e, "collapse");
}

}  // extern "C"
