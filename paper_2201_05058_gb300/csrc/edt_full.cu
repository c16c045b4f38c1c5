// Exact signed EDT of a whole grid (sm_103a): the static map (Sec. 6: the
// environment's exact distance field), the union of the map and the humans'
// primitives at one t (the full per-field recompute that the composite is
// compared against), and a primitive alone on its box (the template of the
// translated primitive field).
//
// Three launches:
//   k_row_bits  one warp per few rows (y, z): the occupancy as 32-bit words
//               (bit l of word w: voxel x = 32 w + l) and, per word, the
//               nearest occupied and free voxel left of it and right of it.
//   k_edt_xy    one CTA per (slice z, 64 columns): the 1-D distance along x of
//               every voxel of its columns from the words and their carries,
//               then the y pass by the block search of blockmin.cuh.  Output:
//               the signed 2-D partial field (int32) of the slice.
//   k_edt_z     one CTA per 64 consecutive columns (x, y) of the partial
//               field: the z pass by the same search, with the float field
//               sign(S) sqrt|S| vox.
// The 1-D row distances never reach memory, so the grid is read once as
// bytes and the 2-D partial field is written and read once.
#include <cuda_runtime.h>

#include "edt_full.cuh"

namespace pcdf {
namespace {

constexpr int kRowWarps = 8;  // k_row_bits: warps per CTA
constexpr int kThreads = 256;   // k_edt_xy, k_edt_z: 8 warps share the blocks of a tile

template <int kMode>
__global__ void __launch_bounds__(32 * kRowWarps)
    k_row_bits(const uint8_t *__restrict__ occ, const __grid_constant__ CapBatch caps, int H, int nx, int ny,
               int nrows, int W, uint32_t *__restrict__ bits, uint2 *__restrict__ carry, int access)
{
    const int row = ((int)blockIdx.x * kRowWarps + (int)(threadIdx.x >> 5)) * full::rows_per_warp(W, access);
    if (row >= nrows)
        return;  // warp-uniform
    full::row_bits_rows<kMode>(occ, caps.caps, H, nx, ny, row, nrows, nrows, W, bits, carry, threadIdx.x & 31, access);
}

// 43 us for a 256^3 map of 60 boxes (85 us with the stack envelopes it
// replaced), 32 us for 317 x 211 x 97 with speckle: instruction issue (67 %
// active).  Four CTAs of 64 registers; held to 48 for five it spills (50 us
// when four took 46).
__global__ void __launch_bounds__(kThreads, 4)
    k_edt_xy(const uint32_t *__restrict__ bits, const uint2 *__restrict__ carry, int nx, int ny, int nz, int W,
             int32_t *__restrict__ mid)
{
    extern __shared__ __align__(16) uint32_t smem[];
    full::edt_xy_block<false>(bits, carry, nx, ny, nz, W, blockIdx.x, blockIdx.y, mid, smem);
}

// 50 us for the 256^3 map in an ncu capture (105 us with the stack envelopes):
// the 12 bytes per voxel alone take 30 us, and it issues on 58 % of the cycles.
template <bool kSdf>
__global__ void __launch_bounds__(kThreads, 4)
    k_edt_z(const int32_t *__restrict__ mid, int32_t *__restrict__ sq, float *__restrict__ sdf, float vox, int n,
            long long ncols, int vec)
{
    extern __shared__ __align__(16) uint32_t smem[];
    full::edt_z_block<kSdf, false>(mid, sq, sdf, vox, n, ncols, (long long)blockIdx.x * full::kTileCols, vec != 0, smem);
}

size_t tile_bytes(int n) { return blockmin::tile_words(n) * sizeof(uint32_t); }

}  // namespace

size_t full_edt_scratch(int nx, int ny, int nz, size_t *bits_off, size_t *carry_off, size_t *mid_off)
{
    const auto al = [](size_t v) { return (v + 255) / 256 * 256; };
    const size_t nw = (size_t)nz * ny * ((nx + 31) / 32);
    *bits_off = 0;
    *carry_off = al(nw * sizeof(uint32_t));
    *mid_off = *carry_off + al(nw * sizeof(uint2));
    return *mid_off + al((size_t)nx * ny * nz * sizeof(int32_t));
}

cudaError_t launch_full_edt(int mode, const uint8_t *occ, const CapBatch *caps, int H, int nx, int ny, int nz,
                            int32_t *sq, float *sdf, float vox, void *ws, cudaStream_t st)
{
    size_t bo, co, mo;
    full_edt_scratch(nx, ny, nz, &bo, &co, &mo);
    uint32_t *bits = (uint32_t *)((char *)ws + bo);
    uint2 *carry = (uint2 *)((char *)ws + co);
    int32_t *mid = (int32_t *)((char *)ws + mo);
    const int W = (nx + 31) / 32;
    const int nrows = ny * nz, access = mode == 0 ? full::row_access(occ, nx) : full::kBytes;
    const int per_cta = kRowWarps * full::rows_per_warp(W, access);
    const unsigned nb = (unsigned)((nrows + per_cta - 1) / per_cta);
    switch (mode) {
    case 0:
        k_row_bits<0><<<nb, 32 * kRowWarps, 0, st>>>(occ, *caps, H, nx, ny, nrows, W, bits, carry, access);
        break;
    case 1:
        k_row_bits<1><<<nb, 32 * kRowWarps, 0, st>>>(occ, *caps, H, nx, ny, nrows, W, bits, carry, access);
        break;
    default:
        k_row_bits<2><<<nb, 32 * kRowWarps, 0, st>>>(occ, *caps, H, nx, ny, nrows, W, bits, carry, access);
        break;
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return e;

    const size_t sxy = tile_bytes(ny);
    if ((e = allow_shared(k_edt_xy)) != cudaSuccess)
        return e;
    const unsigned nt = (unsigned)((nx + full::kTileCols - 1) / full::kTileCols);
    k_edt_xy<<<dim3(nt, (unsigned)nz), kThreads, sxy, st>>>(bits, carry, nx, ny, nz, W, mid);
    if ((e = cudaGetLastError()) != cudaSuccess)
        return e;

    const long long ncols = (long long)nx * ny;
    const unsigned nbz = (unsigned)((ncols + full::kTileCols - 1) / full::kTileCols);
    const size_t sz = tile_bytes(nz);
    // rows of whole 8-byte pairs: two adjacent columns per lane
    const int vec = ncols % 2 == 0 && (((uintptr_t)sq | (uintptr_t)sdf) & 7u) == 0;
    if (sdf) {
        if ((e = allow_shared(k_edt_z<true>)) != cudaSuccess)
            return e;
        k_edt_z<true><<<nbz, kThreads, sz, st>>>(mid, sq, sdf, vox, nz, ncols, vec);
    } else {
        if ((e = allow_shared(k_edt_z<false>)) != cudaSuccess)
            return e;
        k_edt_z<false><<<nbz, kThreads, sz, st>>>(mid, sq, nullptr, vox, nz, ncols, vec);
    }
    return cudaGetLastError();
}

}  // namespace pcdf
