// Predicted composite fields (Sec. 6, Sec. 8) on sm_103a: stand-alone
// kernels and launchers; the algorithms are described in composite.cuh.
#include <cuda_runtime.h>

#include "composite.cuh"

namespace pcdf {
namespace {

// Partial fields of the capsules: one CTA per (slab slice, 64 columns, t).
// 8 warps; like k_edt_xy bound by instruction issue.  3 humans on 256^2, 7
// distinct slices at each of 20 t: 40 us (111 us with an envelope per column
// and thread, whose serial chain left 8 % of the warps active); 4 humans on
// 161 x 115, T = 9: 17 us (82 us).
__global__ void __launch_bounds__(256, 4)
    k_dyn_xy(const __grid_constant__ CapBatch caps, const __grid_constant__ SlabMap map, int H, int nx, int ny,
             int zlo, int S, int t0, int32_t *__restrict__ dyn_mid)
{
    const int ntile = (nx + full::kTileCols - 1) / full::kTileCols;
    const int s = (int)blockIdx.x / ntile, w2 = (int)blockIdx.x % ntile;
    const int t = t0 + (int)blockIdx.y;
    // a slice whose cross-sections equal an earlier slice's is read from that one
    if (map.on && map.rep[t * S + s] != s)
        return;
    extern __shared__ __align__(16) uint32_t sm[];
    full::capsule_xy_block(caps.caps + blockIdx.y * H, H, nx, ny, zlo + s, w2,
                           dyn_mid + ((long long)t * S + s) * nx * ny, sm);
}

// CTAs are ordered t-fastest: those of one column block run together and the
// static block comes from DRAM once.  Three CTAs of 8 warps (80 registers).
// 256^3, T = 20, 3 humans: 463 us for 2.82 GB of outputs and inputs, 90 % of
// the measured copy bandwidth (558 us, and 15 us of column maxima, with an
// envelope per column and thread); 161 x 115 x 83, T = 9: 46 us (88 us).
template <bool kSq, bool kSdfOut, bool kStaticSdf>
__global__ void __launch_bounds__(comp::kThreadsZ, 3)
    k_composite_z(const comp::Composite<kSq, kSdfOut, kStaticSdf> c, const __grid_constant__ SlabMap map, int t0, int nt,
                  int steps)
{
    extern __shared__ __align__(16) uint32_t smem[];
    const int groups = (nt + steps - 1) / steps, g = (int)blockIdx.x % groups;
    comp::Composite<kSq, kSdfOut, kStaticSdf> cc = c;
    cc.rep = map.on ? map.rep : nullptr;
    cc.run(t0 + g * steps, min(steps, nt - g * steps), (long long)(blockIdx.x / groups) * full::kTileCols, smem);
}

__global__ void k_broadcast_static(const int32_t *__restrict__ static_sq, long long V, int t0, int nt,
                                   int32_t *__restrict__ comp_sq, float *__restrict__ comp_sdf, float vox)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += stride) {
        const int32_t s = __ldg(static_sq + v);
        const float f = sq_to_sdf(s, vox);
        for (int t = t0; t < t0 + nt; ++t) {
            if (comp_sq)
                __stcs(comp_sq + (long long)t * V + v, s);
            if (comp_sdf)
                __stcs(comp_sdf + (long long)t * V + v, f);
        }
    }
}

}  // namespace

size_t dyn_xy_words(int ny, int run_rows) { return blockmin::tile_words(ny) + (size_t)run_rows; }

cudaError_t launch_dyn_xy(const CapBatch *caps, const SlabMap *map, int H, int nx, int ny, int zlo, int S, int t0,
                          int n_t, int run_rows, int32_t *dyn_mid, cudaStream_t stream)
{
    if (S <= 0 || n_t <= 0)
        return cudaSuccess;
    cudaError_t e = allow_shared(k_dyn_xy);
    if (e != cudaSuccess)
        return e;
    const unsigned nt = (unsigned)((nx + full::kTileCols - 1) / full::kTileCols);
    k_dyn_xy<<<dim3((unsigned)S * nt, (unsigned)n_t), 256, dyn_xy_words(ny, run_rows) * 4, stream>>>(
        *caps, *map, H, nx, ny, zlo, S, t0, dyn_mid);
    return cudaGetLastError();
}

namespace {

template <bool kSq, bool kSdfOut, bool kStaticSdf>
cudaError_t launch_cz(const comp::Composite<kSq, kSdfOut, kStaticSdf> &c, const SlabMap *map, int t0, int nt,
                      cudaStream_t stream)
{
    auto kern = k_composite_z<kSq, kSdfOut, kStaticSdf>;
    cudaError_t e = allow_shared(kern);
    if (e != cudaSuccess)
        return e;
    // three CTAs per SM share its shared memory
    const int steps = comp::steps_per_cta(c.zlo, c.S, c.nz, nt, 72 * 1024);
    const size_t smem = steps * comp::slab_words(c.zlo, c.S, c.nz) * sizeof(uint32_t);
    const int ntile = (c.V2 + full::kTileCols - 1) / full::kTileCols;
    kern<<<(unsigned)(ntile * ((nt + steps - 1) / steps)), comp::kThreadsZ, smem, stream>>>(c, *map, t0, nt, steps);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_composite_z(const int32_t *static_sq, const float *static_sdf, const int32_t *dyn_mid,
                               const SlabMap *map, int nx, int ny, int nz, int zlo, int S, int t0, int nt,
                               int32_t *comp_sq, float *comp_sdf, float vox, cudaStream_t stream)
{
    const bool sq = comp_sq != nullptr, sd = comp_sdf != nullptr, st = static_sdf != nullptr && sd;
    // two adjacent columns in 8 bytes: every row of every field starts on such a boundary
    const bool vec = nx * ny % 2 == 0 && (((uintptr_t)static_sq | (uintptr_t)(st ? static_sdf : nullptr) |
                                           (uintptr_t)comp_sq | (uintptr_t)comp_sdf | (uintptr_t)dyn_mid) & 7u) == 0;
#define PCDF_CZ(a, b, c)                                                                                            \
    return launch_cz<a, b, c>({static_sq, static_sdf, dyn_mid, nullptr, comp_sq, comp_sdf, nx * ny, nz, zlo, S, vox, \
                               vec},                                                                               \
                              map, t0, nt, stream)
    if (sq && sd && st)
        PCDF_CZ(true, true, true);
    if (sq && sd)
        PCDF_CZ(true, true, false);
    if (sq)
        PCDF_CZ(true, false, false);
    if (st)
        PCDF_CZ(false, true, true);
    PCDF_CZ(false, true, false);
#undef PCDF_CZ
}

cudaError_t launch_broadcast_static(const int32_t *static_sq, long long V, int t0, int nt, int32_t *comp_sq,
                                    float *comp_sdf, float vox, cudaStream_t stream)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    long long nblk = (V + 255) / 256;
    if (nblk > (long long)sms * 8)
        nblk = (long long)sms * 8;
    k_broadcast_static<<<(unsigned)nblk, 256, 0, stream>>>(static_sq, V, t0, nt, comp_sq, comp_sdf, vox);
    return cudaGetLastError();
}

}  // namespace pcdf
