// Many environments of uneven size, horizon and human count in one
// persistent launch (sm_103a).
//
// Every environment needs the static field (row words, the fused x+y pass and
// the z pass of edt_full.cuh) and its T composite fields (capsule x+y pass
// over the slab, fused z pass).  The host cuts all of that
// into work items (environment, stage, tile).  The first persistent launch
// takes the row-pass, capsule, y and z items from a global queue in that
// order; the second takes the composite items (column block, time steps) of
// the single-environment kernel.  Two launches let each have its own register and shared
// memory budget.  An item whose inputs come from an earlier stage of the same
// environment waits (one thread, bounded spin, acquire loads) until the
// completion counter of that stage reaches the stage's item count; finished
// items publish with a release increment.  Because an item only ever waits for
// items that were taken from the queue before it, by CTAs that are already
// running, the queue always drains, whatever the number of resident CTAs.
// A wait that exceeds its bound sets an error word, counts the item as done
// and skips it; the host reads the word with pcdf_batch_error.
//
// The launch needs no host synchronisation and no allocation, so it can be
// captured in a CUDA graph together with the counter reset.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "composite.cuh"
#include "edt_full.cuh"
#include "host.h"

using namespace pcdf::host;

namespace pcdf {
namespace {

constexpr int kFirst = 256;  // threads of the first launch
constexpr int kSecond = 128;  // and of the second: grids of 8 to 16 blocks of slices keep 4 warps busy, not 8
constexpr long long kSpinLimit = 1LL << 22;  // x 256 ns sleep: about one second

enum ItemType : int { kRow = 0, kY = 1, kZ = 2, kDyn = 3, kComp = 4 };

struct BatchItem {
    int type, env, a, b;
};

struct BatchEnv {
    int nx, ny, nz, T, H, zlo, S, W;
    float vox;
    int need[3];  // items of the row, y and z stages
    int vec;      // two columns in 8 bytes (composite items)
    int steps;    // time steps that a composite CTA takes together
    int group;    // and those of a composite item: a multiple
    const uint8_t *occ;
    int32_t *comp_sq;
    uint32_t *bits;   // row words, [nz][ny][W]
    uint2 *carry;     // their carries, [nz][ny][W]
    int32_t *mid;
    int32_t *static_sq;
    int32_t *dyn;
    const uint8_t *rep;   // [T][S] slab slice map (slices of equal capsule cross-sections); NULL: identity
    const CapInfo *caps;  // [T][H]
};

__device__ __forceinline__ int ld_acquire(const int *p)
{
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void add_release(int *p, int v)
{
    asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Wait until *p >= target.  Gives up after about a second, or at once when an
// earlier wait has already failed, so a broken dependency cannot keep the
// kernel alive for long.
__device__ bool wait_ge(const int *p, int target, int *err)
{
    for (long long i = 0; i < kSpinLimit; ++i) {
        if (ld_acquire(p) >= target)
            return true;
        if ((i & 255) == 0 && ld_acquire(err) != 0)
            return false;
        __nanosleep(256);
    }
    atomicExch(err, 1);
    return false;
}

__device__ __forceinline__ void run_rows(const BatchEnv &E, int r0, int r1)
{
    const int lane = threadIdx.x & 31;
    const int access = full::row_access(E.occ, E.nx), per = full::rows_per_warp(E.W, access);
    for (int r = r0 + (threadIdx.x >> 5) * per; r < r1; r += kFirst / 32 * per)
        full::row_bits_rows<0>(E.occ, nullptr, 0, E.nx, E.ny, r, r1, E.ny * E.nz, E.W, E.bits, E.carry, lane, access);
}

// 3 CTAs of 8 warps per SM: the tile of a 320-voxel axis takes 63 KB.  0.71 ms
// for 16 environments (60 M static voxels, 72 M of distinct capsule slices).
__global__ void __launch_bounds__(kFirst, 3)
    k_batched(const BatchEnv *__restrict__ envs, const BatchItem *__restrict__ items, int n_items, int *state,
              int row_rows, int dyn_slices)
{
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ int s_item, s_ok;
    int *head = state, *err = state + 1, *ctr = state + 2;  // ctr[4 * env + stage]
    blockmin::fill_squares(smem);  // every tile begins with them: once for all items
    for (;;) {
        if (threadIdx.x == 0)
            s_item = atomicAdd(head, 1);
        __syncthreads();
        const int it = s_item;
        if (it >= n_items)
            break;
        const BatchItem I = items[it];
        const BatchEnv &E = envs[I.env];
        int *ce = ctr + 4 * I.env;
        if (threadIdx.x == 0) {
            bool ok = true;
            if (I.type == kY)
                ok = wait_ge(ce + kRow, E.need[kRow], err);
            else if (I.type == kZ)
                ok = wait_ge(ce + kY, E.need[kY], err);
            s_ok = ok;
        }
        __syncthreads();
        if (s_ok) {
            switch (I.type) {
            case kRow:
                run_rows(E, I.a, min(I.a + row_rows, E.ny * E.nz));
                break;
            case kY:  // slice I.a, columns from 64 I.b
                full::edt_xy_block<true, true>(E.bits, E.carry, E.nx, E.ny, E.nz, E.W, I.b, I.a, E.mid, smem);
                break;
            case kZ:
                full::edt_z_block<false, true, true>(E.mid, E.static_sq, nullptr, 0.f, E.nz, (long long)E.nx * E.ny,
                                               (long long)I.a, E.nx * E.ny % 2 == 0, smem);
                break;
            case kDyn: {  // time I.a, slices from I.b / 16, columns from 64 (I.b % 16)
                const int s0 = I.b >> 4;
                for (int s = s0; s < min(s0 + dyn_slices, E.S); ++s) {
                    if (E.rep && E.rep[I.a * E.S + s] != s)
                        continue;  // read from the earlier slice of equal cross-sections
                    full::capsule_xy_block<true>(E.caps + (long long)I.a * E.H, E.H, E.nx, E.ny, E.zlo + s, I.b & 15,
                                           E.dyn + ((long long)I.a * E.S + s) * E.nx * E.ny, smem);
                    __syncthreads();
                }
                break;
            }
            default:
                break;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            add_release(ce + I.type, 1);
        }
    }
}

// The composite items, after every static and capsule item has finished (the
// previous launch on the stream): item (env, t, column block) computes time
// steps t .. t + E.group - 1 of 64 consecutive columns, E.steps at a time,
// reading the static block once for them.  Nothing to wait for; if a
// dependency wait of the first launch expired, the items are skipped.  1.30 ms
// for the 16 environments (888 M voxel fields) whose stores alone take 0.52 ms;
// the envelope per column it replaced took 1.75 ms, 8 warps per CTA take 1.52.
__global__ void __launch_bounds__(kSecond, 6)
    k_batched_comp(const BatchEnv *__restrict__ envs, const BatchItem *__restrict__ items, int n_items,
                   const int *__restrict__ err, int *head)
{
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ int s_item;
    if (*err != 0)
        return;  // uniform: every thread reads the same word
    for (;;) {
        if (threadIdx.x == 0)
            s_item = atomicAdd(head, 1);
        __syncthreads();
        const int it = s_item;
        if (it >= n_items)
            break;
        const BatchItem I = items[it];
        const BatchEnv &E = envs[I.env];
        const int t1 = min(I.a + E.group, E.T);
        const comp::Composite<true, false, false> c = {E.static_sq, nullptr, E.dyn, E.rep, E.comp_sq, nullptr,
                                                       E.nx * E.ny, E.nz, E.zlo, E.S, E.vox, E.vec != 0};
        for (int t = I.a; t < t1; t += E.steps) {
            c.run(t, min(E.steps, t1 - t), (long long)I.b, smem);
            __syncthreads();
        }
    }
}

// shared memory words of the first launch's stages, and of a composite item
size_t smem_words_env(const CompositePlan &p, const pcdf_grid &g)
{
    size_t w = std::max(blockmin::tile_words(g.ny), blockmin::tile_words(g.nz));
    if (p.S > 0)
        w = std::max(w, dyn_xy_words(g.ny, p.run_rows));
    return w;
}
constexpr size_t kCompShared = 36 * 1024;  // of a composite CTA: six per SM

}  // namespace
}  // namespace pcdf

struct pcdf_batch {
    pcdf_batch_tiles tiles;
    int n_env = 0;
    std::vector<pcdf_env> user;
    std::vector<pcdf::host::CompositePlan> plans;
    std::vector<pcdf::BatchEnv> desc;   // device pointers filled at upload
    std::vector<size_t> off_bits, off_carry, off_mid, off_static, off_dyn, off_caps, off_rep;
    std::vector<pcdf::BatchItem> items;  // the first launch's items, then the composite items
    int n_first = 0;                     // items of the first launch
    size_t off_desc = 0, off_items = 0, off_state = 0, bytes = 0;
    size_t smem = 0, smem_comp = 0;
    int blocks = 0, blocks_comp = 0;
};

namespace {

void default_tiles(pcdf_batch_tiles &t)
{
    if (t.row_rows <= 0)
        t.row_rows = 32;
    if (t.dyn_slices <= 0)
        t.dyn_slices = 1;
    if (t.comp_t <= 0)
        t.comp_t = 1;
}

int build_plan(const pcdf_env *envs, int n_env, const pcdf_batch_tiles *tiles, pcdf_batch &B)
{
    using namespace pcdf;
    if (n_env < 1 || !envs)
        return fail(PCDF_EINVAL, "n_env must be >= 1 and envs non-NULL");
    B.tiles = tiles ? *tiles : pcdf_batch_tiles{0, 0, 0};
    default_tiles(B.tiles);
    if (B.tiles.row_rows > 4096 || B.tiles.dyn_slices > 512 || B.tiles.comp_t > PCDF_MAX_T)
        return fail(PCDF_EINVAL, "tile shape out of range");
    B.n_env = n_env;
    B.user.assign(envs, envs + n_env);
    B.plans.resize(n_env);
    B.desc.resize(n_env);
    B.off_bits.resize(n_env);
    B.off_carry.resize(n_env);
    B.off_mid.resize(n_env);
    B.off_static.resize(n_env);
    B.off_dyn.resize(n_env);
    B.off_caps.resize(n_env);
    B.off_rep.resize(n_env);
    size_t off = 0, words = 0, words_comp = 0;
    std::vector<BatchItem> rows, dyn, ys, zs, comps;
    for (int e = 0; e < n_env; ++e) {
        const pcdf_env &U = envs[e];
        if (!U.occ || !U.comp_sq)
            return fail(PCDF_EINVAL, "environment %d: occ and comp_sq must be non-NULL", e);
        CompositePlan &p = B.plans[e];
        if (int rc = plan_composite(&U.grid, U.T, U.H, U.caps, p))
            return rc;
        if (p.S > 0 && !p.fused)
            return fail(PCDF_EINVAL, "environment %d: capsule row bound %d too large for the batched kernel", e,
                        p.cap);
        // slabs of more than 438 slices are refused, as they always have been
        // (a composite item once needed 128 columns of them in shared memory)
        const size_t slab = (size_t)128 * (p.S + 2 + (p.S + 31) / 32) * sizeof(uint32_t);
        if (slab > kMaxShared)
            return fail(PCDF_EINVAL, "an environment needs %zu bytes of shared memory (limit 227 KB)", slab);
        const pcdf_grid &g = U.grid;
        const long long V = (long long)g.nx * g.ny * g.nz;
        const size_t nw = (size_t)g.nz * g.ny * ((g.nx + 31) / 32);
        B.off_bits[e] = off;
        off += align_up(nw * sizeof(uint32_t));
        B.off_carry[e] = off;
        off += align_up(nw * sizeof(uint2));
        B.off_mid[e] = off;
        off += align_up((size_t)V * 4);
        B.off_static[e] = off;
        off += align_up((size_t)V * 4);
        B.off_dyn[e] = off;
        off += align_up((size_t)p.slab * 4);
        B.off_caps[e] = off;
        off += align_up(p.ci.size() * sizeof(CapInfo));
        B.off_rep[e] = off;
        off += align_up(p.rep.size());
        words = std::max(words, smem_words_env(p, g));

        BatchEnv &D = B.desc[e];
        std::memset(&D, 0, sizeof(D));
        D.nx = g.nx;
        D.ny = g.ny;
        D.nz = g.nz;
        D.T = U.T;
        D.H = U.H;
        D.zlo = p.zlo;
        D.S = p.S;
        D.W = (g.nx + 31) / 32;
        D.vox = g.vox;
        D.steps = comp::steps_per_cta(p.zlo, p.S, g.nz, U.T, kCompShared);
        // whole runs of the steps that a CTA takes together (items of comp_t = 1,
        // taken four at a time, split them: 9 steps as 3 + 1 + 3 + 1 + 1)
        D.group = (std::max(B.tiles.comp_t, 1) + D.steps - 1) / D.steps * D.steps;
        words_comp = std::max(words_comp, D.steps * comp::slab_words(p.zlo, p.S, g.nz));
        const int nrows = g.ny * g.nz;
        for (int r = 0; r < nrows; r += B.tiles.row_rows)
            rows.push_back({kRow, e, r, 0});
        D.need[kRow] = (nrows + B.tiles.row_rows - 1) / B.tiles.row_rows;
        const int nxb = (g.nx + full::kTileCols - 1) / full::kTileCols;  // column blocks of a slice (<= 8)
        // slices that repeat an earlier one's cross-sections need no item: most of
        // an upright human's, and taking an empty item from the queue costs as much
        // as a small one
        for (int t = 0; t < U.T; ++t)
            for (int s = 0; s < p.S; s += B.tiles.dyn_slices) {
                bool any = p.rep.empty();
                for (int k = s; k < std::min(s + B.tiles.dyn_slices, p.S) && !any; ++k)
                    any = p.rep[(size_t)t * p.S + k] == k;
                if (!any)
                    continue;
                for (int xb = 0; xb < nxb; ++xb)
                    dyn.push_back({kDyn, e, t, s * 16 + xb});
            }
        const long long zcols = (long long)g.nx * g.ny;
        for (int z = 0; z < g.nz; ++z)
            for (int x = 0; x < g.nx; x += full::kTileCols)
                ys.push_back({kY, e, z, x / full::kTileCols});
        D.need[kY] = g.nz * ((g.nx + full::kTileCols - 1) / full::kTileCols);
        for (long long c = 0; c < zcols; c += full::kTileCols)
            zs.push_back({kZ, e, (int)c, 0});
        D.need[kZ] = (int)((zcols + full::kTileCols - 1) / full::kTileCols);
        // composite items t-fastest within a column block: the blocks of one
        // column range run together and share the static column in L2
        for (long long c = 0; c < zcols; c += full::kTileCols)
            for (int t = 0; t < U.T; t += D.group)
                comps.push_back({kComp, e, t, (int)c});
    }
    B.items.clear();
    for (auto *v : {&rows, &dyn, &ys, &zs})
        B.items.insert(B.items.end(), v->begin(), v->end());
    B.n_first = (int)B.items.size();
    B.items.insert(B.items.end(), comps.begin(), comps.end());
    B.off_desc = off;
    off += align_up(sizeof(BatchEnv) * n_env);
    B.off_items = off;
    off += align_up(sizeof(BatchItem) * B.items.size());
    B.off_state = off;
    off += align_up(sizeof(int) * (3 + 4 * (size_t)n_env));
    B.bytes = off;
    B.smem = words * 4;
    B.smem_comp = std::max<size_t>(words_comp * 4, 16);
    if (B.smem > 227 * 1024 || B.smem_comp > 227 * 1024)
        return fail(PCDF_EINVAL, "an environment needs %zu bytes of shared memory (limit 227 KB)",
                    std::max(B.smem, B.smem_comp));
    cudaFuncAttributes a1, a2;
    cudaError_t e = cudaFuncGetAttributes(&a1, k_batched);
    if (e == cudaSuccess)
        e = cudaFuncGetAttributes(&a2, k_batched_comp);
    if (e == cudaSuccess)
        e = allow_shared(k_batched, a1.sharedSizeBytes);
    if (e == cudaSuccess)
        e = allow_shared(k_batched_comp, a2.sharedSizeBytes);
    if (e != cudaSuccess)
        return cuda_fail(e, "batched kernel attributes");
    int dev = 0, sms = 0, per_sm = 0, per_sm_comp = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_batched, kFirst, B.smem);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_comp, k_batched_comp, kSecond, B.smem_comp);
    if (e != cudaSuccess)
        return cuda_fail(e, "batched kernel occupancy");
    B.blocks = std::max(1, sms * std::max(per_sm, 1));
    B.blocks_comp = std::max(1, sms * std::max(per_sm_comp, 1));
    return PCDF_OK;
}

}  // namespace

extern "C" {

int pcdf_batch_create(const pcdf_env *envs, int32_t n_env, const pcdf_batch_tiles *tiles, pcdf_batch **out)
{
    if (!out)
        return fail(PCDF_EINVAL, "out is NULL");
    *out = nullptr;
    pcdf_batch *B = new pcdf_batch();
    if (int rc = build_plan(envs, n_env, tiles, *B)) {
        delete B;
        return rc;
    }
    *out = B;
    return PCDF_OK;
}

void pcdf_batch_destroy(pcdf_batch *b) { delete b; }

int pcdf_batch_workspace_bytes(const pcdf_batch *b, size_t *bytes)
{
    if (!b || !bytes)
        return fail(PCDF_EINVAL, "batch and bytes must be non-NULL");
    *bytes = b->bytes;
    return PCDF_OK;
}

int pcdf_batch_tiles_used(const pcdf_batch *b, pcdf_batch_tiles *tiles)
{
    if (!b || !tiles)
        return fail(PCDF_EINVAL, "batch and tiles must be non-NULL");
    *tiles = b->tiles;
    return PCDF_OK;
}

int pcdf_batch_block_stage(pcdf_batch *b, int32_t env, int32_t stage)
{
    if (!b || env < 0 || env >= b->n_env || stage < 0 || stage > 2)
        return fail(PCDF_EINVAL, "batch, environment %d or stage %d out of range (stages 0 to 2 have waiters)", env,
                    stage);
    b->desc[env].need[stage] = 1 << 30;  // above any item count: the waits on it can only expire
    return PCDF_OK;
}

int pcdf_batch_upload(pcdf_batch *b, void *workspace, size_t workspace_bytes, void *stream)
{
    using namespace pcdf;
    if (!b || !workspace)
        return fail(PCDF_EINVAL, "batch and workspace must be non-NULL");
    if (!aligned(workspace, kAlign))
        return fail(PCDF_EINVAL, "workspace must be %zu-byte aligned", kAlign);
    if (workspace_bytes < b->bytes)
        return fail(PCDF_ENOMEM, "workspace %zu bytes < %zu needed", workspace_bytes, b->bytes);
    char *ws = (char *)workspace;
    cudaStream_t st = (cudaStream_t)stream;
    for (int e = 0; e < b->n_env; ++e) {
        BatchEnv &D = b->desc[e];
        D.occ = b->user[e].occ;
        D.comp_sq = b->user[e].comp_sq;
        D.bits = (uint32_t *)(ws + b->off_bits[e]);
        D.carry = (uint2 *)(ws + b->off_carry[e]);
        D.mid = (int32_t *)(ws + b->off_mid[e]);
        D.static_sq = (int32_t *)(ws + b->off_static[e]);
        D.vec = D.nx * D.ny % 2 == 0 && ((uintptr_t)D.comp_sq & 7u) == 0;  // the workspace's fields are aligned
        D.dyn = (int32_t *)(ws + b->off_dyn[e]);
        D.caps = (const CapInfo *)(ws + b->off_caps[e]);
        const std::vector<uint8_t> &rp = b->plans[e].rep;
        D.rep = rp.empty() ? nullptr : (const uint8_t *)(ws + b->off_rep[e]);
        if (!rp.empty()) {
            cudaError_t err = cudaMemcpyAsync(ws + b->off_rep[e], rp.data(), rp.size(), cudaMemcpyHostToDevice, st);
            if (err != cudaSuccess)
                return cuda_fail(err, "batch upload");
        }
        const std::vector<CapInfo> &ci = b->plans[e].ci;
        if (!ci.empty()) {
            cudaError_t err = cudaMemcpyAsync(ws + b->off_caps[e], ci.data(), ci.size() * sizeof(CapInfo),
                                              cudaMemcpyHostToDevice, st);
            if (err != cudaSuccess)
                return cuda_fail(err, "batch upload");
        }
    }
    cudaError_t err = cudaMemcpyAsync(ws + b->off_desc, b->desc.data(), sizeof(BatchEnv) * b->n_env,
                                      cudaMemcpyHostToDevice, st);
    if (err == cudaSuccess)
        err = cudaMemcpyAsync(ws + b->off_items, b->items.data(), sizeof(BatchItem) * b->items.size(),
                              cudaMemcpyHostToDevice, st);
    if (err != cudaSuccess)
        return cuda_fail(err, "batch upload");
    return PCDF_OK;
}

int pcdf_batch_run(const pcdf_batch *b, void *workspace, void *stream)
{
    using namespace pcdf;
    if (!b || !workspace)
        return fail(PCDF_EINVAL, "batch and workspace must be non-NULL");
    char *ws = (char *)workspace;
    cudaStream_t st = (cudaStream_t)stream;
    int *state = (int *)(ws + b->off_state);
    cudaError_t err = cudaMemsetAsync(state, 0, sizeof(int) * (3 + 4 * (size_t)b->n_env), st);
    if (err != cudaSuccess)
        return cuda_fail(err, "batch counter reset");
    const BatchEnv *desc = (const BatchEnv *)(ws + b->off_desc);
    const BatchItem *items = (const BatchItem *)(ws + b->off_items);
    k_batched<<<b->blocks, kFirst, b->smem, st>>>(desc, items, b->n_first, state, b->tiles.row_rows,
                                                  b->tiles.dyn_slices);
    err = cudaGetLastError();
    if (err != cudaSuccess)
        return cuda_fail(err, "batched launch");
    const int n_comp = (int)b->items.size() - b->n_first;
    k_batched_comp<<<b->blocks_comp, kSecond, b->smem_comp, st>>>(desc, items + b->n_first, n_comp, state + 1,
                                                                  state + 2 + 4 * b->n_env);
    err = cudaGetLastError();
    return err == cudaSuccess ? PCDF_OK : cuda_fail(err, "batched composite launch");
}

int pcdf_batch_error(const pcdf_batch *b, const void *workspace, void *stream, int32_t *code)
{
    if (!b || !workspace || !code)
        return fail(PCDF_EINVAL, "batch, workspace and code must be non-NULL");
    int word = 0;
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t err = cudaMemcpyAsync(&word, (const char *)workspace + b->off_state + sizeof(int), sizeof(int),
                                      cudaMemcpyDeviceToHost, st);
    if (err == cudaSuccess)
        err = cudaStreamSynchronize(st);
    if (err != cudaSuccess)
        return cuda_fail(err, "batch error read");
    *code = word ? PCDF_ETIMEOUT : PCDF_OK;
    return PCDF_OK;
}

int pcdf_batch_autotune_workspace_bytes(const pcdf_env *envs, int32_t n_env, size_t *bytes)
{
    if (!bytes)
        return fail(PCDF_EINVAL, "bytes is NULL");
    // the smallest tiles give the longest item list, hence the largest layout
    pcdf_batch_tiles t{8, 1, 1};
    pcdf_batch B;
    if (int rc = build_plan(envs, n_env, &t, B))
        return rc;
    *bytes = B.bytes;
    return PCDF_OK;
}

int pcdf_batch_autotune(const pcdf_env *envs, int32_t n_env, void *workspace, size_t workspace_bytes, void *stream,
                        int32_t reps, pcdf_batch_tiles *best, float *best_ms)
{
    if (!best)
        return fail(PCDF_EINVAL, "best is NULL");
    cudaStream_t st = (cudaStream_t)stream;
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess)
        return fail(PCDF_ECUDA, "event creation failed");
    float best_t = -1.f;
    int rc = PCDF_OK;
    for (int rr : {8, 32, 128})
        for (int ds : {1, 4})
            for (int ct : {1, 4}) {
                pcdf_batch_tiles t{rr, ds, ct};
                pcdf_batch B;
                if ((rc = build_plan(envs, n_env, &t, B)))
                    goto done;
                if ((rc = pcdf_batch_upload(&B, workspace, workspace_bytes, stream)))
                    goto done;
                if ((rc = pcdf_batch_run(&B, workspace, stream)))  // warm-up
                    goto done;
                float tot = 0.f;
                for (int k = 0; k < std::max(reps, 1); ++k) {
                    cudaEventRecord(e0, st);
                    if ((rc = pcdf_batch_run(&B, workspace, stream)))
                        goto done;
                    cudaEventRecord(e1, st);
                    if (cudaEventSynchronize(e1) != cudaSuccess) {
                        rc = fail(PCDF_ECUDA, "autotune synchronisation failed");
                        goto done;
                    }
                    float ms = 0.f;
                    cudaEventElapsedTime(&ms, e0, e1);
                    tot += ms;
                }
                int32_t code = 0;
                if ((rc = pcdf_batch_error(&B, workspace, stream, &code)))
                    goto done;
                if (code != PCDF_OK) {
                    rc = fail(code, "batched kernel reported a dependency timeout during autotuning");
                    goto done;
                }
                tot /= std::max(reps, 1);
                if (best_t < 0.f || tot < best_t) {
                    best_t = tot;
                    *best = t;
                }
            }
done:
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (rc == PCDF_OK && best_ms)
        *best_ms = best_t;
    return rc;
}

}  // extern "C"
