// Plan and dispatch of the tensor-core decode kernel (mkv_tc_kernel.cuh): operand geometry, tensor maps, launch.
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <new>

#include "mkv_tc_kernel.cuh"

namespace mkv {

extern template cudaError_t tc_launch_group<1>(TcPlan *, const DecodeArgs &, cudaStream_t);
extern template cudaError_t tc_launch_group<2>(TcPlan *, const DecodeArgs &, cudaStream_t);
extern template cudaError_t tc_launch_group<4>(TcPlan *, const DecodeArgs &, cudaStream_t);
extern template cudaError_t tc_launch_group<8>(TcPlan *, const DecodeArgs &, cudaStream_t);
extern template cudaError_t tc_launch_group<16>(TcPlan *, const DecodeArgs &, cudaStream_t);

namespace {

int pad32(int x) { return (x + 31) & ~31; }

}  // namespace

int tc_padded_group(int G)
{
    int g = 1;
    while (g < G) g *= 2;
    return g;
}

// Chunks the recent-query ring is cut into: one MMA takes at most 256 ring rows (N of the instruction, and with
// two accumulator buffers the 512 TMEM columns).
int tc_ring_chunks(int G, int R)
{
    const int rows = R * tc_padded_group(G);
    return rows <= 256 ? 1 : (rows + 255) / 256;
}

namespace {
constexpr int kMaxRingChunks = 8;
// rows of one chunk: the chunks are made equally wide (a multiple of 32, hence of the padded group)
int chunk_rows(int G, int R)
{
    const int rows = R * tc_padded_group(G), nc = tc_ring_chunks(G, R);
    return pad32((rows + nc - 1) / nc);
}
}  // namespace

// Ring slots a step scores: the block that is being filled (DecodeArgs::slab), or with CURRENT normalisation the chunk
// of the ring that holds the new query's slot, whose other chunks are scored beside it.
// Block size: bs * G' rows are scored per key on every step and once more when the block is finished, and a block's
// slab costs 4 bytes per key beside the 512 of its K and V, so wide windows take larger blocks.  32 rows is what one
// TMEM load brings; two blocks of 128 rows are the 256 one MMA takes, but at G' = 16 leave room for two 32 KB stages only, so
// narrow windows take half of that (148 units x 4096 slots, R = 16: 177 us per step with 8 slots, 174 with 4; a layer of 8 units
// x 1056 38 and, on the warp-level kernel, which two blocks of 64 rows fit, 19).
int tc_block_slots(int G, int R, bool current)
{
    const int g = tc_padded_group(G);
    if (current) return tc_ring_chunks(G, R) > 1 ? chunk_rows(G, R) / g : R;
    int bs = R <= 96 ? 8 : R <= 384 ? 16 : 32;
    bs = std::max(bs, 32 / g);
    bs = std::min(bs, (R <= 96 ? 64 : 128) / g);
    return bs < R ? bs : R;
}

// G: the model's GQA ratio; the kernel works with the group padded to a power of two
bool tc_shape_supported(bool f32, int D, int G, int R)
{
    if (f32 || D != kD || G < 1 || G > kMaxGroup || R < 1) return false;
    return tc_ring_chunks(G, R) <= kMaxRingChunks;
}

int tc_grid(int U, int cap, int splits_hint, int n_sm) { return sched_grid(U, cap, splits_hint, n_sm); }

int tc_partials_per_unit(int U, int cap, int grid) { return sched_partials_per_unit(U, cap, grid); }

cudaError_t tc_plan_create(TcPlan **out, const DecodeArgs &a, int grid, unsigned long long wait_limit_cycles, bool prefetch,
                           char *err, size_t err_len)
{
    *out = nullptr;
    TcPlan *p = new (std::nothrow) TcPlan;
    if (!p) return cudaErrorMemoryAllocation;
    memset(p, 0, sizeof(*p));
    int dev = 0, n_sm = 0, max_smem = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) { delete p; return e; }
    TcGeom &g = p->geo;
    const int G = a.G;
    g.nc = a.nc;
    g.qbox = pad32(a.bs * G);
    g.rgpad = a.nblk > 1 && !a.norm_current ? 2 * g.qbox : g.qbox;
    if (a.bs != tc_block_slots(a.Gq, a.R, a.norm_current != 0) || g.rgpad > 256 || (long long)a.bs * a.nblk * g.nc < a.R ||
        (g.nc > 1 && !a.Fc) || (a.nblk > 1 && (g.qbox != a.bs * G || !a.slab || !a.pre || !a.sum_pos))) {
        snprintf(err, err_len, "tensor-core kernel: ring block geometry does not match the shape");
        delete p;
        return cudaErrorInvalidValue;
    }
    g.ng = kComputeGroups;
    g.nb = g.rgpad <= 128 ? 4 : 2;
    g.tmem_cols = 32;
    while (g.tmem_cols < g.nb * g.rgpad) g.tmem_cols *= 2;
    g.grid = grid;
    g.wait_cycles = wait_limit_cycles > 0 ? (long long)wait_limit_cycles : kWaitCycles;
    // Two tiles: what counts is that a CTA's first loads after the wait hit L2 (config 1: 56.1 instead of 57.1 us per
    // step with 1 to 3 tiles).  More is worse - 8 tiles cost 3 us, 32 tiles 10 us - because the prefetches compete
    // with the previous grid's last CTAs.  Prefetching the first item's query ring as well changed nothing.
    // A launch over one layer's few units, whose CTAs hold two tiles or so each, is slower with it (17.9 instead of
    // 16.9 us per call): the caller asks for it on the whole-stack plan only.
    g.prefetch_tiles = prefetch ? 2 : 0;
    // as many 32 KB stages as fit, split between the K ring (short-lived tiles) and the V ring
    int total_stages = 0;
    for (int st = 9; st >= 2; --st) {
        g.sk = 1; g.sv = st - 1;
        if (tc_smem_layout(g, G).total + 1024 <= max_smem) { total_stages = st; break; }
    }
    if (total_stages < 2) {
        snprintf(err, err_len, "tensor-core kernel: shared memory does not fit");
        delete p;
        return cudaErrorInvalidConfiguration;
    }
    g.sk = total_stages >= 7 ? 3 : total_stages >= 5 ? 2 : 1;
    if (g.nc > 1 && total_stages >= 4) g.sk = 2;      // most items of a chunked window read K only
    g.sv = total_stages - g.sk;
    g.smem_bytes = tc_smem_layout(g, G).total + 1024;
    if (!encode_map(&p->tmK, a.K, a.U, a.cap, kTile) || !encode_map(&p->tmV, a.V, a.U, a.cap, kTile) ||
        !encode_map(&p->tmQ, a.ring_q, a.U, a.R * G, g.qbox)) {
        snprintf(err, err_len, "tensor-core kernel: cuTensorMapEncodeTiled failed");
        delete p;
        return cudaErrorInvalidValue;
    }
    *out = p;
    return cudaSuccess;
}

void tc_plan_destroy(TcPlan *plan) { delete plan; }

cudaError_t launch_decode_tc(TcPlan *plan, const DecodeArgs &a, cudaStream_t stream)
{
    switch (a.G) {
        case 1: return tc_launch_group<1>(plan, a, stream);
        case 2: return tc_launch_group<2>(plan, a, stream);
        case 4: return tc_launch_group<4>(plan, a, stream);
        case 8: return tc_launch_group<8>(plan, a, stream);
        case 16: return tc_launch_group<16>(plan, a, stream);
    }
    return cudaErrorInvalidValue;
}

}  // namespace mkv
