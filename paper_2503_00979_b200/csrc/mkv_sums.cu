// The window sums of the cached slots (DecodeArgs::slab, pre) from the arena as it stands.
//
// window_sums_tc_kernel ends the prompt phase of the tensor-core contexts with more than 256 ring rows (gather_sums_tc_kernel
// takes the others): every key is scored against all ring rows,
// block by block from the last block of the ring to the first, so that the sums of the last lap's blocks accumulate in
// a register on the way.  It has the decode kernel's orientation (keys in the TMEM lanes, ring rows as the N operand,
// up to 256 at a time) and the CTA layout of the prompt phase's scoring passes: warps 0-3 and 6-9 are two consumer
// groups on alternate key tiles and accumulator buffers, warp 4 feeds K tiles with TMA, warp 5 issues the MMAs.
// Bound by the kept keys' bytes and R*G exponentials per key (256 units of 2032 slots, 128 rows: 44 us).
#include <string.h>

#include "mkv_common.cuh"
#include "mkv_kernels.h"
#include "mkv_sm100.cuh"

namespace mkv {

namespace {

constexpr int kSumThreads = 320;
constexpr int kSumGroups = 2;
constexpr int kSumMaxRows = 2048;            // ring rows of one launch: their normalisers sit in shared memory
enum SumWait { kSumKEmpty = 31, kSumKFull, kSumTEmpty, kSumTFull, kSumDrain };

struct SumArgs {
    DecodeArgs d;
    long long t;              // the sums are those the step at position t finds
    int n;
    int set_states;           // step states at d.st to set to (t, n)
    int *err;
    int row0, rows;           // ring rows of this launch (whole blocks; the launches of a wide window go from the last
    int last;                 // rows to the first, and the last one leaves sum_pos)
    int piece;                // rows of one MMA operand
    int splits;               // CTAs per unit along the keys
    int tmem_cols, stages;
    long long wait_cycles;
};

__device__ __forceinline__ void set_states(const SumArgs &a)
{
    for (int i = threadIdx.x; i < a.set_states; i += blockDim.x) {
        DevState *s = a.d.st + i;
        s->t = a.t; s->n = a.n; s->steps = 0; s->err = 0; s->done = 0; s->compact = 0;
    }
}

template <int G, int FUSION>
__global__ void __launch_bounds__(kSumThreads, 2)
window_sums_tc_kernel(const __grid_constant__ SumArgs a, const __grid_constant__ CUtensorMap tmK)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const DecodeArgs &d = a.d;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int sp = blockIdx.x, u = blockIdx.y;
    const int PR = a.piece, ST = a.stages;
    const uint32_t sbase = smem_u32(smem);
    const uint32_t q_addr = sbase, kst_addr = sbase + PR * 256;
    float *negc = reinterpret_cast<float *>(smem + PR * 256 + ST * kStageBytes);        // [kSumMaxRows]
    uint64_t *bars = reinterpret_cast<uint64_t *>(negc + kSumMaxRows);
    const uint32_t bar_kfull = smem_u32(bars), bar_kempty = smem_u32(bars + 4);
    const uint32_t bar_tfull = smem_u32(bars + 8), bar_tempty = smem_u32(bars + 10);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 12);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(bars + 13);
    const long long WL = a.wait_cycles;

    const int n = a.n, nt = (n + kTile - 1) / kTile, per = (nt + a.splits - 1) / a.splits;
    const int t0 = sp * per, t1 = min(nt, t0 + per), ntile = max(0, t1 - t0);
    chain_wait();
    if (sp == 0 && u == 0) set_states(a);
    const int blk_rows = d.bs * G, RG = d.R * G, open = open_block(a.t, d.R, d.bs);
    const int npiece = (a.rows + PR - 1) / PR;

    if (tid == 0) {
        prefetch_tensormap(&tmK);
        for (int s = 0; s < ST; ++s) { mbar_init(bar_kfull + 8 * s, 1); mbar_init(bar_kempty + 8 * s, 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(bar_tfull + 8 * b, 1); mbar_init(bar_tempty + 8 * b, 4); }
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 5) tmem_alloc(smem_u32(tmem_slot), (uint32_t)a.tmem_cols);
    for (int i = tid; i < kSumMaxRows; i += kSumThreads) {
        const int row = a.row0 + i;
        negc[i] = i < a.rows && row < RG ? -d.ring_c[(size_t)u * RG + row] : -INFINITY;     // empty and padding rows: weight 0
    }

    int done = 0;               // tiles of the pieces before this one
    for (int pc = npiece - 1; pc >= 0; --pc, done += ntile) {
        // the piece's ring rows, K-major with the 128-byte swizzle (two 64-column panels of PR rows)
        const int r0 = a.row0 + pc * PR, rn = min(PR, a.rows - pc * PR);
        for (int c = tid; c < PR * 16; c += kSumThreads) {
            const int row = c >> 4, ch = c & 15;
            uint4 v = make_uint4(0, 0, 0, 0);
            if (row < rn && r0 + row < RG)
                v = reinterpret_cast<const uint4 *>(static_cast<const __nv_bfloat16 *>(d.ring_q) + ((size_t)u * RG + r0 + row) * kD)[ch];
            *reinterpret_cast<uint4 *>(smem + (uint32_t)((ch >> 3) * (PR * 128) + row * 128 + (((ch & 7) ^ (row & 7)) << 4))) = v;
        }
        fence_proxy_async();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        const uint32_t tmem_base = *tmem_slot;
        bool ok = true;
        if (warp == 4) {
            // ------------------------------------------------ TMA producer of K tiles (one lane)
            if (lane == 0) {
                const uint64_t pol = l2_policy_evict_first();
                int issued = done;
                for (int j = done; j < done + ntile && ok; ++j) {
                    const int s = j % ST;
                    ok = mbar_wait(bar_kempty + 8 * s, (uint32_t)(((j / ST) & 1) ^ 1), abort_flag, kSumKEmpty, WL);
                    if (!ok) break;
                    const int row = (t0 + j - done) * kTile;
                    mbar_expect_tx(bar_kfull + 8 * s, kStageBytes);
                    tma_load_3d(kst_addr + s * kStageBytes, &tmK, 0, row, u, bar_kfull + 8 * s, pol);
                    tma_load_3d(kst_addr + s * kStageBytes + kStageBytes / 2, &tmK, 64, row, u, bar_kfull + 8 * s, pol);
                    issued = j + 1;
                }
                if (!ok) {      // let the copies in flight land before the CTA exits
                    int dummy = 0;
                    for (int j = max(done, issued - ST); j < issued; ++j)
                        mbar_wait(bar_kfull + 8 * (j % ST), (uint32_t)((j / ST) & 1), &dummy, kSumDrain, kWaitCycles);
                }
            }
            __syncwarp();
        } else if (warp == 5) {
            // ------------------------------------------------ MMA issue: D[128 keys x rows] = K_tile . Q^T
            const int np = (rn + 31) & ~31;
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTile >> 4) << 24) | ((uint32_t)(np >> 3) << 17);
            int j = done;
            for (; j < done + ntile; ++j) {
                const int s = j % ST, b = j & 1;
                bool k = mbar_wait(bar_kfull + 8 * s, (uint32_t)((j / ST) & 1), abort_flag, kSumKFull, WL);
                k = k && mbar_wait(bar_tempty + 8 * b, (uint32_t)(((j >> 1) & 1) ^ 1), abort_flag, kSumTEmpty, WL);
                ok = __all_sync(0xffffffffu, k);
                if (!ok) break;
                tc_fence_after();
                if (elect_one()) {
                    const uint32_t d_tmem = tmem_base + (uint32_t)(b * PR);
#pragma unroll
                    for (int ks = 0; ks < kD / 16; ++ks) {
                        const uint64_t ad = smem_desc_sw128(kst_addr + s * kStageBytes + (ks >> 2) * (kStageBytes / 2) + (ks & 3) * 32);
                        const uint64_t bd = smem_desc_sw128(q_addr + (ks >> 2) * (PR * 128) + (ks & 3) * 32);
                        umma_bf16(d_tmem, ad, bd, idesc, ks > 0 ? 1u : 0u);
                    }
                    umma_commit(bar_kempty + 8 * s);
                    umma_commit(bar_tfull + 8 * b);
                }
                __syncwarp();
            }
            {   // every commit is observed before the operand is overwritten, TMEM is freed or the CTA exits
                int dummy = 0;
                for (int i = max(done, j - ST); i < j; ++i)
                    mbar_wait(bar_kempty + 8 * (i % ST), (uint32_t)((i / ST) & 1), &dummy, kSumDrain, kWaitCycles);
                if (!ok)
                    for (int i = max(done, j - 2); i < j; ++i)
                        mbar_wait(bar_tfull + 8 * (i & 1), (uint32_t)((i >> 1) & 1), &dummy, kSumDrain, kWaitCycles);
                __syncwarp();
            }
        } else {
            // ------------------------------------------------ consumers: one key per thread; group g takes the tiles
            // whose running number has its parity (= accumulator buffer g)
            const int grp = warp < 4 ? 0 : 1, lq = (warp & 3) * 32 + lane;
            const uint32_t tlane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(grp * PR);
            const int jtop = (r0 + rn) / blk_rows;                       // block behind this piece's last one
            const bool top = jtop >= d.nblk;
            for (int j = done + (((done & 1) != grp) ? 1 : 0); j < done + ntile && ok; j += kSumGroups) {
                ok = __all_sync(0xffffffffu, mbar_wait(bar_tfull + 8 * grp, (uint32_t)((j >> 1) & 1), abort_flag, kSumTFull, WL));
                if (!ok) break;
                tc_fence_after();
                const int key = (t0 + j - done) * kTile + lq;
                const bool valid = key < n;
                float *slab = d.slab + (size_t)u * d.nblk * d.cap + key, *prep = d.pre + (size_t)u * d.cap + key;
                float acc = !top && valid && jtop > open ? slab[(size_t)jtop * d.cap] : 0.f;
                float pre = !top && valid ? *prep : 0.f;
                float S = 0.f;
                for (int c = ((rn + 31) & ~31) - 32; c >= 0; c -= 32) {
                    uint32_t v[32];
                    tmem_ld32(tlane + (uint32_t)c, v);
                    score_chunk<G, FUSION>(v, negc + pc * PR + c, d.scale2, S);
                    if (c % blk_rows == 0) {
                        take_block(S, (r0 + c) / blk_rows, open, FUSION, slab, d.cap, valid, acc, pre);
                        S = 0.f;
                        __syncwarp();                        // converged again in front of the aligned TMEM load
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_tempty + 8 * grp);
                if (valid) {
                    *prep = pre;
                    if (a.last && pc == 0) d.sum_pos[(size_t)u * d.cap + key] = d.pos[(size_t)u * d.cap + key];
                }
                __syncwarp();
            }
        }
        tc_fence_before();
        __syncthreads();        // the operand's and the accumulators' readers are done
        tc_fence_after();
        if (*abort_flag) break;
    }
    if (warp == 5) tmem_dealloc(*tmem_slot, (uint32_t)a.tmem_cols);
    if (tid == 0 && *abort_flag) atomicCAS(a.err, 0, *abort_flag);
}

// The gather of the kept rows and the window sums in one pass over them, for windows of one operand (up to 256 ring rows):
// what the gather brings from HBM for the arena is scored on the way.  Persistent CTAs, one per SM, with equal shares of the
// units' tiles.  Warps 10-13 fetch the kept K and V rows of a tile into a stage (cp.async, 16-byte chunks at their swizzled
// places; free slots as zeros: the decode kernels read whole tiles and mask afterwards, so a row must hold finite numbers),
// warp 4 stores the stage to the arena with TMA, warp 5 issues the MMAs, and the two consumer groups are those of the
// kernel above; they load the ring's rows whenever the unit changes, while the stages behind them fill.
// Bound by HBM: 266 MB read and written for 256 units of 2032 slots.  As a gather, 81 us, and a second pass over the arena
// for the sums, 44 us, it took 125 us, now 95.
struct GatherArgs {
    SumArgs s;
    const __nv_bfloat16 *k, *v;  // [U][Ps][128] prompt
    int P, Ps;                   // tokens of the longest prompt, of a unit as laid out
    RowMap rowmap;
};
constexpr int kGsThreads = 448;
constexpr int kGsStage = 2 * kStageBytes;      // K and V
constexpr int kGsFetch = 128;                  // fetching threads
enum GsWait { kGsEmpty = 41, kGsFull, kGsTEmpty, kGsTFull, kGsQFull, kGsDrain };

template <int G, int FUSION>
__global__ void __launch_bounds__(kGsThreads, 1)
gather_sums_tc_kernel(const __grid_constant__ GatherArgs ga, const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const SumArgs &a = ga.s;
    const DecodeArgs &d = a.d;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int PR = a.piece, ST = a.stages;
    const uint32_t q_addr = smem_u32(smem), st_addr = q_addr + PR * 256;
    float *negc = reinterpret_cast<float *>(smem + PR * 256 + ST * kGsStage);           // [256]
    uint64_t *bars = reinterpret_cast<uint64_t *>(negc + 256);
    const uint32_t bar_full = smem_u32(bars), bar_empty = smem_u32(bars + 4);
    const uint32_t bar_tfull = smem_u32(bars + 8), bar_tempty = smem_u32(bars + 10), bar_qfull = smem_u32(bars + 12);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 13);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(bars + 14);
    const long long WL = a.wait_cycles;

    const int nt = (d.cap + kTile - 1) / kTile;                // tiles per unit, the free slots' among them
    const long long total = (long long)d.U * nt;
    const long long i0 = total * blockIdx.x / gridDim.x, i1 = total * (blockIdx.x + 1) / gridDim.x;
    const int ntile = (int)(i1 - i0), u0 = (int)(i0 / nt), t0 = (int)(i0 % nt);

    if (tid == 0) {
        prefetch_tensormap(&tmK);
        prefetch_tensormap(&tmV);
        for (int s = 0; s < ST; ++s) { mbar_init(bar_full + 8 * s, kGsFetch); mbar_init(bar_empty + 8 * s, 2); }
        for (int b = 0; b < 2; ++b) { mbar_init(bar_tfull + 8 * b, 1); mbar_init(bar_tempty + 8 * b, 4); }
        mbar_init(bar_qfull, 8);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 5) tmem_alloc(smem_u32(tmem_slot), (uint32_t)a.tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    chain_wait();

    if (warp >= 10) {
        // ------------------------------------------------ fetch: a warp takes 32 rows of a tile, half a warp a row
        const int w = warp - 10, half = lane >> 4, ch = lane & 15;
        int u = u0, t = t0;
        bool ok = true;
        auto position = [&](int uu, int tt) -> int {           // of this lane's row
            const int slot = tt * kTile + w * 32 + lane;
            const int P = ga.P - ga.rowmap(uu), n = min(P, d.C + min(P, d.R));
            return slot < n ? d.pos[(size_t)uu * d.cap + slot] : -1;
        };
        int p = ntile > 0 ? position(u, t) : -1;
        int j = 0;
        for (; j < ntile; ++j) {
            const int s = j % ST;
            const int un = t + 1 == nt ? u + 1 : u, tn = t + 1 == nt ? 0 : t + 1;
            const int p_next = j + 1 < ntile ? position(un, tn) : -1;
            ok = __all_sync(0xffffffffu, mbar_wait(bar_empty + 8 * s, (uint32_t)(((j / ST) & 1) ^ 1), abort_flag, kGsEmpty, WL));
            if (!ok) break;
            const __nv_bfloat16 *ku = ga.k + (size_t)u * ga.Ps * kD + ch * 8, *vu = ga.v + (size_t)u * ga.Ps * kD + ch * 8;
            const uint32_t dst = st_addr + s * kGsStage + (ch >> 3) * (kStageBytes / 2);
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const int r = 2 * i + half, row = w * 32 + r;
                const int pr = __shfl_sync(0xffffffffu, p, r);
                const uint32_t off = dst + row * 128 + (((ch & 7) ^ (row & 7)) << 4);
                const size_t at = (size_t)max(pr, 0) * kD;
                const int bytes = pr >= 0 ? 16 : 0;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(off), "l"(ku + at), "r"(bytes) : "memory");
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(off + kStageBytes), "l"(vu + at), "r"(bytes) : "memory");
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
            if (j > 0) {                                       // the tile before has landed
                asm volatile("cp.async.wait_group 1;" ::: "memory");
                fence_proxy_async();
                mbar_arrive(bar_full + 8 * ((j - 1) % ST));
            }
            u = un; t = tn; p = p_next;
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        if (ok && ntile > 0) {
            fence_proxy_async();
            mbar_arrive(bar_full + 8 * ((ntile - 1) % ST));
        }
    } else if (warp == 4) {
        // ------------------------------------------------ stores to the arena (one lane)
        if (lane == 0) {
            int u = u0, t = t0;
            for (int j = 0; j < ntile; ++j) {
                const int s = j % ST;
                if (!mbar_wait(bar_full + 8 * s, (uint32_t)((j / ST) & 1), abort_flag, kGsFull, WL)) break;
                const uint32_t src = st_addr + s * kGsStage;
                tma_store_3d(&tmK, src, 0, t * kTile, u);
                tma_store_3d(&tmK, src + kStageBytes / 2, 64, t * kTile, u);
                tma_store_3d(&tmV, src + kStageBytes, 0, t * kTile, u);
                tma_store_3d(&tmV, src + kStageBytes + kStageBytes / 2, 64, t * kTile, u);
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                mbar_arrive(bar_empty + 8 * s);
                if (++t == nt) { t = 0; ++u; }
            }
            asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        }
        __syncwarp();
    } else if (warp == 5) {
        // ------------------------------------------------ MMA issue: D[128 keys x rows] = K_tile . Q^T
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTile >> 4) << 24) | ((uint32_t)(PR >> 3) << 17);
        bool ok = true;
        int j = 0, t = t0, runs = 0;
        for (; j < ntile; ++j) {
            const int s = j % ST, b = j & 1;
            bool k = true;
            if (j == 0 || t == 0) k = mbar_wait(bar_qfull, (uint32_t)(runs++ & 1), abort_flag, kGsQFull, WL);
            k = k && mbar_wait(bar_full + 8 * s, (uint32_t)((j / ST) & 1), abort_flag, kGsFull, WL);
            k = k && mbar_wait(bar_tempty + 8 * b, (uint32_t)(((j >> 1) & 1) ^ 1), abort_flag, kGsTEmpty, WL);
            ok = __all_sync(0xffffffffu, k);
            if (!ok) break;
            tc_fence_after();
            if (elect_one()) {
                const uint32_t d_tmem = tmem_base + (uint32_t)(b * PR);
#pragma unroll
                for (int ks = 0; ks < kD / 16; ++ks) {
                    const uint64_t ad = smem_desc_sw128(st_addr + s * kGsStage + (ks >> 2) * (kStageBytes / 2) + (ks & 3) * 32);
                    const uint64_t bd = smem_desc_sw128(q_addr + (ks >> 2) * (PR * 128) + (ks & 3) * 32);
                    umma_bf16(d_tmem, ad, bd, idesc, ks > 0 ? 1u : 0u);
                }
                umma_commit(bar_empty + 8 * s);
                umma_commit(bar_tfull + 8 * b);
            }
            __syncwarp();
            if (++t == nt) t = 0;
        }
        {   // every commit is observed before TMEM is freed and the CTA exits
            int dummy = 0;
            for (int i = max(0, j - ST); i < j; ++i)
                mbar_wait(bar_empty + 8 * (i % ST), (uint32_t)((i / ST) & 1), &dummy, kGsDrain, kWaitCycles);
            if (!ok)
                for (int i = max(0, j - 2); i < j; ++i)
                    mbar_wait(bar_tfull + 8 * (i & 1), (uint32_t)((i >> 1) & 1), &dummy, kGsDrain, kWaitCycles);
            __syncwarp();
        }
    } else {
        // ------------------------------------------------ consumers: one key per thread, groups on alternate tiles
        constexpr int kBar = 1, kN = 256;
        const int grp = warp < 4 ? 0 : 1, ct = warp < 4 ? tid : tid - 64, lq = (warp & 3) * 32 + lane;
        const uint32_t tlane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(grp * PR);
        const int blk_rows = d.bs * G, RG = d.R * G, open = open_block(a.t, d.R, d.bs);
        bool ok = true;
        int u = u0, t = t0;
        for (int j0 = 0; j0 < ntile; ++u, t = 0) {
            const int j1 = min(ntile, j0 + nt - t);            // tiles of this unit
            // every accumulator of the unit before has been read, so its MMAs are done with the operand
            if (group_any<kN>(kBar, !ok)) break;
            for (int c0 = ct; c0 < PR * 16; c0 += 8 * kN) {
                uint4 v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int c = c0 + i * kN, row = c >> 4;
                    v[i] = row < RG && row < PR ? reinterpret_cast<const uint4 *>(static_cast<const __nv_bfloat16 *>(d.ring_q) + ((size_t)u * RG + row) * kD)[c & 15]
                                                : make_uint4(0, 0, 0, 0);
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int c = c0 + i * kN, row = c >> 4, ch = c & 15;
                    if (row < PR) *reinterpret_cast<uint4 *>(smem + (ch >> 3) * (PR * 128) + row * 128 + (((ch & 7) ^ (row & 7)) << 4)) = v[i];
                }
            }
            negc[ct] = ct < RG ? -d.ring_c[(size_t)u * RG + ct] : -INFINITY;         // empty and padding rows: weight 0
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_qfull);
            group_sync(kBar, kN);
            for (int j = j0 + ((j0 & 1) ^ grp); j < j1 && ok; j += 2) {
                const int key = (t + j - j0) * kTile + lq;
                const bool valid = key < a.n;
                const int p = valid ? d.pos[(size_t)u * d.cap + key] : 0;
                ok = __all_sync(0xffffffffu, mbar_wait(bar_tfull + 8 * grp, (uint32_t)((j >> 1) & 1), abort_flag, kGsTFull, WL));
                if (!ok) break;
                tc_fence_after();
                float *slab = d.slab + (size_t)u * d.nblk * d.cap + key;
                float acc = 0.f, pre = 0.f, S = 0.f;
                for (int c = PR - 32; c >= 0; c -= 32) {
                    uint32_t v[32];
                    tmem_ld32(tlane + (uint32_t)c, v);
                    score_chunk<G, FUSION>(v, negc + c, d.scale2, S);
                    if (c % blk_rows == 0) {
                        take_block(S, c / blk_rows, open, FUSION, slab, d.cap, valid, acc, pre);
                        S = 0.f;
                        __syncwarp();                        // converged again in front of the aligned TMEM load
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_tempty + 8 * grp);
                if (valid) {
                    d.pre[(size_t)u * d.cap + key] = pre;
                    d.sum_pos[(size_t)u * d.cap + key] = p;
                }
                __syncwarp();
            }
            j0 = j1;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 5) {
        tc_fence_after();
        tmem_dealloc(tmem_base, (uint32_t)a.tmem_cols);
    }
    if (tid == 0 && *abort_flag) atomicCAS(a.err, 0, *abort_flag);
}

template <int G>
cudaError_t launch_gather_g(const GatherArgs &a, const CUtensorMap &tmK, const CUtensorMap &tmV, cudaStream_t stream)
{
    const SumArgs &s = a.s;
    auto kern = s.d.fusion == kFusionSum ? gather_sums_tc_kernel<G, kFusionSum> : gather_sums_tc_kernel<G, kFusionMax>;
    const int smem = s.piece * 256 + s.stages * kGsStage + 256 * 4 + 256 + 1024;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    const long long tiles = (long long)s.d.U * ((s.d.cap + kTile - 1) / kTile);
    return launch_chained(kern, dim3((unsigned)(tiles < 148 ? tiles : 148)), kGsThreads, smem, stream, a, tmK, tmV);
}

__global__ void set_states_kernel(const __grid_constant__ SumArgs a)
{
    chain_wait();
    set_states(a);
}

template <int G>
cudaError_t launch_sums_g(const SumArgs &a, const CUtensorMap &tm, cudaStream_t stream)
{
    auto kern = a.d.fusion == kFusionSum ? window_sums_tc_kernel<G, kFusionSum> : window_sums_tc_kernel<G, kFusionMax>;
    const int smem = a.piece * 256 + a.stages * kStageBytes + kSumMaxRows * 4 + 256 + 1024;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    return launch_chained(kern, dim3(a.splits, a.d.U), kSumThreads, smem, stream, a, tm);
}

// `d` for a launch over its units u0 .. u0 + count - 1 (grid.y takes 65535 units at most)
DecodeArgs unit_range(const DecodeArgs &d, int D, size_t es, int u0, int count)
{
    DecodeArgs p = d;
    const size_t u = u0;
    p.U = count;
    p.K = static_cast<char *>(d.K) + u * d.cap * D * es;
    p.ring_q = static_cast<char *>(d.ring_q) + u * d.R * d.G * D * es;
    p.ring_c += u * d.R * d.G;
    p.pos += u * d.cap; p.sum_pos += u * d.cap; p.pre += u * d.cap;
    p.slab += u * d.nblk * d.cap;
    return p;
}
constexpr int kMaxGridY = 65535;

// CTAs per unit along the keys.  A CTA pays a set-up (TMEM, barriers, the ring's rows into shared memory) worth about
// `kSetupTiles` key tiles, and the grid runs in waves of `slots` resident CTAs: the split with the fewest tile-times over all waves.
int sums_splits(int units, int n, int rows)
{
    constexpr int kSetupTiles = 3;
    const int nt = (n + kTile - 1) / kTile;
    const int slots = 148 * (rows <= 128 ? 2 : 1);
    int best = 1;
    long long best_cost = -1;
    for (int s = 1; s <= nt && s <= 64; ++s) {
        const long long waves = ((long long)units * s + slots - 1) / slots;
        const long long cost = waves * ((nt + s - 1) / s + kSetupTiles);
        if (best_cost < 0 || cost < best_cost) { best_cost = cost; best = s; }
    }
    return best;
}

}  // namespace

bool gather_sums_supported(const DecodeArgs &d, const void *k, const void *v)
{
    return d.nblk > 1 && d.nblk * d.bs * d.G <= 256 && ((uintptr_t)k & 15) == 0 && ((uintptr_t)v & 15) == 0;
}

cudaError_t launch_gather_sums(const DecodeArgs &d, const void *k, const void *v, int P, int Ps, int n, int *err, cudaStream_t stream)
{
    GatherArgs g;
    memset(&g, 0, sizeof(g));
    SumArgs &a = g.s;
    a.d = d;
    a.t = P; a.n = n; a.err = err;
    a.wait_cycles = kWaitCycles;
    a.piece = d.nblk * d.bs * d.G;
    a.stages = a.piece <= 128 ? 3 : 2;
    a.tmem_cols = 32;
    while (a.tmem_cols < 2 * a.piece) a.tmem_cols *= 2;
    g.k = static_cast<const __nv_bfloat16 *>(k); g.v = static_cast<const __nv_bfloat16 *>(v);
    g.P = P; g.Ps = Ps; g.rowmap = {d.row_shift, d.Hkv, d.B};
    CUtensorMap tmK, tmV;
    if (!encode_map(&tmK, d.K, d.U, d.cap, kTile) || !encode_map(&tmV, d.V, d.U, d.cap, kTile)) return cudaErrorInvalidValue;
    switch (d.G) {
        case 1: return launch_gather_g<1>(g, tmK, tmV, stream);
        case 2: return launch_gather_g<2>(g, tmK, tmV, stream);
        case 4: return launch_gather_g<4>(g, tmK, tmV, stream);
        case 8: return launch_gather_g<8>(g, tmK, tmV, stream);
        case 16: return launch_gather_g<16>(g, tmK, tmV, stream);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_finish_prompt(const DecodeArgs &d, bool sums, long long t, int n, int n_states, int *err, unsigned long long *launches,
                                 cudaStream_t stream)
{
    SumArgs a;
    memset(&a, 0, sizeof(a));
    a.d = d;
    a.t = t; a.n = n; a.err = err;
    a.wait_cycles = kWaitCycles;
    if (d.nblk <= 1 || !sums) {
        a.set_states = n_states;
        ++*launches;
        return launch_chained(set_states_kernel, dim3(1), 32, 0, stream, a);
    }
    const int blk_rows = d.bs * d.G, all = d.nblk * blk_rows;
    a.piece = min(all, 256 / blk_rows * blk_rows);
    a.stages = a.piece <= 128 ? 2 : 3;
    a.tmem_cols = 32;
    while (a.tmem_cols < 2 * a.piece) a.tmem_cols *= 2;
    const int chunk = kSumMaxRows / a.piece * a.piece;
    for (int u0 = 0; u0 < d.U; u0 += kMaxGridY) {
        a.d = unit_range(d, kD, 2, u0, min(kMaxGridY, d.U - u0));
        a.splits = sums_splits(a.d.U, n, a.piece);
        CUtensorMap tm;
        if (!encode_map(&tm, a.d.K, a.d.U, d.cap, kTile)) return cudaErrorInvalidValue;
        for (int row0 = (all - 1) / chunk * chunk; row0 >= 0; row0 -= chunk) {
            a.row0 = row0;
            a.rows = min(chunk, all - row0);
            a.last = row0 == 0;
            a.set_states = a.last && u0 + a.d.U == d.U ? n_states : 0;
            cudaError_t e;
            switch (d.G) {
                case 1: e = launch_sums_g<1>(a, tm, stream); break;
                case 2: e = launch_sums_g<2>(a, tm, stream); break;
                case 4: e = launch_sums_g<4>(a, tm, stream); break;
                case 8: e = launch_sums_g<8>(a, tm, stream); break;
                case 16: e = launch_sums_g<16>(a, tm, stream); break;
                default: e = cudaErrorInvalidValue;
            }
            ++*launches;
            if (e != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

}  // namespace mkv
