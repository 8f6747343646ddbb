// Prompt-phase scoring on the tensor cores (bf16, head_dim 128, GQA group in {1,2,4,8,16}; a window of more than 256
// rows R*G is scored in pieces of up to 256 rows, one launch per piece, the pieces' scores fused in place).
//
// One application of Algorithm 1 to the whole prompt needs, for every older prompt token k, the fused score
// F[k] = sum_r / max_r of S_r[k], S_r[k] = sum over the GQA group of the causal soft-max weight window row r puts
// on k (Eq. 1, Eq. 4-6).  The weights need each row's soft-max normaliser over ALL prompt keys first, so the keys
// are visited twice and nothing of size rows x P ever goes to global memory:
//   statistics  logits[rows x keys] = Qwin . K_tile^T on tcgen05 with the window rows in the TMEM lanes: every thread
//               owns one row and keeps its running (reference, sum) over the keys it may see (causal inside the window).
//   scores      logits^T[keys x rows] = K_tile . Qwin^T with the keys in the lanes (the decode kernel's orientation):
//               every thread owns one key, turns its row of logits into weights exp2(s - c_row), sums them over the
//               group and fuses them over the window; F[k] is written for the candidates (P floats per unit).
//
// One launch does both where the keys are too many to stay in L2 by themselves (prompt_apart_tiles), so that the second visit of a key
// finds it there: its persistent CTAs take items, each a visit of one kind to a run of a unit's key tiles, from one sequence in which the
// scores of a run follow its statistics `lag` runs later - late enough for all of its unit's statistics to be there, early enough for the
// runs in between (some 60 MB, and a unit's own keys) to stay in the 126 MB L2.  Items are handed out by a ticket, in order: an item waits
// only for items that running CTAs hold, so no number of resident CTAs is needed.  The CTA that completes a unit's statistics merges them
// into the normalisers and raises the unit's flag.  Otherwise each visit has a launch, whose items wait for nothing and are every
// CTA's own, and the items of the second merge their unit's statistics.
//
// CTA layout: warp 0 takes the tickets and feeds queries and K tiles with TMA; warps 1 and 3 issue the MMAs into the TMEM
// accumulator buffers; warp 2 waits for the units' flags and fetches their normalisers, ahead of the items that need them;
// warps 4-7 publish statistics; warps 8-23 are four consumer groups (one TMEM lane quarter per warp), to which tiles go in
// turn (with more than 128 window rows to pairs of them, each of which takes half of the rows).  The item descriptors, queries
// (two buffers), K tiles, normalisers and statistics pass through rings of their own, so that nothing drains between items.
// Every wait is bounded; a wait that runs out raises an error word that the host reads after the call.
//
// What bounds it: the MUFU's exponentials, two per key and row: 2048 cycles of a tile's two visits with 128 rows, of 3290 taken for 256
// units x 6144 tokens (159 us at 1.70 GHz: MUFU 73 % busy, tensor pipe 31 %, 441 MB from HBM of which the keys are 403); prompt after
// prompt also the 1000 W of the card (256 x 131072: 3236 us at 1965 MHz, 3717 at 1500 after a second of it).  A launch for each visit is bound by the
// same and by the start of a launch that needs whole SMs: up to two tiles per unit take 3 to 8 us longer than with smaller CTAs, two to an SM.
// Prompt phase in us, one pass of launches over the keys per visit -> now (L2 flushed): 256 units x 6144 tokens, 128 rows, 304 -> 288;
// 64 x 32768, 256 rows, 528 -> 485; 128 x 12291, 800 rows in pieces, 1341 -> 1226; 256 x 131072 3259 -> 3254;
// 112 x 560 91 -> 75.  Taken back: every fourth exponential as a polynomial on the FMA pipe (6144: 285 us cold, but 131072 3850 -> 3910:
// more power); keys kept with evict_last, or without a policy at the second visit (no change, 131072 up to 15 % slower); a row's maximum
// only where a chunk's sum shows that the reference is far below it (no faster, and the exponents of the weights that count rounded coarsely).
#include <stdio.h>

#include <algorithm>

#include "mkv_common.cuh"
#include "mkv_kernels.h"
#include "mkv_schedule.h"
#include "mkv_sm100.cuh"

namespace mkv {

namespace {

constexpr int kPfGroups = 4;                 // consumer groups of four warps
constexpr int kPfFirstConsumer = 8, kPfFirstPublisher = 4;
constexpr int kPfThreads = 32 * (kPfFirstConsumer + 4 * kPfGroups);
constexpr int kPfDesc = 4;                   // item descriptors in flight
constexpr int kPfMerge = 16;                 // statistics merged at a time
enum PfWait { kPfKEmpty = 21, kPfKFull, kPfTEmpty, kPfTFull, kPfDrain, kPfDEmpty, kPfDFull, kPfQEmpty, kPfQFull, kPfNEmpty, kPfNFull,
              kPfSEmpty, kPfSFull, kPfFlag, kPfPair };

// Rows of different lengths go through the same launches (rowmap); a unit has the runs of its own prompt.
struct PfArgs {
    float *part_ml;              // [nb][runs][qrows][2] (max, sum) of a run per window row, log2 domain
    float *ring_c;               // [U][R][G] arena: normaliser of the row of position p in ring slot p % R
    float *Fp;                   // [nb][P] fused scores of the batch's units
    int *done, *flag;            // [nb][1 + clusters of runs] statistics that are there; [nb] 1: the unit's normalisers are in ring_c
    int *ticket, *left;          // next item; CTAs that have finished.  All zero between launches
    int *err;                    // error word (0 = none)
    int ub0, nb;                 // units of this batch
    int P, R, G, C;              // P: tokens of the longest prompt
    RowMap rowmap;               // how much shorter a unit's prompt is
    int Gq;                      // real heads per unit; heads Gq .. G-1 are padding (zero query)
    int rows;                    // window rows of this launch (a unit with a shorter window has fewer); row = (window
                                 // slot - i0) * G + head
    int held;                    // rows of this launch that the window tensor holds (more if it is padded)
    int i0;                      // first window slot of this launch (a wide window is scored piece by piece)
    int accumulate;              // fuse the scores into Fp (a later piece) instead of writing them
    int qrows;                   // rows padded to a multiple of 128 (statistics: MMA M blocks)
    int rpad;                    // rows padded to a multiple of 32 (scores: MMA N)
    int run, runs;               // tiles of a run, runs of the longest prompt
    RunOrder order;              // of the batch's units' runs (order.shift: in this device's memory)
    int items, lag;              // runs of the batch's units, distance of a run's two visits in runs
    int select;                  // 0: nothing has to be selected, the normalisers are all there is to do
    int visit;                   // 0: both visits in this launch; 1, 2: one of them
    int stages, bufs;            // K stages, TMEM accumulator buffers (as many as fit 512 columns)
    float scale2;
    long long wait_cycles;
};

struct PfItem { int kind, ul, tile0, ntile; };        // kind: 0 none left, 1 statistics, 2 scores

struct PfSmem { int q, kst, negc, stat, pair, desc, bars, table, total; };
__host__ __device__ inline PfSmem pf_smem(int qrows, int stages)
{
    PfSmem L;
    int o = 0;
    L.q = o; o += 2 * qrows * 256;
    L.kst = o; o += stages * kStageBytes;
    L.negc = o; o += 2 * 256 * 4;                              // two items' negated normalisers
    L.stat = o; o += 2 * 512 * 8;                              // two items' (max, sum) per accumulator column
    L.pair = o; o += 2 * 128 * 4;                              // scores over the rows from 128 on, of two buffers' keys
    L.desc = o; o += kPfDesc * 16;
    L.bars = o; o += 512;
    L.table = o; o += (kRunTable + 1) * 4;
    L.total = o;
    return L;
}

// The t-th item of the launch.
__device__ __forceinline__ RunVisit pf_item(const PfArgs &a, int t)
{
    if (a.visit != 0 || !a.select) return RunVisit{a.visit == 2 ? 2 : 1, t, t < a.items};
    return prompt_item(t, a.items, a.lag);
}

// The next ticket, or `own`.  (One predicated instruction: with a branch around atomicAdd its result was waited for at once, 2 to 7 % of
// the prompt phase: 448 units x 66 tokens 91 -> 98 us, 256 x 9000 306 -> 312.)
__device__ __forceinline__ int take_ticket(int *count, bool tickets, int own)
{
    int t = own;
    asm volatile("{\n.reg .pred p;\nsetp.ne.s32 p, %2, 0;\n@p atom.global.add.s32 %0, [%1], 1;\n}" : "+r"(t) : "l"(count), "r"((int)tickets) : "memory");
    return t;
}

// Waits for the flag that another CTA raises; bounded like mbar_wait.
__device__ __noinline__ bool pf_flag_wait(const int *flag, volatile int *abort, long long limit)
{
    const long long t0 = clock64();
    for (;;) {
        int v;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
        if (v != 0) return true;
        if (*abort) return false;
        if (clock64() - t0 > limit) { *abort = kPfFlag; return false; }
        __nanosleep(100);
    }
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *map, int x, int y, int z, int w, uint32_t bar, uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
        "[%0], [%1, {%2, %3, %4, %5}], [%6], %7;"
        ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar), "l"(policy) : "memory");
}
__device__ __forceinline__ uint64_t l2_policy_evict_normal()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
    return p;
}


// ---- pairs of floats (f32x2 instructions: half the issue slots)
typedef unsigned long long F32x2;
__device__ __forceinline__ F32x2 pack2(float a, float b) { F32x2 r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b)); return r; }
__device__ __forceinline__ float2 unpack2(F32x2 v) { float2 r; asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v)); return r; }
__device__ __forceinline__ F32x2 fma2(F32x2 a, F32x2 b, F32x2 c) { F32x2 r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }
__device__ __forceinline__ F32x2 add2(F32x2 a, F32x2 b) { F32x2 r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ F32x2 both(float a) { return pack2(a, a); }
__device__ __forceinline__ F32x2 ex2_pair(F32x2 x)
{
    const float2 u = unpack2(x);
    return pack2(ex2f(u.x), ex2f(u.y));
}

// sum over 32 keys of exp2(s * scale2 - m)
__device__ __forceinline__ float sum_chunk(const uint32_t (&v)[32], float scale2, float m)
{
    F32x2 a[2] = {0ull, 0ull};
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const F32x2 s = pack2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
        a[i & 1] = add2(a[i & 1], ex2_pair(fma2(s, both(scale2), both(-m))));
    }
    const float2 t = unpack2(add2(a[0], a[1]));
    return t.x + t.y;
}

// score_chunk of mkv_sm100.cuh in pairs
template <int G, int FUSION>
__device__ __forceinline__ void score_chunk_pairs(const uint32_t (&v)[32], const float *negc, float scale2, float &F)
{
    F32x2 part = 0ull;
#pragma unroll
    for (int j = 0; j < 32; j += 4) {
        const float4 nc = *reinterpret_cast<const float4 *>(negc + j);
        const F32x2 w0 = ex2_pair(fma2(pack2(__uint_as_float(v[j]), __uint_as_float(v[j + 1])), both(scale2), pack2(nc.x, nc.y)));
        const F32x2 w1 = ex2_pair(fma2(pack2(__uint_as_float(v[j + 2]), __uint_as_float(v[j + 3])), both(scale2), pack2(nc.z, nc.w)));
        if (FUSION == kFusionMax && G <= 2) {
            const float2 a = unpack2(w0), b = unpack2(w1);
            F = G == 1 ? fmaxf(fmaxf(F, fmaxf(a.x, a.y)), fmaxf(b.x, b.y)) : fmaxf(F, fmaxf(a.x + a.y, b.x + b.y));
        } else {
            part = add2(part, add2(w0, w1));
            if (FUSION == kFusionMax && (j + 4) % G == 0) {
                const float2 a = unpack2(part);
                F = fmaxf(F, a.x + a.y);
                part = 0ull;
            }
        }
    }
    if (FUSION == kFusionSum) {
        const float2 a = unpack2(part);
        F += a.x + a.y;
    }
}

template <int G, int FUSION>
__global__ void __launch_bounds__(kPfThreads, 1)
prefill_tc_kernel(const __grid_constant__ PfArgs a, const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmQ)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int QR = a.qrows, RB = QR / 128, ST = a.stages, NB = a.bufs;
    const PfSmem L = pf_smem(QR, ST);
    const uint32_t sbase = smem_u32(smem), q_addr = sbase + L.q, kst_addr = sbase + L.kst;
    float *negc_s = reinterpret_cast<float *>(smem + L.negc);              // [2][256]
    float *stat_s = reinterpret_cast<float *>(smem + L.stat);              // [2][NB][QR][2]
    float *pair_s = reinterpret_cast<float *>(smem + L.pair);              // [2][128]
    PfItem *desc = reinterpret_cast<PfItem *>(smem + L.desc);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + L.bars);
    const uint32_t bar_kfull = smem_u32(bars), bar_kempty = smem_u32(bars + 4), bar_tfull = smem_u32(bars + 8), bar_tempty = smem_u32(bars + 12);
    const uint32_t bar_dfull = smem_u32(bars + 16), bar_dempty = smem_u32(bars + 20), bar_qfull = smem_u32(bars + 24), bar_qempty = smem_u32(bars + 26);
    const uint32_t bar_nfull = smem_u32(bars + 28), bar_nempty = smem_u32(bars + 30), bar_sfull = smem_u32(bars + 32), bar_sempty = smem_u32(bars + 34);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 36);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(bars + 37);
    int *last_s = reinterpret_cast<int *>(bars + 38);
    const uint32_t bar_pair = smem_u32(bars + 39);
    int *table = reinterpret_cast<int *>(smem + L.table);                  // RunOrder::place
    const long long WL = a.wait_cycles;

    // a barrier per lane: the launch's start is in the way of the first copies (by thread index, in all warps' code, it cost the consumers
    // three registers and spills)
    if (warp == 0) {
        for (int i = lane; i < 38; i += 32) {
            const int n = i >= 34 ? 4                                   // sempty, pair
                          : i >= 30 ? 4 * kPfGroups                     // nempty, sfull
                          : i >= 28 ? 1                                 // nfull
                          : i >= 26 ? 2                                 // qempty
                          : i >= 24 ? 1                                 // qfull
                          : i >= 20 ? 3 + 4 + 4 * kPfGroups             // dempty: the MMA warps, the normalisers' warp, four publishing and all consumer warps
                          : i >= 16 ? 1                                 // dfull
                          : i >= 12 ? 4 * kPfGroups / NB                // tempty
                                    : 1;                                // tfull, kempty, kfull
            mbar_init(smem_u32(bars) + 8 * (i < 36 ? i : i + 3), (uint32_t)n);
        }
        if (lane == 0) {
            prefetch_tensormap(&tmK);
            prefetch_tensormap(&tmQ);
            *abort_flag = 0;
        }
        fence_barrier_init();
    }
    if (warp == 1) tmem_alloc(smem_u32(tmem_slot), 512);
    // (the rows' lengths were there before the first launch of the chain)
    const int entries = a.order.entries;
    if (entries > 0) {         // (by a warp that has time: ahead of the copying lane's code it slowed that down, 1 to 5 % of a prompt)
        for (int e = tid; e < entries; e += kPfThreads) table[e + 1] = a.order.entry(e);
        __syncthreads();
        if (warp == 2) {
            for (int e0 = 0, sum = 0; e0 < entries; e0 += 32) {
                int v = e0 + lane < entries ? table[e0 + lane + 1] : 0;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int up = __shfl_up_sync(0xffffffffu, v, o);
                    if (lane >= o) v += up;
                }
                if (e0 + lane < entries) table[e0 + lane + 1] = sum + v;
                if (e0 + lane == 0) table[0] = 0;
                sum += __shfl_sync(0xffffffffu, v, 31);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    chain_wait();           // (the prompt is complete: the chain of launches starts behind it in full stream order)

    // the next descriptor, in every role but the producer; `k` counts them
    int k = 0;
    auto take = [&](PfItem &x) -> bool {
        const bool ok = __all_sync(0xffffffffu, mbar_wait(bar_dfull + 8 * (k % kPfDesc), (uint32_t)((k / kPfDesc) & 1), abort_flag, kPfDFull, WL));
        if (!ok) return false;
        x = desc[k % kPfDesc];
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_dempty + 8 * (k % kPfDesc));
        ++k;
        return x.kind != 0;
    };

    if (warp == 0) {
        // ------------------------------------------------ tickets, queries, K tiles (one lane)
        if (lane == 0) {
            // the keys stay in L2 between their two visits, and are not needed there afterwards
            const uint64_t pol_first = l2_policy_evict_normal(), pol_last = l2_policy_evict_first();
            bool ok = true;
            int issued = 0, items = 0, queries = 0;
            // Items are taken by ticket, the next one's on its way while this one is worked on.  In the launches of one visit of two,
            // whose items are few and about as long, a CTA has its own: one that starts early would take two while others get none.  They
            // are one place further on in every round, or the units' shorter last runs could all be the same CTAs'.
            const bool tickets = a.visit == 0;
            int place = (int)blockIdx.x, round0 = 0, ticket = take_ticket(a.ticket, tickets, place);
            while (ok) {
                const int t = ticket;
                place = place + 1 == (int)gridDim.x ? 0 : place + 1;
                round0 += (int)gridDim.x;
                ticket = take_ticket(a.ticket, tickets, round0 + place);
                PfItem x;
                int u = 0;
                const RunVisit v = pf_item(a, t);
                x.kind = v.kind;
                if (v.more) {
                    const RunAt at = a.order.place(v.i, table);
                    const int P = at.P, Rw = min(P, a.R);
                    u = at.unit;
                    x.ul = u - a.ub0;
                    x.tile0 = at.r * a.run;
                    const int nkeys = x.kind == 1 ? P : P - Rw;
                    x.ntile = min(a.run, (nkeys + kTile - 1) / kTile - x.tile0);
                    if (x.kind == 2 && (!a.select || P - Rw <= a.C)) x.ntile = 0;        // a prompt that is kept whole
                    if (x.ntile <= 0) {
                        if (a.visit != 2 || x.tile0 != 0) continue;        // no candidates in the run
                        x.ntile = 0;                                       // (the unit's normalisers are merged)
                    }
                    if (Rw <= a.i0) continue;                              // a piece of the window that the unit does not have
                } else {
                    x.kind = 0;
                }
                const int d = items % kPfDesc;
                ok = mbar_wait(bar_dempty + 8 * d, (uint32_t)(((items / kPfDesc) & 1) ^ 1), abort_flag, kPfDEmpty, WL);
                if (!ok) break;
                desc[d] = x;
                mbar_arrive(bar_dfull + 8 * d);
                ++items;
                if (!v.more) break;
                if (x.ntile == 0) continue;
                const int qs = queries & 1;
                ok = mbar_wait(bar_qempty + 8 * qs, (uint32_t)(((queries >> 1) & 1) ^ 1), abort_flag, kPfQEmpty, WL);
                if (!ok) break;
                // K-major with the 128-byte swizzle the MMA descriptors expect: two 64-column panels of QR rows; heads and window
                // slots that do not exist are zero
                mbar_expect_tx(bar_qfull + 8 * qs, (uint32_t)(QR * 256));
                tma_load_4d(q_addr + qs * QR * 256, &tmQ, 0, 0, a.i0, u, bar_qfull + 8 * qs, pol_first);
                tma_load_4d(q_addr + qs * QR * 256 + QR * 128, &tmQ, 64, 0, a.i0, u, bar_qfull + 8 * qs, pol_first);
                ++queries;
                const uint64_t pol = x.kind == 1 && a.select ? pol_first : pol_last;
                for (int j = 0; j < x.ntile; ++j) {
                    const int s = issued % ST;
                    ok = mbar_wait(bar_kempty + 8 * s, (uint32_t)(((issued / ST) & 1) ^ 1), abort_flag, kPfKEmpty, WL);
                    if (!ok) break;
                    const int row = (x.tile0 + j) * kTile;
                    mbar_expect_tx(bar_kfull + 8 * s, kStageBytes);
                    tma_load_3d(kst_addr + s * kStageBytes, &tmK, 0, row, u, bar_kfull + 8 * s, pol);
                    tma_load_3d(kst_addr + s * kStageBytes + kStageBytes / 2, &tmK, 64, row, u, bar_kfull + 8 * s, pol);
                    ++issued;
                }
            }
            if (!ok) {      // let the copies in flight land before the CTA exits
                int dummy = 0;
                for (int j = max(0, issued - ST); j < issued; ++j)
                    mbar_wait(bar_kfull + 8 * (j % ST), (uint32_t)((j / ST) & 1), &dummy, kPfDrain, kWaitCycles);
                for (int j = max(0, queries - 2); j < queries; ++j)
                    mbar_wait(bar_qfull + 8 * (j & 1), (uint32_t)((j >> 1) & 1), &dummy, kPfDrain, kWaitCycles);
            }
        }
        __syncwarp();
    } else if (warp == 1 || warp == 3) {
        // ------------------------------------------------ MMA issue: the two warps take alternate tiles, as a tile's waits, eight
        // MMAs and commits are a chain of some 1000 cycles.  (One warp, which also made every descriptor from scratch behind
        // `lane == 0`, took 1600 cycles per tile and set the pace: 335 us for 256 units x 6144
        // tokens, 297 now.)
        const int mw = warp >> 1;
        const uint32_t idesc_base = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTile >> 4) << 24);   // M = 128
        const uint32_t idesc1 = idesc_base | ((uint32_t)(kTile >> 3) << 17), idesc2 = idesc_base | ((uint32_t)(a.rpad >> 3) << 17);
        const uint64_t kdesc0 = smem_desc_sw128(kst_addr), qdesc0 = smem_desc_sw128(q_addr);
        const uint32_t q_panel = (uint32_t)(QR * 128) >> 4;
        bool ok = true;
        int T0 = 0, nq = 0, mine = 0;                          // tiles, items with tiles, and this warp's tiles so far
        int s = mw, b = mw;                                    // this warp's next tile's stage and buffer, parities of the waits on them
        uint32_t s_par = 0, b_par = 1;
        PfItem x;
        while (ok && take(x)) {
            if (x.ntile == 0) continue;
            const int qs = nq & 1;
            ok = __all_sync(0xffffffffu, mbar_wait(bar_qfull + 8 * qs, (uint32_t)((nq >> 1) & 1), abort_flag, kPfQFull, WL));
            if (!ok) break;
            ++nq;
            const uint64_t qdesc = qdesc0 + (uint32_t)(qs * QR * 256 >> 4);
            const int P = a.P - a.rowmap(a.ub0 + x.ul), rows = min(a.rows, (min(P, a.R) - a.i0) * G);
            if (rows < min(a.held, QR)) {
                // what lies behind a shorter window's queries is not the prompt's (both warps clear it, each before its own MMAs)
                for (int c = lane; c < (QR - rows) * 16; c += 32)
                    *reinterpret_cast<uint4 *>(smem + L.q + qs * QR * 256 + ((c & 15) >> 3) * (QR * 128) + (rows + (c >> 4)) * 128 + (c & 7) * 16) = make_uint4(0, 0, 0, 0);
                fence_proxy_async();
                __syncwarp();
            }
            const int j0 = (T0 ^ mw) & 1;
            for (int j = j0; j < x.ntile; j += 2) {
                bool w = mbar_wait(bar_kfull + 8 * s, s_par, abort_flag, kPfKFull, WL);
                w = w && mbar_wait(bar_tempty + 8 * b, b_par, abort_flag, kPfTEmpty, WL);
                ok = __all_sync(0xffffffffu, w);
                if (!ok) break;
                tc_fence_after();
                if (elect_one()) {
                    const uint64_t kdesc = kdesc0 + (uint32_t)(s * (kStageBytes >> 4));
                    const uint32_t d_tmem = tmem_base + (uint32_t)(b * QR);
                    if (x.kind == 1) {
                        // rows in the lanes: D[128 rows x 128 keys] = Q_block . K_tile^T, one block of 128 rows at a time
#pragma unroll
                        for (int ks = 0; ks < kD / 16; ++ks)
                            umma_bf16(d_tmem, qdesc + (ks >> 2) * q_panel + (ks & 3) * 2, kdesc + (ks >> 2) * (kStageBytes / 2 >> 4) + (ks & 3) * 2, idesc1,
                                      ks > 0 ? 1u : 0u);
                        if (RB > 1)
#pragma unroll
                            for (int ks = 0; ks < kD / 16; ++ks)
                                umma_bf16(d_tmem + 128, qdesc + (128 * 128 >> 4) + (ks >> 2) * q_panel + (ks & 3) * 2,
                                          kdesc + (ks >> 2) * (kStageBytes / 2 >> 4) + (ks & 3) * 2, idesc1, ks > 0 ? 1u : 0u);
                    } else {
                        // keys in the lanes: D[128 keys x rpad rows] = K_tile . Q^T
#pragma unroll
                        for (int ks = 0; ks < kD / 16; ++ks)
                            umma_bf16(d_tmem, kdesc + (ks >> 2) * (kStageBytes / 2 >> 4) + (ks & 3) * 2, qdesc + (ks >> 2) * q_panel + (ks & 3) * 2, idesc2,
                                      ks > 0 ? 1u : 0u);
                    }
                    umma_commit(bar_kempty + 8 * s);
                    umma_commit(bar_tfull + 8 * b);
                    if (j + 2 >= x.ntile) umma_commit(bar_qempty + 8 * qs);
                }
                __syncwarp();
                ++mine;
                s += 2; b += 2;
                if (s >= ST) { s = mw; s_par ^= 1; }
                if (b >= NB) { b = mw; b_par ^= 1; }
            }
            if (!ok) break;
            if (j0 >= x.ntile && lane == 0) mbar_arrive(bar_qempty + 8 * qs);      // (no tile of this item is this warp's)
            T0 += x.ntile;
        }
        {   // every commit of this warp is observed before TMEM is freed and the CTA exits
            int dummy = 0;
            const int hs = ST / 2, hb = NB / 2;
            for (int i = max(0, mine - hs); i < mine; ++i)
                mbar_wait(bar_kempty + 8 * (mw + 2 * (i % hs)), (uint32_t)((i / hs) & 1), &dummy, kPfDrain, kWaitCycles);
            if (!ok)
                for (int i = max(0, mine - hb); i < mine; ++i)
                    mbar_wait(bar_tfull + 8 * (mw + 2 * (i % hb)), (uint32_t)((i / hb) & 1), &dummy, kPfDrain, kWaitCycles);
            else
                for (int i = max(0, nq - 2); i < nq; ++i)
                    mbar_wait(bar_qempty + 8 * (i & 1), (uint32_t)((i >> 1) & 1), &dummy, kPfDrain, kWaitCycles);
            __syncwarp();
        }
    } else if (warp == 2) {
        // ------------------------------------------------ normalisers of the items that score
        int n = 0;
        PfItem x;
        while (take(x)) {
            if (x.kind != 2 || a.visit == 2) continue;
            const int s = n & 1, u = a.ub0 + x.ul;
            bool w = mbar_wait(bar_nempty + 8 * s, (uint32_t)(((n >> 1) & 1) ^ 1), abort_flag, kPfNEmpty, WL);
            w = w && pf_flag_wait(a.flag + x.ul, abort_flag, WL);
            if (!__all_sync(0xffffffffu, w)) break;
            const int shift = a.rowmap(u), P = a.P - shift, Rw = min(P, a.R), rows = min(a.rows, (Rw - a.i0) * G);
            for (int row = lane; row < a.rpad; row += 32) {
                const int rslot = (P - Rw + a.i0 + row / G + shift) % a.R;       // ring slots follow the common time axis
                negc_s[s * 256 + row] = row < rows ? -__ldcg(a.ring_c + ((size_t)u * a.R + rslot) * G + row % G) : -INFINITY;   // padding: weight 0
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_nfull + 8 * s);
            ++n;
        }
    } else if (warp >= kPfFirstPublisher && warp < kPfFirstConsumer) {
        // ------------------------------------------------ statistics: merged over the consumer groups and published; the CTA that
        // brings a unit's last run merges the runs
        constexpr int kBar = 1;
        const int pt = tid - 32 * kPfFirstPublisher;
        int n = 0, T0 = 0;
        PfItem x;
        while (take(x)) {
            const int s = n & 1, u = a.ub0 + x.ul, b0 = T0;       // (b0: the item's first tile, whose buffer comes first in the sum:
            T0 += x.ntile;                                        // the result does not depend on which CTA took the item when)
            const int shift = a.rowmap(u), P = a.P - shift, Rw = min(P, a.R), rows = min(a.rows, (Rw - a.i0) * G);
            const int nrun = ((P + kTile - 1) / kTile + a.run - 1) / a.run;
            float2 *unit = reinterpret_cast<float2 *>(a.part_ml) + (size_t)x.ul * a.runs * QR;
            auto merged = [&](int row, int first, int step, int end) -> float2 {
                float m = -INFINITY, l = 0.f;
                for (int r0 = first; r0 < end; r0 += 8 * step) {       // eight loads in flight
                    float2 p[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) p[i] = r0 + i * step < end ? __ldcg(unit + (size_t)(r0 + i * step) * QR + row) : make_float2(-INFINITY, 0.f);
                    float mn = m;
#pragma unroll
                    for (int i = 0; i < 8; ++i) mn = fmaxf(mn, p[i].x);
                    if (mn > -INFINITY) {
                        l *= exp2f(m - mn);
#pragma unroll
                        for (int i = 0; i < 8; ++i) l += p[i].y * exp2f(p[i].x - mn);
                        m = mn;
                    }
                }
                return make_float2(m, l);
            };
            // a row's normaliser; a padding head (zero query) takes no part: +inf, weight 0
            auto to_ring = [&](int row, float2 p) -> float {
                const int g = row % G, rslot = (P - Rw + a.i0 + row / G + shift) % a.R;       // ring slots follow the common time axis
                const float c = g < a.Gq ? p.x + log2f(p.y) : INFINITY;
                if (a.visit != 2 || x.tile0 == 0) a.ring_c[((size_t)u * a.R + rslot) * G + g] = c;
                return c;
            };
            if (x.kind == 2) {
                if (a.visit != 2) continue;
                // the statistics are those of the launch before: every item merges its unit's
                if (group_any(kBar, !mbar_wait(bar_nempty + 8 * s, (uint32_t)(((n >> 1) & 1) ^ 1), abort_flag, kPfNEmpty, WL))) break;
                ++n;
                for (int row = pt; row < a.rpad; row += kGroupThreads)
                    negc_s[s * 256 + row] = row < rows ? -to_ring(row, merged(row, 0, 1, nrun)) : -INFINITY;
                group_sync(kBar, kGroupThreads);
                if (pt == 0) mbar_arrive(bar_nfull + 8 * s);
                continue;
            }
            if (group_any(kBar, !mbar_wait(bar_sfull + 8 * s, (uint32_t)((n >> 1) & 1), abort_flag, kPfSFull, WL))) break;
            ++n;
            const float2 *st = reinterpret_cast<const float2 *>(stat_s) + s * 512;
            for (int row = pt; row < QR; row += kGroupThreads) {
                float m = -INFINITY, l = 0.f;
                for (int b = 0; b < NB; ++b) m = fmaxf(m, st[b * QR + row].x);
                for (int b = 0; b < NB; ++b) {
                    const float2 p = st[((b0 + b) & (NB - 1)) * QR + row];
                    if (p.x > -INFINITY) l += p.y * ex2f(p.x - m);
                }
                unit[(size_t)(x.tile0 / a.run) * QR + row] = make_float2(m, l);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_sempty + 8 * s);
            if (a.visit == 1) continue;
            // The last of a cluster of kPfMerge runs merges them into the cluster's first entry, the last cluster merges the clusters:
            // two round trips of loads each, where one pass over all runs took 25 us at 131072 tokens.
            const int ncl = (nrun + kPfMerge - 1) / kPfMerge, cl = x.tile0 / a.run / kPfMerge;
            int *done = a.done + (size_t)x.ul * (1 + (a.runs + kPfMerge - 1) / kPfMerge);
            auto last_of = [&](int *count, int of) -> bool {   // (the group's writes before it are released, the others' acquired)
                group_sync(kBar, kGroupThreads);
                if (pt == 0) {
                    int old;
                    asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;" : "=r"(old) : "l"(count) : "memory");
                    *last_s = old == of - 1;
                    if (old == of - 1) *count = 0;
                }
                group_sync(kBar, kGroupThreads);
                return *last_s != 0;
            };
            if (!last_of(done + 1 + cl, min(kPfMerge, nrun - cl * kPfMerge))) continue;
            if (ncl > 1) {
                for (int row = pt; row < rows; row += kGroupThreads) unit[(size_t)cl * kPfMerge * QR + row] = merged(row, cl * kPfMerge, 1, min(nrun, (cl + 1) * kPfMerge));
                if (!last_of(done, ncl)) continue;
            }
            for (int row = pt; row < rows; row += kGroupThreads) to_ring(row, ncl > 1 ? merged(row, 0, kPfMerge, nrun) : merged(row, 0, 1, nrun));
            group_sync(kBar, kGroupThreads);
            if (pt == 0 && a.select) asm volatile("st.release.gpu.global.s32 [%0], 1;" ::"l"(a.flag + x.ul) : "memory");
        }
    } else if (warp >= kPfFirstConsumer) {
        // ------------------------------------------------ consumers: tile T is in buffer T % NB, the business of the groups grp
        // with grp % NB == T % NB: one of four, or two of four that share its rows (so every phase of a buffer's barrier is waited
        // for, without which its parity would be ambiguous)
        const int grp = (warp - kPfFirstConsumer) >> 2, b = grp % NB, part = grp / NB;
        const int lq = (warp & 3) * 32 + lane;               // lane of the accumulator this thread reads
        const uint32_t tacc = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(b * QR + part * 128);
        bool ok = true;
        int T0 = 0, n_stat = 0, n_score = 0, n_pair = 0;     // tiles, items of the two kinds and tiles whose scores were shared so far
        PfItem x;
        while (ok && take(x)) {
            const int u = a.ub0 + x.ul, P = a.P - a.rowmap(u), Rw = min(P, a.R);
            const int j0 = (b - T0) & (NB - 1);
            if (x.kind == 1) {
                // this thread's row and the last key it may see
                const int row = part * 128 + lq, lim = row < min(a.rows, (Rw - a.i0) * G) ? P - Rw + a.i0 + row / G : -1;
                float m = -INFINITY, l = 0.f;
                for (int j = j0; j < x.ntile; j += NB) {
                    ok = __all_sync(0xffffffffu, mbar_wait(bar_tfull + 8 * b, (uint32_t)(((T0 + j) / NB) & 1), abort_flag, kPfTFull, WL));
                    if (!ok) break;
                    tc_fence_after();
                    const int key0 = (x.tile0 + j) * kTile;
                    for (int c = 0; c < kTile; c += 32) {
                        uint32_t v[32];
                        tmem_ld32(tacc + (uint32_t)c, v);
                        const int kc = key0 + c;
                        if (kc <= lim) {                     // else: nothing this row may see in these 32 keys
                            if (kc + 31 > lim) {             // the row's causal limit falls inside the chunk
#pragma unroll
                                for (int i = 0; i < 32; ++i)
                                    if (kc + i > lim) v[i] = 0xff800000u;        // -inf: weight 0
                            }
                            // The reference is the maximum so far, rounded up: the weights that count have exponents near 0, and factors
                            // between references, here and where sums are merged, are whole powers of two.  The scale is positive, so
                            // the maximum is taken on the raw logits and scaled once.
                            float cm = -INFINITY;
#pragma unroll
                            for (int i = 0; i < 32; ++i) cm = fmaxf(cm, __uint_as_float(v[i]));
                            cm *= a.scale2;
                            if (cm > m) {
                                const float up = ceilf(cm);
                                l *= ex2f(m - up);
                                m = up;
                            }
                            l += sum_chunk(v, a.scale2, m);
                        }
                        __syncwarp();                        // the lanes meet again in front of the aligned TMEM load
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_tempty + 8 * b);
                    __syncwarp();
                }
                if (!ok) break;
                const int s = n_stat & 1;
                ok = __all_sync(0xffffffffu, mbar_wait(bar_sempty + 8 * s, (uint32_t)(((n_stat >> 1) & 1) ^ 1), abort_flag, kPfSEmpty, WL));
                if (!ok) break;
                ++n_stat;
                reinterpret_cast<float2 *>(stat_s)[(s * NB + b) * QR + row] = make_float2(m, l);
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_sfull + 8 * s);
            } else {
                const int s = n_score & 1, nkeys = P - Rw;
                ok = __all_sync(0xffffffffu, mbar_wait(bar_nfull + 8 * s, (uint32_t)((n_score >> 1) & 1), abort_flag, kPfNFull, WL));
                if (!ok) break;
                ++n_score;
                const float *negc = negc_s + s * 256 + part * 128;
                float *Fu = a.Fp + (size_t)x.ul * a.P;
                const int cols = min(128, a.rpad - part * 128);
                for (int j = j0; j < x.ntile; j += NB) {
                    ok = __all_sync(0xffffffffu, mbar_wait(bar_tfull + 8 * b, (uint32_t)(((T0 + j) / NB) & 1), abort_flag, kPfTFull, WL));
                    if (!ok) break;
                    tc_fence_after();
                    float F = 0.f;
                    for (int c = 0; c < cols; c += 32) {
                        uint32_t v[32];
                        tmem_ld32(tacc + (uint32_t)c, v);
                        score_chunk_pairs<G, FUSION>(v, negc + c, a.scale2, F);
                    }
                    tc_fence_before();
                    if (part > 0) {                          // to the group with the first 128 rows
                        pair_s[b * 128 + lq] = F;
                        __syncwarp();
                        if (lane == 0) { mbar_arrive(bar_pair + 8 * b); mbar_arrive(bar_tempty + 8 * b); }
                        __syncwarp();
                        continue;
                    }
                    if (NB < kPfGroups) {
                        // (the buffer is handed back after this, so the other group cannot have moved on to the next one)
                        ok = __all_sync(0xffffffffu, mbar_wait(bar_pair + 8 * b, (uint32_t)(n_pair & 1), abort_flag, kPfPair, WL));
                        if (!ok) break;
                        ++n_pair;
                        const float F1 = pair_s[b * 128 + lq];
                        F = FUSION == kFusionSum ? F + F1 : fmaxf(F, F1);
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_tempty + 8 * b);
                    __syncwarp();
                    const int key = (x.tile0 + j) * kTile + lq;
                    if (key < nkeys) {
                        if (a.accumulate) F = FUSION == kFusionSum ? Fu[key] + F : fmaxf(Fu[key], F);   // Eq. 5 / 6 over the pieces
                        Fu[key] = F;
                    }
                }
                if (!ok) break;
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_nempty + 8 * s);
            }
            T0 += x.ntile;
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
    if (tid == 0 && *abort_flag) atomicCAS(a.err, 0, *abort_flag);
    if (a.visit != 0) return;                                  // (no ticket was taken, no flag is looked at)
    if (tid == 0) {
        __threadfence();
        *last_s = atomicAdd(a.left, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (*last_s) {                                             // the last CTA leaves everything as it was found
        for (int i = tid; i < a.nb; i += kPfThreads) a.flag[i] = 0;
        if (tid == 0) { *a.ticket = 0; *a.left = 0; }
    }
}

template <int G>
cudaError_t launch_scores(const PfArgs &a, const CUtensorMap &tmK, const CUtensorMap &tmQ, int fusion, cudaStream_t stream)
{
    auto kern = fusion == kFusionSum ? prefill_tc_kernel<G, kFusionSum> : prefill_tc_kernel<G, kFusionMax>;
    const int smem = pf_smem(a.qrows, a.stages).total + 1024;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    return launch_chained(kern, dim3((unsigned)std::min(kPromptCtas, a.items)), kPfThreads, smem, stream, a, tmK, tmQ);
}

// The window queries [units][heads][slots][128] as boxes of `slots` window slots x `group` heads x 64 columns: window slot by window
// slot in shared memory
bool encode_window_map(CUtensorMap *m, const void *q, int units, int heads, int slots, int group, int box_slots)
{
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[4] = {(cuuint64_t)kD, (cuuint64_t)heads, (cuuint64_t)slots, (cuuint64_t)units};
    const cuuint64_t strides[3] = {(cuuint64_t)slots * kD * 2, (cuuint64_t)kD * 2, (cuuint64_t)heads * slots * kD * 2};
    const cuuint32_t box[4] = {64, (cuuint32_t)group, (cuuint32_t)box_slots, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(q), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int pf_qrows(int rows) { return rows <= 128 ? 128 : 256; }

}  // namespace

bool prefill_tc_supported(bool f32, int D, int G, int R, const void *k, const void *qwin, int P)
{
    // any window: the pieces need no more than 256 rows at a time (the decode kernel's own limit on the ring, which
    // the stored-profile mode lifts, does not apply here)
    return !f32 && D == kD && G >= 1 && G <= kMaxGroup && R >= 1 && (((uintptr_t)k | (uintptr_t)qwin) & 15) == 0 && P >= 1;
}

int prefill_tc_run(const DecodeArgs &a, int P, const int *row_shift) { return prompt_run(row_shift, P, a.Hkv, a.B, a.U, std::min(P, a.R) * a.G, P - std::min(P, a.R) > a.C); }

static int pf_runs(int P, int run) { return ((P + kTile - 1) / kTile + run - 1) / run; }

size_t prefill_tc_words_per_unit(int P, int run) { return 2 + (pf_runs(P, run) + kPfMerge - 1) / kPfMerge; }

size_t prefill_tc_floats_per_unit(int P, int Rw, int G, int run)
{
    // scores, statistics, words of state
    return (size_t)P + (size_t)pf_runs(P, run) * pf_qrows(Rw * G) * 2 + prefill_tc_words_per_unit(P, run);
}

// Window-row normalisers into ring_c and, if `select`, fused scores of the prompt's older tokens into Fp [nb][P] for units
// ub0 .. ub0+nb-1.  `part` holds the statistics of `units` >= nb units; `words`: prefill_tc_words_per_unit words a unit and two more that are
// zero, and are again afterwards; `err` is a zeroed error word.
cudaError_t run_prefill_scores_tc(const DecodeArgs &a, const void *k, const void *qwin, int P, int Ps, const int *row_shift, int ub0, int nb, int units, int run, bool select,
                                  float *Fp, float *part, int *words, int *err, unsigned long long *launches, cudaStream_t stream)
{
    CUtensorMap tmK, tmQ;
    if (!encode_map(&tmK, const_cast<void *>(k), a.U, Ps, kTile)) return cudaErrorInvalidValue;
    const int Rw = P < a.R ? P : a.R, slots_per_piece = 256 / a.G;
    const int Rws = Ps < a.R ? Ps : a.R;
    PfArgs pa = {};
    pa.part_ml = part; pa.ring_c = a.ring_c; pa.Fp = Fp;
    pa.flag = words; pa.ticket = words + units; pa.left = pa.ticket + 1; pa.done = pa.left + 1; pa.err = err;
    pa.ub0 = ub0; pa.nb = nb; pa.P = P; pa.C = a.C; pa.rowmap = {a.row_shift, a.Hkv, a.B}; pa.G = a.G; pa.R = a.R; pa.Gq = a.Gq;
    pa.run = run; pa.runs = pf_runs(P, run);
    pa.order = run_order(row_shift, P, a.Hkv, a.B, run, ub0, nb, &pa.items);
    pa.order.shift = a.row_shift;
    pa.select = select ? 1 : 0;
    pa.scale2 = a.scale2;
    pa.wait_cycles = kWaitCycles;
    pa.lag = prompt_lag(pa.items, pa.runs);
    // One launch per visit where the batch's keys stay in L2 by themselves, the second of which merges the statistics: the normalisers
    // then take the end of a launch instead of a chain of tickets and a flag.  Not where nothing is selected, as the second visit then has
    // nothing else to do (32 units x 600 tokens 59 -> 62), unless there are fewer tiles than SMs.
    int tiles;
    run_order(row_shift, P, a.Hkv, a.B, 1, ub0, nb, &tiles);
    const bool apart = tiles <= (select ? prompt_apart_tiles(Rw * a.G) : kPromptCtas);
    // up to 256 window rows per launch; the rows of a wider window are taken in pieces of whole window
    // slots, whose normalisers are independent and whose scores fuse associatively (Eq. 5 / 6)
    for (int i0 = 0; i0 < Rw; i0 += slots_per_piece) {
        pa.i0 = i0;
        pa.accumulate = i0 > 0 ? 1 : 0;
        pa.rows = std::min(slots_per_piece, Rw - i0) * a.G;
        pa.held = (Rws - i0) * a.G;
        pa.rpad = (pa.rows + 31) & ~31;
        pa.qrows = pf_qrows(pa.rows);
        pa.stages = pa.qrows == 128 ? 4 : 2;
        pa.bufs = 512 / pa.qrows;
        if (!encode_window_map(&tmQ, qwin, a.U, a.Gq, Rws, a.G, pa.qrows / a.G)) return cudaErrorInvalidValue;
        for (pa.visit = apart ? 1 : 0; pa.visit <= (apart ? 2 : 0); ++pa.visit) {
            cudaError_t e = cudaErrorInvalidValue;
            switch (a.G) {
                case 1: e = launch_scores<1>(pa, tmK, tmQ, a.fusion, stream); break;
                case 2: e = launch_scores<2>(pa, tmK, tmQ, a.fusion, stream); break;
                case 4: e = launch_scores<4>(pa, tmK, tmQ, a.fusion, stream); break;
                case 8: e = launch_scores<8>(pa, tmK, tmQ, a.fusion, stream); break;
                case 16: e = launch_scores<16>(pa, tmK, tmQ, a.fusion, stream); break;
            }
            if (e != cudaSuccess) return e;
            ++*launches;
        }
    }
    return cudaSuccess;
}

}  // namespace mkv
