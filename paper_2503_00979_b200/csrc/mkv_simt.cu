// Warp-level decode kernel: any dtype (bf16 / f32), head_dim 64 or 128, any GQA group and window size.  It is the
// kernel of the f32 mode, of head_dim 64 and of windows beyond the tcgen05 kernel's range, the low-latency kernel of
// small launches (one layer of a small batch) of the tcgen05 contexts, and an on-device cross-check of that kernel.
//
// A unit is one CTA's, or a cluster's of up to sixteen CTAs, each with a contiguous range of the cached keys.  The
// warps of a CTA take tiles of 32 keys (f32: 16) in turn and do not wait for one another; a warp copies its tile into shared memory of
// its own (cp.async, 16-byte chunks swizzled by row), the next K tile while P.V runs and the next V tile while it is
// scored.  Per tile:
//   scores   logits of the tile's keys against the resident ring rows: bf16 on mma.sync (keys are the rows of the
//            A operand), f32 with two lanes per key.  The rows turn into frozen weights exp2(s - c_row), are summed over
//            the GQA group and fused over the window (Eq. 4-6, Algorithm 1).  Resident are the block of ring slots that
//            is being filled and, on the step that opens it, the block before it; the rest of the window comes from the
//            sums in slab and pre (DecodeArgs::slab).  Without kept sums (CURRENT normalisation, windows of more than
//            kMaxBlocks blocks) the whole ring passes through, kRows rows at a time.
//   attend   logits and soft-max of the new query over the tile, continued online, and P.V (Eq. 1): bf16 on mma.sync
//            with P in three bf16 terms (24 mantissa bits), f32 with one slice of the head dimension per lane.
// The warps' partials are merged in shared memory; the CTAs of a cluster then exchange theirs through distributed shared
// memory, each writes a slice of the output, adds the new row's term to the scores of its own keys and finds their
// minimum; a second exchange elects the slot that is evicted (Eq. 7).  Scores stay in shared memory while a CTA's range
// is short enough.
//
// Bound by HBM for bf16 and, nearly, by FMA issue for f32; small launches by their chain of latencies.  Of those
// everything that does not need the new query (state, tiles, ring rows, their scoring) may run before the launch before
// this one has ended, when that launch works on another layer (DecodeArgs::early).
//
// Measured: 512 units x 1056 slots, bf16, d = 64, R*G = 128: 65 us per step (all rows scored with scalar FMAs, CTA barriers
// per tile: 838).  2 units x 80 slots, f32, d = 64: 10.6 us (30.6).  One layer of 8 units x 2032 slots, bf16, d = 128, as a
// cluster of 16 CTAs per unit: 11.6 us per call in a sequence of layers (17.2 on the tcgen05 kernel).
#include "mkv_common.cuh"
#include "mkv_kernels.h"
#include "mkv_sm100.cuh"

namespace mkv {

namespace {

constexpr int kRound = 128;          // keys a CTA takes in one round of its warps: 4 x 32 (bf16) or 8 x 16 (f32)
constexpr int kMaxCluster = 16;      // CTAs per unit
constexpr int kMaxBlocks = 64;       // beyond this many blocks the sums would outgrow the rows they save

// 16-byte chunk `ch` of row `row` in a tile of rows of ROWB bytes
template <int ROWB> __device__ __forceinline__ uint32_t swz(int row, int ch)
{
    return (uint32_t)(row * ROWB + ((ch ^ (row & 7)) << 4));
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, bool live)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(live ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}

// p in three bf16 terms
__device__ __forceinline__ void split3(float x, float y, uint32_t (&t)[3])
{
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
        const float2 f = __bfloat1622float2(h);
        x -= f.x; y -= f.y;
        t[i] = *reinterpret_cast<const uint32_t *>(&h);
    }
}

template <typename T, int D, int GP> struct SimtSmem {
    static constexpr int kt = sizeof(T) == 2 ? 32 : 16;        // keys per warp tile
    static constexpr int warps = kRound / kt, threads = 32 * warps;
    // CTAs per SM.  Two or more leave room for the next layer's launch beside this one's; at 128-wide bf16 heads that takes
    // every byte there is, hence `keys`.
    static constexpr int ctas = sizeof(T) == 2 ? (D == 64 ? 4 : 2) : (D == 64 ? 2 : 1);
    static constexpr int row = D * (int)sizeof(T);             // bytes of a K, V or query row
    static constexpr int tile = kt * row;
    static constexpr int stage = 2 * tile;                     // K and V, per warp; later its partial output [GP][D] floats
    static constexpr int st_w = GP * kt + 4 * GP + 32;         // floats per warp: logits or weights, factors, references, F
    static constexpr int rows = sizeof(T) == 2 && D == 128 ? 128 : 64;     // resident ring rows
    static constexpr int qn_rows = GP > 8 ? GP : 8;            // the new query's rows
    static constexpr int keys = GP == 4 ? 224 : GP > 4 ? 256 : 512;        // keys whose scores stay in shared memory
    static constexpr int q = 0;
    static constexpr int qn = q + rows * row;
    static constexpr int stages = qn + qn_rows * row;
    static constexpr int negc = stages + warps * stage;
    static constexpr int stw = negc + rows * 4;
    static constexpr int wml = stw + warps * st_w * 4;
    static constexpr int cml = wml + warps * GP * 2 * 4;      // partial (m, l) of each CTA of the cluster [16][GP][2]
    static constexpr int co = cml + kMaxCluster * GP * 2 * 4;  // partial outputs, this CTA's slice of each [16][slice]
    static constexpr int cred = co + (GP * D + kMaxCluster) * 4 + 16;      // (rank key, slot) of each CTA of the cluster
    static constexpr int loc = cred + kMaxCluster * 16;        // scores, positions, logits of the CTA's keys
    static constexpr int fin = loc + (2 + GP) * keys * 4;      // q [GP][D], k_new [D], v_new [D], self, m, l, c [GP], reduction
    static constexpr int total = fin + (GP * D + 2 * D + 4 * GP + 3 * warps) * 4;
    static_assert(stage >= GP * D * 4, "a warp's partial fits its stage");
    static_assert(total <= 227 * 1024 && (GP > 4 || ctas * (total + 1024) <= 228 * 1024), "shared memory");
};

// epilogue scratch inside the `fin` area
template <int D, int GP, int W> struct Fin {
    float *q, *k, *v, *self, *m, *l, *c;
    unsigned long long *red_key;
    int *red_slot;
    __device__ explicit Fin(float *p)
    {
        q = p; k = q + GP * D; v = k + D;
        self = v + D; m = self + GP; l = m + GP; c = l + GP;
        red_key = reinterpret_cast<unsigned long long *>(c + GP);
        red_slot = reinterpret_cast<int *>(red_key + W);
    }
};

// distributed shared memory of the cluster
__device__ __forceinline__ uint32_t mapa(uint32_t addr, int rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, float v)
{
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void st_cluster64(uint32_t addr, unsigned long long v)
{
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// GP: the group padded to a power of two (padding heads: zero query, weight 0).  CHECK: DecodeArgs::check_moved (compiled apart, as it costs a layer's call 0.4 us).
template <typename T, int D, int GP, bool CHECK>
__global__ void __launch_bounds__(SimtSmem<T, D, GP>::threads, GP > 8 ? 1 : SimtSmem<T, D, GP>::ctas)
decode_simt_kernel(const __grid_constant__ DecodeArgs a, const int nsplit)
{
    using L = SimtSmem<T, D, GP>;
    constexpr bool BF = sizeof(T) == 2;
    constexpr int kKT = L::kt, kWarps = L::warps, kThreads = L::threads;
    constexpr int CH = L::row / 16, EP = 16 / (int)sizeof(T);   // chunks per row, elements per chunk
    extern __shared__ __align__(1024) unsigned char smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int Gs = a.G, G = a.Gq, R = a.R;                      // heads per ring slot and scratch row as laid out, real heads
    const int u = blockIdx.x / nsplit, sp = blockIdx.x % nsplit;
    const uint32_t q_s = smem_u32(smem + L::q), qn_s = smem_u32(smem + L::qn);
    const uint32_t k_s = smem_u32(smem + L::stages) + warp * L::stage, v_s = k_s + L::tile;
    float *negc = reinterpret_cast<float *>(smem + L::negc);
    float *st_w = reinterpret_cast<float *>(smem + L::stw) + warp * L::st_w;     // [g][key]
    float *fac = st_w + GP * kKT, *mref = fac + GP, *fsm = st_w + GP * kKT + 4 * GP;
    float *wml = reinterpret_cast<float *>(smem + L::wml);
    const Fin<D, GP, kWarps> fin(reinterpret_cast<float *>(smem + L::fin));

    if (nsplit > 1) cluster_arrive();      // waited for before the first access to another CTA's memory
    // see the tcgen05 kernel: the grid before this one is complete behind the wait, the next one may start and park there.
    // (Every grid releases the next one after its own wait, so the grid before the one before this one is complete here
    // already: with DecodeArgs::early nothing in flight can still write this launch's units or their state.)
    if (!a.early) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
    const long long t = __ldcg(&a.st->t);
    const int n = __ldcg(&a.st->n), steps_done = __ldcg(&a.st->steps);
    const bool evict_all = step_scores(t, n, steps_done, R, a.C, a.T);
    // the unit's own fill and policy decision (they differ from the uniform ones only between batch rows whose
    // prompts had different lengths); the splits are laid out over the largest fill
    const UnitStep us = unit_step(a, u, t, n, steps_done, evict_all);
    const bool evict = us.evict;
    int active;                                                 // (CTAs with keys; the others of a cluster take part all the same)
    const int per = split_len(n, nsplit, 32, &active);
    const int k0 = min(n, sp * per), k1 = min(us.n, k0 + per);
    const int ntile = (min(n, k0 + per) - k0 + kKT - 1) / kKT;
    // (positions fit in 32 bits; 64-bit divisions would take most of a microsecond here)
    const int rs_new = (int)((unsigned)t % (unsigned)R), jb = rs_new / a.bs;
    const bool kept = a.nblk > 1, fold = kept && jb * a.bs == rs_new;
    const int j_old = rs_new == 0 ? a.nblk - 1 : jb - 1;        // fold: the finished block
    // ring slots that pass through: the open block (the whole ring without kept sums)
    const bool score = evict || fold;
    constexpr int slots_per = L::rows / GP;
    const int s_begin = score ? jb * a.bs : rs_new, s_end = score ? min(R, (jb + 1) * a.bs) : rs_new + 1;
    const T *Ku = static_cast<const T *>(a.K) + (size_t)u * a.cap * D, *Vu = static_cast<const T *>(a.V) + (size_t)u * a.cap * D;
    const int *pos = a.pos + (size_t)u * a.cap;
    float *slab = kept ? a.slab + (size_t)u * a.nblk * a.cap : nullptr, *pre = kept ? a.pre + (size_t)u * a.cap : nullptr;
    bool moved = false;                                         // a slot holds another token than its window sums belong to
    // scores, logits and positions of this CTA's keys: in shared memory if they fit (index key - k0), else in the arena
    // (CURRENT normalisation reads the logits there)
    const bool local = per <= L::keys && !a.norm_current;
    float *Fu = a.F + (size_t)u * a.cap + k0;
    float *Fk = local ? reinterpret_cast<float *>(smem + L::loc) : Fu;
    int *pk = reinterpret_cast<int *>(smem + L::loc) + L::keys;                 // local only
    float *sk = local ? reinterpret_cast<float *>(smem + L::loc) + 2 * L::keys : a.s_new + (size_t)u * Gs * a.cap + k0;
    const int sk_stride = local ? L::keys : a.cap;

    auto load_tile = [&](uint32_t dst, const T *base, int it) {
        if (it < ntile) {
            const int key0 = k0 + it * kKT;
#pragma unroll
            for (int i = 0; i < kKT * CH / 32; ++i) {
                const int c = i * 32 + lane, row = c / CH, ch = c % CH;
                const bool live = key0 + row < k1;
                cp_async16(dst + swz<L::row>(row, ch), base + (size_t)(live ? key0 + row : 0) * D + ch * EP, live);
            }
        }
        cp_async_commit();
    };

    float mrun[GP], lsum[GP > 2 ? GP : 2];                    // bf16: lsum[nt] of the fragment layout
    constexpr int NT = GP > 8 ? 2 : 1, DB = D / 16, DC = D / 32;
    float acc[BF ? NT * DB * 4 : GP * DC];
#pragma unroll
    for (int g = 0; g < GP; ++g) mrun[g] = -INFINITY;
#pragma unroll
    for (int i = 0; i < (GP > 2 ? GP : 2); ++i) lsum[i] = 0.f;
#pragma unroll
    for (int i = 0; i < (BF ? NT * DB * 4 : GP * DC); ++i) acc[i] = 0.f;
    const int gid = lane >> 2, tig = lane & 3;
    bool first_tile = true, q_here = false;

    for (int s0 = s_begin; s0 < s_end; s0 += slots_per) {
        const int s1 = min(s_end, s0 + slots_per);
        const bool attend = rs_new >= s0 && rs_new < s1;       // the pass in which the new query attends
        // rows of this pass: the slots s0 .. s1 - 1, padded to whole n-tiles, then the finished block's (fold)
        const int nA = (s1 - s0) * GP, rA = (nA + 7) & ~7;
        const int f0 = j_old * a.bs, nB = fold ? (min(R, f0 + a.bs) - f0) * GP : 0, nrow = score ? rA + ((nB + 7) & ~7) : 0;
        if (s0 != s_begin) __syncthreads();                    // the rows of the pass before are done with
        for (int i = tid; i < nrow * CH; i += kThreads) {      // (copy groups in order: rows, K, V)
            const int row = i / CH, ch = i % CH;
            const bool inA = row < nA, inB = row >= rA && row < rA + nB;
            const int rr = inA ? row : row - rA, slot = (inA ? s0 : f0) + rr / GP, g = rr % GP;
            const bool there = (inA || inB) && g < G;
            const T *src = static_cast<const T *>(a.ring_q) + (there ? (((size_t)u * R + slot) * Gs + g) * D + ch * EP : 0);
            cp_async16(q_s + (BF ? swz<L::row>(row, ch) : (uint32_t)(row * L::row + ch * 16)), src, there);
        }
        cp_async_commit();
        load_tile(k_s, Ku, warp);
        if (attend) load_tile(v_s, Vu, warp); else cp_async_commit();
        for (int row = tid; row < nrow; row += kThreads) {
            const bool inA = row < nA, inB = row >= rA && row < rA + nB;
            const int rr = inA ? row : row - rA, slot = (inA ? s0 : f0) + rr / GP, g = rr % GP;
            // the slot of the row that leaves the window, padding: weight 0
            negc[row] = (inA || inB) && g < G && slot != rs_new ? -a.ring_c[((size_t)u * R + slot) * Gs + g] : -INFINITY;
        }
        cp_async_wait<2>();                           // the rows
        __syncthreads();

        // the first round ends with the new query's arrival; every warp takes part in it, with or without a tile
        for (int it = warp, round = 0; it < ntile || round == 0; it += kWarps, ++round) {
            const bool live = it < ntile;
            const int kl = it * kKT + lane % kKT, key = k0 + kl;
            const bool valid = live && key < k1 && lane < kKT;   // f32: two lanes per key, the lower one speaks for it
            float F = 0.f;
            if (live) {
                float f_pre = 0.f, f_rest = 0.f;               // the rest of the window's fused score
                if (kept && score && valid) {
                    if (jb > (fold ? 1 : 0)) f_pre = __ldcg(pre + key);
                    if ((jb > 0 || !fold) && jb + 1 < a.nblk) f_rest = __ldcg(slab + (size_t)(jb + 1) * a.cap + key);
                    f_rest = fuse(a.fusion, f_rest, f_pre);
                }
                if (local && evict && valid) pk[kl] = pos[key];
                if (CHECK && valid) moved |= pos[key] != __ldcg(a.sum_pos + (size_t)u * a.cap + key);
                cp_async_wait<1>();
                __syncwarp();
                // ---------------- fused scores over the resident rows
                float S = 0.f;
                if constexpr (BF) {
                    uint32_t af[2][D / 16][4];
                    if (score) {
#pragma unroll
                        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                            for (int ks = 0; ks < D / 16; ++ks) ldmatrix_x4(k_s + swz<L::row>(mt * 16 + (lane & 15), ks * 2 + (lane >> 4)), af[mt][ks]);
                    }
                    float fk[2][2] = {{0.f, 0.f}, {0.f, 0.f}}, pend[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
                    auto to_lanes = [&]() {                    // a key's score from the four lanes of its fragment row to lane = key
#pragma unroll
                        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                float x = fk[mt][h];
                                x = fuse(a.fusion, x, __shfl_xor_sync(0xffffffffu, x, 1));
                                x = fuse(a.fusion, x, __shfl_xor_sync(0xffffffffu, x, 2));
                                if (tig == 0) fsm[mt * 16 + gid + h * 8] = x;
                                fk[mt][h] = 0.f;
                            }
                        __syncwarp();
                        const float x = fsm[lane];
                        __syncwarp();
                        return x;
                    };
#pragma unroll 1
                    for (int nt = 0; nt < nrow / 8; ++nt) {
                        float c[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
                        for (int kp = 0; kp < D / 32; ++kp) {
                            uint32_t b[4];
                            ldmatrix_x4(q_s + swz<L::row>(nt * 8 + (lane & 7), kp * 4 + (lane >> 3)), b);
#pragma unroll
                            for (int mt = 0; mt < 2; ++mt) {
                                mma_bf16_16816(c[mt], af[mt][2 * kp], b[0], b[1]);
                                mma_bf16_16816(c[mt], af[mt][2 * kp + 1], b[2], b[3]);
                            }
                        }
                        if (nt * 8 == rA) F = to_lanes();      // the open block is done, the finished one follows
                        const int r = nt * 8 + tig * 2;
                        const float n0 = negc[r], n1 = negc[r + 1];
#pragma unroll
                        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                const float w0 = exp2f(fmaf(c[mt][2 * h], a.scale2, n0)), w1 = exp2f(fmaf(c[mt][2 * h + 1], a.scale2, n1));
                                if (a.fusion == kFusionSum) {
                                    fk[mt][h] += w0 + w1;
                                } else if (GP == 1) {
                                    fk[mt][h] = fmaxf(fk[mt][h], fmaxf(w0, w1));
                                } else {
                                    float x = w0 + w1;
                                    if (GP >= 4) x += __shfl_xor_sync(0xffffffffu, x, 1);
                                    if (GP >= 8) x += __shfl_xor_sync(0xffffffffu, x, 2);
                                    if (GP == 16) {
                                        pend[mt][h] += x;
                                        x = pend[mt][h];
                                        if ((nt & 1) == 0) continue;
                                        pend[mt][h] = 0.f;
                                    }
                                    fk[mt][h] = fmaxf(fk[mt][h], x);
                                }
                            }
                    }
                    if (score) { const float x = to_lanes(); if (nrow > rA) S = x; else F = x; }
                } else {
                    const unsigned char *qb = smem + L::q;
                    const unsigned char *kb = smem + L::stages + warp * L::stage;
                    constexpr int RB = GP > 8 ? GP : 8;        // rows at a time: whole slots
#pragma unroll 1
                    for (int r0 = 0; r0 < nrow; r0 += RB) {
                        float x[RB];
#pragma unroll
                        for (int r = 0; r < RB; ++r) x[r] = 0.f;
#pragma unroll 4
                        for (int ch = lane / kKT; ch < CH; ch += 2) {              // each of a key's two lanes takes every other chunk
                            const float4 kv = *reinterpret_cast<const float4 *>(kb + swz<L::row>(lane % kKT, ch));
#pragma unroll
                            for (int r = 0; r < RB; ++r) {
                                const float4 qv = *reinterpret_cast<const float4 *>(qb + (r0 + r) * L::row + ch * 16);
                                x[r] += kv.x * qv.x + kv.y * qv.y + kv.z * qv.z + kv.w * qv.w;
                            }
                        }
#pragma unroll
                        for (int r = 0; r < RB; ++r) x[r] += __shfl_xor_sync(0xffffffffu, x[r], 16);
                        float f = 0.f;
#pragma unroll
                        for (int r = 0; r < RB; r += GP) {
                            float Sr = 0.f;
#pragma unroll
                            for (int g = 0; g < GP; ++g) Sr += exp2f(fmaf(x[r + g], a.scale2, negc[r0 + r + g]));
                            f = fuse(a.fusion, f, Sr);
                        }
                        if (r0 < rA) F = fuse(a.fusion, F, f); else S = fuse(a.fusion, S, f);
                    }
                }
                if (fold && valid) {                           // the finished block of the ring, scored for good
                    float *sb = slab + key;
                    sb[(size_t)j_old * a.cap] = S;
                    if (jb > 0) {
                        pre[key] = fuse(a.fusion, f_pre, S);
                    } else {                                   // a lap ends: its single blocks become the sums of all later ones
                        for (int i0 = a.nblk - 2; i0 >= 1; i0 -= 4) {
                            float v[4];
#pragma unroll
                            for (int b = 0; b < 4; ++b) v[b] = i0 - b >= 1 ? __ldcg(sb + (size_t)(i0 - b) * a.cap) : 0.f;
#pragma unroll
                            for (int b = 0; b < 4; ++b)
                                if (i0 - b >= 1) {
                                    S = fuse(a.fusion, S, v[b]);
                                    sb[(size_t)(i0 - b) * a.cap] = S;
                                }
                        }
                    }
                    f_rest = fuse(a.fusion, f_rest, S);
                }
                if (evict && valid) {
                    F = fuse(a.fusion, F, s0 == s_begin ? f_rest : Fk[kl]);
                    Fk[kl] = F;
                }
            }
            if (!q_here) {
                q_here = true;
                if (a.early) {
                    asm volatile("griddepcontrol.wait;" ::: "memory");
                    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
                }
                // the new token's tensors: query rows for the logits, everything as floats for the epilogue.  All loads
                // are issued before the first of them is waited for.
                const T *q = static_cast<const T *>(a.q) + (size_t)u * G * D;
                const bool aligned = (reinterpret_cast<uintptr_t>(q) & 15) == 0;
                constexpr int KI = (2 * D + kThreads - 1) / kThreads;
                float kv[KI];
#pragma unroll
                for (int j = 0; j < KI; ++j) {
                    const int i = tid + j * kThreads;
                    kv[j] = i < D ? ldf(static_cast<const T *>(a.k_new) + (size_t)u * D + i)
                          : i < 2 * D ? ldf(static_cast<const T *>(a.v_new) + (size_t)u * D + i - D) : 0.f;
                }
                constexpr int QI = (L::qn_rows * CH + kThreads - 1) / kThreads;
                __align__(16) T e[QI][EP];
#pragma unroll
                for (int j = 0; j < QI; ++j) {
                    const int i = tid + j * kThreads, row = i / CH, ch = i % CH;
                    *reinterpret_cast<uint4 *>(e[j]) = make_uint4(0, 0, 0, 0);
                    if (row < G) {
                        if (aligned) {
                            *reinterpret_cast<uint4 *>(e[j]) = reinterpret_cast<const uint4 *>(q + (size_t)row * D)[ch];
                        } else {
#pragma unroll
                            for (int x = 0; x < EP; ++x) e[j][x] = q[(size_t)row * D + ch * EP + x];
                        }
                    }
                }
#pragma unroll
                for (int j = 0; j < QI; ++j) {
                    const int i = tid + j * kThreads, row = i / CH, ch = i % CH;
                    if (row < L::qn_rows)
                        *reinterpret_cast<uint4 *>(smem + L::qn + (BF ? swz<L::row>(row, ch) : (uint32_t)(row * L::row + ch * 16))) = *reinterpret_cast<uint4 *>(e[j]);
                    if (row < GP)
#pragma unroll
                        for (int x = 0; x < EP; ++x) fin.q[row * D + ch * EP + x] = ldf(e[j] + x);
                }
#pragma unroll
                for (int j = 0; j < KI; ++j)                   // (v lies behind k)
                    if (tid + j * kThreads < 2 * D) fin.k[tid + j * kThreads] = kv[j];
                __syncthreads();
                if (tid == 0) {
                    // Every thread holds its copy of the step state (and has used it): the last CTA to get here advances it
                    // for the next launch.  No fence: nothing is published, and one would wait for this warp's stores.
                    if (atomicAdd(&a.st->done, 1u) == gridDim.x - 1) advance_state(a, t, n, steps_done, evict_all);
                }
            }
            if (!live) break;
            // ---------------- logits of the new query
            float s2[GP];
            if (attend) {
                if constexpr (BF) {
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt) {
                        float c[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
                        for (int kp = 0; kp < D / 32; ++kp) {
                            uint32_t b[4];
                            ldmatrix_x4(qn_s + swz<L::row>(nt * 8 + (lane & 7), kp * 4 + (lane >> 3)), b);
#pragma unroll
                            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                                for (int h = 0; h < 2; ++h) {
                                    uint32_t af[4];
                                    ldmatrix_x4(k_s + swz<L::row>(mt * 16 + (lane & 15), (2 * kp + h) * 2 + (lane >> 4)), af);
                                    mma_bf16_16816(c[mt], af, b[2 * h], b[2 * h + 1]);
                                }
                        }
#pragma unroll
                        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const int g = nt * 8 + tig * 2 + (e & 1);
                                if (g < GP) st_w[g * kKT + mt * 16 + gid + (e >> 1) * 8] = c[mt][e] * a.scale2;
                            }
                    }
                    __syncwarp();
#pragma unroll
                    for (int g = 0; g < GP; ++g) s2[g] = st_w[g * kKT + lane];
                } else {
                    const unsigned char *kb = smem + L::stages + warp * L::stage;
#pragma unroll
                    for (int g = 0; g < GP; ++g) s2[g] = 0.f;
#pragma unroll 4
                    for (int ch = lane / kKT; ch < CH; ch += 2) {
                        const float4 kv = *reinterpret_cast<const float4 *>(kb + swz<L::row>(lane % kKT, ch));
#pragma unroll
                        for (int g = 0; g < GP; ++g) {
                            const float4 qv = *reinterpret_cast<const float4 *>(smem + L::qn + g * L::row + ch * 16);
                            s2[g] += kv.x * qv.x + kv.y * qv.y + kv.z * qv.z + kv.w * qv.w;
                        }
                    }
#pragma unroll
                    for (int g = 0; g < GP; ++g) s2[g] = (s2[g] + __shfl_xor_sync(0xffffffffu, s2[g], 16)) * a.scale2;
                }
            }
            __syncwarp();                                      // the K tile has been read
            load_tile(k_s, Ku, it + kWarps);
            if (!attend) {
                cp_async_commit();                             // keeps the count of copy groups
                continue;
            }
            // ---------------- online soft-max of the new row over this warp's keys (Eq. 1)
            bool changed = false;
#pragma unroll
            for (int g = 0; g < GP; ++g) {
                const float s = valid ? s2[g] : -INFINITY;
                if (valid && evict && g < G) sk[(size_t)g * sk_stride + kl] = s;
                const float mn = fmaxf(mrun[g], warp_max(s));
                const float f = mn == mrun[g] ? 1.f : exp2f(mrun[g] - mn);
                changed |= mn != mrun[g];
                mrun[g] = mn;
                if constexpr (BF) {
                    st_w[g * kKT + lane] = s;
                    if (lane == 0) { fac[g] = f; mref[g] = mn == -INFINITY ? 0.f : mn; }
                } else {
                    const float p = mn == -INFINITY ? (s == -INFINITY ? 0.f : s) : exp2f(s - mn);        // (s -inf or NaN: NaN stays)
                    if (lane < kKT) st_w[g * kKT + lane] = p;
                    lsum[g] = lsum[g] * f + p;
                    if (f != 1.f && !first_tile)
#pragma unroll
                        for (int c = 0; c < DC; ++c) acc[g * DC + c] *= f;
                }
            }
            cp_async_wait<1>();                                // this tile's V (the next K may still be on its way)
            __syncwarp();
            if constexpr (BF) {
                if (changed && !first_tile) {
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt) {
                        const int gr = gid + 8 * nt, gc = tig * 2 + 8 * nt;
                        const float fr = gr < GP ? fac[gr] : 0.f, f0_ = gc < GP ? fac[gc] : 0.f, f1_ = gc + 1 < GP ? fac[gc + 1] : 0.f;
                        lsum[nt] *= fr;
#pragma unroll
                        for (int i = 0; i < DB; ++i) {
                            float *x = acc + (nt * DB + i) * 4;
                            x[0] *= f0_; x[1] *= f1_; x[2] *= f0_; x[3] *= f1_;
                        }
                    }
                }
                // O^T[d][g] += V^T[d][keys] . P^T[keys][g]
#pragma unroll
                for (int ks = 0; ks < 2; ++ks) {
                    uint32_t b0[NT][3], b1[NT][3];
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt) {
                        const int gr = gid + 8 * nt;
                        const bool lv = gr < GP;
                        const int grc = lv ? gr : 0;
                        const float *p = st_w + grc * kKT + ks * 16 + tig * 2;
                        const float m = mref[grc];
                        float p0 = exp2f(p[0] - m), p1 = exp2f(p[1] - m), p2 = exp2f(p[8] - m), p3 = exp2f(p[9] - m);
                        p0 = lv ? p0 : 0.f; p1 = lv ? p1 : 0.f; p2 = lv ? p2 : 0.f; p3 = lv ? p3 : 0.f;
                        lsum[nt] += (p0 + p1) + (p2 + p3);
                        split3(p0, p1, b0[nt]);
                        split3(p2, p3, b1[nt]);
                    }
                    __syncwarp();
                    const int mat = lane >> 3, krow = ks * 16 + (mat >> 1) * 8 + (lane & 7);
#pragma unroll
                    for (int db = 0; db < DB; ++db) {
                        uint32_t af[4];
                        ldmatrix_x4_trans(v_s + swz<L::row>(krow, db * 2 + (mat & 1)), af);
#pragma unroll
                        for (int nt = 0; nt < NT; ++nt) {
                            float(&o)[4] = *reinterpret_cast<float(*)[4]>(acc + (nt * DB + db) * 4);
#pragma unroll
                            for (int x = 0; x < 3; ++x) mma_bf16_16816(o, af, b0[nt][x], b1[nt][x]);
                        }
                    }
                }
            } else {
                const unsigned char *vb = smem + L::stages + warp * L::stage + L::tile;
#pragma unroll 1
                for (int j0 = 0; j0 < kKT; j0 += 8) {
                    float v[8][DC];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        if constexpr (DC == 2) {
                            const float2 x = *reinterpret_cast<const float2 *>(vb + swz<L::row>(j0 + j, lane >> 1) + (lane & 1) * 8);
                            v[j][0] = x.x; v[j][1] = x.y;
                        } else {
                            const float4 x = *reinterpret_cast<const float4 *>(vb + swz<L::row>(j0 + j, lane));
                            v[j][0] = x.x; v[j][1] = x.y; v[j][2] = x.z; v[j][3] = x.w;
                        }
                    }
#pragma unroll
                    for (int g = 0; g < GP; ++g) {
                        const float4 pa = *reinterpret_cast<const float4 *>(st_w + g * kKT + j0), pb = *reinterpret_cast<const float4 *>(st_w + g * kKT + j0 + 4);
                        const float p[8] = {pa.x, pa.y, pa.z, pa.w, pb.x, pb.y, pb.z, pb.w};
#pragma unroll
                        for (int j = 0; j < 8; ++j)
#pragma unroll
                            for (int c = 0; c < DC; ++c) acc[g * DC + c] += p[j] * v[j][c];
                    }
                }
            }
            __syncwarp();                                      // the V tile and st_w have been read
            load_tile(v_s, Vu, it + kWarps);
            first_tile = false;
        }
        cp_async_wait<0>();
    }

    // ---------------- this warp's partial (m, l, O), the stage's memory being free now
    __syncwarp();
    float *wo = reinterpret_cast<float *>(smem + L::stages + warp * L::stage);
    if constexpr (BF) {
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            const int gr = gid + 8 * nt, gc = tig * 2 + 8 * nt;
            float l = lsum[nt];
            l += __shfl_xor_sync(0xffffffffu, l, 1);
            l += __shfl_xor_sync(0xffffffffu, l, 2);
            float m = -INFINITY;
#pragma unroll
            for (int g = 0; g < GP; ++g) m = g == gr ? mrun[g] : m;
            if (tig == 0 && gr < GP) { wml[(warp * GP + gr) * 2] = m; wml[(warp * GP + gr) * 2 + 1] = l; }
#pragma unroll
            for (int db = 0; db < DB; ++db) {
                const float *x = acc + (nt * DB + db) * 4;
                if (gc < GP) { wo[gc * D + db * 16 + gid] = x[0]; wo[gc * D + db * 16 + gid + 8] = x[2]; }
                if (gc + 1 < GP) { wo[(gc + 1) * D + db * 16 + gid] = x[1]; wo[(gc + 1) * D + db * 16 + gid + 8] = x[3]; }
            }
        }
    } else {
#pragma unroll
        for (int g = 0; g < GP; ++g) {
            const float l = warp_sum(lsum[g]);
            if (lane == 0) { wml[(warp * GP + g) * 2] = mrun[g]; wml[(warp * GP + g) * 2 + 1] = l; }
#pragma unroll
            for (int c = 0; c < DC; ++c) wo[g * D + lane * DC + c] = acc[g * DC + c];
        }
    }
    // self-inclusive Eq. 1: one more logit per head
    for (int g = warp; g < GP; g += kWarps) {
        float x = 0.f;
        for (int i = lane; i < D; i += 32) x += fin.q[g * D + i] * fin.k[i];
        x = warp_sum(x);
        if (lane == 0) fin.self[g] = x * a.scale2;
    }
    __syncthreads();
    // ---------------- merge of the warps' partials; output element idx belongs to the CTA idx / slice of the cluster
    const int slice = (GP * D + nsplit - 1) / nsplit;
    float *co = reinterpret_cast<float *>(smem + L::co);       // [cluster rank][slice]
    float *cml = reinterpret_cast<float *>(smem + L::cml);     // [cluster rank][GP][2]
    if (nsplit > 1) cluster_wait();                            // every CTA of the cluster has started
    for (int idx = tid; idx < GP * D; idx += kThreads) {
        const int g = idx / D;
        float m = -INFINITY;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) m = fmaxf(m, wml[(w * GP + g) * 2]);
        float o = 0.f, l = 0.f;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const float mw = wml[(w * GP + g) * 2], lw = wml[(w * GP + g) * 2 + 1];
            if (lw != 0.f) {                                             // a warp with keys (NaN if they are not numbers)
                const float f = exp2f(mw - m);
                o += reinterpret_cast<const float *>(smem + L::stages + w * L::stage)[idx] * f;
                l += lw * f;
            }
        }
        const int r = idx / slice, at = sp * slice + idx - r * slice;
        if (nsplit == 1) co[at] = o; else st_cluster(mapa(smem_u32(co + at), r), o);
        if (idx % D < nsplit) {                                // thread x of the head's row tells CTA x
            float *p = cml + (sp * GP + g) * 2;
            if (nsplit == 1) { p[0] = m; p[1] = l; }
            else { st_cluster(mapa(smem_u32(p), idx % D), m); st_cluster(mapa(smem_u32(p + 1), idx % D), l); }
        }
    }
    __syncwarp();
    if (nsplit > 1) { cluster_arrive(); cluster_wait(); } else __syncthreads();
    // soft-max statistics of the unit: sixteen lanes per head, one per CTA of the cluster; a CTA's factor takes the place of
    // its maximum
    for (int g0 = 0; g0 < GP; g0 += kThreads / kMaxCluster) {
        const int g = g0 + tid / kMaxCluster, r = tid % kMaxCluster;
        const bool live = g < GP, mine = live && r < nsplit;
        const float mr = mine ? cml[(r * GP + g) * 2] : -INFINITY, lr = mine ? cml[(r * GP + g) * 2 + 1] : 0.f, ms = live ? fin.self[g] : 0.f;
        float m = fmaxf(mr, ms);
#pragma unroll
        for (int o = kMaxCluster / 2; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        const float f = mr > -INFINITY ? exp2f(mr - m) : 0.f, fs = exp2f(ms - m);
        float l = lr * f + (r == 0 ? fs : 0.f);
#pragma unroll
        for (int o = kMaxCluster / 2; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (mine) cml[(r * GP + g) * 2] = f;
        if (live && r == 0) {
            fin.m[g] = fs;
            fin.l[g] = l;
            fin.c[g] = g < G ? m + log2f(l) : INFINITY;
        }
    }
    __syncthreads();
    T *out = static_cast<T *>(a.out) + (size_t)u * G * D;
    for (int i = tid; i < slice && sp * slice + i < G * D; i += kThreads) {
        const int idx = sp * slice + i, g = idx / D;
        float o = fin.m[g] * fin.v[idx % D];
#pragma unroll
        for (int r = 0; r < kMaxCluster; ++r)
            if (r < nsplit) o += co[r * slice + i] * cml[(r * GP + g) * 2];
        stf(out + idx, o / fin.l[g]);
    }
    if (CHECK && __syncthreads_or(moved)) {
        resum_moved<T, D>(a, u, k0, k1, rs_new, Fk, warp, kWarps, lane);
        __syncthreads();
    }
    // ---------------- Algorithm 1 / Eq. 7: add the new row's term to the scores of this CTA's keys, evict the minimum
    int e_slot = us.n, e_pos = -1;
    if (evict) {
        const long long thr = t - us.shift - R;
        unsigned long long best = ~0ull;
        int bslot = -1;
        constexpr int B = 4;                                   // slots per thread and round, their loads in flight together
        for (int kb = tid; kb < k1 - k0; kb += B * kThreads) {
            int p[B];
            float f0[B], x[B];
#pragma unroll
            for (int b = 0; b < B; ++b) {
                const int k = kb + b * kThreads;
                p[b] = k < k1 - k0 ? (local ? pk[k] : pos[k0 + k]) : 0x7fffffff;
                f0[b] = k < k1 - k0 ? Fk[k] : 0.f;
                x[b] = 0.f;
            }
#pragma unroll
            for (int g = 0; g < GP; ++g) {
                if (g >= G) break;
#pragma unroll
                for (int b = 0; b < B; ++b) {
                    const int k = kb + b * kThreads;
                    x[b] += exp2f((k < k1 - k0 ? sk[(size_t)g * sk_stride + k] : -INFINITY) - fin.c[g]);
                }
            }
#pragma unroll
            for (int b = 0; b < B; ++b) {
                const int k = kb + b * kThreads;
                if (k >= k1 - k0) continue;
                float f = -1.f;                                // window slot: not a candidate
                if ((long long)p[b] <= thr) {
                    f = fuse(a.fusion, f0[b], x[b]);
                    const unsigned long long key = rank_key(__float_as_uint(f), p[b]);
                    if (key < best) { best = key; bslot = k0 + k; }
                }
                Fu[k] = f;
            }
        }
        {   // the warp's smallest key: smallest score, then smallest inverted position (all keys differ)
            const unsigned hi = __reduce_min_sync(0xffffffffu, (unsigned)(best >> 32));
            const unsigned lo = __reduce_min_sync(0xffffffffu, (unsigned)(best >> 32) == hi ? (unsigned)best : 0xffffffffu);
            const unsigned long long wb = ((unsigned long long)hi << 32) | lo;
            bslot = __shfl_sync(0xffffffffu, bslot, __ffs(__ballot_sync(0xffffffffu, best == wb)) - 1);
            best = wb;
        }
        if (lane == 0) { fin.red_key[warp] = best; fin.red_slot[warp] = bslot; }
        __syncthreads();
        best = fin.red_key[0]; bslot = fin.red_slot[0];
#pragma unroll
        for (int w = 1; w < kWarps; ++w)
            if (fin.red_key[w] < best) { best = fin.red_key[w]; bslot = fin.red_slot[w]; }
        if (nsplit > 1) {                                      // CTA 0 elects the minimum and updates the cache
            unsigned long long *red = reinterpret_cast<unsigned long long *>(smem + L::cred);
            if (tid == 0) {
                st_cluster64(mapa(smem_u32(red + 2 * sp), 0), best);
                st_cluster64(mapa(smem_u32(red + 2 * sp + 1), 0), (unsigned long long)(unsigned)bslot);
            }
            __syncwarp();
            cluster_arrive();
            cluster_wait();
            if (sp != 0) return;
            best = red[0]; bslot = (int)red[1];
            for (int r = 1; r < nsplit; ++r)
                if (red[2 * r] < best) { best = red[2 * r]; bslot = (int)red[2 * r + 1]; }
        }
        e_slot = bslot;
        e_pos = (int)(0xFFFFFFFFu - (unsigned)(best & 0xFFFFFFFFull));     // the rank key carries the position
        if (a.T > 1) {          // coarse-grained eviction: append now, the compaction launch evicts
            e_slot = us.n;
            e_pos = -1;
        } else if (a.norm_current) {
            renormalise_after_eviction<T, D>(a, u, e_slot, rs_new, fin.c, reinterpret_cast<float *>(smem + L::q), tid, kThreads, 0);
        }
    } else if (sp != 0) {
        return;
    }
    if (e_slot >= a.cap) {      // no free slot: refuse to write beyond the unit's rows
        if (tid == 0) atomicCAS(&a.st->err, 0, (int)kErrCacheOverflow);
        return;
    }
    T *Kd = static_cast<T *>(a.K) + ((size_t)u * a.cap + e_slot) * D;
    T *Vd = static_cast<T *>(a.V) + ((size_t)u * a.cap + e_slot) * D;
    for (int i = tid; i < D; i += kThreads) {                  // (the floats are exact copies of the T values)
        stf(Kd + i, fin.k[i]);
        stf(Vd + i, fin.v[i]);
    }
    T *rq = static_cast<T *>(a.ring_q) + ((size_t)u * R + rs_new) * Gs * D;
    for (int i = tid; i < Gs * D; i += kThreads) stf(rq + i, fin.q[i]);
    if (tid < Gs) a.ring_c[((size_t)u * R + rs_new) * Gs + tid] = fin.c[tid];
    if (tid == 0) {
        a.pos[(size_t)u * a.cap + e_slot] = (int)(t - us.shift);
        if (kept) a.sum_pos[(size_t)u * a.cap + e_slot] = (int)(t - us.shift);
        if (e_pos < 0) a.F[(size_t)u * a.cap + e_slot] = -1.f;     // appended: a window slot
        a.evicted_pos[u] = e_pos;
    }
}

template <typename T, int D, int GP, bool CHECK>
cudaError_t launch_simt_g(const DecodeArgs &a, int nsplit, cudaStream_t stream)
{
    auto kern = decode_simt_kernel<T, D, GP, CHECK>;
    const int smem = SimtSmem<T, D, GP>::total;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess && nsplit > 8) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.U * nsplit);
    cfg.blockDim = dim3(SimtSmem<T, D, GP>::threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = nsplit;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = nsplit > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kern, a, nsplit);
}

template <typename T, int D, bool CHECK>
cudaError_t launch_simt_t(const DecodeArgs &a, int nsplit, cudaStream_t stream)
{
    switch (tc_padded_group(a.G)) {
        case 1: return launch_simt_g<T, D, 1, CHECK>(a, nsplit, stream);
        case 2: return launch_simt_g<T, D, 2, CHECK>(a, nsplit, stream);
        case 4: return launch_simt_g<T, D, 4, CHECK>(a, nsplit, stream);
        case 8: return launch_simt_g<T, D, 8, CHECK>(a, nsplit, stream);
        case 16: return launch_simt_g<T, D, 16, CHECK>(a, nsplit, stream);
    }
    return cudaErrorInvalidValue;
}

template <bool CHECK>
cudaError_t launch_simt_c(const DecodeArgs &a, int nsplit, bool f32, int D, cudaStream_t stream)
{
    if (f32) return D == 64 ? launch_simt_t<float, 64, CHECK>(a, nsplit, stream) : launch_simt_t<float, 128, CHECK>(a, nsplit, stream);
    return D == 64 ? launch_simt_t<__nv_bfloat16, 64, CHECK>(a, nsplit, stream) : launch_simt_t<__nv_bfloat16, 128, CHECK>(a, nsplit, stream);
}

}  // namespace

cudaError_t launch_decode_simt(const DecodeArgs &a, int nsplit, bool f32, int D, cudaStream_t stream)
{
    if (nsplit > kMaxCluster) return cudaErrorInvalidValue;
    return a.check_moved ? launch_simt_c<true>(a, nsplit, f32, D, stream) : launch_simt_c<false>(a, nsplit, f32, D, stream);
}

// Rows of a block are scored on every step and once more when it is finished: 16 where they cost scalar FMAs, 32 on the
// matrix instructions, as long as that makes no more than kMaxBlocks blocks.  0: no sums are kept.
int simt_block_slots(bool f32, int G, int R)
{
    const int g = tc_padded_group(G);
    int bs = (f32 ? 16 : 32) / g;
    if (bs < 1) bs = 1;
    while ((R + bs - 1) / bs > kMaxBlocks && 4 * bs * g <= 64) bs *= 2;        // two blocks are resident
    return (R + bs - 1) / bs > kMaxBlocks ? 0 : bs < R ? bs : R;
}

// Whether a launch over U units of a tcgen05 context is better off here, as clusters of as many CTAs as a unit has rounds of
// tiles: CTAs per unit, or 0.  (us per call, tcgen05 kernel -> here; R * G' = 128)
// - A layer's call starts ahead of the end of the one before it, so its chain of latencies is what counts: 8 units x 96 / 512 /
//   2048 / 4096 slots at G' = 4: 8.1 -> 7.2 / 11.0 -> 7.8 / 14.9 -> 10.9 / 20.0 -> 16.8.  The next layer's CTAs find room beside
//   this one's up to one CTA per SM.  At G' > 4 a CTA takes a whole SM: half as many leave that room (8 units x 1056, 72 CTAs:
//   19.9 -> 13.3), and more are worth it from 4 tiles per unit on while all clusters are resident at once: on the chip's seven
//   larger groups of SMs and the smaller eighth (12 units of 8 CTAs 19.6 -> 15.3, 14: 19.7 -> 16.1, 22 of 6: 19.7 -> 18.1; not so 16 of
//   8: 20.0 -> 26.5, 18 of 7: 19.9 -> 27.7, 16 of 9: 20.7 -> 26.6, 64 of 2: 14.4 -> 17.3).
// - A launch of the whole stack starts from nothing here, while the tcgen05 kernel sets itself up ahead of its wait and gives
//   units of up to eight tiles a CTA per tile: 8 units x 256 / 512 / 768: 9.2 -> 13.0 / 11.2 -> 12.9 / 12.2 -> 12.9.  Longer ones
//   it merges from several tiles per CTA, or more partials: 1056 / 2048: 13.8 -> 13.0 / 14.7 -> 14.0 (G' = 8: 20.0 -> 17.3 at 1056).
int simt_small_splits(int U, int G, int R, int bs, int nblk, int cap, bool layer)
{
    const int g = tc_padded_group(G);
    if ((nblk > 1 ? 2 : 1) * bs * g > SimtSmem<__nv_bfloat16, 128, 1>::rows) return 0;
    const int rounds = (cap + kRound - 1) / kRound, s = rounds < kMaxCluster ? rounds : kMaxCluster;
    if (!layer && rounds <= 8) return 0;
    const bool fits = (long long)U * s <= (g > 4 ? 74 : 148) || (layer && g > 4 && s >= 4 && U <= 18 / s * 7 + 11 / s);
    return fits && rounds <= 2 * kMaxCluster ? s : 0;
}

// CTAs per unit: enough to fill the chip (two CTAs per SM), at least one round of tiles each.
int simt_default_splits(int U, int cap)
{
    int s = (2 * 148 + U - 1) / U;
    const int max_s = (cap + kRound - 1) / kRound;
    if (s > max_s) s = max_s;
    if (s > kMaxCluster) s = kMaxCluster;
    return s < 1 ? 1 : s;
}

}  // namespace mkv
