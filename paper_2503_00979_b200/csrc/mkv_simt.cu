// Warp-level decode kernel: any dtype (bf16 / f32), head_dim 64 or 128, any GQA group and window size.  It is the
// kernel of the f32 mode, of head_dim 64 and of windows beyond the tcgen05 kernel's range, and serves as an on-device
// cross-check of that kernel.
//
// One CTA handles one (unit, split): a contiguous range of the unit's cached keys.  Its eight warps take 32-key tiles in
// turn and do not wait for one another; a warp copies its tile into shared memory of its own (cp.async, 16-byte chunks
// swizzled by row), the next K tile while P.V runs and the next V tile while it is scored.  Per tile:
//   scores   logits of the tile's keys against the resident ring rows: bf16 on mma.sync (keys are the rows of the
//            A operand), f32 with one key per lane.  Rows other than the new query turn into frozen weights
//            exp2(s - c_row), are summed over the GQA group and fused over the window (Eq. 4-6, Algorithm 1).  Resident
//            are the block of ring slots that is being filled and, on the step that opens it, the block before it; the
//            rest of the window comes from the sums in slab and pre (DecodeArgs::slab).  Without kept sums (CURRENT
//            normalisation, windows of more than kMaxBlocks blocks) the whole ring passes through, kRows rows at a time.
//   attend   soft-max of the new query over the tile, continued online, and P.V (Eq. 1): bf16 on mma.sync with P in
//            three bf16 terms (24 mantissa bits), f32 with one slice of the head dimension per lane.
// The warps' partials are merged in shared memory; the CTA that finishes a unit last merges the splits, adds the new
// row's term to the scores, selects and appends (Eq. 7).
//
// Bound by HBM for bf16 and, nearly, by FMA issue for f32.  The kernel before it scored all R*G rows with scalar FMAs and
// met at CTA barriers for every 32 keys: 512 units x 1056 slots, bf16, d = 64, R*G = 128 took 837 us per step, now
// 67 (issue slots 42 % busy, 1600 instructions per warp tile); 2 units x 80 slots, f32, d = 64 30.6, now 12.2.
#include "mkv_common.cuh"
#include "mkv_kernels.h"
#include "mkv_sm100.cuh"

namespace mkv {

namespace {

constexpr int kWarps = 8;
constexpr int kThreads = 32 * kWarps;
constexpr int kKT = 32;              // keys per warp tile
constexpr int kRows = 64;            // resident ring rows
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
    static constexpr int row = D * (int)sizeof(T);             // bytes of a K, V or query row
    static constexpr int tile = kKT * row;
    static constexpr bool v_staged = sizeof(T) == 2;
    static constexpr int stage = tile * (v_staged ? 2 : 1);    // per warp; later the warp's partial output [GP][D] floats
    static constexpr int st_w = GP * kKT + 4 * GP + kKT;       // floats per warp: logits or weights, factors, references, F
    static constexpr int q = 0;
    static constexpr int stages = q + kRows * row;
    static constexpr int negc = stages + kWarps * stage;
    static constexpr int stw = negc + kRows * 4;
    static constexpr int wml = stw + kWarps * st_w * 4;
    static constexpr int fin = wml + kWarps * GP * 2 * 4;      // q [GP][D], k_new [D], v_new [D], self, m, l, c [GP], reduction
    static constexpr int total = fin + (GP * D + 2 * D + 4 * GP + D + 3 * 32) * 4;
    static_assert(stage >= GP * D * 4, "a warp's partial fits its stage");
};

// epilogue scratch inside the `fin` area
template <int D, int GP> struct Fin {
    float *q, *k, *v, *self, *m, *l, *c, *krow;
    unsigned long long *red_key;
    int *red_slot;
    __device__ explicit Fin(float *p)
    {
        q = p; k = q + GP * D; v = k + D;
        self = v + D; m = self + GP; l = m + GP; c = l + GP;
        krow = c + GP;
        red_key = reinterpret_cast<unsigned long long *>(krow + D);
        red_slot = reinterpret_cast<int *>(red_key + 32);
    }
};

// Epilogue of a unit (the whole CTA).  One split: the merged partial is in shared memory (cml [GP][2], osm [GP][D]);
// several: in global memory, written by other CTAs, read past L1.
template <typename T, int D, int GP>
__device__ void finish_unit(const DecodeArgs &a, int u, long long t, int n, int nseg, bool evict, int shift, const Fin<D, GP> &s,
                            const float *cml, const float *osm, int tid)
{
    const int G = a.G, lane = tid & 31, warp = tid >> 5;
    const float *pml = a.part_ml + (size_t)u * a.splits * G * 2;
    const float *po = a.part_o + (size_t)u * a.splits * G * D;
    if (tid < G) {
        float m = s.self[tid], l;
        if (nseg == 1) {
            m = fmaxf(m, cml[tid * 2]);
            l = exp2f(s.self[tid] - m) + cml[tid * 2 + 1] * exp2f(cml[tid * 2] - m);
        } else {
            for (int i = 0; i < nseg; ++i) m = fmaxf(m, __ldcg(pml + (i * G + tid) * 2));
            l = exp2f(s.self[tid] - m);
            for (int i = 0; i < nseg; ++i) l += __ldcg(pml + (i * G + tid) * 2 + 1) * exp2f(__ldcg(pml + (i * G + tid) * 2) - m);
        }
        s.m[tid] = m;
        s.l[tid] = l;
        s.c[tid] = m + log2f(l);
    }
    __syncthreads();
    T *out = static_cast<T *>(a.out) + (size_t)u * G * D;
    for (int idx = tid; idx < G * D; idx += kThreads) {
        const int g = idx / D, dd = idx % D;
        const float m = s.m[g];
        float o = exp2f(s.self[g] - m) * s.v[dd];
        if (nseg == 1) {
            o += osm[idx] * exp2f(cml[g * 2] - m);
        } else {
            for (int i0 = 0; i0 < nseg; i0 += 4) {
                float v[4], w[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    v[i] = i0 + i < nseg ? __ldcg(po + ((i0 + i) * G + g) * D + dd) : 0.f;
                    w[i] = i0 + i < nseg ? __ldcg(pml + ((i0 + i) * G + g) * 2) : -INFINITY;
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) o += v[i] * exp2f(w[i] - m);
            }
        }
        stf(out + idx, o / s.l[g]);
    }
    // Algorithm 1 / Eq. 7: add the new row's term to the fused scores, evict the minimum
    int *pos = a.pos + (size_t)u * a.cap;
    float *F = a.F + (size_t)u * a.cap;
    const int rs = (int)(t % a.R);
    int e_slot = n, e_pos = -1;
    if (evict) {
        const float *sn = a.s_new + (size_t)u * G * a.cap;
        const long long thr = t - shift - a.R;
        unsigned long long best = ~0ull;
        int bslot = -1;
        constexpr int B = 4;
        for (int kb = tid; kb < n; kb += B * kThreads) {
            int p[B];
            float f0[B], x[B];
#pragma unroll
            for (int b = 0; b < B; ++b) {
                const int k = kb + b * kThreads;
                p[b] = k < n ? pos[k] : 0x7fffffff;
                f0[b] = k < n ? __ldcg(F + k) : 0.f;
                x[b] = 0.f;
            }
#pragma unroll
            for (int g = 0; g < GP; ++g) {
                if (g >= G) break;
#pragma unroll
                for (int b = 0; b < B; ++b) {
                    const int k = kb + b * kThreads;
                    x[b] += exp2f((k < n ? __ldcg(sn + (size_t)g * a.cap + k) : -INFINITY) - s.c[g]);
                }
            }
#pragma unroll
            for (int b = 0; b < B; ++b) {
                const int k = kb + b * kThreads;
                if (k >= n) continue;
                if ((long long)p[b] <= thr) {
                    const float f = fuse(a.fusion, f0[b], x[b]);
                    F[k] = f;
                    const unsigned long long key = rank_key(__float_as_uint(f), p[b]);
                    if (key < best) { best = key; bslot = k; }
                } else {
                    F[k] = -1.f;   // window slot: not a candidate
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long ok = __shfl_xor_sync(0xffffffffu, best, o);
            const int os = __shfl_xor_sync(0xffffffffu, bslot, o);
            if (ok < best) { best = ok; bslot = os; }
        }
        if (lane == 0) { s.red_key[warp] = best; s.red_slot[warp] = bslot; }
        __syncthreads();
        best = s.red_key[0]; bslot = s.red_slot[0];
#pragma unroll
        for (int w = 1; w < kWarps; ++w)
            if (s.red_key[w] < best) { best = s.red_key[w]; bslot = s.red_slot[w]; }
        e_slot = bslot;
        e_pos = (int)(0xFFFFFFFFu - (unsigned)(best & 0xFFFFFFFFull));     // the rank key carries the position
        if (a.T > 1) {          // coarse-grained eviction: append now, the compaction launch evicts
            e_slot = n;
            e_pos = -1;
            if (tid == 0 && n < a.cap) F[n] = -1.f;
        } else if (a.norm_current) {
            renormalise_after_eviction<T, D>(a, u, e_slot, rs, s.c, s.krow, tid, kThreads, 0);
        }
    }
    if (e_slot >= a.cap) {      // no free slot: refuse to write beyond the unit's rows
        if (tid == 0) { atomicCAS(&a.st->err, 0, (int)kErrCacheOverflow); a.ticket[u] = 0; }
        return;
    }
    T *Kd = static_cast<T *>(a.K) + ((size_t)u * a.cap + e_slot) * D;
    T *Vd = static_cast<T *>(a.V) + ((size_t)u * a.cap + e_slot) * D;
    if (tid < D) stf(Kd + tid, s.k[tid]);                    // (the floats are exact copies of the T values)
    else if (tid < 2 * D) stf(Vd + tid - D, s.v[tid - D]);
    T *rq = static_cast<T *>(a.ring_q) + ((size_t)u * a.R + rs) * G * D;
    for (int i = tid; i < G * D; i += kThreads) stf(rq + i, s.q[i]);
    if (tid < G) a.ring_c[((size_t)u * a.R + rs) * G + tid] = s.c[tid];
    if (tid == 0) {
        pos[e_slot] = (int)(t - shift);
        if (a.nblk > 1) a.sum_pos[(size_t)u * a.cap + e_slot] = (int)(t - shift);
        a.evicted_pos[u] = e_pos;
        a.ticket[u] = 0;
    }
}

// GP: the group padded to a power of two (padding heads: zero query, weight 0)
template <typename T, int D, int GP>
__global__ void __launch_bounds__(kThreads, D == 64 ? 2 : 1) decode_simt_kernel(const __grid_constant__ DecodeArgs a, const int nsplit)
{
    using L = SimtSmem<T, D, GP>;
    constexpr bool BF = sizeof(T) == 2;
    constexpr int CH = L::row / 16, EP = 16 / (int)sizeof(T);   // chunks per row, elements per chunk
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ int is_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int G = a.G, R = a.R;
    const int u = blockIdx.x / nsplit, sp = blockIdx.x % nsplit;
    const uint32_t q_s = smem_u32(smem + L::q), k_s = smem_u32(smem + L::stages) + warp * L::stage, v_s = k_s + L::tile;
    float *negc = reinterpret_cast<float *>(smem + L::negc);
    float *st_w = reinterpret_cast<float *>(smem + L::stw) + warp * L::st_w;     // [g][key]
    float *fac = st_w + GP * kKT, *mref = fac + GP, *fsm = mref + GP;
    float *wml = reinterpret_cast<float *>(smem + L::wml);
    const Fin<D, GP> fin(reinterpret_cast<float *>(smem + L::fin));

    // see the tcgen05 kernel: the grid before this one is complete behind the wait, the next one may start and park there
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const long long t = a.st->t;
    const int n = a.st->n, steps_done = a.st->steps;
    // the new token's tensors, as floats (read once; the epilogue writes them to the cache)
    {
        const T *q = static_cast<const T *>(a.q) + (size_t)u * G * D;
        for (int i = tid; i < GP * D; i += kThreads) fin.q[i] = i < G * D ? ldf(q + i) : 0.f;
        if (tid < D) fin.k[tid] = ldf(static_cast<const T *>(a.k_new) + (size_t)u * D + tid);
        else if (tid < 2 * D) fin.v[tid - D] = ldf(static_cast<const T *>(a.v_new) + (size_t)u * D + tid - D);
    }
    const bool evict_all = step_scores(t, n, steps_done, R, a.C, a.T);
    // the unit's own fill and policy decision (they differ from the uniform ones only between batch rows whose
    // prompts had different lengths); the splits are laid out over the largest fill
    const UnitStep us = unit_step(a, u, t, n, steps_done, evict_all);
    const bool evict = us.evict;
    int active;
    const int per = split_len(n, nsplit, kKT, &active);
    const int k0 = sp * per, k1 = min(us.n, k0 + per);
    const int ntile = (max(0, min(n, k0 + per) - k0) + kKT - 1) / kKT;
    const int rs_new = (int)(t % R);
    const bool kept = a.nblk > 1, fold = step_opens_block(t, R, a.bs, a.nblk);
    const int jb = rs_new / a.bs, j_old = open_block(t, R, a.bs);
    // ring slots that pass through: the open block (the whole ring without kept sums), or the new query's alone
    const bool score = evict || fold;
    const int slots_per = kRows / GP;
    const int s_begin = score ? jb * a.bs : rs_new, s_end = score ? min(R, (jb + 1) * a.bs) : rs_new + 1;
    const T *Ku = static_cast<const T *>(a.K) + (size_t)u * a.cap * D, *Vu = static_cast<const T *>(a.V) + (size_t)u * a.cap * D;
    float *s_new = a.s_new + (size_t)u * G * a.cap, *Fu = a.F + (size_t)u * a.cap;
    float *slab = kept ? a.slab + (size_t)u * a.nblk * a.cap : nullptr, *pre = kept ? a.pre + (size_t)u * a.cap : nullptr;

    auto load_tile = [&](uint32_t dst, const T *base, int it) {
        if (it < ntile) {
            const int key0 = k0 + it * kKT;
#pragma unroll
            for (int i = 0; i < CH; ++i) {
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
    bool first_tile = true;

    for (int s0 = s_begin; s0 < s_end; s0 += slots_per) {
        const int s1 = min(s_end, s0 + slots_per);
        const bool attend = rs_new >= s0 && rs_new < s1;       // this pass holds the new query
        load_tile(k_s, Ku, warp);
        if (BF) {
            if (attend) load_tile(v_s, Vu, warp); else cp_async_commit();
        }
        // rows of this pass: the slots s0 .. s1 - 1, padded to whole n-tiles, then the finished block's (fold)
        const int nA = (s1 - s0) * GP, rA = (nA + 7) & ~7;
        const int f0 = j_old * a.bs, nB = fold ? (min(R, f0 + a.bs) - f0) * GP : 0, nrow = rA + ((nB + 7) & ~7);
        const int rl0 = (rs_new - s0) * GP;                    // the new query's rows (attend)
        const T *ring_q = static_cast<const T *>(a.ring_q) + (size_t)u * R * G * D;
        if (s0 != s_begin) __syncthreads();                    // the rows of the pass before are done with
        for (int i = tid; i < nrow * CH; i += kThreads) {
            const int row = i / CH, ch = i % CH;
            const bool inA = row < nA, inB = row >= rA && row < rA + nB;
            const int rr = inA ? row : row - rA, slot = (inA ? s0 : f0) + rr / GP, g = rr % GP;
            uint4 v = make_uint4(0, 0, 0, 0);
            if ((inA || inB) && g < G) {
                const T *src = slot == rs_new ? static_cast<const T *>(a.q) + ((size_t)u * G + g) * D : ring_q + ((size_t)slot * G + g) * D;
                // (the caller's q need not be 16-byte aligned)
                if (slot == rs_new && (reinterpret_cast<uintptr_t>(a.q) & 15) != 0) {
                    T *e = reinterpret_cast<T *>(&v);
#pragma unroll
                    for (int x = 0; x < EP; ++x) e[x] = src[ch * EP + x];
                } else {
                    v = reinterpret_cast<const uint4 *>(src)[ch];
                }
            }
            *reinterpret_cast<uint4 *>(smem + L::q + (BF ? swz<L::row>(row, ch) : (uint32_t)(row * L::row + ch * 16))) = v;
        }
        for (int row = tid; row < nrow; row += kThreads) {
            const bool inA = row < nA, inB = row >= rA && row < rA + nB;
            const int rr = inA ? row : row - rA, slot = (inA ? s0 : f0) + rr / GP, g = rr % GP;
            negc[row] = (inA || inB) && g < G && slot != rs_new ? -a.ring_c[((size_t)u * R + slot) * G + g] : -INFINITY;
        }
        __syncthreads();
        if (s0 == s_begin && tid == 0) {
            // Every thread holds its copy of the step state: the last CTA to get here advances it for the next launch.
            __threadfence();
            if (atomicAdd(&a.st->done, 1u) == gridDim.x - 1) advance_state(a, t, n, steps_done, evict_all);
        }

        for (int it = warp; it < ntile; it += kWarps) {
            const int key = k0 + it * kKT + lane;
            const bool valid = key < k1;
            float f_pre = 0.f, f_rest = 0.f;                   // the rest of the window's fused score
            if (kept && score && valid) {
                if (jb > (fold ? 1 : 0)) f_pre = __ldcg(pre + key);
                if ((jb > 0 || !fold) && jb + 1 < a.nblk) f_rest = __ldcg(slab + (size_t)(jb + 1) * a.cap + key);
                f_rest = fuse(a.fusion, f_rest, f_pre);
            }
            cp_async_wait<BF ? 1 : 0>();
            __syncwarp();
            // ---------------- logits and fused scores
            float F = 0.f, S = 0.f;
            float s2[GP];
            if constexpr (BF) {
                uint32_t af[2][D / 16][4];
#pragma unroll
                for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks) ldmatrix_x4(k_s + swz<L::row>(mt * 16 + (lane & 15), ks * 2 + (lane >> 4)), af[mt][ks]);
                float fk[2][2] = {{0.f, 0.f}, {0.f, 0.f}}, pend[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
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
                    const int r = nt * 8 + tig * 2;
                    if (attend && nt * 8 < rl0 + GP && nt * 8 + 8 > rl0) {             // uniform over the warp
#pragma unroll
                        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const int g = r + (e & 1) - rl0;
                                if (g >= 0 && g < GP) st_w[g * kKT + mt * 16 + gid + (e >> 1) * 8] = c[mt][e] * a.scale2;
                            }
                    }
                    if (!score) continue;
                    if (nt * 8 == rA) {                        // the open block is done, the finished one follows
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
                        F = fsm[lane];
                        __syncwarp();
                    }
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
                if (score) {
#pragma unroll
                    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            float x = fk[mt][h];
                            x = fuse(a.fusion, x, __shfl_xor_sync(0xffffffffu, x, 1));
                            x = fuse(a.fusion, x, __shfl_xor_sync(0xffffffffu, x, 2));
                            if (tig == 0) fsm[mt * 16 + gid + h * 8] = x;
                        }
                }
                __syncwarp();
                if (score) { if (nrow > rA) S = fsm[lane]; else F = fsm[lane]; }
                if (attend)
#pragma unroll
                    for (int g = 0; g < GP; ++g) s2[g] = st_w[g * kKT + lane];
            } else {
                const unsigned char *qb = smem + L::q;
                const unsigned char *kb = smem + L::stages + warp * L::stage;
                constexpr int RB = GP > 8 ? GP : 8;            // rows at a time: whole slots
                for (int r0 = 0; r0 < nrow; r0 += RB) {
                    float x[RB];
#pragma unroll
                    for (int r = 0; r < RB; ++r) x[r] = 0.f;
#pragma unroll 4
                    for (int ch = 0; ch < CH; ++ch) {
                        const float4 kv = *reinterpret_cast<const float4 *>(kb + swz<L::row>(lane, ch));
#pragma unroll
                        for (int r = 0; r < RB; ++r) {
                            const float4 qv = *reinterpret_cast<const float4 *>(qb + (r0 + r) * L::row + ch * 16);
                            x[r] += kv.x * qv.x + kv.y * qv.y + kv.z * qv.z + kv.w * qv.w;
                        }
                    }
                    if (attend && r0 < rl0 + GP && r0 + RB > rl0)
#pragma unroll
                        for (int r = 0; r < RB; ++r)
                            if (r0 + r >= rl0 && r0 + r < rl0 + GP) st_w[(r0 + r - rl0) * kKT + lane] = x[r] * a.scale2;
                    if (!score) continue;
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
                if (attend)
#pragma unroll
                    for (int g = 0; g < GP; ++g) s2[g] = st_w[g * kKT + lane];
            }
            __syncwarp();                                      // the K tile has been read
            load_tile(k_s, Ku, it + kWarps);
            if (score && valid) {
                if (fold) {                                    // the finished block of the ring, scored for good
                    float *sk = slab + key;
                    sk[(size_t)j_old * a.cap] = S;
                    if (jb > 0) {
                        pre[key] = fuse(a.fusion, f_pre, S);
                    } else {                                   // a lap ends: its single blocks become the sums of all later ones
                        for (int i0 = a.nblk - 2; i0 >= 1; i0 -= 4) {
                            float v[4];
#pragma unroll
                            for (int b = 0; b < 4; ++b) v[b] = i0 - b >= 1 ? __ldcg(sk + (size_t)(i0 - b) * a.cap) : 0.f;
#pragma unroll
                            for (int b = 0; b < 4; ++b)
                                if (i0 - b >= 1) {
                                    S = fuse(a.fusion, S, v[b]);
                                    sk[(size_t)(i0 - b) * a.cap] = S;
                                }
                        }
                    }
                    f_rest = fuse(a.fusion, f_rest, S);
                }
                if (evict) {
                    F = fuse(a.fusion, F, s0 == s_begin ? f_rest : Fu[key]);
                    Fu[key] = F;
                }
            }
            if (!attend) {
                if (BF) cp_async_commit();                     // keeps the count of copy groups
                continue;
            }
            // ---------------- online soft-max of the new row over this warp's keys (Eq. 1)
            bool changed = false;
#pragma unroll
            for (int g = 0; g < GP; ++g) {
                const float s = valid ? s2[g] : -INFINITY;
                s2[g] = s;
                if (valid && evict && g < G) s_new[(size_t)g * a.cap + key] = s;
                const float mn = fmaxf(mrun[g], warp_max(s));
                const float f = mn == mrun[g] ? 1.f : exp2f(mrun[g] - mn);
                changed |= mn != mrun[g];
                mrun[g] = mn;
                if constexpr (BF) {
                    st_w[g * kKT + lane] = s;
                    if (lane == 0) { fac[g] = f; mref[g] = mn == -INFINITY ? 0.f : mn; }
                } else {
                    const float p = mn == -INFINITY ? 0.f : exp2f(s - mn);
                    st_w[g * kKT + lane] = p;
                    lsum[g] = lsum[g] * f + p;
                    if (f != 1.f && !first_tile)
#pragma unroll
                        for (int c = 0; c < DC; ++c) acc[g * DC + c] *= f;
                }
            }
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
                cp_async_wait<1>();                            // this tile's V (the next K may still be on its way)
                __syncwarp();
                // O^T[d][g] += V^T[d][keys] . P^T[keys][g]
#pragma unroll
                for (int ks = 0; ks < 2; ++ks) {
                    uint32_t b0[NT][3], b1[NT][3];
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt) {
                        const int gr = gid + 8 * nt;
                        const bool live = gr < GP;
                        const int grc = live ? gr : 0;
                        const float *p = st_w + grc * kKT + ks * 16 + tig * 2;
                        const float m = mref[grc];
                        float p0 = exp2f(p[0] - m), p1 = exp2f(p[1] - m), p2 = exp2f(p[8] - m), p3 = exp2f(p[9] - m);
                        p0 = live ? p0 : 0.f; p1 = live ? p1 : 0.f; p2 = live ? p2 : 0.f; p3 = live ? p3 : 0.f;
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
                __syncwarp();                                  // the V tile has been read
                load_tile(v_s, Vu, it + kWarps);
            } else {
                const float *Vp = reinterpret_cast<const float *>(Vu) + (size_t)(k0 + it * kKT) * D + lane * DC;
                const int cnt = min(kKT, k1 - (k0 + it * kKT));
#pragma unroll
                for (int j0 = 0; j0 < kKT; j0 += 8) {
                    float v[8][DC];
#pragma unroll
                    for (int j = 0; j < 8; ++j)
#pragma unroll
                        for (int c = 0; c < DC; c += 2) {
                            const float2 x = j0 + j < cnt ? *reinterpret_cast<const float2 *>(Vp + (size_t)(j0 + j) * D + c) : make_float2(0.f, 0.f);
                            v[j][c] = x.x; v[j][c + 1] = x.y;
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
                __syncwarp();                                  // st_w is free again
            }
            first_tile = false;
        }
        cp_async_wait<0>();
    }

    // self-inclusive Eq. 1: one more logit per head
    for (int g = warp; g < GP; g += kWarps) {
        float x = 0.f;
        for (int i = lane; i < D; i += 32) x += fin.q[g * D + i] * fin.k[i];
        x = warp_sum(x);
        if (lane == 0) fin.self[g] = x * a.scale2;
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
    __syncthreads();
    if (k0 >= n) return;                                       // no keys for this split (only ever the state was counted)
    // merge of the eight partials: element idx is read and written by the same thread
    float *osm = reinterpret_cast<float *>(smem + L::q);       // [GP][D] in the query rows' place
    static_assert(kRows * L::row >= GP * D * 4, "the merged output fits the query rows");
    float *cml = reinterpret_cast<float *>(smem + L::negc);    // [GP][2]
    for (int idx = tid; idx < GP * D; idx += kThreads) {
        const int g = idx / D;
        float m = -INFINITY;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) m = fmaxf(m, wml[(w * GP + g) * 2]);
        float o = 0.f;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const float mw = wml[(w * GP + g) * 2];
            if (mw > -INFINITY) o += reinterpret_cast<const float *>(smem + L::stages + w * L::stage)[idx] * exp2f(mw - m);
        }
        osm[idx] = o;
        if (idx % D == 0) {
            float l = 0.f;
            for (int w = 0; w < kWarps; ++w) {
                const float mw = wml[(w * GP + g) * 2];
                if (mw > -INFINITY) l += wml[(w * GP + g) * 2 + 1] * exp2f(mw - m);
            }
            cml[g * 2] = m;
            cml[g * 2 + 1] = l;
        }
    }
    __syncthreads();
    if (active > 1) {
        float *pml = a.part_ml + ((size_t)u * a.splits + sp) * G * 2, *po = a.part_o + ((size_t)u * a.splits + sp) * G * D;
        for (int idx = tid; idx < G * D; idx += kThreads) po[idx] = osm[idx];
        if (tid < 2 * G) pml[tid] = cml[tid];
        __threadfence();
        __syncthreads();
        if (tid == 0) is_last = atomicAdd(&a.ticket[u], 1) == active - 1;
        __syncthreads();
        if (!is_last) return;
        __threadfence();
    }
    finish_unit<T, D, GP>(a, u, t, us.n, active, evict, us.shift, fin, cml, osm, tid);
}

template <typename T, int D, int GP>
cudaError_t launch_simt_g(const DecodeArgs &a, int nsplit, cudaStream_t stream)
{
    auto kern = decode_simt_kernel<T, D, GP>;
    const int smem = SimtSmem<T, D, GP>::total;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.U * nsplit);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, a, nsplit);
}

template <typename T, int D>
cudaError_t launch_simt_t(const DecodeArgs &a, int nsplit, cudaStream_t stream)
{
    switch (tc_padded_group(a.G)) {
        case 1: return launch_simt_g<T, D, 1>(a, nsplit, stream);
        case 2: return launch_simt_g<T, D, 2>(a, nsplit, stream);
        case 4: return launch_simt_g<T, D, 4>(a, nsplit, stream);
        case 8: return launch_simt_g<T, D, 8>(a, nsplit, stream);
        case 16: return launch_simt_g<T, D, 16>(a, nsplit, stream);
    }
    return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_decode_simt(const DecodeArgs &a, int nsplit, bool f32, int D, cudaStream_t stream)
{
    if (f32) return D == 64 ? launch_simt_t<float, 64>(a, nsplit, stream) : launch_simt_t<float, 128>(a, nsplit, stream);
    return D == 64 ? launch_simt_t<__nv_bfloat16, 64>(a, nsplit, stream) : launch_simt_t<__nv_bfloat16, 128>(a, nsplit, stream);
}

// Rows of a block are scored on every step and once more when it is finished: 16 where they cost scalar FMAs, 32 on the
// matrix instructions, as long as that makes no more than kMaxBlocks blocks.  0: no sums are kept.
int simt_block_slots(bool f32, int G, int R)
{
    const int g = tc_padded_group(G);
    int bs = (f32 ? 16 : 32) / g;
    if (bs < 1) bs = 1;
    while ((R + bs - 1) / bs > kMaxBlocks && 4 * bs * g <= kRows) bs *= 2;
    return (R + bs - 1) / bs > kMaxBlocks ? 0 : bs < R ? bs : R;
}

// CTAs per unit: enough to fill the chip (two CTAs per SM), at least one round of tiles (256 keys) each.
int simt_default_splits(int U, int cap)
{
    int s = (2 * 148 + U - 1) / U;
    const int max_s = (cap + kWarps * kKT - 1) / (kWarps * kKT);
    if (s > max_s) s = max_s;
    return s < 1 ? 1 : s;
}

}  // namespace mkv
