// Prompt phase of MorphKV (set-up, not part of the per-token hot path).
//
// The paper states no prefill procedure; this is one application of Algorithm 1 with the
// whole prompt as the cache G_i: the last Rw = min(R, P) prompt tokens are the window, each
// window row's attention profile is its causal soft-max over all prompt keys (Eq. 1), every
// older prompt token gets the fused score of Eq. 4-6 (group sum first), and the C best are
// kept beside the window (Eq. 7).  The selection is a block-wide radix select over
// (score, position) keys, so ties keep the lower position deterministically.
#include <mutex>

#include "mkv_common.cuh"
#include "mkv_kernels.h"

namespace mkv {

namespace {

constexpr int kPT = 256;    // threads per CTA
constexpr int kPK = 32;     // keys per tile
constexpr int kPR = 64;     // window rows per sub-block
constexpr size_t kScratchWords = 3;      // ticket, finished CTAs and error word of the scoring kernels

__device__ __forceinline__ void ld4(const float *p, float (&o)[4])
{
    const float4 v = *reinterpret_cast<const float4 *>(p);
    o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
}
__device__ __forceinline__ void ld4(const __nv_bfloat16 *p, float (&o)[4])
{
    const uint2 v = *reinterpret_cast<const uint2 *>(p);
    o[0] = __uint_as_float(v.x << 16); o[1] = __uint_as_float(v.x & 0xffff0000u);
    o[2] = __uint_as_float(v.y << 16); o[3] = __uint_as_float(v.y & 0xffff0000u);
}

// (launched in full stream order: what it waits for is complete for the kernels behind it too)
__global__ void init_arena_kernel(DecodeArgs a, int *words, int n_words)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < (size_t)n_words) words[i] = 0;
    const size_t ncap = (size_t)a.U * a.cap;
    if (i < ncap) { a.pos[i] = -1; a.F[i] = 0.f; }
    if (i < ncap && a.nblk > 1) a.sum_pos[i] = -1;
    if (i < (size_t)a.U * a.R * a.G) a.ring_c[i] = INFINITY;   // empty ring row: weight 0
    if (i < (size_t)a.U) { a.ticket[i] = 0; a.evicted_pos[i] = -1; }
}

// S[ub][row = i*G + g][j] = log2-domain logit of window row (i, g) against prompt key j,
// -inf where j lies after the row's own position (causal mask).
template <typename T, int D>
__global__ void __launch_bounds__(kPT) prefill_logits_kernel(const T *__restrict__ k, const T *__restrict__ qwin,
                                                             float *__restrict__ S, int ub0, int P, int Rw, int G,
                                                             float scale2, int Ps, int Rws, RowMap rowmap)
{
    // P, Rw: of the longest prompt, which S is laid out for.  Ps, Rws: tokens per unit in k and entries per head in qwin
    // as laid out by the caller (P and Rw unless the batch rows' prompts have different lengths and the tensors are
    // padded)
    extern __shared__ __align__(16) float psm[];
    float *Ks = psm, *Qs = psm + kPK * (D + 4), *Ssm = Qs + kPR * (D + 4);
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int u = ub0 + blockIdx.y, kt = blockIdx.x * kPK;
    const int Srows = Rw * G, SP = P;
    P -= rowmap(u);
    Rw = min(Rw, P);
    const int rows = Rw * G;
    if (kt >= P) return;
    constexpr int KS = D + 4, C4 = D / 4;
    const T *Ku = k + (size_t)u * Ps * D;
    for (int idx = tid; idx < kPK * C4; idx += kPT) {
        const int key = idx / C4, c4 = idx % C4;
        float v[4] = {0.f, 0.f, 0.f, 0.f};
        if (kt + key < P) ld4(Ku + (size_t)(kt + key) * D + c4 * 4, v);
        *reinterpret_cast<float4 *>(Ks + key * KS + c4 * 4) = make_float4(v[0], v[1], v[2], v[3]);
    }
    for (int r0 = 0; r0 < rows; r0 += kPR) {
        const int nr = min(kPR, rows - r0);
        __syncthreads();
        for (int idx = tid; idx < nr * C4; idx += kPT) {
            const int rl = idx / C4, c4 = idx % C4;
            const int row = r0 + rl, i = row / G, g = row % G;
            float v[4];
            ld4(qwin + (((size_t)u * G + g) * Rws + i) * D + c4 * 4, v);
            *reinterpret_cast<float4 *>(Qs + rl * KS + c4 * 4) = make_float4(v[0], v[1], v[2], v[3]);
        }
        __syncthreads();
        float acc[2][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) { acc[0][i] = 0.f; acc[1][i] = 0.f; }
        const float *ka = Ks + ty * KS, *kb = Ks + (ty + 16) * KS;
        const float *qr[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) qr[i] = Qs + ((tx + 16 * i) < nr ? (tx + 16 * i) : 0) * KS;
#pragma unroll 4
        for (int dd = 0; dd < D; dd += 4) {
            const float4 x = *reinterpret_cast<const float4 *>(ka + dd);
            const float4 y = *reinterpret_cast<const float4 *>(kb + dd);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 qv = *reinterpret_cast<const float4 *>(qr[i] + dd);
                acc[0][i] += x.x * qv.x + x.y * qv.y + x.z * qv.z + x.w * qv.w;
                acc[1][i] += y.x * qv.x + y.y * qv.y + y.z * qv.z + y.w * qv.w;
            }
        }
#pragma unroll
        for (int kk = 0; kk < 2; ++kk)
#pragma unroll
            for (int i = 0; i < 4; ++i) Ssm[(ty + 16 * kk) * (kPR + 1) + tx + 16 * i] = acc[kk][i] * scale2;
        __syncthreads();
        for (int idx = tid; idx < nr * kPK; idx += kPT) {
            const int rl = idx / kPK, key = idx % kPK;
            const int j = kt + key;
            if (j >= P) continue;
            const int row = r0 + rl;
            const int rpos = P - Rw + row / G;           // absolute position of the window row
            S[((size_t)blockIdx.y * Srows + row) * SP + j] = (j <= rpos) ? Ssm[key * (kPR + 1) + rl] : -INFINITY;
        }
    }
}

// c = max + log2(sum exp2(s - max)) of one window row; stored in the ring row p % R.
__global__ void __launch_bounds__(kPT) prefill_rowstats_kernel(const float *__restrict__ S, float *__restrict__ ring_c,
                                                               int ub0, int P, int Rw, int G, int Gs, int R, RowMap rowmap)
{
    __shared__ float red[kPT / 32];
    __shared__ float bc;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int row = blockIdx.x, u = ub0 + blockIdx.y;
    const float *s = S + ((size_t)blockIdx.y * Rw * G + row) * P;
    const int shift = rowmap(u);
    P -= shift;
    Rw = min(Rw, P);
    if (row >= Rw * G) return;
    float m = -INFINITY;
    for (int j = tid; j < P; j += kPT) m = fmaxf(m, s[j]);
    m = warp_max(m);
    if (lane == 0) red[warp] = m;
    __syncthreads();
    if (tid == 0) { float x = red[0]; for (int w = 1; w < kPT / 32; ++w) x = fmaxf(x, red[w]); bc = x; }
    __syncthreads();
    m = bc;
    float l = 0.f;
    for (int j = tid; j < P; j += kPT) l += exp2f(s[j] - m);
    l = warp_sum(l);
    __syncthreads();
    if (lane == 0) red[warp] = l;
    __syncthreads();
    if (tid == 0) {
        float x = 0.f;
        for (int w = 0; w < kPT / 32; ++w) x += red[w];
        const int i = row / G, g = row % G;
        const int rslot = (P - Rw + i + shift) % R;     // ring slots are assigned on the context's common time axis
        ring_c[((size_t)u * R + rslot) * Gs + g] = m + log2f(x);     // Gs: heads per ring slot (G padded)
    }
}

// Eq. 4-6 with Algorithm 1's group sum: F[j] for every older prompt token j < P - Rw.
__global__ void __launch_bounds__(kPT) prefill_fuse_kernel(const float *__restrict__ S, const float *__restrict__ ring_c,
                                                           float *__restrict__ Fp, int ub0, int P, int Rw, int G, int Gs,
                                                           int R, int fusion, RowMap rowmap)
{
    extern __shared__ float cs[];   // [Rw * G]
    const int u = ub0 + blockIdx.y, Srows = Rw * G, SP = P, shift = rowmap(u);
    P -= shift;
    Rw = min(Rw, P);
    const int rows = Rw * G;
    for (int row = threadIdx.x; row < rows; row += kPT) {
        const int rslot = (P - Rw + row / G + shift) % R;
        cs[row] = ring_c[((size_t)u * R + rslot) * Gs + row % G];
    }
    __syncthreads();
    const int j = blockIdx.x * kPT + threadIdx.x;
    if (j >= P - Rw) return;
    const float *s = S + (size_t)blockIdx.y * Srows * SP + j;
    float F = 0.f;
    for (int i = 0; i < Rw; ++i) {
        float Sr = 0.f;
        for (int g = 0; g < G; ++g) Sr += exp2f(s[(size_t)(i * G + g) * SP] - cs[i * G + g]);
        F = fuse(fusion, F, Sr);
    }
    Fp[(size_t)blockIdx.y * SP + j] = F;
}

// Top-C of the M = P - Rw older tokens by (F descending, position ascending): a radix select on the 64-bit rank keys finds
// the C-th best, then an order-preserving compaction lists the kept positions, followed by the window positions.
//
// One CTA per unit; a warp owns a run of the keys, so that the compaction needs one scan over the warps and no barrier per
// round.  The digits are 12 bits wide: the first takes sign, exponent and three bits of the mantissa, after which a bucket mostly holds a few hundredths of the keys; those move to a list in shared memory, on which the other digits
// work.  The keys are read from memory once if a warp's run fits in its registers (up to 8192 keys), else once per digit
// until the bucket fits the list (the first digit as a rule; more where many scores tie), and twice more.
// Bound by latency for short prompts, by L2 for long ones.  With 8-bit digits, every one of them over all keys, and a
// compaction of 1024 keys per round between barriers: 31 us for 256 units of 6112 keys and 306 us for 131040, now 17 and 101.
constexpr int kSelRun = 8;       // keys a lane holds at a time
constexpr int kSelList = 3072;   // keys of a bucket that fit the list
// T threads per CTA: 1024, or 512 for many units of short prompts, whose CTAs are bound by their barriers (2048 units x 1900 keys
// on average: 60 -> 48 us).
template <int kSelT>
__global__ void __launch_bounds__(kSelT, 2048 / kSelT) prefill_select_kernel(const float *__restrict__ Fp, int *__restrict__ pos, int ub0,
                                                                  int P, int Rw, int C, int cap, RowMap rowmap)
{
    constexpr int kW = kSelT / 32, kChunk = 32 * kSelRun, kBins = 4096, kPer = kBins / kSelT;
    __shared__ unsigned int hist[kBins];
    __shared__ unsigned long long list[kSelList];
    __shared__ int wtot[kW], wkeep[kW];
    __shared__ unsigned long long prefix_s;
    __shared__ int remaining_s, count_s, n_list;
    chain_wait();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int u = ub0 + blockIdx.x;
    const float *F = Fp + (size_t)blockIdx.x * P;
    int *upos = pos + (size_t)u * cap;
    P -= rowmap(u);
    Rw = min(Rw, P);
    const int M = P - Rw;
    if (M <= C) {               // a shorter row whose whole prompt fits
        for (int i = tid; i < P; i += kSelT) upos[i] = i;
        return;
    }
    const int run = (M + kW * kChunk - 1) / (kW * kChunk) * kChunk;      // keys of a warp
    const int j0 = warp * run, j1 = min(M, j0 + run);
    const bool held = run == kChunk;
    unsigned int v[kSelRun];
    auto load = [&](int c0) {                                            // lane l holds keys c0 + 32 i + l
#pragma unroll
        for (int i = 0; i < kSelRun; ++i) {
            const int j = c0 + 32 * i + lane;
            v[i] = j < j1 ? __float_as_uint(F[j]) : 0u;
        }
    };
    if (held) load(j0);
    if (tid == 0) n_list = 0;
    unsigned long long prefix = 0;       // the key bits found so far, at their place
    int remaining = C, hi = 64, shift = 52;      // the bits from `hi` up are known, the digit is hi - 1 .. shift
    bool listed = false, exact = false;
    while (true) {
        // ---- histogram of the digit among the keys that share the prefix
        for (int i = tid; i < kBins; i += kSelT) hist[i] = 0;
        __syncthreads();
        const unsigned int mask = (1u << (hi - shift)) - 1u;
        if (listed) {
            for (int i = tid; i < n_list; i += kSelT)
                if ((list[i] ^ prefix) >> hi == 0) atomicAdd(&hist[(unsigned)(list[i] >> shift) & mask], 1u);
        } else {
            for (int c0 = j0; c0 < j1; c0 += kChunk) {
                if (!held) load(c0);
#pragma unroll
                for (int i = 0; i < kSelRun; ++i) {
                    const int j = c0 + 32 * i + lane;
                    const unsigned long long key = rank_key(v[i], j);
                    if (j < j1 && (hi == 64 || (key ^ prefix) >> hi == 0)) atomicAdd(&hist[(unsigned)(key >> shift) & mask], 1u);
                }
            }
        }
        __syncthreads();
        // ---- the bucket that holds the `remaining`-th best key: above < remaining <= above + its count, with `above` the
        // keys in higher buckets.  A thread owns kPer adjacent buckets; exactly one bucket qualifies.
        int own = 0;
#pragma unroll
        for (int b = 0; b < kPer; ++b) own += (int)hist[tid * kPer + b];
        int incl = own;                                                  // sum over this warp's threads >= tid
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int up = __shfl_down_sync(0xffffffffu, incl, o);
            if (lane + o < 32) incl += up;
        }
        if (lane == 0) wtot[warp] = incl;
        __syncthreads();
        int wsum = lane > warp && lane < kW ? wtot[lane] : 0;
        wsum = (int)__reduce_add_sync(0xffffffffu, (unsigned)wsum);
        int above = wsum + incl - own;
        if (above < remaining && remaining <= above + own) {
#pragma unroll
            for (int b = kPer - 1; b >= 0; --b) {
                const int h = (int)hist[tid * kPer + b];
                if (above < remaining && remaining <= above + h) {
                    prefix_s = prefix | (unsigned long long)(tid * kPer + b) << shift;
                    remaining_s = remaining - above;
                    count_s = h;
                }
                above += h;
            }
        }
        __syncthreads();
        prefix = prefix_s;
        remaining = remaining_s;
        const int count = count_s;
        __syncthreads();
        // the bucket fills the remaining places exactly: all of it is kept, the finer digits are not needed
        exact = count == remaining;
        if (exact || shift == 0) break;
        if (!listed && count <= kSelList) {
            // ---- the bucket moves to the list; what lies above it is kept
            int keep = 0;
            for (int c0 = j0; c0 < j1; c0 += kChunk) {
                if (!held) load(c0);
#pragma unroll
                for (int i = 0; i < kSelRun; ++i) {
                    const int j = c0 + 32 * i + lane;
                    const unsigned long long key = rank_key(v[i], j);
                    const bool in = j < j1;
                    keep += __popc(__ballot_sync(0xffffffffu, in && key >> shift > prefix >> shift));
                    const unsigned int bal = __ballot_sync(0xffffffffu, in && key >> shift == prefix >> shift);
                    if (bal != 0) {
                        int at = 0;
                        if (lane == 0) at = atomicAdd(&n_list, __popc(bal));
                        at = __shfl_sync(0xffffffffu, at, 0);
                        if (bal >> lane & 1) list[at + __popc(bal & ((1u << lane) - 1u))] = key;
                    }
                }
            }
            if (lane == 0) wkeep[warp] = keep;
            listed = true;
            __syncthreads();
        }
        hi = shift;
        shift = max(0, shift - 12);
    }
    // every key >= prefix is kept (the bits below the last digit are zero in it): how many of each warp's
    if (listed) {
        for (int i = tid; i < n_list; i += kSelT)
            if (list[i] >= prefix) atomicAdd(&wkeep[(0xFFFFFFFFu - (unsigned)list[i]) / (unsigned)run], 1);
    } else {
        int keep = 0;
        for (int c0 = j0; c0 < j1; c0 += kChunk) {
            if (!held) load(c0);
#pragma unroll
            for (int i = 0; i < kSelRun; ++i) {
                const int j = c0 + 32 * i + lane;
                keep += __popc(__ballot_sync(0xffffffffu, j < j1 && rank_key(v[i], j) >= prefix));
            }
        }
        if (lane == 0) wkeep[warp] = keep;
    }
    __syncthreads();
    int base = (int)__reduce_add_sync(0xffffffffu, lane < warp ? (unsigned)wkeep[lane] : 0u);
    for (int c0 = j0; c0 < j1; c0 += kChunk) {
        if (!held) load(c0);
#pragma unroll
        for (int i = 0; i < kSelRun; ++i) {
            const int j = c0 + 32 * i + lane;
            const bool keep = j < j1 && rank_key(v[i], j) >= prefix;
            const unsigned int bal = __ballot_sync(0xffffffffu, keep);
            if (keep) upos[base + __popc(bal & ((1u << lane) - 1u))] = j;
            base += __popc(bal);
        }
    }
    for (int i = tid; i < Rw; i += kSelT) upos[C + i] = M + i;
}

// The window sums (DecodeArgs::slab) of the kept slots from the window-row logits S, which the scoring without the tensor
// cores leaves behind: 32 slots per CTA, the ring's blocks shared out among its warps and then run along by one of them.
// Bound by latency for few units, by L2 for many.  (One thread per slot for all blocks: a prompt of
// 4000 tokens into 2 units of 1200 slots, d = 64, 800 rows, took 342 us, now 243; without the sums it takes 232.)
constexpr int kSumSlots = 32, kSumWarps = 8, kMaxSumBlocks = 64;
__global__ void __launch_bounds__(32 * kSumWarps) prefill_sums_kernel(const float *__restrict__ S, DecodeArgs a, int ub0, int P, int Rw, int Gs,
                                                                      RowMap rowmap)
{
    extern __shared__ float cs[];   // [R * Gq]
    __shared__ float blk[kMaxSumBlocks][kSumSlots];
    const int u = ub0 + blockIdx.y, G = a.Gq, Srows = Rw * G, SP = P, shift = rowmap(u), open = open_block(P, a.R, a.bs);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    P -= shift;
    Rw = min(Rw, P);
    for (int i = threadIdx.x; i < a.R * G; i += blockDim.x) cs[i] = a.ring_c[((size_t)u * a.R + i / G) * Gs + i % G];
    __syncthreads();
    const int k = blockIdx.x * kSumSlots + lane;
    const size_t at = (size_t)u * a.cap + k;
    const int p = k < a.cap ? a.pos[at] : -1;
    const int r0 = (P - Rw + shift) % a.R;                                // ring slot of the first window row
    if (p >= 0) {
        const float *s = S + (size_t)blockIdx.y * Srows * SP + p;
        for (int j = warp; j < a.nblk; j += kSumWarps) {
            float F = 0.f;
            for (int r = j * a.bs; r < min(a.R, (j + 1) * a.bs); ++r) {
                const int i = r - r0 + (r < r0 ? a.R : 0);                // window row in ring slot r
                if (i >= Rw) continue;
                float Sr = 0.f;
                for (int g = 0; g < G; ++g) Sr += exp2f(s[(size_t)(i * G + g) * SP] - cs[r * G + g]);
                F = fuse(a.fusion, F, Sr);
            }
            blk[j][lane] = F;
        }
    }
    __syncthreads();
    if (warp != 0 || k >= a.cap) return;
    a.sum_pos[at] = p;
    if (p < 0) return;                                                    // free
    float acc = 0.f, pre = 0.f;
    for (int j = a.nblk - 1; j >= 0; --j) take_block(blk[j][lane], j, open, a.fusion, a.slab + (size_t)u * a.nblk * a.cap + k, a.cap, true, acc, pre);
    a.pre[at] = pre;
}

__global__ void prefill_identity_pos_kernel(int *pos, int U, int n, int cap, RowMap rowmap)
{
    chain_wait();
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (size_t)U * n) return;
    if ((int)(i % n) < n - rowmap((int)(i / n))) pos[(i / n) * cap + (i % n)] = (int)(i % n);
}

// K/V rows of the kept prompt positions into the arena, 16 bytes per thread.  The free slots n .. cap-1 are cleared: the
// decode kernels read whole tiles and mask afterwards, so a row must hold finite numbers.  (Bound by HBM: 266 MB read
// and written in 80 us for 256 units of 2032 slots.  Clearing the whole arena first, as two memsets, wrote every kept
// row twice.)
constexpr int kMaxGridY = 65535;
template <typename T, int D>
__global__ void prefill_gather_kernel(const T *__restrict__ k, const T *__restrict__ v, DecodeArgs a, int P, int Ps, RowMap rowmap)
{
    constexpr int CH = D * sizeof(T) / 16;
    const int u = blockIdx.x;
    P -= rowmap(u);
    const int n = min(P, a.C + min(P, a.R));
    for (int idx = blockIdx.y * blockDim.x + threadIdx.x; idx < a.cap * CH; idx += gridDim.y * blockDim.x) {   // (more than once beyond kMaxGridY only)
        const int slot = idx / CH, c = idx % CH;
        uint4 *Kd = reinterpret_cast<uint4 *>(static_cast<T *>(a.K) + ((size_t)u * a.cap + slot) * D) + c;
        uint4 *Vd = reinterpret_cast<uint4 *>(static_cast<T *>(a.V) + ((size_t)u * a.cap + slot) * D) + c;
        if (slot >= n) {
            *Kd = make_uint4(0, 0, 0, 0);
            *Vd = make_uint4(0, 0, 0, 0);
            continue;
        }
        const int p = a.pos[(size_t)u * a.cap + slot];
        const uint4 *ks = reinterpret_cast<const uint4 *>(k + ((size_t)u * Ps + p) * D) + c;
        const uint4 *vs = reinterpret_cast<const uint4 *>(v + ((size_t)u * Ps + p) * D) + c;
        *Kd = *ks;
        *Vd = *vs;
    }
}

// window queries into their ring rows (row p % R); the rows that a prompt shorter than the window leaves empty are zero
template <typename T, int D>
__global__ void prefill_ring_kernel(const T *__restrict__ qwin, DecodeArgs a, int P, int Rws, RowMap rowmap)
{
    chain_wait();
    const int u = blockIdx.x, G = a.G, Gq = a.Gq, shift = rowmap(u);
    P -= shift;
    const int Rw = min(P, a.R);                         // heads Gq .. G-1 of a ring slot are padding (zero query)
    T *rq = static_cast<T *>(a.ring_q) + (size_t)u * a.R * G * D;
    for (int idx = threadIdx.x; idx < a.R * G * D; idx += blockDim.x) {
        const int dd = idx % D, g = (idx / D) % G, i = idx / (D * G);
        const int rslot = (P - Rw + i + shift) % a.R;
        if (g < Gq && i < Rw) rq[((size_t)rslot * G + g) * D + dd] = qwin[(((size_t)u * Gq + g) * Rws + i) * D + dd];
        else stf(rq + ((size_t)rslot * G + g) * D + dd, 0.f);
    }
}

// the same, 16 bytes at a time and four in flight per thread (q_window 16-byte aligned; 2048 units of 128 rows 34 -> 23 us)
template <typename T, int D>
__global__ void prefill_ring_vec_kernel(const T *__restrict__ qwin, DecodeArgs a, int P, int Rws, RowMap rowmap)
{
    chain_wait();
    constexpr int CH = D * sizeof(T) / 16;
    const int u = blockIdx.x, G = a.G, Gq = a.Gq, shift = rowmap(u);
    P -= shift;
    const int Rw = min(P, a.R);
    const uint4 *src = reinterpret_cast<const uint4 *>(qwin) + (size_t)u * Gq * Rws * CH;
    uint4 *dst = reinterpret_cast<uint4 *>(a.ring_q) + (size_t)u * a.R * G * CH;
    for (int idx0 = (int)blockIdx.y * 4 * blockDim.x + threadIdx.x; idx0 < a.R * G * CH; idx0 += gridDim.y * 4 * blockDim.x) {
        uint4 v[4];
        int at[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int idx = idx0 + j * blockDim.x, c = idx % CH, g = (idx / CH) % G, i = idx / (CH * G);
            at[j] = idx < a.R * G * CH ? ((P - Rw + i + shift) % a.R * G + g) * CH + c : -1;
            v[j] = at[j] >= 0 && g < Gq && i < Rw ? src[(g * Rws + i) * CH + c] : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (at[j] >= 0) dst[at[j]] = v[j];
    }
}

// The prompt phase on a scratch area of `scratch_floats` floats (the window-row logits S and the fused scores of
// as many units as fit go through it, batch after batch).  Every element a kernel reads was written earlier in the
// same batch, so what the area held before never matters.
// CURRENT normalisation after the prompt-phase selection: each window row's normaliser is taken again over the
// tokens that were kept and that the row may see, c = log2 sum exp2(s), from the arena as it stands (kept K rows,
// their positions, the ring's queries).  One CTA per (window row, unit).
template <typename T, int D>
__global__ void __launch_bounds__(kPT) prefill_renorm_kernel(DecodeArgs a, int P, RowMap rowmap)
{
    __shared__ float qs[D];
    __shared__ float red[kPT / 32];
    __shared__ float bc;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int u = blockIdx.y, G = a.G, row = blockIdx.x, i = row / G, g = row % G, shift = rowmap(u);
    P -= shift;
    const int Rw = min(P, a.R), n = a.C + Rw;
    if (i >= Rw || P <= n) return;                                    // everything was kept
    const int rpos = P - Rw + i, rslot = (rpos + shift) % a.R;
    float *c_out = a.ring_c + ((size_t)u * a.R + rslot) * G + g;
    if (*c_out == INFINITY) return;                                   // padding head
    const T *q = static_cast<const T *>(a.ring_q) + (((size_t)u * a.R + rslot) * G + g) * D;
    for (int d = tid; d < D; d += kPT) qs[d] = ldf(q + d);
    __syncthreads();
    const T *K = static_cast<const T *>(a.K) + (size_t)u * a.cap * D;
    const int *pos = a.pos + (size_t)u * a.cap;
    float s[8];       // up to 8 slots per thread per round
    float m = -INFINITY, l = 0.f;
    for (int k0 = 0; k0 < n; k0 += 8 * kPT) {
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const int k = k0 + b * kPT + tid;
            s[b] = -INFINITY;
            if (k < n && pos[k] <= rpos) {
                float acc = 0.f;
                for (int d = 0; d < D; ++d) acc += qs[d] * ldf(K + (size_t)k * D + d);
                s[b] = acc * a.scale2;
            }
        }
        float cm = m;
#pragma unroll
        for (int b = 0; b < 8; ++b) cm = fmaxf(cm, s[b]);
        if (cm > m) { l *= exp2f(m - cm); m = cm; }
        if (m > -INFINITY)
#pragma unroll
            for (int b = 0; b < 8; ++b) l += exp2f(s[b] - m);
    }
    float bm = warp_max(m);
    if (lane == 0) red[warp] = bm;
    __syncthreads();
    if (tid == 0) { float x = red[0]; for (int w = 1; w < kPT / 32; ++w) x = fmaxf(x, red[w]); bc = x; }
    __syncthreads();
    bm = bc;
    float bl = warp_sum(m > -INFINITY ? l * exp2f(m - bm) : 0.f);
    __syncthreads();
    if (lane == 0) red[warp] = bl;
    __syncthreads();
    if (tid == 0) {
        float x = 0.f;
        for (int w = 0; w < kPT / 32; ++w) x += red[w];
        *c_out = bm + log2f(x);
    }
}

template <typename T, int D>
cudaError_t run_prefill_t(const DecodeArgs &a, const T *k, const T *v, const T *qwin, int P, cudaStream_t stream,
                          unsigned long long *launches, float *S, size_t scratch_floats, int *host_err, int n_states, int padded_len,
                          const int *row_shift)
{
    // With prompts of different lengths (a.row_shift) P is the longest one and the tensors are padded to padded_len
    // tokens; the ring slots follow the common time axis, on which every row ends at P.
    const RowMap rowmap = {a.row_shift, a.Hkv, a.B};
    const int Ps = padded_len, Rws = min(Ps, a.R);
    const int U = a.U, G = a.G, R = a.R, C = a.C;
    // the CUDA-core scoring kernels work on the model's Gq heads per window position (rows of S); the ring keeps G
    // heads per slot, the padding heads with normaliser +inf from init_arena_kernel
    const int Rw = P < R ? P : R, rows = Rw * a.Gq;
    const bool select = P - Rw > C;
    const int n = select ? C + Rw : P;
    if (n > a.cap) return cudaErrorInvalidValue;
    // bf16 / head_dim 128 shapes score on the tensor cores (no rows x P table); the
    // others materialise the window-row logits S [rows][P] per unit and reduce them with CUDA-core kernels
    // (the arena's group must be the padded one: a context that runs the CUDA-core decode kernel keeps G as it is)
    const bool tc = prefill_tc_supported(sizeof(T) == 4, D, a.Gq, R, k, qwin, P) && tc_padded_group(a.Gq) == G;
    const int tc_run = tc ? prefill_tc_run(a, P, row_shift) : 0;
    const size_t per_unit = tc ? prefill_tc_floats_per_unit(P, Rw, G, tc_run) : (size_t)rows * P + P;   // floats
    const size_t fixed = tc ? kScratchWords : 1;
    if (per_unit + fixed > scratch_floats) return cudaErrorInvalidConfiguration;
    size_t ub = (scratch_floats - fixed) / per_unit;
    if (ub > (size_t)U) ub = U;
    if (ub > 65535) ub = 65535;
    // tensor-core path: the window rows' statistics, the scores, and the words of state, zero at the start, that end with the error word
    const size_t unit_words = tc ? prefill_tc_words_per_unit(P, tc_run) : 0;
    float *part = S, *Fp = S + ub * (tc ? per_unit - P - unit_words : (size_t)rows * P);
    const int n_words = (int)(ub * unit_words + fixed);
    int *words = reinterpret_cast<int *>(Fp + ub * (size_t)P), *err_word = words + n_words - 1;

    const size_t logits_smem = (size_t)(kPK * (D + 4) + kPR * (D + 4) + kPK * (kPR + 1)) * sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(prefill_logits_kernel<T, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)logits_smem);
    if (e != cudaSuccess) return e;
    const size_t init_n = max(max((size_t)U * a.cap, (size_t)U * R * G), (size_t)n_words);
    init_arena_kernel<<<(unsigned)((init_n + 255) / 256), 256, 0, stream>>>(a, words, n_words);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const bool waits = tc || a.nblk > 1;            // kernels with bounded waits are launched
    constexpr int CH = D * sizeof(T) / 16;
    e = ((uintptr_t)qwin & 15) == 0
        ? launch_chained(prefill_ring_vec_kernel<T, D>, dim3(U, min(kMaxGridY, (R * G * CH + 1023) / 1024)), 256, 0, stream, qwin, a, P, Rws, rowmap)
        : launch_chained(prefill_ring_kernel<T, D>, dim3(U), 256, 0, stream, qwin, a, P, Rws, rowmap);
    if (e != cudaSuccess) return e;
    *launches += 2;
    if (!select) {
        e = launch_chained(prefill_identity_pos_kernel, dim3((unsigned)(((size_t)U * n + 255) / 256)), 256, 0, stream, a.pos, U, n, a.cap, rowmap);
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    // the window sums: on the tensor cores at the end, or from the logits S where there are any
    const bool sums_tc = sizeof(T) == 2 && D == 128 && tc_padded_group(a.Gq) == G;
    for (int ub0 = 0; ub0 < U; ub0 += (int)ub) {
        const int nb = min((int)ub, U - ub0);
        if (tc) {
            e = run_prefill_scores_tc(a, k, qwin, P, Ps, row_shift, ub0, nb, (int)ub, tc_run, select, Fp, part, words, err_word, launches, stream);
            if (e != cudaSuccess) return e;
        } else {
            prefill_logits_kernel<T, D><<<dim3((P + kPK - 1) / kPK, nb), kPT, logits_smem, stream>>>(k, qwin, S, ub0, P, Rw,
                                                                                                 a.Gq, a.scale2, Ps, Rws, rowmap);
            prefill_rowstats_kernel<<<dim3(rows, nb), kPT, 0, stream>>>(S, a.ring_c, ub0, P, Rw, a.Gq, G, R, rowmap);
            *launches += 2;
        }
        if (select) {
            if (!tc) {
                prefill_fuse_kernel<<<dim3((P - Rw + kPT - 1) / kPT, nb), kPT, rows * sizeof(float), stream>>>(
                    S, a.ring_c, Fp, ub0, P, Rw, a.Gq, G, R, a.fusion, rowmap);
                ++*launches;
            }
            e = nb > 2 * 148 && P - Rw <= 512 * kSelRun ? launch_chained(prefill_select_kernel<512>, dim3(nb), 512, 0, stream, Fp, a.pos, ub0, P, Rw, C, a.cap, rowmap)
                                                       : launch_chained(prefill_select_kernel<1024>, dim3(nb), 1024, 0, stream, Fp, a.pos, ub0, P, Rw, C, a.cap, rowmap);
            if (e != cudaSuccess) return e;
            ++*launches;
        }
        if (a.nblk > 1 && !sums_tc) {
            if (a.nblk > kMaxSumBlocks) return cudaErrorInvalidValue;
            prefill_sums_kernel<<<dim3((a.cap + kSumSlots - 1) / kSumSlots, nb), 32 * kSumWarps, R * a.Gq * sizeof(float), stream>>>(S, a, ub0, P, Rw, G, rowmap);
            ++*launches;
        }
    }
    // (the gather may take the window sums along, for which it needs the ring)
    const bool sums_along = sums_tc && gather_sums_supported(a, k, v);
    e = cudaSuccess;
    if (sums_along) e = launch_gather_sums(a, k, v, P, Ps, n, err_word, stream);
    else prefill_gather_kernel<T, D><<<dim3(U, min(kMaxGridY, (a.cap * CH + 255) / 256)), 256, 0, stream>>>(k, v, a, P, Ps, rowmap);
    if (e != cudaSuccess) return e;
    if (a.norm_current && select) {
        prefill_renorm_kernel<T, D><<<dim3(Rw * G, U), kPT, 0, stream>>>(a, P, rowmap);
        ++*launches;
    }
    ++*launches;
    e = cudaGetLastError();
    if (e == cudaSuccess) e = launch_finish_prompt(a, sums_tc && !sums_along, P, n, n_states, err_word, launches, stream);
    // a bounded wait that ran out: the word comes back with the stream's end if there is pinned memory for it
    int werr = 0;
    if (waits && host_err != nullptr && e == cudaSuccess) e = cudaMemcpyAsync(host_err, err_word, sizeof(int), cudaMemcpyDeviceToHost, stream);
    const cudaError_t e2 = cudaStreamSynchronize(stream);
    if (e != cudaSuccess || e2 != cudaSuccess) return e != cudaSuccess ? e : e2;
    if (waits) {
        if (host_err != nullptr) werr = *host_err;
        else e = cudaMemcpy(&werr, err_word, sizeof(int), cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) return e;
        if (werr != 0) return cudaErrorLaunchTimeout;
    }
    return cudaSuccess;
}

cudaError_t dispatch_prefill(const DecodeArgs &a, bool f32, int D, const void *k, const void *v, const void *q_window, int P,
                             cudaStream_t stream, unsigned long long *launches, float *S, size_t scratch_floats, int *host_err, int n_states,
                             int padded_len, const int *row_shift)
{
    if (f32) {
        auto kk = static_cast<const float *>(k), vv = static_cast<const float *>(v), qq = static_cast<const float *>(q_window);
        return D == 64 ? run_prefill_t<float, 64>(a, kk, vv, qq, P, stream, launches, S, scratch_floats, host_err, n_states, padded_len, row_shift)
                       : run_prefill_t<float, 128>(a, kk, vv, qq, P, stream, launches, S, scratch_floats, host_err, n_states, padded_len, row_shift);
    }
    auto kk = static_cast<const __nv_bfloat16 *>(k), vv = static_cast<const __nv_bfloat16 *>(v),
         qq = static_cast<const __nv_bfloat16 *>(q_window);
    return D == 64 ? run_prefill_t<__nv_bfloat16, 64>(a, kk, vv, qq, P, stream, launches, S, scratch_floats, host_err, n_states, padded_len, row_shift)
                   : run_prefill_t<__nv_bfloat16, 128>(a, kk, vv, qq, P, stream, launches, S, scratch_floats, host_err, n_states, padded_len, row_shift);
}

// ---- scratch of mkv_prefill_static -------------------------------------------------------------------------
// A fixed device array that every GPU loading this library holds until the process exits.  16 MiB: one unit of a
// 4096-token prompt with R*G = 128 window rows needs 2.1 MB, so the units go through it a few at a time.
constexpr size_t kStaticScratchFloats = (size_t)4 << 20;
static __device__ __align__(256) float g_prefill_scratch[kStaticScratchFloats];

constexpr int kMaxDevices = 64;
static float *g_scratch_addr[kMaxDevices];   // device address of the array, per device ordinal
static std::mutex g_scratch_mutex;

// The array's name is only a host-side handle here; a kernel needs its device address, which the runtime hands out
// per device.  Looked up once per device, with that device current.
cudaError_t static_scratch_address(int device, float **out)
{
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    if (dev != device) return cudaErrorInvalidDevice;          // the context lives on another device than the current one
    std::lock_guard<std::mutex> lock(g_scratch_mutex);
    if (!g_scratch_addr[dev]) {
        float *ptr = nullptr;
        e = cudaGetSymbolAddress((void **)&ptr, g_prefill_scratch);
        if (e != cudaSuccess) return e;
        g_scratch_addr[dev] = ptr;
    }
    *out = g_scratch_addr[dev];
    return cudaSuccess;
}

}  // namespace

cudaError_t run_prefill(const DecodeArgs &a, bool f32, int D, const void *k, const void *v, const void *q_window, int P,
                        cudaStream_t stream, unsigned long long *launches, PrefillScratch *scratch, int n_states,
                        int padded_len, const int *row_shift)
{
    const int Rw = P < a.R ? P : a.R;
    const bool tc = prefill_tc_supported(f32, D, a.Gq, a.R, k, q_window, P) && tc_padded_group(a.Gq) == a.G;
    const size_t per_unit = (tc ? prefill_tc_floats_per_unit(P, Rw, a.G, prefill_tc_run(a, P, row_shift))
                                : (size_t)Rw * a.G * P + P) * sizeof(float);
    size_t ub = ((size_t)1 << 30) / per_unit;
    if (ub < 1) ub = 1;
    if (ub > (size_t)a.U) ub = a.U;
    if (ub > 65535) ub = 65535;
    const size_t need = ub * per_unit + kScratchWords * sizeof(float);
    // The scratch belongs to the context and is kept until the context is destroyed: it only grows.
    // (Allocating and freeing it around every prompt put a cudaFree of up to 1 GiB right in front
    // of the first decode launches.)
    if (scratch->bytes < need) {
        if (scratch->ptr) cudaFree(scratch->ptr);
        scratch->ptr = nullptr;
        scratch->bytes = 0;
        const cudaError_t e = cudaMalloc(&scratch->ptr, need);
        if (e != cudaSuccess) { scratch->ptr = nullptr; return e; }
        scratch->bytes = need;
    }
    if (!scratch->host_err && cudaMallocHost(reinterpret_cast<void **>(&scratch->host_err), sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        scratch->host_err = nullptr;
    }
    return dispatch_prefill(a, f32, D, k, v, q_window, P, stream, launches, static_cast<float *>(scratch->ptr),
                            scratch->bytes / sizeof(float), scratch->host_err, n_states, padded_len, row_shift);
}

namespace {
// rows_dst / rows_src: the states' per-row fills ([2][B] ints per state, see DecodeArgs::row_n), or nullptr
__global__ void copy_state_kernel(DevState *dst, int n_dst, const DevState *src, int *rows_dst, const int *rows_src,
                                  int row_ints)
{
    const DevState s = *src;
    __syncthreads();            // src may be one of the destinations
    for (int i = threadIdx.x; i < n_dst; i += blockDim.x) { dst[i] = s; dst[i].done = 0; }
    if (rows_dst != nullptr && rows_dst != rows_src)
        for (int i = threadIdx.x; i < n_dst * row_ints; i += blockDim.x) rows_dst[i] = rows_src[i % row_ints];
}
}  // namespace

cudaError_t launch_copy_state(DevState *dst, int n_dst, const DevState *src, cudaStream_t stream, int *rows_dst,
                              const int *rows_src, int row_ints)
{
    copy_state_kernel<<<1, 64, 0, stream>>>(dst, n_dst, src, rows_dst, rows_src, row_ints);
    return cudaGetLastError();
}

size_t prefill_static_max_floats() { return kStaticScratchFloats; }

cudaError_t run_prefill_static(const DecodeArgs &a, bool f32, int D, const void *k, const void *v, const void *q_window,
                               int P, cudaStream_t stream, unsigned long long *launches, int device, int n_states)
{
    float *S = nullptr;
    const cudaError_t e = static_scratch_address(device, &S);
    if (e != cudaSuccess) return e;
    return dispatch_prefill(a, f32, D, k, v, q_window, P, stream, launches, S, kStaticScratchFloats, nullptr, n_states, P, nullptr);
}

}  // namespace mkv
