// Coarse-grained eviction (the paper's appendix on running the policy every T-th step): the decode
// step that scored has appended its token like any other step and left the final fused score of
// every slot in F (-1 for the slots of the recent window).  This launch then applies Eq. 7 once:
// it drops the E = n - (C + R) lowest-ranked candidates (lower fused score first, on equal scores
// the later position first, so that the lower position is the one kept) and moves the survivors
// that sit beyond slot C + R into the freed slots, which restores a dense prefix of C + R slots.
// One CTA of 1024 threads per unit, each thread holding a few slots' rank keys; launched after the
// decode steps that ran the policy, and a no-op unless the device state says a compaction is pending.
//
// Selection without a loop over the evicted: the threads form groups of GL lanes, and the E-th smallest of the groups' minima
// bounds the E smallest keys from above; the few keys up to it move to a list, where each counts the smaller ones.  (Bound by
// latency: E block-wide minima one after the other, two barriers each, a serial sort of the holes, and a launch in full stream
// order took 22.7 us for 256 units of 2040 slots and E = 8, now 10.9.)
#include "mkv_common.cuh"
#include "mkv_kernels.h"

namespace mkv {

namespace {

constexpr int kCT = 1024;         // threads per CTA

// KPT slots per thread, held in registers (indices are compile-time constants after unrolling)
template <typename T, int D, int KPT>
__global__ void __launch_bounds__(kCT, KPT <= 4 ? 2 : 1) compact_kernel(DecodeArgs a)
{
    // at least as many groups as tokens can be evicted (64), and 64 groups' keys fit the list
    constexpr int GL = KPT <= 4 ? 16 : KPT == 8 ? 8 : 4, NGR = kCT / GL, kList = 64 * GL * KPT;
    static_assert(kList <= 4096 && NGR >= 64, "groups");
    __shared__ unsigned long long group_min[NGR], bound_s;
    __shared__ unsigned long long list[kList];
    __shared__ unsigned short list_slot[kList];          // (16 slots per thread at most)
    __shared__ int ev_slot[64];          // evicted slots, in eviction order
    __shared__ int holes[64], movers[64];
    __shared__ int n_list, n_holes;
    chain_wait();
    const int tid = threadIdx.x;
    const int u = blockIdx.x;
    const bool pending = a.st->compact != 0;
    const int n = a.st->n;                       // tokens cached after the step's append
    const int keep = a.C + a.R;
    const int E = n - keep;
    if (pending && E > 0) {
        int *pos = a.pos + (size_t)u * a.cap;
        float *F = a.F + (size_t)u * a.cap;
        // every thread's candidates as rank keys (window slots carry F = -1 and never compete)
        unsigned long long key[KPT];
#pragma unroll
        for (int i = 0; i < KPT; ++i) {
            const int k = tid + i * kCT;
            unsigned long long v = ~0ull;
            if (k < n) {
                const float f = F[k];
                if (f >= 0.f) v = rank_key(__float_as_uint(f), pos[k]);
            }
            key[i] = v;
        }
        unsigned long long low = key[0];
#pragma unroll
        for (int i = 1; i < KPT; ++i) low = key[i] < low ? key[i] : low;
#pragma unroll
        for (int o = GL / 2; o > 0; o >>= 1) {
            const unsigned long long x = __shfl_xor_sync(0xffffffffu, low, o);
            low = x < low ? x : low;
        }
        if (tid % GL == 0) group_min[tid / GL] = low;
        if (tid < 64) ev_slot[tid] = -1;
        if (tid == 0) n_list = n_holes = 0;
        __syncthreads();
        if (tid < NGR) {                            // (groups without candidates tie: the earlier one first)
            const unsigned long long mine = group_min[tid];
            int rank = 0;
            for (int g = 0; g < NGR; ++g) rank += group_min[g] < mine || (group_min[g] == mine && g < tid);
            if (rank == E - 1) bound_s = mine;
        }
        __syncthreads();
        const unsigned long long bound = bound_s;
#pragma unroll
        for (int i = 0; i < KPT; ++i)
            if (key[i] <= bound && key[i] != ~0ull) {
                const int at = atomicAdd(&n_list, 1);
                list[at] = key[i];
                list_slot[at] = (unsigned short)(tid + i * kCT);
            }
        __syncthreads();
        const int m = n_list;
        for (int i = tid; i < m; i += kCT) {
            const unsigned long long mine = list[i];
            int rank = 0;
            for (int j = 0; j < m; ++j) rank += list[j] < mine;
            if (rank < E) ev_slot[rank] = list_slot[i];
        }
        __syncthreads();
        // holes: evicted slots inside the kept prefix; movers: surviving slots beyond it (both ascending, as many of one as of
        // the other)
        if (tid < E) {
            const int s = ev_slot[tid];
            if (s >= 0 && s < keep) {
                int at = 0;
                for (int e = 0; e < E; ++e) at += ev_slot[e] >= 0 && ev_slot[e] < s;
                holes[at] = s;
                atomicAdd(&n_holes, 1);
            }
        } else if (tid >= 64 && tid < 64 + E) {
            const int k = keep + tid - 64;
            bool gone = false;
            int before = 0;
            for (int e = 0; e < E; ++e) {
                gone |= ev_slot[e] == k;
                before += ev_slot[e] >= keep && ev_slot[e] < k;
            }
            if (!gone) movers[k - keep - before] = k;
        }
        __syncthreads();
        const int nh = n_holes;
        constexpr int CH = D * (int)sizeof(T) / 16;
        uint4 *K = reinterpret_cast<uint4 *>(static_cast<T *>(a.K) + (size_t)u * a.cap * D);
        uint4 *V = reinterpret_cast<uint4 *>(static_cast<T *>(a.V) + (size_t)u * a.cap * D);
        for (int idx = tid; idx < 2 * nh * CH; idx += kCT) {
            const int i = idx / (2 * CH), c = idx % CH;
            uint4 *X = idx / CH % 2 ? V : K;
            X[(size_t)holes[i] * CH + c] = X[(size_t)movers[i] * CH + c];
        }
        __syncthreads();
        if (tid < nh) { pos[holes[tid]] = pos[movers[tid]]; F[holes[tid]] = F[movers[tid]]; }
        if (a.nblk > 1) {           // the window sums move with their slot
            float *slab = a.slab + (size_t)u * a.nblk * a.cap, *pre = a.pre + (size_t)u * a.cap;
            for (int idx = tid; idx < nh * (a.nblk + 1); idx += kCT) {
                const int i = idx % nh, j = idx / nh;
                float *row = j < a.nblk ? slab + (size_t)j * a.cap : pre;
                row[holes[i]] = row[movers[i]];
            }
            if (tid < nh) a.sum_pos[(size_t)u * a.cap + holes[tid]] = a.sum_pos[(size_t)u * a.cap + movers[tid]];
        }
        __syncthreads();
        for (int k = keep + tid; k < n; k += kCT) {
            pos[k] = -1;
            F[k] = 0.f;
            if (a.nblk > 1) a.sum_pos[(size_t)u * a.cap + k] = -1;
        }
        if (tid == 0) a.evicted_pos[u] = -1;
    }
    // the last CTA publishes the new fill (all CTAs have read the state by then)
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        if (atomicAdd(&a.st->done, 1u) == gridDim.x - 1) {
            if (pending && E > 0) a.st->n = keep;
            a.st->compact = 0;
            a.st->done = 0;
            __threadfence();
        }
    }
}

}  // namespace

template <typename T, int D>
static cudaError_t launch_compact_t(const DecodeArgs &a, cudaStream_t stream)
{
    const int per = (a.cap + kCT - 1) / kCT;
    if (per <= 2) return launch_chained(compact_kernel<T, D, 2>, dim3(a.U), kCT, 0, stream, a);
    if (per <= 4) return launch_chained(compact_kernel<T, D, 4>, dim3(a.U), kCT, 0, stream, a);
    if (per <= 8) return launch_chained(compact_kernel<T, D, 8>, dim3(a.U), kCT, 0, stream, a);
    return launch_chained(compact_kernel<T, D, 16>, dim3(a.U), kCT, 0, stream, a);
}

cudaError_t launch_compact(const DecodeArgs &a, bool f32, int D, cudaStream_t stream)
{
    if (a.T > 64 || (a.cap + kCT - 1) / kCT > 16) return cudaErrorInvalidConfiguration;
    if (f32) return D == 64 ? launch_compact_t<float, 64>(a, stream) : launch_compact_t<float, 128>(a, stream);
    return D == 64 ? launch_compact_t<__nv_bfloat16, 64>(a, stream) : launch_compact_t<__nv_bfloat16, 128>(a, stream);
}

}  // namespace mkv
