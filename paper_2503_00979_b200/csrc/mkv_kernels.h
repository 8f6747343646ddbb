// Host-callable launchers of the MorphKV kernels (internal to the library).
#pragma once

#include "mkv_common.cuh"

namespace mkv {

// Warp-level decode step (any supported shape).  `nsplit` CTAs per unit, at most 16.
cudaError_t launch_decode_simt(const DecodeArgs &a, int nsplit, bool f32, int D, cudaStream_t stream);
int simt_block_slots(bool f32, int G, int R);      // slots per block of the ring (DecodeArgs::bs), 0: no sums are kept
int simt_default_splits(int U, int cap);
int simt_small_splits(int U, int G, int R, int bs, int nblk, int cap, bool layer);   // CTAs per unit for a small tcgen05-context launch, 0: not small

// Coarse-grained eviction (evict_interval > 1): drops everything beyond the top C after a step that scored and
// restores the dense prefix of C + R slots; a no-op after the other steps.  Launched after every decode step.
cudaError_t launch_compact(const DecodeArgs &a, bool f32, int D, cudaStream_t stream);

// Tensor-core (tcgen05) decode step: bf16, head_dim 128, GQA group padded to {1,2,4,8,16}.  A window of up to
// 256 ring rows (R * padded group) is one MMA operand; a larger one is cut into tc_ring_chunks() chunks of equal
// width, and a unit then appears in the kernel's schedule once per chunk (U * chunks "virtual units": pass that
// count to tc_grid() and tc_partials_per_unit()).  The plan holds the TMA tensor maps of a context's arena and
// the launch geometry; `a.splits` must be tc_partials_per_unit() of the grid (every CTA that holds tiles of a
// unit leaves one partial).
bool tc_shape_supported(bool f32, int D, int G, int R);
int tc_padded_group(int G);
int tc_ring_chunks(int G, int R);
int tc_block_slots(int G, int R, bool current);   // slots per block of the ring (DecodeArgs::bs)
int tc_grid(int U, int cap, int splits_hint, int n_sm);
int tc_partials_per_unit(int U, int cap, int grid);
struct TcPlan;
// `prefetch`: CTAs ask for the first tiles of their range into L2 while the previous launch drains.
cudaError_t tc_plan_create(TcPlan **plan, const DecodeArgs &a, int grid, unsigned long long wait_limit_cycles, bool prefetch,
                           char *err, size_t err_len);
void tc_plan_destroy(TcPlan *plan);
cudaError_t launch_decode_tc(TcPlan *plan, const DecodeArgs &a, cudaStream_t stream);

// Prompt phase: fills the arena (K, V, pos, ring) and the n_states step states at a.st from a prompt of P
// tokens.  `a` supplies the arena pointers and shape; q/k_new/v_new/out are ignored.
// *launches is advanced per kernel launched.
// Device scratch of the prompt phase, owned by the context (allocated on first use, grown when a
// longer prompt needs more, released with the context).
struct PrefillScratch {
    void *ptr;
    size_t bytes;
    int *host_err;       // pinned word (nullptr: none could be had)
};
// With prompts of different lengths in the batch (a.row_shift; `row_shift`: the same [B] numbers on the host, else nullptr) P is
// the longest prompt's length; the tensors are padded to padded_len tokens (P otherwise).
cudaError_t run_prefill(const DecodeArgs &a, bool f32, int D, const void *k, const void *v, const void *q_window,
                        int P, cudaStream_t stream, unsigned long long *launches, PrefillScratch *scratch, int n_states,
                        int padded_len, const int *row_shift);

// Tensor-core scoring of the prompt phase (mkv_prefill_tc.cu): window-row normalisers into ring_c and fused scores of the
// older tokens into Fp [nb][P].
bool prefill_tc_supported(bool f32, int D, int G, int R, const void *k, const void *qwin, int P);
int prefill_tc_run(const DecodeArgs &a, int P, const int *row_shift);       // key tiles of an item
size_t prefill_tc_words_per_unit(int P, int run);
size_t prefill_tc_floats_per_unit(int P, int Rw, int G, int run);
cudaError_t run_prefill_scores_tc(const DecodeArgs &a, const void *k, const void *qwin, int P, int Ps, const int *row_shift, int ub0, int nb, int units, int run, bool select,
                                  float *Fp, float *part, int *words, int *err, unsigned long long *launches, cudaStream_t stream);

// The same prompt phase with its scratch in a fixed device array of prefill_static_max_floats()
// floats instead of a temporary allocation; cudaErrorInvalidConfiguration if one unit's
// (R*G + 1) * P floats do not fit.
size_t prefill_static_max_floats();
cudaError_t run_prefill_static(const DecodeArgs &a, bool f32, int D, const void *k, const void *v, const void *q_window,
                               int P, cudaStream_t stream, unsigned long long *launches, int device, int n_states);

// The gather of the kept prompt rows into the arena and the window sums in one launch (windows of up to 256 ring rows on the
// tensor cores); a.pos and the ring are there.
bool gather_sums_supported(const DecodeArgs &a, const void *k, const void *v);
cudaError_t launch_gather_sums(const DecodeArgs &a, const void *k, const void *v, int P, int Ps, int n, int *err, cudaStream_t stream);
// Last launch(es) of the prompt phase: if `sums`, the window sums of every slot, where the context keeps them, for the
// step at position t of n cached tokens, and the n_states step states at a.st.  `err`: word in which a wait that runs out is
// reported.
cudaError_t launch_finish_prompt(const DecodeArgs &a, bool sums, long long t, int n, int n_states, int *err, unsigned long long *launches,
                                 cudaStream_t stream);

// Copies one step state over n_dst others (the whole-stack state and the per-layer states are brought level when
// a context switches between whole-stack and per-layer calls).
cudaError_t launch_copy_state(DevState *dst, int n_dst, const DevState *src, cudaStream_t stream, int *rows_dst = nullptr,
                              const int *rows_src = nullptr, int row_ints = 0);

}  // namespace mkv
