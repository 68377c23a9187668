// Launchers shared between the API translation unit and the kernel files.
#pragma once
#include <memory>

#include "common.cuh"
#include "ssd_scalars.cuh"

namespace swimba {

// K1a: router logits, softmax over all E, top-k (indices + un-renormalised weights).
// When counts is given (zeroed beforehand) the (token, slot) pairs are also grouped by expert:
// perm[e * cap + i], i < counts[e], lists the entries t*k + j routed to expert e.
// zero_out (may be NULL): a [T, zero_bytes_per_token] buffer the kernel clears on the way (the
// mixed streams, when the projection adds its slots in place).  scalars.l2 != NULL: the call also
// produces the SSD step sizes and tile log-decays of the same forward (they depend on dt only and
// run beside the router, inside its launch or as a kernel in front of it).  pi_out (may be NULL):
// the softmax over all E, [T,E].
int launch_router(LaunchCtx &ctx, int dtype, const void *u, const void *W_r, int64_t T, int F,
                  int E, int k, int32_t *idx, float *w, int *counts, int *perm, int64_t cap,
                  int sm_count, void *zero_out, int zero_bytes_per_token, const ScalarsArgs &scalars,
                  float *pi_out = nullptr);

// K1b (tensor cores): grouped GEMM over the per-expert lists + slot sum.  `workspace` is sized
// by expert_gemm_workspace_bytes and holds the histogram (zeroed by the caller before the
// router runs), the per-expert lists (capacity T each) and the per-slot projections.
size_t expert_gemm_workspace_bytes(int64_t T, int S, int E, int k);
bool expert_gemm_supported(int F, int S);
bool expert_gemm_adds_rows(int k);   // true: BC must be zero before launch_expert_gemm runs
int *expert_gemm_counts(void *workspace);
int *expert_gemm_perm(void *workspace);
// slots_out (may be NULL): [T*k, S] bf16; when given, the projection of (token t, slot j), scaled by
// its router weight (w NULL: 1), is stored in row t*k + j and nothing is mixed (BC is not touched); slots_f32: as
// fp32 rows.
int launch_expert_gemm(LaunchCtx &ctx, const void *u, const void *W_e, const float *w, int64_t T,
                       int F, int S, int E, int k, int sm_count, void *BC, void *workspace,
                       void *slots_out = nullptr, bool slots_f32 = false);

// BC[t, :] = sum_j w[t,j] slots[t*k + j, :], bf16 (w NULL: 1).
int launch_mix_slots(LaunchCtx &ctx, const void *slots, const float *w, int64_t T, int S, int k, int sm_count, void *BC);

// The same products on CTA pairs, 256 x 256 tiles, persistent: calls with enough tiles (pair_gemm_usable).
// perm == NULL: the T rows of A as they lie (E = k = 1, no weights); out rows are ld_out elements apart.
// tail (dense rows only): columns tail_col .. S-1 (tail_col % 32 == 0) go there as fp32, [T, S - tail_col].
bool pair_gemm_usable(int64_t rows, int F, int S, int E, int sm_count);
int launch_pair_gemm(LaunchCtx &ctx, const void *A, const void *W, const int *perm, const int *counts,
                     const float *w_slot, int64_t T, int F, int S, int E, int k, bool add_rows, int sm_count,
                     void *out, int64_t ld_out, float *tail = nullptr, int tail_col = 0);

// K1b (SIMT): project the k selected experts and mix.  BC is written in `dtype`, or as float
// per slot-sum when bc_fp32 is set.
int launch_project_mix_simt(LaunchCtx &ctx, int dtype, const void *u, const void *W_e,
                            const int32_t *idx, const float *w, int64_t T, int F, int S, int E,
                            int k, void *BC, bool bc_fp32);
// The same without the mix: row t*k + j of slots_out (dtype) = w[t,j] * W_e[idx[t,j]] u_t (w NULL: 1).
int launch_project_slots_simt(LaunchCtx &ctx, int dtype, const void *u, const void *W_e,
                              const int32_t *idx, const float *w, int64_t T, int F, int S, int E,
                              int k, void *slots_out);

// General injection (expert-specific SSM inputs) helpers, all dtype-generic streaming kernels:
//   assemble: BCj[t, :] = [ slots[t*k + j, 0:GN] | sum_j' slots[t*k + j', GN:2GN] ]
//   accumulate: y += y_add (dtype, fp32 sum), h += h_add (float); either pair may be NULL
int launch_assemble_slot_streams(LaunchCtx &ctx, int dtype, const void *slots, int64_t T, int S, int k,
                                 int j, void *BCj);
int launch_accumulate(LaunchCtx &ctx, int dtype, void *y, const void *y_add, int64_t ny, float *h,
                      const float *h_add, int64_t nh);

// K1 for at most a few hundred tokens (decode): one or two short kernels, no lists in global memory.
// idx [T,k], w [T,k] and the fp32 streams BC are written: [T,S] mixed, or, where front_small_slots says so,
// [T,k,S] per slot (weights applied), summed by the reader.  The kernel behind starts only after everything
// in front of this call has completed, so it may read what earlier calls wrote before its own wait.
// front_small_faster: whether it is, beside the router and the grouped product (with fp32 slots).
constexpr int FRONT_SMALL_TOKENS = 256;      // per call
bool front_small_supported(int dtype, int64_t T, int F, int S, int E, int k);
bool front_small_faster(int64_t T, int F, int S, int E, int k);
bool front_small_slots(int64_t T, int S, int E, int k);
int launch_front_small(LaunchCtx &ctx, const void *u, const void *W_r, const void *W_e, int64_t T, int F,
                       int S, int E, int k, int sm_count, int32_t *idx, float *w, float *BC);
// The same kernels for short calls of the forward: BC [T,S] bf16; scalars as in launch_router.
bool front_short_supported(int dtype, int64_t T, int F, int S, int E, int k);
int launch_front_short(LaunchCtx &ctx, const void *u, const void *W_r, const void *W_e, int64_t T, int F, int S, int E,
                       int k, int sm_count, int32_t *idx, float *w, void *BC, const ScalarsArgs &scalars);

// K2/K3 (tensor cores): tiled SSD with the carried state kept on chip; bf16, P == 64, N == 128.
bool ssd_tiles_supported(int dtype, int P, int N);
size_t ssd_workspace_bytes(int B, int L, int H, int G, int chunk, int sm_count);
// Tokens per segment the tile path cuts a sequence into (a multiple of 128; >= L: one segment).
int ssd_segment_len(int B, int L, int H, int G, int chunk, int sm_count);
// Clears up to four regions (16-byte aligned, sizes multiples of 16; null: none) as the first kernel of a gradient call;
// the kernel behind it may be launched programmatically and waits with grid_dep_wait.  Four memsets in its place cost
// 8 us more at 4 x 8192 tokens (795 -> 787): mostly the gaps between them.  A forward clears its histogram alone and keeps the memset: with this kernel and the router launched behind it
// programmatically calls went anywhere between 0.973 and 1.034 of their rate.
struct ZeroRegions { void *p[4]; size_t bytes[4]; };
int launch_zero(LaunchCtx &ctx, const ZeroRegions &z, int sm_count);

// scalars_done: the step sizes and tile log-decays (ssd_scalars_args over the same workspace) have
// already been produced earlier in the stream (launch_router with scalars, or launch_ssd_scalars).  early:
// x and h0 were complete before the first kernel of the same call.
// runs: what ssd_long_runs says of the call (false for kernels that take the records of the tile kernel).
ScalarsArgs ssd_scalars_args(const float *dt, const float *A, const float *dt_bias, int B, int L, int H,
                             void *workspace, bool runs);
// Whether the full pass of such a call goes to the kernel for long runs of tiles.
bool ssd_long_runs(int B, int L, int H, int G, int chunk, int sm_count);
int launch_ssd_scalars(LaunchCtx &ctx, const ScalarsArgs &args);
size_t ssd_scalars_bytes(int B, int L, int H);       // of the arrays ssd_scalars_args lays out
// Chains nseg segment states per (sequence, head): states [B,nseg,H,P,N] holds local end states on entry
// and, for all but the first segment (keep_first: for all), entry states on exit (P = 64, N = 128).
int launch_segment_scan(LaunchCtx &ctx, float *states, const float *decay, const float *h0, int B, int nseg, int H,
                        bool keep_first);
int launch_ssd_tiles(LaunchCtx &ctx, const void *x, const void *BC, const float *dt, const float *A,
                     const float *dt_bias, const float *D, const float *h0, int B, int L, int H, int G,
                     int chunk, int sm_count, void *y, float *h_final, void *workspace,
                     bool scalars_done, bool early);

// One bf16 stream of G*N entries per token, rows ld elements apart.
struct SsdStream {
    const void *p;
    int64_t ld;
};
// The same with the injection and readout streams given apart; add: y and h_final are added to.
int launch_ssd_tiles_streams(LaunchCtx &ctx, const void *x, const SsdStream &Bs, const SsdStream &Cs, const float *dt,
                             const float *A, const float *dt_bias, const float *D, const float *h0, int B, int L,
                             int H, int G, int chunk, int sm_count, void *y, float *h_final, void *workspace,
                             bool scalars_done, bool add, bool early);
// The general form on the tile kernel: k evaluations (one per slot) added up; cmix: T*G*N bf16 scratch.
int launch_ssd_slots_tiles(LaunchCtx &ctx, const void *x_slots, const void *BC_slots, const float *dt, const float *A,
                           const float *dt_bias, const float *h0, int B, int L, int H, int G, int k, int chunk,
                           int sm_count, void *y, float *h_final, void *cmix, void *workspace);

// The same over a packed batch: nseq sequences back to back in [T, ...] arrays, sequence b holding
// tokens cu[b] .. cu[b+1]-1 (cu is a HOST array of nseq + 1 entries).  h0 / h_final are [nseq, H, P, N].
// A call makes its plan once (host work only), uploads the plan's tables in front of the router, has
// the step sizes computed beside it (ssd_packed_scalars_args) and launches the rest behind the mix.
struct PackedPlan;
std::shared_ptr<const PackedPlan> ssd_packed_plan(const int32_t *cu, int nseq, int H, int G, int chunk, int sm_count);
size_t ssd_packed_workspace_bytes(const PackedPlan &plan, int H);
int ssd_packed_segments(const PackedPlan &plan);
int ssd_packed_upload(LaunchCtx &ctx, const PackedPlan &plan, int H, void *workspace);
ScalarsArgs ssd_packed_scalars_args(const PackedPlan &plan, const float *dt, const float *A, const float *dt_bias,
                                    int64_t T, int H, void *workspace);
int launch_ssd_tiles_packed(LaunchCtx &ctx, const PackedPlan &plan, const void *x, const void *BC, const float *dt,
                            const float *A, const float *dt_bias, const float *D, const float *h0, int64_t T, int H,
                            int G, void *y, float *h_final, void *workspace);

// Sequence-sharded evaluation (every rank holds L consecutive tokens of each of B sequences), in two
// halves around the exchange of the ranks' summaries.  summary: state-only pass + local scan from a
// zero entry state; sum_state [B,H,P,N] and sum_decay [B,H] receive the shard's end state and the
// product of a_t over the shard; the workspace keeps the step sizes and the zero-entry segment
// states for the second half.  finish: all_state [R,B,H,P,N] / all_decay [R,B,H] are the gathered
// summaries in rank order; the state entering this rank's shard is chained from h0 through the
// ranks in front, y [B,L,H,P] is produced and h_end [B,H,P,N] (may be NULL) is the state after the
// shard's last token.
size_t ssd_shard_workspace_bytes(int B, int L, int H, int G, int chunk, int sm_count);
ScalarsArgs ssd_shard_scalars_args(const float *dt, const float *A, const float *dt_bias, int B, int L, int H,
                                   int G, int chunk, int sm_count, void *workspace);
int launch_ssd_shard_summary(LaunchCtx &ctx, const void *x, const void *BC, const float *dt, const float *A,
                             const float *dt_bias, int B, int L, int H, int G, int chunk, int sm_count,
                             float *sum_state, float *sum_decay, void *workspace, bool scalars_done);
int launch_ssd_shard_finish(LaunchCtx &ctx, const void *x, const void *BC, const float *D, const float *h0,
                            const float *all_state, const float *all_decay, int rank, int B, int L, int H, int G,
                            int chunk, int sm_count, void *y, float *h_end, void *workspace);

// Backward for the trained weights (router and expert matrices).
// adjoint: both passes of the recurrence's adjoint; dBC [T,S] fp32 (zeroed by the caller) receives
// dBtilde | dCtilde.  weight_grads: dpi / dg (dg [T,E] scratch) from the softmax over all E (pi [T,E], left by
// launch_router) and the unscaled slot projections slots [T*k,S] (dtype; overwritten when perm is given),
// then dW_r [E,F] and dW_e [E,S,F] (fp32, zeroed by the caller, accumulated with atomics).  perm / counts:
// the per-expert lists of launch_router (bf16; the gradient of the expert matrices then runs on the tensor
// cores), or NULL.
bool ssd_adjoint_supported(int P, int N);
int launch_ssd_adjoint(LaunchCtx &ctx, int dtype, const void *x, const void *dy, const void *BC, const float *dt,
                       const float *A, const float *dt_bias, const float *h0, int B, int L, int H, int P, int N,
                       int G, float *dBC);
// The same adjoint on tensor cores (bf16, P = 64, N = 128).  The step sizes and tile log-decays of the
// workspace (ssd_adjoint_scalars_args) are produced earlier in the stream; dBC (zeroed) is added to.
size_t ssd_adjoint_tiles_workspace_bytes(int B, int L, int H, int G, int sm_count);
ScalarsArgs ssd_adjoint_scalars_args(const float *dt, const float *A, const float *dt_bias, int B, int L, int H,
                                     void *workspace);
int launch_ssd_adjoint_tiles(LaunchCtx &ctx, const void *x, const void *dy, const void *BC, const float *h0, int B,
                             int L, int H, int G, int sm_count, float *dBC, void *workspace);
int launch_weight_grads(LaunchCtx &ctx, int dtype, const void *u, void *slots, const int32_t *idx, const float *w,
                        const float *dBC, int64_t Tn, int F, int S, int E, int k, const float *pi, float *dg,
                        const int *perm, const int *counts, int sm_count, float *dW_r, float *dW_e);
int launch_pair_outer(LaunchCtx &ctx, const void *g, const void *u, const int *perm, const int *counts, int64_t T,
                      int F, int S, int E, int k, int sm_count, float *dW);

// One warp waiting on a barrier nobody signals, with the given limit (see swimba_selftest_wait).
// out_dev: three 64-bit words on the device.
int launch_wait_selftest(LaunchCtx &ctx, long long limit_cycles, long long *out_dev);

// The rest of the block: causal depthwise convolution + SiLU over the channels [x' (D columns of a
// matrix with row stride ldx) | B'C' (S)], gated RMS norm, step-size columns to fp32.
int launch_conv_silu(LaunchCtx &ctx, int dtype, const void *xp, int64_t ldx, const void *bcp, const float *cw,
                     const float *cb, const void *state_in, int B, int L, int D, int S, int K, void *x,
                     void *bc, void *state_out);
int launch_gated_rmsnorm(LaunchCtx &ctx, int dtype, const void *y, const void *z, int64_t ldz, const float *wt,
                         int64_t T, int D, int ngroups, float eps, void *out);
int launch_dt_columns(LaunchCtx &ctx, int dtype, const void *zxdt, int64_t ld, int off, int64_t T, int H, float *dt);

// Chunked CUDA-core evaluation of the recurrence (fp32 arithmetic): the fp32 path and the bf16 shapes
// the tile kernel does not take.
int launch_ssd_sequential(LaunchCtx &ctx, int dtype, const void *x, const void *BC, const float *dt, const float *A,
                          const float *dt_bias, const float *D, const float *h0, int B, int L, int H, int P, int N,
                          int G, int sm_count, void *y, float *h_final);

// Sequences of a few tokens in a packed batch (bf16 streams, P = 64, N = 128), stepped token by token:
// seq_tab[i] = (first token, tokens, sequence index, 0), a device array of n entries; x, BC, dt, y are
// the packed arrays, h0 / h_final (may be NULL) are indexed by the sequence.
int launch_step_sequences(LaunchCtx &ctx, const void *x, const void *BC, const float *dt, const float *A,
                          const float *dt_bias, const float *D, const float *h0, const int4 *seq_tab, int n, int H,
                          int G, void *y, float *h_final);

// K4: one-token state update, state[B,H,P,N] in place.
// BC [B,bc_slots,S] is fp32 when bc_fp32, else bf16; the slots are summed.  early: what was
// launched in front lets this kernel in only after the previous writer of the states has completed
// (launch_front_small), so that they may be read before the dependency wait.
int launch_decode_update(LaunchCtx &ctx, int dtype, const void *x, void *BC, bool bc_fp32, int bc_slots, bool early,
                         const float *dt, const float *A, const float *dt_bias, const float *D,
                         float *state, int B, int H, int P, int N, int G, int sm_count, void *y);

}  // namespace swimba
