// What the two kernels over 128-token tiles share (k2_ssd.cu, which picks by RUN_TILES, and k2_run.cu): sizes and parameters.
#pragma once
#include "internal.h"
#include "ssd_scalars.cuh"
#include "tc05.cuh"

namespace swimba {

constexpr int ST = 128;                 // tokens per tile
constexpr int SP = 64;                  // head dim these kernels are built for
constexpr int SN = 128;                 // state size these kernels are built for
constexpr int NHD = 2;                  // heads per CTA
constexpr uint32_t SLAB = 16384;        // 128 rows x 128 bytes

struct SeqDesc {            // one sequence of a packed batch
    int tok0, len;          // first token in the packed arrays, tokens
    int tile0, seg0;        // first 128-token tile / first segment of the sequence in the batch-wide lists
};

struct SsdParams {
    const float *l2;        // [B,H,Lpad] log2-decay accumulated inside the 128-token tile
    const TileScalars *rec; // [B,H,Lpad/128] per-tile weights and block ends
    const TileAux *aux;     // run kernel: [B,H,Lpad/128]
    const float *D;
    const float *h_in;      // initial states: [B,H,P,N] (nseg == 1) or [B,nseg,H,P,N]; may be null
    const float *h_first;   // seg_states >= 2: states entering the first segments, [B,H,P,N]; may be null
    float *h_out;           // ssd_tiles_kernel: h_final [B,H,P,N] (last segment writes) or null
                            // ssd_state_kernel: local end states [B,nseg,H,P,N]
    float *seg_decay;       // ssd_state_kernel: [B,nseg,H] product of a_t over the segment
    int L, Lpad, H, G, nseg, seg_len;
    int split_tiles;        // > 0 (nseg == 1): every (sequence, head pair) is worked by two CTAs, see
                            // ssd_tiles_kernel
    int *d_status;
    // Packed batch (sequences of different lengths back to back in one [T, ...] array): seqs has one
    // entry per sequence plus a closing one, items lists the (sequence, segment) pairs of this launch
    // (grid.x), the scalar arrays are laid out [H, tiles of the batch], and the per-segment state
    // arrays are indexed by seqs[b].seg0 + segment.  seg_states: h_in / ssd_state_kernel's h_out are those
    // per-segment arrays (else h_in is [sequences, H, P, N]); 2: a sequence's first segment starts from
    // h_first instead; 3: so does a sequence of one segment (in-place states: the first of several reads
    // the scan's copy, since the last one writes over h_first in the same launch).  y: base of the output (ragged last
    // tiles are stored row by row).  Null seqs: dense [B, L].
    const SeqDesc *seqs;
    const int2 *items;
    int ntile_total, seg_states;
    void *y;
    // 1: y and h_out are added to, not overwritten (the slots behind the first of the general form)
    int add;
    // 1: x and the initial states are not written by anything in the same call, so that they may be read before
    // the dependency wait (everything in front of the call has completed when its first kernel runs)
    int early;
};

// pairs of heads never straddle a B/C group
__host__ __device__ inline int pairs_per_group(int H, int G) { return (H / G + NHD - 1) / NHD; }

// The run kernel (k2_run.cu) in place of the tile kernel, for dense launches whose CTAs walk RUN_TILES tiles and more.
bool ensure_ssd_run();
void launch_ssd_run(LaunchCtx &ctx, dim3 grid, const CUtensorMap &tm_b, const CUtensorMap &tm_c, const CUtensorMap &tm_x,
                    const CUtensorMap &tm_y, const SsdParams &p);

}  // namespace swimba
