// Adjoint of the recurrence on tensor cores (bf16, P = 64, N = 128): given dy, the gradients of
// sum(dy * y) with respect to the mixed streams,
//   dCtilde_t = sum_h dy_t[h]^T H_t[h],     dBtilde_s = Delta_s sum_h x_s[h]^T lambda_s[h],
// H the forward states (Theorem 1), lambda_s = sum_{t>=s} (prod_{r=s+1..t} a_r) dy_t Ctilde_t^T.
// Inside a 128-token tile, with l the log-decay accumulated from the tile's start,
//   M_h[t,s] = exp(l_t - l_s) Delta_s (dy_t . x_s)  for s <= t, else 0,
//   Y^_t = exp(l_t) dy_t,   X^_s = exp(l_last - l_s) Delta_s x_s,
// both gradients use the same matrix and the same two scaled operands:
//   dCtilde = (sum_h M_h)   Btilde + sum_h Y^_h Hin_h       Hin:  state entering the tile
//   dBtilde = (sum_h M_h)^T Ctilde + sum_h X^_h Lout_h      Lout: adjoint state entering it from behind
//   Hin  <- exp(l_last) Hin  + X^^T Btilde   (towards later tiles)
//   Lout <- exp(l_last) Lout + Y^^T Ctilde   (towards earlier tiles)
// so that the heads are summed BEFORE the products with Btilde / Ctilde.  Two kernels:
//   adjoint_states_kernel  walks the tiles (one CTA per sequence, four heads and direction), carries the
//                          states in fp32 registers and stores both at every tile boundary as bf16;
//   adjoint_tiles_kernel   one CTA per (tile, group, share of its heads) sums over the heads in tensor
//                          memory and registers and adds dBtilde | dCtilde to dBC.
// What bounds them: HBM.  Both read x and dy once; the boundary states (32 KB per head and tile) are
// written once and read once.  4 x 8192 tokens of 64 heads: 214 us (5.0 TB/s) and 220 us (4.9 TB/s; 251 us
// while the mask chose its factor entry by entry, exponentials included); two
// evaluations of the forward's tile kernel on a virtual layer of 2H heads, with its operands re-arranged
// and its per-head outputs summed by kernels of their own, took 1960 us.
#include <algorithm>

#include "internal.h"
#include "ssd_scalars.cuh"
#include "tc05.cuh"

namespace swimba {

namespace {
constexpr int AT = 128, AP = 64, AN = 128;          // tokens per tile, head dim, state size
constexpr uint32_t ASLAB = 16384;                   // 128 rows x 128 bytes

__device__ __forceinline__ void tma_store_3d(const CUtensorMap *m, const void *src, int c0, int c1, int c2)
{
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];" ::"l"(m),
                 "r"(tc::smem_u32(src)), "r"(c0), "r"(c1), "r"(c2)
                 : "memory");
}
// Eight bf16 values times (w_hi + w_lo), rounded once.
__device__ __forceinline__ uint4 scale8(const uint4 &v, __nv_bfloat162 w_hi, __nv_bfloat162 w_lo)
{
    const uint32_t in[4] = {v.x, v.y, v.z, v.w};
    uint32_t o[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const __nv_bfloat162 xv = *reinterpret_cast<const __nv_bfloat162 *>(&in[e]);
        const __nv_bfloat162 pr = __hfma2(w_hi, xv, __hmul2(w_lo, xv));
        o[e] = *reinterpret_cast<const uint32_t *>(&pr);
    }
    return make_uint4(o[0], o[1], o[2], o[3]);
}
// A weight as a two-term bf16 sum: from the record's packed word, or from a log2 value.
__device__ __forceinline__ void weight_of_word(uint32_t wp, __nv_bfloat162 &hi, __nv_bfloat162 &lo)
{
    const uint32_t h = __byte_perm(wp, 0, 0x1010), l = __byte_perm(wp, 0, 0x3232);
    hi = *reinterpret_cast<const __nv_bfloat162 *>(&h);
    lo = *reinterpret_cast<const __nv_bfloat162 *>(&l);
}
__device__ __forceinline__ void weight_of_log(float l2, __nv_bfloat162 &hi, __nv_bfloat162 &lo)
{
    const float w = tc::ex2_approx(l2);
    const __nv_bfloat16 h = __float2bfloat16_rn(w);
    const __nv_bfloat16 l = __float2bfloat16_rn(w - __bfloat162float(h));
    hi = __halves2bfloat162(h, h);
    lo = __halves2bfloat162(l, l);
}

struct AdjParams {
    const float *l2;           // [B,H,Lpad]
    const TileScalars *rec;    // [B,H,nt]
    const float *h0;           // [B,H,P,N] or null
    float *seg_states;         // [2B,nseg,H,P,N] fp32, segments in walking order (see below)
    float *seg_decay;          // [2B,nseg,H]
    int L, nt, H, G, B, nseg, seg_tiles;
    int nsplit;                // adjoint_tiles_kernel: shares a group's heads are cut into
    float *dBC;
    int *d_status;
};

// ------------------------------------------------------------------------------ boundary states
constexpr int AQ = 4;                                   // heads per CTA
constexpr int AH = 64;                                  // tokens per ring stage: half a tile
constexpr int AS_STAGES = 3;
constexpr uint32_t AHSLAB = ASLAB / 2;
constexpr uint32_t AS_STAGE_BYTES = (2 + AQ) * AHSLAB;  // U0 U1 V0 .. V3
constexpr uint32_t AS_OUT = AS_STAGES * AS_STAGE_BYTES; // staged states, one slab per head
constexpr uint32_t AS_SMALL = AS_OUT + AQ * ASLAB;
constexpr int AS_THREADS = 32 * (4 * AQ + 2);
struct __align__(16) AdjStateSmall {
    uint64_t full[AS_STAGES], scaled[AS_STAGES], empty[AS_STAGES], upd[2];
    uint32_t tmem_slot;
    int abort_flag;
};
__host__ __device__ inline int adj_quads(int H, int G) { return (H / G + AQ - 1) / AQ; }
}  // namespace

// grid = (segments x 2 B, groups x head quads); walk z = x / segments: z < B forward in time (V = x,
// U = Btilde, states Hin), z >= B backward (V = dy, U = Ctilde, states Lout).  SUMMARY: from a zero state, only the segment's end
// state and total decay leave (first pass of walks that are cut into segments); else the state in front of
// every tile, in walking order, goes out as bf16 rows [n][p].
template <bool SUMMARY>
__global__ void __launch_bounds__(AS_THREADS, 1)
adjoint_states_kernel(const __grid_constant__ CUtensorMap tmap_bc, const __grid_constant__ CUtensorMap tmap_x,
                      const __grid_constant__ CUtensorMap tmap_dy, const __grid_constant__ CUtensorMap tmap_st,
                      const AdjParams prm)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    AdjStateSmall *sm = (AdjStateSmall *)(smem + AS_SMALL);
    int *abort_flag = &sm->abort_flag;
    int *d_status = prm.d_status;
    if ((tc::smem_u32(smem) & 1023u) != 0) {
        if (threadIdx.x == 0) atomicCAS(d_status, 0, SWIMBA_ERR_DEVICE_BOUNDS);
        return;
    }
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int H = prm.H, HG = H / prm.G, qpg = adj_quads(H, prm.G), nt = prm.nt;
    const int gsegs = SUMMARY ? prm.nseg - 1 : prm.nseg;    const int seg = blockIdx.x % gsegs, z = blockIdx.x / gsegs, g = blockIdx.y / qpg, qd = blockIdx.y % qpg;
    const int dir = z >= prm.B ? 1 : 0, b = z - dir * prm.B;
    const int head0 = g * HG + qd * AQ, nh = min(AQ, HG - qd * AQ);
    const int q0 = seg * prm.seg_tiles, nq = min(prm.seg_tiles, nt - q0);     // tiles of the walk
    const int nupd = SUMMARY ? nq : nq - 1;                                  // tiles whose update is needed
    auto tile_at = [&](int q) { return dir ? nt - 1 - (q0 + q) : q0 + q; };

    if (tid == 0) {
        for (int s = 0; s < AS_STAGES; ++s) {
            tc::mbar_init(&sm->full[s], 1);
            tc::mbar_init(&sm->scaled[s], 128 * nh);
            tc::mbar_init(&sm->empty[s], 1);
        }
        tc::mbar_init(&sm->upd[0], 1);
        tc::mbar_init(&sm->upd[1], 1);
        *abort_flag = 0;
        tc::fence_mbar_init();
    }
    if (warp == 4 * AQ + 1) {
        tc::tmem_alloc(&sm->tmem_slot, 512);
        tc::tmem_relinquish();
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = sm->tmem_slot;
    grid_dep_launch();
    grid_dep_wait();

    const int uwarp = __shfl_sync(0xffffffffu, warp, 0);
    if (uwarp == 4 * AQ) {
        // ------------------------------------------------------------------ TMA producer
        const bool leader = tc::elect_one();
        const CUtensorMap *tm_v = dir ? &tmap_dy : &tmap_x;
        const int ucol = (dir ? prm.G + g : g) * AN;
        for (int n = 0; n < 2 * nupd; ++n) {
            const int s = n % AS_STAGES;
            tc::mbar_wait(&sm->empty[s], ((n / AS_STAGES) & 1) ^ 1, abort_flag, d_status);
            if (leader) {
                uint8_t *stg = smem + s * AS_STAGE_BYTES;
                const int t0 = tile_at(n >> 1) * AT + (n & 1) * AH;
                tc::mbar_arrive_expect_tx(&sm->full[s], (2 + nh) * AHSLAB);
                tc::tma_load_3d(stg, &tmap_bc, &sm->full[s], ucol, t0, b);
                tc::tma_load_3d(stg + AHSLAB, &tmap_bc, &sm->full[s], ucol + 64, t0, b);
                for (int hd = 0; hd < nh; ++hd)
                    tc::tma_load_4d(stg + (2 + hd) * AHSLAB, tm_v, &sm->full[s], 0, head0 + hd, t0, b);
            }
            __syncwarp();
        }
    } else if (uwarp == 4 * AQ + 1) {
        // ------------------------------------------------------------------ MMA issuer
        const bool leader = tc::elect_one();
        const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem, 0);
        const uint32_t id = tc::idesc_bf16(128, 64 * nh, 1, 1);          // both operands MN-major
        for (int n = 0; n < 2 * nupd; ++n) {
            const int s = n % AS_STAGES, q = n >> 1;
            tc::mbar_wait(&sm->scaled[s], (n / AS_STAGES) & 1, abort_flag, d_status);
            tc::tc_fence_after();
            if (leader) {
                const uint32_t base = tc::smem_u32(smem + s * AS_STAGE_BYTES);
                const uint64_t dU = tc::smem_desc_sw128(base, AHSLAB, 1024);
                const uint64_t dV = tc::smem_desc_sw128(base + 2 * AHSLAB, AHSLAB, 1024);
#pragma unroll
                for (int kk = 0; kk < AH / 16; ++kk)
                    tc::mma_ss(tmem_u + (q & 1) * 256, tc::smem_desc_advance(dU, kk * 2048),
                               tc::smem_desc_advance(dV, kk * 2048), id, ((n & 1) | kk) != 0);
                tc::mma_commit(&sm->empty[s]);
                if (n & 1) tc::mma_commit(&sm->upd[q & 1]);
            }
            __syncwarp();
        }
    } else if ((uwarp >> 2) < nh) {
        // ------------------------------------------------------------------ compute warps: four per head
        const int hd = warp >> 2, wq = warp & 3, h = head0 + hd;
        const int i = wq * 32 + lane;                                   // state index n
        const int64_t row = ((int64_t)b * H + h) * nt;                   // record of tile 0
        const int64_t srow_seg = (((int64_t)z * prm.nseg + seg) * H + h) * (AP * AN);
        float st[AP];
        {
            const float *src = nullptr;
            if (!SUMMARY) {
                if (seg > 0) src = prm.seg_states + srow_seg;
                else if (dir == 0 && prm.h0) src = prm.h0 + ((int64_t)b * H + h) * (AP * AN);
            }
#pragma unroll
            for (int p = 0; p < AP; ++p) st[p] = src ? src[p * AN + i] : 0.f;
        }
        uint8_t *s_out = smem + AS_OUT + hd * ASLAB;
        const uint32_t tm = tmem + ((uint32_t)(wq * 32) << 16) + 64 * hd;
        // this thread's share of a stage: token row i / 2, four of its eight 16-byte chunks
        const int srow = i >> 1, shalf = i & 1;
        auto load_word = [&](int q, int half) {
            const int64_t r = row + tile_at(q);
            return dir ? __float_as_uint(prm.l2[r * AT + half * AH + srow]) : prm.rec[r].wp[half * AH + srow];
        };
        uint32_t word[2] = {0u, 0u};
        float end = 0.f, end_next = 0.f, total = 0.f;                    // log2 decay of tile q - 1, q; of the walk
        if (nupd > 0) {
            word[0] = load_word(0, 0);
            word[1] = load_word(0, 1);
            end_next = prm.rec[row + tile_at(0)].ends[3];
        }
        auto update = [&](int q) {                                       // st <- 2^end st + U^T V of tile q
            tc::mbar_wait(&sm->upd[q & 1], (q >> 1) & 1, abort_flag, d_status);
            tc::tc_fence_after();
            const float dec = tc::ex2_approx(end);
            total += end;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint32_t d[16];
                tc::tmem_ld16(tm + (q & 1) * 256 + 16 * c, d);
                tc::tmem_ld_wait();
#pragma unroll
                for (int e = 0; e < 16; ++e) st[16 * c + e] = fmaf(dec, st[16 * c + e], __uint_as_float(d[e]));
            }
            tc::tc_fence_before();
        };
        for (int q = 0; q < nq; ++q) {
            if (q < nupd) {
                const uint32_t w0 = word[0], w1 = word[1];
                if (q + 1 < nupd) { word[0] = load_word(q + 1, 0); word[1] = load_word(q + 1, 1); }
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    const int n = 2 * q + half, s = n % AS_STAGES;
                    __nv_bfloat162 hi, lo;
                    if (dir) weight_of_log(__uint_as_float(half ? w1 : w0), hi, lo);
                    else weight_of_word(half ? w1 : w0, hi, lo);
                    tc::mbar_wait(&sm->full[s], (n / AS_STAGES) & 1, abort_flag, d_status);
                    uint8_t *v = smem + s * AS_STAGE_BYTES + (2 + hd) * AHSLAB;
                    uint4 xr[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c) xr[c] = *reinterpret_cast<const uint4 *>(v + tc::sw128_offset(srow, 4 * shalf + c));
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        *reinterpret_cast<uint4 *>(v + tc::sw128_offset(srow, 4 * shalf + c)) = scale8(xr[c], hi, lo);
                    tc::fence_proxy_async_smem();
                    tc::mbar_arrive(&sm->scaled[s]);
                }
            }
            if (q > 0) update(q - 1);
            end = end_next;                                              // tile q's decay
            if (q + 1 < nupd) end_next = prm.rec[row + tile_at(q + 1)].ends[3];
            if (!SUMMARY) {
                // the state in front of tile q, as rows [n][p]
                if (i == 0) tc::bulk_wait_read_all();                    // the previous one has left the slab
                tc::named_bar_sync(1 + hd, 128);
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    *reinterpret_cast<uint4 *>(s_out + tc::sw128_offset(i, c)) =
                        make_uint4(tc::pack_bf16x2(st[8 * c], st[8 * c + 1]), tc::pack_bf16x2(st[8 * c + 2], st[8 * c + 3]),
                                   tc::pack_bf16x2(st[8 * c + 4], st[8 * c + 5]), tc::pack_bf16x2(st[8 * c + 6], st[8 * c + 7]));
                tc::fence_proxy_async_smem();
                tc::named_bar_sync(1 + hd, 128);
                if (i == 0) {
                    tma_store_3d(&tmap_st, s_out, 0, 0, (z * nt + tile_at(q)) * H + h);
                    tc::bulk_commit_group();
                }
            }
        }
        if (SUMMARY) {
            if (nq > 0) update(nq - 1);
            float *dst = prm.seg_states + srow_seg;
#pragma unroll
            for (int p = 0; p < AP; ++p) dst[p * AN + i] = st[p];
            if (i == 0) prm.seg_decay[((int64_t)z * prm.nseg + seg) * H + h] = tc::ex2_approx(total);
        } else if (i == 0) {
            tc::bulk_wait_read_all();
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == 4 * AQ + 1) tc::tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------------------ head sums per tile
namespace {
constexpr int AC_STAGES = 3;
constexpr uint32_t AC_STAGE_BYTES = 4 * ASLAB;           // X dY Hin Lout, or Btilde (2 slabs) Ctilde (2 slabs)
constexpr uint32_t AC_SMALL = AC_STAGES * AC_STAGE_BYTES;
constexpr int AC_THREADS = 32 * 18;
constexpr uint32_t AC_ROW = AN * 4 + 16;                 // staged fp32 output row
constexpr uint32_t TC_DC = 0, TC_DB = 128, TC_S = 256;   // tensor memory columns
struct __align__(16) AdjTileSmall {
    TileScalars sc[AC_STAGES];
    float l2[AC_STAGES][AT];
    uint64_t full[AC_STAGES], scaled[AC_STAGES], empty[AC_STAGES], s_full[2], s_free[2], heads_done, m_ready, out_full;
    uint32_t tmem_slot;
    int abort_flag;
};
static_assert(2 * AT * AC_ROW <= AC_STAGES * AC_STAGE_BYTES, "the staged outputs reuse the ring");
}  // namespace

// grid = (tiles x shares, G, B)
__global__ void __launch_bounds__(AC_THREADS, 1)
adjoint_tiles_kernel(const __grid_constant__ CUtensorMap tmap_bc, const __grid_constant__ CUtensorMap tmap_x,
                     const __grid_constant__ CUtensorMap tmap_dy, const __grid_constant__ CUtensorMap tmap_st,
                     const AdjParams prm)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    AdjTileSmall *sm = (AdjTileSmall *)(smem + AC_SMALL);
    int *abort_flag = &sm->abort_flag;
    int *d_status = prm.d_status;
    if ((tc::smem_u32(smem) & 1023u) != 0) {
        if (threadIdx.x == 0) atomicCAS(d_status, 0, SWIMBA_ERR_DEVICE_BOUNDS);
        return;
    }
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int H = prm.H, HG = H / prm.G, nt = prm.nt;
    const int tile = blockIdx.x / prm.nsplit, share = blockIdx.x % prm.nsplit, g = blockIdx.y, b = blockIdx.z;
    const int ha = (int)((int64_t)HG * share / prm.nsplit), hb = (int)((int64_t)HG * (share + 1) / prm.nsplit);
    const int head0 = g * HG + ha, nheads = hb - ha;                   // (nsplit <= HG: at least one)
    const int t0 = tile * AT;

    if (tid == 0) {
        for (int s = 0; s < AC_STAGES; ++s) {
            tc::mbar_init(&sm->full[s], 1);
            tc::mbar_init(&sm->scaled[s], 512);
            tc::mbar_init(&sm->empty[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            tc::mbar_init(&sm->s_full[s], 1);
            tc::mbar_init(&sm->s_free[s], 512);
        }
        tc::mbar_init(&sm->heads_done, 1);
        tc::mbar_init(&sm->m_ready, 512);
        tc::mbar_init(&sm->out_full, 1);
        *abort_flag = 0;
        tc::fence_mbar_init();
    }
    if (warp == 17) {
        tc::tmem_alloc(&sm->tmem_slot, 512);
        tc::tmem_relinquish();
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = sm->tmem_slot;
    grid_dep_launch();
    grid_dep_wait();

    const int uwarp = __shfl_sync(0xffffffffu, warp, 0);
    const int slot_bc = nheads % AC_STAGES, slot_m = (nheads + 1) % AC_STAGES;
    if (uwarp == 16) {
        // ------------------------------------------------------------------ TMA producer
        const bool leader = tc::elect_one();
        for (int n = 0; n <= nheads; ++n) {
            const int s = n % AC_STAGES;
            tc::mbar_wait(&sm->empty[s], ((n / AC_STAGES) & 1) ^ 1, abort_flag, d_status);
            if (leader) {
                uint8_t *stg = smem + s * AC_STAGE_BYTES;
                uint64_t *bar = &sm->full[s];
                if (n < nheads) {
                    const int h = head0 + n;
                    const int64_t r = ((int64_t)b * H + h) * nt + tile;
                    tc::mbar_arrive_expect_tx(bar, 4 * ASLAB + (uint32_t)sizeof(TileScalars) + AT * 4);
                    tc::tma_load_4d(stg, &tmap_x, bar, 0, h, t0, b);
                    tc::tma_load_4d(stg + ASLAB, &tmap_dy, bar, 0, h, t0, b);
                    tc::bulk_load(&sm->sc[s], prm.rec + r, (uint32_t)sizeof(TileScalars), bar);
                    tc::bulk_load(sm->l2[s], prm.l2 + r * AT, AT * 4, bar);
                    tc::tma_load_3d(stg + 2 * ASLAB, &tmap_st, bar, 0, 0, (b * nt + tile) * H + h);
                    tc::tma_load_3d(stg + 3 * ASLAB, &tmap_st, bar, 0, 0, ((prm.B + b) * nt + tile) * H + h);
                } else {
                    tc::mbar_arrive_expect_tx(bar, 4 * ASLAB);
                    tc::tma_load_3d(stg, &tmap_bc, bar, g * AN, t0, b);
                    tc::tma_load_3d(stg + ASLAB, &tmap_bc, bar, g * AN + 64, t0, b);
                    tc::tma_load_3d(stg + 2 * ASLAB, &tmap_bc, bar, (prm.G + g) * AN, t0, b);
                    tc::tma_load_3d(stg + 3 * ASLAB, &tmap_bc, bar, (prm.G + g) * AN + 64, t0, b);
                }
            }
            __syncwarp();
        }
    } else if (uwarp == 17) {
        // ------------------------------------------------------------------ MMA issuer
        const bool leader = tc::elect_one();
        const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem, 0);
        const uint32_t base = tc::smem_u32(smem);
        const uint64_t dk = tc::smem_desc_sw128(base, 16, 1024);             // K-major
        const uint64_t dmn = tc::smem_desc_sw128(base, ASLAB, 1024);         // MN-major, two slabs
        constexpr uint32_t id_kk = tc::idesc_bf16(128, 128, 0, 0);
        auto issue_s = [&](int n) {                                          // S = dY X^T
            const int s = n % AC_STAGES;
            tc::mbar_wait(&sm->full[s], (n / AC_STAGES) & 1, abort_flag, d_status);
            if (n >= 2) tc::mbar_wait(&sm->s_free[n & 1], ((n - 2) >> 1) & 1, abort_flag, d_status);
            tc::tc_fence_after();
            if (leader) {
                const uint64_t dX = tc::smem_desc_advance(dk, s * AC_STAGE_BYTES), dY = tc::smem_desc_advance(dX, ASLAB);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                    tc::mma_ss(tmem_u + TC_S + (n & 1) * 128, tc::smem_desc_advance(dY, kk * 32),
                               tc::smem_desc_advance(dX, kk * 32), id_kk, kk > 0);
                tc::mma_commit(&sm->s_full[n & 1]);
            }
            __syncwarp();
        };
        issue_s(0);
        if (nheads > 1) issue_s(1);
        for (int n = 0; n < nheads; ++n) {
            const int s = n % AC_STAGES;
            tc::mbar_wait(&sm->scaled[s], (n / AC_STAGES) & 1, abort_flag, d_status);
            tc::tc_fence_after();
            if (leader) {
                const uint64_t dX = tc::smem_desc_advance(dk, s * AC_STAGE_BYTES), dY = tc::smem_desc_advance(dX, ASLAB);
                const uint64_t dH = tc::smem_desc_advance(dX, 2 * ASLAB), dL = tc::smem_desc_advance(dX, 3 * ASLAB);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    tc::mma_ss(tmem_u + TC_DC, tc::smem_desc_advance(dY, kk * 32), tc::smem_desc_advance(dH, kk * 32),
                               id_kk, (n | kk) != 0);
                    tc::mma_ss(tmem_u + TC_DB, tc::smem_desc_advance(dX, kk * 32), tc::smem_desc_advance(dL, kk * 32),
                               id_kk, (n | kk) != 0);
                }
                tc::mma_commit(&sm->empty[s]);
                if (n == nheads - 1) tc::mma_commit(&sm->heads_done);
            }
            __syncwarp();
            if (n + 2 < nheads) issue_s(n + 2);
        }
        // dC += M Btilde, dB += M^T Ctilde
        tc::mbar_wait(&sm->full[slot_bc], (nheads / AC_STAGES) & 1, abort_flag, d_status);
        tc::mbar_wait(&sm->m_ready, 0, abort_flag, d_status);
        tc::tc_fence_after();
        if (leader) {
            const uint32_t om = slot_m * AC_STAGE_BYTES, ob = slot_bc * AC_STAGE_BYTES;
            constexpr uint32_t id_c = tc::idesc_bf16(128, 128, 0, 1), id_b = tc::idesc_bf16(128, 128, 1, 1);
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) {
                tc::mma_ss(tmem_u + TC_DC, tc::smem_desc_advance(dk, om + (kk >> 2) * ASLAB + (kk & 3) * 32),
                           tc::smem_desc_advance(dmn, ob + kk * 2048), id_c, 1);
                tc::mma_ss(tmem_u + TC_DB, tc::smem_desc_advance(dmn, om + kk * 2048),
                           tc::smem_desc_advance(dmn, ob + 2 * ASLAB + kk * 2048), id_b, 1);
            }
            tc::mma_commit(&sm->out_full);
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------------ compute warps
        // scaling: thread = (row tid / 4, two of its eight 16-byte chunks) of both operands;
        // M: warp = (row block wq, column block cq) of 32 x 32
        const int srow = tid >> 2, sch = (tid & 3) * 2;
        const int wq = warp & 3, cq = warp >> 2, i = wq * 32 + lane;
        const uint32_t lane_base = tmem + ((uint32_t)(wq * 32) << 16);
        uint64_t acc[16];                                    // two fp32 sums each
#pragma unroll
        for (int e = 0; e < 16; ++e) acc[e] = 0;
        for (int n = 0; n < nheads; ++n) {
            const int s = n % AC_STAGES;
            tc::mbar_wait(&sm->full[s], (n / AC_STAGES) & 1, abort_flag, d_status);
            uint8_t *sx = smem + s * AC_STAGE_BYTES, *sy = sx + ASLAB;
            const TileScalars *sc = &sm->sc[s];
            const float *l2s = sm->l2[s];
            uint4 xv[2], yv[2];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const uint32_t off = tc::sw128_offset(srow, sch + c);
                xv[c] = *reinterpret_cast<const uint4 *>(sx + off);
                yv[c] = *reinterpret_cast<const uint4 *>(sy + off);
            }
            __nv_bfloat162 xh, xl, yh, yl;
            weight_of_word(sc->wp[srow], xh, xl);
            weight_of_log(l2s[srow], yh, yl);
            const float l_i = l2s[i];
            const float l_end = sc->ends[cq];
            // S has been formed from the unscaled rows: they can be overwritten
            tc::mbar_wait(&sm->s_full[n & 1], (n >> 1) & 1, abort_flag, d_status);
            tc::tc_fence_after();
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const uint32_t off = tc::sw128_offset(srow, sch + c);
                *reinterpret_cast<uint4 *>(sx + off) = scale8(xv[c], xh, xl);
                *reinterpret_cast<uint4 *>(sy + off) = scale8(yv[c], yh, yl);
            }
            if (cq <= wq) {
                const uint32_t sa = lane_base + TC_S + (n & 1) * 128 + cq * 32;
                const float *cb = sc->cb + cq * 32;
                const float up = l_i - l_end;          // row factor 2^up: <= 1 below the diagonal blocks
                // a diagonal block's row factor is >= 1 and below 2^96: it is applied as a product.  Columns of a block
                // that decays by more come without a factor: their exponents are formed per entry (where <= 0)
                const float l_beg = cq == 0 ? 0.f : sc->ends[cq - 1];
                const bool prod = !block_fast(l_beg, l_end);
                const float rf = tc::ex2_approx(prod ? up : 0.f);
                const uint64_t rf2 = tc::f32x2(rf, rf);
                uint32_t v[32];
                tc::tmem_ld32(sa, v);
                tc::tmem_ld_wait();
                if (cq == wq) {
#pragma unroll
                    for (int e = 0; e < 32; ++e) v[e] = e <= lane ? v[e] : 0u;
                }
                if (prod) {
#pragma unroll
                    for (int e = 0; e < 32; e += 4) {
                        const ulonglong2 w4 = *reinterpret_cast<const ulonglong2 *>(cb + e);
                        acc[e / 2] = tc::f32x2_fma(tc::f32x2(__uint_as_float(v[e]), __uint_as_float(v[e + 1])),
                                                   tc::f32x2_mul(w4.x, rf2), acc[e / 2]);
                        acc[e / 2 + 1] = tc::f32x2_fma(tc::f32x2(__uint_as_float(v[e + 2]), __uint_as_float(v[e + 3])),
                                                       tc::f32x2_mul(w4.y, rf2), acc[e / 2 + 1]);
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < 32; e += 2) {
                        // (behind the diagonal the exponent is positive: the entry there is zero, its factor must be finite)
                        const float *lc = l2s + cq * 32;
                        const float f0 = cq < wq || e <= lane ? cb[e] * tc::ex2_approx(l_i - lc[e]) : 0.f;
                        const float f1 = cq < wq || e + 1 <= lane ? cb[e + 1] * tc::ex2_approx(l_i - lc[e + 1]) : 0.f;
                        acc[e / 2] = tc::f32x2_fma(tc::f32x2(__uint_as_float(v[e]), __uint_as_float(v[e + 1])),
                                                   tc::f32x2(f0, f1), acc[e / 2]);
                    }
                }
            }
            tc::tc_fence_before();
            tc::fence_proxy_async_smem();
            tc::mbar_arrive(&sm->scaled[s]);
            tc::mbar_arrive(&sm->s_free[n & 1]);
        }
        // ---- M (bf16) as two slabs of 64 columns; the slot is free once all heads' products are done
        tc::mbar_wait(&sm->heads_done, 0, abort_flag, d_status);
        {
            uint8_t *m = smem + slot_m * AC_STAGE_BYTES + (cq >> 1) * ASLAB;
#pragma unroll
            for (int c = 0; c < 4; ++c)
                *reinterpret_cast<uint4 *>(m + tc::sw128_offset(i, (cq & 1) * 4 + c)) =
                    make_uint4(tc::f32x2_bf16(acc[4 * c]), tc::f32x2_bf16(acc[4 * c + 1]), tc::f32x2_bf16(acc[4 * c + 2]),
                               tc::f32x2_bf16(acc[4 * c + 3]));
        }
        tc::fence_proxy_async_smem();
        tc::mbar_arrive(&sm->m_ready);
        // ---- results: staged rows, added to dBC (other shares of the heads add to the same rows)
        tc::mbar_wait(&sm->out_full, 0, abort_flag, d_status);
        tc::tc_fence_after();
#pragma unroll
        for (int mat = 0; mat < 2; ++mat) {
            uint8_t *dst = smem + mat * AT * AC_ROW + i * AC_ROW + cq * 128;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                uint32_t v[16];
                tc::tmem_ld16(lane_base + (mat ? TC_DB : TC_DC) + cq * 32 + 16 * c, v);
                tc::tmem_ld_wait();
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    *reinterpret_cast<uint4 *>(dst + 64 * c + 16 * e) = make_uint4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
            }
        }
        tc::tc_fence_before();
        tc::fence_proxy_async_smem();
        tc::named_bar_sync(1, 512);
        if (tid < 2 * AT) {
            const int mat = tid >> 7, r = tid & 127;
            if (t0 + r < prm.L)
                tc::bulk_reduce_add_f32(prm.dBC + ((int64_t)b * prm.L + t0 + r) * (2 * prm.G * AN) + (mat ? g : prm.G + g) * AN,
                                    smem + mat * AT * AC_ROW + r * AC_ROW, AN * 4);
            tc::bulk_commit_group();
            tc::bulk_wait_read_all();
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == 17) tc::tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------------------ host side
namespace {
// Segments of the state walks.  One CTA carries four heads of a sequence in one direction; where that
// leaves most SMs idle the walks are cut, which costs a summary pass over the same rows: two passes of
// 1/nseg against one, so from three segments on.
int adj_seg_tiles(int B, int nt, int H, int G, int sm_count)
{
    const int64_t ctas = 2 * (int64_t)B * G * adj_quads(H, G);
    const int64_t nseg = sm_count / ctas;
    if (nseg < 3 || nt < 6) return nt;
    const int st = (int)ceil_div64(nt, nseg);
    return st < 2 ? 2 : st;
}
// States at segment starts (of all heads each) that a call reserves: at least what any call with no more
// sequences of no more tokens takes (at most `cut` sequences are few enough to be cut).
int64_t adj_segment_states(int B, int nt, int H, int G, int sm_count)
{
    const int64_t quads = (int64_t)G * adj_quads(H, G);
    const int64_t cut = std::min<int64_t>(B, sm_count / (6 * quads));
    return nt < 6 ? 0 : std::min<int64_t>(2 * cut * ceil_div(nt, 2), sm_count / quads);
}
struct AdjLayout {
    size_t scal, states, seg_states, seg_decay, total;
    int nt, seg_tiles, nseg;
};
AdjLayout adj_layout(int B, int L, int H, int G, int sm_count)
{
    auto up = [](size_t v) { return (v + 255) / 256 * 256; };
    AdjLayout l;
    l.nt = ceil_div(L, AT);
    l.seg_tiles = adj_seg_tiles(B, l.nt, H, G, sm_count);
    l.nseg = ceil_div(l.nt, l.seg_tiles);
    const size_t nstates = (size_t)adj_segment_states(B, l.nt, H, G, sm_count);
    size_t off = 0;
    l.scal = off;   off += ssd_scalars_bytes(B, L, H);
    l.states = off; off += up((size_t)2 * B * l.nt * H * AN * AP * 2);
    l.seg_states = off; off += up(nstates * H * AN * AP * sizeof(float));
    l.seg_decay = off;  off += up(nstates * H * sizeof(float));
    l.total = off;
    return l;
}
// Shares the heads of a tile are cut into: whole rounds of CTAs, each costing its heads plus about three
// heads' time for the products with Btilde / Ctilde and the results.
int adj_split(int64_t tiles, int HG, int sm_count)
{
    int best = 1;
    int64_t best_cost = -1;
    for (int ns = 1; ns <= HG && ns <= 16; ++ns) {
        const int64_t cost = ceil_div64(tiles * ns, sm_count) * (ceil_div(HG, ns) + 3);
        if (best_cost < 0 || cost < best_cost) { best_cost = cost; best = ns; }
    }
    return best;
}
}  // namespace

size_t ssd_adjoint_tiles_workspace_bytes(int B, int L, int H, int G, int sm_count)
{
    return adj_layout(B, L, H, G, sm_count).total;
}

ScalarsArgs ssd_adjoint_scalars_args(const float *dt, const float *A, const float *dt_bias, int B, int L, int H,
                                     void *workspace)
{
    return ssd_scalars_args(dt, A, dt_bias, B, L, H, workspace, false);
}

int launch_ssd_adjoint_tiles(LaunchCtx &ctx, const void *x, const void *dy, const void *BC, const float *h0, int B,
                             int L, int H, int G, int sm_count, float *dBC, void *workspace)
{
    if (B <= 0 || L <= 0) return SWIMBA_OK;
    const AdjLayout lay = adj_layout(B, L, H, G, sm_count);
    char *ws = (char *)workspace;
    const int S = 2 * G * AN;
    CUtensorMap bc_h, bc_t, x_h, x_t, dy_h, dy_t, st;
    {
        const uint64_t d3[3] = {(uint64_t)S, (uint64_t)L, (uint64_t)B};
        const uint64_t s3[2] = {(uint64_t)S * 2, (uint64_t)L * S * 2};
        const uint64_t d4[4] = {(uint64_t)AP, (uint64_t)H, (uint64_t)L, (uint64_t)B};
        const uint64_t s4[3] = {(uint64_t)AP * 2, (uint64_t)H * AP * 2, (uint64_t)L * H * AP * 2};
        const uint32_t b3h[3] = {64, AH, 1}, b3t[3] = {64, AT, 1}, b4h[4] = {AP, 1, AH, 1}, b4t[4] = {AP, 1, AT, 1};
        const uint64_t ds[3] = {(uint64_t)AP, (uint64_t)AN, (uint64_t)2 * B * lay.nt * H};
        const uint64_t ss[2] = {(uint64_t)AP * 2, (uint64_t)AP * AN * 2};
        const uint32_t bs[3] = {AP, AN, 1};
        if (!encode_tmap_bf16_cached(ctx.tmaps, &bc_h, BC, 3, d3, s3, b3h) ||
            !encode_tmap_bf16_cached(ctx.tmaps, &bc_t, BC, 3, d3, s3, b3t) ||
            !encode_tmap_bf16_cached(ctx.tmaps, &x_h, x, 4, d4, s4, b4h) ||
            !encode_tmap_bf16_cached(ctx.tmaps, &x_t, x, 4, d4, s4, b4t) ||
            !encode_tmap_bf16_cached(ctx.tmaps, &dy_h, dy, 4, d4, s4, b4h) ||
            !encode_tmap_bf16_cached(ctx.tmaps, &dy_t, dy, 4, d4, s4, b4t) ||
            !encode_tmap_bf16_cached(ctx.tmaps, &st, ws + lay.states, 3, ds, ss, bs))
            return SWIMBA_ERR_CUDA;
    }
    const size_t smem_s = AS_SMALL + sizeof(AdjStateSmall), smem_t = AC_SMALL + sizeof(AdjTileSmall);
    if (!ensure_dynamic_smem((const void *)adjoint_states_kernel<true>, smem_s) ||
        !ensure_dynamic_smem((const void *)adjoint_states_kernel<false>, smem_s) ||
        !ensure_dynamic_smem((const void *)adjoint_tiles_kernel, smem_t))
        return SWIMBA_ERR_CUDA;
    AdjParams p;
    const ScalarsArgs sa = ssd_scalars_args(nullptr, nullptr, nullptr, B, L, H, ws + lay.scal, false);
    p.l2 = sa.l2; p.rec = sa.rec; p.h0 = h0;
    p.seg_states = (float *)(ws + lay.seg_states); p.seg_decay = (float *)(ws + lay.seg_decay);
    p.L = L; p.nt = lay.nt; p.H = H; p.G = G; p.B = B; p.nseg = lay.nseg; p.seg_tiles = lay.seg_tiles;
    p.nsplit = adj_split((int64_t)B * lay.nt * G, H / G, sm_count);
    p.dBC = dBC;
    p.d_status = ctx.d_status;
    const unsigned quads = (unsigned)(G * adj_quads(H, G));
    if (lay.nseg > 1) {
        ctx.begin(STAGE_ADJOINT_STATES);
        launch_kernel(adjoint_states_kernel<true>, dim3((unsigned)(lay.nseg - 1) * 2u * B, quads), dim3(AS_THREADS), smem_s,
                      ctx.stream, true, bc_h, x_h, dy_h, st, p);
        ctx.end();
        for (int dir = 0; dir < 2; ++dir) {
            const int rc = launch_segment_scan(ctx, p.seg_states + (size_t)dir * B * lay.nseg * H * AN * AP,
                                               p.seg_decay + (size_t)dir * B * lay.nseg * H, dir == 0 ? h0 : nullptr, B,
                                               lay.nseg, H, false);
            if (rc != SWIMBA_OK) return rc;
        }
    }
    ctx.begin(STAGE_ADJOINT_STATES);
    launch_kernel(adjoint_states_kernel<false>, dim3((unsigned)lay.nseg * 2u * B, quads), dim3(AS_THREADS), smem_s, ctx.stream,
                  true, bc_h, x_h, dy_h, st, p);
    ctx.end();
    ctx.begin(STAGE_SSD_ADJOINT);
    launch_kernel(adjoint_tiles_kernel, dim3((unsigned)(lay.nt * p.nsplit), (unsigned)G, (unsigned)B), dim3(AC_THREADS),
                  smem_t, ctx.stream, true, bc_t, x_t, dy_t, st, p);
    ctx.end();
    return cudaGetLastError() == cudaSuccess ? SWIMBA_OK : SWIMBA_ERR_CUDA;
}

}  // namespace swimba
