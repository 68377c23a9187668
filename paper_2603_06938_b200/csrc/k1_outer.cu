// Gradient of the expert matrices on CTA pairs (tcgen05, cta_group::2):
//   dW_e[e][s, f] += sum over the (token, slot) entries r routed to e of  g_r[s] u_t(r)[f],
// g_r = pi_{t,e} dBC_t as bf16 rows by entry (written by dpi_dg_kernel), u the token features.  Both
// operands are gathered rows with the contraction index (the entry) as the row, i.e. MN-major tiles; a
// 256 (s) x 256 (f) tile of one expert's matrix per pair, 64 entries per step.
//
// Work split: the steps of all tiles, expert by expert, form one line that is cut into as many equal runs
// as there are pairs (an expert's list can be any length); a run adds its part of a tile in fp32 at every
// tile boundary it meets.  That balances the pairs to a step and keeps the additions to about one more
// tile per pair, where runs of fixed length would add the whole matrix once per 1000 entries.
// What bounds it: the rows gathered from L2, 64 KB per step and pair against 512 cycles of tensor time.
// 65536 entries of 8 experts, S = 256, F = 2048: mma.sync tiles of 128 x 128 over runs of 4096 tokens
// 711 us, this kernel 75 us (0.92 PFLOP/s).
#include "internal.h"
#include "pair.cuh"

namespace swimba {

namespace {
constexpr int PO_BM = 256, PO_BN = 256, PO_BK = 64, PO_STAGES = 5;
constexpr uint32_t PO_SLAB = 64 * 128;                       // 64 entries x 64 columns
constexpr uint32_t PO_STAGE_BYTES = 4 * PO_SLAB;             // per CTA: 128 columns of g, 128 of u
constexpr int PO_COLS = 64;                                  // columns of a staged output row
constexpr uint32_t PO_ROW = PO_COLS * 4 + 16;
constexpr uint32_t PO_OUT = PO_STAGES * PO_STAGE_BYTES;
constexpr uint32_t PO_SMALL = PO_OUT + 128 * PO_ROW;
constexpr int PO_LIST = 16;                                  // steps whose list entries are held
constexpr int PO_EPI_WARP = 4, PO_GATHER_WARP = 8, PO_GATHER = 256;
constexpr int PO_THREADS = 32 * PO_GATHER_WARP + PO_GATHER;

struct __align__(16) OuterSmall {
    int list[PO_LIST][PO_BK + 4];                            // list entries of the steps ahead (from the 16-byte
                                                             // boundary at or below the first one on)
    uint64_t full[PO_STAGES], empty[PO_STAGES], gathered[PO_STAGES], acc_full[2], acc_empty[2];
    uint64_t list_full[PO_LIST], list_free[PO_LIST];
    uint32_t tmem_slot;
    int abort_flag;
    int64_t step_end[SWIMBA_MAX_EXPERTS];                    // steps of experts 0 .. e, summed
    int cnt[SWIMBA_MAX_EXPERTS];
};

struct OuterArgs {
    const __nv_bfloat16 *g, *u;       // [T*k, S], [T, F]
    const int *perm, *counts;         // (up to 256 bytes behind the last list are read, not used)
    int64_t cap;
    float *dW;                        // [E, S, F]
    int E, F, S, k, check;
    int *d_status;
};
}  // namespace

__global__ void __launch_bounds__(PO_THREADS, 1)
pair_outer_kernel(const OuterArgs p)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    OuterSmall *sm = (OuterSmall *)(smem + PO_SMALL);
    int *abort_flag = &sm->abort_flag;
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const uint32_t rank = tc::cluster_rank();
    const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
    if ((tc::smem_u32(smem) & 1023u) != 0) {      // (the same in both CTAs)
        if (tid == 0) atomicCAS(p.d_status, 0, SWIMBA_ERR_DEVICE_BOUNDS);
        return;
    }
    if (tid == 0) {
        for (int s = 0; s < PO_STAGES; ++s) {
            tc::mbar_init(&sm->full[s], 2);                 // the gathered rows of either CTA
            tc::mbar_init(&sm->gathered[s], PO_GATHER);
            tc::mbar_init(&sm->empty[s], 1);
        }
        for (int s = 0; s < PO_LIST; ++s) {
            tc::mbar_init(&sm->list_full[s], 1);
            tc::mbar_init(&sm->list_free[s], PO_GATHER / 32);
        }
        for (int s = 0; s < 2; ++s) {
            tc::mbar_init(&sm->acc_full[s], 1);
            tc::mbar_init(&sm->acc_empty[s], 2 * 4);
        }
        *abort_flag = 0;
        tc::fence_mbar_init();
    }
    if (warp == 1) tc::pair_tmem_alloc(&sm->tmem_slot);
    grid_dep_launch();
    grid_dep_wait();
    const int ns = ceil_div(p.S, PO_BM), nf = ceil_div(p.F, PO_BN);
    if (warp == 2) {
        int c[2];
        int64_t n[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            c[q] = 2 * lane + q < p.E ? p.counts[2 * lane + q] : 0;
            if (p.check && (c[q] < 0 || c[q] > p.cap)) {
                atomicCAS(p.d_status, 0, SWIMBA_ERR_DEVICE_BOUNDS);
                c[q] = 0;
            }
            n[q] = (int64_t)((c[q] + PO_BK - 1) / PO_BK) * ns * nf;
        }
        int64_t incl = n[0] + n[1];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t nb = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += nb;
        }
        sm->step_end[2 * lane] = incl - n[1];
        sm->step_end[2 * lane + 1] = incl;
        sm->cnt[2 * lane] = c[0];
        sm->cnt[2 * lane + 1] = c[1];
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::cluster_sync();
    tc::tc_fence_after();
    const uint32_t tmem = sm->tmem_slot;
    const int64_t total = sm->step_end[SWIMBA_MAX_EXPERTS - 1];
    const int64_t run_a = total * pair / npairs, run_b = total * (pair + 1) / npairs;

    // Part of a tile at step `pos` of the line: expert, first row and column, first step, steps.
    struct Part { int e, cnt, s0, f0, k0, n; };
    auto part_at = [&](int64_t pos) {
        Part r;
        const unsigned lo = __ballot_sync(0xffffffffu, sm->step_end[lane] > pos);
        if (lo) r.e = __ffs(lo) - 1;
        else r.e = 32 + __ffs(__ballot_sync(0xffffffffu, sm->step_end[32 + lane] > pos)) - 1;
        r.cnt = sm->cnt[r.e];
        const int ks = (r.cnt + PO_BK - 1) / PO_BK;
        const int64_t local = pos - (r.e > 0 ? sm->step_end[r.e - 1] : 0);
        const int tile = (int)(local / ks);
        r.k0 = (int)(local - (int64_t)tile * ks);
        r.s0 = (tile / nf) * PO_BM;
        r.f0 = (tile % nf) * PO_BN;
        r.n = (int)min((int64_t)(ks - r.k0), run_b - pos);
        return r;
    };

    if (warp == 1 && rank == 0) {
        // ------------------------------------------------------------------ products (first CTA)
        const bool elected = tc::elect_one();
        const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem, 0);
        const uint64_t d0 = tc::smem_desc_sw128(tc::smem_u32(smem), PO_SLAB, 1024);
        constexpr uint32_t idesc = tc::idesc_bf16(PO_BM, PO_BN, 1, 1);        // both operands MN-major
        uint32_t n = 0, it = 0;
        for (int64_t pos = run_a; pos < run_b; ++it) {
            const Part pt = part_at(pos);
            const uint32_t buf = it & 1, acc = tmem_u + buf * PO_BN;
            tc::mbar_wait(&sm->acc_empty[buf], ((it >> 1) & 1) ^ 1, abort_flag, p.d_status);
            tc::tc_fence_after();
            for (int j = 0; j < pt.n; ++j, ++n) {
                const uint32_t s = n % PO_STAGES;
                tc::mbar_wait(&sm->full[s], (n / PO_STAGES) & 1, abort_flag, p.d_status);
                tc::tc_fence_after();
                if (elected) {
                    const uint64_t dA = tc::smem_desc_advance(d0, s * PO_STAGE_BYTES);
                    const uint64_t dB = tc::smem_desc_advance(dA, 2 * PO_SLAB);
#pragma unroll
                    for (int kk = 0; kk < PO_BK / 16; ++kk)
                        tc::pair_mma(acc, tc::smem_desc_advance(dA, kk * 2048), tc::smem_desc_advance(dB, kk * 2048),
                                     idesc, (j | kk) != 0);
                    tc::pair_commit(&sm->empty[s]);
                    if (j == pt.n - 1) tc::pair_commit(&sm->acc_full[buf]);
                }
                __syncwarp();
            }
            pos += pt.n;
        }
    } else if (warp == 2) {
        // ------------------------------------------------------------------ gathered rows -> products
        const bool elected = tc::elect_one();
        const uint32_t nsteps = (uint32_t)(run_b - run_a);
        for (uint32_t n = 0; n < nsteps; ++n) {
            const uint32_t s = n % PO_STAGES;
            tc::mbar_wait(&sm->gathered[s], (n / PO_STAGES) & 1, abort_flag, p.d_status);
            tc::fence_proxy_async_smem();
            if (elected) {
                if (rank == 0) tc::mbar_arrive(&sm->full[s]);
                else tc::remote_arrive(tc::leader_addr(&sm->full[s]));
            }
            __syncwarp();
        }
    } else if (warp == 3) {
        // ------------------------------------------------------------------ lists, PO_LIST steps ahead
        // (by bulk copies: ordinary loads return behind the gather warps' copies in flight, however far
        // ahead they are issued, and hold the pipeline at a fraction of its depth: 150 us)
        const bool elected = tc::elect_one();
        uint32_t n = 0;
        for (int64_t pos = run_a; pos < run_b;) {
            const Part pt = part_at(pos);
            for (int j = 0; j < pt.n; ++j, ++n) {
                const uint32_t q = n % PO_LIST;
                tc::mbar_wait(&sm->list_free[q], ((n / PO_LIST) & 1) ^ 1, abort_flag, p.d_status);
                if (elected) {
                    const int64_t first = (int64_t)pt.e * p.cap + (int64_t)(pt.k0 + j) * PO_BK;
                    const uint32_t bytes = PO_BK * 4 + ((first & 3) ? 16 : 0);
                    tc::mbar_arrive_expect_tx(&sm->list_full[q], bytes);
                    tc::bulk_load(sm->list[q], p.perm + (first & ~(int64_t)3), bytes, &sm->list_full[q]);
                }
                __syncwarp();
            }
            pos += pt.n;
        }
    } else if (warp >= PO_GATHER_WARP) {
        // ------------------------------------------------------------------ row gather (both CTAs)
        // thread -> 16-byte chunk `ch` of the 256 bytes of rows r0, r0 + 16, r0 + 32, r0 + 48, both operands
        const int gt = tid - 32 * PO_GATHER_WARP, ch = gt & 15, r0 = gt >> 4;
        uint32_t n = 0;
        for (int64_t pos = run_a; pos < run_b;) {
            const Part pt = part_at(pos);
            const int sc = pt.s0 + (int)rank * 128 + ch * 8, fc = pt.f0 + (int)rank * 128 + ch * 8;
            const bool s_in = sc < p.S, f_in = fc < p.F;
            const __nv_bfloat16 *g0 = p.g + sc, *u0 = p.u + fc;
            const int shift = (int)(((int64_t)pt.e * p.cap) & 3);
            for (int j = 0; j < pt.n; ++j, ++n) {
                const uint32_t s = n % PO_STAGES, q = n % PO_LIST;
                tc::mbar_wait(&sm->list_full[q], (n / PO_LIST) & 1, abort_flag, p.d_status);
                int ent[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = r0 + 16 * i;
                    ent[i] = (pt.k0 + j) * PO_BK + r < pt.cnt ? sm->list[q][shift + r] : -1;
                    if (p.check && (ent[i] < -1 || ent[i] >= p.cap * p.k)) {
                        atomicCAS(p.d_status, 0, SWIMBA_ERR_DEVICE_BOUNDS);
                        ent[i] = -1;
                    }
                }
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&sm->list_free[q]);
                tc::mbar_wait(&sm->empty[s], ((n / PO_STAGES) & 1) ^ 1, abort_flag, p.d_status);
                const uint32_t base = tc::smem_u32(smem + s * PO_STAGE_BYTES) + (ch >> 3) * PO_SLAB;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint32_t off = tc::sw128_offset(r0 + 16 * i, ch & 7);
                    const bool gi = ent[i] >= 0 && s_in, ui = ent[i] >= 0 && f_in;
                    const int tok = p.k == 2 ? ent[i] >> 1 : ent[i] / p.k;
                    tc::cp_async16(base + off, gi ? g0 + (int64_t)ent[i] * p.S : p.g, gi ? 16u : 0u);
                    tc::cp_async16(base + 2 * PO_SLAB + off, ui ? u0 + (int64_t)tok * p.F : p.u, ui ? 16u : 0u);
                }
                tc::cp_async_arrive(&sm->gathered[s]);
            }
            pos += pt.n;
        }
        tc::cp_async_commit();
        tc::cp_async_wait<0>();
    } else if (warp >= PO_EPI_WARP) {
        // ------------------------------------------------------------------ additions: thread = row s
        const int q = warp - PO_EPI_WARP;
        uint8_t *srow = smem + PO_OUT + (uint32_t)(q * 32 + lane) * PO_ROW;
        uint32_t it = 0;
        for (int64_t pos = run_a; pos < run_b; ++it) {
            const Part pt = part_at(pos);
            const uint32_t buf = it & 1;
            const int row = pt.s0 + (int)rank * 128 + q * 32 + lane;
            float *dst = p.dW + ((int64_t)pt.e * p.S + row) * p.F + pt.f0;
            const int ncols = min(PO_BN, p.F - pt.f0);
            tc::mbar_wait(&sm->acc_full[buf], (it >> 1) & 1, abort_flag, p.d_status);
            tc::tc_fence_after();
            const uint32_t acc = tmem + buf * PO_BN + ((uint32_t)(q * 32) << 16);
#pragma unroll 1
            for (int c = 0; c < ncols; c += PO_COLS) {
                tc::bulk_wait_read_all();
                __syncwarp();
#pragma unroll
                for (int hf = 0; hf < PO_COLS / 32; ++hf) {
                    uint32_t v[32];
                    tc::tmem_ld32(acc + c + 32 * hf, v);
                    tc::tmem_ld_wait();
                    uint4 *d4 = reinterpret_cast<uint4 *>(srow + hf * 128);
#pragma unroll
                    for (int i = 0; i < 8; ++i) d4[i] = make_uint4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                }
                tc::fence_proxy_async_smem();
                if (row < p.S) tc::bulk_reduce_add_f32(dst + c, srow, (uint32_t)min(PO_COLS, ncols - c) * 4);
                tc::bulk_commit_group();
            }
            tc::tc_fence_before();
            __syncwarp();
            if (lane == 0) tc::remote_arrive(tc::leader_addr(&sm->acc_empty[buf]));
            pos += pt.n;
        }
        tc::bulk_wait_read_all();
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::cluster_sync();
    tc::tc_fence_after();
    if (warp == 1) tc::pair_tmem_dealloc(tmem);
}

int launch_pair_outer(LaunchCtx &ctx, const void *g, const void *u, const int *perm, const int *counts, int64_t T,
                      int F, int S, int E, int k, int sm_count, float *dW)
{
    OuterArgs p;
    p.g = (const __nv_bfloat16 *)g; p.u = (const __nv_bfloat16 *)u;
    p.perm = perm; p.counts = counts; p.cap = T; p.dW = dW;
    p.E = E; p.F = F; p.S = S; p.k = k;
    p.check = ctx.check_indices ? 1 : 0;
    p.d_status = ctx.d_status;
    const size_t smem = PO_SMALL + sizeof(OuterSmall);
    if (!ensure_dynamic_smem((const void *)pair_outer_kernel, smem)) return SWIMBA_ERR_CUDA;
    // no more pairs than steps
    int64_t pairs = (ceil_div64(T * k, PO_BK) + E) * ceil_div(S, PO_BM) * ceil_div(F, PO_BN);
    if (pairs > sm_count / 2) pairs = sm_count / 2;
    ctx.begin(STAGE_DW_EXPERT);
    launch_kernel_cluster(pair_outer_kernel, dim3((unsigned)(2 * pairs)), dim3(PO_THREADS), smem, ctx.stream, true, 2u, p);
    ctx.end();
    return cudaGetLastError() == cudaSuccess ? SWIMBA_OK : SWIMBA_ERR_CUDA;
}

}  // namespace swimba
