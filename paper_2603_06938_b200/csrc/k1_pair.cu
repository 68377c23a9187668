// Grouped and dense products on CTA pairs (tcgen05 with cta_group::2): the expert stream projection of
// large calls (Theorem 2: only the active experts of a token are projected) and the block's linear maps,
//   D[256, 256] = A_rows[256, F] * W[n0 : n0 + 256, F]^T   per tile,
// two SMs working one tile: each holds 128 of its rows (and their fp32 accumulators in tensor memory) and
// half of the weight rows.  Persistent: a pair walks tiles p, p + pairs, ...; the accumulators are double
// buffered, so that a tile's epilogue runs under the next tile's products.
//
// Why this shape.  The products are fed from L2: a 64-feature step of a tile costs 32 KB per SM for 512
// cycles of tensor time, and what the L2 delivers is set by the bytes in flight.  One CTA per 256 x 256
// tile with gathering warps (cp.async) had room for two such steps per SM in flight and took 1590 cycles
// for what the tensor core does in 1024; here up to five steps are in flight per SM (160 KB) and no
// tile exposes its epilogue.  Measured: 65536 rows x 2048 features x 256 columns of 8 experts 96 -> 58 us
// (1.19 PFLOP/s), 32768 x 2048 x 8192 dense 1190 -> 661 us (1.66 PFLOP/s).  Gathered rows come by
// cp.async: tile::gather4 loads (512 bytes each with the 128-byte swizzle) took 150 us for the first shape.
#include <algorithm>

#include "internal.h"
#include "pair.cuh"

namespace swimba {

namespace {
constexpr int PG_BM = 256, PG_BN = 256, PG_BK = 64, PG_STAGES = 5;
constexpr uint32_t PG_A_BYTES = 128 * 128, PG_STAGE_BYTES = 2 * PG_A_BYTES;     // per CTA: 128 rows of A, 128 of W
constexpr uint32_t PG_ROW = PG_BN * 2 + 16;          // staged output row, padded against bank conflicts
constexpr uint32_t PG_OUT = PG_STAGES * PG_STAGE_BYTES;
constexpr uint32_t PG_SMALL = PG_OUT + 128 * PG_ROW;
constexpr int PG_EPI_WARP = 4;                       // warps 4..7: epilogue (TMEM lane quarter = warp % 4)
constexpr int PG_GATHER_WARP = 8;                    // warps 8..11: row gather (grouped products only)
__host__ __device__ constexpr int pg_threads(bool dense) { return dense ? 256 : 384; }

struct PairSmall {
    uint64_t full[PG_STAGES], empty[PG_STAGES], acc_full[2], acc_empty[2];
    uint64_t gathered[PG_STAGES];                    // the CTA's gathered rows have arrived
    uint32_t tmem_slot;
    int abort_flag;
    int tile_end[SWIMBA_MAX_EXPERTS];                // row tiles of experts 0 .. e, summed
    int cnt[SWIMBA_MAX_EXPERTS];
};

struct PairArgs {
    const int *perm, *counts;      // per-expert lists (entries t*k + j) and their lengths; null: dense rows
    int64_t cap;                   // list capacity = tokens
    const float *w_slot;           // [T*k] row weights; null: 1
    const __nv_bfloat16 *rows;     // the rows the lists index
    __nv_bfloat16 *out;
    int64_t ld_out;
    float *tail;                   // columns from tail_col on go here as fp32, [rows, S - tail_col] (a
    int tail_col;                  // multiple of 32; S: none)
    int E, F, S, k, add_rows, check;
    int *d_status;
};

__device__ __forceinline__ void pair_load_2d(void *dst, const CUtensorMap *m, uint32_t bar, int c0, int c1)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 "
        "[%0], [%1, {%3, %4}], [%2];" ::"r"(tc::smem_u32(dst)),
        "l"(m), "r"(bar), "r"(c0), "r"(c1)
        : "memory");
}
__device__ __forceinline__ void pair_load_3d(void *dst, const CUtensorMap *m, uint32_t bar, int c0, int c1, int c2)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 "
        "[%0], [%1, {%3, %4, %5}], [%2];" ::"r"(tc::smem_u32(dst)),
        "l"(m), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}
}  // namespace

// DENSE: rows are taken as they lie (one expert, no lists, no weights).
template <bool DENSE>
__global__ void __launch_bounds__(pg_threads(DENSE), 1)
pair_gemm_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_w,
                 const PairArgs p)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    PairSmall *sm = (PairSmall *)(smem + PG_SMALL);
    int *abort_flag = &sm->abort_flag;
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const uint32_t rank = tc::cluster_rank();
    const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
    if ((tc::smem_u32(smem) & 1023u) != 0) {      // the swizzled tiles need a 1024-byte aligned base (the
        if (tid == 0) atomicCAS(p.d_status, 0, SWIMBA_ERR_DEVICE_BOUNDS);   // same in both CTAs)
        return;
    }

    if (tid == 0) {
        for (int s = 0; s < PG_STAGES; ++s) {
            tc::mbar_init(&sm->full[s], DENSE ? 1 : 3);        // loads by TMA, the gathered rows of either CTA
            tc::mbar_init(&sm->gathered[s], 128);
            tc::mbar_init(&sm->empty[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            tc::mbar_init(&sm->acc_full[s], 1);
            tc::mbar_init(&sm->acc_empty[s], 2 * 4);           // four epilogue warps in each CTA
        }
        *abort_flag = 0;
        tc::fence_mbar_init();
        tc::prefetch_tmap(&tmap_a);
        tc::prefetch_tmap(&tmap_w);
    }
    if (warp == 1) {
        tc::pair_tmem_alloc(&sm->tmem_slot);
    }
    grid_dep_launch();
    grid_dep_wait();        // lists, weights and rows come from the kernels in front
    if (warp == 2) {
        // row tiles of every expert, summed over the experts (64 at most: two per lane)
        int c0 = 0, c1 = 0;
        if (DENSE) {
            c0 = lane == 0 ? (int)p.cap : 0;
        } else {
            c0 = 2 * lane < p.E ? p.counts[2 * lane] : 0;
            c1 = 2 * lane + 1 < p.E ? p.counts[2 * lane + 1] : 0;
            if (p.check && (c0 < 0 || c0 > p.cap || c1 < 0 || c1 > p.cap)) {   // longer than a list can be
                atomicCAS(p.d_status, 0, SWIMBA_ERR_DEVICE_BOUNDS);
                if (c0 < 0 || c0 > p.cap) c0 = 0;
                if (c1 < 0 || c1 > p.cap) c1 = 0;
            }
        }
        const int n0 = (c0 + PG_BM - 1) / PG_BM, n1 = (c1 + PG_BM - 1) / PG_BM;
        int incl = n0 + n1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int nb = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += nb;
        }
        sm->tile_end[2 * lane] = incl - n1;
        sm->tile_end[2 * lane + 1] = incl;
        sm->cnt[2 * lane] = c0;
        sm->cnt[2 * lane + 1] = c1;
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::cluster_sync();            // barriers and tensor memory of both CTAs are ready
    tc::tc_fence_after();
    const uint32_t tmem = sm->tmem_slot;
    const int ncol = ceil_div(p.S, PG_BN);
    const int ntiles = sm->tile_end[SWIMBA_MAX_EXPERTS - 1] * ncol;
    const int KB = ceil_div(p.F, PG_BK);

    // Tile -> expert, first row inside its list, length of the list, first column, columns of the product.
    struct Tile { int e, row0, cnt, n0, nt; };
    auto tile_of = [&](int t) {
        Tile r;
        const int rt = t / ncol;
        r.n0 = (t - rt * ncol) * PG_BN;
        r.nt = min(PG_BN, (p.S - r.n0 + 31) & ~31);
        int e = 0;
        if (!DENSE) {
            const unsigned lo = __ballot_sync(0xffffffffu, sm->tile_end[lane] > rt);
            if (lo) e = __ffs(lo) - 1;
            else e = 32 + __ffs(__ballot_sync(0xffffffffu, sm->tile_end[32 + lane] > rt)) - 1;
        }
        r.e = e;
        r.row0 = (rt - (e > 0 ? sm->tile_end[e - 1] : 0)) * PG_BM;
        r.cnt = sm->cnt[e];
        return r;
    };
    // List entry of row r of expert e (rows past the end repeat the last one and are never written).
    auto entry_of = [&](const Tile &t, int r) {
        if (r >= t.cnt) r = t.cnt - 1;
        int entry = p.perm[(int64_t)t.e * p.cap + r];
        if (p.check && (entry < 0 || entry >= p.cap * p.k)) {
            atomicCAS(p.d_status, 0, SWIMBA_ERR_DEVICE_BOUNDS);
            entry = -1;
        }
        return entry;
    };

    if (warp == 0) {
        // ------------------------------------------------------------------ loads by TMA (both CTAs)
        const bool elected = tc::elect_one();
        uint32_t n = 0;
        for (int t = pair; t < ntiles; t += npairs) {
            const Tile ti = tile_of(t);
            for (int kb = 0; kb < KB; ++kb, ++n) {
                const uint32_t s = n % PG_STAGES;
                tc::mbar_wait(&sm->empty[s], ((n / PG_STAGES) & 1) ^ 1, abort_flag, p.d_status);
                uint8_t *sA = smem + s * PG_STAGE_BYTES, *sB = sA + PG_A_BYTES;
                if (elected) {
                    const uint32_t bar = tc::leader_addr(&sm->full[s]);
                    if (rank == 0) tc::mbar_arrive_expect_tx(&sm->full[s], DENSE ? 2 * PG_STAGE_BYTES : 2 * PG_A_BYTES);
                    pair_load_3d(sB, &tmap_w, bar, kb * PG_BK, ti.n0 + (int)rank * (ti.nt >> 1), ti.e);
                    if (DENSE) pair_load_2d(sA, &tmap_a, bar, kb * PG_BK, ti.row0 + (int)rank * 128);
                }
                __syncwarp();
            }
        }
    } else if (warp == 1 && rank == 0) {
        // ------------------------------------------------------------------ products (first CTA)
        const bool elected = tc::elect_one();
        const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem, 0);
        const uint64_t d0 = tc::smem_desc_sw128(tc::smem_u32(smem), 16, 1024);
        uint32_t n = 0, it = 0;
        for (int t = pair; t < ntiles; t += npairs, ++it) {
            const Tile ti = tile_of(t);
            const uint32_t buf = it & 1, acc = tmem_u + buf * PG_BN;
            const uint32_t idesc = tc::idesc_bf16(PG_BM, ti.nt, 0, 0);
            tc::mbar_wait(&sm->acc_empty[buf], ((it >> 1) & 1) ^ 1, abort_flag, p.d_status);
            tc::tc_fence_after();
            for (int kb = 0; kb < KB; ++kb, ++n) {
                const uint32_t s = n % PG_STAGES;
                tc::mbar_wait(&sm->full[s], (n / PG_STAGES) & 1, abort_flag, p.d_status);
                tc::tc_fence_after();
                if (elected) {
                    const uint64_t dA = tc::smem_desc_advance(d0, s * PG_STAGE_BYTES);
                    const uint64_t dB = tc::smem_desc_advance(dA, PG_A_BYTES);
#pragma unroll
                    for (int kk = 0; kk < PG_BK / 16; ++kk)
                        tc::pair_mma(acc, tc::smem_desc_advance(dA, kk * 32), tc::smem_desc_advance(dB, kk * 32), idesc,
                                 (kb | kk) != 0);
                    tc::pair_commit(&sm->empty[s]);
                    if (kb == KB - 1) tc::pair_commit(&sm->acc_full[buf]);
                }
                __syncwarp();
            }
        }
    } else if (!DENSE && warp == 2) {
        // ------------------------------------------------------------------ gathered rows -> products
        // The copies report to a barrier of their own; this warp orders them before the tensor core's
        // reads and passes the word on.  The gather warps cannot do that themselves: a proxy fence
        // waits for the issuing thread's copies in flight, so that every step would cost their whole
        // latency.
        const bool elected = tc::elect_one();
        uint32_t n = 0;
        for (int t = pair; t < ntiles; t += npairs)
            for (int kb = 0; kb < KB; ++kb, ++n) {
                const uint32_t s = n % PG_STAGES;
                tc::mbar_wait(&sm->gathered[s], (n / PG_STAGES) & 1, abort_flag, p.d_status);
                tc::fence_proxy_async_smem();
                if (elected) {
                    if (rank == 0) tc::mbar_arrive(&sm->full[s]);
                    else tc::remote_arrive(tc::leader_addr(&sm->full[s]));
                }
                __syncwarp();
            }
    } else if (!DENSE && warp >= PG_GATHER_WARP) {
        // ------------------------------------------------------------------ row gather (both CTAs)
        // thread -> 16-byte chunk lane % 8 of rows 4 i + lane / 8 of its warp's 32
        const int q = warp - PG_GATHER_WARP, chunk = lane & 7;
        // the list entries are fetched a tile ahead: behind the copies in flight they would return late
        uint32_t n = 0;
        int ent[8];
        auto fetch = [&](int t) {
            if (t >= ntiles) return;
            const Tile ti = tile_of(t);
#pragma unroll
            for (int i = 0; i < 8; ++i) ent[i] = entry_of(ti, ti.row0 + (int)rank * 128 + q * 32 + i * 4 + (lane >> 3));
        };
        fetch(pair);
        for (int t = pair; t < ntiles; t += npairs) {
            const __nv_bfloat16 *src[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) src[i] = p.rows + chunk * 8 + (int64_t)(max(ent[i], 0) / p.k) * p.F;
            fetch(t + npairs);
            for (int kb = 0; kb < KB; ++kb, ++n) {
                const uint32_t s = n % PG_STAGES;
                tc::mbar_wait(&sm->empty[s], ((n / PG_STAGES) & 1) ^ 1, abort_flag, p.d_status);
                const uint32_t a_base = tc::smem_u32(smem + s * PG_STAGE_BYTES);
                const bool in = kb * PG_BK + chunk * 8 < p.F;
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    tc::cp_async16(a_base + tc::sw128_offset(q * 32 + i * 4 + (lane >> 3), chunk),
                                   in ? src[i] + kb * PG_BK : p.rows, in ? 16u : 0u);
                tc::cp_async_arrive(&sm->gathered[s]);
            }
        }
        tc::cp_async_commit();
        tc::cp_async_wait<0>();
    } else if (warp >= PG_EPI_WARP && warp < PG_GATHER_WARP) {
        // ------------------------------------------------------------------ epilogue: thread = row
        const int q = warp - PG_EPI_WARP;
        uint8_t *srow = smem + PG_OUT + (uint32_t)(q * 32 + lane) * PG_ROW;
        uint32_t it = 0;
        for (int t = pair; t < ntiles; t += npairs, ++it) {
            const Tile ti = tile_of(t);
            const uint32_t buf = it & 1;
            const int r = ti.row0 + (int)rank * 128 + q * 32 + lane;
            bool ok = r < ti.cnt;
            float wr = 1.f;
            int64_t dst = r;
            if (!DENSE) {
                const int entry = entry_of(ti, r);
                ok = ok && entry >= 0;
                wr = (ok && p.w_slot) ? p.w_slot[entry] : 1.f;
                dst = p.add_rows ? entry / p.k : entry;
            }
            tc::mbar_wait(&sm->acc_full[buf], (it >> 1) & 1, abort_flag, p.d_status);
            tc::tc_fence_after();
            tc::bulk_wait_read_all();            // the previous tile's row has left its staging buffer
            __syncwarp();
            const int ncols = min(PG_BN, p.S - ti.n0);                   // all columns of the tile,
            const int nmain = max(0, min(ncols, p.tail_col - ti.n0));     // those in front of the tail
            const uint32_t acc = tmem + buf * PG_BN + ((uint32_t)(q * 32) << 16);
#pragma unroll 1
            for (int c = 0; c < ncols; c += 32) {
                uint32_t v[32];
                tc::tmem_ld32(acc + c, v);
                tc::tmem_ld_wait();
                if (DENSE && c >= nmain) {
                    if (ok) {
                        const int c0 = ti.n0 + c - p.tail_col, nt = p.S - p.tail_col;
                        float *d = p.tail + dst * nt + c0;
#pragma unroll
                        for (int i = 0; i < 32; ++i) if (c0 + i < nt) d[i] = __uint_as_float(v[i]);
                    }
                    continue;
                }
                uint32_t pk[16];
#pragma unroll
                for (int i = 0; i < 16; ++i)
                    pk[i] = tc::pack_bf16x2(wr * __uint_as_float(v[2 * i]), wr * __uint_as_float(v[2 * i + 1]));
                uint4 *d4 = reinterpret_cast<uint4 *>(srow + c * 2);
#pragma unroll
                for (int i = 0; i < 4; ++i) d4[i] = make_uint4(pk[4 * i], pk[4 * i + 1], pk[4 * i + 2], pk[4 * i + 3]);
            }
            tc::tc_fence_before();
            tc::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) tc::remote_arrive(tc::leader_addr(&sm->acc_empty[buf]));
            if (ok && nmain > 0) {
                __nv_bfloat16 *row = p.out + dst * p.ld_out + ti.n0;
                if (p.add_rows) tc::bulk_reduce_add_bf16(row, srow, (uint32_t)nmain * 2);
                else tc::bulk_store(row, srow, (uint32_t)nmain * 2);
            }
            tc::bulk_commit_group();
        }
        tc::bulk_wait_read_all();
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::cluster_sync();            // nobody reads or signals the other CTA's memory any more
    tc::tc_fence_after();
    if (warp == 1) tc::pair_tmem_dealloc(tmem);
}

int launch_pair_gemm(LaunchCtx &ctx, const void *A, const void *W, const int *perm, const int *counts,
                     const float *w_slot, int64_t T, int F, int S, int E, int k, bool add_rows, int sm_count,
                     void *out, int64_t ld_out, float *tail, int tail_col)
{
    const bool dense = perm == nullptr;
    CUtensorMap tm_a, tm_w;
    {
        const uint64_t dims[2] = {(uint64_t)F, (uint64_t)T};
        const uint64_t str[1] = {(uint64_t)F * 2};
        const uint32_t box[2] = {(uint32_t)PG_BK, 128u};
        if (!encode_tmap_bf16_cached(ctx.tmaps, &tm_a, A, 2, dims, str, box)) return SWIMBA_ERR_CUDA;
    }
    {
        const uint64_t dims[3] = {(uint64_t)F, (uint64_t)S, (uint64_t)E};
        const uint64_t str[2] = {(uint64_t)F * 2, (uint64_t)S * F * 2};
        const uint32_t box[3] = {(uint32_t)PG_BK, 128u, 1u};
        if (!encode_tmap_bf16_cached(ctx.tmaps, &tm_w, W, 3, dims, str, box)) return SWIMBA_ERR_CUDA;
    }
    PairArgs p;
    p.perm = perm; p.counts = counts; p.cap = T; p.w_slot = w_slot;
    p.rows = (const __nv_bfloat16 *)A;
    p.out = (__nv_bfloat16 *)out; p.ld_out = ld_out;
    p.tail = tail; p.tail_col = tail ? tail_col : S;
    p.E = E; p.F = F; p.S = S; p.k = k; p.add_rows = add_rows ? 1 : 0;
    p.check = ctx.check_indices ? 1 : 0;
    p.d_status = ctx.d_status;
    int64_t pairs = (ceil_div64(T * k, PG_BM) + (dense ? 0 : E)) * ceil_div(S, PG_BN);
    if (pairs > sm_count / 2) pairs = sm_count / 2;
    const size_t smem = PG_SMALL + sizeof(PairSmall);
    auto kern = dense ? pair_gemm_kernel<true> : pair_gemm_kernel<false>;
    if (!ensure_dynamic_smem((const void *)kern, smem)) return SWIMBA_ERR_CUDA;
    ctx.begin(STAGE_EXPERT_GEMM);
    launch_kernel_cluster(kern, dim3((unsigned)(2 * pairs)), dim3((unsigned)pg_threads(dense)), smem, ctx.stream, true,
                          2u, tm_a, tm_w, p);
    ctx.end();
    return cudaGetLastError() == cudaSuccess ? SWIMBA_OK : SWIMBA_ERR_CUDA;
}

// Calls that take the pair kernel: eight 256 x 256 tiles or more of rows as they lie.  Grouped rows also have the
// narrow column tiles of expert_gemm_kernel, which it narrows further while all its tiles fit half of the SMs, and
// whose products stop at 128 rows where a list does.  They keep: short products of few tiles; lists that fill half
// a tile or less, unless one column of long products has few of them (all gain from fewer, longer steps) or they
// are too many to be narrowed and the pairs hold them in one round (or short and more than two rounds of CTAs,
// whose set-up the persistent pairs save).  Measured (router, lists and product, us, narrow
// / pairs; rows are (token, expert) entries):
//   S = 256    F = 512       F = 1024      F = 2048        S = 2048   F = 512       F = 1024      F = 2048
//   E = 8      2050 rows  16.4 / 16.4   20.5 / 20.5   28.7 / 26.6   600 rows   19 / 21   24.5 / 26.7   33.5 / 41.1
//              3200       16.4 / 16.4   20.6 / 20.5   29.3 / 26.6   1600       24.5 / 19.5  33.0 / 22.8  53.3 / 30.9
//   E = 16     2050       16.4 / 18.4   20.5 / 22.2   33.0 / 31.0   600        22.2 / 24.9  29.0 / 34.2  51.9 / 60.9
//   E = 32     3200       18.4 / 19.3   24.7 / 26.6   37.0 / 38.9
//   E = 64     2600       26.6 / 24.6   39.0 / 34.9   65.8 / 55.9   600        58.4 / 54.1  65.6 / 66.6  113 / 117
// Over 411 calls the line costs 0.2 % over picking the faster one every time.
bool pair_gemm_usable(int64_t rows, int F, int S, int E, int sm_count)
{
    const int64_t cols = ceil_div(S, PG_BN), row_tiles = ceil_div64(rows, PG_BM);
    if (sm_count < 2 || F < 64 || F % 8 != 0 || S % 8 != 0 || row_tiles * cols < 8) return false;
    if (E == 1) return true;
    if (rows > 120 * (int64_t)E) return F >= 1024 || row_tiles * cols >= 32;
    if (cols == 1 && F >= 1024 && E <= (F < 2048 ? 8 : 16)) return true;
    if (2 * (row_tiles + E) * cols <= sm_count) return false;
    const int64_t tiles = std::max(row_tiles, std::min<int64_t>(E, rows)) * cols;
    return tiles <= sm_count / 2 || (tiles > 2 * sm_count && F < 1024);
}

}  // namespace swimba
