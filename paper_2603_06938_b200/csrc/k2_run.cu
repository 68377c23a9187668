// The chunked SSD evaluation of k2_ssd.cu for CTAs that walk many tiles in a row (same division of the work, same
// products; names of the products and of the factors as there).  What the tile loop there waits for is, as far as counters
// and bytes tell, shared memory's data pipe: of a tile's 5500 cycles 4300 are counted as wavefronts of the CUDA cores and of
// the tensor cores' operands, TMA's 128 KB are another 1000.  So here
//   - w.X goes from the x slab to the tensor memory by ldmatrix and is MMA 4's A operand (no scaled copy in shared
//     memory), Ctilde is copied to tensor memory once and is the A operand of MMA 1 and MMA 3;
//   - G is read once for both heads, masked in place and in the fragment layout (8 weights a head and thread);
//   - exp(l_i - l_s) = 2^(l_i - ref) 2^(ref - l_s) with one reference a tile (ssd_scalars.cuh): one product an entry, no
//     scaling of Ctilde Hprev^T (the bf16 state copy decays to the reference), the row factor in the epilogue;
//   - w.X of the next tile is made while MMA 2 runs, y replaces x in place, x is three tiles ahead.
// A tile takes 4350 cycles: 3300 counted as wavefronts (2050 of the CUDA cores, 1240 operands), 1000 for TMA by its bytes, so that
// the pipe is the bound again.  A CTA takes 2000 to 3500 more to start and to drain: runs of fewer than RUN_TILES tiles stay
// with the other kernel.
#include "ssd_tiles.cuh"

namespace swimba {

namespace {
constexpr int NCW = 16;                 // compute warps
constexpr int WARP_TMA = NCW, WARP_MMA = NCW + 1;
constexpr int RUN_THREADS = 32 * (NCW + 2);

// shared memory map (bytes from the 1024-aligned base): Btilde of two tiles, Ctilde of one (two slabs each), x of
// three tiles, which y replaces in place, and the bf16 states of both heads.  A copy from L2 takes 2000 cycles
// here, from HBM up to 4000: with one Btilde tile less, or x two tiles deep, they were waited for.
constexpr int B_SLOTS = 2, X_SLOTS = 3;
constexpr int Y_BARS = 3;               // (the store of a tile is waited for while two more may be staged)
constexpr uint32_t SM_B = 0;
constexpr uint32_t SM_C = B_SLOTS * 2 * SLAB;
constexpr uint32_t SM_X = SM_C + 2 * SLAB;
constexpr uint32_t SM_H = SM_X + X_SLOTS * NHD * SLAB;
constexpr uint32_t SM_SMALL = SM_H + 2 * SLAB;

// TMEM columns: G, which the masked tiles of both heads overwrite in place; Y; dH; w.X; Ctilde.  (w.X of every
// second leading tile takes Y's place, which those do not use.)
constexpr uint32_t TM_G = 0, TM_Y = 128, TM_DH = 256, TM_XP = 384, TM_C = 448, TM_COLS = 512;

struct __align__(8) RunBars {
    uint64_t b_full[B_SLOTS], b_empty[B_SLOTS], c_full, c_empty;
    uint64_t x_full[X_SLOTS], xp_full[2], xp_free[2], y_staged[Y_BARS];
    uint64_t rec_free, m_full, g_full, yd_full, dh_full;
};

// What this kernel keeps of a tile's record: the column weights, the block ends, what follows from them, and the row
// factors.  Every warp takes what it needs into registers as soon as the record is there, a tile ahead of its
// use: room for one.
struct __align__(16) TileRec {
    float cb[ST], ends[4];
    TileAux aux;
    float row[ST];
};

struct __align__(16) RunSmall {
    TileRec sc[NHD];         // copied in by the TMA warp
    RunBars bars;
    // split launch: per warp, log2 decay over all leading tiles, and over those worked so far: summed in the same order, so
    // that the difference is 0 at the last one (a remainder counted down keeps every subtraction's rounding)
    float run_total[NCW], run_done[NCW];
    uint32_t tmem_slot;
    int abort_flag;
};

}  // namespace

__device__ __forceinline__ uint64_t f32x2_bits(uint32_t a, uint32_t b)
{
    return tc::f32x2(__uint_as_float(a), __uint_as_float(b));
}

// Weights of a thread's eight columns (or tokens) of a 32-wide block.
struct BlockWeights { uint64_t v[4]; };
__device__ __forceinline__ void load_weights(BlockWeights &w, const float *s_cb, int lane)
{
#pragma unroll
    for (int r = 0; r < 4; ++r) w.v[r] = *reinterpret_cast<const uint64_t *>(s_cb + 8 * r + 2 * (lane & 3));
}

// Their decay to the end of the block, where the record has Delta alone and l in place of row factors (block_fast).
__device__ __forceinline__ void decay_weights(BlockWeights &w, const TileRec *rec, int block, int lane)
{
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const float2 l = *reinterpret_cast<const float2 *>(&rec->row[32 * block + 8 * r + 2 * (lane & 3)]);
        w.v[r] = tc::f32x2_mul(w.v[r], tc::f32x2(tc::ex2_approx(rec->ends[block] - l.x), tc::ex2_approx(rec->ends[block] - l.y)));
    }
}

// w . X of one warp, from the X slab to the A operand of MMA 4 in tensor memory: lanes p0 .. p0+31 (channels of
// the head), tokens s0 .. s0+31 (16 columns, two to a column).  wx: weights of tokens s0 + 8 c + 2 (t % 4) and
// the one behind; x' = w x with the weight as a two-term bf16 sum (rounded once).
__device__ __forceinline__ void scale_to_tmem(const uint8_t *s_x, const BlockWeights &wx, int p0, int s0, int lane,
                                              uint32_t taddr)
{
    uint32_t a[4][4];              // [8 tokens][8 channels], the fragment layout of ldmatrix
    const uint32_t src = tc::smem_u32(s_x) + tc::sw128_offset(s0 + (lane & 7), (p0 >> 3) + (lane >> 3));
#pragma unroll
    for (int c = 0; c < 4; ++c) tc::ldmatrix_x4_trans(src + c * 1024, a[c][0], a[c][1], a[c][2], a[c][3]);
    const uint64_t minus = tc::f32x2(-1.f, -1.f);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const uint64_t w = wx.v[c];
        const uint32_t hi_u = tc::f32x2_bf16(w);
        const uint32_t lo_u = tc::f32x2_bf16(tc::f32x2_fma(f32x2_bits(hi_u << 16, hi_u & 0xffff0000u), minus, w));
        const __nv_bfloat162 w_hi2 = *reinterpret_cast<const __nv_bfloat162 *>(&hi_u);
        const __nv_bfloat162 w_lo2 = *reinterpret_cast<const __nv_bfloat162 *>(&lo_u);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const __nv_bfloat162 xv = *reinterpret_cast<const __nv_bfloat162 *>(&a[c][m]);
            const __nv_bfloat162 pr = __hfma2(w_hi2, xv, __hmul2(w_lo2, xv));
            a[c][m] = *reinterpret_cast<const uint32_t *>(&pr);
        }
    }
    const uint32_t lo[8] = {a[0][0], a[0][1], a[1][0], a[1][1], a[2][0], a[2][1], a[3][0], a[3][1]};
    const uint32_t hi[8] = {a[0][2], a[0][3], a[1][2], a[1][3], a[2][2], a[2][3], a[3][2], a[3][3]};
    tc::tmem_st_16x128b_x4(taddr, lo);
    tc::tmem_st_16x128b_x4(taddr + (16u << 16), hi);
}

// Decay mask of a 32 x 32 block in place, M = G cb as bf16 pairs, in the fragment layout: this thread has rows t / 4 + 8 k
// and columns 8 r + 2 (t % 4) and the one behind, so that it needs 8 weights a head (a row per thread would
// need all 32, read as broadcasts: a fourth of the kernel's shared-memory wavefronts).  16 columns of G become 8
// of the first head's M and 8 of the second one's, which is what a K step of MMA 2 takes.  The row factor comes
// with the epilogue.
// Entries of rows k = 0, 1 (t / 4 + 8 k) and columns 16 c .. 16 c + 15 for one head: a K step's four registers.  DIAG: the
// 16 x 16 block on the diagonal; `keep` the bits that a row keeps of the pair in its own 8 x 8 block.
template <bool DIAG>
__device__ __forceinline__ void mask_step(uint32_t taddr, const uint32_t (&g)[16], const BlockWeights &w, int c, uint32_t keep)
{
    uint32_t o[4];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int e = 4 * (2 * c + r) + 2 * k;
            o[2 * r + k] = tc::f32x2_bf16(tc::f32x2_mul(f32x2_bits(g[e], g[e + 1]), w.v[2 * c + r]));
        }
    if (DIAG) {
        o[0] &= keep;
        o[2] = 0u;
        o[3] &= keep;
    }
    tc::tmem_st_16x128b_x2(taddr + 16 * c, o[0], o[1], o[2], o[3]);
}

template <bool DIAG>
__device__ __forceinline__ void mask_block(uint32_t taddr, const BlockWeights (&w)[2], uint32_t keep)
{
#pragma unroll
    for (int half = 0; half < 2; ++half) {                    // rows 0 .. 15, 16 .. 31
        const uint32_t ta = taddr + ((uint32_t)(16 * half) << 16);
        uint32_t g[16];
        tc::tmem_ld_16x256b_x4(ta, g);
        tc::tmem_ld_wait();
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            if (!DIAG) {
                mask_step<false>(ta + 8 * q, g, w[q], 0, 0u);
                mask_step<false>(ta + 8 * q, g, w[q], 1, 0u);
            } else if (half == 0) {
                mask_step<true>(ta + 8 * q, g, w[q], 0, keep);
                tc::tmem_st_16x128b_x2(ta + 8 * q + 16, 0u, 0u, 0u, 0u);
            } else {
                mask_step<false>(ta + 8 * q, g, w[q], 0, 0u);
                mask_step<true>(ta + 8 * q, g, w[q], 1, keep);
            }
        }
    }
}

// The same where this row block of a head decays by 2^-96 and more (block_fast; heads in `fast`, one bit each): that head's
// entries carry the row factor 2^lr, which lane t has for row t.  On the diagonal the weights are Delta and exponents
// are formed entry by entry, those kept all <= 0; rows and columns are the same tokens there.  4 x 8192 tokens of
// 64 heads, one of them like that: 235 us (200 without, 218 in the tile kernel); with l and Delta read from global memory where
// they are used 440.
__device__ __forceinline__ void mask_block_entries(uint32_t taddr, const BlockWeights (&w)[2], const float (&lr)[2], int fast,
                                                   bool diag, uint32_t keep, int lane)
{
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        const uint32_t ta = taddr + ((uint32_t)(16 * half) << 16);
        uint32_t g[16];
        tc::tmem_ld_16x256b_x4(ta, g);
        tc::tmem_ld_wait();
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const bool entries = diag && (fast >> q & 1);
            const float l = fast >> q & 1 ? lr[q] : 0.f;
            float row[2];                                    // l of rows k, their factor where the weights have one
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                row[k] = __shfl_sync(0xffffffffu, l, 16 * half + 8 * k + (lane >> 2));
                if (!entries) row[k] = tc::ex2_approx(row[k]);
            }
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                if (diag && c > half) {                      // (above the diagonal)
                    tc::tmem_st_16x128b_x2(ta + 8 * q + 16 * c, 0u, 0u, 0u, 0u);
                    continue;
                }
                uint32_t o[4];
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    float col[2] = {0.f, 0.f};
                    if (entries) {
#pragma unroll
                        for (int e = 0; e < 2; ++e) col[e] = __shfl_sync(0xffffffffu, l, 16 * c + 8 * r + 2 * (lane & 3) + e);
                    }
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        const uint64_t f = entries ? tc::f32x2(tc::ex2_approx(row[k] - col[0]), tc::ex2_approx(row[k] - col[1]))
                                                   : tc::f32x2(row[k], row[k]);
                        const int e = 4 * (2 * c + r) + 2 * k;
                        o[2 * r + k] = tc::f32x2_bf16(tc::f32x2_mul(f32x2_bits(g[e], g[e + 1]), tc::f32x2_mul(w[q].v[2 * c + r], f)));
                    }
                }
                if (diag && c == half) {                     // the 16 x 16 block on the diagonal
                    o[0] &= keep;
                    o[2] = 0u;
                    o[3] &= keep;
                }
                tc::tmem_st_16x128b_x2(ta + 8 * q + 16 * c, o[0], o[1], o[2], o[3]);
            }
        }
    }
}

template <bool SPLIT>
__global__ void __launch_bounds__(RUN_THREADS, 1)
ssd_run_kernel(const __grid_constant__ CUtensorMap tmap_b, const __grid_constant__ CUtensorMap tmap_c,
                 const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_y,
                 const SsdParams prm)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    RunSmall *sm = (RunSmall *)(smem + SM_SMALL);
    RunBars *bars = &sm->bars;
    int *abort_flag = &sm->abort_flag;
    int *d_status = prm.d_status;
    if ((tc::smem_u32(smem) & 1023u) != 0) {      // the swizzled tiles need a 1024-byte aligned base
        if (threadIdx.x == 0) atomicCAS(d_status, 0, SWIMBA_ERR_DEVICE_BOUNDS);
        return;
    }

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // Split launch (grid = [B, head pairs, 2]; used when one CTA per (sequence, head pair) would
    // leave SMs idle): the CTAs of the first z-plane, which start first, walk the whole
    // sequence but evaluate the first split_tiles tiles for their end state only (about half the
    // cost of a full tile) and produce y from there on; the CTAs of the second plane produce y of
    // those first tiles.  No CTA waits for another.
    const bool head_part = SPLIT && blockIdx.z == 1;             // y of the leading tiles only
    const int seg = SPLIT ? 0 : blockIdx.x, b = SPLIT ? blockIdx.x : blockIdx.z;
    const int L = prm.L, nseg = prm.nseg;
    const int H = prm.H;
    const int seg_base = b * prm.nseg;               // index of the sequence's first segment
    const int64_t rec_base = (int64_t)b * H * (prm.Lpad / ST);   // tile record of head 0, tile 0: + h * rec_hstride
    const int rec_hstride = prm.Lpad / ST;
    const int HG = H / prm.G, ppg = pairs_per_group(H, prm.G);
    const int pair = blockIdx.y;
    const int g = pair / ppg, pr = pair % ppg;
    const int head0 = g * HG + pr * NHD;
    const int nh = min(NHD, HG - pr * NHD);          // heads this CTA really has
    const int t_begin = seg * prm.seg_len;
    const int t_end = head_part ? min(L, prm.split_tiles * ST) : min(L, t_begin + prm.seg_len);
    const int ntiles = (t_end - t_begin + ST - 1) / ST;
    // leading tiles that only carry the state forward (tile j is a full tile iff j >= n_pre;
    // barriers that only full tiles use count their phases in full tiles, jf = j - n_pre)
    const int n_pre = SPLIT ? (head_part ? 0 : min(prm.split_tiles, ntiles)) : 0;

    if (tid == 0) {
        for (int s = 0; s < B_SLOTS; ++s) {
            tc::mbar_init(&bars->b_full[s], 1);
            tc::mbar_init(&bars->b_empty[s], 1);
        }
        tc::mbar_init(&bars->c_full, 1);
        tc::mbar_init(&bars->c_empty, 1);
        for (int s = 0; s < X_SLOTS; ++s) tc::mbar_init(&bars->x_full[s], 1);
        for (int s = 0; s < Y_BARS; ++s) tc::mbar_init(&bars->y_staged[s], NCW);
        for (int s = 0; s < 2; ++s) {
            tc::mbar_init(&bars->xp_full[s], NCW);
            tc::mbar_init(&bars->xp_free[s], 1);
        }
        tc::mbar_init(&bars->rec_free, NCW);
        tc::mbar_init(&bars->m_full, NCW);
        tc::mbar_init(&bars->g_full, 1);
        tc::mbar_init(&bars->yd_full, 1);
        tc::mbar_init(&bars->dh_full, 1);
        *abort_flag = 0;
        tc::fence_mbar_init();
    }
    if (warp == WARP_MMA) {
        tc::tmem_alloc(&sm->tmem_slot, TM_COLS);
        tc::tmem_relinquish();
    }
    if (warp == WARP_TMA && lane == 0) {
        tc::prefetch_tmap(&tmap_b);
        tc::prefetch_tmap(&tmap_c);
        tc::prefetch_tmap(&tmap_x);
        tc::prefetch_tmap(&tmap_y);
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = sm->tmem_slot;
    grid_dep_launch();

    // Warp index as a value the compiler knows to be warp-uniform.
    const int uwarp = __shfl_sync(0xffffffffu, warp, 0);
    if (uwarp == WARP_TMA) {
        // ------------------------------------------------------------------ TMA producer, y stores
        // (the whole warp runs the loop; one elected lane issues the copies)
        const bool leader = tc::elect_one();
        auto load_x = [&](int j) {                           // x and, on the same barrier, the tile's record
            const int s = j % X_SLOTS;
            tc::mbar_arrive_expect_tx(&bars->x_full[s], nh * (SLAB + (uint32_t)sizeof(TileRec)));
            for (int hd = 0; hd < nh; ++hd)
                tc::tma_load_4d(smem + SM_X + (s * NHD + hd) * SLAB, &tmap_x, &bars->x_full[s], 0, head0 + hd,
                                t_begin + j * ST, b);
        };
        auto load_rec = [&](int j) {
            for (int hd = 0; hd < nh; ++hd) {
                const int64_t r = rec_base + (int64_t)(head0 + hd) * rec_hstride + t_begin / ST + j;
                tc::bulk_load(sm->sc[hd].cb, prm.rec[r].cb, (ST + 4) * sizeof(float), &bars->x_full[j % X_SLOTS]);
                tc::bulk_load(&sm->sc[hd].aux, prm.aux + r, (uint32_t)sizeof(TileAux), &bars->x_full[j % X_SLOTS]);
                tc::bulk_load(sm->sc[hd].row, prm.l2 + r * ST, ST * sizeof(float), &bars->x_full[j % X_SLOTS]);
            }
        };
        // a stream's tile: Btilde waits for MMA 4 of the tile before the last, Ctilde for the last one's copy
        auto load_stream = [&](const CUtensorMap *m, int j, uint8_t *dst, uint64_t *full_bar) {
            tc::mbar_arrive_expect_tx(full_bar, 2 * SLAB);
            tc::tma_load_3d(dst, m, full_bar, g * SN, t_begin + j * ST, b);
            tc::tma_load_3d(dst + SLAB, m, full_bar, g * SN + 64, t_begin + j * ST, b);
        };
        auto load_b = [&](int j) {
            const int s = j & 1;
            tc::mbar_wait(&bars->b_empty[s], ((j >> 1) & 1) ^ 1, abort_flag, d_status);
            if (leader) load_stream(&tmap_b, j, smem + SM_B + s * 2 * SLAB, &bars->b_full[s]);
            __syncwarp();
        };
        auto load_c = [&](int j) {                           // (full tiles only)
            const int jf = SPLIT ? j - n_pre : j;
            tc::mbar_wait(&bars->c_empty, (jf & 1) ^ 1, abort_flag, d_status);
            if (leader) load_stream(&tmap_c, j, smem + SM_C, &bars->c_full);
            __syncwarp();
        };
        // the y tiles staged over x of tile j (rows past the end of the sequence are clipped by the tensor map)
        auto store_y = [&](int j) {
            const int jf = SPLIT ? j - n_pre : j;
            tc::mbar_wait(&bars->y_staged[jf % Y_BARS], (jf / Y_BARS) & 1, abort_flag, d_status);
            if (leader) {
                for (int q = 0; q < nh; ++q) {
                    const uint8_t *s_y = smem + SM_X + ((j % X_SLOTS) * NHD + q) * SLAB;
                    if (prm.add) tc::tma_reduce_add_4d(&tmap_y, s_y, 0, head0 + q, t_begin + j * ST, b);
                    else tc::tma_store_4d(&tmap_y, s_y, 0, head0 + q, t_begin + j * ST, b);
                }
                tc::bulk_commit_group();
            }
            __syncwarp();
        };
        const int ahead = min(X_SLOTS, ntiles);
        if (!prm.early) grid_dep_wait();
        if (leader)
            for (int j = 0; j < ahead; ++j) load_x(j);
        if (prm.early) grid_dep_wait();
        if (leader)
            if (ntiles > 0) load_rec(0);
        __syncwarp();
        if (ntiles > 0) load_b(0);
        if (ntiles > 0 && n_pre == 0) load_c(0);
        if (ntiles > 1) {
            load_b(1);
            tc::mbar_wait(&bars->rec_free, 0, abort_flag, d_status);
            if (leader) load_rec(1);
            __syncwarp();
        }
        for (int j = 0; j < ntiles; ++j) {                   // while tile j is worked
            if (j + 1 < ntiles && (!SPLIT || j + 1 >= n_pre)) load_c(j + 1);
            // the tile in front gives back its x slot: a full one once its y has gone out; a leading one's w.X was
            // done when the record of tile j was taken, which has been waited for.  (Not on xp_full: two tiles share
            // a barrier there, and tile j + 1, whose record is out, could have completed its phase too.)
            if (j > 0 && (!SPLIT || j > n_pre)) store_y(j - 1);
            if (j + 2 < ntiles) load_b(j + 2);
            if (leader && j > 0 && j - 1 + X_SLOTS < ntiles) {
                tc::bulk_wait_read_all();
                load_x(j - 1 + X_SLOTS);
            }
            __syncwarp();
            if (j + 2 < ntiles) {                            // (the next tile's record has been taken)
                tc::mbar_wait(&bars->rec_free, (j + 1) & 1, abort_flag, d_status);
                if (leader) load_rec(j + 2);
                __syncwarp();
            }
        }
        if (ntiles > n_pre) store_y(ntiles - 1);
        if (leader) tc::bulk_wait_read_all();
    } else if (uwarp == WARP_MMA) {
        // ------------------------------------------------------------------ MMA issuer
        // The whole warp runs the loop and the waits; one elected lane issues the MMAs and the
        // commits.  The order of issue is relied upon where PTX promises it: products into one accumulator in one
        // shape, a product behind a copy.  Everything else that follows in the same columns waits for a commit:
        // MMA 2 (another shape than MMA 3) and the copy of the next Ctilde for MMA 3, MMA 1 for MMA 2, whose masked tile
        // it overwrites.
        grid_dep_wait();
        const bool leader = tc::elect_one();
        // The products against the shared Ctilde / Btilde tiles (MMA 1, 3, 4) are issued for both heads at once:
        // the shared operand is read from shared memory once instead of once per head.
        constexpr uint32_t id_g = tc::idesc_bf16(128, 128, 0, 0);         // C (TMEM) x B (K-major)
        constexpr uint32_t id_x = tc::idesc_bf16(128, 64, 0, 1);          // M (TMEM) x X (MN-major)
        constexpr uint32_t id_h = tc::idesc_bf16(128, 128, 0, 1);         // w.X (TMEM) x B (MN-major)
        const uint32_t id_y = nh == 2 ? tc::idesc_bf16(128, 128, 0, 0) : tc::idesc_bf16(128, 64, 0, 0);   // C (TMEM) x H, K-major
        const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem, 0);
        // descriptors of the first K step; later steps and slots advance the address field
        const uint64_t dC = tc::smem_desc_sw128(tc::smem_u32(smem + SM_C), 16, 1024);        // K-major
        const uint64_t dB = tc::smem_desc_sw128(tc::smem_u32(smem + SM_B), 16, 1024);        // K-major
        const uint64_t dBt = tc::smem_desc_sw128(tc::smem_u32(smem + SM_B), SLAB, 1024);     // MN-major
        const uint64_t dH = tc::smem_desc_sw128(tc::smem_u32(smem + SM_H), 16, 1024);
        const uint64_t dX0 = tc::smem_desc_sw128(tc::smem_u32(smem + SM_X), SLAB, 1024);
        // MMA 1 of tile j: G = Ctilde Btilde^T (K = state index), for both heads, over the masked tile in front of it.
        // Ctilde is copied to tensor memory first, as soon as MMA 3 of the tile in front has read the last one:
        // MMA 1 and MMA 3 would each read it from shared memory.
        auto copy_c = [&](int j) {
            const int jf = SPLIT ? j - n_pre : j;
            tc::mbar_wait(&bars->c_full, jf & 1, abort_flag, d_status);
            tc::tc_fence_after();
            if (leader) {
                const uint64_t d = tc::smem_desc_fresh(dC);
#pragma unroll
                for (int kk = 0; kk < 8; ++kk)
                    tc::tmem_copy_128x256b(tmem_u + TM_C + kk * 8, tc::smem_desc_advance(d, (kk >> 2) * SLAB + (kk & 3) * 32));
                tc::mma_commit(&bars->c_empty);
            }
            __syncwarp();
        };
        auto issue_g = [&](int j) {
            tc::mbar_wait(&bars->b_full[j & 1], (j >> 1) & 1, abort_flag, d_status);
            tc::tc_fence_after();
            if (leader) {
                const uint64_t d = tc::smem_desc_fresh(tc::smem_desc_advance(dB, (j & 1) * 2 * SLAB));
#pragma unroll
                for (int kk = 0; kk < 8; ++kk)
                    tc::mma_ts(tmem_u + TM_G, tmem_u + TM_C + kk * 8,
                               tc::smem_desc_advance(d, (kk >> 2) * SLAB + (kk & 3) * 32), id_g, kk > 0);
                tc::mma_commit(&bars->g_full);
            }
            __syncwarp();
        };
        if (n_pre == 0 && ntiles > 0) {
            copy_c(0);
            issue_g(0);
        }
        for (int j = 0; j < ntiles; ++j) {
            const bool full = !SPLIT || j >= n_pre;
            const int jf = SPLIT ? j - n_pre : j;
            if (!full) tc::mbar_wait(&bars->b_full[j & 1], (j >> 1) & 1, abort_flag, d_status);
            // MMA 4: dH[p,n] = sum_s (w_s x_s[p]) Btilde[s,n]   (K = token; A = w.X in TMEM, both heads' channels).  It
            // and MMA 1 run ahead: under the epilogue of the tile in front.
            tc::mbar_wait(&bars->xp_full[j & 1], (j >> 1) & 1, abort_flag, d_status);
            tc::tc_fence_after();
            if (leader) {
                const uint64_t d = tc::smem_desc_fresh(tc::smem_desc_advance(dBt, (j & 1) * 2 * SLAB));
                const uint32_t xp = tmem_u + (!full && (j & 1) ? TM_Y : TM_XP);
#pragma unroll
                for (int kk = 0; kk < 8; ++kk)             // (leading tiles accumulate)
                    tc::mma_ts(tmem_u + TM_DH, xp + kk * 8, tc::smem_desc_advance(d, kk * 2048),
                               id_h, (kk > 0) || (!full && j > 0));
                if (j == n_pre - 1) tc::mma_commit(&bars->dh_full);
                if (!full) tc::mma_commit(&bars->xp_free[j & 1]);
                tc::mma_commit(&bars->b_empty[j & 1]);
            }
            __syncwarp();
            if (full) {
                // MMA 3: Y = Ctilde Hprev^T  (K = state index; B = bf16 states, rows = channels; they are stored before
                // w.X of this tile), once the tile in front has read its Y
                if (jf > 0) tc::mbar_wait(&bars->y_staged[(jf - 1) % Y_BARS], ((jf - 1) / Y_BARS) & 1, abort_flag, d_status);
                tc::tc_fence_after();
                if (leader) {
                    const uint64_t d = tc::smem_desc_fresh(dH);
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)
                        tc::mma_ts(tmem_u + TM_Y, tmem_u + TM_C + kk * 8,
                                   tc::smem_desc_advance(d, (kk >> 2) * SLAB + (kk & 3) * 32), id_y, kk > 0);
                    tc::mma_commit(&bars->dh_full);          // (MMA 4 and 3: the state may be advanced, its copy replaced)
                }
                __syncwarp();
                tc::mbar_wait(&bars->dh_full, (jf + (SPLIT && n_pre > 0 ? 1 : 0)) & 1, abort_flag, d_status);
                if (j + 1 < ntiles) copy_c(j + 1);
                // MMA 2: Y += M X per head (A = masked tile in TMEM, 16 tokens every 16 columns)
                tc::mbar_wait(&bars->m_full, jf & 1, abort_flag, d_status);
                tc::tc_fence_after();
                if (leader) {
                    for (int q = 0; q < nh; ++q) {
                        const uint64_t dX = tc::smem_desc_fresh(tc::smem_desc_advance(dX0, ((j % X_SLOTS) * NHD + q) * SLAB));
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk)
                            tc::mma_ts(tmem_u + TM_Y + q * 64, tmem_u + TM_G + kk * 16 + q * 8,
                                       tc::smem_desc_advance(dX, kk * 2048), id_x, 1);
                    }
                    tc::mma_commit(&bars->yd_full);
                }
                __syncwarp();
                if (j + 1 < ntiles) tc::mbar_wait(&bars->yd_full, jf & 1, abort_flag, d_status);
            }
            // MMA 1 of the next tile needs no state
            if (j + 1 < ntiles && j + 1 >= n_pre) {
                if (!full) copy_c(j + 1);
                issue_g(j + 1);
            }
        }
    } else {
        // ------------------------------------------------------------------ compute warps
        // Warp (row block wq, share sub).  State and w.X: 32 channels of head wq / 2, the share 32 state indices / 32
        // tokens.  Mask: a block of 32 rows and 32 columns, both heads.  Epilogue: row i is a
        // token, the share one half of one head's channels.
        const int wq = uwarp & 3, sub = uwarp >> 2;
        const int i = wq * 32 + lane;
        const int hs = wq >> 1;                              // state: head of the pair
        const int he = sub >> 1, hf = sub & 1;               // epilogue: head of the pair, half of its channels
        const bool has_s = hs < nh, has_e = he < nh;
        const uint32_t lane_base = tmem + ((uint32_t)(wq * 32) << 16);
        const uint32_t tm_g = lane_base + TM_G + 32 * sub, tm_y = lane_base + TM_Y + 32 * sub;
        const uint32_t tm_dh = lane_base + TM_DH + 32 * sub;
        // 16-byte chunk c of this thread's part of row i, in the x and y slabs: base ^ 16 c
        const uint32_t row_off = tc::sw128_offset(i, 4 * hf);
        // of a pair of columns c, c + 1 = 2 (t % 4) of an 8 x 8 diagonal block, the bf16 halves that row t / 4 keeps
        const int below = (lane >> 2) - 2 * (lane & 3);
        const uint32_t keep = below < 0 ? 0u : (below == 0 ? 0xffffu : 0xffffffffu);
        const float Dh = prm.D && has_e ? prm.D[head0 + he] : 0.f;
        auto arrive = [&](uint64_t *bar) {                   // one arrival per warp, behind all lanes' work
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(bar);
        };
        // fp32 master copy of the state, rows (channels) 32 wq .. and columns (state indices) 32 sub .. in the fragment
        // layout: pair 8 m + 4 k + r is row 16 m + 8 k + t / 4, columns 8 r + 2 (t % 4) and the one behind.  (A row per
        // thread makes every access to the states in global memory touch 32 lines: 3 us at either end of a CTA.)
        uint64_t Hst[16];
        // its bf16 copy, MMA 3 operand of the next tile, decayed by f
        const uint32_t s_h = tc::smem_u32(smem + SM_H + (sub >> 1) * SLAB) +
                             tc::sw128_offset(32 * wq + (lane & 7), 4 * hf + (lane >> 3));
        auto store_h = [&](float f) {
            const uint64_t f2 = tc::f32x2(f, f);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint32_t o[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) o[r] = tc::f32x2_bf16(tc::f32x2_mul(f2, Hst[4 * q + r]));
                tc::stmatrix_x4(s_h + q * 1024, o[0], o[1], o[2], o[3]);
            }
            tc::fence_proxy_async_smem();
        };
        // offset of pair 8 m + 4 k + r inside the pair of heads' states, from this thread's first one
        auto h_off = [&](int e) { return 8 * (e >> 2) * SN + 8 * (e & 3); };
        const int h_mine = (32 * (wq & 1) + (lane >> 2)) * SN + 32 * sub + 2 * (lane & 3);
        {
            const bool first = seg == 0 && (prm.seg_states == 2 || (prm.seg_states == 3 && nseg == 1));
            const float *h_in = first ? prm.h_first : prm.h_in;
            // (states of earlier segments come from the scan in front; given ones go past L1)
            const bool wait = !prm.early || (prm.seg_states && !first);
            if (wait) grid_dep_wait();
#pragma unroll
            for (int q = 0; q < 16; ++q) Hst[q] = 0;
            if (h_in && has_s) {
                const int64_t row = (prm.seg_states && !first) ? ((int64_t)seg_base + seg) * H + head0 + hs
                                                               : (int64_t)b * H + head0 + hs;
                const float *src = h_in + row * SP * SN + h_mine;
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    const float2 v = __ldcg(reinterpret_cast<const float2 *>(src + h_off(e)));
                    Hst[e] = tc::f32x2(v.x, v.y);
                }
            }
        }
        grid_dep_wait();         // the step sizes, the streams
        // The leading tiles of a split launch are one long contraction: with every token weighted by its
        // decay up to the END OF THE RUN (exponent <= 0), (w . X)^T Btilde accumulates over all tiles of
        // the run in tensor memory and the state is touched once, at the run's last tile:
        //   H_end = 2^(sum of l_last over the run) H_in + sum_tiles (w' . X)^T Btilde.
        if (SPLIT && n_pre > 0 && has_s) {
            const TileScalars *rec0 = prm.rec + rec_base + (int64_t)(head0 + hs) * rec_hstride + t_begin / ST;
            float total = 0.f;
            for (int jr = 0; jr < n_pre; ++jr) total += rec0[jr].ends[3];
            const float dec = tc::ex2_approx(total);
#pragma unroll
            for (int q = 0; q < 16; ++q) Hst[q] = tc::f32x2_mul(Hst[q], tc::f32x2(dec, dec));
            sm->run_total[uwarp] = total;
            sm->run_done[uwarp] = 0.f;
            __syncwarp();
        }

        // What a tile's record means for this thread, taken when the record arrives:
        struct Prep {
            BlockWeights w[2];     // mask: weights of its columns, both heads
            BlockWeights wx;       // w.X: weights of its tokens (the same ones)
            float dec;             // decay of the state over the tile
            float row;             // epilogue: y = row Y + D x
            float pre;             // != 1: Y = Ctilde Hprev^T is multiplied by it before M X is added
            int fast;              // heads with MASK_ENTRIES for these rows, one bit each; of them, if any:
            float lr[2];           // l of row 32 wq + lane, relative to the block's start (garbage for the others)
        };
        const TileRec *const sc0 = &sm->sc[0], *const sc1 = &sm->sc[nh - 1];
        const TileRec *const scs = hs ? sc1 : sc0, *const sce = he ? sc1 : sc0;
        auto take_rec = [&](int j, Prep &p) {
            const float blocks0 = sc0->aux.blocks, blocks1 = sc1->aux.blocks;
            load_weights(p.w[0], sc0->cb + 32 * sub, lane);
            load_weights(p.w[1], sc1->cb + 32 * sub, lane);
            p.row = sce->row[i];
            p.dec = scs->aux.total;
            p.pre = 1.f;
            p.fast = 0;
            float lead = 1.f;                                // leading tiles: from the end of the tile to the end of the run
            if (SPLIT && j < n_pre) {
                const float done = sm->run_done[uwarp] + scs->ends[3];
                __syncwarp();
                sm->run_done[uwarp] = done;
                lead = tc::ex2_approx(sm->run_total[uwarp] - done);
                p.dec = 1.f;
            }
            // w.X: from where the column weights refer to, to the end of the tile
            auto take_wx = [&](float f, const BlockWeights &w0, const BlockWeights &w1) {
                const uint64_t f2 = tc::f32x2(f, f);
#pragma unroll
                for (int r = 0; r < 4; ++r) p.wx.v[r] = tc::f32x2_mul(f2, hs ? w1.v[r] : w0.v[r]);
            };
            if (blocks0 == 0.f && blocks1 == 0.f) {
                take_wx(scs->aux.from_ref * lead, p.w[0], p.w[1]);
            } else {
                int m0 = blocks0 == 0.f ? MASK_TILE : MASK_BLOCKS, m1 = blocks1 == 0.f ? MASK_TILE : MASK_BLOCKS;
                const float Lw0 = wq ? sc0->ends[wq - 1] : 0.f, Lw1 = wq ? sc1->ends[wq - 1] : 0.f;
                // (weights of a fast block's columns come without their decay: w.X needs it, its own rows do not)
                BlockWeights w0 = p.w[0], w1 = p.w[1];
                if (blocks0 == 2.f) {
                    m0 = mask_mode(sc0->ends, wq);
                    if (mask_mode(sc0->ends, sub) == MASK_ENTRIES) decay_weights(w0, sc0, sub, lane);
                }
                if (blocks1 == 2.f) {
                    m1 = mask_mode(sc1->ends, wq);
                    if (mask_mode(sc1->ends, sub) == MASK_ENTRIES) decay_weights(w1, sc1, sub, lane);
                }
                const int me = he ? m1 : m0;
                take_wx(((hs ? blocks1 : blocks0) != 0.f ? tc::ex2_approx(scs->ends[3] - scs->ends[sub]) : scs->aux.from_ref) * lead,
                        w0, w1);
                const float f0 = m0 == MASK_TILE ? 1.f : tc::ex2_approx(Lw0 - sc0->ends[sub]);
                const float f1 = m1 == MASK_TILE ? 1.f : tc::ex2_approx(Lw1 - sc1->ends[sub]);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    if (!(sub == wq && m0 == MASK_ENTRIES)) p.w[0].v[r] = tc::f32x2_mul(w0.v[r], tc::f32x2(f0, f0));
                    if (!(sub == wq && m1 == MASK_ENTRIES)) p.w[1].v[r] = tc::f32x2_mul(w1.v[r], tc::f32x2(f1, f1));
                }
                if (me == MASK_BLOCKS) p.pre = tc::ex2_approx(he ? Lw1 : Lw0);
                if (me == MASK_ENTRIES) { p.pre = tc::ex2_approx(p.row); p.row = 1.f; }
                if (m0 == MASK_ENTRIES || m1 == MASK_ENTRIES) {
                    p.fast = (m0 == MASK_ENTRIES ? 1 : 0) | (m1 == MASK_ENTRIES ? 2 : 0);
                    p.lr[0] = sc0->row[i] - Lw0;
                    p.lr[1] = sc1->row[i] - Lw1;
                }
            }
            tc::fence_proxy_async_smem();                    // (the record is refilled by a copy next)
            arrive(&bars->rec_free);
        };
        // w . X of tile j (rows of the X slab -> A operand of MMA 4)
        auto scale_x = [&](int j, int sx, const BlockWeights &wx) {
            uint32_t xp = lane_base + 16 * sub + TM_XP;
            const bool lead = SPLIT && j < n_pre;
            if (lead) {
                if (j & 1) xp += TM_Y - TM_XP;
                // (its columns are free once the product before the previous tile's has read them)
                if (j > 1) tc::mbar_wait(&bars->xp_free[j & 1], ((j >> 1) & 1) ^ 1, abort_flag, d_status);
                tc::tc_fence_after();
            }
            if (has_s) scale_to_tmem(smem + SM_X + (sx * NHD + hs) * SLAB, wx, 32 * (wq & 1), 32 * sub, lane, xp);
            if (lead) tc::fence_proxy_async_smem();          // (the x slot is refilled by a copy next)
            tc::tmem_st_wait();
            tc::tc_fence_before();
            arrive(&bars->xp_full[j & 1]);
        };
        Prep cur;
        if (ntiles > 0) {
            tc::mbar_wait(&bars->x_full[0], 0, abort_flag, d_status);
            if (n_pre == 0) store_h(scs->aux.to_ref);
            take_rec(0, cur);
            scale_x(0, 0, cur.wx);
        }

        int sx = 0, sx_next = 0;                             // x slots of this tile and of the next one
        uint32_t x_ph = 0;
        for (int j = 0; j < ntiles; ++j, sx = sx_next) {
            sx_next = sx + 1;
            if (sx_next == X_SLOTS) { sx_next = 0; x_ph ^= 1; }
            const bool full = !SPLIT || j >= n_pre;
            const int jf = SPLIT ? j - n_pre : j;
            const uint32_t dh_ph = (full ? jf + (SPLIT && n_pre > 0 ? 1 : 0) : 0) & 1;
            if (full) {
                // ---- decay mask: G (fp32, TMEM) -> M of both heads (bf16, TMEM)
                tc::mbar_wait(&bars->g_full, jf & 1, abort_flag, d_status);
                tc::tc_fence_after();
                if (sub > wq) {
                    uint32_t zero[16];
#pragma unroll
                    for (int q = 0; q < 16; ++q) zero[q] = 0u;
                    tc::tmem_st16(tm_g, zero);
                    tc::tmem_st16(tm_g + 16, zero);
                } else if (cur.fast) {
                    mask_block_entries(tm_g, cur.w, cur.lr, cur.fast, sub == wq, keep, lane);
                } else if (sub < wq) {
                    mask_block<false>(tm_g, cur.w, 0u);
                } else {
                    mask_block<true>(tm_g, cur.w, keep);
                }
                // (one answer for the warp, tensor memory being accessed by whole warps: with MASK_ENTRIES the factor is each
                // row's own, and 1 for rows that nothing has decayed in front of)
                if (__any_sync(0xffffffffu, cur.pre != 1.f)) {
                    // ---- Y = Ctilde Hprev^T scaled in place
                    tc::mbar_wait(&bars->dh_full, dh_ph, abort_flag, d_status);
                    tc::tc_fence_after();
                    const uint64_t e2 = tc::f32x2(cur.pre, cur.pre);
                    uint32_t yo[2][16];
                    tc::tmem_ld16(tm_y, yo[0]);
                    tc::tmem_ld16(tm_y + 16, yo[1]);
                    tc::tmem_ld_wait();
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh) {
#pragma unroll
                        for (int q = 0; q < 16; q += 2) {
                            const float2 v = tc::f32x2_get(tc::f32x2_mul(e2, f32x2_bits(yo[hh][q], yo[hh][q + 1])));
                            yo[hh][q] = __float_as_uint(v.x);
                            yo[hh][q + 1] = __float_as_uint(v.y);
                        }
                        tc::tmem_st16(tm_y + 16 * hh, yo[hh]);
                    }
                }
                tc::tmem_st_wait();
                tc::tc_fence_before();
                arrive(&bars->m_full);
            }

            // ---- state: H = exp(l_last) H + dH; of the leading tiles only at the last one, with the decay of the
            // whole run
            float h_next = 1.f;
            if (j + 1 < ntiles) {
                tc::mbar_wait(&bars->x_full[sx_next], x_ph, abort_flag, d_status);
                h_next = scs->aux.to_ref;
            }
            if (full || j == n_pre - 1) {
                tc::mbar_wait(&bars->dh_full, dh_ph, abort_flag, d_status);
                tc::tc_fence_after();
                const uint64_t dec2 = tc::f32x2(cur.dec, cur.dec);
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    uint32_t dh[16];
                    tc::tmem_ld_16x256b_x4(tm_dh + ((uint32_t)(16 * m) << 16), dh);
                    tc::tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 8; ++e) {            // (its registers: columns r first, then rows k)
                        const int k = e >> 2, r = e & 3;
                        Hst[8 * m + e] = tc::f32x2_fma(dec2, Hst[8 * m + e],
                                                       f32x2_bits(dh[4 * r + 2 * k], dh[4 * r + 2 * k + 1]));
                    }
                }
                if (j + 1 < ntiles) store_h(h_next);           // (MMA 3 has read the old copy)
                tc::tc_fence_before();
            }
            // ---- w . X of the next tile while MMA 2 runs
            const float row = cur.row;
            if (j + 1 < ntiles) {
                take_rec(j + 1, cur);
                scale_x(j + 1, sx_next, cur.wx);
            }
            if (full) {
                // ---- epilogue: y_i = row Y_i + D x_i, staged for the TMA store where x_i stood
                uint8_t *s_y = smem + SM_X + (sx * NHD + he) * SLAB;
                tc::mbar_wait(&bars->yd_full, jf & 1, abort_flag, d_status);
                tc::tc_fence_after();
                if (has_e) {
                    const uint64_t D2 = tc::f32x2(Dh, Dh), r2 = tc::f32x2(row, row);
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh) {
                        uint32_t yd[16];
                        tc::tmem_ld16(tm_y + 16 * hh, yd);
                        uint4 xr[2];
#pragma unroll
                        for (int c = 0; c < 2; ++c)
                            xr[c] = *reinterpret_cast<const uint4 *>(s_y + (row_off ^ ((2 * hh + c) << 4)));
                        tc::tmem_ld_wait();
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            const uint32_t xw[4] = {xr[c].x, xr[c].y, xr[c].z, xr[c].w};
                            uint32_t o[4];
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                const int e = 8 * c + 2 * q;
                                o[q] = tc::f32x2_bf16(tc::f32x2_fma(
                                    D2, f32x2_bits(xw[q] << 16, xw[q] & 0xffff0000u),
                                    tc::f32x2_mul(r2, f32x2_bits(yd[e], yd[e + 1]))));
                            }
                            *reinterpret_cast<uint4 *>(s_y + (row_off ^ ((2 * hh + c) << 4))) = make_uint4(o[0], o[1], o[2], o[3]);
                        }
                    }
                }
                tc::tc_fence_before();
                tc::fence_proxy_async_smem();
                arrive(&bars->y_staged[jf % Y_BARS]);
            }
        }

        // ---- final state
        if (prm.h_out && seg == nseg - 1 && !head_part && has_s) {
            float *dst = prm.h_out + ((int64_t)b * prm.H + head0 + hs) * SP * SN + h_mine;
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                float2 v = tc::f32x2_get(Hst[e]);
                float2 *p = reinterpret_cast<float2 *>(dst + h_off(e));
                if (prm.add) {
                    const float2 w = *p;
                    v.x += w.x; v.y += w.y;
                }
                *p = v;
            }
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == WARP_MMA) tc::tmem_dealloc(tmem, TM_COLS);
}


bool ensure_ssd_run()
{
    const size_t smem = SM_SMALL + sizeof(RunSmall);
    return ensure_dynamic_smem((const void *)ssd_run_kernel<false>, smem) &&
           ensure_dynamic_smem((const void *)ssd_run_kernel<true>, smem);
}

void launch_ssd_run(LaunchCtx &ctx, dim3 grid, const CUtensorMap &tm_b, const CUtensorMap &tm_c, const CUtensorMap &tm_x,
                    const CUtensorMap &tm_y, const SsdParams &p)
{
    launch_kernel(p.split_tiles > 0 ? ssd_run_kernel<true> : ssd_run_kernel<false>, grid, dim3(RUN_THREADS),
                  SM_SMALL + sizeof(RunSmall), ctx.stream, true, tm_b, tm_c, tm_x, tm_y, p);
}

}  // namespace swimba
