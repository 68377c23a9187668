// K1 for a handful of tokens (the decode step: one token per sequence).  With at most a few
// hundred tokens the routing / projection stage moves almost nothing besides the expert matrices
// (Theorem 2: only the active experts are touched), so what counts is latency: no histogram, no
// per-expert lists in global memory, no tile table, short kernels chained by programmatic dependent
// launch.
//   router_small_kernel   four warps per token: logits in fp32 with a fixed summation order, softmax
//                         over all E, the k largest kept with their softmax values, NOT renormalised
//                         (router softmax equation and the sentence after it); clears the token's
//                         row of the fp32 mixed streams
//   project_small_kernel  one CTA per (expert, 16 rows of its matrix, share of the tokens): finds the tokens routed to
//                         its expert by scanning the k * T routing entries, streams its 16 x F slice
//                         of W_e once, multiplies it with those tokens' features on the tensor cores
//                         (mma.sync m16n8k16, features split over the eight warps and added in a
//                         fixed order) and adds pi_{t,e} times the result into the token's row of
//                         the mixed streams (Theorem 1).  With k <= 2 a row receives at most two
//                         additions onto zero, so the sum does not depend on their order; with more
//                         experts the rows go to slots (t, j), which the update sums in order.
// At most SM_FUSED tokens (and not too many CTAs): every CTA of the projection computes the few logits itself (the router
// matrix and the tokens are in L2, and a dependent launch costs more than they do); the rows go to slots,
// since no kernel in front could clear the mixed streams.  A decode step of one token, 64 heads, 8 experts,
// F = 2048: router and projection apart 14.7 us, one kernel (and the states read under it) 8.5 us.
#include <algorithm>

#include "internal.h"

namespace swimba {

namespace {
constexpr int SM_MAX_E = 16;        // experts the small router holds in registers
constexpr int SM_MAX_T = FRONT_SMALL_TOKENS;
constexpr int SM_ROWS = 16;         // rows of W_e per CTA (the M of m16n8k16)
constexpr int SM_WARPS = 8;
constexpr int SM_NT = 4;            // 8-token column tiles worked per pass
constexpr int SM_FUSED = 4;         // tokens up to which the projection routes as well

// k rounds of arg-max over the logits (ties to the lower index); returns the next expert.  Logits that compare
// with nothing (NaN) leave the lowest expert not taken yet: a token never picks one twice, so that an
// expert's list holds no more entries than there are tokens.
__device__ __forceinline__ int next_expert(const float (&g)[SM_MAX_E], int E, unsigned taken)
{
    int best = __ffs(~taken) - 1;
    float bv = -INFINITY;
#pragma unroll
    for (int e = 0; e < SM_MAX_E; ++e)
        if (e < E && !((taken >> e) & 1u) && g[e] > bv) { bv = g[e]; best = e; }
    return best;
}
}  // namespace

__global__ void __launch_bounds__(256)
router_small_kernel(const __nv_bfloat16 *__restrict__ u, const __nv_bfloat16 *__restrict__ W_r, int Ttok,
                    int F, int E, int k, int32_t *__restrict__ idx, float *__restrict__ w,
                    float4 *__restrict__ bc_zero, int bc_vec_per_token, const ScalarsArgs scalars)
{
    // two tokens per block, four warps per token (a quarter of the features each, partial logits
    // added in warp order)
    __shared__ float s_part[2][4][SM_MAX_E];
    grid_dep_wait();        // the previous step's update may still be reading the mixed streams
    grid_dep_launch();
    if ((int)blockIdx.x >= (Ttok + 1) / 2) {
        // SSD step sizes and tile log-decays of the same call (they depend on dt only)
        ssd_scalars_block<false>(scalars, blockIdx.x - (Ttok + 1) / 2);
        return;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int tl = warp >> 2, part = warp & 3;
    const int t = blockIdx.x * 2 + tl;
    const bool live = t < Ttok;
    float acc[SM_MAX_E];
#pragma unroll
    for (int e = 0; e < SM_MAX_E; ++e) acc[e] = 0.f;
    if (live) {
        for (int v = part * 32 + lane; v < bc_vec_per_token; v += 128)
            bc_zero[(int64_t)t * bc_vec_per_token + v] = make_float4(0.f, 0.f, 0.f, 0.f);
        const __nv_bfloat16 *urow = u + (int64_t)t * F;
        const int fq = F / 4;                               // (a multiple of 8)
#pragma unroll 2
        for (int f = part * fq + lane * 8; f < (part + 1) * fq; f += 256) {
            float uv[8];
            load8(urow + f, uv);
#pragma unroll
            for (int e = 0; e < SM_MAX_E; ++e) {
                if (e < E) {
                    float wv[8];
                    load8(W_r + (int64_t)e * F + f, wv);
#pragma unroll
                    for (int i = 0; i < 8; ++i) acc[e] = fmaf(wv[i], uv[i], acc[e]);
                }
            }
        }
    }
    // sixteen sums over the lanes by halving exchanges: expert 8 b4 + 4 b3 + 2 b2 + b1 ends on the lanes
    // whose bits 4 .. 1 are b4 .. b1 (unused experts are zero)
    static_assert(SM_MAX_E == 16, "the reduction is for sixteen values");
#pragma unroll
    for (int o = 16, m = 8; m >= 1; o >>= 1, m >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int q = 0; q < m; ++q) {
            const float send = up ? acc[q] : acc[q + m], keep = up ? acc[q + m] : acc[q];
            acc[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 1);
    if ((lane & 1) == 0) s_part[tl][part][lane >> 1] = acc[0];
    __syncthreads();
    if (!live || part != 0) return;
#pragma unroll
    for (int e = 0; e < SM_MAX_E; ++e)
        acc[e] = e < E ? ((s_part[tl][0][e] + s_part[tl][1][e]) + s_part[tl][2][e]) + s_part[tl][3][e] : -INFINITY;
    // softmax over all E, then k rounds of arg-max; every lane holds the same values, lane 0 writes
    float m = acc[0];
#pragma unroll
    for (int e = 1; e < SM_MAX_E; ++e) m = fmaxf(m, acc[e]);
    float den = 0.f, pe[SM_MAX_E];
#pragma unroll
    for (int e = 0; e < SM_MAX_E; ++e) {
        pe[e] = e < E ? expf(acc[e] - m) : 0.f;
        den += pe[e];
    }
    const float inv = 1.f / den;
    unsigned taken = 0u;
    for (int j = 0; j < k; ++j) {
        const int best = next_expert(acc, E, taken);
        taken |= 1u << best;
        float pb = 0.f;
#pragma unroll
        for (int e = 0; e < SM_MAX_E; ++e) if (e == best) pb = pe[e];
        if (lane == 0) {
            idx[(int64_t)t * k + j] = best;
            w[(int64_t)t * k + j] = pb * inv;
        }
    }
}

__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                               uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// How the rows leave: added to BC[t, :] (fp32, cleared before), stored to slots BC[(t*k + j), :] (fp32), or,
// for the forward's bf16 streams, stored (one expert per token) or added (two; 0 + a + b does not depend on
// the order).  FUSED (slots): the routing is computed here, by every CTA for itself; the first CTA writes it
// to idx / w.
enum { ROWS_ADD = 0, ROWS_SLOTS = 1, ROWS_BF16 = 2 };
template <int ROWS, bool FUSED>
__global__ void __launch_bounds__(256)
project_small_kernel(const __nv_bfloat16 *__restrict__ u, const __nv_bfloat16 *__restrict__ W_r,
                     const __nv_bfloat16 *__restrict__ W_e, int32_t *__restrict__ idx, float *__restrict__ w, int Ttok,
                     int F, int S, int E, int k, int share, void *__restrict__ BCv, int check, int *d_status)
{
    float *BC = reinterpret_cast<float *>(BCv);
    __shared__ int s_tok[SM_MAX_T], s_out[SM_MAX_T];
    __shared__ float s_wgt[SM_MAX_T];
    __shared__ int s_count;
    __shared__ float s_red[SM_WARPS][SM_ROWS][8 * SM_NT + 1];
    __shared__ float s_logit[FUSED ? SM_FUSED : 1][SM_MAX_E];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int e = blockIdx.y, row0 = blockIdx.x * SM_ROWS;
    if (tid == 0) s_count = 0;
    __syncthreads();
    // (this kernel runs at all only because every router block is past its wait: what the next kernel reads
    // before its own wait is complete)
    if (!FUSED) grid_dep_launch();
    // 32-feature steps of this warp: the first (steps % 8) warps take one more
    const int g = lane >> 2, tq = lane & 3;
    const int steps = F >> 5, base_n = steps / SM_WARPS, extra = steps % SM_WARPS;
    const int nsteps = base_n + (warp < extra ? 1 : 0), f_warp = (warp * base_n + min(warp, extra)) * 32;
    const __nv_bfloat16 *wrow0 = W_e + ((int64_t)e * S + row0 + g) * F + f_warp + tq * 8;
    const __nv_bfloat16 *wrow1 = wrow0 + (int64_t)8 * F;
    // The matrix slice does not depend on the routing: when a warp's share fits in registers (F up to
    // 2048) it is fetched before the wait, under the tail of the kernel in front, and serves every pass.
    // (Fused, only the few active experts' slices are wanted: fetched once the routing is known.)
    const bool resident = !FUSED && base_n + (extra ? 1 : 0) <= 8;
    uint4 a0[8], a1[8];
    if (resident) {
#pragma unroll
        for (int st = 0; st < 8; ++st) {
            if (st < nsteps) {
                a0[st] = *reinterpret_cast<const uint4 *>(wrow0 + st * 32);
                a1[st] = *reinterpret_cast<const uint4 *>(wrow1 + st * 32);
            }
        }
    }
    grid_dep_wait();        // routing entries (fused: the previous step's readers of the slots)
    if (FUSED) {
        grid_dep_launch();
        // one warp per (token, expert) logit in turn; every CTA sums in the same order
        for (int q = warp; q < Ttok * E; q += SM_WARPS) {
            const int t = q / E, ee = q - t * E;
            const __nv_bfloat16 *ur = u + (int64_t)t * F, *wr = W_r + (int64_t)ee * F;
            float acc = 0.f;
#pragma unroll 4
            for (int f = lane * 8; f < F; f += 256) {
                float uv[8], wv[8];
                load8(ur + f, uv);
                load8(wr + f, wv);
#pragma unroll
                for (int i = 0; i < 8; ++i) acc = fmaf(wv[i], uv[i], acc);
            }
            acc = warp_sum(acc);
            if (lane == 0) s_logit[t][ee] = acc;
        }
        __syncthreads();
        if (tid < Ttok) {
            float lg[SM_MAX_E], pe[SM_MAX_E], m = -INFINITY, den = 0.f;
#pragma unroll
            for (int q = 0; q < SM_MAX_E; ++q) {
                lg[q] = q < E ? s_logit[tid][q] : -INFINITY;
                m = fmaxf(m, lg[q]);
            }
#pragma unroll
            for (int q = 0; q < SM_MAX_E; ++q) {
                pe[q] = q < E ? expf(lg[q] - m) : 0.f;
                den += pe[q];
            }
            const float inv = 1.f / den;
            unsigned taken = 0u;
            for (int j = 0; j < k; ++j) {
                const int best = next_expert(lg, E, taken);
                taken |= 1u << best;
                float pb = 0.f;
#pragma unroll
                for (int q = 0; q < SM_MAX_E; ++q) if (q == best) pb = pe[q];
                if (best == e) {
                    const int slot = atomicAdd(&s_count, 1);
                    s_tok[slot] = tid;
                    s_out[slot] = tid * k + j;
                    s_wgt[slot] = pb * inv;
                }
                if (blockIdx.x == 0 && blockIdx.y == 0) {
                    idx[tid * k + j] = best;
                    w[tid * k + j] = pb * inv;
                }
            }
        }
    } else {
        // tokens of this CTA's share routed to its expert (a token picks an expert at most once); the order
        // of the list does not matter: every entry ends in its own output row
        const int t_beg = blockIdx.z * share, t_end = min(Ttok, t_beg + share);
        for (int i = t_beg * k + tid; i < t_end * k; i += blockDim.x) {
            const int ei = idx[i];
            if (check && (ei < 0 || ei >= E)) atomicCAS(d_status, 0, SWIMBA_ERR_DEVICE_BOUNDS);
            if (ei == e) {
                const int slot = atomicAdd(&s_count, 1);
                if (slot < SM_MAX_T) {
                    s_tok[slot] = i / k;
                    s_out[slot] = ROWS == ROWS_SLOTS ? i : i / k;
                    s_wgt[slot] = w[i];
                }
            }
        }
    }
    __syncthreads();
    const int count = min(s_count, SM_MAX_T);
    if (count == 0) return;
    for (int n0 = 0; n0 < count; n0 += 8 * SM_NT) {
        float acc[SM_NT][4];
#pragma unroll
        for (int q = 0; q < SM_NT; ++q)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[q][i] = 0.f;
        // 32 features per step, up to eight steps in flight: a lane holds 8 consecutive features of
        // its two matrix rows and of its token of every column tile; the first four feed one
        // m16n8k16, the last four the next (the contraction may run over the features in any
        // order, as long as both operands agree)
        for (int s0 = 0; s0 < nsteps; s0 += 8) {
            const int nst = min(8, nsteps - s0), f0 = s0 * 32;
#pragma unroll
            for (int st = 0; st < 8; ++st) {
                if (!resident && st < nst) {
                    a0[st] = *reinterpret_cast<const uint4 *>(wrow0 + f0 + st * 32);
                    a1[st] = *reinterpret_cast<const uint4 *>(wrow1 + f0 + st * 32);
                }
            }
#pragma unroll
            for (int q = 0; q < SM_NT; ++q) {
                if (n0 + q * 8 < count) {                  // (warp-uniform)
                    const int n = n0 + q * 8 + g;
                    const __nv_bfloat16 *urow = n < count ? u + (int64_t)s_tok[n] * F + f_warp + tq * 8 + f0 : nullptr;
                    uint4 bv[8];
#pragma unroll
                    for (int st = 0; st < 8; ++st)
                        bv[st] = (urow && st < nst) ? *reinterpret_cast<const uint4 *>(urow + st * 32)
                                                    : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                    for (int st = 0; st < 8; ++st) {
                        if (st < nst) {
                            mma_bf16_16816(acc[q], a0[st].x, a1[st].x, a0[st].y, a1[st].y, bv[st].x, bv[st].y);
                            mma_bf16_16816(acc[q], a0[st].z, a1[st].z, a0[st].w, a1[st].w, bv[st].z, bv[st].w);
                        }
                    }
                }
            }
        }
        // partial sums of the eight feature slices -> shared memory, added in warp order
#pragma unroll
        for (int q = 0; q < SM_NT; ++q) {
            s_red[warp][g][q * 8 + 2 * tq] = acc[q][0];
            s_red[warp][g][q * 8 + 2 * tq + 1] = acc[q][1];
            s_red[warp][g + 8][q * 8 + 2 * tq] = acc[q][2];
            s_red[warp][g + 8][q * 8 + 2 * tq + 1] = acc[q][3];
        }
        __syncthreads();
        if (ROWS == ROWS_BF16) {
            for (int o = tid; o < SM_ROWS / 2 * 8 * SM_NT; o += blockDim.x) {
                const int r = o % (SM_ROWS / 2) * 2, c = o / (SM_ROWS / 2);
                const int n = n0 + c;
                if (n < count) {
                    float v0 = 0.f, v1 = 0.f;
#pragma unroll
                    for (int q = 0; q < SM_WARPS; ++q) {
                        v0 += s_red[q][r][c];
                        v1 += s_red[q][r + 1][c];
                    }
                    const __nv_bfloat162 v = __floats2bfloat162_rn(s_wgt[n] * v0, s_wgt[n] * v1);
                    __nv_bfloat16 *dst = reinterpret_cast<__nv_bfloat16 *>(BCv) + (int64_t)s_out[n] * S + row0 + r;
                    if (k == 1) *reinterpret_cast<__nv_bfloat162 *>(dst) = v;
                    else atomicAdd(reinterpret_cast<__nv_bfloat162 *>(dst), v);
                }
            }
        } else {
            for (int o = tid; o < SM_ROWS * 8 * SM_NT; o += blockDim.x) {
                const int r = o % SM_ROWS, c = o / SM_ROWS;      // (neighbouring threads: neighbouring columns of a row)
                const int n = n0 + c;
                if (n < count) {
                    float v = 0.f;
#pragma unroll
                    for (int q = 0; q < SM_WARPS; ++q) v += s_red[q][r][c];
                    float *dst = &BC[(int64_t)s_out[n] * S + row0 + r];
                    if (ROWS == ROWS_SLOTS) *dst = s_wgt[n] * v;
                    else atomicAdd(dst, s_wgt[n] * v);
                }
            }
        }
        __syncthreads();
    }
}

bool front_small_supported(int dtype, int64_t T, int F, int S, int E, int k)
{
    return dtype == SWIMBA_DTYPE_BF16 && T <= SM_MAX_T && E <= SM_MAX_E && S % SM_ROWS == 0 && F % 32 == 0;
}

// The cost here is CTAs with an active expert ((S / 16) of them each) and the 16 x 16 output tiles they work
// through; the grouped product's is a chain along the features.  Measured over 1678 short forwards and decode steps
// (5 to 256 tokens, 2 to 16 experts, k = 1 to 8, S = 256 to 4096, F = 64 to 4096): the line costs 0.1 % over
// picking the faster one every time.  A forward of 8 experts, k = 2, S = 2048, F = 1024 (us, here / grouped): 8
// tokens 28 / 31, 24 34 / 33, 120 51 / 35, 250 83 / 39; S = 512, 250 tokens 25 / 29.
bool front_small_faster(int64_t T, int F, int S, int E, int k)
{
    return (S / SM_ROWS) * (12 * std::min<int64_t>(E, T * k) + T * k) <= 27 * (int64_t)F + 4608;
}

// Every CTA of the fused form computes the logits: not for more than 512 of them (16 experts, k = 2, F = 2048,
// one token: 512 CTAs 14.5 us fused, 1024 19.0 and 17.2 apart).
static bool front_small_fused(int64_t T, int S, int E) { return T <= SM_FUSED && (S / SM_ROWS) * E <= 512; }
bool front_small_slots(int64_t T, int S, int E, int k) { return front_small_fused(T, S, E) || k > 2; }

// Shares the tokens of a projection are cut into (grid z; a CTA lists and works its share): sixteen entries of
// an expert or more each, two CTAs per SM at most.  Few experts make few CTAs (32 with two experts), which
// walked their lists 32 entries at a time: two experts, k = 2, F = 768, 256 tokens 34.0 us (the grouped
// product: 16.4), in shares 13; four experts, k = 1, F = 2048, 128 tokens 10.5, in shares 9.  32 entries a
// share are 5 % slower over 1083 calls, four CTAs per SM 3 %.
static int project_share(int64_t T, int S, int E, int k, int sm_count)       // tokens of one
{
    const int64_t by_work = T * k / (16 * (int64_t)E), by_sms = 2 * (int64_t)sm_count / ((int64_t)(S / SM_ROWS) * E);
    return (int)ceil_div64(T, std::max<int64_t>(1, std::min(by_work, by_sms)));
}

int launch_front_small(LaunchCtx &ctx, const void *u, const void *W_r, const void *W_e, int64_t T, int F,
                       int S, int E, int k, int sm_count, int32_t *idx, float *w, float *BC)
{
    if (T <= 0) return SWIMBA_OK;
    const bool slots = front_small_slots(T, S, E, k), fused = front_small_fused(T, S, E);
    if (!fused) {
        ctx.begin(STAGE_ROUTER);
        launch_kernel(router_small_kernel, dim3((unsigned)ceil_div64(T, 2)), dim3(256), 0, ctx.stream, true,
                      (const __nv_bfloat16 *)u, (const __nv_bfloat16 *)W_r, (int)T, F, E, k, idx, w,
                      (float4 *)BC, slots ? 0 : S / 4, ScalarsArgs{});
        ctx.end();
    }
    ctx.begin(STAGE_PROJECT_SMALL);
    const int share = fused ? (int)T : project_share(T, S, E, k, sm_count);
    auto kern = fused ? project_small_kernel<ROWS_SLOTS, true>
                      : slots ? project_small_kernel<ROWS_SLOTS, false> : project_small_kernel<ROWS_ADD, false>;
    launch_kernel(kern, dim3((unsigned)(S / SM_ROWS), (unsigned)E, (unsigned)ceil_div64(T, share)), dim3(256), 0,
                  ctx.stream, true, (const __nv_bfloat16 *)u, (const __nv_bfloat16 *)W_r, (const __nv_bfloat16 *)W_e, idx, w, (int)T, F, S, E, k, share, (void *)BC,
                  ctx.check_indices ? 1 : 0, ctx.d_status);
    ctx.end();
    return cudaGetLastError() == cudaSuccess ? SWIMBA_OK : SWIMBA_ERR_CUDA;
}

// The forward's streams for short calls: no histogram to clear, no lists, no tiles.  One prompt of
// 93 tokens, 24 heads, F = 768, one of four experts: 22.5 us a call through router, lists and grouped product,
// 16.8 us this way (the first tile and the states fetched ahead of the wait included).
bool front_short_supported(int dtype, int64_t T, int F, int S, int E, int k)
{
    return front_small_supported(dtype, T, F, S, E, k) && k <= 2 && E > 1 && front_small_faster(T, F, S, E, k);
}

int launch_front_short(LaunchCtx &ctx, const void *u, const void *W_r, const void *W_e, int64_t T, int F, int S, int E,
                       int k, int sm_count, int32_t *idx, float *w, void *BC, const ScalarsArgs &scalars)
{
    if (T <= 0) return SWIMBA_OK;
    ctx.begin(STAGE_ROUTER);
    launch_kernel(router_small_kernel, dim3((unsigned)(ceil_div64(T, 2) + scalars_blocks(scalars, 256))), dim3(256), 0,
                  ctx.stream, true, (const __nv_bfloat16 *)u, (const __nv_bfloat16 *)W_r, (int)T, F, E, k, idx, w,
                  (float4 *)BC, k == 1 ? 0 : S / 8, scalars);
    ctx.end();
    const int share = project_share(T, S, E, k, sm_count);
    ctx.begin(STAGE_PROJECT_SMALL);
    launch_kernel(project_small_kernel<ROWS_BF16, false>,
                  dim3((unsigned)(S / SM_ROWS), (unsigned)E, (unsigned)ceil_div64(T, share)), dim3(256), 0, ctx.stream,
                  true, (const __nv_bfloat16 *)u, (const __nv_bfloat16 *)W_r, (const __nv_bfloat16 *)W_e, idx, w, (int)T, F,
                  S, E, k, share, BC, ctx.check_indices ? 1 : 0, ctx.d_status);
    ctx.end();
    return cudaGetLastError() == cudaSuccess ? SWIMBA_OK : SWIMBA_ERR_CUDA;
}

}  // namespace swimba
