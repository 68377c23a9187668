// The recurrence on the CUDA cores (selective-SSM equation with the channelwise convention; Theorem 1):
// the chunked fp32 path of the forward, packed sequences of a few tokens stepped token by token, and K4,
// the one-token decode update.
#include <algorithm>
#include <type_traits>

#include "internal.h"
#include "tc05.cuh"

namespace swimba {

// Chunked evaluation on the CUDA cores (fp32 arithmetic throughout): the fp32 path of the forward and
// the bf16 shapes that the tensor-core kernel does not take.  A cluster of up to eight CTAs owns one
// (sequence, head); every CTA takes a run of CK_Q consecutive tokens, all CTAs at once:
//   S_c[n,p] = sum_s w_s Btilde_s[n] x_s[p],  w_s = Delta_s exp(l_last - l_s)     local end state
//   G[i,s]   = (Ctilde_i . Btilde_s) Delta_s exp(l_i - l_s)  for s <= i, else 0
// then the local end states and decays are exchanged through distributed shared memory,
//   H <- decay_r H + S_r  over the runs in front of this one,
// and  y_i = exp(l_i) Ctilde_i^T H + sum_s G[i,s] x_s + D x_i.  Longer sequences repeat this with the
// carried state (every CTA keeps its own copy).  All exponents are <= 0 and are formed from cumulative
// sums in fp64, so a product of decays is rounded once.
// With few heads, the latency of a handful of dependent phases (load, G and S, exchange, y) bounds it; with as
// many as fill the SMs, shared memory, and every further CTA of a cluster costs an exchange of whole states.  So
// a cluster is no larger than lets all of them run at once, and a cluster of one adds its run to the state in
// place.  Up to a CTA per SM they may have 128 registers each, 64 (four CTAs per SM) beyond.  A forward in fp32,
// a step per token / always eight CTAs / this way: 8 heads of 256 tokens (P = 64, N = 16) 184 / 25 / 23 us, 512
// heads of 1024 (P = 64, N = 128) 3.6 / 4.6 / 2.8 ms, 512 heads of 1024 (P = 64, N = 256) 5.8 / 12.1 / 4.7 ms, 128
// heads of 1000 (P = 64, N = 16) 697 / 157 / 130 us.  Over 430 shapes 0.77 of the faster of the other two, none
// slower.
constexpr int CK_Q = 32;          // tokens per CTA and round
constexpr int CK_THREADS = 256;
constexpr int CK_MAX_CLUSTER = 8;
constexpr int CK_FILL = 4;        // CTAs per SM (fewer where shared memory holds fewer)

namespace {
__device__ __forceinline__ float4 ck_load4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ float4 ck_load4(const __nv_bfloat16 *p)
{
    const uint2 raw = *reinterpret_cast<const uint2 *>(p);
    return make_float4(__uint_as_float(raw.x << 16), __uint_as_float(raw.x & 0xffff0000u),
                       __uint_as_float(raw.y << 16), __uint_as_float(raw.y & 0xffff0000u));
}
__device__ __forceinline__ void ck_store4(float *p, const float (&v)[4])
{
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void ck_store4(__nv_bfloat16 *p, const float (&v)[4])
{
    *reinterpret_cast<uint2 *>(p) = make_uint2(tc::pack_bf16x2(v[0], v[1]), tc::pack_bf16x2(v[2], v[3]));
}
__device__ __forceinline__ uint32_t cluster_addr(uint32_t local, uint32_t rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}
__device__ __forceinline__ float4 cluster_load4(uint32_t addr)
{
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ float cluster_load(uint32_t addr)
{
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void fma4(float4 &acc, float a, const float4 &v)
{
    acc.x = fmaf(a, v.x, acc.x);
    acc.y = fmaf(a, v.y, acc.y);
    acc.z = fmaf(a, v.z, acc.z);
    acc.w = fmaf(a, v.w, acc.w);
}

// Offsets in floats; rows padded to whole float4s.  One CTA adds its run to the state in place and needs no S.
struct ChunkSmem {
    int B, C, x, G, S, H, total;
};
__host__ __device__ inline ChunkSmem chunk_smem(int P, int N, int ncta)
{
    const int Pp = (P + 3) & ~3;
    ChunkSmem m;
    int off = 0;
    m.B = off; off += CK_Q * (N + 4);
    m.C = off; off += CK_Q * (N + 4);
    m.x = off; off += CK_Q * Pp;
    m.G = off; off += CK_Q * (CK_Q + 4);
    m.H = off; off += N * Pp;
    m.S = off; off += ncta > 1 ? N * Pp : 0;
    m.total = off;
    return m;
}
}  // namespace

// MULTI: a cluster of ncta > 1 CTAs.  PER_SM: CTAs that share an SM, and with it the registers.
template <typename T, bool MULTI, int PER_SM>
__global__ void __launch_bounds__(CK_THREADS, PER_SM)
ssd_chunk_kernel(const T *__restrict__ x, const T *__restrict__ BC, const float *__restrict__ dt,
                 const float *__restrict__ A, const float *__restrict__ dt_bias, const float *__restrict__ D,
                 const float *__restrict__ h0, int L, int H, int P, int N, int G, int cluster, T *__restrict__ y,
                 float *__restrict__ h_final)
{
    const int ncta = MULTI ? cluster : 1;
    extern __shared__ __align__(16) float csm[];
    __shared__ double s_l[CK_Q];
    __shared__ float s_delta[CK_Q], s_w[CK_Q], s_e[CK_Q];
    __shared__ float s_decay;
    const ChunkSmem m = chunk_smem(P, N, ncta);
    float *sB = csm + m.B, *sC = csm + m.C, *sx = csm + m.x, *sG = csm + m.G, *sS = csm + m.S, *sH = csm + m.H;
    const int Pp = (P + 3) & ~3, pq = Pp >> 2, Nr = N + 4, Gr = CK_Q + 4;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = (int)(blockIdx.x % ncta);
    const int64_t bh = blockIdx.x / ncta;
    const int b = (int)(bh / H), h = (int)(bh % H);
    const int g = h / (H / G), S = 2 * G * N;
    const bool vec = (P & 3) == 0;
    grid_dep_launch();
    grid_dep_wait();
    const double Ah = (double)A[h];
    const float bias = dt_bias[h], Dh = D ? D[h] : 0.f;
    const float *h0p = h0 ? h0 + bh * P * N : nullptr;
    // A warp's share of a state: 8 state indexes x 16 channels, whole 32-byte sectors of [p][n] in global memory
    // and two-way bank conflicts on rows [n][p] (with the state index along all lanes: 32-way; 16 tokens of 512
    // heads, P = 32, N = 128: 75 -> 50 us a call)
    auto state_tiles = [&](auto f) {
        const int nct = (pq + 3) >> 2;
        for (int i = warp; i < (N >> 3) * nct; i += CK_THREADS / 32) {
            const int n = (i / nct) * 8 + (lane >> 3) * 2 + (lane & 1), p = (i % nct) * 16 + ((lane >> 1) & 3) * 4;
            if (p < Pp) f(n, p);
        }
    };
    bool has_state = h0p != nullptr;         // (zero otherwise: no product with it)
    const int nrounds = ceil_div(L, CK_Q * ncta);
    for (int rd = 0; rd < nrounds; ++rd) {
        const int t0 = (rd * ncta + rank) * CK_Q;
        const int nt = max(0, min(CK_Q, L - t0));
        const int64_t tok0 = (int64_t)b * L + t0;
        // ---- this run's rows; rows past the end are zero
        for (int i = tid; i < CK_Q * (N >> 2); i += CK_THREADS) {
            const int tt = i / (N >> 2), c = (i - tt * (N >> 2)) * 4;
            float4 vb = make_float4(0.f, 0.f, 0.f, 0.f), vc = vb;
            if (tt < nt) {
                const T *row = BC + (tok0 + tt) * S + g * N + c;
                vb = ck_load4(row);
                vc = ck_load4(row + G * N);
            }
            *reinterpret_cast<float4 *>(sB + tt * Nr + c) = vb;
            *reinterpret_cast<float4 *>(sC + tt * Nr + c) = vc;
        }
#pragma unroll 2
        for (int i = tid; i < CK_Q * pq; i += CK_THREADS) {
            const int tt = i / pq, c = (i - tt * pq) * 4;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (tt < nt) {
                const T *row = x + ((tok0 + tt) * H + h) * P + c;
                if (vec) {
                    v = ck_load4(row);
                } else {
                    v.x = to_f32<T>(row[0]);
                    if (c + 1 < P) v.y = to_f32<T>(row[1]);
                    if (c + 2 < P) v.z = to_f32<T>(row[2]);
                    if (c + 3 < P) v.w = to_f32<T>(row[3]);
                }
            }
            *reinterpret_cast<float4 *>(sx + tt * Pp + c) = v;
        }
        if (warp == 0) {
            const float d = lane < nt ? softplus_f((dt ? dt[(tok0 + lane) * H + h] : 0.f) + bias) : 0.f;
            double l = (double)d * Ah;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const double nb = __shfl_up_sync(0xffffffffu, l, o);
                if (lane >= o) l += nb;
            }
            const double l_last = __shfl_sync(0xffffffffu, l, 31);
            s_l[lane] = l;
            s_delta[lane] = d;
            s_w[lane] = d * expf((float)(l_last - l));
            s_e[lane] = expf((float)l);
            if (lane == 31) s_decay = expf((float)l);
        }
        if (rd == 0 && has_state) {          // the given state, [p][n] -> [n][p]
            state_tiles([&](int n, int p) {
                float v[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) v[q] = p + q < P ? h0p[(int64_t)(p + q) * N + n] : 0.f;
                *reinterpret_cast<float4 *>(sH + n * Pp + p) = make_float4(v[0], v[1], v[2], v[3]);
            });
        } else if (rd == 0) {
            for (int i = tid; i < N * pq; i += CK_THREADS) reinterpret_cast<float4 *>(sH)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        __syncthreads();
        // ---- local end state, two state rows x four channels per thread and step: to S, or (a cluster of one)
        // added to the decayed state
        const int nt8 = (nt + 7) & ~7;
        auto end_state = [&]() {
            for (int i = tid; i < (N >> 1) * pq; i += CK_THREADS) {
                const int nn = (i / pq) * 2, c = (i % pq) * 4;
                float4 a0 = make_float4(0.f, 0.f, 0.f, 0.f), a1 = a0;
#pragma unroll 8
                for (int s = 0; s < nt8; ++s) {
                    const float w = s_w[s];
                    const float2 bv = *reinterpret_cast<const float2 *>(sB + s * Nr + nn);
                    const float4 xv = *reinterpret_cast<const float4 *>(sx + s * Pp + c);
                    fma4(a0, w * bv.x, xv);
                    fma4(a1, w * bv.y, xv);
                }
                float *dst = MULTI ? sS : sH;
                if (!MULTI) {
                    fma4(a0, s_decay, *reinterpret_cast<const float4 *>(sH + nn * Pp + c));
                    fma4(a1, s_decay, *reinterpret_cast<const float4 *>(sH + (nn + 1) * Pp + c));
                }
                *reinterpret_cast<float4 *>(dst + nn * Pp + c) = a0;
                *reinterpret_cast<float4 *>(dst + (nn + 1) * Pp + c) = a1;
            }
        };
        if (MULTI) end_state();
        // ---- G: warp = rows i, lane = column s
        for (int i = warp; i < nt8; i += CK_THREADS / 32) {
            float v = 0.f;
            if (lane <= i) {
                const float4 *cr = reinterpret_cast<const float4 *>(sC + i * Nr);
                const float4 *br = reinterpret_cast<const float4 *>(sB + lane * Nr);
                float4 d4 = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
                for (int c = 0; c < (N >> 2); ++c) {
                    const float4 cv = cr[c], bv = br[c];
                    d4.x = fmaf(cv.x, bv.x, d4.x);
                    d4.y = fmaf(cv.y, bv.y, d4.y);
                    d4.z = fmaf(cv.z, bv.z, d4.z);
                    d4.w = fmaf(cv.w, bv.w, d4.w);
                }
                v = ((d4.x + d4.y) + (d4.z + d4.w)) * s_delta[lane] * expf((float)(s_l[i] - s_l[lane]));
            }
            sG[i * Gr + lane] = v;
        }
        if (MULTI) tc::cluster_sync();
        else __syncthreads();
        // ---- state entering this run: the runs in front of it, in order
        const uint32_t s_addr = tc::smem_u32(sS), d_addr = tc::smem_u32(&s_decay);
        for (int r = 0; r < rank; ++r) {
            const float dr = cluster_load(cluster_addr(d_addr, r));
            const uint32_t ra = cluster_addr(s_addr, r);
#pragma unroll 4
            for (int i = tid; i < N * pq; i += CK_THREADS) {
                float4 cur = reinterpret_cast<float4 *>(sH)[i];
                const float4 v = cluster_load4(ra + i * 16);
                cur.x = fmaf(dr, cur.x, v.x);
                cur.y = fmaf(dr, cur.y, v.y);
                cur.z = fmaf(dr, cur.z, v.z);
                cur.w = fmaf(dr, cur.w, v.w);
                reinterpret_cast<float4 *>(sH)[i] = cur;
            }
        }
        __syncthreads();
        // ---- y: two tokens x four channels per thread and step
        has_state |= rank > 0;
        for (int i = tid; i < (CK_Q / 2) * pq; i += CK_THREADS) {
            const int i0 = (i / pq) * 2, c = (i % pq) * 4;
            if (i0 >= nt) continue;
            float4 a0 = make_float4(0.f, 0.f, 0.f, 0.f), a1 = a0;
#pragma unroll 2
            for (int n = 0; n < (has_state ? N : 0); n += 4) {
                const float4 c0 = *reinterpret_cast<const float4 *>(sC + i0 * Nr + n);
                const float4 c1 = *reinterpret_cast<const float4 *>(sC + (i0 + 1) * Nr + n);
                const float cv0[4] = {c0.x, c0.y, c0.z, c0.w}, cv1[4] = {c1.x, c1.y, c1.z, c1.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float4 hv = *reinterpret_cast<const float4 *>(sH + (n + q) * Pp + c);
                    fma4(a0, cv0[q], hv);
                    fma4(a1, cv1[q], hv);
                }
            }
            const float e0 = s_e[i0], e1 = s_e[i0 + 1];
            a0.x *= e0; a0.y *= e0; a0.z *= e0; a0.w *= e0;
            a1.x *= e1; a1.y *= e1; a1.z *= e1; a1.w *= e1;
            // columns up to the diagonal and none behind it (G's zeros there would meet later tokens' infinities)
            int s = 0;
            for (; s + 4 <= i0; s += 4) {
                const float4 g0 = *reinterpret_cast<const float4 *>(sG + i0 * Gr + s);
                const float4 g1 = *reinterpret_cast<const float4 *>(sG + (i0 + 1) * Gr + s);
                const float gv0[4] = {g0.x, g0.y, g0.z, g0.w}, gv1[4] = {g1.x, g1.y, g1.z, g1.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float4 xv = *reinterpret_cast<const float4 *>(sx + (s + q) * Pp + c);
                    fma4(a0, gv0[q], xv);
                    fma4(a1, gv1[q], xv);
                }
            }
            if (s < i0) {
                const float2 g0 = *reinterpret_cast<const float2 *>(sG + i0 * Gr + s);
                const float2 g1 = *reinterpret_cast<const float2 *>(sG + (i0 + 1) * Gr + s);
                const float4 x0 = *reinterpret_cast<const float4 *>(sx + s * Pp + c);
                const float4 x1 = *reinterpret_cast<const float4 *>(sx + (s + 1) * Pp + c);
                fma4(a0, g0.x, x0);
                fma4(a1, g1.x, x0);
                fma4(a0, g0.y, x1);
                fma4(a1, g1.y, x1);
            }
            const float4 xi0 = *reinterpret_cast<const float4 *>(sx + i0 * Pp + c);
            const float4 xi1 = *reinterpret_cast<const float4 *>(sx + (i0 + 1) * Pp + c);
            const float2 gd = *reinterpret_cast<const float2 *>(sG + (i0 + 1) * Gr + i0);
            fma4(a0, sG[i0 * Gr + i0], xi0);
            fma4(a1, gd.x, xi0);
            fma4(a1, gd.y, xi1);
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                if (i0 + r >= nt) break;
                float4 v = r ? a1 : a0;
                fma4(v, Dh, r ? xi1 : xi0);
                T *dst = y + ((tok0 + i0 + r) * H + h) * P + c;
                const float o[4] = {v.x, v.y, v.z, v.w};
                if (vec) {
                    ck_store4(dst, o);
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (c + q < P) dst[q] = from_f32<T>(o[q]);
                }
            }
        }
        // ---- the state after this round (carried on, or the call's end state)
        if (rd + 1 < nrounds || (h_final && rank == 0)) {
            has_state = true;
            __syncthreads();                                 // (y has read the entry state)
            if (!MULTI) end_state();
            else for (int r = rank; r < ncta; ++r) {
                const float dr = cluster_load(cluster_addr(d_addr, r));
                const uint32_t ra = cluster_addr(s_addr, r);
#pragma unroll 4
                for (int i = tid; i < N * pq; i += CK_THREADS) {
                    float4 cur = reinterpret_cast<float4 *>(sH)[i];
                    const float4 v = cluster_load4(ra + i * 16);
                    cur.x = fmaf(dr, cur.x, v.x);
                    cur.y = fmaf(dr, cur.y, v.y);
                    cur.z = fmaf(dr, cur.z, v.z);
                    cur.w = fmaf(dr, cur.w, v.w);
                    reinterpret_cast<float4 *>(sH)[i] = cur;
                }
            }
        }
        // the local end states have been read by everyone (and no CTA leaves while it is being read)
        if (MULTI) tc::cluster_sync();
        else __syncthreads();
    }
    if (h_final && rank == 0) {
        float *dst = h_final + bh * P * N;
        state_tiles([&](int n, int p) {
            const float4 h4 = *reinterpret_cast<const float4 *>(sH + n * Pp + p);
            const float v[4] = {h4.x, h4.y, h4.z, h4.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) if (p + q < P) dst[(int64_t)(p + q) * N + n] = v[q];
        });
    }
}

template <typename T>
static int launch_chunk_t(LaunchCtx &ctx, const void *x, const void *BC, const float *dt, const float *A,
                          const float *dt_bias, const float *D, const float *h0, int B, int L, int H, int P, int N,
                          int G, int sm_count, void *y, float *h_final)
{
    // as many CTAs per (sequence, head) as it has runs of CK_Q tokens, a power of two up to eight (the
    // portable cluster size), as long as they all run at once
    const size_t per_cta = (size_t)chunk_smem(P, N, 2).total * sizeof(float) + 2048;
    const int64_t room = (int64_t)sm_count * std::min<int64_t>(CK_FILL, std::max<int64_t>(1, 228 * 1024 / per_cta));
    int ncta = 1;
    while (ncta < CK_MAX_CLUSTER && ncta * CK_Q < L && 2 * ncta * (int64_t)B * H <= room) ncta <<= 1;
    const size_t smem = (size_t)chunk_smem(P, N, ncta).total * sizeof(float);
    const bool few = (int64_t)B * H * ncta <= (ncta > 1 ? 1 : 2) * (int64_t)sm_count;
    auto kern = ncta > 1 ? (few ? ssd_chunk_kernel<T, true, 2> : ssd_chunk_kernel<T, true, 4>)
                         : (few ? ssd_chunk_kernel<T, false, 2> : ssd_chunk_kernel<T, false, 4>);
    if (smem > 40 * 1024 && !ensure_dynamic_smem((const void *)kern, smem)) return SWIMBA_ERR_CUDA;
    ctx.begin(STAGE_SSD_SEQUENTIAL);
    launch_kernel_cluster(kern, dim3((unsigned)((int64_t)B * H * ncta)), dim3(CK_THREADS), smem, ctx.stream, true,
                          (unsigned)ncta, (const T *)x, (const T *)BC, dt, A, dt_bias, D, h0, L, H, P, N, G, ncta,
                          (T *)y, h_final);
    ctx.end();
    return cudaGetLastError() == cudaSuccess ? SWIMBA_OK : SWIMBA_ERR_CUDA;
}

int launch_ssd_sequential(LaunchCtx &ctx, int dtype, const void *x, const void *BC, const float *dt, const float *A,
                          const float *dt_bias, const float *D, const float *h0, int B, int L, int H, int P, int N,
                          int G, int sm_count, void *y, float *h_final)
{
    if (B <= 0 || L <= 0) return SWIMBA_OK;
    if (dtype == SWIMBA_DTYPE_FP32)
        return launch_chunk_t<float>(ctx, x, BC, dt, A, dt_bias, D, h0, B, L, H, P, N, G, sm_count, y, h_final);
    return launch_chunk_t<__nv_bfloat16>(ctx, x, BC, dt, A, dt_bias, D, h0, B, L, H, P, N, G, sm_count, y, h_final);
}

// ------------------------------------------------------------------------------------------
// K4: decode.  The state [B,H,P,N] fp32 is read and written exactly once: the kernel is a pure
// HBM stream (128 sequences of 64 heads, 537 MB in and out: 92 us, 5.8 TB/s).  One warp owns ROWS consecutive channels p of one (b,h); a row is N floats read
// as float4 per lane, all ROWS loads are issued before any use.  (A ring of 4 KB pieces per warp in shared
// memory, filled and emptied by bulk copies, took 95 us with neighbouring warps on neighbouring pieces and
// 103 us with a contiguous run per warp; asking L2 for the first 16 to 80 MB of the states under the front
// end cost 3 to 8 us: the previous step's last writes still occupy HBM then.)
// ------------------------------------------------------------------------------------------
constexpr int DEC_ROWS = 8;

__device__ __forceinline__ float4 load_bc4(const float *p, int v)
{
    return reinterpret_cast<const float4 *>(p)[v];
}
__device__ __forceinline__ float4 load_bc4(const __nv_bfloat16 *p, int v)
{
    const uint2 raw = reinterpret_cast<const uint2 *>(p)[v];
    return make_float4(__uint_as_float(raw.x << 16), __uint_as_float(raw.x & 0xffff0000u),
                       __uint_as_float(raw.y << 16), __uint_as_float(raw.y & 0xffff0000u));
}

// A sequence's mixed streams are bc_slots rows of BC: MULTI, to be summed in order here; else the first one.
// EARLY: small launches with rows of at most 128 entries, in which every warp has one piece of work and
// its state rows are fetched before the dependency wait, under the projection (large ones run out of
// registers that way: 92 -> 139 us at 128 sequences of 64 heads).
template <typename T, typename TBC, bool MULTI, bool EARLY>
__global__ void __launch_bounds__(256, 2)
decode_update_kernel(const T *__restrict__ x, const TBC *__restrict__ BC,
                     const float *__restrict__ dt, const float *__restrict__ A,
                     const float *__restrict__ dt_bias, const float *__restrict__ D,
                     float *__restrict__ state, int B, int H, int P, int N, int G, int bc_slots,
                     T *__restrict__ y)
{
    const int lane = threadIdx.x & 31;
    const int S = 2 * G * N;
    const int pgroups = ceil_div(P, DEC_ROWS);
    const int64_t nwork = (int64_t)B * H * pgroups;
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    const int nv = N >> 2;   // groups of 4 state entries per row
    int64_t wk = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    float4 s[DEC_ROWS];
    if (EARLY && wk < nwork && lane < nv) {
        // (the kernel in front lets this one in only behind its own wait: the previous step's update, the
        // last writer of the states, has completed; the loads go past L1, which may hold older lines)
        const int pg = (int)(wk % pgroups);
#pragma unroll
        for (int r = 0; r < DEC_ROWS; ++r)
            if (pg * DEC_ROWS + r < P)
                s[r] = __ldcg(reinterpret_cast<const float4 *>(state + ((wk / pgroups) * P + pg * DEC_ROWS + r) * N) + lane);
    }
    grid_dep_wait();      // the mixed streams come from the projection kernel
    for (; wk < nwork; wk += nwarps) {
        const int pg = (int)(wk % pgroups);
        const int64_t bh = wk / pgroups;
        const int h = (int)(bh % H), b = (int)(bh / H);
        const int g = h / (H / G);
        const float delta = softplus_f((dt ? dt[bh] : 0.f) + dt_bias[h]);
        const float a = expf(delta * A[h]);
        const float Dh = D ? D[h] : 0.f;
        const TBC *Bp = BC + (int64_t)b * bc_slots * S + g * N;
        const TBC *Cp = Bp + G * N;
        float xv[DEC_ROWS], acc[DEC_ROWS];
#pragma unroll
        for (int r = 0; r < DEC_ROWS; ++r) {
            const int p = pg * DEC_ROWS + r;
            xv[r] = (p < P) ? to_f32<T>(x[bh * P + p]) : 0.f;
            acc[r] = 0.f;
        }
        for (int v = lane; v < nv; v += 32) {
            if (!EARLY) {
#pragma unroll
                for (int r = 0; r < DEC_ROWS; ++r) {
                    const int p = pg * DEC_ROWS + r;
                    if (p < P)
                        s[r] = __ldcs(reinterpret_cast<const float4 *>(state + (bh * P + p) * N) + v);
                }
            }
            float4 bb = load_bc4(Bp, v), cc = load_bc4(Cp, v);
            if (MULTI) {
#pragma unroll 1
                for (int j = 1; j < bc_slots; ++j) {
                    const float4 bj = load_bc4(Bp + (int64_t)j * S, v), cj = load_bc4(Cp + (int64_t)j * S, v);
                    bb.x += bj.x; bb.y += bj.y; bb.z += bj.z; bb.w += bj.w;
                    cc.x += cj.x; cc.y += cj.y; cc.z += cj.z; cc.w += cj.w;
                }
            }
#pragma unroll
            for (int r = 0; r < DEC_ROWS; ++r) {
                const int p = pg * DEC_ROWS + r;
                if (p < P) {
                    const float dx = delta * xv[r];
                    s[r].x = fmaf(a, s[r].x, dx * bb.x);
                    s[r].y = fmaf(a, s[r].y, dx * bb.y);
                    s[r].z = fmaf(a, s[r].z, dx * bb.z);
                    s[r].w = fmaf(a, s[r].w, dx * bb.w);
                    acc[r] = fmaf(cc.x, s[r].x, acc[r]);
                    acc[r] = fmaf(cc.y, s[r].y, acc[r]);
                    acc[r] = fmaf(cc.z, s[r].z, acc[r]);
                    acc[r] = fmaf(cc.w, s[r].w, acc[r]);
                    __stcs(reinterpret_cast<float4 *>(state + (bh * P + p) * N) + v, s[r]);
                }
            }
            if (EARLY) break;
        }
#pragma unroll
        for (int r = 0; r < DEC_ROWS; ++r) {
            const float tot = warp_sum(acc[r]);
            const int p = pg * DEC_ROWS + r;
            if (lane == r && p < P) y[bh * P + p] = from_f32<T>(tot + Dh * xv[r]);
        }
        if (EARLY) break;
    }
}

// Decode tokens riding in a packed prefill batch: the same stream of states for the listed sequences,
// out of place (h0 -> h_final), with up to four tokens applied while the rows are in registers.  Bound by
// HBM like the decode update: 57 one-token sequences of 64 heads move 239 MB of states; one block per
// (sequence, head) that staged its tokens in shared memory took 72 us, a warp per eight rows 43 us (5.6 TB/s).
__global__ void __launch_bounds__(256)
step_sequences_kernel(const __nv_bfloat16 *__restrict__ x, const __nv_bfloat16 *__restrict__ BC,
                      const float *__restrict__ dt, const float *__restrict__ A, const float *__restrict__ dt_bias,
                      const float *__restrict__ D, const float *__restrict__ h0, const int4 *__restrict__ seq_tab,
                      int n, int H, int G, __nv_bfloat16 *__restrict__ y, float *__restrict__ h_final)
{
    constexpr int P = 64, N = 128, PG = P / DEC_ROWS;
    grid_dep_launch();
    const int lane = threadIdx.x & 31, S = 2 * G * N;
    const int64_t nwork = (int64_t)n * H * PG, nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    grid_dep_wait();      // the table, the mixed streams
    for (int64_t wk = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); wk < nwork; wk += nwarps) {
        const int pg = (int)(wk % PG), h = (int)((wk / PG) % H);
        const int4 e = seq_tab[wk / ((int64_t)PG * H)];
        const int g = h / (H / G);
        const int64_t row0 = ((int64_t)e.z * H + h) * P + pg * DEC_ROWS;
        float4 s[DEC_ROWS];
#pragma unroll
        for (int r = 0; r < DEC_ROWS; ++r)
            s[r] = h0 ? __ldcs(reinterpret_cast<const float4 *>(h0 + (row0 + r) * N) + lane)
                      : make_float4(0.f, 0.f, 0.f, 0.f);
        const float Ah = A[h], bias = dt_bias[h], Dh = D ? D[h] : 0.f;
        for (int tt = 0; tt < e.y; ++tt) {
            const int64_t tok = e.x + tt;
            const float delta = softplus_f((dt ? dt[tok * H + h] : 0.f) + bias);
            const float a = expf(delta * Ah);
            const float4 bb = load_bc4(BC + tok * S + g * N, lane), cc = load_bc4(BC + tok * S + (G + g) * N, lane);
            float xv[DEC_ROWS];
            load8(x + (tok * H + h) * P + pg * DEC_ROWS, xv);
            float mine = 0.f;
#pragma unroll
            for (int r = 0; r < DEC_ROWS; ++r) {
                const float dx = delta * xv[r];
                s[r].x = fmaf(a, s[r].x, dx * bb.x);
                s[r].y = fmaf(a, s[r].y, dx * bb.y);
                s[r].z = fmaf(a, s[r].z, dx * bb.z);
                s[r].w = fmaf(a, s[r].w, dx * bb.w);
                float acc = cc.x * s[r].x;
                acc = fmaf(cc.y, s[r].y, acc);
                acc = fmaf(cc.z, s[r].z, acc);
                acc = fmaf(cc.w, s[r].w, acc);
                const float tot = warp_sum(acc) + Dh * xv[r];
                if (lane == r) mine = tot;
            }
            if (lane < DEC_ROWS) y[(tok * H + h) * P + pg * DEC_ROWS + lane] = from_f32<__nv_bfloat16>(mine);
        }
        if (h_final) {
#pragma unroll
            for (int r = 0; r < DEC_ROWS; ++r) __stcs(reinterpret_cast<float4 *>(h_final + (row0 + r) * N) + lane, s[r]);
        }
    }
}

int launch_step_sequences(LaunchCtx &ctx, const void *x, const void *BC, const float *dt, const float *A,
                          const float *dt_bias, const float *D, const float *h0, const int4 *seq_tab, int n, int H,
                          int G, void *y, float *h_final)
{
    if (n <= 0) return SWIMBA_OK;
    const int64_t blocks = ceil_div64((int64_t)n * H * (64 / DEC_ROWS), 8);
    ctx.begin(STAGE_SSD_SEQUENTIAL);
    launch_kernel(step_sequences_kernel, dim3((unsigned)blocks), dim3(256), 0, ctx.stream, true,
                  (const __nv_bfloat16 *)x, (const __nv_bfloat16 *)BC, dt, A, dt_bias, D, h0, seq_tab, n, H, G,
                  (__nv_bfloat16 *)y, h_final);
    ctx.end();
    return cudaGetLastError() == cudaSuccess ? SWIMBA_OK : SWIMBA_ERR_CUDA;
}

// The first row of every sequence's k rows becomes their sum, in order.
__global__ void __launch_bounds__(256)
sum_slots_kernel(float *__restrict__ BC, int64_t T, int S, int k)
{
    grid_dep_launch();
    grid_dep_wait();
    const int vpr = S >> 2;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= T * vpr) return;
    float4 *p = reinterpret_cast<float4 *>(BC) + (i / vpr) * k * vpr + i % vpr;
    float4 sum = p[0];
    for (int j = 1; j < k; ++j) {
        const float4 v = p[(int64_t)j * vpr];
        sum.x += v.x; sum.y += v.y; sum.z += v.z; sum.w += v.w;
    }
    p[0] = sum;
}

template <typename T, typename TBC>
static int launch_decode_t(LaunchCtx &ctx, const void *x, void *BC, const float *dt, const float *A,
                           const float *dt_bias, const float *D, float *state, int B, int H, int P, int N, int G,
                           int bc_slots, bool early, int sm_count, void *y)
{
    const int64_t nwork = (int64_t)B * H * ceil_div(P, DEC_ROWS);
    const int warps = 8;
    int64_t blocks = ceil_div64(nwork, warps);
    const int64_t cap = (int64_t)sm_count * 8;
    // one piece of work per warp, and all of them resident (two blocks of 256 threads per SM)
    early = early && N <= 128 && blocks <= 2 * (int64_t)sm_count;
    if (blocks > cap) blocks = cap;
    // Every warp of a sequence would sum its rows again, H ceil(P / 8) of them.  Where that reads more than a
    // launch costs (20 MB out of L2; 5 or 80 MB in the rule are 1 and 2 % slower over 435 calls), a kernel of
    // its own sums them once: 256 sequences of 64 heads, 16 experts, k = 8, F = 1024 283 us, now 205.
    bool multi = bc_slots > 1;
    if constexpr (std::is_same<TBC, float>::value) {
        if (multi && nwork * (bc_slots - 1) * 2 * N * (int64_t)sizeof(float) > 20 << 20) {
            const int S = 2 * G * N;
            ctx.begin(STAGE_SLOT_SUM);
            launch_kernel(sum_slots_kernel, dim3((unsigned)ceil_div64((int64_t)B * (S / 4), 256)), dim3(256), 0, ctx.stream,
                          true, (float *)BC, (int64_t)B, S, bc_slots);
            ctx.end();
            multi = false;
        }
    }
    auto kern = !multi ? (early ? decode_update_kernel<T, TBC, false, true> : decode_update_kernel<T, TBC, false, false>)
                              : (early ? decode_update_kernel<T, TBC, true, true> : decode_update_kernel<T, TBC, true, false>);
    ctx.begin(STAGE_DECODE_UPDATE);
    launch_kernel(kern, dim3((unsigned)blocks), dim3(warps * 32), 0, ctx.stream, true, (const T *)x, (const TBC *)BC, dt, A, dt_bias, D, state, B, H, P, N,
                  G, bc_slots, (T *)y);
    ctx.end();
    return cudaGetLastError() == cudaSuccess ? SWIMBA_OK : SWIMBA_ERR_CUDA;
}

int launch_decode_update(LaunchCtx &ctx, int dtype, const void *x, void *BC, bool bc_fp32, int bc_slots, bool early,
                         const float *dt, const float *A, const float *dt_bias, const float *D,
                         float *state, int B, int H, int P, int N, int G, int sm_count, void *y)
{
    if (B <= 0) return SWIMBA_OK;
    if (dtype == SWIMBA_DTYPE_FP32)
        return launch_decode_t<float, float>(ctx, x, BC, dt, A, dt_bias, D, state, B, H, P, N, G, bc_slots, early, sm_count, y);
    if (bc_fp32)
        return launch_decode_t<__nv_bfloat16, float>(ctx, x, BC, dt, A, dt_bias, D, state, B, H, P, N, G, bc_slots, early,
                                                     sm_count, y);
    return launch_decode_t<__nv_bfloat16, __nv_bfloat16>(ctx, x, BC, dt, A, dt_bias, D, state, B, H, P, N, G, bc_slots, early,
                                                         sm_count, y);
}

}  // namespace swimba
