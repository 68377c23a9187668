// The rest of the block around the mixer (Section "Swimba layer": the in-projection becomes a
// mixture of experts and the rest of the Mamba-2 layer is kept unchanged): causal depthwise
// convolution + SiLU on the [x | B | C] stream, the gated RMS norm rmsnorm(y * silu(z)) * weight,
// and the conversion of the step-size columns of the shared in-projection to fp32.  All three are
// streaming kernels (every element read and written once).
#include "internal.h"

namespace swimba {

namespace {
constexpr int CV_K = 4;        // widest convolution window
constexpr int CV_CH = 4;       // channels per thread
template <typename T> __host__ __device__ constexpr int cv_strip() { return sizeof(T) == 2 ? 16 : 8; }  // tokens per thread

// (bf16 results: the quotient by __fdividef, 2 ulp of fp32 against the 2^-8 of the store; fp32 results
// by the full-precision division, whose ten-odd instructions bounded the bf16 convolution)
template <typename T> __device__ __forceinline__ float silu_f(float v) { return v / (1.f + __expf(-v)); }
template <> __device__ __forceinline__ float silu_f<__nv_bfloat16>(float v) { return __fdividef(v, 1.f + __expf(-v)); }

template <typename T> __device__ __forceinline__ void store8(T *p, const float (&v)[8]);
template <> __device__ __forceinline__ void store8<float>(float *p, const float (&v)[8]) {
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<float4 *>(p + 4) = make_float4(v[4], v[5], v[6], v[7]);
}
template <> __device__ __forceinline__ void store8<__nv_bfloat16>(__nv_bfloat16 *p, const float (&v)[8]) {
    uint32_t o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __nv_bfloat162 q = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
        o[i] = *reinterpret_cast<const uint32_t *>(&q);
    }
    *reinterpret_cast<uint4 *>(p) = make_uint4(o[0], o[1], o[2], o[3]);
}
// Four consecutive elements: raw registers of a load, their widening, the store of four results.
__device__ __forceinline__ void load_raw4(const float *p, float4 &r) { r = *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ void load_raw4(const __nv_bfloat16 *p, uint2 &r) { r = *reinterpret_cast<const uint2 *>(p); }
__device__ __forceinline__ void unpack4(const float4 &r, float (&v)[4]) { v[0] = r.x; v[1] = r.y; v[2] = r.z; v[3] = r.w; }
__device__ __forceinline__ void unpack4(const uint2 &r, float (&v)[4]) {
    v[0] = __uint_as_float(r.x << 16); v[1] = __uint_as_float(r.x & 0xffff0000u);
    v[2] = __uint_as_float(r.y << 16); v[3] = __uint_as_float(r.y & 0xffff0000u);
}
template <typename T> struct Raw4;
template <> struct Raw4<float> { typedef float4 type; };
template <> struct Raw4<__nv_bfloat16> { typedef uint2 type; };
__device__ __forceinline__ void store4(float *p, const float (&v)[4]) { *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]); }
__device__ __forceinline__ void store4(__nv_bfloat16 *p, const float (&v)[4]) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]), b = __floats2bfloat162_rn(v[2], v[3]);
    *reinterpret_cast<uint2 *>(p) = make_uint2(*reinterpret_cast<const uint32_t *>(&a), *reinterpret_cast<const uint32_t *>(&b));
}
}  // namespace

// out[b,t,c] = silu(bias[c] + sum_{i<K} w[c,i] in[b, t-(K-1)+i, c]) over the channels c of
// [x' (D, rows of stride ldx) | B'C' (S)]; tokens before the call come from state_in[b,K-1,C]
// (zeros when null).  A thread owns CV_CH channels and a strip of tokens whose rows are all loaded
// before its window slides along them; the thread of a sequence's last strip also writes state_out.
// Bound by instruction issue and by the warps that fit: 32768 x 4352 channels, bf16: 8 channels x 8 tokens
// a thread with the full-precision division 247 us, __fdividef 182 us, 4 channels x 16 tokens 153 us, held
// to 80 registers (three blocks) 137 us (4.2 TB/s); 12 tokens 147 us, 24 tokens in two blocks 139 us.
template <typename T>
__global__ void __launch_bounds__(256, 3)
conv_silu_kernel(const T *__restrict__ xp, int64_t ldx, const T *__restrict__ bcp, const float *__restrict__ cw,
                 const float *__restrict__ cb, const T *__restrict__ state_in, int B, int L, int D, int S,
                 int K, T *__restrict__ x, T *__restrict__ bc, T *__restrict__ state_out)
{
    constexpr int STRIP = cv_strip<T>();
    grid_dep_launch();
    grid_dep_wait();
    const int C = D + S, ngrp = C / CV_CH;
    const int nstrip = ceil_div(L, STRIP);
    const int64_t item = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (item >= (int64_t)B * nstrip * ngrp) return;
    const int grp = (int)(item % ngrp);
    const int strip = (int)((item / ngrp) % nstrip);
    const int b = (int)(item / ((int64_t)ngrp * nstrip));
    const int c0 = grp * CV_CH;
    const bool from_x = c0 < D;
    const int64_t lds = from_x ? ldx : (int64_t)S;
    const T *src = (from_x ? xp + c0 : bcp + (c0 - D)) + (int64_t)b * L * lds;
    const int64_t ldd = from_x ? (int64_t)D : (int64_t)S;
    const int t0 = strip * STRIP, t1 = min(L, t0 + STRIP);
    T *dst = (from_x ? x + c0 : bc + (c0 - D)) + ((int64_t)b * L + t0) * ldd;
    typename Raw4<T>::type raw[STRIP];
    {
        const T *p = src + (int64_t)t0 * lds;
#pragma unroll
        for (int r = 0; r < STRIP; ++r, p += lds)
            if (t0 + r < t1) load_raw4(p, raw[r]);
    }
    // token at position tt of this sequence (tt may be negative: before the call)
    auto fetch = [&](int tt, float (&v)[CV_CH]) {
        typename Raw4<T>::type q;
        if (tt >= 0) {
            load_raw4(src + (int64_t)tt * lds, q);
            unpack4(q, v);
        } else if (state_in && tt >= -(K - 1)) {
            load_raw4(state_in + ((int64_t)b * (K - 1) + (K - 1 + tt)) * C + c0, q);
            unpack4(q, v);
        } else {
#pragma unroll
            for (int i = 0; i < CV_CH; ++i) v[i] = 0.f;
        }
    };
    float win[CV_K][CV_CH];
#pragma unroll
    for (int j = 0; j < CV_K - 1; ++j) fetch(t0 - (CV_K - 1) + j, win[j]);
    // taps aligned to the end of a window of CV_K: tap j multiplies the token CV_K-1-j steps back
    float wt[CV_K][CV_CH], bias[CV_CH];
#pragma unroll
    for (int q = 0; q < CV_CH; ++q) {
        bias[q] = cb ? cb[c0 + q] : 0.f;
        if (K == CV_K) {
            const float4 t4 = *reinterpret_cast<const float4 *>(cw + (int64_t)(c0 + q) * CV_K);
            wt[0][q] = t4.x; wt[1][q] = t4.y; wt[2][q] = t4.z; wt[3][q] = t4.w;
        } else {
#pragma unroll
            for (int j = 0; j < CV_K; ++j) {
                const int i = j - (CV_K - K);
                wt[j][q] = i >= 0 ? cw[(int64_t)(c0 + q) * K + i] : 0.f;
            }
        }
    }
#pragma unroll
    for (int r = 0; r < STRIP; ++r) {
        if (t0 + r >= t1) break;
        unpack4(raw[r], win[(r + CV_K - 1) % CV_K]);
        float o[CV_CH];
#pragma unroll
        for (int q = 0; q < CV_CH; ++q) {
            float acc = bias[q];
#pragma unroll
            for (int j = 0; j < CV_K; ++j) acc = fmaf(wt[j][q], win[(r + j) % CV_K][q], acc);
            o[q] = silu_f<T>(acc);
        }
        store4(dst, o);
        dst += ldd;
    }
    if (state_out && strip == nstrip - 1) {
        for (int i = 0; i < K - 1; ++i) {
            float v[CV_CH];
            fetch(L - (K - 1) + i, v);
            store4(state_out + ((int64_t)b * (K - 1) + i) * C + c0, v);
        }
    }
}

// out[t, g-th group] = v / sqrt(mean(v^2) + eps) * weight,  v = y * silu(z); one block per
// (token, group).  A thread holds its GN_VEC chunks of 8 channels in registers from the first load to the
// store (groups of up to 8 GN_VEC GN_THREADS channels; longer ones go over the row again), so that every
// element is read once and all loads are in flight together.  32768 x 4096, bf16: two passes over the row
// 233 us (3.4 TB/s), this form 133 us (6.1 TB/s); 128 threads with four chunks each 160 us (64 registers,
// fewer warps).
constexpr int GN_THREADS = 256, GN_VEC = 2;
template <typename T>
__global__ void __launch_bounds__(GN_THREADS, 6)
gated_rmsnorm_kernel(const T *__restrict__ y, const T *__restrict__ z, int64_t ldz, const float *__restrict__ wt,
                     int D, int ngroups, float eps, T *__restrict__ out)
{
    grid_dep_launch();
    grid_dep_wait();
    __shared__ float s_part[8];
    const int gs = D / ngroups;
    const int64_t t = blockIdx.x / ngroups;
    const int g = blockIdx.x % ngroups;
    const T *yr = y + t * D + g * gs;
    const T *zr = z + t * ldz + g * gs;
    float v[GN_VEC][8];
    float ss = 0.f;
    {
        typename Raw8<T>::type ry[GN_VEC], rz[GN_VEC];
#pragma unroll
        for (int i = 0; i < GN_VEC; ++i) {
            const int c = (i * GN_THREADS + threadIdx.x) * 8;
            if (c < gs) {
                load_raw8(yr + c, ry[i]);
                load_raw8(zr + c, rz[i]);
            }
        }
#pragma unroll
        for (int i = 0; i < GN_VEC; ++i) {
            const int c = (i * GN_THREADS + threadIdx.x) * 8;
            if (c < gs) {
                float yv[8], zv[8];
                unpack8(ry[i], yv);
                unpack8(rz[i], zv);
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    v[i][q] = yv[q] * silu_f<T>(zv[q]);
                    ss = fmaf(v[i][q], v[i][q], ss);
                }
            }
        }
    }
    for (int c = (GN_VEC * GN_THREADS + threadIdx.x) * 8; c < gs; c += GN_THREADS * 8) {
        float yv[8], zv[8];
        load8(yr + c, yv);
        load8(zr + c, zv);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float x = yv[q] * silu_f<T>(zv[q]);
            ss = fmaf(x, x, ss);
        }
    }
    ss = warp_sum(ss);
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = ss;
    __syncthreads();
    const float tot = ((s_part[0] + s_part[1]) + (s_part[2] + s_part[3])) + ((s_part[4] + s_part[5]) + (s_part[6] + s_part[7]));
    const float r = rsqrtf(tot / gs + eps);
    T *orow = out + t * D + g * gs;
    const float *wg = wt + g * gs;
#pragma unroll
    for (int i = 0; i < GN_VEC; ++i) {
        const int c = (i * GN_THREADS + threadIdx.x) * 8;
        if (c < gs) {
            float wv[8], o[8];
            load8(wg + c, wv);
#pragma unroll
            for (int q = 0; q < 8; ++q) o[q] = v[i][q] * r * wv[q];
            store8<T>(orow + c, o);
        }
    }
    for (int c = (GN_VEC * GN_THREADS + threadIdx.x) * 8; c < gs; c += GN_THREADS * 8) {
        float yv[8], zv[8], o[8];
        load8(yr + c, yv);
        load8(zr + c, zv);
#pragma unroll
        for (int q = 0; q < 8; ++q) o[q] = yv[q] * silu_f<T>(zv[q]) * r * wg[c + q];
        store8<T>(orow + c, o);
    }
}

// dt[t, h] (float) = zxdt[t, off + h]
template <typename T>
__global__ void __launch_bounds__(256)
dt_columns_kernel(const T *__restrict__ zxdt, int64_t ld, int off, int64_t Ttok, int H, float *__restrict__ dt)
{
    grid_dep_wait();
    const int64_t n = Ttok * H;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dt[i] = to_f32<T>(zxdt[(i / H) * ld + off + (int)(i % H)]);
}

template <typename T>
static void launch_conv_t(LaunchCtx &ctx, const void *xp, int64_t ldx, const void *bcp, const float *cw, const float *cb,
                          const void *state_in, int B, int L, int D, int S, int K, void *x, void *bc, void *state_out)
{
    const int64_t items = (int64_t)B * ceil_div(L, cv_strip<T>()) * ((D + S) / CV_CH);
    launch_kernel(conv_silu_kernel<T>, dim3((unsigned)ceil_div64(items, 256)), dim3(256), 0, ctx.stream, true,
                  (const T *)xp, ldx, (const T *)bcp, cw, cb, (const T *)state_in, B, L, D, S, K, (T *)x, (T *)bc,
                  (T *)state_out);
}

int launch_conv_silu(LaunchCtx &ctx, int dtype, const void *xp, int64_t ldx, const void *bcp, const float *cw,
                     const float *cb, const void *state_in, int B, int L, int D, int S, int K, void *x,
                     void *bc, void *state_out)
{
    if (B <= 0 || L <= 0) return SWIMBA_OK;
    ctx.begin(STAGE_CONV);
    if (dtype == SWIMBA_DTYPE_FP32)
        launch_conv_t<float>(ctx, xp, ldx, bcp, cw, cb, state_in, B, L, D, S, K, x, bc, state_out);
    else
        launch_conv_t<__nv_bfloat16>(ctx, xp, ldx, bcp, cw, cb, state_in, B, L, D, S, K, x, bc, state_out);
    ctx.end();
    return cudaGetLastError() == cudaSuccess ? SWIMBA_OK : SWIMBA_ERR_CUDA;
}

int launch_gated_rmsnorm(LaunchCtx &ctx, int dtype, const void *y, const void *z, int64_t ldz, const float *wt,
                         int64_t T, int D, int ngroups, float eps, void *out)
{
    if (T <= 0) return SWIMBA_OK;
    const dim3 grid((unsigned)(T * ngroups)), block(GN_THREADS);
    ctx.begin(STAGE_GATED_NORM);
    if (dtype == SWIMBA_DTYPE_FP32)
        launch_kernel(gated_rmsnorm_kernel<float>, grid, block, 0, ctx.stream, true, (const float *)y, (const float *)z,
                      ldz, wt, D, ngroups, eps, (float *)out);
    else
        launch_kernel(gated_rmsnorm_kernel<__nv_bfloat16>, grid, block, 0, ctx.stream, true, (const __nv_bfloat16 *)y,
                      (const __nv_bfloat16 *)z, ldz, wt, D, ngroups, eps, (__nv_bfloat16 *)out);
    ctx.end();
    return cudaGetLastError() == cudaSuccess ? SWIMBA_OK : SWIMBA_ERR_CUDA;
}

int launch_dt_columns(LaunchCtx &ctx, int dtype, const void *zxdt, int64_t ld, int off, int64_t T, int H, float *dt)
{
    if (T <= 0) return SWIMBA_OK;
    int64_t blocks = ceil_div64(T * H, 256);
    if (blocks > 148 * 8) blocks = 148 * 8;
    ctx.begin(STAGE_DT_COLUMNS);
    if (dtype == SWIMBA_DTYPE_FP32)
        dt_columns_kernel<float><<<(unsigned)blocks, 256, 0, ctx.stream>>>((const float *)zxdt, ld, off, T, H, dt);
    else
        dt_columns_kernel<__nv_bfloat16><<<(unsigned)blocks, 256, 0, ctx.stream>>>((const __nv_bfloat16 *)zxdt, ld, off, T, H, dt);
    ctx.end();
    return cudaGetLastError() == cudaSuccess ? SWIMBA_OK : SWIMBA_ERR_CUDA;
}

}  // namespace swimba
