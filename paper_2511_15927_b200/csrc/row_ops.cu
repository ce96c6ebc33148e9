// Small row-wise kernels around the mixer: embedding gather, RMSNorm, the gated norm's rstd, arg-max
// over the vocabulary, the carried conv state.  All are bandwidth-trivial next to the GEMMs and the scan.
#include "dm_internal.h"
#include "tc_ptx.cuh"

namespace dm {
namespace {

template <typename T> __device__ __forceinline__ float ldf(const T *p);
template <> __device__ __forceinline__ float ldf<float>(const float *p) { return *p; }
template <> __device__ __forceinline__ float ldf<__nv_bfloat16>(const __nv_bfloat16 *p) { return __bfloat162float(*p); }
template <typename T> __device__ __forceinline__ void stf(T *p, float v);
template <> __device__ __forceinline__ void stf<float>(float *p, float v) { *p = v; }
template <> __device__ __forceinline__ void stf<__nv_bfloat16>(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }

__device__ __forceinline__ float block_sum(float v, float *red) {
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    float t = 0.f;
    for (int i = 0; i < nwarp; ++i) t += red[i];      // same order in every thread: deterministic
    return t;
}

// One warp per row: the lanes read the row's per-head sums side by side, then reduce in a fixed order.
__global__ void rstd_kernel(const float *__restrict__ ssq, float *__restrict__ rstd, int rows, int H, float inv_n, float eps) {
    pdl_wait();
    pdl_trigger();
    const int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (r >= rows) return;
    float s = 0.f;
    for (int h = lane; h < H; h += 32) s += ssq[(int64_t)r * H + h];
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) rstd[r] = rsqrtf(s * inv_n + eps);
}

template <typename T>
__global__ void embed_kernel(const T *__restrict__ embed, const int32_t *__restrict__ tokens, float *__restrict__ r, int d, int vocab) {
    pdl_wait();
    pdl_trigger();
    const int64_t t = blockIdx.x;
    int id = tokens[t];
    id = id < 0 ? 0 : (id >= vocab ? vocab - 1 : id);      // ids are validated on the host side of the tests; clamp keeps reads in bounds
    const T *e = embed + (int64_t)id * d;
    constexpr int PER = 16 / (int)sizeof(T);                // channels per 16-byte load, where the rows allow it
    if (d % PER == 0 && (reinterpret_cast<uintptr_t>(embed) & 15u) == 0) {
        for (int c = threadIdx.x * PER; c < d; c += blockDim.x * PER) {
            const uint4 v = __ldg(reinterpret_cast<const uint4 *>(e + c));
            const T *x = reinterpret_cast<const T *>(&v);
#pragma unroll
            for (int i = 0; i < PER; i += 4) *reinterpret_cast<float4 *>(r + t * d + c + i) = make_float4(ldf(x + i), ldf(x + i + 1), ldf(x + i + 2), ldf(x + i + 3));
        }
    } else {
        for (int c = threadIdx.x; c < d; c += blockDim.x) r[t * d + c] = ldf(e + c);
    }
}

// The two row kernels below keep the token's channels in registers between the statistics and the output (one read
// of r): thread i holds channels 4 (i + 256 k) .. +3 for k < ROW_K, which covers d <= 4096; wider rows are re-read.
constexpr int ROW_THREADS = 256, ROW_K = 4;

template <typename T> __device__ __forceinline__ void st4(T *p, float a, float b, float c, float d);
template <> __device__ __forceinline__ void st4<float>(float *p, float a, float b, float c, float d) { *reinterpret_cast<float4 *>(p) = make_float4(a, b, c, d); }
template <> __device__ __forceinline__ void st4<__nv_bfloat16>(__nv_bfloat16 *p, float a, float b, float c, float d) {
    __nv_bfloat162 lo = __floats2bfloat162_rn(a, b), hi = __floats2bfloat162_rn(c, d);
    *reinterpret_cast<uint2 *>(p) = make_uint2(*reinterpret_cast<uint32_t *>(&lo), *reinterpret_cast<uint32_t *>(&hi));
}

// eight consecutive channels, the first a multiple of 8
template <typename T> __device__ __forceinline__ void st8(T *p, float a, float b, float c, float d, float e, float f, float g, float h);
template <> __device__ __forceinline__ void st8<float>(float *p, float a, float b, float c, float d, float e, float f, float g, float h) { st4(p, a, b, c, d); st4(p + 4, e, f, g, h); }
template <> __device__ __forceinline__ void st8<__nv_bfloat16>(__nv_bfloat16 *p, float a, float b, float c, float d, float e, float f, float g, float h) {
    const __nv_bfloat162 v[4] = {__floats2bfloat162_rn(a, b), __floats2bfloat162_rn(c, d), __floats2bfloat162_rn(e, f), __floats2bfloat162_rn(g, h)};
    const uint32_t *w = reinterpret_cast<const uint32_t *>(v);
    *reinterpret_cast<uint4 *>(p) = make_uint4(w[0], w[1], w[2], w[3]);
}

template <typename T>
__global__ void __launch_bounds__(ROW_THREADS)
rmsnorm_kernel(const float *__restrict__ r, const T *__restrict__ w, T *__restrict__ u, int d, float eps) {
    pdl_wait();
    pdl_trigger();
    __shared__ float red[32];
    const int64_t t = blockIdx.x;
    const float *row = r + t * d;
    const bool fast = (d & 3) == 0 && d <= 4 * ROW_THREADS * ROW_K;
    float4 v[ROW_K];
    float s = 0.f;
    if (fast) {
#pragma unroll
        for (int k = 0; k < ROW_K; ++k) {
            const int c = 4 * (threadIdx.x + ROW_THREADS * k);
            v[k] = c < d ? *reinterpret_cast<const float4 *>(row + c) : make_float4(0.f, 0.f, 0.f, 0.f);
            s = fmaf(v[k].x, v[k].x, s); s = fmaf(v[k].y, v[k].y, s); s = fmaf(v[k].z, v[k].z, s); s = fmaf(v[k].w, v[k].w, s);
        }
    } else {
        for (int c = threadIdx.x; c < d; c += blockDim.x) { const float x = row[c]; s = fmaf(x, x, s); }
    }
    s = block_sum(s, red);
    const float rs = rsqrtf(s / (float)d + eps);
    if (fast) {
#pragma unroll
        for (int k = 0; k < ROW_K; ++k) {
            const int c = 4 * (threadIdx.x + ROW_THREADS * k);
            if (c < d) st4(u + t * d + c, v[k].x * rs * ldf(w + c), v[k].y * rs * ldf(w + c + 1), v[k].z * rs * ldf(w + c + 2), v[k].w * rs * ldf(w + c + 3));
        }
    } else {
        for (int c = threadIdx.x; c < d; c += blockDim.x) stf(u + t * d + c, row[c] * rs * ldf(w + c));
    }
}

// u[t, :] = gamma[b, :] * (r[t, :] - mean) / sqrt(var + eps) + beta[b, :], b = t / L  (App. A.1, Eq. "AdaLN");
// gamma and beta are rows of the per-sequence modulation table (row pitch ld_mod).
template <typename T>
__global__ void __launch_bounds__(ROW_THREADS)
adaln_kernel(const float *__restrict__ r, const float *__restrict__ gamma, const float *__restrict__ beta, int64_t ld_mod,
             T *__restrict__ u, int L, int d, float eps) {
    pdl_wait();
    pdl_trigger();
    __shared__ float red[32];
    const int64_t t = blockIdx.x, b = t / L;
    const float *row = r + t * d, *g = gamma + b * ld_mod, *be = beta + b * ld_mod;
    const bool fast = (d & 3) == 0 && d <= 4 * ROW_THREADS * ROW_K;
    float4 v[ROW_K];
    float s = 0.f;
    if (fast) {
#pragma unroll
        for (int k = 0; k < ROW_K; ++k) {
            const int c = 4 * (threadIdx.x + ROW_THREADS * k);
            v[k] = c < d ? *reinterpret_cast<const float4 *>(row + c) : make_float4(0.f, 0.f, 0.f, 0.f);
            s += (v[k].x + v[k].y) + (v[k].z + v[k].w);
        }
    } else {
        for (int c = threadIdx.x; c < d; c += blockDim.x) s += row[c];
    }
    const float mu = block_sum(s, red) / (float)d;
    float q = 0.f;
    if (fast) {
#pragma unroll
        for (int k = 0; k < ROW_K; ++k) {
            const int c = 4 * (threadIdx.x + ROW_THREADS * k);
            if (c < d) {
                const float a0 = v[k].x - mu, a1 = v[k].y - mu, a2 = v[k].z - mu, a3 = v[k].w - mu;
                q = fmaf(a0, a0, q); q = fmaf(a1, a1, q); q = fmaf(a2, a2, q); q = fmaf(a3, a3, q);
            }
        }
    } else {
        for (int c = threadIdx.x; c < d; c += blockDim.x) { const float x = row[c] - mu; q = fmaf(x, x, q); }
    }
    const float rs = rsqrtf(block_sum(q, red) / (float)d + eps);
    if (fast) {
#pragma unroll
        for (int k = 0; k < ROW_K; ++k) {
            const int c = 4 * (threadIdx.x + ROW_THREADS * k);
            if (c < d)
                st4(u + t * d + c, fmaf(g[c], (v[k].x - mu) * rs, be[c]), fmaf(g[c + 1], (v[k].y - mu) * rs, be[c + 1]),
                    fmaf(g[c + 2], (v[k].z - mu) * rs, be[c + 2]), fmaf(g[c + 3], (v[k].w - mu) * rs, be[c + 3]));
        }
    } else {
        for (int c = threadIdx.x; c < d; c += blockDim.x) stf(u + t * d + c, fmaf(g[c], (row[c] - mu) * rs, be[c]));
    }
}

// The same with a warp per row, its channels in the lanes' registers (8 (lane + 32 k) .. +7, k < K8): every load of a row is in flight at once and the statistics need no
// block barrier.  Bound by the stream of rows (4 bytes in, 2 out per channel).  8192 rows of 1920: 34 us with a block per row, 24 us.  For d up to 2048 in whole groups of 8; the
// kernel above takes the rest (a wider row no longer fits a warp's registers).
constexpr int AW_K8 = 8, AW_ROWS = 4;
template <typename T>
__global__ void __launch_bounds__(32 * AW_ROWS)
adaln_warp_kernel(const float *__restrict__ r, const float *__restrict__ gamma, const float *__restrict__ beta, int64_t ld_mod, T *__restrict__ u, int T_rows, int L, int d, float eps) {
    pdl_wait();
    pdl_trigger();
    const int lane = threadIdx.x & 31;
    const int64_t t = (int64_t)blockIdx.x * AW_ROWS + (threadIdx.x >> 5);
    if (t >= T_rows) return;
    const float *row = r + t * d, *g = gamma + t / L * ld_mod, *be = beta + t / L * ld_mod;
    float4 v[2 * AW_K8];
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < AW_K8; ++k) {
        const int c = 8 * (lane + 32 * k);
        v[2 * k] = v[2 * k + 1] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (c < d) { v[2 * k] = *reinterpret_cast<const float4 *>(row + c); v[2 * k + 1] = *reinterpret_cast<const float4 *>(row + c + 4); }
    }
#pragma unroll
    for (int k = 0; k < 2 * AW_K8; ++k) s += (v[k].x + v[k].y) + (v[k].z + v[k].w);
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    const float mu = s / (float)d;
    float q = 0.f;
#pragma unroll
    for (int k = 0; k < AW_K8; ++k) {
        if (8 * (lane + 32 * k) >= d) break;
#pragma unroll
        for (int e = 2 * k; e < 2 * k + 2; ++e) {
            v[e].x -= mu; v[e].y -= mu; v[e].z -= mu; v[e].w -= mu;
            q = fmaf(v[e].x, v[e].x, q); q = fmaf(v[e].y, v[e].y, q); q = fmaf(v[e].z, v[e].z, q); q = fmaf(v[e].w, v[e].w, q);
        }
    }
    for (int off = 16; off > 0; off >>= 1) q += __shfl_xor_sync(0xffffffffu, q, off);
    const float rs = rsqrtf(q / (float)d + eps);
#pragma unroll
    for (int k = 0; k < AW_K8; ++k) {
        const int c = 8 * (lane + 32 * k);
        if (c >= d) break;
        const float4 g0 = __ldg(reinterpret_cast<const float4 *>(g + c)), g1 = __ldg(reinterpret_cast<const float4 *>(g + c + 4));
        const float4 b0 = __ldg(reinterpret_cast<const float4 *>(be + c)), b1 = __ldg(reinterpret_cast<const float4 *>(be + c + 4));
        const float4 x = v[2 * k], y = v[2 * k + 1];
        st8(u + t * d + c, fmaf(g0.x, x.x * rs, b0.x), fmaf(g0.y, x.y * rs, b0.y), fmaf(g0.z, x.z * rs, b0.z), fmaf(g0.w, x.w * rs, b0.w),
            fmaf(g1.x, y.x * rs, b1.x), fmaf(g1.y, y.y * rs, b1.y), fmaf(g1.z, y.z * rs, b1.z), fmaf(g1.w, y.w * rs, b1.w));
    }
}

// mod[b, j] = bias[j] + sum_c w[j, c] tau[b, c]: the modulation vectors of one layer (App. A.1: (gamma, beta) = W_cond tau).
// A warp computes MOD_R consecutive outputs of MOD_B sequences: a weight is read once for all of them, the first MOD_C columns before the kernel before this one has
// finished.  Bound by latency: 8 sequences, 11520 outputs of 128 columns (3 MB of weights): 8 us; with a warp per output element, whose lanes did 4
// products between five shuffles, 15 us.
constexpr int MOD_R = 4, MOD_B = 8, MOD_C = 128;
template <typename T>
__global__ void __launch_bounds__(256)
modulation_kernel(const float *__restrict__ tau, const T *__restrict__ w, const float *__restrict__ bias, float *__restrict__ mod, int n_out, int d_c, int B) {
    const int j0 = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * MOD_R, lane = threadIdx.x & 31, b0 = blockIdx.y * MOD_B;
    float wv[MOD_C / 32][MOD_R];
#pragma unroll
    for (int i = 0; i < MOD_C / 32; ++i)
#pragma unroll
        for (int r = 0; r < MOD_R; ++r) wv[i][r] = j0 + r < n_out && 32 * i + lane < d_c ? ldf(w + (int64_t)(j0 + r) * d_c + 32 * i + lane) : 0.f;
    pdl_wait();
    pdl_trigger();
    if (j0 >= n_out) return;
    float acc[MOD_R * MOD_B];
#pragma unroll
    for (int i = 0; i < MOD_R * MOD_B; ++i) acc[i] = 0.f;
    auto column = [&](int c, const float (&x)[MOD_R]) {
#pragma unroll
        for (int b = 0; b < MOD_B; ++b) {
            const float t = b0 + b < B && c < d_c ? __ldg(tau + (int64_t)(b0 + b) * d_c + c) : 0.f;
#pragma unroll
            for (int r = 0; r < MOD_R; ++r) acc[r * MOD_B + b] = fmaf(x[r], t, acc[r * MOD_B + b]);
        }
    };
#pragma unroll
    for (int i = 0; i < MOD_C / 32; ++i) column(32 * i + lane, wv[i]);
    for (int c = MOD_C + lane; c < d_c + lane; c += 32) {          // (every lane takes every step: the sums below are the warp's)
        float x[MOD_R];
#pragma unroll
        for (int r = 0; r < MOD_R; ++r) x[r] = j0 + r < n_out && c < d_c ? ldf(w + (int64_t)(j0 + r) * d_c + c) : 0.f;
        column(c, x);
    }
    // sums over the lanes, halving the number of values a lane holds at each step: lane l ends with value l
    static_assert(MOD_R * MOD_B == 32, "one value per lane");
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const bool up = lane & off;
#pragma unroll
        for (int i = 0; i < off; ++i) {
            const float other = __shfl_xor_sync(0xffffffffu, up ? acc[i] : acc[i + off], off);
            acc[i] = (up ? acc[i + off] : acc[i]) + other;
        }
    }
    const int j = j0 + lane / MOD_B, b = b0 + lane % MOD_B;
    if (j < n_out && b < B) mod[(int64_t)b * n_out + j] = acc[0] + (bias ? bias[j] : 0.f);
}

template <typename T>
__global__ void argmax_kernel(const T *__restrict__ logits, int32_t *__restrict__ out, int V) {
    __shared__ float bv[32];
    __shared__ int bi[32];
    const int64_t t = blockIdx.x;
    float best = -INFINITY; int idx = 0x7fffffff;
    const T *row = logits + t * V;
    constexpr int PER = 16 / (int)sizeof(T);            // elements per 16-byte load
    if ((reinterpret_cast<uintptr_t>(row) & 15u) == 0) {
        const int nvec = V / PER;
        for (int i = threadIdx.x; i < nvec; i += blockDim.x) {
            const uint4 q = *reinterpret_cast<const uint4 *>(row + (int64_t)i * PER);
            const T *e = reinterpret_cast<const T *>(&q);
#pragma unroll
            for (int j = 0; j < PER; ++j) {                 // increasing v inside the thread: strict > keeps the lowest index
                const float x = ldf(e + j);
                if (x > best) { best = x; idx = i * PER + j; }
            }
        }
        for (int v = nvec * PER + threadIdx.x; v < V; v += blockDim.x) {
            const float x = ldf(row + v);
            if (x > best || (x == best && v < idx)) { best = x; idx = v; }
        }
    } else {
        for (int v = threadIdx.x; v < V; v += blockDim.x) {
            const float x = ldf(row + v);
            if (x > best || (x == best && v < idx)) { best = x; idx = v; }
        }
    }
    for (int off = 16; off > 0; off >>= 1) {
        const float ob = __shfl_xor_sync(0xffffffffu, best, off);
        const int oi = __shfl_xor_sync(0xffffffffu, idx, off);
        if (ob > best || (ob == best && oi < idx)) { best = ob; idx = oi; }
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
    if (lane == 0) { bv[warp] = best; bi[warp] = idx; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < nwarp; ++i)
            if (bv[i] > best || (bv[i] == best && bi[i] < idx)) { best = bv[i]; idx = bi[i]; }
        out[t] = idx == 0x7fffffff ? 0 : idx;
    }
}

// Row r (0..k-2) of the new conv state of batch row b is row L + r - (k-1) of the block when that is
// >= 0, otherwise row (k-1) + (L + r - (k-1)) of the old state (or zero).
template <typename T>
__global__ void conv_state_kernel(const T *__restrict__ zx, const T *__restrict__ conv_in, T *__restrict__ conv_out,
                                  int L, int k, int d_inner, int conv_ch, int d_in_proj) {
    pdl_wait();
    pdl_trigger();
    const int b = blockIdx.y, r = blockIdx.z;
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= conv_ch) return;
    const int src = L + r - (k - 1);
    T v;
    if (src >= 0) v = zx[((int64_t)b * L + src) * d_in_proj + d_inner + c];
    else if (conv_in) v = conv_in[((int64_t)b * (k - 1) + (k - 1 + src)) * conv_ch + c];
    else { stf(&v, 0.f); }
    conv_out[((int64_t)b * (k - 1) + r) * conv_ch + c] = v;
}

// g0 <- s0 g0 + s1 g1, one block of threads per row (tied projections: the sum of the directions before the shared out_proj);
// 16-byte accesses when the rows allow it (VEC = elements per 16 bytes, or 1)
template <typename T, int VEC>
__global__ void __launch_bounds__(256) combine_kernel(T *__restrict__ g0, const T *__restrict__ g1, const float *__restrict__ r0,
                                                       const float *__restrict__ r1, int64_t rows, int d_inner) {
    for (int64_t t = blockIdx.x; t < rows; t += gridDim.x) {
        const float s0 = r0 ? r0[t] : 1.f, s1 = r1 ? r1[t] : 1.f;
        T *a = g0 + t * d_inner;
        const T *b = g1 + t * d_inner;
        for (int c = threadIdx.x * VEC; c < d_inner; c += blockDim.x * VEC) {
            if constexpr (VEC == 1) {
                stf(a + c, fmaf(s0, ldf(a + c), s1 * ldf(b + c)));
            } else {
                uint4 va = *reinterpret_cast<const uint4 *>(a + c);
                const uint4 vb = __ldg(reinterpret_cast<const uint4 *>(b + c));
                uint32_t *wa = reinterpret_cast<uint32_t *>(&va);
                const uint32_t *wb = reinterpret_cast<const uint32_t *>(&vb);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if constexpr (sizeof(T) == 2) {
                        const float lo = fmaf(s0, __uint_as_float(wa[e] << 16), s1 * __uint_as_float(wb[e] << 16));
                        const float hi = fmaf(s0, __uint_as_float(wa[e] & 0xFFFF0000u), s1 * __uint_as_float(wb[e] & 0xFFFF0000u));
                        const __nv_bfloat162 pk = __floats2bfloat162_rn(lo, hi);
                        wa[e] = *reinterpret_cast<const uint32_t *>(&pk);
                    } else {
                        wa[e] = __float_as_uint(fmaf(s0, __uint_as_float(wa[e]), s1 * __uint_as_float(wb[e])));
                    }
                }
                *reinterpret_cast<uint4 *>(a + c) = va;
            }
        }
    }
}

}  // namespace

cudaError_t rstd_from_ssq(const float *ssq, float *rstd, int rows, int H, int d_inner, float eps, cudaStream_t s) {
    return launch_chain(rstd_kernel, (rows + 7) / 8, 256, 0, s, 0, ssq, rstd, rows, H, 1.f / (float)d_inner, eps);
}

cudaError_t embed_gather(const void *embed, int dtype, const int32_t *tokens, float *r, int T, int d, int vocab, cudaStream_t s) {
    if (dtype == DM_BF16) return launch_chain(embed_kernel<__nv_bfloat16>, T, 256, 0, s, 0, static_cast<const __nv_bfloat16 *>(embed), tokens, r, d, vocab);
    return launch_chain(embed_kernel<float>, T, 256, 0, s, 0, static_cast<const float *>(embed), tokens, r, d, vocab);
}

cudaError_t rmsnorm_rows(const float *r, const void *w, void *u, int dtype, int T, int d, float eps, cudaStream_t s) {
    if (dtype == DM_BF16) return launch_chain(rmsnorm_kernel<__nv_bfloat16>, T, 256, 0, s, 0, r, static_cast<const __nv_bfloat16 *>(w), static_cast<__nv_bfloat16 *>(u), d, eps);
    return launch_chain(rmsnorm_kernel<float>, T, 256, 0, s, 0, r, static_cast<const float *>(w), static_cast<float *>(u), d, eps);
}

cudaError_t adaln_rows(const float *r, const float *gamma, const float *beta, int64_t ld_mod, void *u, int dtype, int T, int L, int d,
                       float eps, cudaStream_t s) {
    const bool al = !((reinterpret_cast<uintptr_t>(r) | reinterpret_cast<uintptr_t>(gamma) | reinterpret_cast<uintptr_t>(beta) | reinterpret_cast<uintptr_t>(u)) & 15u);
    if (d % 8 == 0 && ld_mod % 4 == 0 && d <= 8 * 32 * AW_K8 && al) {
        const int grid = (T + AW_ROWS - 1) / AW_ROWS;
        if (dtype == DM_BF16) return launch_chain(adaln_warp_kernel<__nv_bfloat16>, grid, 32 * AW_ROWS, 0, s, 0, r, gamma, beta, ld_mod, static_cast<__nv_bfloat16 *>(u), T, L, d, eps);
        return launch_chain(adaln_warp_kernel<float>, grid, 32 * AW_ROWS, 0, s, 0, r, gamma, beta, ld_mod, static_cast<float *>(u), T, L, d, eps);
    }
    if (dtype == DM_BF16) return launch_chain(adaln_kernel<__nv_bfloat16>, T, 256, 0, s, 0, r, gamma, beta, ld_mod, static_cast<__nv_bfloat16 *>(u), L, d, eps);
    return launch_chain(adaln_kernel<float>, T, 256, 0, s, 0, r, gamma, beta, ld_mod, static_cast<float *>(u), L, d, eps);
}

cudaError_t modulation_rows(const float *tau, const void *w_cond, const float *b_cond, float *mod, int dtype, int B, int n_out, int d_c,
                            cudaStream_t s) {
    const dim3 grid((n_out + 8 * MOD_R - 1) / (8 * MOD_R), (B + MOD_B - 1) / MOD_B);
    if (dtype == DM_BF16) return launch_chain(modulation_kernel<__nv_bfloat16>, grid, 256, 0, s, 0, tau, static_cast<const __nv_bfloat16 *>(w_cond), b_cond, mod, n_out, d_c, B);
    return launch_chain(modulation_kernel<float>, grid, 256, 0, s, 0, tau, static_cast<const float *>(w_cond), b_cond, mod, n_out, d_c, B);
}

cudaError_t argmax_rows(const void *logits, int dtype, int32_t *out, int T, int V, cudaStream_t s) {
    if (dtype == DM_BF16) argmax_kernel<<<T, 256, 0, s>>>(static_cast<const __nv_bfloat16 *>(logits), out, V);
    else argmax_kernel<<<T, 256, 0, s>>>(static_cast<const float *>(logits), out, V);
    count_launch();
    return cudaGetLastError();
}

cudaError_t conv_state_update(const void *zx_fwd, const void *conv_in, void *conv_out, int dtype, int B, int L,
                              int k, int d_inner, int conv_ch, int d_in_proj, cudaStream_t s) {
    dim3 grid((conv_ch + 255) / 256, B, k - 1);
    if (dtype == DM_BF16)
        return launch_chain(conv_state_kernel<__nv_bfloat16>, grid, 256, 0, s, 0, static_cast<const __nv_bfloat16 *>(zx_fwd), static_cast<const __nv_bfloat16 *>(conv_in),
                                               static_cast<__nv_bfloat16 *>(conv_out), L, k, d_inner, conv_ch, d_in_proj);
    return launch_chain(conv_state_kernel<float>, grid, 256, 0, s, 0, static_cast<const float *>(zx_fwd), static_cast<const float *>(conv_in),
                                               static_cast<float *>(conv_out), L, k, d_inner, conv_ch, d_in_proj);
}

cudaError_t combine_directions(void *g0, const void *g1, const float *rstd0, const float *rstd1, int dtype, int64_t T, int d_inner, cudaStream_t s) {
    const int64_t most = 8 * (int64_t)tc::sm_count();
    const int blocks = (int)(T < most ? T : most);
    const size_t es = dtype_size(dtype);
    const bool vec = ((size_t)d_inner * es) % 16 == 0 && ((reinterpret_cast<uintptr_t>(g0) | reinterpret_cast<uintptr_t>(g1)) & 15u) == 0;
    if (dtype == DM_BF16) {
        auto *a = static_cast<__nv_bfloat16 *>(g0);
        auto *b = static_cast<const __nv_bfloat16 *>(g1);
        if (vec) combine_kernel<__nv_bfloat16, 8><<<blocks, 256, 0, s>>>(a, b, rstd0, rstd1, T, d_inner);
        else combine_kernel<__nv_bfloat16, 1><<<blocks, 256, 0, s>>>(a, b, rstd0, rstd1, T, d_inner);
    } else {
        auto *a = static_cast<float *>(g0);
        auto *b = static_cast<const float *>(g1);
        if (vec) combine_kernel<float, 4><<<blocks, 256, 0, s>>>(a, b, rstd0, rstd1, T, d_inner);
        else combine_kernel<float, 1><<<blocks, 256, 0, s>>>(a, b, rstd0, rstd1, T, d_inner);
    }
    count_launch();
    return cudaGetLastError();
}

}  // namespace dm
