// CUDA-core GEMMs with fp32 accumulation.  They serve the fp32 I/O mode (whose 1e-4 tolerance rules out
// reduced-precision tensor products) and shapes the tensor-core kernel does not take.
//   gemm_simple_kernel   64 x 64 tiles, any type and alignment: large fp32 products, and bf16 ones whose rows TMA cannot address
//   gemm_f32_kernel      32 x 32 tiles, fp32 with 16-byte rows, for products that leave the 64 x 64 kernel with fewer CTAs than two per SM.
//                        Such a product is bound by the latency of its K loop: the four pairs of warps of a CTA take a quarter of the K steps each,
//                        fetched asynchronously two steps ahead, and add up through shared memory at the end.  Two products (both directions'
//                        in_proj) share a launch, or are summed in it (both out_proj, half of the warps each).  256 x 552 x 128 twice: 48 us
//                        (two launches of the 64 x 64 kernel) -> 11 us; 256 x 128 x 256 twice, summed: 96 -> 15 us.
#include "dm_internal.h"
#include "tc_ptx.cuh"

namespace dm {
namespace {

constexpr int BM = 64, BN = 64, BK = 16, TM = 4, TN = 4;   // 256 threads, 4x4 outputs each

template <typename T> __device__ __forceinline__ float to_f32(T v);
template <> __device__ __forceinline__ float to_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }

template <typename TIn, typename TOut>
__global__ void __launch_bounds__(256)
gemm_simple_kernel(const TIn *__restrict__ A, int64_t lda, const TIn *__restrict__ B, int64_t ldb,
                   TOut *C, int64_t ldc, int M, int N, int K,
                   const float *__restrict__ row_scale, const float *addend, int64_t ld_add, int silu_cols,
                   const float *__restrict__ col_bias, int gelu, const float *__restrict__ col_scale, int cs_rows, int64_t ld_cs, const int *__restrict__ m_dev, int m_off,
                   const float *__restrict__ rs_ssq, int rs_n, float rs_inv, float rs_eps) {
    if (m_dev) M = min(M, max(0, *m_dev - m_off));
    __shared__ float As[BK][BM + 4];
    __shared__ float Bs[BK][BN + 4];
    const int tid = threadIdx.x;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const int tx = tid % 16, ty = tid / 16;
    float acc[TM][TN] = {};
    for (int k0 = 0; k0 < K; k0 += BK) {
        // 64 rows x 16 k per operand = 1024 elements, 4 per thread; consecutive threads walk k
        for (int e = tid; e < BM * BK; e += 256) {
            const int r = e / BK, kk = e % BK;
            const int gm = m0 + r, gk = k0 + kk;
            As[kk][r] = (gm < M && gk < K) ? to_f32(A[(int64_t)gm * lda + gk]) : 0.f;
            const int gn = n0 + r;
            Bs[kk][r] = (gn < N && gk < K) ? to_f32(B[(int64_t)gn * ldb + gk]) : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            float a[TM], b[TN];
#pragma unroll
            for (int i = 0; i < TM; ++i) a[i] = As[kk][ty * TM + i];
#pragma unroll
            for (int j = 0; j < TN; ++j) b[j] = Bs[kk][tx * TN + j];
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int gm = m0 + ty * TM + i;
        if (gm >= M) continue;
        float sc = row_scale ? row_scale[gm] : 1.f;
        if (rs_ssq) {
            float q = 0.f;
            for (int j = 0; j < rs_n; ++j) q += rs_ssq[(int64_t)gm * rs_n + j];
            sc = rsqrtf(q * rs_inv + rs_eps);
        }
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            const int gn = n0 + tx * TN + j;
            if (gn >= N) continue;
            float v = acc[i][j] * sc;
            if (col_bias) v += col_bias[gn];
            if (gn < silu_cols) v = v / (1.f + __expf(-v));
            if (gelu) v = 0.5f * v * (1.f + tanhf(0.7978845608028654f * (v + 0.044715f * v * v * v)));
            if (col_scale) v *= col_scale[(int64_t)(gm / cs_rows) * ld_cs + gn];
            if (addend) v += addend[(int64_t)gm * ld_add + gn];
            if constexpr (sizeof(TOut) == 4) C[(int64_t)gm * ldc + gn] = v;
            else C[(int64_t)gm * ldc + gn] = __float2bfloat16_rn(v);
        }
    }
}

template <typename TIn, typename TOut>
cudaError_t launch(const GemmArgs &a, cudaStream_t s) {
    dim3 grid((a.N + BN - 1) / BN, (a.M + BM - 1) / BM);
    gemm_simple_kernel<TIn, TOut><<<grid, 256, 0, s>>>(
        static_cast<const TIn *>(a.A), a.lda, static_cast<const TIn *>(a.B), a.ldb,
        static_cast<TOut *>(a.C), a.ldc, a.M, a.N, a.K, a.row_scale, a.addend, a.ld_add, a.silu_cols,
        a.col_bias, a.gelu, a.col_scale, a.cs_rows > 0 ? a.cs_rows : 1, a.ld_cs > 0 ? a.ld_cs : a.N, a.m_dev, a.m_off,
        a.rs_ssq, a.rs_n, a.rs_inv, a.rs_eps);
    count_launch();
    return cudaGetLastError();
}

constexpr int FT = 32, FK = 32, FLD = FK + 4, FG = 4;        // tile, K step, row pitch in shared memory (conflict-free float4 reads of 8 rows), K groups
constexpr int FOP = FT * FLD;                                 // floats of one operand tile
constexpr size_t F32_SMEM = (size_t)FG * 2 * 2 * FOP * sizeof(float);
struct F32Problems { GemmArgs p[2]; };

// grid: (N tiles, M tiles, problems); sum: one problem's worth of tiles, both products added into problem 1's output
__global__ void __launch_bounds__(256)
gemm_f32_kernel(const __grid_constant__ F32Problems pr, const int sum) {
    extern __shared__ __align__(16) float fsm[];
    pdl_wait();
    pdl_trigger();
    const int tid = threadIdx.x, g = tid >> 6, t = tid & 63, tx = t & 7, ty = t >> 3;
    const int per = sum ? FG / 2 : FG, prob = sum ? g / per : (int)blockIdx.z, gi = sum ? g % per : g;      // K groups per product
    const GemmArgs &a = pr.p[prob], &o = pr.p[sum ? 1 : prob];
    const int M = a.m_dev ? min(a.M, max(0, *a.m_dev - a.m_off)) : a.M, N = a.N, K = a.K;
    const int m0 = blockIdx.y * FT, n0 = blockIdx.x * FT;
    float *st = fsm + g * 4 * FOP;                             // this group's two stages of (A, B)
    const float *A = static_cast<const float *>(a.A), *B = static_cast<const float *>(a.B);
    const int steps = (K + FK - 1) / FK, mine = gi < steps ? (steps - 1 - gi) / per + 1 : 0;
    auto fetch = [&](int i) {                                  // K step gi + i * per: 32 rows x 32 floats of each operand, 16 bytes at a time
        float *as = st + (i & 1) * 2 * FOP, *bs = as + FOP;
        const int k0 = (gi + i * per) * FK;
#pragma unroll
        for (int u = t; u < FT * FK / 4; u += 64) {
            const int r = u / (FK / 4), c = (u % (FK / 4)) * 4, left = K - k0 - c;
            const uint32_t nb = left >= 4 ? 16u : left > 0 ? 4u * left : 0u;
            const uint32_t na = m0 + r < M ? nb : 0u, nbb = n0 + r < N ? nb : 0u;
            tc::cp_async16(as + r * FLD + c, na ? A + (int64_t)(m0 + r) * a.lda + k0 + c : A, na);
            tc::cp_async16(bs + r * FLD + c, nbb ? B + (int64_t)(n0 + r) * a.ldb + k0 + c : B, nbb);
        }
    };
    float acc[4][4] = {};
    if (mine > 0) fetch(0);
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (mine > 1) fetch(1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    for (int i = 0; i < mine; ++i) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        tc::named_sync(1 + g, 64);
        const float *as = st + (i & 1) * 2 * FOP, *bs = as + FOP;
#pragma unroll
        for (int k = 0; k < FK; k += 4) {
            float4 av[4], bv[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                av[j] = *reinterpret_cast<const float4 *>(as + (ty + 8 * j) * FLD + k);
                bv[j] = *reinterpret_cast<const float4 *>(bs + (tx + 8 * j) * FLD + k);
            }
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
                for (int y = 0; y < 4; ++y) {
                    acc[x][y] = fmaf(av[x].x, bv[y].x, acc[x][y]); acc[x][y] = fmaf(av[x].y, bv[y].y, acc[x][y]);
                    acc[x][y] = fmaf(av[x].z, bv[y].z, acc[x][y]); acc[x][y] = fmaf(av[x].w, bv[y].w, acc[x][y]);
                }
        }
        tc::named_sync(1 + g, 64);
        if (i + 2 < mine) fetch(i + 2);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    tc::cp_async_wait_all();
    __syncthreads();
    float *red = fsm;                                          // [FG][FT][FT + 1]
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) red[(g * FT + ty + 8 * x) * (FT + 1) + tx + 8 * y] = acc[x][y];
    __syncthreads();
    const int row = tid >> 3, gm = m0 + row, c0 = (tid & 7) * 4;
    if (gm >= M) return;
    auto scale_of = [&](const GemmArgs &q) {
        if (q.row_scale) return q.row_scale[gm];
        if (!q.rs_ssq) return 1.f;
        float s = 0.f;
        for (int j = 0; j < q.rs_n; ++j) s += __ldg(q.rs_ssq + (int64_t)gm * q.rs_n + j);
        return rsqrtf(s * q.rs_inv + q.rs_eps);
    };
    const float s_lo = scale_of(pr.p[sum ? 0 : prob]), s_hi = sum ? scale_of(pr.p[1]) : s_lo;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int gn = n0 + c0 + j;
        if (gn >= N) break;
        const float *q = red + row * (FT + 1) + c0 + j;
        constexpr int GP = FT * (FT + 1);
        float v = fmaf(q[0] + q[GP], s_lo, (q[2 * GP] + q[3 * GP]) * s_hi);
        if (o.col_bias) v += o.col_bias[gn];
        if (gn < o.silu_cols) v = v / (1.f + __expf(-v));
        if (o.gelu) v = 0.5f * v * (1.f + tanhf(0.7978845608028654f * (v + 0.044715f * v * v * v)));
        if (o.col_scale) v *= o.col_scale[(int64_t)(gm / o.cs_rows) * o.ld_cs + gn];
        if (o.addend) v += o.addend[(int64_t)gm * o.ld_add + gn];
        if (o.c_dtype == DM_F32) static_cast<float *>(o.C)[(int64_t)gm * o.ldc + gn] = v;
        else static_cast<__nv_bfloat16 *>(o.C)[(int64_t)gm * o.ldc + gn] = __float2bfloat16_rn(v);
    }
}

}  // namespace

bool gemm_f32_supports(const GemmArgs &a, int n) {
    if (a.in_dtype != DM_F32 || a.u || a.M <= 0 || a.N <= 0 || a.K <= 0 || a.lda % 4 || a.ldb % 4) return false;
    if ((reinterpret_cast<uintptr_t>(a.A) | reinterpret_cast<uintptr_t>(a.B)) & 15u) return false;
    // fewer than two 64 x 64 tiles per SM; beyond, that kernel reads half as much shared memory per product
    return (int64_t)((a.M + BM - 1) / BM) * ((a.N + BN - 1) / BN) * n < 2 * tc::sm_count();
}

// n = 1 or 2 products of the same sizes; sum: both into b's output
cudaError_t gemm_f32(const GemmArgs &a, const GemmArgs *b, bool sum, cudaStream_t s) {
    F32Problems pr{{a, b ? *b : a}};
    for (GemmArgs &q : pr.p) {
        if (q.cs_rows <= 0) q.cs_rows = 1;
        if (q.ld_cs <= 0) q.ld_cs = q.N;
    }
    cudaError_t e = cudaFuncSetAttribute(gemm_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F32_SMEM);
    if (e != cudaSuccess) return e;
    return launch_chain(gemm_f32_kernel, dim3((a.N + FT - 1) / FT, (a.M + FT - 1) / FT, b && !sum ? 2 : 1), 256, F32_SMEM, s, 0, pr, sum ? 1 : 0);
}

cudaError_t gemm_simple(const GemmArgs &a, cudaStream_t s) {
    if (a.M <= 0 || a.N <= 0 || a.K <= 0 || a.u) return cudaErrorInvalidValue;
    if ((a.M + BM - 1) / BM > 65535) return cudaErrorInvalidValue;
    if (gemm_f32_supports(a, 1)) return gemm_f32(a, nullptr, false, s);
    if (a.in_dtype == DM_F32) {
        return a.c_dtype == DM_F32 ? launch<float, float>(a, s) : launch<float, __nv_bfloat16>(a, s);
    }
    return a.c_dtype == DM_F32 ? launch<__nv_bfloat16, float>(a, s) : launch<__nv_bfloat16, __nv_bfloat16>(a, s);
}

}  // namespace dm
