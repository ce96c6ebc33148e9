// Fused depthwise conv + SiLU, discretisation, selective scan and gate on the CUDA cores, both
// directions in one launch.  One CTA owns one (batch row, direction, head) and walks the sequence in
// logical time (left-to-right for the forward layer, right-to-left for the reverse layer: the reverse
// layer is the same operator on the reversed sequence, done here by index arithmetic only).
//
// The CTA is split in two groups that work on different chunks of TC tokens at the same time:
//   scan threads (the first P * LPC):  the state h[p][n] of the head lives in their registers: channel p is served
//       by LPC adjacent lanes, each holding N / LPC states; the C-contraction is finished with warp shuffles.  They
//       run the token loop of chunk i from shared memory and leave y_t = h_t C_t + D x_t there.
//   loader threads (the last 128 or 256):  meanwhile one half of them start the copies of chunk i+2 (x, z, B', C': TMA, straight to shared memory)
//       and prepare chunk i+1 (conv + SiLU of this head's x channels, Delta and the decay), the other half write chunk i-1's gated output
//       (g = y SiLU(z) [* norm_w], per-head sum of squares).
// One __syncthreads per chunk hands the buffers over.  B' and C' (conv + SiLU of the B and C columns, shared by all heads) come from a small launch
// of their own.  What bounds it is the chain of L tokens in each of the 2 B H CTAs: at 8 heads of 32, d_state 16, L = 256 a chunk of 32 tokens takes 2.9 k clocks, in
// the scan threads and in the preparing ones alike, and both launches 25 us; with one synchronous loader group, which waited for memory three
// times a chunk, it was 74 us.
//
// This is the exact (fp32) form of the recurrence: the kernel for fp32 I/O (whose 1e-4 tolerance rules out bf16
// products) and for d_state above 128; bf16 I/O with d_state <= 128 runs the chunked kernels of scan_ssd.cu, block
// decoding with carried state included.
#include "dm_internal.h"
#include "tc_ptx.cuh"

namespace dm {
namespace {

using namespace tc;

template <typename T> __device__ __forceinline__ float ldf(const T *p);
template <> __device__ __forceinline__ float ldf<float>(const float *p) { return __ldg(p); }
template <> __device__ __forceinline__ float ldf<__nv_bfloat16>(const __nv_bfloat16 *p) {
    return __bfloat162float(*p);
}
template <typename T> __device__ __forceinline__ void stf(T *p, float v);
template <> __device__ __forceinline__ void stf<float>(float *p, float v) { *p = v; }
template <> __device__ __forceinline__ void stf<__nv_bfloat16>(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }

__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(__nv_bfloat16 v) { return __bfloat162float(v); }
inline size_t es_of(const ScanArgs &a) { return dtype_size(a.dtype); }

__device__ __forceinline__ float silu_f(float v) { return __fdividef(v, 1.f + __expf(-v)); }     // ~1e-6 relative: inside the fp32 tolerance
__device__ __forceinline__ float softplus_f(float v) { return fmaxf(v, 0.f) + log1pf(expf(-fabsf(v))); }

// B' and C' of every token: conv + SiLU of the 2N shared columns, in logical time order semantics (the reverse layer
// looks at later rows), fp32, layout [dir][B*L][2N].  Thread = one column of one run of BC_ROWS consecutive tokens, all its loads in flight at
// once: the launch is a handful of CTAs and one round trip to memory (runs of 32 tokens took 19 us at L = 256).
constexpr int BC_ROWS = 8;
template <typename T>
__global__ void __launch_bounds__(256)
bc_prep_kernel(const ScanArgs a, const int dir0, float *__restrict__ bc) {
    pdl_wait();
    pdl_trigger();
    const int N2 = 2 * a.N, L = a.L, k = a.k;
    const int dir = dir0 + blockIdx.z, b = blockIdx.y;
    const bool rev = dir == 1;
    const ScanDir &w = a.dir[dir];
    const int64_t T_all = (int64_t)a.B * L;
    const T *zx = static_cast<const T *>(a.zx) + ((int64_t)(a.zx_tied ? 0 : dir) * T_all + (int64_t)b * L) * a.d_in_proj;
    const T *conv_in = (!rev && a.conv_in) ? static_cast<const T *>(a.conv_in) + (int64_t)b * (k - 1) * a.conv_ch : nullptr;
    float *out = bc + ((int64_t)dir * T_all + (int64_t)b * L) * N2;
    const bool has_bias = (a.flags & DM_FLAG_CONV_BIAS) && w.conv_b != nullptr;
    const int task = blockIdx.x * blockDim.x + threadIdx.x, col = task % N2, tau0 = task / N2 * BC_ROWS, cc = a.d_inner + col;
    if (tau0 >= L) return;
    float v[BC_ROWS + 3];                                  // pre-conv values of tau0 - 3 .. tau0 + BC_ROWS - 1
#pragma unroll
    for (int i = 0; i < BC_ROWS + 3; ++i) {
        const int tau = tau0 + i - 3;
        v[i] = 0.f;
        if (tau >= 0 && tau < L) v[i] = ldf(zx + (int64_t)(rev ? L - 1 - tau : tau) * a.d_in_proj + a.d_inner + cc);
        else if (tau < 0 && conv_in && k - 1 + tau >= 0) v[i] = ldf(conv_in + (int64_t)(k - 1 + tau) * a.conv_ch + cc);
    }
    float wl[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) wl[m] = m < k ? ldf(static_cast<const T *>(w.conv_w) + (int64_t)cc * k + (k - 1 - m)) : 0.f;
    const float bias = has_bias ? ldf(static_cast<const T *>(w.conv_b) + cc) : 0.f;
#pragma unroll
    for (int i = 0; i < BC_ROWS; ++i) {
        const int tau = tau0 + i;
        if (tau >= L) break;
        float r = fmaf(wl[3], v[i], bias);
        r = fmaf(wl[2], v[i + 1], r); r = fmaf(wl[1], v[i + 2], r); r = fmaf(wl[0], v[i + 3], r);
        out[(int64_t)(rev ? L - 1 - tau : tau) * N2 + col] = silu_f(r);
    }
}

// Shared memory (bytes).  A raw stage holds one chunk as it comes from memory: [B' | C'] fp32 [TC][2N], x [TC + 3][P] (3 rows of history first) and z [TC][P] of
// type T; RAW of them: chunk i - 1 (its z), i (B', C'), i + 1 (x) and i + 2 (in flight).  Then, for two chunks each: conv'd x and y [TC][P], Delta and the decay [TC].
constexpr int RAW = 4;
__host__ __device__ constexpr int lanes_per_channel(int n) { return n / 4 < 8 ? n / 4 : 8; }
__host__ __device__ constexpr int loaders(int p, int n) { return p * lanes_per_channel(n) > 256 ? 128 : 256; }      // loader threads
struct SeqSmem {
    int TC, P, N, es;
    __host__ __device__ int xoff() const { return TC * 2 * N * 4; }                                              // a multiple of 128, as TMA wants its tiles
    __host__ __device__ int zoff() const { return xoff() + up128((TC + 3) * P * es); }
    __host__ __device__ int raw_bytes() const { return zoff() + up128(TC * P * es); }
    __host__ __device__ static int up128(int v) { return (v + 127) / 128 * 128; }
    __host__ __device__ int cooked() const { return RAW * raw_bytes(); }
    __host__ __device__ int cooked_floats() const { return TC * (2 * P + 2); }
    __host__ __device__ size_t total() const { return (size_t)cooked() + 2 * (size_t)cooked_floats() * 4; }
};

// P channels and N states of a head; LPC = lanes per channel, NQ = float4 groups of state per lane
template <typename T, int P, int N>
__global__ void __launch_bounds__(P * lanes_per_channel(N) + loaders(P, N))
scan_seq_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_z, const __grid_constant__ ScanArgs a, const int dir0, const int TC, const int hold, const float *__restrict__ bc_all, int *status) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ uint64_t bars[RAW];                     // raw stage has landed
    __shared__ int abort_word;
    volatile int *abort_flag = &abort_word;
    pdl_wait();
    pdl_trigger();
    constexpr int LPC = lanes_per_channel(N), NQ = N / (4 * LPC), NS = P * LPC, NL = loaders(P, N), NP = NL / 2;       // NS: scan threads, NL: loader threads, NP of them preparing
    const int L = a.L, k = a.k;
    const int h = blockIdx.x, b = blockIdx.z;
    const int dir = dir0 + blockIdx.y;                 // 0 = left-to-right, 1 = right-to-left
    const bool rev = dir == 1;
    const int tid = threadIdx.x;
    const SeqSmem lay{TC, P, N, (int)sizeof(T)};
    const int raw_bytes = lay.raw_bytes(), xoff = lay.xoff(), zoff = lay.zoff(), cooked_floats = lay.cooked_floats();
    auto raw_of = [&](int ci) { return smem + (ci % RAW) * raw_bytes; };
    auto xs_of = [&](int ci) { return reinterpret_cast<float *>(smem + RAW * raw_bytes) + (ci & 1) * cooked_floats; };      // x', then y, Delta, decay

    const ScanDir &w = a.dir[dir];
    const T *conv_w = static_cast<const T *>(w.conv_w);
    const T *conv_b = static_cast<const T *>(w.conv_b);
    const T *norm_w = static_cast<const T *>(w.norm_w);
    const bool has_bias = (a.flags & DM_FLAG_CONV_BIAS) && conv_b != nullptr;
    const bool norm_on = (a.flags & DM_FLAG_GATED_RMSNORM) != 0;

    const int64_t T_all = (int64_t)a.B * L;
    const T *zx = static_cast<const T *>(a.zx) + ((int64_t)(a.zx_tied ? 0 : dir) * T_all + (int64_t)b * L) * a.d_in_proj;
    T *gout = static_cast<T *>(a.g) + ((int64_t)dir * T_all + (int64_t)b * L) * a.d_inner;
    float *ssq = a.ssq ? a.ssq + ((int64_t)dir * T_all + (int64_t)b * L) * a.H : nullptr;
    const T *conv_in = (!rev && a.conv_in) ? static_cast<const T *>(a.conv_in) + (int64_t)b * (k - 1) * a.conv_ch : nullptr;
    const float *bc = bc_all + ((int64_t)dir * T_all + (int64_t)b * L) * (2 * N);
    const int nchunks = (L + TC - 1) / TC;
    const int sg = rev ? -1 : 1, x0 = rev ? TC - 1 : 3, z0 = rev ? TC - 1 : 0;      // token i of a chunk is row x0 + sg i of its x tile, z0 + sg i of its z tile
    if (tid == 0) {
        for (int i = 0; i < RAW; ++i) mbar_init(&bars[i], 1);
        abort_word = 0;
        mbar_fence_init();
    }
    __syncthreads();

    // gated output of chunk ci: one warp per token, lanes over the channels; by warps lw = 0..nwarp-1
    constexpr int CPL = P / 32;                        // channels per lane
    float nw[CPL];
#pragma unroll
    for (int e = 0; e < CPL; ++e) nw[e] = (norm_on && norm_w) ? ldf(norm_w + h * P + (tid & 31) + 32 * e) : 1.f;
    auto finish = [&](int ci, int lw, int nwarp, int lane) {
        const int tau0 = ci * TC, tc = min(TC, L - tau0);
        const T *zs = reinterpret_cast<const T *>(raw_of(ci) + zoff);
        const float *ys = xs_of(ci) + TC * P;
        constexpr int FU = 8 / CPL;                              // tokens in flight per warp
        for (int i0 = lw; i0 < tc; i0 += FU * nwarp) {
            float gv[FU][CPL], sacc[FU];
#pragma unroll
            for (int u = 0; u < FU; ++u) {
                const int i = min(i0 + u * nwarp, tc - 1);
                sacc[u] = 0.f;
#pragma unroll
                for (int e = 0; e < CPL; ++e) {
                    const int c = lane + 32 * e;
                    gv[u][e] = ys[i * P + c] * silu_f(to_f(zs[(z0 + sg * i) * P + c]));
                    sacc[u] = fmaf(gv[u][e], gv[u][e], sacc[u]);
                }
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
                for (int u = 0; u < FU; ++u) sacc[u] += __shfl_xor_sync(0xffffffffu, sacc[u], off);
            }
#pragma unroll
            for (int u = 0; u < FU; ++u) {
                const int i = i0 + u * nwarp;
                if (i >= tc) break;
                const int t = rev ? L - 1 - (tau0 + i) : tau0 + i;
#pragma unroll
                for (int e = 0; e < CPL; ++e) stf(gout + (int64_t)t * a.d_inner + h * P + lane + 32 * e, gv[u][e] * nw[e]);
                if (lane == 0 && ssq) ssq[(int64_t)t * a.H + h] = sacc[u];
            }
        }
    };

    if (tid >= NS + NP) {
        // ------------------------------------------------------------------ finishing half of the loader group
        const int lt = tid - NS - NP;
        __syncthreads();
        for (int ci = 0; ci < nchunks; ++ci) {
            if (ci > 0) finish(ci - 1, lt >> 5, NP / 32, lt & 31);
            __syncthreads();
        }
    } else if (tid >= NS) {
        // ------------------------------------------------------------------ preparing half
        const int lt = tid - NS;
        const float Ah = -expf(w.A_log[h]);
        const float dtb = w.dt_bias[h];
        // Everything chunk ci needs from memory: a tile of x with the three rows before it in time, one of z (rows outside the sequence become zeros) and
        // the run of [B' | C'], in physical order.  (16-byte copies by the threads took 1000 clocks a chunk to issue, and held up the
        // shared-memory reads behind them.)
        bool ok = true;
        int limit = nchunks;                               // copies are started for the chunks below it
        auto fetch = [&](int ci) {
            if (ci >= limit || lt != 0) return;
            if (ci == hold) return;                        // (left out, for the self-test)
            uint8_t *st = raw_of(ci);
            uint64_t *bar = &bars[ci % RAW];
            const int tau0 = ci * TC, tc = min(TC, L - tau0), bt = a.zx_tied ? b : dir * a.B + b, t0 = rev ? L - TC - tau0 : tau0;
            mbar_expect_tx(bar, (uint32_t)((2 * TC + 3) * P * sizeof(T) + tc * 2 * N * 4));
            tma_load_3d(st + xoff, &map_x, a.d_inner + h * P, rev ? t0 : t0 - 3, bt, bar);
            tma_load_3d(st + zoff, &map_z, h * P, t0, bt, bar);
            bulk_load(st, bc + (int64_t)(rev ? L - tau0 - tc : tau0) * 2 * N, tc * 2 * N * 4, bar);
        };
        // the carried rows before the sequence (the tile has zeros there)
        auto carry = [&](int ci) {
            const int neg = 3 - min(3, ci * TC);               // rows of this chunk's history that are before the sequence
            if (!conv_in || neg <= 0) return;
            T *xt = reinterpret_cast<T *>(raw_of(ci) + xoff);
            for (int u = lt; u < neg * P; u += NP) {
                const int r = u / P, c = u - r * P, src = k - 1 - neg + r;      // tile row r = token r - neg before the first one
                if (src >= 0) xt[r * P + c] = conv_in[(int64_t)src * a.conv_ch + h * P + c];
            }
            named_sync(1, NP);
        };
        auto landed = [&](int ci) { ok = mbar_wait(&bars[ci % RAW], (ci / RAW) & 1, abort_flag, status) && ok; };      // (gives up after its limit, then at once: the loop still ends)
        auto dt_of = [&](int ci) {                         // raw step size of token lt of the chunk (TC <= NP)
            const int tau = ci * TC + lt;
            return (lt < TC && tau < L) ? ldf(zx + (int64_t)(rev ? L - 1 - tau : tau) * a.d_in_proj + a.d_inner + a.conv_ch + h) : 0.f;
        };
        // conv + SiLU of this head's channels, Delta and decay: task = (channel, run of tokens); with P = 32 or 64 a thread keeps its channel
        constexpr int nseg = NP / P;
        const int col = lt % P, cc = h * P + col, seg = lt / P;
        float wl[4];                                       // wl[m] multiplies the row m steps back in time
#pragma unroll
        for (int m = 0; m < 4; ++m) wl[m] = m < k ? ldf(conv_w + (int64_t)cc * k + (k - 1 - m)) : 0.f;
        const float bias = has_bias ? ldf(conv_b + cc) : 0.f;
        auto prepare = [&](int ci, float dt_raw) {
            const int tc = min(TC, L - ci * TC);
            float *xs = xs_of(ci), *dl = xs + 2 * TC * P, *da = dl + TC;
            const T *xc = reinterpret_cast<const T *>(raw_of(ci) + xoff) + x0 * P + col;
            const int sP = sg * P;                             // xc[i * sP] = pre-conv value at token i of the chunk
            const int len = (tc + nseg - 1) / nseg, i0 = seg * len, i1 = min(tc, i0 + len);
            if (i0 < i1) {
                float h1 = to_f(xc[(i0 - 1) * sP]), h2 = to_f(xc[(i0 - 2) * sP]), h3 = to_f(xc[(i0 - 3) * sP]);
#pragma unroll 4
                for (int i = i0; i < i1; ++i) {
                    const float cur = to_f(xc[i * sP]);
                    float v = fmaf(wl[3], h3, bias);
                    v = fmaf(wl[2], h2, v); v = fmaf(wl[1], h1, v); v = fmaf(wl[0], cur, v);
                    xs[i * P + col] = silu_f(v);
                    h3 = h2; h2 = h1; h1 = cur;
                }
            }
            if (lt < tc) {
                const float dlt = softplus_f(dt_raw + dtb);
                dl[lt] = dlt;
                da[lt] = expf(dlt * Ah);
            }
        };
        fetch(0);
        fetch(1);
        float dt_cur = dt_of(0), dt_next = dt_of(1);
        landed(0);
        carry(0);
        prepare(0, dt_cur);
        __syncthreads();
        if (!ok) limit = 0;                                // a wait of this thread has given up: no more copies
        for (int ci = 0; ci < nchunks; ++ci) {
            fetch(ci + 2);                                 // its stage held chunk ci - 2, finished before the last barrier
            dt_cur = dt_next;
            dt_next = dt_of(ci + 2);
            if (ci + 1 < nchunks) { landed(ci + 1); if (!ok) limit = min(limit, ci + 1); carry(ci + 1); prepare(ci + 1, dt_cur); }
            __syncthreads();
        }
        // after a wait that gave up: no copy of this CTA may still be in flight when it leaves
        if (lt == 0 && !ok)
            for (int c = limit; c < min(nchunks, limit + 2); ++c) mbar_wait_quiet(&bars[c % RAW], (c / RAW) & 1, 100000000ull);
    } else {
        // ------------------------------------------------------------------ scan group
        const int p = tid / LPC, j = tid - p * LPC;
        const float Dh = (a.flags & DM_FLAG_D_SKIP) ? w.D[h] : 0.f;
        // state slice of this lane: float4 index f = q*LPC + j, q = 0..NQ-1
        float hst[4 * NQ];
        if (!rev && a.ssm_in) {
            const float *h0 = a.ssm_in + (((int64_t)b * a.H + h) * P + p) * N;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const float4 v = *reinterpret_cast<const float4 *>(h0 + (q * LPC + j) * 4);
                hst[4 * q] = v.x; hst[4 * q + 1] = v.y; hst[4 * q + 2] = v.z; hst[4 * q + 3] = v.w;
            }
        } else {
#pragma unroll
            for (int q = 0; q < 4 * NQ; ++q) hst[q] = 0.f;
        }
        __syncthreads();
        for (int ci = 0; ci < nchunks; ++ci) {
            const int tc = min(TC, L - ci * TC);
            const float *xs = xs_of(ci), *dl = xs + 2 * TC * P, *da = dl + TC;
            mbar_wait(&bars[ci % RAW], (ci / RAW) & 1, abort_flag, status);      // (the loaders have waited for it already)
            const float *BC = reinterpret_cast<const float *>(raw_of(ci)) + (rev ? tc - 1 : 0) * 2 * N;
            float *ys = xs_of(ci) + TC * P;
            // h_t = a_t h_{t-1} + Delta_t x_t (x) B_t ;  y_t = h_t C_t + D x_t.  Only h depends on the token before: several tokens' loads and
            // contractions are in flight together
            // (all loads of U tokens first: one warp per scheduler has to overlap their latency by itself)
            constexpr int U = NQ == 1 ? 8 : NQ == 2 ? 4 : NQ == 4 ? 2 : 1;
            auto tokens = [&](int i, int n) {                  // tokens i .. i + n - 1, n <= U
                float av[U], xv[U], dx[U], acc[U];
                float4 bv[U][NQ], cv[U][NQ];
#pragma unroll
                for (int e = 0; e < U; ++e) {
                    const int ie = e < n ? i + e : i;
                    const float4 *B4 = reinterpret_cast<const float4 *>(BC + sg * ie * 2 * N) + j, *C4 = B4 + N / 4;
                    av[e] = da[ie]; xv[e] = xs[ie * P + p]; dx[e] = dl[ie];
#pragma unroll
                    for (int q = 0; q < NQ; ++q) { bv[e][q] = B4[q * LPC]; cv[e][q] = C4[q * LPC]; }
                }
#pragma unroll
                for (int e = 0; e < U; ++e) {
                    dx[e] *= xv[e];
                    if (e >= n) { av[e] = 1.f; dx[e] = 0.f; }
                    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;      // four partial sums keep the dependent chain short
#pragma unroll
                    for (int q = 0; q < NQ; ++q) {
                        hst[4 * q + 0] = fmaf(av[e], hst[4 * q + 0], dx[e] * bv[e][q].x); a0 = fmaf(hst[4 * q + 0], cv[e][q].x, a0);
                        hst[4 * q + 1] = fmaf(av[e], hst[4 * q + 1], dx[e] * bv[e][q].y); a1 = fmaf(hst[4 * q + 1], cv[e][q].y, a1);
                        hst[4 * q + 2] = fmaf(av[e], hst[4 * q + 2], dx[e] * bv[e][q].z); a2 = fmaf(hst[4 * q + 2], cv[e][q].z, a2);
                        hst[4 * q + 3] = fmaf(av[e], hst[4 * q + 3], dx[e] * bv[e][q].w); a3 = fmaf(hst[4 * q + 3], cv[e][q].w, a3);
                    }
                    acc[e] = (a0 + a1) + (a2 + a3);
                }
#pragma unroll
                for (int off = LPC >> 1; off > 0; off >>= 1) {
#pragma unroll
                    for (int e = 0; e < U; ++e) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], off);
                }
                if (j == 0) {
#pragma unroll
                    for (int e = 0; e < U; ++e) if (e < n) ys[(i + e) * P + p] = fmaf(Dh, xv[e], acc[e]);
                }
            };
            int i = 0;
            for (; i + U <= tc; i += U) tokens(i, U);
            if (i < tc) tokens(i, tc - i);
            __syncthreads();
        }
        if (!rev && a.ssm_out) {
            float *ho = a.ssm_out + (((int64_t)b * a.H + h) * P + p) * N;
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                *reinterpret_cast<float4 *>(ho + (q * LPC + j) * 4) =
                    make_float4(hst[4 * q], hst[4 * q + 1], hst[4 * q + 2], hst[4 * q + 3]);
        }
    }
    finish(nchunks - 1, tid >> 5, blockDim.x >> 5, tid & 31);    // last chunk: everybody (the loop's last barrier made y visible)
}

// The in_proj output [2 B][L][d_in_proj] in boxes of `rows` x P channels, no swizzle.
bool make_map_rows(CUtensorMap *m, const ScanArgs &a, int rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t es = es_of(a), d[3] = {(cuuint64_t)a.d_in_proj, (cuuint64_t)a.L, (cuuint64_t)2 * a.B}, st[2] = {a.d_in_proj * es, a.L * a.d_in_proj * es};
    const cuuint32_t b[3] = {(cuuint32_t)a.P, (cuuint32_t)rows, 1}, e[3] = {1, 1, 1};
    return fn(m, a.dtype == DM_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void *>(a.zx), d, st, b, e,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

typedef void (*Kern)(const CUtensorMap, const CUtensorMap, const ScanArgs, const int, const int, const int, const float *, int *);
template <typename T> Kern kernel_for(int P, int N) {
    switch (N) {
        case 16: return P == 32 ? scan_seq_kernel<T, 32, 16> : scan_seq_kernel<T, 64, 16>;
        case 32: return P == 32 ? scan_seq_kernel<T, 32, 32> : scan_seq_kernel<T, 64, 32>;
        case 64: return P == 32 ? scan_seq_kernel<T, 32, 64> : scan_seq_kernel<T, 64, 64>;
        case 128: return P == 32 ? scan_seq_kernel<T, 32, 128> : scan_seq_kernel<T, 64, 128>;
        case 256: return P == 32 ? scan_seq_kernel<T, 32, 256> : scan_seq_kernel<T, 64, 256>;
        default: return nullptr;
    }
}

}  // namespace

size_t scan_seq_workspace_bytes(const ScanArgs &a) {
    return align_up((size_t)2 * a.B * a.L * 2 * a.N * sizeof(float));      // B', C' of both directions, fp32
}

cudaError_t scan_sequential(const ScanArgs &a, void *ws, cudaStream_t s) {
    if (!ws) return cudaErrorInvalidValue;
    if (a.N % 16 || a.P % 32) return cudaErrorNotSupported;
    if (a.P != 32 && a.P != 64) return cudaErrorNotSupported;
    // 16-byte rows for TMA: true of every workspace and configuration the entry points let through
    if ((int64_t)a.d_in_proj * es_of(a) % 16 || (int64_t)a.d_inner * es_of(a) % 16 || (int64_t)a.conv_ch * es_of(a) % 16) return cudaErrorNotSupported;
    const int ndir = (a.dir_mask == DM_DIR_BOTH) ? 2 : 1;
    const int dir0 = (a.dir_mask == DM_DIR_REV) ? 1 : 0;
    int TC = a.chunk > 0 ? a.chunk : 32;
    if (TC > a.L) TC = a.L;
    if (TC > 64) TC = 64;                               // one preparing thread per token's step size
    size_t smem;
    for (;;) {
        smem = SeqSmem{TC, a.P, a.N, (int)es_of(a)}.total();
        if (smem <= 200 * 1024 || TC == 1) break;
        TC = (TC + 1) / 2;
    }
    const Kern kern = a.dtype == DM_BF16 ? kernel_for<__nv_bfloat16>(a.P, a.N) : kernel_for<float>(a.P, a.N);
    if (!kern) return cudaErrorNotSupported;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    CUtensorMap mx, mz;
    if (!make_map_rows(&mx, a, TC + 3) || !make_map_rows(&mz, a, TC)) return cudaErrorInvalidValue;
    int *status = device_status_ptr();
    if (!status) return cudaErrorUnknown;
    float *bc = static_cast<float *>(ws);
    const int tasks = (a.L + BC_ROWS - 1) / BC_ROWS * 2 * a.N, bt = tasks >= 256 * sm_count() ? 256 : 64;        // small CTAs while they do not fill the GPU
    dim3 pgrid((tasks + bt - 1) / bt, a.B, ndir);
    e = a.dtype == DM_BF16 ? launch_chain(bc_prep_kernel<__nv_bfloat16>, pgrid, bt, 0, s, 0, a, dir0, bc) : launch_chain(bc_prep_kernel<float>, pgrid, bt, 0, s, 0, a, dir0, bc);
    if (e != cudaSuccess) return e;
    dim3 grid(a.H, ndir, a.B);
    chain_spread((int64_t)pgrid.x * pgrid.y * pgrid.z, (int64_t)a.H * ndir * a.B, sm_count());
    return launch_chain(kern, grid, a.P * lanes_per_channel(a.N) + loaders(a.P, a.N), smem, s, 0, mx, mz, a, dir0, TC, scan_selftest_withheld() ? 2 : -1, bc, status);
}

}  // namespace dm
