// Shared by the chunked scan kernels (scan_ssd.cu, scan_step.cu): arguments, the arithmetic of conv and step size, mma.sync helpers.
#pragma once

#include "dm_internal.h"
#include "tc_ptx.cuh"

namespace dm {
namespace ssd {

using namespace tc;

constexpr int N = 128;                // d_state (a smaller one is zero-padded)
constexpr int Q = 128;                // tokens per chunk
constexpr int QB = 32;                // tokens per sub-chunk of the short-block and narrow-state kernels
constexpr int PREP_THREADS = 512;     // threads of a prep CTA
constexpr int NLD = N + 8;            // row pitch (elements) of C', B' and state tiles: 16-byte rows, conflict-free ldmatrix

struct SsdArgs {
    int B, L, H, d_inner, d_in_proj, conv_ch, k, flags, nch, Lp;
    int Nr;                      // d_state of the model (<= N); B', C' and the state are zero-padded to N
    int Pr;                      // headdim of the model: P, or P / 2 (the CTA then carries the next head's channels as unused padding)
    int zx_tied;                 // both directions read the in_proj output of direction 0 (shared projections)
    __nv_bfloat16 *g;            // [2][B*L][d_inner] gated output (written with plain stores when Pr < P, else through map_g)
    const __nv_bfloat16 *zx;
    float *ssq;                  // [2][B*L][ssq_parts] sums of squares of the gated output, or NULL
    int ssq_parts;               // H, or (narrow-state kernel) one per 32 channels
    const float *dA;             // [2][B][H][2][Lp]: Lambda, Lambda' (log2 units)
    const float *ssm_in; float *ssm_out;
    const __nv_bfloat16 *conv_in;  // [B][k-1][conv_ch] pre-conv rows before the first token (left-to-right layer), or NULL
    ScanDir dir[2];
};

__device__ __forceinline__ float silu_fast(float v) { const float hv = 0.5f * v; return fmaf(hv, tanh_fast(hv), hv); }     // SiLU(v) = v/2 + v/2 tanh(v/2)
// Arithmetic shared by the two forms of the prep work (the launch of its own below and the prep role inside the scan
// launch), so that both give the same bits.
// conv + SiLU of one bf16 channel pair: r[m] = the pre-conv pair m steps back in time, wl[e][m] its weight
__device__ __forceinline__ uint32_t prep_conv_pair(const float (&wl)[2][4], const float (&bias)[2], const uint32_t (&r)[4]) {
    float v0 = bias[0], v1 = bias[1];
#pragma unroll
    for (int m = 3; m >= 0; --m) {
        v0 = fmaf(wl[0][m], bf16_lo(r[m]), v0);
        v1 = fmaf(wl[1][m], bf16_hi(r[m]), v1);
    }
    return pack_bf16(silu_fast(v0), silu_fast(v1));
}
// softplus(dt + bias) = max(v, 0) + log1p(exp(-|v|)) with the fast exponential and logarithm: log1p by its series where 1 + e
// would round e away (e < 2^-7: error below e^4 / 4), by log(1 + e) elsewhere.  Relative error of Delta about 1e-6, far inside
// what the bf16 path needs.
__device__ __forceinline__ float prep_delta(float dt, float dt_bias) {
    const float v = dt + dt_bias;
    const float e = __expf(-fabsf(v));
    const float l = e < 0.0078125f ? e * fmaf(e, fmaf(e, 0.33333334f, -0.5f), 1.f) : __logf(1.f + e);
    return fmaxf(v, 0.f) + l;
}
// One warp, one head, one 128-token chunk: d[e] = Delta of the token 4 lane + e in the direction's time order.
// SUB = false: writes Lambda (inclusive cumulative Delta A in that order, log2 units) of physical chunk row r to dl[r] and Lambda' = Lambda - log2 Delta to dl[Lp + r].
// SUB = true (narrow-state kernel): Lambda starts again at every sub-chunk of QB tokens, and dl holds [physical sub-chunk][Lambda, Lambda'][QB] in time order.
template <bool SUB>
__device__ __forceinline__ void prep_lambda_head(const float (&d)[4], float A_log, bool rev, int lane, float *dl, int Lp) {
    const float Ah = -expf(A_log) * 1.4426950408889634f;
    float cum[4];
    cum[0] = d[0] * Ah; cum[1] = fmaf(d[1], Ah, cum[0]); cum[2] = fmaf(d[2], Ah, cum[1]); cum[3] = fmaf(d[3], Ah, cum[2]);
    float run = cum[3];
    const int at = SUB ? lane & (QB / 4 - 1) : lane;             // this lane's place in its scan
#pragma unroll
    for (int off = 1; off < (SUB ? QB / 4 : 32); off <<= 1) {
        const float up = __shfl_up_sync(0xffffffffu, run, off);
        if (at >= off) run += up;
    }
    const float base = run - cum[3];                             // sum over the lanes before this one
    float lam[4], lamp[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) { lam[e] = base + cum[e]; lamp[e] = lam[e] - __log2f(d[e]); }    // Delta = 0 (padding): Lambda' = +inf
    if (SUB) {
        const int sub = lane / (QB / 4);
        float *p = dl + (rev ? Q / QB - 1 - sub : sub) * 2 * QB + 4 * at;
        *reinterpret_cast<float4 *>(p) = make_float4(lam[0], lam[1], lam[2], lam[3]);
        *reinterpret_cast<float4 *>(p + QB) = make_float4(lamp[0], lamp[1], lamp[2], lamp[3]);
        return;
    }
    const int rlo = rev ? Q - 4 - 4 * lane : 4 * lane;           // lowest physical row of this lane's four
    const float4 v0 = rev ? make_float4(lam[3], lam[2], lam[1], lam[0]) : make_float4(lam[0], lam[1], lam[2], lam[3]);
    const float4 v1 = rev ? make_float4(lamp[3], lamp[2], lamp[1], lamp[0]) : make_float4(lamp[0], lamp[1], lamp[2], lamp[3]);
    *reinterpret_cast<float4 *>(dl + rlo) = v0;
    *reinterpret_cast<float4 *>(dl + Lp + rlo) = v1;
}
// Delta and the cumulative log-decays of heads [h0, h0 + 64) over the chunk that starts at row r0, by a CTA of PREP_THREADS; dsm: [64][Q] floats.
// dA: [seq][H][2][Lp], or [seq][H][Lp / QB][2][QB] with SUB (the same place for a chunk of Q tokens but for the order inside)
template <bool SUB>
__device__ __forceinline__ void prep_decay(const SsdArgs &a, float *__restrict__ dA, int dir, int b, int r0, int h0, float *dsm) {
    const bool rev = dir == 1;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const ScanDir &w = a.dir[dir];
    const int64_t seq = (int64_t)dir * a.B + b;
    {
        const int row = tid & (Q - 1), hg = tid / Q * 16, t = r0 + row, hb = h0 + hg;
        // the dt columns start on a 16-byte boundary (all widths are multiples of 8), and the rows are padded to one
        const __nv_bfloat16 *src = a.zx + (((int64_t)(a.zx_tied ? 0 : dir) * a.B + b) * a.L + t) * a.d_in_proj + a.d_inner + a.conv_ch + hb;
        uint4 v[2] = {make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u)};
#pragma unroll
        for (int i = 0; i < 2; ++i) if (t < a.L && hb + 8 * i < a.H) v[i] = __ldg(reinterpret_cast<const uint4 *>(src) + i);
        float bias[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) bias[j] = hb + j < a.H ? __ldg(w.dt_bias + hb + j) : 0.f;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const uint32_t word = reinterpret_cast<const uint32_t *>(v)[j >> 1];
            const float dt = (j & 1) ? bf16_hi(word) : bf16_lo(word);
            dsm[(hg + j) * Q + row] = t < a.L ? prep_delta(dt, bias[j]) : 0.f;
        }
    }
    __syncthreads();
#pragma unroll 2
    for (int hh = warp; hh < 64; hh += PREP_THREADS / 32) {
        const int h = h0 + hh;
        if (h >= a.H) break;
        const float4 q = *reinterpret_cast<const float4 *>(dsm + hh * Q + (rev ? Q - 4 - 4 * lane : 4 * lane));
        const float d[4] = {rev ? q.w : q.x, rev ? q.z : q.y, rev ? q.y : q.z, rev ? q.x : q.w};
        prep_lambda_head<SUB>(d, __ldg(w.A_log + h), rev, lane, dA + ((seq * a.H + h) * 2) * a.Lp + (SUB ? 2 * r0 : r0), a.Lp);
    }
}
// Eight consecutive bf16 of a read-only array, two to a word; at any address (callers' weight vectors carry no alignment rule)
__device__ __forceinline__ uint4 ld8_bf16(const __nv_bfloat16 *p) {
    if ((reinterpret_cast<uintptr_t>(p) & 15u) == 0) return __ldg(reinterpret_cast<const uint4 *>(p));
    const unsigned short *q = reinterpret_cast<const unsigned short *>(p);
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = (uint32_t)__ldg(q + 2 * i) | ((uint32_t)__ldg(q + 2 * i + 1) << 16);
    return make_uint4(w[0], w[1], w[2], w[3]);
}

}  // namespace ssd

// One block of up to QB tokens per sequence in one launch: see scan_step.cu (which takes 16-byte aligned states and norm weights).
bool scan_step_supports(const ssd::SsdArgs &a);
cudaError_t scan_step(const ssd::SsdArgs &a, int headdim, int ndir, int dir0, cudaStream_t s);
// Sequences of more than two sub-chunks with d_state 16, in chains of `width` channels (scan_narrow_width; heads: of all sequences and directions): see scan_narrow.cu.
// bc: [2][B][L][32] bf16, dl: [2][B][H][Lp / 32][2][32] fp32 of scratch.  The sums of squares do not depend on the width, so that a row's result does not depend on how many others share the
// call: a.ssq_parts is d_inner / 32, or H where heads are as wide as the chains.
bool scan_narrow_shape(int d_state);
int scan_narrow_width(int headdim, int64_t heads, bool skip);
cudaError_t scan_narrow(const ssd::SsdArgs &a, __nv_bfloat16 *bc, float *dl, int ndir, int dir0, int width, cudaStream_t s);

}  // namespace dm
