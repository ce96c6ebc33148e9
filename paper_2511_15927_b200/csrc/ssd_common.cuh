// Shared by the chunked scan kernels (scan_ssd.cu, scan_step.cu): arguments, the arithmetic of conv and step size, mma.sync helpers.
#pragma once

#include "dm_internal.h"
#include "tc_ptx.cuh"

namespace dm {
namespace ssd {

using namespace tc;

constexpr int N = 128;                // d_state (a smaller one is zero-padded)
constexpr int QB = 32;                // tokens per sub-chunk of the short-block kernels
constexpr int NLD = N + 8;            // row pitch (elements) of C', B' and state tiles: 16-byte rows, conflict-free ldmatrix

struct SsdArgs {
    int B, L, H, d_inner, d_in_proj, conv_ch, k, flags, nch, Lp;
    int Nr;                      // d_state of the model (<= N); B', C' and the state are zero-padded to N
    int Pr;                      // headdim of the model: P, or P / 2 (the CTA then carries the next head's channels as unused padding)
    int zx_tied;                 // both directions read the in_proj output of direction 0 (shared projections)
    __nv_bfloat16 *g;            // [2][B*L][d_inner] gated output (written with plain stores when Pr < P, else through map_g)
    const __nv_bfloat16 *zx;
    float *ssq;
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

}  // namespace dm
