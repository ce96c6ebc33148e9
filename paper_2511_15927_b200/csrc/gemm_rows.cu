// The GEMM for up to 128 rows (decoding a few sequences): such a product is a read of its weights, so the roles are swapped -- a tile is 128 rows
// of the weight matrix (the M side of tcgen05.mma) times all the tokens (its N side, 16 to 128), D^T = B A^T -- and what matters is that
// every SM has weight bytes in flight all the time.  Where the tiles are few they are cut along K over the CTAs of a cluster; the partial sums go to their owner's shared memory
// (each CTA of the cluster owns a share of the tokens), which adds them, applies the epilogue and stores them: lanes are
// consecutive output columns.  sum: the cluster's CTAs are halves over two products (both directions' out_proj) that are added with each product's row scale.
// Weights from HBM, with tokens as the M side and 128 x 128 tiles before: 32 x 16112 x 1920 18.2 -> 16.3 us, 32 x 1920 x 3840 20.2 -> 8.5 us, 32 x 50304 x 1920
// 50.6 -> 37.1 us (5.2 TB/s).  Inside a pass over 24 layers (one sequence, hybrid), where every kernel's instructions have left the chip since its last launch: 942 us, 925 us with
// the weights marked as read once (the instructions then stay in L2), 902 us with a warp that runs the epilogue's code ahead of time, 849 us with 126 uncut tiles
// in place of 252 halves of K (the exchange costs 2 us and a CTA already fills its SM's share of the bandwidth).
//
// Warp 0 issues the TMA loads, warp 1 the MMAs, the next EW (4 or 8) are the epilogue and a last one brings its code: one TMEM lane quarter each, tokens shared out between the two
// warps of a quarter.  Waits and abort as in gemm_pair.cu: every mbarrier wait is bounded, and the CTAs of a cluster leave together.
#include <array>

#include "gemm_epi.cuh"

namespace dm {
namespace {

using namespace tc;

constexpr int BF = 128, BK = 64, MAX_STAGES = 8, MAX_CS = 8;
constexpr uint32_t W_BYTES = BF * BK * 2;

struct __align__(8) Bars {
    uint64_t full[MAX_STAGES], empty[MAX_STAGES], done;
    uint32_t tmem_base;
    int abort;
    float scale[2][128];           // row scale of this CTA's tokens, per product
    float red[4][128];             // sums of squares of 32 columns each
};

struct RowsArgs {
    EpiArgs p[2];
    int sum, cs, ks;               // CTAs per cluster, K shares per product
    int nt, stages, tiles_n;       // nt: tokens rounded up to 16
    uint32_t tmem_cols;
};

__device__ __forceinline__ void st_cluster_f32(uint32_t addr, float v) { asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory"); }

// G tokens from t on (n of them exist), one output column: bias, activation, gate, residual, output, the next norm's input.  What does not apply is skipped
// for all of them at once, and loads come before the arithmetic: a warp has its scheduler almost to itself here, an instruction costs about six clocks.
template <int G>
__device__ __forceinline__ void emit(const EpiArgs &ep, int t, int n, int col, bool in, float bias, float uw, float (&v)[G]) {
    if (!in) {
#pragma unroll
        for (int g = 0; g < G; ++g) v[g] = 0.f;
        return;
    }
    float add[G];
    if (ep.addend) {
        const float *p = ep.addend + (int64_t)t * ep.ld_add + col;
#pragma unroll
        for (int g = 0; g < G; ++g, p += ep.ld_add) add[g] = g < n ? *p : 0.f;
    }
    if (ep.col_bias) {
#pragma unroll
        for (int g = 0; g < G; ++g) v[g] += bias;
    }
    if (col < ep.silu_cols) {
#pragma unroll
        for (int g = 0; g < G; ++g) { const float hv = 0.5f * v[g]; v[g] = fmaf(hv, tanh_fast(hv), hv); }      // SiLU(v) = v/2 + v/2 tanh(v/2)
    }
    if (ep.gelu) {
#pragma unroll
        for (int g = 0; g < G; ++g) { const float x = v[g], hx = 0.5f * x; v[g] = fmaf(hx, tanh_fast(0.7978845608028654f * fmaf(0.044715f * x, x * x, x)), hx); }
    }
    if (ep.col_scale) {
        float cs[G];
#pragma unroll
        for (int g = 0; g < G; ++g) cs[g] = g < n ? __ldg(ep.col_scale + (int64_t)((t + g) / ep.cs_rows) * ep.ld_cs + col) : 1.f;
#pragma unroll
        for (int g = 0; g < G; ++g) v[g] *= cs[g];
    }
    if (ep.addend) {
#pragma unroll
        for (int g = 0; g < G; ++g) v[g] += add[g];
    }
    if (ep.c_is_f32) {
        float *p = static_cast<float *>(ep.C) + (int64_t)t * ep.ldc + col;
#pragma unroll
        for (int g = 0; g < G; ++g, p += ep.ldc) if (g < n) *p = v[g];
    } else {
        __nv_bfloat16 *p = static_cast<__nv_bfloat16 *>(ep.C) + (int64_t)t * ep.ldc + col;
#pragma unroll
        for (int g = 0; g < G; ++g, p += ep.ldc) if (g < n) *p = __float2bfloat16_rn(v[g]);
    }
    if (ep.u) {
        __nv_bfloat16 *p = ep.u + (int64_t)t * ep.N + col;
#pragma unroll
        for (int g = 0; g < G; ++g, p += ep.N) if (g < n) *p = __float2bfloat16_rn(v[g] * uw);
    }
}

template <int EW>
__global__ void __launch_bounds__(96 + 32 * EW, EW == 4 ? 2 : 1)
gemm_rows_kernel(const __grid_constant__ CUtensorMap map_x0, const __grid_constant__ CUtensorMap map_w0,
                 const __grid_constant__ CUtensorMap map_x1, const __grid_constant__ CUtensorMap map_w1,
                 const __grid_constant__ RowsArgs ra, int *status) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const int nt = ra.nt, S = ra.stages, cs = ra.cs, tpc = nt / cs;
    const uint32_t stage = W_BYTES + (uint32_t)nt * (BK * 2);
    float *recv = reinterpret_cast<float *>(smem + S * stage);               // [source CTA][own token][BF]  (clusters only)
    Bars *bars = reinterpret_cast<Bars *>(smem + S * stage + (cs > 1 ? (uint32_t)nt * BF * 4 : 0u));
    volatile int *abort_flag = &bars->abort;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = cs > 1 ? (int)cluster_ctarank() : 0, cid = blockIdx.x / cs, tile = cid % ra.tiles_n;
    const int prod = ra.sum ? rank / ra.ks : cid / ra.tiles_n, kr = rank % ra.ks;
    const EpiArgs &ep = ra.p[ra.sum ? 1 : prod];                             // output, addend, ...
    if (ep.m_dev) pdl_wait();                                                // (the row count comes from a kernel before this one)
    const int M = ep.m_dev ? min(ep.M, max(0, *ep.m_dev - ep.m_off)) : ep.M;
    const int kblocks = (ep.K + BK - 1) / BK, kb0 = kr * kblocks / ra.ks, nk = (kr + 1) * kblocks / ra.ks - kb0;
    const int n0 = tile * BF;

    if (threadIdx.x == 0) {
        for (int i = 0; i < S; ++i) { mbar_init(&bars->full[i], 1); mbar_init(&bars->empty[i], 1); }
        mbar_init(&bars->done, 1);
        bars->abort = 0;
        mbar_fence_init();
    }
    if (threadIdx.x == 64) { prefetch_map(prod ? &map_w1 : &map_w0); prefetch_map(prod ? &map_x1 : &map_x0); }
    if (warp == 1) tmem_alloc(&bars->tmem_base, ra.tmem_cols);
    __syncwarp();
    fence_before();
    if (cs > 1) cluster_sync(); else __syncthreads();                        // (no CTA of a cluster writes to one that has not started)
    fence_after();
    const uint32_t tmem = bars->tmem_base;

    bool ok = true;
    if (warp == 0) {
        const bool leader = elect_one();
        const CUtensorMap *mx = prod ? &map_x1 : &map_x0, *mw = prod ? &map_w1 : &map_w0;
        const uint64_t once = l2_evict_first();
        int s = 0;
        uint32_t ph = 1;
        // the weights of the first stages are on their way before the kernel before this one has finished
        const int ahead = min(S, nk);
        if (leader)
            for (int i = 0; i < ahead; ++i) {
                mbar_expect_tx(&bars->full[i], stage);
                tma_load_2d_hint(smem + i * stage, mw, (kb0 + i) * BK, n0, &bars->full[i], once);
            }
        __syncwarp();
        pdl_wait();
        pdl_trigger();
        for (int i = 0; i < nk; ++i) {
            if (!(ok = mbar_wait(&bars->empty[s], ph, abort_flag, status))) break;
            if (leader) {
                uint8_t *sw = smem + s * stage;
                if (i >= ahead) {
                    mbar_expect_tx(&bars->full[s], stage);
                    tma_load_2d_hint(sw, mw, (kb0 + i) * BK, n0, &bars->full[s], once);
                }
                tma_load_2d(sw + W_BYTES, mx, (kb0 + i) * BK, 0, &bars->full[s]);
            }
            __syncwarp();
            if (++s == S) { s = 0; ph ^= 1; }
        }
        if (!ok) sleep_ns(100000000ull);                                     // aborting: the loads already issued get time to land
    } else if (warp == 1) {
        const bool leader = elect_one();
        pdl_wait();                                                          // (the limit of the waits below counts from here)
        const uint32_t idesc = idesc_bf16(BF, nt, 0, 0), d0 = desc_lo_k(smem_u32(smem));
        int s = 0;
        uint32_t ph = 0;
        for (int i = 0; i < nk; ++i) {
            if (!(ok = mbar_wait(&bars->full[s], ph, abort_flag, status))) break;
            fence_after();
            const uint32_t dw = d0 + s * (stage >> 4), dx = dw + (W_BYTES >> 4);
            if (leader) {
#pragma unroll
                for (int k = 0; k < BK / 16; ++k) {
                    if (i == 0 && k == 0) umma_ss<0>(tmem, dw, dx, idesc); else umma_ss<1>(tmem, dw + 2 * k, dx + 2 * k, idesc);
                }
                umma_commit(&bars->empty[s]);
                if (i == nk - 1) umma_commit(&bars->done);
            }
            __syncwarp();
            if (++s == S) { s = 0; ph ^= 1; }
        }
    } else {
        const int ew = warp - 2, q = warp & 3, f = q * 32 + lane, col = n0 + f;      // this thread's output column of the tile
        const bool in = col < ep.N;
        const float bias = in && ep.col_bias ? ep.col_bias[col] : 0.f;
        const float uw = in && ep.u ? __bfloat162float(ep.u_w[col]) : 0.f;
        // The last warp does the same without a token (real = false: no wait, no load of activations, no store), as soon as the CTA starts: it brings the instructions.  They come from memory --
        // the weights of a pass have gone through L2 since the last launch --, all SMs wait for each line of them, and after the products nothing would hide that.
        const bool real = ew < EW;
        {
            if (real) pdl_wait();
            const int Mp = real ? M : 0;
            // row scales of this CTA's tokens, while the products run: a warp per (product, token)
            const int first = ra.sum ? 0 : prod, items = (ra.sum ? 2 : 1) * tpc;
            for (int i = real ? ew : items - 1; i < items; i += EW) {
                const int pi = i / tpc, tl = i - pi * tpc, t = rank * tpc + tl;
                const EpiArgs &e = ra.p[first + pi];
                float sc = 1.f;
                if (t < Mp && e.row_scale) sc = e.row_scale[t];
                else if (e.rs_ssq) {
                    float v = 0.f;
                    for (int j = lane; j < e.rs_n; j += 32) v += t < Mp ? __ldg(e.rs_ssq + (int64_t)t * e.rs_n + j) : 0.f;
                    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
                    sc = rsqrtf(v * e.rs_inv + e.rs_eps);
                }
                if (lane == 0 && real) bars->scale[pi][tl] = sc;
            }
            if (real) {
                named_sync(1, 32 * EW);                                      // the scales are there for all of these warps
                ok = __all_sync(0xffffffffu, mbar_wait(&bars->done, 0, abort_flag, status));
                fence_after();
            }
            if (cs > 1) {                                                    // this CTA's partial sums to the owners of the tokens
                for (int c0 = real ? 16 * (ew >> 2) : 0; c0 < nt && ok; c0 += 4 * EW) {
                    uint32_t r[16];
                    tmem_ld_x16(tmem + ((uint32_t)(q * 32) << 16) + c0, r);
                    tmem_wait_ld();
                    int owner = c0 / tpc, tl = c0 - owner * tpc;
                    uint32_t dst = cluster_addr(recv + (rank * tpc) * BF + f, owner);
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        if (real) st_cluster_f32(dst + tl * (BF * 4), __uint_as_float(r[j]));
                        if (++tl == tpc && owner + 1 < cs) { tl = 0; ++owner; dst = cluster_addr(recv + (rank * tpc) * BF + f, owner); }
                    }
                    if (!real) break;
                }
                __syncwarp();
                if (real) cluster_sync();                                    // every partial sum has arrived; nobody's shared memory is written any more
            }
            // ------------------------------------------------------------ the CTA's tokens: sum, epilogue, store
            const bool go = !real || !*abort_flag;
            auto squares = [&](const auto &v, int tl, int n) {               // the next norm's sums over this warp's 32 columns
                if (!ep.u) return;
#pragma unroll
                for (int g = 0; g < (int)(sizeof(v) / sizeof(float)); ++g) {
                    float ss = v[g] * v[g];
#pragma unroll
                    for (int off = 16; off > 0; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
                    if (lane == 0 && g < n && real) bars->red[q][tl + g] = ss;
                }
            };
            if (cs == 1) {
                for (int c0 = real ? 16 * (ew >> 2) : 0; c0 < nt && c0 < M && go; c0 += 4 * EW) {
                    uint32_t r[16];
                    float v[16];
                    tmem_ld_x16(tmem + ((uint32_t)(q * 32) << 16) + c0, r);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]) * bars->scale[0][c0 + j];
                    emit(ep, c0, min(16, Mp - c0), col, in, bias, uw, v);
                    squares(v, c0, 16);
                    if (!real) break;
                }
            } else {
                const int half = ra.sum ? ra.ks : cs;                        // sources [0, half) are product 0 (or the only one)
                constexpr int G = 4;
                for (int tl = real ? G * (ew >> 2) : 0; tl < tpc && go; tl += G * (EW / 4)) {
                    const int t = rank * tpc + tl;
                    if (t >= M) break;
                    float v[G] = {};
#pragma unroll
                    for (int r = 0; r < MAX_CS; ++r) {
                        if (r >= cs) break;
#pragma unroll
                        for (int g = 0; g < G; ++g) {
                            const int tg = min(tl + g, tpc - 1);
                            v[g] = fmaf(recv[(r * tpc + tg) * BF + f], bars->scale[r < half ? 0 : 1][tg], v[g]);
                        }
                    }
                    emit(ep, t, min(min(G, tpc - tl), Mp - t), col, in, bias, uw, v);
                    squares(v, tl, tpc - tl);
                    if (!real) break;
                }
            }
            if (ep.u && go) {
                if (real) named_sync(1, 32 * EW);
                const int parts = (ep.N + 63) / 64;
                for (int i = real ? threadIdx.x - 64 : lane; i < 2 * tpc; i += 32 * EW) {  // (half of the tile, token)
                    const int hf = i / tpc, tl = i - hf * tpc, t = rank * tpc + tl;
                    if (t < Mp && n0 / 64 + hf < parts) ep.u_ssq[(int64_t)t * parts + n0 / 64 + hf] = bars->red[2 * hf][tl] + bars->red[2 * hf + 1][tl];
                }
            }
        }
    }
    if ((warp < 2 || warp == 2 + EW) && cs > 1) {
        __syncwarp();
        cluster_sync();                                                      // (the epilogue warps' turn is after their sums are sent)
    }
    __syncwarp();
    fence_before();
    __syncthreads();
    if (warp == 1) {
        fence_after();
        tmem_dealloc(tmem, ra.tmem_cols);
    }
}

// The same for more uncut tiles than two to an SM (the vocabulary's projection): every CTA takes each gridDim.x-th tile, with two accumulator buffers, so that a tile's epilogue runs
// under the next one's products and the ring of stages never empties.  Bound by the weights' way from HBM.  A CTA per tile / this kernel: 128 x 50304 x 1024 37.8 / 26.2 us, 128 x 50304 x 2048
// 51.3 / 41.2, 64 x 50304 x 1024 28.1 / 23.7, 16 rows 24.0 / 20.9 (4.9 TB/s).  A kernel of its own: as an option of the one above its loop cost the launches of a decoding pass 1 to 2 us each.
// Warps 0 and 1 as above, the next EW are the epilogue.  (No next norm's input: nothing that wide is normed.)
struct __align__(8) LoopBars {
    uint64_t full[MAX_STAGES], empty[MAX_STAGES], done[2], drained[2];
    uint32_t tmem_base;
    int abort;
    float scale[2][128];           // row scale of every token, per product
};

template <int EW>
__global__ void __launch_bounds__(64 + 32 * EW, EW == 4 ? 2 : 1)
gemm_rows_loop_kernel(const __grid_constant__ CUtensorMap map_x0, const __grid_constant__ CUtensorMap map_w0,
                      const __grid_constant__ CUtensorMap map_x1, const __grid_constant__ CUtensorMap map_w1,
                      const __grid_constant__ RowsArgs ra, const int items, int *status) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const int nt = ra.nt, S = ra.stages, nprob = items / ra.tiles_n;
    const uint32_t stage = W_BYTES + (uint32_t)nt * (BK * 2);
    LoopBars *bars = reinterpret_cast<LoopBars *>(smem + S * stage);
    volatile int *abort_flag = &bars->abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const EpiArgs &e0 = ra.p[0];                                             // (sizes are common to both products)
    if (e0.m_dev) pdl_wait();                                                // (the row count comes from a kernel before this one)
    const int M = e0.m_dev ? min(e0.M, max(0, *e0.m_dev - e0.m_off)) : e0.M;
    const int kblocks = (e0.K + BK - 1) / BK;

    if (threadIdx.x == 0) {
        for (int i = 0; i < S; ++i) { mbar_init(&bars->full[i], 1); mbar_init(&bars->empty[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&bars->done[i], 1); mbar_init(&bars->drained[i], EW); }
        bars->abort = 0;
        mbar_fence_init();
    }
    if (threadIdx.x == 64) { prefetch_map(&map_w0); prefetch_map(&map_x0); }
    if (warp == 1) tmem_alloc(&bars->tmem_base, 2 * ra.tmem_cols);
    __syncwarp();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = bars->tmem_base;

    bool ok = true;
    if (warp == 0) {
        const bool leader = elect_one();
        const uint64_t once = l2_evict_first();
        int s = 0;
        uint32_t ph = 1;
        // the weights of the first stages are on their way before the kernel before this one has finished
        const int ahead = min(S, kblocks);
        if (leader)
            for (int i = 0; i < ahead; ++i) {
                mbar_expect_tx(&bars->full[i], stage);
                tma_load_2d_hint(smem + i * stage, (int)blockIdx.x < ra.tiles_n ? &map_w0 : &map_w1, i * BK, (int)blockIdx.x % ra.tiles_n * BF, &bars->full[i], once);
            }
        __syncwarp();
        pdl_wait();
        pdl_trigger();
        for (int item = blockIdx.x; item < items && ok; item += gridDim.x) {
            const bool second = item >= ra.tiles_n;
            const CUtensorMap *mx = second ? &map_x1 : &map_x0, *mw = second ? &map_w1 : &map_w0;
            const int n0 = (second ? item - ra.tiles_n : item) * BF;
            for (int i = 0; i < kblocks; ++i) {
                if (!(ok = mbar_wait(&bars->empty[s], ph, abort_flag, status))) break;
                if (leader) {
                    uint8_t *sw = smem + s * stage;
                    if (item != (int)blockIdx.x || i >= ahead) {
                        mbar_expect_tx(&bars->full[s], stage);
                        tma_load_2d_hint(sw, mw, i * BK, n0, &bars->full[s], once);
                    }
                    tma_load_2d(sw + W_BYTES, mx, i * BK, 0, &bars->full[s]);
                }
                __syncwarp();
                if (++s == S) { s = 0; ph ^= 1; }
            }
        }
        if (!ok) sleep_ns(100000000ull);                                     // aborting: the loads already issued get time to land
    } else if (warp == 1) {
        const bool leader = elect_one();
        pdl_wait();                                                          // (the limit of the waits below counts from here)
        const uint32_t idesc = idesc_bf16(BF, nt, 0, 0), d0 = desc_lo_k(smem_u32(smem));
        int s = 0, n = 0;
        uint32_t ph = 0;
        for (int item = blockIdx.x; item < items && ok; item += gridDim.x, ++n) {
            if (n > 1 && !(ok = mbar_wait(&bars->drained[n & 1], ((n >> 1) - 1) & 1, abort_flag, status))) break;
            fence_after();
            const uint32_t d_tmem = tmem + (n & 1) * ra.tmem_cols;
            for (int i = 0; i < kblocks; ++i) {
                if (!(ok = mbar_wait(&bars->full[s], ph, abort_flag, status))) break;
                fence_after();
                const uint32_t dw = d0 + s * (stage >> 4), dx = dw + (W_BYTES >> 4);
                if (leader) {
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k) {
                        if (i == 0 && k == 0) umma_ss<0>(d_tmem, dw, dx, idesc); else umma_ss<1>(d_tmem, dw + 2 * k, dx + 2 * k, idesc);
                    }
                    umma_commit(&bars->empty[s]);
                    if (i == kblocks - 1) umma_commit(&bars->done[n & 1]);
                }
                __syncwarp();
                if (++s == S) { s = 0; ph ^= 1; }
            }
        }
    } else {
        const int ew = warp - 2, q = warp & 3, f = q * 32 + lane;             // f: this thread's output column of the tile
        pdl_wait();
        for (int i = ew; i < nprob * nt; i += EW) {                          // row scales, while the products run: a warp per (product, token)
            const int pi = i / nt, t = i - pi * nt;
            const EpiArgs &e = ra.p[pi];
            float sc = 1.f;
            if (t < M && e.row_scale) sc = e.row_scale[t];
            else if (e.rs_ssq) {
                float v = 0.f;
                for (int j = lane; j < e.rs_n; j += 32) v += t < M ? __ldg(e.rs_ssq + (int64_t)t * e.rs_n + j) : 0.f;
                for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
                sc = rsqrtf(v * e.rs_inv + e.rs_eps);
            }
            if (lane == 0) bars->scale[pi][t] = sc;
        }
        named_sync(1, 32 * EW);                                              // the scales are there for all of these warps
        int n = 0;
        for (int item = blockIdx.x; item < items; item += gridDim.x, ++n) {
            const int prod = item >= ra.tiles_n ? 1 : 0, col = (item - prod * ra.tiles_n) * BF + f;
            const EpiArgs &ep = ra.p[prod];
            const bool in = col < ep.N;
            const float bias = in && ep.col_bias ? ep.col_bias[col] : 0.f;
            if (!__all_sync(0xffffffffu, mbar_wait(&bars->done[n & 1], (n >> 1) & 1, abort_flag, status))) break;
            fence_after();
            for (int c0 = 16 * (ew >> 2); c0 < nt && c0 < M; c0 += 4 * EW) {
                uint32_t r[16];
                float v[16];
                tmem_ld_x16(tmem + (n & 1) * ra.tmem_cols + ((uint32_t)(q * 32) << 16) + c0, r);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]) * bars->scale[prod][c0 + j];
                emit(ep, c0, min(16, M - c0), col, in, bias, 0.f, v);
            }
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->drained[n & 1]);
        }
    }
    __syncwarp();
    fence_before();
    __syncthreads();
    if (warp == 1) {
        fence_after();
        tmem_dealloc(tmem, 2 * ra.tmem_cols);
    }
}

}  // namespace

// Clusters of 2^i CTAs that are resident at once with one CTA per SM (of eight: 15 on 148 SMs; the GPU's parts hold uneven numbers of SMs).
static int resident_clusters(int cs) {
    static const std::array<int, 4> n = [] {
        std::array<int, 4> r{};
        const int smem = 226 * 1024;
        if (cudaFuncSetAttribute(gemm_rows_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return r;
        for (int i = 0; i < 4; ++i) {
            cudaLaunchConfig_t cfg{};
            cfg.gridDim = dim3(1 << i); cfg.blockDim = dim3(352); cfg.dynamicSmemBytes = smem;
            cudaLaunchAttribute at;
            at.id = cudaLaunchAttributeClusterDimension;
            at.val.clusterDim.x = 1 << i; at.val.clusterDim.y = 1; at.val.clusterDim.z = 1;
            cfg.attrs = &at; cfg.numAttrs = 1;
            if (cudaOccupancyMaxActiveClusters(&r[i], gemm_rows_kernel<8>, &cfg) != cudaSuccess) r[i] = 0;
        }
        return r;
    }();
    return n[cs == 8 ? 3 : cs == 4 ? 2 : cs == 2 ? 1 : 0];
}

// b == NULL: one product; sum: s_a A_a B_a^T + s_b A_b B_b^T into b's output; else two products of equal sizes side by side.
cudaError_t gemm_rows_launch(const GemmArgs &a, const GemmArgs *b, bool sum, cudaStream_t s) {
    RowsArgs ra{};
    ra.p[0] = epi_of(a);
    ra.p[1] = b ? epi_of(*b) : ra.p[0];
    ra.sum = sum ? 1 : 0;
    ra.nt = (a.M + 15) / 16 * 16;
    ra.tiles_n = (a.N + BF - 1) / BF;
    const int items = ra.tiles_n * (b && !sum ? 2 : 1), kblocks = (a.K + BK - 1) / BK, per = sum ? 2 : 1;      // per: products of a cluster
    const int slots = (ra.nt <= 64 ? 2 : 1) * sm_count();                    // (more tokens: the partial sums of a CTA take 40 KB and more)
    // K shares: powers of two while less than three fifths of the SMs have a CTA (beyond that the exchange costs more than the idle SMs: 90 and 126 CTAs beat 180 and 252), the grid fits
    // the GPU at once and a share keeps four steps
    int ks = 1;
    while (items * per * ks < sm_count() * 3 / 5 && 2 * ks * per <= MAX_CS && items * per * 2 * ks <= slots && kblocks >= 8 * ks && ra.nt % (2 * ks * per) == 0) ks *= 2;
    uint32_t cols = 32;
    while (cols < (uint32_t)ra.nt) cols *= 2;
    ra.tmem_cols = cols;
    // Two CTAs per SM where not all clusters are resident with one and the stages stay at least three deep (128 x 25000 x 1920: 25.5 us, 32.4 in two rounds of one CTA; four where tiles are taken
    // in turn: 128 x 50304 x 2048 41.2 us with one CTA of seven stages per SM, 44.5 with two of three);
    // else one CTA may use all of the SM, with twice the epilogue warps, and a cut of K that does not fit one round is halved.  (16 clusters of eight CTAs, the summed
    // out_proj of d_model 2048, ran in two rounds: 24 layers of 32 tokens 1003 -> 846 us, one layer of 100 tokens 53 -> 47 us.)
    const size_t stage = W_BYTES + (size_t)ra.nt * BK * 2;
    const bool loop = ks * per == 1 && items > 2 * sm_count() && !a.u && !(b && b->u);
    size_t fixed;
    bool two;
    for (;; ks /= 2) {
        ra.ks = ks;
        ra.cs = ks * per;
        fixed = (ra.cs > 1 ? (size_t)ra.nt * BF * 4 : 0) + (loop ? sizeof(LoopBars) : sizeof(Bars)) + 1024;
        const bool fits = items <= resident_clusters(ra.cs);
        two = !fits && fixed + (loop ? 4 : 3) * stage <= 113 * 1024;
        if (fits || two || ks == 1) break;
    }
    const int ctas = loop ? (two ? 2 : 1) * sm_count() : items * ra.cs;
    const int stages = (int)(((two ? 113 : 226) * 1024 - fixed) / stage);
    ra.stages = stages > MAX_STAGES ? MAX_STAGES : stages;
    const size_t smem = fixed + ra.stages * stage;
    CUtensorMap mx[2], mw[2];
    if (!make_map_2d(&mx[0], a.A, a.M, a.K, a.lda, ra.nt) || !make_map_2d(&mw[0], a.B, a.N, a.K, a.ldb, BF)) return cudaErrorInvalidValue;
    mx[1] = mx[0]; mw[1] = mw[0];
    if (b && (!make_map_2d(&mx[1], b->A, b->M, b->K, b->lda, ra.nt) || !make_map_2d(&mw[1], b->B, b->N, b->K, b->ldb, BF))) return cudaErrorInvalidValue;
    int *status = device_status_ptr();
    if (!status) return cudaErrorUnknown;
    if (loop) {
        auto kern = two ? gemm_rows_loop_kernel<4> : gemm_rows_loop_kernel<8>;
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
        return e != cudaSuccess ? e : launch_chain(kern, dim3(ctas), dim3(two ? 192 : 320), smem, s, 0, mx[0], mw[0], mx[1], mw[1], ra, items, status);
    }
    auto kern = two ? gemm_rows_kernel<4> : gemm_rows_kernel<8>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
    if (e != cudaSuccess) return e;
    return launch_chain(kern, dim3(ctas), dim3(two ? 224 : 352), smem, s, ra.cs, mx[0], mw[0], mx[1], mw[1], ra, status);
}

}  // namespace dm
