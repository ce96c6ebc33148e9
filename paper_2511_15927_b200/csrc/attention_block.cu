// Attention for few queries per sequence (the active block of block-autoregressive decoding, Sec. 4.3): 32 queries of one head against the
// committed prefix in the key/value cache and the block's own keys, which this launch also appends to the cache.
// Bound by reading the cache (2 * d * 2 bytes per key against 4 * 32 * d products): the keys of a (head, sequence) are split over the CTAs of a
// cluster, so that few heads and one sequence still fill the GPU, and each CTA streams its share through a ring of asynchronous 16-byte
// copies.  The 32 x keys products are a quarter of a tcgen05 tile and run on mma.sync instead: eight warps take 16 queries and 16 of a tile's 64 keys
// each, with running maxima of their own, and P goes from the accumulators of Q K^T straight into the A operand of P V.  At the end the warps' and
// then the CTAs' (m, l, O) are combined through shared and distributed shared memory: no second launch, no partials in memory.
// What bounds it now is mma.sync itself: a 16 x 8 x 16 product takes 32 clocks of an SM quarter, 40 of them per 16 keys and head.
// 24 heads of 80, 8192 + 32 keys, block of 32: 30 us for one sequence (149 us on the 128-query kernel, one CTA per head), 79 us for four (150 us).
#include "dm_internal.h"
#include "tc_ptx.cuh"

namespace dm {
namespace {

using namespace tc;

constexpr int BQ = 32, KT = 64, STAGES = 4, NT = 256;
constexpr int WK = KT / 4;                         // keys of a tile per warp: a pair of warps (two times 16 queries) shares them
constexpr int MAX_SPLIT = 8;                       // portable cluster size

template <int DH> struct Smem {
    static constexpr int LD = DH + 8;              // row pitch (bf16): 16-byte rows, conflict-free ldmatrix
    static constexpr uint32_t TILE = KT * LD * 2;  // one K or V tile
    static constexpr uint32_t q = 0, kv = q + BQ * LD * 2, total = kv + STAGES * 2 * TILE;
    // after the main loop the ring's bytes hold the warps' O, then this CTA's O (fp32), maxima and sums
    static constexpr uint32_t ow = kv, mw = ow + 4 * BQ * DH * 4, lw = mw + 4 * BQ * 4, oc = lw + 4 * BQ * 4, mc = oc + BQ * DH * 4, lc = mc + BQ * 4, end = lc + BQ * 4;
    static_assert(end <= total && kv % 16 == 0 && ow % 16 == 0 && oc % 16 == 0, "the combine's arrays fit the ring");
};

struct BlockAttnArgs {
    const __nv_bfloat16 *qkv;            // [B * Lq, 3 d]
    __nv_bfloat16 *kc, *vc;              // [B, cap, d] or NULL (keys and values are the block's own only)
    __nv_bfloat16 *out;                  // [B * Lq, d]
    int Lq, d, len, cap;                 // len: committed rows of the cache (0 without one)
    float scale_log2;                    // log2(e) / sqrt(DH)
};

__device__ __forceinline__ float ld_cluster_f32(uint32_t cluster_addr) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(cluster_addr) : "memory");
    return v;
}
__device__ __forceinline__ float2 ld_cluster_f32x2(uint32_t cluster_addr) {
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(cluster_addr) : "memory");
    return v;
}

// grid: (split, heads * query blocks, B), cluster (split, 1, 1)
template <int DH>
__global__ void __launch_bounds__(NT, 2)
attention_block_kernel(const BlockAttnArgs a, int H, int split) {
    using S = Smem<DH>;
    constexpr int LD = S::LD, U = DH / 8, KS = DH / 16, NO = DH / 8;       // 16-byte pieces per row, K steps of Q K^T, 8-column tiles of O
    extern __shared__ __align__(16) uint8_t sm[];
    pdl_wait();
    pdl_trigger();
    const uint32_t base = smem_u32(sm);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gr = lane >> 2, qc = lane & 3;
    const int rank = blockIdx.x, h = blockIdx.y % H, q0 = blockIdx.y / H * BQ, b = blockIdx.z;
    const int Lk = a.len + a.Lq, ntiles = (Lk + KT - 1) / KT, per = (ntiles + split - 1) / split;
    const int t0 = min(ntiles, rank * per), t1 = min(ntiles, t0 + per);
    const __nv_bfloat16 *own = a.qkv + (int64_t)b * a.Lq * 3 * a.d + h * DH;             // this head's Q columns of the sequence's first row
    const __nv_bfloat16 *kc = a.kc ? a.kc + (int64_t)b * a.cap * a.d + h * DH : nullptr, *vc = a.vc ? a.vc + (int64_t)b * a.cap * a.d + h * DH : nullptr;

    // this thread's 16-byte pieces of a K or V tile: (row, column) do not change from tile to tile
    constexpr int PIECES = (KT * U + NT - 1) / NT;
    int prow[PIECES], pcol[PIECES];
#pragma unroll
    for (int i = 0; i < PIECES; ++i) { const int u = tid + i * NT; prow[i] = u / U; pcol[i] = (u - prow[i] * U) * 8; }
    auto fetch = [&](int t, int st) {              // K and V rows of tile t; rows past the last key become zeros
        const uint32_t ks = base + S::kv + st * 2 * S::TILE;
        const int k0 = t * KT;
        if (k0 + KT <= a.len) {                    // all of it in the cache
            const __nv_bfloat16 *pk = kc + (int64_t)k0 * a.d, *pv = vc + (int64_t)k0 * a.d;
#pragma unroll
            for (int i = 0; i < PIECES; ++i) {
                if (KT * U % NT != 0 && i == PIECES - 1 && prow[i] >= KT) break;
                const uint32_t off = (prow[i] * LD + pcol[i]) * 2, g = (uint32_t)(prow[i] * a.d + pcol[i]);
                cp_async16(ks + off, pk + g, 16);
                cp_async16(ks + S::TILE + off, pv + g, 16);
            }
            return;
        }
#pragma unroll
        for (int i = 0; i < PIECES; ++i) {
            if (KT * U % NT != 0 && i == PIECES - 1 && prow[i] >= KT) break;
            const int key = k0 + prow[i];
            const __nv_bfloat16 *pk = own, *pv = own;
            if (key < a.len) { pk = kc + (int64_t)key * a.d + pcol[i]; pv = vc + (int64_t)key * a.d + pcol[i]; }
            else if (key < Lk) { pk = own + (int64_t)(key - a.len) * 3 * a.d + a.d + pcol[i]; pv = pk + a.d; }
            const uint32_t nb = key < Lk ? 16 : 0, off = (prow[i] * LD + pcol[i]) * 2;
            cp_async16(ks + off, pk, nb);
            cp_async16(ks + S::TILE + off, pv, nb);
        }
    };
    auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };

    // queries, with the first tile's group
    for (int u = tid; u < BQ * U; u += NT) {
        const int r = u / U, c = (u - r * U) * 8;
        const bool ok = q0 + r < a.Lq;
        cp_async16(base + S::q + (r * LD + c) * 2, ok ? own + (int64_t)(q0 + r) * 3 * a.d + c : own, ok ? 16 : 0);
    }
#pragma unroll
    for (int i = 0; i < STAGES - 1; ++i) {
        if (t0 + i < t1) fetch(t0 + i, i);
        commit();
    }
    // the block's keys and values go to rows [len, len + Lq) of the cache (nobody in this launch reads them there)
    if (kc && q0 == 0 && rank == split - 1) {
        for (int u = tid; u < a.Lq * U; u += NT) {
            const int r = u / U, c = (u - r * U) * 8;
            const uint4 k4 = *reinterpret_cast<const uint4 *>(own + (int64_t)r * 3 * a.d + a.d + c), v4 = *reinterpret_cast<const uint4 *>(own + (int64_t)r * 3 * a.d + 2 * a.d + c);
            *reinterpret_cast<uint4 *>(a.kc + ((int64_t)b * a.cap + a.len + r) * a.d + h * DH + c) = k4;
            *reinterpret_cast<uint4 *>(a.vc + ((int64_t)b * a.cap + a.len + r) * a.d + h * DH + c) = v4;
        }
    }
    const int mt = warp & 1, kg = warp >> 1;       // this warp's 16 queries and its quarter of a tile's keys
    uint32_t qf[KS][4];
    float o[NO][4], m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};
#pragma unroll
    for (int n = 0; n < NO; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[n][e] = 0.f;
    for (int t = t0; t < t1; ++t) {
        const int st = (t - t0) % STAGES;
        asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
        __syncthreads();                           // tile t has landed for every thread; everyone is done with the stage the next copy fills
        if (t + STAGES - 1 < t1) fetch(t + STAGES - 1, (t - t0 + STAGES - 1) % STAGES);
        commit();
        if (t == t0) {
#pragma unroll
            for (int k = 0; k < KS; ++k) ldmatrix_x4(qf[k][0], qf[k][1], qf[k][2], qf[k][3], base + S::q + ((16 * mt + (lane & 15)) * LD + 16 * k + (lane >> 4) * 8) * 2);
        }
        const uint32_t ks = base + S::kv + st * 2 * S::TILE + WK * kg * LD * 2, vs = ks + S::TILE;
        // S = Q K^T: 16 queries x WK keys
        float s[WK / 8][4];
#pragma unroll
        for (int n = 0; n < WK / 8; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) s[n][e] = 0.f;
#pragma unroll
        for (int k = 0; k < KS; ++k)
#pragma unroll
            for (int n2 = 0; n2 < WK / 16; ++n2) {
                uint32_t kb[4];                    // keys 0-7 of the 16: channels 16 k + (0-7, 8-15); keys 8-15 likewise
                ldmatrix_x4(kb[0], kb[1], kb[2], kb[3], ks + ((16 * n2 + (lane & 7) + (lane >> 4) * 8) * LD + 16 * k + ((lane >> 3) & 1) * 8) * 2);
                mma_bf16_16816(s[2 * n2], qf[k][0], qf[k][1], qf[k][2], qf[k][3], kb[0], kb[1]);
                mma_bf16_16816(s[2 * n2 + 1], qf[k][0], qf[k][1], qf[k][2], qf[k][3], kb[2], kb[3]);
            }
        const int kleft = Lk - t * KT - WK * kg;    // valid keys of this warp's share
        if (kleft < WK) {
#pragma unroll
            for (int n = 0; n < WK / 8; ++n)
#pragma unroll
                for (int e = 0; e < 2; ++e)
                    if (8 * n + 2 * qc + e >= kleft) s[n][e] = s[n][e + 2] = -INFINITY;
        }
        // running maximum; P = 2^(s - m) as the A operand of P V
        float alpha[2];
        bool moved = false;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            float mx = -INFINITY;
#pragma unroll
            for (int n = 0; n < WK / 8; ++n) mx = fmaxf(mx, fmaxf(s[n][2 * r], s[n][2 * r + 1]));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
            const float mn = fmaxf(m[r], mx * a.scale_log2), ref = mn == -INFINITY ? 0.f : mn;      // no valid key yet: everything stays zero
            alpha[r] = ex2f(m[r] - ref);
            moved |= alpha[r] != 1.f;
            m[r] = mn;
            float sum = 0.f;
#pragma unroll
            for (int n = 0; n < WK / 8; ++n)
#pragma unroll
                for (int e = 0; e < 2; ++e) { s[n][2 * r + e] = ex2f(fmaf(s[n][2 * r + e], a.scale_log2, -ref)); sum += s[n][2 * r + e]; }
            l[r] = fmaf(l[r], alpha[r], sum);
        }
        if (__any_sync(0xffffffffu, moved)) {
#pragma unroll
            for (int n = 0; n < NO; ++n) { o[n][0] *= alpha[0]; o[n][1] *= alpha[0]; o[n][2] *= alpha[1]; o[n][3] *= alpha[1]; }
        }
#pragma unroll
        for (int k2 = 0; k2 < WK / 16; ++k2) {
            const uint32_t pf[4] = {pack_bf16(s[2 * k2][0], s[2 * k2][1]), pack_bf16(s[2 * k2][2], s[2 * k2][3]),
                                    pack_bf16(s[2 * k2 + 1][0], s[2 * k2 + 1][1]), pack_bf16(s[2 * k2 + 1][2], s[2 * k2 + 1][3])};
#pragma unroll
            for (int n2 = 0; n2 < NO / 2; ++n2) {
                uint32_t vb[4];                    // 16 keys x channels 16 n2 + (0-7, 8-15), transposed
                ldmatrix_x4_t(vb[0], vb[1], vb[2], vb[3], vs + ((16 * k2 + (lane & 15)) * LD + 16 * n2 + (lane >> 4) * 8) * 2);
                mma_bf16_16816(o[2 * n2], pf[0], pf[1], pf[2], pf[3], vb[0], vb[1]);
                mma_bf16_16816(o[2 * n2 + 1], pf[0], pf[1], pf[2], pf[3], vb[2], vb[3]);
            }
        }
    }
    cp_async_wait_all();
    __syncthreads();                               // the ring is free: its bytes take the partial results
    float *ow = reinterpret_cast<float *>(sm + S::ow), *mw = reinterpret_cast<float *>(sm + S::mw), *lw = reinterpret_cast<float *>(sm + S::lw);
    float *oc = reinterpret_cast<float *>(sm + S::oc), *mc = reinterpret_cast<float *>(sm + S::mc), *lc = reinterpret_cast<float *>(sm + S::lc);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int row = 16 * mt + 8 * r + gr;
        float ls = l[r];
        ls += __shfl_xor_sync(0xffffffffu, ls, 1);
        ls += __shfl_xor_sync(0xffffffffu, ls, 2);
        if (qc == 0) { mw[kg * BQ + row] = m[r]; lw[kg * BQ + row] = ls; }
#pragma unroll
        for (int n = 0; n < NO; ++n)
            *reinterpret_cast<float2 *>(ow + (kg * BQ + row) * DH + 8 * n + 2 * qc) = make_float2(o[n][2 * r], o[n][2 * r + 1]);
    }
    __syncthreads();
    for (int e = tid; e < BQ * DH / 2; e += NT) {
        const int row = e / (DH / 2), c = (e - row * (DH / 2)) * 2;
        float mm = mw[row];
#pragma unroll
        for (int w = 1; w < 4; ++w) mm = fmaxf(mm, mw[w * BQ + row]);
        const float ref = mm == -INFINITY ? 0.f : mm;
        float x = 0.f, y = 0.f, ls = 0.f;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const float f = ex2f(mw[w * BQ + row] - ref);
            const float2 v = *reinterpret_cast<const float2 *>(ow + (w * BQ + row) * DH + c);
            x = fmaf(f, v.x, x); y = fmaf(f, v.y, y); ls = fmaf(f, lw[w * BQ + row], ls);
        }
        *reinterpret_cast<float2 *>(oc + row * DH + c) = make_float2(x, y);
        if (c == 0) { mc[row] = mm; lc[row] = ls; }
    }
    cluster_sync();                                // every CTA's (m, l, O) is in its shared memory
    // rows of the block are shared out over the cluster
    const int rows = BQ / split;
    for (int e = tid; e < rows * DH / 2; e += NT) {
        const int row = rank * rows + e / (DH / 2), c = (e % (DH / 2)) * 2;
        // every CTA's values are asked for before the first one is used: a remote load takes hundreds of clocks
        float mr[MAX_SPLIT], lr[MAX_SPLIT], mm = -INFINITY;
        float2 v[MAX_SPLIT];
#pragma unroll
        for (int k = 0; k < MAX_SPLIT; ++k) {
            const int kk = min(k, split - 1);
            mr[k] = ld_cluster_f32(cluster_addr(mc + row, kk));
            lr[k] = ld_cluster_f32(cluster_addr(lc + row, kk));
            v[k] = ld_cluster_f32x2(cluster_addr(oc + row * DH + c, kk));
        }
#pragma unroll
        for (int k = 0; k < MAX_SPLIT; ++k) mm = fmaxf(mm, mr[k]);
        float x = 0.f, y = 0.f, ls = 0.f;
#pragma unroll
        for (int k = 0; k < MAX_SPLIT; ++k) {
            const float f = k < split ? ex2f(mr[k] - mm) : 0.f;
            x = fmaf(f, v[k].x, x); y = fmaf(f, v[k].y, y); ls = fmaf(f, lr[k], ls);
        }
        if (q0 + row < a.Lq)
            *reinterpret_cast<uint32_t *>(a.out + ((int64_t)b * a.Lq + q0 + row) * a.d + h * DH + c) = pack_bf16(x / ls, y / ls);
    }
    cluster_sync();                                // nobody leaves while its shared memory may still be read
}

template <int DH>
cudaError_t launch(const BlockAttnArgs &a, int B, int H, cudaStream_t s) {
    const int qb = (a.Lq + BQ - 1) / BQ, Lk = a.len + a.Lq, ctas = B * H * qb;
    int split = 1;      // enough CTAs for all SMs, and no CTA with less than two tiles of keys
    while (split < MAX_SPLIT && ctas * split < sm_count() && Lk >= 2 * KT * 2 * split) split *= 2;
    cudaError_t e = cudaFuncSetAttribute(attention_block_kernel<DH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Smem<DH>::total);
    if (e != cudaSuccess) return e;
    return launch_chain(attention_block_kernel<DH>, dim3(split, H * qb, B), NT, Smem<DH>::total, s, split, a, H, split);
}

}  // namespace

cudaError_t attention_block(const void *qkv, void *out, int B, int Lq, int d, int n_heads, void *k_cache, void *v_cache, int cache_len, int cache_cap, cudaStream_t s) {
    const int dh = d / n_heads;
    BlockAttnArgs a{static_cast<const __nv_bfloat16 *>(qkv), static_cast<__nv_bfloat16 *>(k_cache), static_cast<__nv_bfloat16 *>(v_cache),
                    static_cast<__nv_bfloat16 *>(out), Lq, d, k_cache ? cache_len : 0, k_cache ? cache_cap : 0, 1.4426950408889634f / sqrtf((float)dh)};
    return dh == 64 ? launch<64>(a, B, n_heads, s) : launch<80>(a, B, n_heads, s);
}

}  // namespace dm
