// Bidirectional multi-head attention for the hybrid variant (Sec. 3.3: one attention mixer every N mixer blocks):
//     O_h = softmax(Q_h K_h^T / sqrt(d_h)) V_h        full (non-causal), no position encoding, d_h = 64 or 80.
// One CTA per (256 queries, head, sequence), as two streams (NS = 2) of 128 queries that share the key and value tiles; the running-maximum form
// of the softmax, so the L x L score matrix never leaves the SM:
//     warp 0       TMA loads: the two Q tiles once, K and V tiles through a ring
//     warp 1       issues, per key tile and stream, S = Q K^T (both operands K-major in shared memory, fp32 accumulator in TMEM) and
//                  O += P V (A = P from TMEM as bf16, B = V [key][d_h] MN-major)
//     warps 4-7, 8-11   softmax of stream 0 and 1, one query row per thread: the row of S into registers, maximum, P = 2^(s - m) as bf16 into TMEM
//                  and its sum; at the end O / l -> bf16 -> global
// S(j + 1) of a stream is issued as soon as its softmax warps hold S(j) in registers (P has TMEM columns of its own), so the products run
// under the softmax, and the two streams fall out of step by themselves: while one waits, the other one has the exponential unit.  What bounds
// it is that unit: 128 x 128 exponentials take 1024 clocks of an SM, their products 512.  With the projections around it, B=4, L=4096, 16 heads of 64: 495 us (740 us with
// one stream per CTA, two CTAs per SM); B=8, L=1024, 24 heads of 80: 258 us (407 us).
// P and O are relative to the row's exact running maximum: O is read back and scaled in every tile in which a row of the warp finds a new one.  (Raising the maximum only when it was exceeded by 2^8
// saved 2 to 5 % of a call -- 4 x 4096, 16 heads of 64, projections included 471 us instead of 495 -- but the largest weight of a row is then no longer the exact 1 that bf16 holds without rounding:
// error against 64 bits 5.69e-3 instead of 5.60e-3.)
// Heads of 80 channels (the paper's 1.3B hybrid, d = 1920 with 24 heads): every Q, K, V tile is two 64-column sub-tiles, the head's
// channels 0..63 and the 64 columns from channel 64 on, of which the products use the first 16 (the rest belongs to the next head, or is
// the zero fill beyond the tensor, and is never read): one more K step of 16 for S, one more product of 16 columns for O.  Key tiles of 96 there:
// S, P and O of two streams then fit the 512 TMEM columns.
// The last CTA of a sequence may have queries for its first stream only: the second one then issues and computes nothing.
// Up to 128 queries per sequence, more (head, sequence) pairs than SMs: CTAs of one stream, key tiles of 64, two to an SM, so that one's set-up and latencies are covered by the other.
// 16 sequences, 16 heads of 64, a block of 100 after 2048 keys, projections included: 97 us with both streams running, 71 with one stream (64 sequences of 128 after 512 keys: 153, 115).
// Fewer pairs: the two-stream form, whose larger key tiles take fewer steps (1 sequence, 8192 keys: 13 % faster).
// Every wait is bounded; on expiry the CTA stores DM_ERR_TIMEOUT in the device status word and leaves.
// Few queries (block decoding) go to attention_block.cu where block_pays says so.
#include "dm_internal.h"
#include "tc_ptx.cuh"

namespace dm {
using namespace tc;
namespace {

constexpr int BQ = 128, SUB = 64;                           // SUB: columns of a sub-tile (128 bytes: one swizzle atom)

// NT: sub-tiles per operand tile; 1 = heads of 64 channels, 2 = heads of 80.  NS: query streams
template <int NT, int NS> struct Cfg {
    static constexpr int DH = NT == 1 ? 64 : 80, BK = NS == 1 ? 64 : NT == 1 ? 128 : 96, STAGES = NT == 1 ? 4 : NS == 1 ? 2 : 3, NTHREADS = 128 + 128 * NS;
    static constexpr uint32_t QTILE = BQ * 128, KTILE = BK * 128, Q_BYTES = NT * QTILE, KV_BYTES = NT * KTILE;
    static constexpr uint32_t OFF_K = NS * Q_BYTES, OFF_V = OFF_K + STAGES * KV_BYTES, OFF_BAR = OFF_V + STAGES * KV_BYTES, SMEM = OFF_BAR + 1024 + 1024;
    static constexpr uint32_t TM_P = NS * BK, TM_O = TM_P + NS * BK / 2, TM_COLS = 256 * NS;      // S of stream s at s BK, its P at TM_P + s BK / 2, its O at TM_O + s DH
    static_assert(TM_O + NS * DH <= TM_COLS && SMEM * (3 - NS) <= 232448, "TMEM and shared memory budget");
};

struct Bars {
    uint64_t q_full, k_full[4], k_empty[4], v_full[4], v_empty[4], s_full[2], s_empty[2], p_full[2], o_done[2];
    uint32_t tmem_base;
    int abort;
};

struct AttnArgs {
    int B, Lq, Lk, d, H;         // Lq queries per sequence attend to Lk keys
    int kx0, vx0;                // column of head 0's keys / values in their tensor maps
    __nv_bfloat16 *out;          // [B*Lq, d]
    float scale_log2;            // log2(e) / sqrt(d_h)
};

template <int NT, int NS>
__global__ void __launch_bounds__(Cfg<NT, NS>::NTHREADS, 3 - NS)
attention_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                 const __grid_constant__ CUtensorMap map_v, const AttnArgs a, int *status) {
    using C = Cfg<NT, NS>;
    constexpr int DH = C::DH, BK = C::BK, STAGES = C::STAGES;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    Bars *bars = reinterpret_cast<Bars *>(smem + C::OFF_BAR);
    volatile int *abort_flag = &bars->abort;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int q0 = blockIdx.x * NS * BQ, h = blockIdx.y, b = blockIdx.z;
    const int n_kv = (a.Lk + BK - 1) / BK, ns = NS == 2 && a.Lq - q0 > BQ ? 2 : 1;      // streams that have queries

    if (tid == 0) {
        mbar_init(&bars->q_full, 1);
        for (int i = 0; i < STAGES; ++i) {
            mbar_init(&bars->k_full[i], 1); mbar_init(&bars->k_empty[i], 1);
            mbar_init(&bars->v_full[i], 1); mbar_init(&bars->v_empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {              // one arrival per softmax warp of the stream
            mbar_init(&bars->s_full[i], 1); mbar_init(&bars->s_empty[i], 4);
            mbar_init(&bars->p_full[i], 4); mbar_init(&bars->o_done[i], 1);
        }
        bars->abort = 0;
        mbar_fence_init();
    }
    if (warp == 1) tmem_alloc(&bars->tmem_base, C::TM_COLS);
    fence_before();
    __syncthreads();
    fence_after();
    pdl_wait();
    pdl_trigger();
    const uint32_t tmem = bars->tmem_base;
    auto WAIT = [&](uint64_t *bar, uint32_t parity) { return mbar_wait(bar, parity, abort_flag, status); };

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            mbar_expect_tx(&bars->q_full, ns * C::Q_BYTES);
            for (int i = 0; i < ns; ++i)
#pragma unroll
                for (int u = 0; u < NT; ++u) tma_load_3d(smem + i * C::Q_BYTES + u * C::QTILE, &map_q, h * DH + u * SUB, q0 + i * BQ, b, &bars->q_full);
            int issued_k = 0, issued_v = 0;
            for (int j = 0; j < n_kv; ++j) {
                const int st = j % STAGES;
                const uint32_t ph = (j / STAGES) & 1;
                if (!WAIT(&bars->k_empty[st], ph ^ 1)) break;
                mbar_expect_tx(&bars->k_full[st], C::KV_BYTES);
#pragma unroll
                for (int u = 0; u < NT; ++u) tma_load_3d(smem + C::OFF_K + st * C::KV_BYTES + u * C::KTILE, &map_k, a.kx0 + h * DH + u * SUB, j * BK, b, &bars->k_full[st]);
                issued_k = j + 1;
                if (!WAIT(&bars->v_empty[st], ph ^ 1)) break;
                mbar_expect_tx(&bars->v_full[st], C::KV_BYTES);
#pragma unroll
                for (int u = 0; u < NT; ++u) tma_load_3d(smem + C::OFF_V + st * C::KV_BYTES + u * C::KTILE, &map_v, a.vx0 + h * DH + u * SUB, j * BK, b, &bars->v_full[st]);
                issued_v = j + 1;
            }
            if (*abort_flag) {             // aborting: bounded wait for the loads still in flight
                mbar_wait_quiet(&bars->q_full, 0, 100000000ull);
                for (int j = max(0, issued_k - STAGES); j < issued_k; ++j) mbar_wait_quiet(&bars->k_full[j % STAGES], (j / STAGES) & 1, 100000000ull);
                for (int j = max(0, issued_v - STAGES); j < issued_v; ++j) mbar_wait_quiet(&bars->v_full[j % STAGES], (j / STAGES) & 1, 100000000ull);
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer: the warp walks the loop, one elected lane issues
        const bool leader = elect_one();
        const uint32_t dQ0 = desc_lo_k(smem_u32(smem)), dK0 = desc_lo_k(smem_u32(smem + C::OFF_K)), dV0 = desc_lo_mn(smem_u32(smem + C::OFF_V), C::KTILE);
        constexpr uint32_t I_S = idesc_bf16(128, BK, 0, 0), I_O = idesc_bf16(128, 64, 0, 1), I_O16 = idesc_bf16(128, 16, 0, 1);
        auto issue_s = [&](int j, int s) -> bool {        // S of stream s <- Q K(j)^T, once the softmax has taken S(j - 1) out of TMEM
            if (j > 0 && !WAIT(&bars->s_empty[s], (uint32_t)((j - 1) & 1))) return false;
            fence_after();
            const uint32_t dQ = dQ0 + s * (C::Q_BYTES >> 4), dK = dK0 + (j % STAGES) * (C::KV_BYTES >> 4), ts = tmem + s * BK;
            if (leader) {
                umma_ss<0>(ts, dQ, dK, I_S);
#pragma unroll
                for (int kk = 1; kk < 4; ++kk) umma_ss<1>(ts, dQ + 2 * kk, dK + 2 * kk, I_S);
                if constexpr (NT == 2) umma_ss<1>(ts, dQ + (C::QTILE >> 4), dK + (C::KTILE >> 4), I_S);      // channels 64..79: one K step of the second sub-tiles
                umma_commit(&bars->s_full[s]);
                if (s == ns - 1) umma_commit(&bars->k_empty[j % STAGES]);
            }
            __syncwarp();
            return true;
        };
        auto issue_pv = [&](int j, int s) -> bool {       // O of stream s (+)= P(j) V(j)
            if (!WAIT(&bars->p_full[s], (uint32_t)(j & 1))) return false;
            fence_after();
            const uint32_t dV = dV0 + (j % STAGES) * (C::KV_BYTES >> 4), tp = tmem + C::TM_P + s * (BK / 2), to = tmem + C::TM_O + s * DH;
            if (leader) {
                if (j == 0) umma_ts<0>(to, tp, dV, I_O); else umma_ts<1>(to, tp, dV, I_O);
#pragma unroll
                for (int kk = 1; kk < BK / 16; ++kk) umma_ts<1>(to, tp + 8 * kk, dV + kk * 128, I_O);
                if constexpr (NT == 2) {                  // channels 64..79: the first 16 columns of the second sub-tile
                    const uint32_t dV2 = dV + (C::KTILE >> 4);
                    if (j == 0) umma_ts<0>(to + 64, tp, dV2, I_O16); else umma_ts<1>(to + 64, tp, dV2, I_O16);
#pragma unroll
                    for (int kk = 1; kk < BK / 16; ++kk) umma_ts<1>(to + 64, tp + 8 * kk, dV2 + kk * 128, I_O16);
                }
                umma_commit(&bars->o_done[s]);            // phase j: O holds tiles 0..j and P(j) has been read
                if (s == ns - 1) umma_commit(&bars->v_empty[j % STAGES]);
            }
            __syncwarp();
            return true;
        };
        bool ok = WAIT(&bars->q_full, 0) && WAIT(&bars->k_full[0], 0) && issue_s(0, 0) && (ns < 2 || issue_s(0, 1));
        for (int j = 0; j < n_kv && ok; ++j) {
            const bool more = j + 1 < n_kv;
            if (more) ok = WAIT(&bars->k_full[(j + 1) % STAGES], ((j + 1) / STAGES) & 1);
            ok = ok && WAIT(&bars->v_full[j % STAGES], (j / STAGES) & 1);
            for (int s = 0; s < ns && ok; ++s) ok = (!more || issue_s(j + 1, s)) && issue_pv(j, s);
        }
    } else if (warp >= 4 && warp < 4 + 4 * ns) {
        // ------------------------------------------------------------ softmax, O scaling, output
        const int s = (warp - 4) >> 2;                            // stream
        const int q = warp & 3;                                   // TMEM lane quarter of this warp
        const uint32_t tlane = tmem + ((uint32_t)(q * 32) << 16), ts = tlane + s * BK, tp = tlane + C::TM_P + s * (BK / 2), to = tlane + C::TM_O + s * DH;
        float m = 0.f;
        f32x2 l2 = pk2(0.f, 0.f);
        bool ok = true;
        for (int j = 0; j < n_kv; ++j) {
            ok = WAIT(&bars->s_full[s], (uint32_t)(j & 1));
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            fence_after();
            uint32_t r[BK];
#pragma unroll
            for (int c0 = 0; c0 < BK; c0 += 32) tmem_ld_x32(ts + c0, r + c0);
            tmem_wait_ld();
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->s_empty[s]);
            const int valid = a.Lk - j * BK;                      // keys of this tile inside the sequence
            if (valid < BK) {
#pragma unroll
                for (int i = 0; i < BK; ++i) if (i >= valid) r[i] = __float_as_uint(-INFINITY);
            }
            float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
            for (int i = 0; i < BK; ++i) mx[i & 3] = fmaxf(mx[i & 3], __uint_as_float(r[i]));
            const float mj = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * a.scale_log2;
            float alpha = 1.f;
            if (j == 0) m = mj;
            else if (mj > m) { alpha = ex2f(m - mj); m = mj; }
            // P V of the previous tile has read P (and completed O for a scaling)
            if (j > 0) {
                ok = WAIT(&bars->o_done[s], (uint32_t)((j - 1) & 1));
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                fence_after();
            }
            const f32x2 sc2 = pk2(a.scale_log2, a.scale_log2), nm2 = pk2(-m, -m);
            l2 = mul2(l2, pk2(alpha, alpha));
#pragma unroll
            for (int c0 = 0; c0 < BK; c0 += 32) {
                uint32_t pk[16];
#pragma unroll
                for (int i = 0; i < 32; i += 2) {
                    float x, y;
                    upk2(fma2(pk2(__uint_as_float(r[c0 + i]), __uint_as_float(r[c0 + i + 1])), sc2, nm2), x, y);
                    const float p0 = ex2f(x), p1 = ex2f(y);
                    l2 = add2(l2, pk2(p0, p1));
                    pk[i >> 1] = pack_bf16(p0, p1);
                }
                tmem_st_x16(tp + (c0 >> 1), pk);
            }
            if (__any_sync(0xffffffffu, alpha != 1.f)) {          // O moves to the new maximum
                uint32_t t[DH];
#pragma unroll
                for (int c0 = 0; c0 + 32 <= DH; c0 += 32) tmem_ld_x32(to + c0, t + c0);
                if constexpr (DH % 32) tmem_ld_x16(to + DH - 16, t + DH - 16);
                tmem_wait_ld();
                const f32x2 a2 = pk2(alpha, alpha);
#pragma unroll
                for (int i = 0; i < DH; i += 2) {
                    float x, y;
                    upk2(mul2(pk2(__uint_as_float(t[i]), __uint_as_float(t[i + 1])), a2), x, y);
                    t[i] = __float_as_uint(x); t[i + 1] = __float_as_uint(y);
                }
#pragma unroll
                for (int c0 = 0; c0 + 32 <= DH; c0 += 32) tmem_st_x32(to + c0, t + c0);
                if constexpr (DH % 32) tmem_st_x16(to + DH - 16, t + DH - 16);
            }
            tmem_wait_st();
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->p_full[s]);
        }
        if (ok) {
            ok = WAIT(&bars->o_done[s], (uint32_t)((n_kv - 1) & 1));
            ok = __all_sync(0xffffffffu, ok);
        }
        if (ok) {
            fence_after();
            float l, lh;
            upk2(l2, l, lh);
            const float inv = 1.f / (l + lh);
            const int t = q0 + s * BQ + q * 32 + lane;
            __nv_bfloat16 *orow = a.out + ((int64_t)b * a.Lq + t) * a.d + h * DH;
#pragma unroll
            for (int c0 = 0; c0 < DH; c0 += 16) {
                uint32_t r[16], w[8];
                tmem_ld_x16(to + c0, r);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 8; ++i) w[i] = pack_bf16(__uint_as_float(r[2 * i]) * inv, __uint_as_float(r[2 * i + 1]) * inv);
                if (t < a.Lq) st_global_256(orow + c0, w);        // heads start on 32-byte boundaries: 16 channels are one sector
            }
        }
    }
    // ---------------------------------------------------------------- teardown
    __syncwarp();
    fence_before();
    __syncthreads();
    if (warp == 1) {
        fence_after();
        tmem_dealloc(tmem, C::TM_COLS);
    }
}

// The block's keys and values (columns [d, 3 d) of qkv [B*G, 3 d]) go to rows [len, len + G) of the caches [B, cap, d].
__global__ void kv_append_kernel(const __nv_bfloat16 *__restrict__ qkv, __nv_bfloat16 *__restrict__ kc, __nv_bfloat16 *__restrict__ vc,
                                 int G, int d, int len, int cap) {
    const int t = blockIdx.x, b = blockIdx.y;
    const uint4 *src = reinterpret_cast<const uint4 *>(qkv + ((int64_t)b * G + t) * 3 * d + d);
    uint4 *dk = reinterpret_cast<uint4 *>(kc + ((int64_t)b * cap + len + t) * d), *dv = reinterpret_cast<uint4 *>(vc + ((int64_t)b * cap + len + t) * d);
    const int n = d / 8;                                   // 16-byte pieces per row (d is a multiple of 16)
    for (int i = threadIdx.x; i < n; i += blockDim.x) { dk[i] = src[i]; dv[i] = src[n + i]; }
}

}  // namespace

bool attention_supports(int dtype, int d, int n_heads) {
    return dtype == DM_BF16 && n_heads > 0 && (d == n_heads * 64 || d == n_heads * 80) && encode_fn() != nullptr;
}

// Few queries: which kernel.  attention_block.cu splits the keys of a (head, sequence) over the GPU, but its products run on mma.sync, for blocks of 32 queries that each read all keys; the
// kernel above takes 128 queries at the price of 33, with a CTA per pair.  Measured, projections included (block kernel / this one), by pairs, 148 SMs:
//   48 queries after 2048 keys, heads of 64: 64 pairs 41 / 46 us, 96 56 / 47, 128 57 / 49, 256 92 / 63, 1024 275 / 163; heads of 80: 48 pairs 49 / 50, 72 53 / 53, 96 74 / 55, 384 163 / 103
static bool block_pays(int64_t pairs, int Lq) {
    if (Lq > ATTN_BLOCK_MAX_Q) return false;
    return Lq <= 32 || 8 * pairs < 5 * sm_count();
}

// qkv [B*Lq, 3 d] bf16 (columns [Q | K | V], heads contiguous inside each), out [B*Lq, d] bf16.
// k_cache == NULL: keys and values are the K and V columns of qkv (Lk = Lq).  Otherwise the block's keys and values are
// first appended at rows [cache_len, cache_len + Lq) of k_cache, v_cache [B, cache_cap, d], and the queries attend to the
// first cache_len + Lq rows of the caches.
cudaError_t attention_forward(const void *qkv, void *out, int B, int Lq, int d, int n_heads, void *k_cache, void *v_cache,
                              int cache_len, int cache_cap, cudaStream_t s) {
    if (!attention_supports(DM_BF16, d, n_heads) || B <= 0 || Lq <= 0 || B > 65535 || n_heads > 65535) return cudaErrorNotSupported;
    const bool cached = k_cache != nullptr;
    if (cached && (!v_cache || cache_len < 0 || cache_len + Lq > cache_cap)) return cudaErrorInvalidValue;
    const int Lk = cached ? cache_len + Lq : Lq;
    const int64_t pairs = (int64_t)B * n_heads;
    if (block_pays(pairs, Lq)) return attention_block(qkv, out, B, Lq, d, n_heads, k_cache, v_cache, cache_len, cache_cap, s);
    const int streams = Lq <= BQ && pairs > sm_count() ? 1 : 2;
    CUtensorMap mq, mk, mv;
    const int dh = d / n_heads;
    const uint32_t box[3] = {(uint32_t)SUB, (uint32_t)BQ, 1}, box_kv[3] = {(uint32_t)SUB, (uint32_t)(streams == 1 ? Cfg<1, 1>::BK : dh == 64 ? Cfg<1, 2>::BK : Cfg<2, 2>::BK), 1};
    {
        const uint64_t dims[3] = {(uint64_t)3 * d, (uint64_t)Lq, (uint64_t)B};
        const uint64_t str[2] = {(uint64_t)3 * d, (uint64_t)Lq * 3 * d};
        if (!make_map_bf16(&mq, qkv, 3, dims, str, box) || !make_map_bf16(&mk, qkv, 3, dims, str, box_kv)) return cudaErrorInvalidValue;
        mv = mk;
    }
    if (cached) {
        // the maps end at the last valid key: the rest of a tile is filled with zeros, whatever the cache holds there
        const uint64_t dims[3] = {(uint64_t)d, (uint64_t)Lk, (uint64_t)B};
        const uint64_t str[2] = {(uint64_t)d, (uint64_t)cache_cap * d};
        if (!make_map_bf16(&mk, k_cache, 3, dims, str, box_kv) || !make_map_bf16(&mv, v_cache, 3, dims, str, box_kv)) return cudaErrorInvalidValue;
        kv_append_kernel<<<dim3(Lq, B), 128, 0, s>>>(static_cast<const __nv_bfloat16 *>(qkv), static_cast<__nv_bfloat16 *>(k_cache),
                                                      static_cast<__nv_bfloat16 *>(v_cache), Lq, d, cache_len, cache_cap);
        count_launch();
        cudaError_t e0 = cudaGetLastError();
        if (e0 != cudaSuccess) return e0;
    }
    int *status = device_status_ptr();
    if (!status) return cudaErrorUnknown;
    AttnArgs a{B, Lq, Lk, d, n_heads, cached ? 0 : d, cached ? 0 : 2 * d, static_cast<__nv_bfloat16 *>(out), 1.4426950408889634f / sqrtf((float)dh)};
    const dim3 grid((Lq + streams * BQ - 1) / (streams * BQ), n_heads, B);
    auto go = [&](auto kern, uint32_t threads, uint32_t smem) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        return e != cudaSuccess ? e : launch_chain(kern, grid, threads, smem, s, 0, mq, mk, mv, a, status);
    };
    if (streams == 1)
        return dh == 64 ? go(attention_kernel<1, 1>, Cfg<1, 1>::NTHREADS, Cfg<1, 1>::SMEM) : go(attention_kernel<2, 1>, Cfg<2, 1>::NTHREADS, Cfg<2, 1>::SMEM);
    return dh == 64 ? go(attention_kernel<1, 2>, Cfg<1, 2>::NTHREADS, Cfg<1, 2>::SMEM) : go(attention_kernel<2, 2>, Cfg<2, 2>::NTHREADS, Cfg<2, 2>::SMEM);
}

}  // namespace dm
