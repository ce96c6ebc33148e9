// Fused conv + scan + gate for one block of up to 32 tokens per sequence (the active block of block-autoregressive decoding, Sec. 4.3): one launch, products
// on mma.sync m16n8k16 tiles, with the identities of scan_ssd.cu over a single sub-chunk.
// A CTA of 4 * PP threads takes several tiles (PP channels: a head, or two of 32) of one (batch row, direction), one after the other.  What the heads share -- B' and C' (conv + SiLU), S = C' B'^T,
// and the decays, all from the raw in_proj rows -- it computes once; per tile:
//   conv    x' = SiLU(conv(x)) as bf16 [j][p] (COMMIT: also w_j x'_j);  W_ij = S_ij 2^(Lambda_i - Lambda'_j) [+ D on the diagonal] for j not after i, else 0
//   y       Yb = C' h^T (K = d_state; the B operand is packed from the fp32 state in shared memory), rows scaled by 2^Lambda_i, then += W x' into
//           the same accumulators: warp = 16 tokens x 16 channels
//   state   (COMMIT, left-to-right) h <- 2^Lambda_last h + (w o x')^T B', straight to memory: warp = 16 channels x 64 states
//   gate    through shared memory to a (token, 8 channels) layout: g = y SiLU(z), sum of squares, * norm_w, 16-byte stores
// x tiles and states arrive by TMA, one instruction each, issued as soon as the head before has read its own; z and the head's weights wait in registers.
// B' and C' columns are stored so that a lane's four values of a 16-wide k step are four consecutive states: a lane reads and writes the state as float4.
// Bound by latencies: about 550 instructions per warp and head between two barriers, 24 warps per SM (16 with COMMIT), an issue slot used 41 % of the time.
// A layer's scan stage, 16 sequences, 64 heads of 64, d_state 128: 33 us -> 29 us (the prep launch of 8 us and a CTA per head, 25 us, before); with the state written out
// 54 -> 49 us.  24 layers 2293 -> 2222 us, one layer with the state committed 111 -> 106 us, 24 layers of one sequence 977 -> 957 us.
// (States through asynchronous 16-byte copies of the threads, B operands as 8-byte reads: 750 instructions per head and no gain over the two launches.)
#include "ssd_common.cuh"

namespace dm {
namespace {

using namespace ssd;

// tiles (of PP channels: a head, or two of half that width) per CTA at most: the decays of their heads are kept.  7: what shared memory leaves three CTAs of 64-wide tiles to an SM.  16 with COMMIT:
// eight cost 6 to 7 % of a committed layer of 16 to 24 sequences of 64 heads, 32 gain nothing.
template <bool COMMIT> constexpr int HG_MAX = COMMIT ? 16 : 7;
constexpr int KG = N / 16;             // 16-wide groups of states
constexpr int XR = QB + 4;             // rows of a raw tile: three of history, one unused
constexpr int SLD = QB + 4;            // row pitch (fp32) of S
constexpr int WTL = QB + 8;            // row pitch (bf16) of W
// CTAs per SM
template <int PP, int HW, bool COMMIT> constexpr int RES = PP == 32 ? (COMMIT ? 3 : 4) : COMMIT || HW == 32 ? 2 : 3;

// Tiles per CTA and CTAs per batch row of either direction
struct StepSplit { int hg[2], groups[2]; };

template <int PP, int HW, bool COMMIT> struct StepSmem {
    static constexpr int HPT = PP / HW;            // heads per tile
    static constexpr int XLD = PP + 8;             // row pitch (bf16) of x' and w o x'
    static constexpr int XRAW = XR * PP * 2, NRAW = 2 * N / PP;            // a raw tile of PP channels; tiles of B and C
    static constexpr int STATE = KG * PP * 16 * 4;                         // [16-state group][p][16]; the raw B, C tiles before that
    static constexpr int st = 0, xr = st + (STATE > NRAW * XRAW ? STATE : NRAW * XRAW), ct = xr + XRAW, bt = ct + QB * NLD * 2, ss = bt + QB * NLD * 2, xt = ss + QB * SLD * 4,
                         wt = xt + QB * XLD * 2, ys = wt + HPT * QB * WTL * 2, lam = ys + QB * PP * 4, bars = lam + HG_MAX<COMMIT> * HPT * 2 * QB * 4, wxt = bars + 64, total = wxt + (COMMIT ? QB * XLD * 2 : 0);
    static_assert(xr % 128 == 0 && XRAW % 128 == 0, "TMA tiles");
    static_assert(ct % 16 == 0 && bt % 16 == 0 && ss % 16 == 0 && xt % 16 == 0 && wt % 16 == 0 && ys % 16 == 0 && lam % 16 == 0 && wxt % 16 == 0, "16-byte tiles");
};

__device__ __forceinline__ void prefetch_3d(const CUtensorMap *map, int x, int y, int z) {
    asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(map), "r"(x), "r"(y), "r"(z) : "memory");
}

template <int PP, int HW, bool COMMIT>
__global__ void __launch_bounds__(4 * PP, RES<PP, HW, COMMIT>)
ssd_step_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_s, const __grid_constant__ SsdArgs a, const StepSplit sp, int *status) {
    using M = StepSmem<PP, HW, COMMIT>;
    constexpr int HPT = M::HPT, NT = 4 * PP, U8 = PP / 8, MT = PP / 16, XLD = M::XLD, CP2 = PP / 2;
    extern __shared__ __align__(128) uint8_t sm[];
    __nv_bfloat16 (*Ct)[NLD] = reinterpret_cast<__nv_bfloat16 (*)[NLD]>(sm + M::ct);      // C' rows [i][n], columns permuted (see perm)
    __nv_bfloat16 (*Bt)[NLD] = reinterpret_cast<__nv_bfloat16 (*)[NLD]>(sm + M::bt);      // B' rows [j][n], likewise
    float (*Ss)[SLD] = reinterpret_cast<float (*)[SLD]>(sm + M::ss);
    __nv_bfloat16 (*Xt)[XLD] = reinterpret_cast<__nv_bfloat16 (*)[XLD]>(sm + M::xt);      // x' [j][p]
    __nv_bfloat16 (*WXt)[XLD] = reinterpret_cast<__nv_bfloat16 (*)[XLD]>(sm + M::wxt);    // w_j x'_j [j][p]   (COMMIT)
    __nv_bfloat16 (*Wt)[QB][WTL] = reinterpret_cast<__nv_bfloat16 (*)[QB][WTL]>(sm + M::wt);      // W [i][j] of either head of the tile
    float (*ys)[PP] = reinterpret_cast<float (*)[PP]>(sm + M::ys);
    float (*lams)[2][QB] = reinterpret_cast<float (*)[2][QB]>(sm + M::lam);               // Lambda, Lambda' of every head
    const float *Hs = reinterpret_cast<const float *>(sm + M::st);                        // incoming state of the tile: group g, channel p at (g * PP + p) * 16
    const __nv_bfloat16 *xraw = reinterpret_cast<const __nv_bfloat16 *>(sm + M::xr);
    uint64_t *bar_bc = reinterpret_cast<uint64_t *>(sm + M::bars), *bar_x = bar_bc + 1, *bar_s = bar_bc + 2;
    volatile int *abort_flag = reinterpret_cast<volatile int *>(bar_bc + 3);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gr = lane >> 2, qc = lane & 3;
    // CTA -> (batch row, direction, group of heads)
    const int per = sp.groups[0] + sp.groups[1], b = blockIdx.x / per, j = blockIdx.x - b * per, dir = j >= sp.groups[0];
    const int hg = dir ? sp.hg[1] : sp.hg[0], h0 = (dir ? j - sp.groups[0] : j) * hg, nh = min(hg, a.H / HPT - h0);       // h0, nh: tiles
    const bool rev = dir == 1;
    const int L = a.L, k = a.k;
    const int64_t seq = (int64_t)dir * a.B + b;
    const ScanDir &w = a.dir[dir];
    const int zseq = (a.zx_tied ? 0 : dir) * a.B + b;
    const __nv_bfloat16 *zx = a.zx + (int64_t)zseq * L * a.d_in_proj;
    const __nv_bfloat16 *conv_w = static_cast<const __nv_bfloat16 *>(w.conv_w), *conv_b = static_cast<const __nv_bfloat16 *>(w.conv_b);
    const __nv_bfloat16 *conv_in = !rev && a.conv_in ? a.conv_in + (int64_t)b * (k - 1) * a.conv_ch : nullptr;
    const bool has_bias = (a.flags & DM_FLAG_CONV_BIAS) && conv_b, norm_on = (a.flags & DM_FLAG_GATED_RMSNORM) && w.norm_w, has_d = (a.flags & DM_FLAG_D_SKIP) != 0;
    const bool update = COMMIT && !rev && a.ssm_out != nullptr, have_state = !rev && a.ssm_in != nullptr;
    const bool cw_vec = k == 4 && (reinterpret_cast<uintptr_t>(conv_w) & 15u) == 0;       // a channel pair's taps are one 16-byte load

    // ---- a channel pair's taps (newest first, two channels interleaved per word) and biases
    struct Taps { uint32_t w[4]; float b0, b1; };
    auto taps_of = [&](int ch) {
        Taps t;
        if (cw_vec) {
            const uint4 v = __ldg(reinterpret_cast<const uint4 *>(conv_w + (int64_t)ch * 4));
            t.w[3] = __byte_perm(v.x, v.z, 0x5410); t.w[2] = __byte_perm(v.x, v.z, 0x7632);       // v.x, v.y: taps (0, 1), (2, 3) of the first channel
            t.w[1] = __byte_perm(v.y, v.w, 0x5410); t.w[0] = __byte_perm(v.y, v.w, 0x7632);
        } else {
            const unsigned short *c = reinterpret_cast<const unsigned short *>(conv_w) + (int64_t)ch * k;
#pragma unroll
            for (int m = 0; m < 4; ++m) t.w[m] = m < k ? (uint32_t)__ldg(c + k - 1 - m) | ((uint32_t)__ldg(c + k + k - 1 - m) << 16) : 0u;
        }
        t.b0 = has_bias ? __bfloat162float(conv_b[ch]) : 0.f;
        t.b1 = has_bias ? __bfloat162float(conv_b[ch + 1]) : 0.f;
        return t;
    };
    // the pair of conv channels ch, ch + 1, m tokens before the sequence: the carried rows, or zeros
    auto carried = [&](int ch, int m) {
        return conv_in && m < k ? __ldg(reinterpret_cast<const uint32_t *>(conv_in + (int64_t)(k - 1 - m) * a.conv_ch + ch)) : 0u;
    };
    // conv + SiLU of one pair along n tokens from physical row i0 on: row(i) = the raw pair of chunk row i, history included; before(m) = the pair m tokens before the
    // sequence; out(i, pair of results)
    auto filter = [&](const Taps &t, int i0, int n, auto row, auto before, auto out) {
        f32x2 wl[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) wl[m] = mul2(bf2_to_f2(t.w[m]), pk2(0.5f, 0.5f));     // halved: SiLU(v) = v/2 + v/2 tanh(v/2)
        const f32x2 cb = pk2(0.5f * t.b0, 0.5f * t.b1);
        const int s = rev ? -1 : 1, first = rev ? i0 + n - 1 : i0;
        uint32_t r1 = row(first - s), r2 = row(first - 2 * s), r3 = row(first - 3 * s);
        if (conv_in && i0 == 0) { r1 = before(1); r2 = before(2); r3 = before(3); }
        f32x2 h1 = bf2_to_f2(r1), h2 = bf2_to_f2(r2), h3 = bf2_to_f2(r3);
#pragma unroll 4
        for (int e = 0; e < n; ++e) {
            const int i = first + e * s;
            const f32x2 cur = bf2_to_f2(row(i));
            f32x2 hh = fma2(wl[3], h3, cb);
            hh = fma2(wl[2], h2, hh); hh = fma2(wl[1], h1, hh); hh = fma2(wl[0], cur, hh);
            float ha, hb;
            upk2(hh, ha, hb);
            out(i, fma2(hh, pk2(tanh_fast(ha), tanh_fast(hb)), hh));
            h3 = h2; h2 = h1; h1 = cur;
        }
    };
    // per-head registers: taps and carried rows of the thread's conv pair, gate and norm weights of its epilogue channels, D
    const int cp2 = tid % CP2, rg = tid / CP2;         // conv: channel pair, group of four rows
    const int ei = tid / U8, ec = (tid % U8) * 8;      // epilogue: token, first of 8 channels
    struct Head { Taps t; uint4 z, nw; float D[HPT]; uint32_t c[3]; };
    auto weights_of = [&](Head &q, int h) {
        q.t = taps_of(h * PP + 2 * cp2);
        q.nw = norm_on ? __ldg(reinterpret_cast<const uint4 *>(static_cast<const __nv_bfloat16 *>(w.norm_w) + h * PP + ec)) : make_uint4(0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u);
#pragma unroll
        for (int e = 0; e < HPT; ++e) q.D[e] = has_d ? __ldg(w.D + h * HPT + e) : 0.f;
    };
    auto rows_of = [&](Head &q, int h) {               // (z holds SiLU(z): the in_proj epilogue applied it)
        q.z = ei < L ? __ldg(reinterpret_cast<const uint4 *>(zx + (int64_t)ei * a.d_in_proj + h * PP + ec)) : make_uint4(0u, 0u, 0u, 0u);
        if (conv_in && rg == 0) {
#pragma unroll
            for (int m = 0; m < 3; ++m) q.c[m] = carried(h * PP + 2 * cp2, m + 1);
        }
    };
    const int rofs = rev ? 0 : 3;                      // tile row of chunk row 0: the history lies before it (->) or behind the sequence (<-)
    auto fetch_x = [&](int h) {                        // one thread; rows outside the sequence arrive as zeros
        mbar_expect_tx(bar_x, M::XRAW);
        tma_load_3d(sm + M::xr, &map_x, a.d_inner + h * PP, -rofs, zseq, bar_x);
    };
    auto fetch_state = [&](int h) {                    // one thread
        mbar_expect_tx(bar_s, M::STATE);
        tma_load_3d(sm + M::st, &map_s, 0, (b * (a.H / HPT) + h) * PP, 0, bar_s);
    };
    // column of state n in the tiles of B' and C': within 16, a lane's operand values (2 q, 2 q + 1, 8 + 2 q, 9 + 2 q) are the states 4 q .. 4 q + 3
    auto perm = [](int n) { return (n & ~15) + ((n & 2) << 2) + ((n & 12) >> 1) + (n & 1); };

    // ================================================================ what the heads share
    constexpr int RUN = QB * N / NT;                                    // a thread filters RUN rows of one pair of B or C channels
    const int cp = tid & (N - 1), isC = cp >= N / 2, pi = cp & (N / 2 - 1), bch = (isC ? a.Nr : 0) + 2 * pi;      // bch: channel among the raw 2 Nr
    const bool valid = 2 * pi < a.Nr;                                   // beyond the model's d_state: zeros
    // weights (and, into L2, states): nothing of the launch before this one is in them
    const Taps tbc = taps_of(a.d_inner + (valid ? bch : 0));
    Head cur{}, nxt{};
    weights_of(cur, h0);
    if (tid == 0) {
        mbar_init(bar_bc, 1); mbar_init(bar_x, 1); mbar_init(bar_s, 1);
        *abort_flag = 0;
        mbar_fence_init();
        if (have_state)
            for (int i = 0; i < nh; ++i) prefetch_3d(&map_s, 0, (b * (a.H / HPT) + h0 + i) * PP, 0);
    }
    const float dtb0 = warp < nh * HPT ? w.dt_bias[h0 * HPT + warp] : 0.f, al0 = warp < nh * HPT ? w.A_log[h0 * HPT + warp] : 0.f;      // (its first head's)
    pdl_wait();
    pdl_trigger();
    if (tid == 0) {
        const int nraw = (2 * a.Nr + PP - 1) / PP;
        mbar_expect_tx(bar_bc, nraw * M::XRAW);
        for (int i = 0; i < nraw; ++i) tma_load_3d(sm + M::st + i * M::XRAW, &map_x, 2 * a.d_inner + i * PP, -rofs, zseq, bar_bc);
        fetch_x(h0);
    }
    // decays: a warp per head, lane = token in time order; Lambda of physical row r, log2 units (rows past the sequence have Delta = 0)
    if (warp < nh * HPT) {
        for (int hd = warp; hd < nh * HPT; hd += NT / 32) {
            const int h = h0 * HPT + hd, r = rev ? QB - 1 - lane : lane;
            const float d = r < L ? prep_delta(__bfloat162float(zx[(int64_t)r * a.d_in_proj + a.d_inner + a.conv_ch + h]), hd == warp ? dtb0 : w.dt_bias[h]) : 0.f;
            float cum = d * (-expf(hd == warp ? al0 : w.A_log[h]) * 1.4426950408889634f);
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const float up = __shfl_up_sync(0xffffffffu, cum, off);
                if (lane >= off) cum += up;
            }
            lams[hd][0][r] = cum;
            lams[hd][1][r] = cum - __log2f(d);                          // Delta = 0 (padding): Lambda' = +inf
        }
    }
    rows_of(cur, h0);
    __syncthreads();                                                    // the barriers are initialised
    {
        mbar_wait(bar_bc, 0, abort_flag, status);                       // (a wait that gave up makes all later ones return at once)
        const uint32_t *raw = reinterpret_cast<const uint32_t *>(sm + M::st + (bch / PP) * M::XRAW) + (bch % PP) / 2 + rofs * (PP / 2);
        uint32_t *dst = reinterpret_cast<uint32_t *>(&(isC ? Ct : Bt)[0][perm(2 * pi)]);
        const int r0 = tid / N * RUN;
        if (valid) {
            filter(tbc, r0, RUN, [&](int i) { return raw[i * (PP / 2)]; }, [&](int m) { return carried(a.d_inner + bch, m); },
                   [&](int i, f32x2 o) { dst[i * (NLD / 2)] = f2_to_bf2(o); });
        } else {
            for (int i = r0; i < r0 + RUN; ++i) dst[i * (NLD / 2)] = 0u;
        }
        __syncthreads();
        if (tid == 0 && have_state) fetch_state(h0);                    // over the raw rows
        // S = C' B'^T: warp = 16 rows i x 16 columns j
        if (warp < 4) {
            const int mt = warp & 1, sh = warp >> 1;
            float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
            for (int k0 = 0; k0 < N; k0 += 16) {
                uint32_t a0, a1, a2, a3, b0, b1, b2, b3;
                ldmatrix_x4(a0, a1, a2, a3, &Ct[16 * mt + (lane & 15)][k0 + (lane >> 4) * 8]);
                ldmatrix_x4(b0, b1, b2, b3, &Bt[16 * sh + (lane >> 4) * 8 + (lane & 7)][k0 + ((lane >> 3) & 1) * 8]);
                mma_bf16_16816(acc[0], a0, a1, a2, a3, b0, b1);
                mma_bf16_16816(acc[1], a0, a1, a2, a3, b2, b3);
            }
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) {
                *reinterpret_cast<float2 *>(&Ss[16 * mt + gr][16 * sh + 8 * nt + 2 * qc]) = make_float2(acc[nt][0], acc[nt][1]);
                *reinterpret_cast<float2 *>(&Ss[16 * mt + gr + 8][16 * sh + 8 * nt + 2 * qc]) = make_float2(acc[nt][2], acc[nt][3]);
            }
        }
    }
    // ================================================================ the heads
    for (int hd = 0; hd < nh; ++hd) {
        const int h = h0 + hd;                                          // tile
        const float (*lm)[2][QB] = &lams[hd * HPT];                     // Lambda, Lambda' of its heads
        if (hd + 1 < nh) { weights_of(nxt, h + 1); rows_of(nxt, h + 1); }
        mbar_wait(bar_x, hd & 1, abort_flag, status);
        // ---- conv: thread = channel pair, four rows
        {
            const uint32_t *xr = reinterpret_cast<const uint32_t *>(xraw) + rofs * (PP / 2) + cp2;
            const float (&lh)[2][QB] = lm[2 * cp2 / HW];
            const float last = COMMIT ? lh[0][QB - 1] : 0.f;
            filter(cur.t, 4 * rg, 4, [&](int i) { return xr[i * (PP / 2)]; }, [&](int m) { return cur.c[m - 1]; }, [&](int i, f32x2 o) {
                *reinterpret_cast<uint32_t *>(&Xt[i][2 * cp2]) = f2_to_bf2(o);
                if (COMMIT && update) {
                    const float wj = ex2f(last - lh[1][i]);                 // rows past the sequence: 2^-inf = 0
                    *reinterpret_cast<uint32_t *>(&WXt[i][2 * cp2]) = f2_to_bf2(mul2(o, pk2(wj, wj)));
                }
            });
        }
        if (hd == 0) __syncthreads();                                   // S is there
        // ---- mask: thread = (row i, four columns)
#pragma unroll
        for (int e = 0; e < HPT; ++e)
        for (int u = tid; u < QB * QB / 4; u += NT) {
            const int i = u >> 3, j0 = (u & 7) * 4;
            const float li = lm[e][0][i];
            const float4 s4 = *reinterpret_cast<const float4 *>(&Ss[i][j0]), lp4 = *reinterpret_cast<const float4 *>(&lm[e][1][j0]);
            const float sv[4] = {s4.x, s4.y, s4.z, s4.w}, lpv[4] = {lp4.x, lp4.y, lp4.z, lp4.w};
            float wv[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int jj = j0 + q;
                const bool ok = rev ? jj >= i : jj <= i;                // (rows past the sequence: Lambda' = inf)
                wv[q] = fmaf(sv[q], ex2f(ok ? li - lpv[q] : -INFINITY), i == jj ? cur.D[e] : 0.f);      // 2^-inf = 0: no branch around the exponential
            }
            *reinterpret_cast<uint2 *>(&Wt[e][i][j0]) = make_uint2(pack_bf16(wv[0], wv[1]), pack_bf16(wv[2], wv[3]));
        }
        if (have_state) mbar_wait(bar_s, hd & 1, abort_flag, status);
        __syncthreads();
        if (tid == 0 && hd + 1 < nh) fetch_x(h + 1);
        // ---- y: warp = tokens [16 ymt, +16) x channels [16 ynh, +16)
        {
            const int ymt = warp & 1, ynh = warp >> 1, sub = 16 * ynh / HW;
            float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
            if (have_state) {
                const float *hp = Hs + (16 * ynh + gr) * 16 + 4 * qc;
#pragma unroll
                for (int g = 0; g < KG; ++g) {
                    uint32_t a0, a1, a2, a3;
                    ldmatrix_x4(a0, a1, a2, a3, &Ct[16 * ymt + (lane & 15)][16 * g + (lane >> 4) * 8]);
#pragma unroll
                    for (int nt = 0; nt < 2; ++nt) {
                        const float4 v = *reinterpret_cast<const float4 *>(hp + (g * PP + 8 * nt) * 16);
                        mma_bf16_16816(acc[nt], a0, a1, a2, a3, pack_bf16(v.x, v.y), pack_bf16(v.z, v.w));
                    }
                }
                const float e0 = ex2f(lm[sub][0][16 * ymt + gr]), e1 = ex2f(lm[sub][0][16 * ymt + gr + 8]);
#pragma unroll
                for (int nt = 0; nt < 2; ++nt) { acc[nt][0] *= e0; acc[nt][1] *= e0; acc[nt][2] *= e1; acc[nt][3] *= e1; }
            }
#pragma unroll
            for (int k0 = 0; k0 < QB; k0 += 16) {
                uint32_t a0, a1, a2, a3, b0, b1, b2, b3;
                ldmatrix_x4(a0, a1, a2, a3, &Wt[sub][16 * ymt + (lane & 15)][k0 + (lane >> 4) * 8]);
                ldmatrix_x4_t(b0, b1, b2, b3, &Xt[k0 + (lane & 15)][16 * ynh + (lane >> 4) * 8]);
                mma_bf16_16816(acc[0], a0, a1, a2, a3, b0, b1);
                mma_bf16_16816(acc[1], a0, a1, a2, a3, b2, b3);
            }
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) {
                const int col = 16 * ynh + 8 * nt + 2 * qc, row = 16 * ymt + gr;
                *reinterpret_cast<float2 *>(&ys[row][col]) = make_float2(acc[nt][0], acc[nt][1]);
                *reinterpret_cast<float2 *>(&ys[row + 8][col]) = make_float2(acc[nt][2], acc[nt][3]);
            }
        }
        if (COMMIT && update) {
            // ---- state after the block: channels [16 smt, +16) x states [64 snh, +64) per warp; a lane's values of a 16-state group are four consecutive states
            const int smt = warp % MT, snh = warp / MT, p0 = 16 * smt + gr;
            const float dec = ex2f(lm[16 * smt / HW][0][QB - 1]);
            float acc[8][4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float4 v0 = make_float4(0.f, 0.f, 0.f, 0.f), v1 = v0;
                if (have_state) {
                    const float *hp = Hs + ((4 * snh + u) * PP + p0) * 16 + 4 * qc;
                    v0 = *reinterpret_cast<const float4 *>(hp);
                    v1 = *reinterpret_cast<const float4 *>(hp + 8 * 16);
                }
                acc[2 * u][0] = v0.x * dec; acc[2 * u][1] = v0.y * dec; acc[2 * u + 1][0] = v0.z * dec; acc[2 * u + 1][1] = v0.w * dec;
                acc[2 * u][2] = v1.x * dec; acc[2 * u][3] = v1.y * dec; acc[2 * u + 1][2] = v1.z * dec; acc[2 * u + 1][3] = v1.w * dec;
            }
#pragma unroll
            for (int k0 = 0; k0 < QB; k0 += 16) {
                uint32_t a0, a1, a2, a3;                    // A = (w o x')^T [p][j] read transposed from [j][p]
                ldmatrix_x4_t(a0, a1, a2, a3, &WXt[k0 + (lane & 7) + ((lane >> 4) & 1) * 8][16 * smt + ((lane >> 3) & 1) * 8]);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    uint32_t b0, b1, b2, b3;                // B = B' [j][n] read transposed
                    ldmatrix_x4_t(b0, b1, b2, b3, &Bt[k0 + (lane & 15)][64 * snh + 16 * u + (lane >> 4) * 8]);
                    mma_bf16_16816(acc[2 * u], a0, a1, a2, a3, b0, b1);
                    mma_bf16_16816(acc[2 * u + 1], a0, a1, a2, a3, b2, b3);
                }
            }
            float *ho = a.ssm_out + (((int64_t)b * (a.H / HPT) + h) * PP + p0) * a.Nr + 4 * qc;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int n = 64 * snh + 16 * u;
                if (n < a.Nr) {                             // columns beyond the model's d_state are padding
                    *reinterpret_cast<float4 *>(ho + n) = make_float4(acc[2 * u][0], acc[2 * u][1], acc[2 * u + 1][0], acc[2 * u + 1][1]);
                    *reinterpret_cast<float4 *>(ho + (int64_t)8 * a.Nr + n) = make_float4(acc[2 * u][2], acc[2 * u][3], acc[2 * u + 1][2], acc[2 * u + 1][3]);
                }
            }
        }
        __syncthreads();
        if (tid == 0 && hd + 1 < nh && have_state) fetch_state(h + 1);
        // ---- gate: thread = (token ei, channels ec .. ec + 7)
        {
            const float zf[8] = {bf16_lo(cur.z.x), bf16_hi(cur.z.x), bf16_lo(cur.z.y), bf16_hi(cur.z.y), bf16_lo(cur.z.z), bf16_hi(cur.z.z), bf16_lo(cur.z.w), bf16_hi(cur.z.w)};
            const float nw[8] = {bf16_lo(cur.nw.x), bf16_hi(cur.nw.x), bf16_lo(cur.nw.y), bf16_hi(cur.nw.y), bf16_lo(cur.nw.z), bf16_hi(cur.nw.z), bf16_lo(cur.nw.w), bf16_hi(cur.nw.w)};
            const float4 y0 = *reinterpret_cast<const float4 *>(&ys[ei][ec]), y1 = *reinterpret_cast<const float4 *>(&ys[ei][ec + 4]);
            const float yv[8] = {y0.x, y0.y, y0.z, y0.w, y1.x, y1.y, y1.z, y1.w};
            float g[8], sq = 0.f;
#pragma unroll
            for (int e = 0; e < 8; ++e) { g[e] = yv[e] * zf[e]; sq = fmaf(g[e], g[e], sq); g[e] *= nw[e]; }
#pragma unroll
            for (int off = 1; off < U8 / HPT; off <<= 1) sq += __shfl_xor_sync(0xffffffffu, sq, off);
            if (ei < L) {
                *reinterpret_cast<uint4 *>(a.g + (seq * L + ei) * a.d_inner + h * PP + ec) =
                    make_uint4(pack_bf16(g[0], g[1]), pack_bf16(g[2], g[3]), pack_bf16(g[4], g[5]), pack_bf16(g[6], g[7]));
                if (a.ssq && ec % HW == 0) a.ssq[(seq * L + ei) * a.H + h * HPT + ec / HW] = sq;
            }
        }
        cur = nxt;
    }
    // after a wait that gave up: no copy of this CTA may still be in flight when it leaves
    if (*abort_flag && tid == 0) {
        mbar_wait_quiet(bar_bc, 0, WAIT_LIMIT_NS);
        mbar_wait_quiet(bar_x, (nh - 1) & 1, WAIT_LIMIT_NS);
        if (have_state) mbar_wait_quiet(bar_s, (nh - 1) & 1, WAIT_LIMIT_NS);
    }
}

// tensor of three dimensions (strides in elements), no swizzle
bool make_map_plain(CUtensorMap *m, CUtensorMapDataType t, int es, const void *base, const cuuint64_t (&d)[3], const cuuint64_t (&st)[2], const cuuint32_t (&b)[3]) {
    const cuuint64_t sb[2] = {st[0] * es, st[1] * es};
    const cuuint32_t e[3] = {1, 1, 1};
    return encode_fn()(m, t, 3, const_cast<void *>(base), d, sb, b, e, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int PP, int HW, bool COMMIT>
cudaError_t launch(const SsdArgs &a, int ndir, int dir0, cudaStream_t s) {
    using M = StepSmem<PP, HW, COMMIT>;
    const int tiles = a.H / M::HPT;
    static_assert((M::total + 1024) * RES<PP, HW, COMMIT> <= 233472, "the CTAs of an SM fit its shared memory");
    int *status = device_status_ptr();
    if (!status) return cudaErrorUnknown;
    CUtensorMap mx, ms{};
    {
        const cuuint64_t d[3] = {(cuuint64_t)a.d_in_proj, (cuuint64_t)a.L, (cuuint64_t)2 * a.B}, st[2] = {(cuuint64_t)a.d_in_proj, (cuuint64_t)a.L * a.d_in_proj};
        const cuuint32_t box[3] = {PP, (cuuint32_t)XR, 1};
        if (!make_map_plain(&mx, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, a.zx, d, st, box)) return cudaErrorInvalidValue;
    }
    if (a.ssm_in) {                                  // [16-state group][row][16]
        const cuuint64_t d[3] = {16, (cuuint64_t)a.B * tiles * PP, (cuuint64_t)a.Nr / 16}, st[2] = {(cuuint64_t)a.Nr, 16};
        const cuuint32_t box[3] = {16, PP, KG};
        if (!make_map_plain(&ms, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, a.ssm_in, d, st, box)) return cudaErrorInvalidValue;
    }
    cudaError_t e = cudaFuncSetAttribute(ssd_step_kernel<PP, HW, COMMIT>, cudaFuncAttributeMaxDynamicSharedMemorySize, M::total);
    if (e != cudaSuccess) return e;
    // As many CTAs as are resident at once, so that what the heads share is computed as seldom as one round allows, and shared out between the directions by what a head costs:
    // a left-to-right one reads its state, and with COMMIT writes it (16 sequences of 64 heads: 4.0 us against 2.8, and 4.2 against 1.9; with equal shares the SMs that happened to
    // get left-to-right CTAs only finished at 27 and 43 us, the others at 19 and 18;
    // one layer with the state committed 103 -> 96 us, 24 layers 2191 -> 2118 us).  The same costs serve smaller states and 32-wide heads: with equal ones a committed layer of 16 sequences took
    // 56 us instead of 51 at d_state 16 and 97 instead of 87 with 120 heads of 32, with ones scaled to the state's bytes 56 at d_state 16; without a commit all are level (24 sequences of 64
    // heads: equal shares 110 us, these 115).
    StepSplit sp{};
    const int slots = sm_count() * RES<PP, HW, COMMIT> / a.B, cap = HG_MAX<COMMIT>;
    const int cost[2] = {!a.ssm_in && !COMMIT ? 10 : COMMIT ? 22 : 14, 10};
    auto groups_of = [&](int hg) { return (tiles + hg - 1) / hg; };
    if (ndir == 1) {
        const int most = slots < 1 ? 1 : slots > tiles ? tiles : slots, hg = groups_of(most);
        sp.hg[dir0] = hg > cap ? cap : hg;
    } else {
        int best = 0;
        for (int f = 1; f <= cap; ++f) {                 // heads per left-to-right CTA
            const int left = slots - groups_of(f);
            if (left < 1) continue;
            const int r = groups_of(left > tiles ? tiles : left), t = f * cost[0] > r * cost[1] ? f * cost[0] : r * cost[1];
            if (r <= cap && (!best || t < best)) { best = t; sp.hg[0] = f; sp.hg[1] = r; }
        }
        if (!best) { sp.hg[1] = cap; sp.hg[0] = cap * cost[1] / cost[0]; }      // more than one round
    }
    for (int d = 0; d < 2; ++d) sp.groups[d] = sp.hg[d] ? groups_of(sp.hg[d]) : 0;
    return launch_chain(ssd_step_kernel<PP, HW, COMMIT>, dim3((sp.groups[0] + sp.groups[1]) * a.B), 4 * PP, M::total, s, 0, mx, ms, a, sp, status);
}

}  // namespace

// (norm weights that are not 16-byte aligned go to the prep launch and ssd_block_kernel: reading them either way here cost 1 % of a decoding pass of 16 sequences)
bool scan_step_supports(const ssd::SsdArgs &a) {
    if (a.flags & DM_FLAG_GATED_RMSNORM)
        for (const ScanDir &d : a.dir)
            if (reinterpret_cast<uintptr_t>(d.norm_w) & 15u) return false;
    return a.L <= QB && !((reinterpret_cast<uintptr_t>(a.ssm_in) | reinterpret_cast<uintptr_t>(a.ssm_out)) & 15u) && (int64_t)a.B * a.H * 64 < (1ll << 31);
}

cudaError_t scan_step(const ssd::SsdArgs &a, int headdim, int ndir, int dir0, cudaStream_t s) {
    const bool commit = a.ssm_out != nullptr;
    if (headdim == 64) return commit ? launch<64, 64, true>(a, ndir, dir0, s) : launch<64, 64, false>(a, ndir, dir0, s);
    // heads of 32: two to a tile, so that eight warps share the work that all heads have in common (24 layers, 120 heads, one sequence: 848 -> 794 us, four: 689 -> 656 us in 16 layers)
    if (a.H % 2 == 0) return commit ? launch<64, 32, true>(a, ndir, dir0, s) : launch<64, 32, false>(a, ndir, dir0, s);
    return commit ? launch<32, 32, true>(a, ndir, dir0, s) : launch<32, 32, false>(a, ndir, dir0, s);
}

}  // namespace dm
