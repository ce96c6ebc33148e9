// Fused conv + scan + gate for sequences of d_state 16: the identities of scan_ssd.cu over sub-chunks of 32 tokens, with every product on mma.sync tiles and the intermediates in registers (34 words a thread of whole heads spill).
// At d_state 16 the tcgen05 kernel's chunk of 128 tokens does eight times the state work the model has and a mask of 128 x 128 per 64 channels; at 32 tokens the mask is a fourth of that per
// channel, the state of a head of 64 is 32 registers per lane, and one warp can carry a tile of 32 tokens x 64 (or 32) channels from its raw rows to its gated output, meeting other warps only
// where it takes the state over.
// A CTA is one chain (batch row, direction, head or half a head): tile warps, of which warp w of n takes the tiles w, w + n, ... in the direction's time order, and a state warp.  A tile:
//     loads    x rows with their conv history, [B' | C'] rows and decays by TMA into the warp's own buffers, the next tile's as soon as this one's have been read; z a step later
//     conv     lane = 4 channels x 8 or 16 rows, results as bf16 over the raw rows, rows in time order
//     St       the tile's own contribution to the state, x'^T (w o B'), left in shared memory for the state warp
//     S, W     C' B'^T; its accumulators, masked and weighted, are the B operand of the next product as they stand
//     chain    waits for the state before the tile: the state warp keeps the state in registers and, tile by tile, leaves its bf16 copy and takes h <- 2^Lambda_last h + St
//     y, gate  y^T = 2^Lambda_i (h_in C'^T) + D x'^T + x'^T W^T, 16 channels at a time; z enters in the accumulators' layout (ldmatrix.trans), g = y SiLU(z), sums of squares, * norm_w; out through
//              stmatrix.trans and a TMA store
// Time order is a matter of row addresses (<- reads its rows backwards), so that the mask is the same for both directions.
// The launch before (narrow_prep) leaves B' | C' as bf16 rows of 32 columns and the decays relative to each sub-chunk.
// Bound by the shared-memory pipe (54 % of its wavefronts on average, 65 % on an SM with two chains) and by latencies at 20 warps an SM: 1750 instructions per warp and tile of 64 channels, an issue
// slot used half of the time.  Prep and scan, 32 heads of 64: 4 x 4096 tokens 196 us on the tcgen05 kernel, 142 here (2.9 TB/s of the rows' traffic where a copy reaches 6.5); 1 x 32768 736 -> 345, 8 x 512
// 81 -> 49, 1 x 4096 99 -> 49.  With the state handed from tile warp to tile warp a step of the chain took 800 to 1800 clocks and the scan of 1 x 32768 436 us, where it took 300; through mbarriers 515.
#include <climits>

#include "ssd_common.cuh"

namespace dm {
namespace {

using namespace ssd;

constexpr int NS = 16;                       // d_state
constexpr int XR = QB + 3;                   // raw rows of a tile with the conv's history
constexpr int PER_SM = 4;                    // CTAs per SM at most

// Tiles of MT x 16 channels: rows of 64 or 128 bytes with the swizzle of that width (tiles aligned to eight rows)
template <int MT> struct Tile {
    static constexpr int CW = 16 * MT, RB = 2 * CW;
    static constexpr int WARPS = 20;                             // (16 of 128 registers: level, 32 x 128 tokens 6 % slower; 24 of 80 for half heads: 8 % slower on one long sequence) resident on an SM, by registers: in CTAs of WARPS / 1 .. 4, one of them the state warp
    static constexpr int QR = CW / 4, RG = 32 / QR, RPG = QB / RG;      // conv: lanes to a row (4 channels each), groups of rows, rows of a group
    // a warp's buffers
    static constexpr uint32_t X = 0, LAM = XR * RB, E = LAM + 256, Z = (E + 256 + 8 * RB - 1) / (8 * RB) * (8 * RB), BC = Z + QB * RB, SLOT = BC + QB * 64;
    static constexpr uint32_t TX_X = XR * RB + QB * 64 + 256, TX_Z = QB * RB;
    static constexpr uint32_t ST = X;                            // over x' once that is in registers: St, then the state's copy, 512 bytes (a 16-byte piece of each lane) at a time
    static_assert(LAM % 16 == 0 && BC % 512 == 0 && SLOT % (8 * RB) == 0, "slot layout");
    // 16-byte piece p of row r lies at piece p ^ swz(r)
    static __host__ __device__ constexpr uint32_t swz(uint32_t r) { return RB == 64 ? (r >> 1) & 3 : r & 7; }
};
template <int MT> struct Shared {
    float conv[5][16 * MT];                  // taps by steps back in time, then the bias; all halved (SiLU(v) = v/2 + v/2 tanh(v/2))
    float norm_w[16 * MT];
    uint64_t x[Tile<MT>::WARPS], z[Tile<MT>::WARPS];
    int ready[Tile<MT>::WARPS];              // by tile warp: 1 + the last tile whose St it left
    int done;                                // tiles whose incoming state is there
    int abort;
};
template <int MT> constexpr size_t smem_bytes(int nw) { return 1024 + (size_t)(nw - 1) * Tile<MT>::SLOT + sizeof(Shared<MT>); }

__device__ __forceinline__ void prefetch_tile(const CUtensorMap *map, int x, int y, int z) {
    asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(map), "r"(x), "r"(y), "r"(z) : "memory");
}
__device__ __forceinline__ float2 lds2(uint32_t addr) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr));
    return v;
}
__device__ __forceinline__ float lds1(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ float4 lds4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ void sts1(uint32_t addr, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory"); }

// Non-volatile, so that the compiler may mix products with what surrounds them
__device__ __forceinline__ void mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// v = hi + lo to 16 bits.  Where v is infinite its rest is NaN: the minimum makes it a number that leaves the infinity alone
__device__ __forceinline__ void split_bf16(f32x2 v, uint32_t &hi, uint32_t &lo) {
    hi = f2_to_bf2(v);
    const uint32_t r = f2_to_bf2(fma2(pk2(-1.f, -1.f), bf2_to_f2(hi), v));
    const __nv_bfloat162 c = __hmin2(*reinterpret_cast<const __nv_bfloat162 *>(&r), __float2bfloat162_rn(0x1p100f));
    lo = *reinterpret_cast<const uint32_t *>(&c);
}
__device__ __forceinline__ void raise_flag(uint32_t addr, int v) { asm volatile("st.release.cta.shared::cta.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }
// Bounded wait until a counter in shared memory has reached `target` (same abort protocol as mbar_wait).  A plain load is answered in a third of the time an mbarrier's probe takes, and these waits
// are the chain's serial part.
__device__ __forceinline__ bool flag_reached(uint32_t addr, int target, volatile int *abort_flag, int *status) {
    auto seen = [&] {
        int v;
        asm volatile("ld.acquire.cta.shared::cta.s32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
        return v >= target;
    };
    if (seen()) return true;
    const uint64_t t0 = globaltimer_ns();
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 256; ++i)
            if (seen()) return true;
        if (*abort_flag) return false;
        if (globaltimer_ns() - t0 > WAIT_LIMIT_NS) {
            *abort_flag = 1;
            atomicExch(status, (int)DM_ERR_TIMEOUT);
            return false;
        }
    }
}

// Eight sums per lane (of tokens 8 i + 2 qc + e) over the lanes of equal qc: halves exchanged, so that each lane ends with one token's sum
__device__ __forceinline__ float token_sum(const f32x2 (&sq)[4], int lane) {
    float v[4][2], u[2][2], t[2];
#pragma unroll
    for (int i = 0; i < 4; ++i) upk2(sq[i], v[i][0], v[i][1]);
    const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int e = 0; e < 2; ++e) u[i][e] = (b4 ? v[2 + i][e] : v[i][e]) + __shfl_xor_sync(0xffffffffu, b4 ? v[i][e] : v[2 + i][e], 16);
#pragma unroll
    for (int e = 0; e < 2; ++e) t[e] = (b3 ? u[1][e] : u[0][e]) + __shfl_xor_sync(0xffffffffu, b3 ? u[0][e] : u[1][e], 8);
    return (b2 ? t[1] : t[0]) + __shfl_xor_sync(0xffffffffu, b2 ? t[0] : t[1], 4);
}

// The state warp: 16 x 16 tiles [channels][states] in the accumulators' layout.  PARTS: bf16 numbers to an entry of the state's copy.
// held: tile at which it waits for a flag that nobody raises (self-test), or -1
template <int MT, int PARTS>
__device__ __forceinline__ void state_role(const uint8_t *slots, Shared<MT> *sh, int nt, int nsub, const float *h_in, float *h_out, int held, int *status) {
    using T = Tile<MT>;
    const int lane = threadIdx.x & 31, gr = lane >> 2, qc = lane & 3;
    volatile int *abort_flag = &sh->abort;
    const uint32_t sb = smem_u32(slots), ready = smem_u32(sh->ready), done = smem_u32(&sh->done);
    float h[MT][2][4];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) h[m][n][e] = h_in ? h_in[(16 * m + gr + (e >> 1) * 8) * NS + 8 * n + 2 * qc + (e & 1)] : 0.f;
    int w = 0;
    const int last = held < 0 ? nsub : min(held, nsub);                          // (asked for in the loop, the chain's serial part, `held` cost 5 % of the scan: 1 x 32768 tokens 375 / 393 us)
    for (int k = 0; k < last; ++k) {
        const uint32_t slot = sb + w * T::SLOT;
        if (!__all_sync(0xffffffffu, flag_reached(ready + 4 * w, k + 1, abort_flag, status))) return;
        float4 st[MT][2];
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int n = 0; n < 2; ++n) st[m][n] = lds4(slot + T::ST + lane * 16 + (2 * m + n) * 512);
        const float dec = lds1(slot + T::E + (QB - 1) * 4);
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            uint32_t c[2][4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const f32x2 v = pk2(h[m][e >> 1][(e & 1) * 2], h[m][e >> 1][(e & 1) * 2 + 1]);
                if constexpr (PARTS == 2) split_bf16(v, c[0][e], c[1][e]);
                else c[0][e] = f2_to_bf2(v);
            }
#pragma unroll
            for (int u = 0; u < PARTS; ++u)
                asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(slot + T::ST + lane * 16 + (PARTS * m + u) * 512), "r"(c[u][0]), "r"(c[u][1]), "r"(c[u][2]), "r"(c[u][3]) : "memory");
        }
        __syncwarp();
        if (lane == 0) raise_flag(done, k + 1);
        const f32x2 dec2 = pk2(dec, dec);
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int n = 0; n < 2; ++n) {
                upk2(fma2(dec2, pk2(h[m][n][0], h[m][n][1]), pk2(st[m][n].x, st[m][n].y)), h[m][n][0], h[m][n][1]);
                upk2(fma2(dec2, pk2(h[m][n][2], h[m][n][3]), pk2(st[m][n].z, st[m][n].w)), h[m][n][2], h[m][n][3]);
            }
        if (++w == nt) w = 0;
    }
    if (last < nsub) { flag_reached(done, INT_MAX, abort_flag, status); return; }
    if (h_out) {
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int n = 0; n < 2; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) h_out[(16 * m + gr + (e >> 1) * 8) * NS + 8 * n + 2 * qc + (e & 1)] = h[m][n][e];
    }
}

// The state's copy is bf16, of which the history of every tile is read: without the D skip beside it that made y up to 1 % less accurate than the 128-token kernel's (which takes more of the history
// through its mask), so that the copy has two parts there (6 to 8 % of a layer's time).  With the skip, D x' is added in fp32 instead of in W, for which the scan takes the same time (5 x 4096 tokens of 32
// heads: 5 % more), and y is 9 % more accurate than that kernel's.
template <int MT, int PARTS, bool REV>
__device__ __forceinline__ void chain(const CUtensorMap &map_x, const CUtensorMap &map_z, const CUtensorMap &map_bc, const CUtensorMap &map_g, const SsdArgs &a,
                                      const float *__restrict__ dl, uint8_t *slots, Shared<MT> *sh, int grp, int b, int held, int *status) {
    using T = Tile<MT>;
    constexpr int CW = T::CW, RB = T::RB;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gr = lane >> 2, qc = lane & 3, nt = (blockDim.x >> 5) - 1;      // nt: tile warps
    const int L = a.L, nsub = (L + QB - 1) / QB, seq = (REV ? a.B : 0) + b, zseq = a.zx_tied ? b : seq, ch0 = grp * CW, h = ch0 / a.Pr;
    volatile int *abort_flag = &sh->abort;
    uint8_t *const slot = slots + warp * T::SLOT;
    const uint32_t sb = smem_u32(slot), conv_w = smem_u32(&sh->conv[0][0]), stp = sb + T::ST + lane * 16;
    uint64_t *const bx = &sh->x[warp], *const bz = &sh->z[warp];
    const float *dl_head = dl + ((int64_t)seq * a.H + h) * 2 * a.Lp;
    const float D1 = (a.flags & DM_FLAG_D_SKIP) ? a.dir[REV ? 1 : 0].D[h] : 0.f;
    const f32x2 Dh = pk2(D1, D1);
    if (warp == nt) {
        const int64_t state0 = (((int64_t)b * a.H + h) * a.Pr + ch0 % a.Pr) * NS;
        state_role<MT, PARTS>(slots, sh, nt, nsub, !REV && a.ssm_in ? a.ssm_in + state0 : nullptr, !REV && a.ssm_out ? a.ssm_out + state0 : nullptr, held, status);
        return;
    }

    auto WAIT = [&](uint64_t *bar, uint32_t parity) { return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, status)); };
    auto first_row = [&](int k) { return (REV ? nsub - 1 - k : k) * QB; };         // of the k-th tile in time
    auto load_x = [&](int k) {
        const int r0 = first_row(k);
        mbar_expect_tx(bx, T::TX_X);
        tma_load_3d(slot + T::X, &map_x, a.d_inner + ch0, REV ? r0 : r0 - 3, zseq, bx);
        tma_load_3d(slot + T::BC, &map_bc, 0, r0, seq, bx);
        bulk_load(slot + T::LAM, dl_head + (int64_t)(r0 / QB) * 2 * QB, 2 * QB * 4, bx);
    };
    auto load_z = [&](int k) {
        mbar_expect_tx(bz, T::TX_Z);
        tma_load_3d(slot + T::Z, &map_z, ch0, first_row(k), zseq, bz);
    };

    const int cg = lane / T::QR, cq = lane % T::QR;                               // conv: rows RPG cg + .., channels 4 cq ..
    auto conv_at = [&](uint32_t row) { return (uint32_t)(((cq >> 1) ^ T::swz(row)) << 4) + (cq & 1) * 8 + row * RB; };       // (row: without the group's, which leave the swizzle alone)
    uint32_t xo, zo, bco, bno;
    {
        const int ri = (lane & 7) + ((lane >> 3) & 1) * 8, rj = (lane & 7) + (lane >> 4) * 8, ra = REV ? QB - 1 - ri : ri, rb = REV ? QB - 1 - rj : rj, lo = (lane >> 3) & 1;
        xo = sb + T::X + rj * RB + ((lo ^ T::swz(rj)) << 4);                      // x'^T (rows in time order): pieces p lo | hi, then rows j lo | hi
        zo = sb + T::Z + rb * RB + ((lo ^ T::swz(rb)) << 4);                      // z^T: pieces p lo | hi, then two i tiles
        bco = sb + T::BC + ra * 64 + (((lane >> 4) ^ ((ra >> 1) & 3)) << 4);      // rows lo | hi, then pieces: B'^T of St; ^ 32: C'
        bno = sb + T::BC + rb * 64 + ((lo ^ ((rb >> 1) & 3)) << 4);               // pieces lo | hi, then rows: B' of S
    }
    constexpr uint32_t BC16 = REV ? (uint32_t)(-16 * 64) : 16 * 64, Z16 = REV ? (uint32_t)(-16 * RB) : 16 * RB;      // 16 rows later in time

    if (lane == 0 && warp < nsub) load_x(warp);
    int it = 0;
    for (int k = warp; k < nsub; k += nt, ++it) {
        const int r0 = first_row(k);
        if (!WAIT(bx, it & 1)) break;
        // ---- conv: a group's rows in time order, history first
        if (!REV && k == 0 && a.conv_in) {                                        // rows before the sequence: the carried conv state (the load left zeros)
            for (int u = lane; u < 3 * CW / 2; u += 32) {
                const int r = u / (CW / 2), c = u % (CW / 2), m = a.k - 1 + r - 3;
                if (m >= 0)
                    *reinterpret_cast<uint32_t *>(slot + T::X + r * RB + (((c >> 2) ^ T::swz(r)) << 4) + (c & 3) * 4) =
                        *reinterpret_cast<const uint32_t *>(a.conv_in + ((int64_t)b * (a.k - 1) + m) * a.conv_ch + ch0 + 2 * c);
            }
            __syncwarp();
        }
        uint2 raw[T::RPG + 3];
#pragma unroll
        for (int u = 0; u < T::RPG + 3; ++u) {
            const uint32_t ad = sb + T::X + conv_at(REV ? QB + 2 - u : u) + (REV ? -cg : cg) * (T::RPG * RB);
            asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(raw[u].x), "=r"(raw[u].y) : "r"(ad));
        }
        const float lam_t = lds1(sb + T::LAM + lane * 4), lamp_t = lds1(sb + T::LAM + QB * 4 + lane * 4);
        const float lam_last = lds1(sb + T::LAM + (QB - 1) * 4);
        __syncwarp();                                                             // the rows are in registers: x' goes over them
        if (lane == 0) {
            bulk_wait_read0();                                                    // the last tile's output has left the z buffer
            load_z(k);
            if (k + nt < nsub) prefetch_tile(&map_x, a.d_inner + ch0, first_row(k + nt), zseq);
        }
        sts1(sb + T::E + lane * 4, ex2f(lam_t));
        sts1(sb + T::E + QB * 4 + lane * 4, ex2f(lam_last - lamp_t));             // w_j
        {
            f32x2 wt[5][2];
#pragma unroll
            for (int m = 0; m < 5; ++m) {
                const float4 v = lds4(conv_w + m * CW * 4 + cq * 16);
                wt[m][0] = pk2(v.x, v.y); wt[m][1] = pk2(v.z, v.w);
            }
            f32x2 w0[2], w1[2], w2[2];                                            // the three rows before
            w2[0] = bf2_to_f2(raw[0].x); w2[1] = bf2_to_f2(raw[0].y);
            w1[0] = bf2_to_f2(raw[1].x); w1[1] = bf2_to_f2(raw[1].y);
            w0[0] = bf2_to_f2(raw[2].x); w0[1] = bf2_to_f2(raw[2].y);
#pragma unroll
            for (int t = 0; t < T::RPG; ++t) {
                const f32x2 cur[2] = {bf2_to_f2(raw[t + 3].x), bf2_to_f2(raw[t + 3].y)};
                uint32_t o[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    f32x2 hv = fma2(wt[3][e], w2[e], wt[4][e]);
                    hv = fma2(wt[2][e], w1[e], hv); hv = fma2(wt[1][e], w0[e], hv); hv = fma2(wt[0][e], cur[e], hv);
                    float ha, hb;
                    upk2(hv, ha, hb);
                    o[e] = f2_to_bf2(fma2(hv, pk2(tanh_fast(ha), tanh_fast(hb)), hv));
                    w2[e] = w1[e]; w1[e] = w0[e]; w0[e] = cur[e];
                }
                asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(sb + T::X + conv_at(t) + cg * (T::RPG * RB)), "r"(o[0]), "r"(o[1]) : "memory");
            }
        }
        __syncwarp();
        // ---- St = x'^T (w o B')
        uint32_t xa[MT][2][4];
        {
            // B' comes rounded to bf16, and rounding w o B' once more made the state 11 % less accurate than the 128-token kernel's (which rounds w o x' once): w o B' is the sum of two bf16 numbers
            // (1 to 2 % of a layer's time)
            uint32_t wb[2][4], wc[2][4];                                          // [16 rows j][(j lo, n lo), (j hi, n lo), (j lo, n hi), (j hi, n hi)]
#pragma unroll
            for (int kt = 0; kt < 2; ++kt) {
                ldmatrix_x4_t(wb[kt][0], wb[kt][1], wb[kt][2], wb[kt][3], bco + kt * BC16);
                const float2 wl = lds2(sb + T::E + QB * 4 + (16 * kt + 2 * qc) * 4), wh = lds2(sb + T::E + QB * 4 + (16 * kt + 8 + 2 * qc) * 4);
#pragma unroll
                for (int e = 0; e < 4; ++e) split_bf16(mul2(bf2_to_f2(wb[kt][e]), (e & 1) ? pk2(wh.x, wh.y) : pk2(wl.x, wl.y)), wb[kt][e], wc[kt][e]);
            }
#pragma unroll
            for (int m = 0; m < MT; ++m) {
#pragma unroll
                for (int kt = 0; kt < 2; ++kt) ldmatrix_x4_t(xa[m][kt][0], xa[m][kt][1], xa[m][kt][2], xa[m][kt][3], (xo ^ (32 * m)) + kt * 16 * RB);
            }
            __syncwarp();                                                         // x' is in registers: St goes over it
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int n = 0; n < 2; ++n) {
                    float st[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                    for (int kt = 0; kt < 2; ++kt) mma(st, xa[m][kt], wc[kt][2 * n], wc[kt][2 * n + 1]);
#pragma unroll
                    for (int kt = 0; kt < 2; ++kt) mma(st, xa[m][kt], wb[kt][2 * n], wb[kt][2 * n + 1]);
                    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(stp + (2 * m + n) * 512), "f"(st[0]), "f"(st[1]), "f"(st[2]), "f"(st[3]) : "memory");
                }
            __syncwarp();
            if (lane == 0) raise_flag(smem_u32(&sh->ready[warp]), k + 1);
        }
        // ---- S, W: C' tiles of 16 rows (the same registers are A operand here and B operand of Yb)
        uint32_t cf[2][4], wf[4][4];                                              // W: (8 rows i, 8 columns j) as the B operand of y^T = x'^T W^T
        f32x2 ei[4];
        {
            uint32_t bf[2][4];
            ldmatrix_x4(cf[0][0], cf[0][1], cf[0][2], cf[0][3], bco ^ 32);
            ldmatrix_x4(cf[1][0], cf[1][1], cf[1][2], cf[1][3], (bco ^ 32) + BC16);
            ldmatrix_x4(bf[0][0], bf[0][1], bf[0][2], bf[0][3], bno);
            ldmatrix_x4(bf[1][0], bf[1][1], bf[1][2], bf[1][3], bno + BC16);
            float2 lp[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) lp[j] = lds2(sb + T::LAM + QB * 4 + (8 * j + 2 * qc) * 4);
#pragma unroll
            for (int i = 0; i < 4; ++i) { const float2 v = lds2(sb + T::E + (8 * i + 2 * qc) * 4); ei[i] = pk2(v.x, v.y); }
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                float s[4][4];
#pragma unroll
                for (int j = 0; j < 2 * mt + 2; ++j) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) s[j][e] = 0.f;
                    mma(s[j], cf[mt], bf[j >> 1][(j & 1) * 2], bf[j >> 1][(j & 1) * 2 + 1]);
                }
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    const int i = 2 * mt + hf;
                    const float li = lds1(sb + T::LAM + (8 * i + gr) * 4);
#pragma unroll
                    for (int j = 0; j <= i; ++j) {
                        float e0 = li - lp[j].x, e1 = li - lp[j].y;
                        if (j == i) { e0 = 2 * qc <= gr ? e0 : -INFINITY; e1 = 2 * qc + 1 <= gr ? e1 : -INFINITY; }      // 2^-inf = 0 after i
                        float v0 = s[j][2 * hf] * ex2f(e0), v1 = s[j][2 * hf + 1] * ex2f(e1);
                        wf[i][j] = pack_bf16(v0, v1);
                    }
                }
            }
        }
        // ---- the state before the tile: A operand of Yb
        if (!__all_sync(0xffffffffu, flag_reached(smem_u32(&sh->done), k + 1, abort_flag, status))) break;
        uint32_t hb[MT][PARTS][4];
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int u = 0; u < PARTS; ++u)
                asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(hb[m][u][0]), "=r"(hb[m][u][1]), "=r"(hb[m][u][2]), "=r"(hb[m][u][3]) : "r"(stp + (PARTS * m + u) * 512));
        fence_proxy_async();
        __syncwarp();                                                             // all but z has been read: the next tile's may come
        if (lane == 0 && k + nt < nsub) {
            load_x(k + nt);
            prefetch_tile(&map_z, ch0, first_row(k + nt), zseq);
        }
        // ---- y and the gate, 16 channels at a time
        if (!WAIT(bz, it & 1)) break;
        f32x2 sq[4];
        float part[MT / 2];                                                       // this lane's token: sums of squares of 32 channels each
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            if (m % 2 == 0) {
#pragma unroll
                for (int i = 0; i < 4; ++i) sq[i] = pk2(0.f, 0.f);
            }
            float y[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) y[i][e] = 0.f;
#pragma unroll
            for (int u = PARTS - 1; u >= 0; --u)
#pragma unroll
                for (int i = 0; i < 4; ++i) mma(y[i], hb[m][u], cf[i >> 1][i & 1], cf[i >> 1][2 + (i & 1)]);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t *xi = &xa[m][i >> 1][(i & 1) * 2];                 // (the A operand's words are laid out as the accumulators)
                const f32x2 lo = pk2(y[i][0], y[i][1]), hi = pk2(y[i][2], y[i][3]);
                upk2(PARTS == 1 ? fma2(ei[i], lo, mul2(Dh, bf2_to_f2(xi[0]))) : mul2(ei[i], lo), y[i][0], y[i][1]);
                upk2(PARTS == 1 ? fma2(ei[i], hi, mul2(Dh, bf2_to_f2(xi[1]))) : mul2(ei[i], hi), y[i][2], y[i][3]);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) mma(y[i], xa[m][0], wf[i][0], i > 0 ? wf[i][1] : 0u);
#pragma unroll
            for (int i = 2; i < 4; ++i) mma(y[i], xa[m][1], wf[i][2], i > 2 ? wf[i][3] : 0u);
            const float nl = sh->norm_w[16 * m + gr], nh = sh->norm_w[16 * m + 8 + gr];
            const f32x2 nl2 = pk2(nl, nl), nh2 = pk2(nh, nh);
#pragma unroll
            for (int ip = 0; ip < 2; ++ip) {
                const uint32_t ad = (zo ^ (32 * m)) + ip * Z16;
                uint32_t z[4];                                                    // (i tile 2 ip, p lo | hi), (i tile 2 ip + 1, p lo | hi)
                ldmatrix_x4_t(z[0], z[1], z[2], z[3], ad);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int i = 2 * ip + (e >> 1);
                    const f32x2 g = mul2(pk2(y[i][(e & 1) * 2], y[i][(e & 1) * 2 + 1]), bf2_to_f2(z[e]));
                    sq[i] = fma2(g, g, sq[i]);
                    z[e] = f2_to_bf2(mul2(g, (e & 1) ? nh2 : nl2));
                }
                stmatrix_x4_t(ad, z[0], z[1], z[2], z[3]);
            }
            if (m % 2 && m < MT - 1 && a.ssq) part[m / 2] = token_sum(sq, lane);
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) {
            tma_store_3d(&map_g, slot + T::Z, ch0, r0, seq);
            bulk_commit();
        }
        if (a.ssq) {
            part[MT / 2 - 1] = token_sum(sq, lane);
            const int i = ((lane >> 3) << 3) + 2 * qc + ((lane >> 2) & 1), row = r0 + (REV ? QB - 1 - i : i);      // token_sum's
            float *dst = a.ssq + ((int64_t)seq * L + row) * a.ssq_parts;
            if (row < L) {
                if constexpr (MT == 2) dst[grp] = part[0];
                else if (a.ssq_parts > a.H) *reinterpret_cast<float2 *>(dst + 2 * grp) = make_float2(part[0], part[1]);
                else dst[grp] = part[0] + part[1];
            }
        }
    }
    if (*abort_flag && lane == 0 && warp < nsub) {                                // aborting: bounded wait for the loads still in flight
        // whichever phase is open: a load that has landed completes it, and a phase without a load runs into the limit
        mbar_wait_quiet(bx, it & 1, 100000000ull);
        mbar_wait_quiet(bx, (it & 1) ^ 1, 100000000ull);
        mbar_wait_quiet(bz, it & 1, 100000000ull);
    }
    if (lane == 0) bulk_wait0();
}

template <int MT, int PARTS>
__global__ void __launch_bounds__(Tile<MT>::WARPS * 32, 1)
narrow_scan_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_z, const __grid_constant__ CUtensorMap map_bc,
                   const __grid_constant__ CUtensorMap map_g, const __grid_constant__ SsdArgs a, const float *__restrict__ dl, int ndir, int dir0, int held, int *status) {
    using T = Tile<MT>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *slots = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const int tid = threadIdx.x, nt = (blockDim.x >> 5) - 1;
    Shared<MT> *sh = reinterpret_cast<Shared<MT> *>(slots + nt * T::SLOT);
    const int G = a.d_inner / T::CW, grp = blockIdx.x % G, dir = dir0 + (blockIdx.x / G) % ndir, b = blockIdx.x / (G * ndir);
    const ScanDir &w = a.dir[dir];
    if (tid == 0) {
        for (int i = 0; i < nt; ++i) { mbar_init(&sh->x[i], 1); mbar_init(&sh->z[i], 1); sh->ready[i] = 0; }
        sh->done = 0;
        sh->abort = 0;
        mbar_fence_init();
    }
    for (int i = tid; i < T::CW; i += blockDim.x) {
        const int c = grp * T::CW + i;
        const __nv_bfloat16 *cw = static_cast<const __nv_bfloat16 *>(w.conv_w) + (int64_t)c * a.k;
        for (int m = 0; m < 4; ++m) sh->conv[m][i] = m < a.k ? 0.5f * __bfloat162float(cw[a.k - 1 - m]) : 0.f;
        sh->conv[4][i] = (a.flags & DM_FLAG_CONV_BIAS) && w.conv_b ? 0.5f * __bfloat162float(static_cast<const __nv_bfloat16 *>(w.conv_b)[c]) : 0.f;
        sh->norm_w[i] = (a.flags & DM_FLAG_GATED_RMSNORM) && w.norm_w ? __bfloat162float(static_cast<const __nv_bfloat16 *>(w.norm_w)[c]) : 1.f;
    }
    __syncthreads();
    pdl_wait();
    pdl_trigger();
    if (dir == 1) chain<MT, PARTS, true>(map_x, map_z, map_bc, map_g, a, dl, slots, sh, grp, b, held, status);
    else chain<MT, PARTS, false>(map_x, map_z, map_bc, map_g, a, dl, slots, sh, grp, b, held, status);
}

// B' and C' (conv + SiLU) as bf16 rows [B' 16 | C' 16], and the decays of every sub-chunk.  A CTA takes the 128 rows of a chunk (a thread: a channel pair over four rows) or the decays of 64 heads
// over them.
__global__ void __launch_bounds__(PREP_THREADS)
narrow_prep_kernel(const __grid_constant__ SsdArgs a, __nv_bfloat16 *__restrict__ bc, float *__restrict__ dl, int dir0) {
    __shared__ __align__(16) float sm[64 * Q];
    pdl_wait();
    pdl_trigger();
    const int per = 1 + (a.H + 63) / 64, c = blockIdx.x / per, part = blockIdx.x - c * per, b = blockIdx.y;
    const int dir = dir0 + blockIdx.z, r0 = (dir == 1 ? a.nch - 1 - c : c) * Q;
    if (part > 0) { prep_decay<true>(a, dl, dir, b, r0, (part - 1) * 64, sm); return; }
    constexpr int RUN = Q * NS / PREP_THREADS;                       // rows of a thread
    const bool rev = dir == 1;
    const int tid = threadIdx.x, pi = tid & (NS - 1), L = a.L, k = a.k;
    const int cc = a.d_inner + 2 * pi;                               // conv channel of the pair's first member (B, then C)
    const int64_t seq = (int64_t)dir * a.B + b;
    const ScanDir &w = a.dir[dir];
    const uint32_t *col = reinterpret_cast<const uint32_t *>(a.zx + ((int64_t)(a.zx_tied ? 0 : dir) * a.B + b) * L * a.d_in_proj + a.d_inner + cc);
    const int64_t ld32 = a.d_in_proj / 2;
    const int lo = r0 + tid / NS * RUN, first = rev ? lo + RUN - 1 : lo, step = rev ? -1 : 1;
    const uint32_t *cin = (!rev && a.conv_in) ? reinterpret_cast<const uint32_t *>(a.conv_in + (int64_t)b * (k - 1) * a.conv_ch + cc) : nullptr;
    uint32_t raw[RUN + 3];
#pragma unroll
    for (int i = 0; i < RUN + 3; ++i) {
        const int t = first + (i - 3) * step;
        raw[i] = (t >= 0 && t < L) ? __ldg(col + (int64_t)t * ld32) : 0u;
        if (cin && t < 0 && k - 1 + t >= 0) raw[i] = __ldg(cin + (int64_t)(k - 1 + t) * (a.conv_ch / 2));
    }
    float wl[2][4], bias[2] = {0.f, 0.f};
    const __nv_bfloat16 *cw = static_cast<const __nv_bfloat16 *>(w.conv_w) + (int64_t)cc * k;
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int m = 0; m < 4; ++m) wl[e][m] = m < k ? __bfloat162float(cw[e * k + k - 1 - m]) : 0.f;
    if ((a.flags & DM_FLAG_CONV_BIAS) && w.conv_b) {
        bias[0] = __bfloat162float(static_cast<const __nv_bfloat16 *>(w.conv_b)[cc]);
        bias[1] = __bfloat162float(static_cast<const __nv_bfloat16 *>(w.conv_b)[cc + 1]);
    }
    uint32_t *dst = reinterpret_cast<uint32_t *>(bc) + seq * L * NS + pi;
#pragma unroll
    for (int i = 0; i < RUN; ++i) {
        const int t = first + i * step;
        const uint32_t win[4] = {raw[i + 3], raw[i + 2], raw[i + 1], raw[i]};
        const uint32_t pk = prep_conv_pair(wl, bias, win);
        if (t < L) dst[(int64_t)t * NS] = pk;
    }
}

template <int MT>
cudaError_t launch(const SsdArgs &a, __nv_bfloat16 *bc, float *dl, int ndir, int dir0, cudaStream_t s) {
    using T = Tile<MT>;
    const int nsub = (a.L + QB - 1) / QB;
    CUtensorMap mx, mz, mb, mg;
    auto map = [&](CUtensorMap *m, const void *p, int64_t ld, int cols, int rows) {
        const uint64_t dims[3] = {(uint64_t)ld, (uint64_t)a.L, (uint64_t)2 * a.B}, str[2] = {(uint64_t)ld, (uint64_t)a.L * ld};
        const uint32_t box[3] = {(uint32_t)cols, (uint32_t)rows, 1};
        return make_map_bf16(m, p, 3, dims, str, box, cols == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B);
    };
    if (!map(&mx, a.zx, a.d_in_proj, T::CW, XR) || !map(&mz, a.zx, a.d_in_proj, T::CW, QB) || !map(&mb, bc, 2 * NS, 2 * NS, QB) || !map(&mg, a.g, a.d_inner, T::CW, QB))
        return cudaErrorInvalidValue;
    int *status = device_status_ptr();
    if (!status) return cudaErrorUnknown;
    const dim3 pgrid(a.nch * (1 + (a.H + 63) / 64), a.B, ndir);
    cudaError_t e = launch_chain(narrow_prep_kernel, pgrid, PREP_THREADS, 0, s, 0, a, bc, dl, dir0);
    if (e != cudaSuccess) return e;
    // as many warps to a chain as leave all chains resident, up to PER_SM of them to an SM.  One to two chains to an SM are launched without overlap behind a prep grid that fills the GPU (chain_spread): 4 x 4096
    // tokens of 32 heads 402 -> 399 us a layer; behind smaller grids the overlap is worth 3 us (8 x 512: 124 / 128).  With more chains every SM is filled either way: 2 % apart at most, in both directions
    // (overlap / none: 5 x 4096 603 / 599, 8 x 2048 440 / 433, 4 x 1024 of 120 heads of 32 379 / 383).
    const int64_t chains = (int64_t)(a.d_inner / T::CW) * ndir * a.B;
    const int sms = sm_count();
    const int per_sm = chains > (int64_t)PER_SM * sms ? PER_SM : (int)((chains + sms - 1) / sms);
    int nw = T::WARPS / per_sm;
    if (nw > nsub + 1) nw = nsub + 1;
    auto kern = (a.flags & DM_FLAG_D_SKIP) ? narrow_scan_kernel<MT, 1> : narrow_scan_kernel<MT, 2>;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes<MT>(T::WARPS));
    if (e != cudaSuccess) return e;
    if (per_sm == 2) chain_spread((int64_t)pgrid.x * pgrid.y * pgrid.z, chains, sms);      // several CTAs to an SM, but not packed
    return launch_chain(kern, (unsigned)chains, 32 * nw, smem_bytes<MT>(nw), s, 0, mx, mz, mb, mg, a, dl, ndir, dir0, scan_selftest_withheld() ? 2 : -1, status);
}

}  // namespace

bool scan_narrow_shape(int d_state) { return d_state == NS; }
// Few chains: heads of 64 are split, so that twice as many SMs have one.  Everywhere else the whole head is the better tile, since mask, decays, B' and C' serve twice the channels.  A layer with half heads /
// whole ones, by heads of all sequences and directions: 64 1 x 1024 tokens 52 / 57 us, 1 x 4096 121 / 138; 72 65 / 69, 158 / 175; 76 1 x 512 54 / 55, 1 x 2048 110 / 106; 80 1 x 4096 208 / 195;
// 128 2 x 2048 127 / 123; 256 4 x 4096 412 / 399.
// Without the D skip the state's copy has two parts and a whole head's registers spill: halves always (2 x 2048 131 / 134 us, 4 x 4096 436 / 446, 5 x 4096 572 / 604).
int scan_narrow_width(int headdim, int64_t heads, bool skip) { return headdim == 64 && skip && 2 * heads > sm_count() ? 64 : 32; }

cudaError_t scan_narrow(const ssd::SsdArgs &a, __nv_bfloat16 *bc, float *dl, int ndir, int dir0, int width, cudaStream_t s) {
    return width == 64 ? launch<4>(a, bc, dl, ndir, dir0, s) : launch<2>(a, bc, dl, ndir, dir0, s);
}

}  // namespace dm
