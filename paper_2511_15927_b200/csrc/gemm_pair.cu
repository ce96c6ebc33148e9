// The GEMM for more than 128 rows (the choice is in gemm_tcgen05.cu), on pairs of CTAs (tcgen05 cta_group::2): the two SMs of a pair work on one 256-row
// tile, each holding half of its rows of A and of its accumulators, and each loading half of B -- the tensor cores read the other half
// out of the partner's shared memory.  Per product that is two thirds of the operand traffic (L2 to shared memory) of a single CTA's 128 x 256
// tile.  Bound by the tensor cores under the power limit on large products (about 1.3 GHz in a long run): 16384 x 8512 x 2048 in 438 us =
// 1.30 PFLOP/s, 364 us = 1.57 PFLOP/s after a pause (single-CTA 128 x 256 tiles: 500 and 410 us); by the operand stream from L2, 14 to 15 TB/s over
// all SMs, on small ones (512 x 17024 x 2048: 31 us).
//
// Persistent, one CTA per SM, warp roles per CTA: warp 0 issues this CTA's TMA loads (A: its 128 rows, B: its half of the columns), which
// report to the first CTA's barrier; warp 1 of the first CTA issues the MMAs of the pair; warps 2-9 drain this CTA's accumulators.
// Tile order: the larger operand is streamed from HBM once, the other one stays in L2 (n_fast: consecutive tiles step along N).
//
// Every mbarrier wait is bounded, in both CTAs; on expiry the CTA stores DM_ERR_TIMEOUT in the device status word, lets its loads land and frees TMEM; the CTAs of a pair leave together.
#include <cstring>

#include "gemm_epi.cuh"

namespace dm {
namespace {

using namespace tc;

constexpr int BM = 128, BK = 64;             // rows of A per CTA and row block, K step
constexpr int NTHREADS = 64 + 8 * 32;
constexpr int MAX_STAGES = 8;

// 256 rows x BN columns per pair.  Stage of one CTA: 128 rows of A and BN / 2 rows of B.
template <int BN> struct Tile {
    static constexpr uint32_t A_BYTES = BM * BK * 2, B_BYTES = BN / 2 * BK * 2, STAGE = A_BYTES + B_BYTES, NARROW = A_BYTES + B_BYTES / 2;     // (NARROW: of a narrow tile)
    static constexpr int STAGES = BN == 128 ? 8 : 6;
    static constexpr uint32_t TMEM_COLS = 2 * BN;               // two accumulator buffers
};

// Operands of up to two problems: A in boxes of 128 rows, B in boxes of BN / 2 rows, and (256-column tiles) of 64 for the narrow ones.
struct OpMaps { CUtensorMap a[2], b[2], bn[2]; };

// The tiles of a launch, in the order in which the pairs take them: tile i goes to pair i % npairs.  Tiles are 256 rows x BN columns; with BN = 256 a last column tile of at most 128 columns is
// narrow (256 x 128: 0.74 of a wide tile's time, see gemm_tcgen05.cu), and so are the halves into which the wide tiles of an incomplete last round are cut where that ends
// earlier.  Narrow ones come last.  (16384 x 1024, 256 wide tiles for 74 pairs: 222 wide and 68 halves, 3.74 rounds instead of 4.  All tiles of one width / these, one layer: 1 x 1024
// tokens at d_model 1920 124 / 120 us, 3 x 1111 343 / 330; 1 x 6000 at 1024 270 / 259; 8 x 1024 at 2048 731 / 719; 4 conditioned layers of 3 x 700 at 1920 1571 / 1528.  Level or up to 1 % slower
// where the rounds come out even, as 8 x 2048.)
struct TileAt { int mb, prob, n0; bool narrow; };
template <int BN> struct Tiles {
    int tiles_m, wn, wn_all, whole, halves, total, n_fast;     // row tiles; wide columns per problem, over all problems; uncut wide tiles; halves; all tiles
    int cost;                                                  // of the launch, in hundredths of a round of 256-column tiles
    __host__ __device__ Tiles(int M, int N, int nprob, int npairs, int n_fast) : n_fast(n_fast) {
        const int rem = N % BN, strip = BN == 256 && rem > 0 && rem <= 128;
        tiles_m = (M + 2 * BM - 1) / (2 * BM);
        wn = N / BN + (rem > 0 && !strip);
        wn_all = wn * nprob;
        const int wide = tiles_m * wn_all, narrow = strip ? tiles_m * nprob : 0;
        int cut = 0;
        const int r = wide % npairs, more = r > 0 ? narrow - (npairs - r) : narrow;      // narrow tiles that find no pair idle in the last round of wide ones
        int last = (r > 0 ? 100 : 0) + (more > 0 ? 74 * ((more + npairs - 1) / npairs) : 0);
        if (BN == 256 && r > 0) {
            const int cut_up = 74 * ((2 * r + narrow + npairs - 1) / npairs);
            if (cut_up < last) { cut = r; last = cut_up; }
        }
        cost = BN == 256 ? 100 * (wide / npairs) + last : 74 * ((wide + npairs - 1) / npairs);
        whole = wide - cut;
        halves = 2 * cut;
        total = whole + halves + narrow;
    }
    __device__ __forceinline__ TileAt at(int i) const {
        TileAt t;
        int w = i, half = 0;
        t.narrow = BN == 256 && i >= whole;
        if (BN == 256 && i >= whole + halves) {                // the last columns
            const int j = i - whole - halves;
            t.prob = j / tiles_m; t.mb = j - t.prob * tiles_m; t.n0 = wn * BN;
            return t;
        }
        if (t.narrow) { w = whole + ((i - whole) >> 1); half = (i - whole) & 1; }
        t.mb = n_fast ? w / wn_all : w % tiles_m;
        const int cb = n_fast ? w % wn_all : w / tiles_m;
        t.prob = cb / wn;
        t.n0 = (cb - t.prob * wn) * BN + half * (BN / 2);
        return t;
    }
};

struct __align__(8) Bars {
    uint64_t full[MAX_STAGES], empty[MAX_STAGES], tmem_full[2], tmem_empty[2], add_full[8];
    uint32_t tmem_base;
    int abort;
};

// How a tile leaves the kernel:
//   DIRECT  every lane reads and writes its own row: for outputs whose rows do not start on 16-byte boundaries
//   TMA     32 rows x 128 bytes at a time through 4 KB of shared memory per warp: the addend arrives and the results leave as whole 128-byte lines (a lane
//           storing 32 bytes of its own row makes a transaction of its own of each: 16384 x 4160 x 1024 spent 8.6 k clocks per tile on that
//           where its products take 8.2 k)
//   SUM     TMA, and the two problems are summed (s_0 A_0 B_0^T + s_1 A_1 B_1^T into problem 1's output): a pair runs both on a tile, one after the other in the
//           two accumulator buffers; the epilogue warps take the first product out of TMEM into registers (128 per thread, scaled by its
//           rows' factor, the addend added) while the second one runs, so the sum costs no pass over memory and the buffers still alternate
//   TMA_HALF  TMA for a bf16 output with an addend, 32 columns at a time (a form of its own: as a branch it cost the projections of a layer 1 %)
enum { DIRECT = 0, TMA = 1, SUM = 2, TMA_HALF = 3 };
template <int BN, int MODE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(NTHREADS, 1)
gemm_pair_kernel(const __grid_constant__ OpMaps op, const __grid_constant__ IoMaps io, const __grid_constant__ EpiPair epp, int *status) {
    using T = Tile<BN>;
    constexpr int STAGES = T::STAGES;
    const EpiArgs &ep = epp.p[0];              // sizes are common to all problems
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    Bars *bars = reinterpret_cast<Bars *>(smem + STAGES * T::STAGE + (MODE == DIRECT ? 0 : 8 * STG_BYTES));
    volatile int *abort_flag = &bars->abort;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
    if (ep.m_dev) pdl_wait();                  // (the row count comes from a kernel before this one)
    const int M_eff = ep.m_dev ? min(ep.M, max(0, *ep.m_dev - ep.m_off)) : ep.M;
    constexpr int NSUB = MODE == SUM ? 2 : 1;                  // products per tile
    const Tiles<BN> tiles(M_eff, ep.N, MODE == SUM ? 1 : epp.nprob, npairs, epp.n_fast);       // separate problems sit side by side along N
    const int num_tiles = tiles.total;
    const int kblocks = (ep.K + BK - 1) / BK;

    if (threadIdx.x == 0) {
        for (int i = 0; i < STAGES; ++i) { mbar_init(&bars->full[i], 1); mbar_init(&bars->empty[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&bars->tmem_full[i], 1); mbar_init(&bars->tmem_empty[i], 16); }     // 8 epilogue warps of both CTAs
        for (int i = 0; i < 8; ++i) mbar_init(&bars->add_full[i], 1);
        bars->abort = 0;
        mbar_fence_init();
    }
    if (threadIdx.x == 64) {                   // the maps are on their way while the barriers and TMEM are set up
        prefetch_map(&op.a[0]); prefetch_map(&op.b[0]);
        if (epp.nprob > 1) { prefetch_map(&op.a[1]); prefetch_map(&op.b[1]); }
    }
    if (warp == 1) tmem_alloc_2cta(&bars->tmem_base, T::TMEM_COLS);
    fence_before();
    cluster_sync();                            // barriers of both CTAs are initialised before either one signals the other's
    fence_after();
    const uint32_t tmem_base = bars->tmem_base;

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer (the warp walks the loop, one elected lane issues)
        {
            const bool leader = elect_one();
            uint32_t it = 0;
            bool ok = true;
            // the first stages' share of B (weights) is on its way before the kernel before this one has finished
            const uint32_t ahead = pair < num_tiles ? min(STAGES, kblocks) : 0;
            if (leader && ahead > 0) {
                const TileAt t = tiles.at(pair);
                const int n0 = t.n0 + (int)rank * (t.narrow ? BN / 4 : BN / 2);
                for (uint32_t s = 0; s < ahead; ++s) {
                    if (rank == 0) mbar_expect_tx(&bars->full[s], t.narrow ? 2 * T::NARROW : 2 * T::STAGE);
                    tma_load_2d_pair(smem + s * T::STAGE + T::A_BYTES, t.narrow ? &op.bn[t.prob] : &op.b[t.prob], (int)s * BK, n0, cluster_addr(&bars->full[s], 0));
                }
            }
            __syncwarp();
            pdl_wait();
            pdl_trigger();
            for (int tile = pair; tile < num_tiles && ok; tile += npairs) {
                const TileAt t = tiles.at(tile);
                const int m0 = t.mb * 2 * BM + (int)rank * BM, n0 = t.n0 + (int)rank * (t.narrow ? BN / 4 : BN / 2);
                for (int sub = 0; sub < NSUB && ok; ++sub) {
                    const int prob = t.prob + sub;
                    const CUtensorMap *ma = &op.a[prob], *mb = t.narrow ? &op.bn[prob] : &op.b[prob];
                    for (int kb = 0; kb < kblocks; ++kb, ++it) {
                        const uint32_t s = it % STAGES, ph = (it / STAGES) & 1u;
                        if (!(ok = mbar_wait(&bars->empty[s], ph ^ 1u, abort_flag, status))) break;
                        uint8_t *sa = smem + s * T::STAGE, *sb = sa + T::A_BYTES;
                        const uint32_t full = cluster_addr(&bars->full[s], 0);
                        if (leader) {
                            if (rank == 0 && it >= ahead) mbar_expect_tx(&bars->full[s], t.narrow ? 2 * T::NARROW : 2 * T::STAGE);        // both CTAs' loads
                            tma_load_2d_pair(sa, ma, kb * BK, m0, full);
                            if (it >= ahead) tma_load_2d_pair(sb, mb, kb * BK, n0, full);
                        }
                        __syncwarp();
                    }
                }
            }
            if (!ok) sleep_ns(100000000ull);       // aborting: the loads already issued get time to land before the pair goes away
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer (a warp of the first CTA walks the loop, one elected lane issues: the
        // operand descriptors then live in uniform registers and an MMA takes about 25 clocks to issue; from a single-lane branch it takes
        // about 80, which held every k-block at 600 clocks where its products take 512)
        if (rank == 0) {
            const bool leader = elect_one();
            const uint32_t desc_a0 = desc_lo_k(smem_u32(smem));
            uint32_t it = 0, tcount = 0;
            bool ok = true;
            pdl_wait();                                        // (the limit of the waits below counts from here)
            for (int tile = pair; tile < num_tiles && ok; tile += npairs) {
                const uint32_t idesc = tiles.at(tile).narrow ? idesc_bf16(2 * BM, BN / 2, 0, 0) : idesc_bf16(2 * BM, BN, 0, 0);
                for (int sub = 0; sub < NSUB && ok; ++sub, ++tcount) {
                    const uint32_t buf = tcount & 1u, bph = (tcount >> 1) & 1u;
                    if (!(ok = mbar_wait(&bars->tmem_empty[buf], bph ^ 1u, abort_flag, status))) break;
                    fence_after();
                    const uint32_t d_tmem = tmem_base + buf * BN;
                    for (int kb = 0; kb < kblocks; ++kb, ++it) {
                        const uint32_t s = it % STAGES, ph = (it / STAGES) & 1u;
                        if (!(ok = mbar_wait(&bars->full[s], ph, abort_flag, status))) break;
                        fence_after();
                        const uint32_t da = desc_a0 + s * (T::STAGE >> 4), db = da + (T::A_BYTES >> 4);
                        if (leader) {
    #pragma unroll
                            for (int k = 0; k < BK / 16; ++k)          // 32 bytes along K per MMA: +2 in 16-byte units
                                umma_ss_2cta(d_tmem, da + 2 * k, db + 2 * k, idesc, (kb | k) != 0);
                            umma_commit_2cta(&bars->empty[s]);         // frees the stage in both CTAs when these MMAs have read it
                        }
                        __syncwarp();
                    }
                    if (ok && leader) umma_commit_2cta(&bars->tmem_full[buf]);
                    __syncwarp();
                }
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue: 8 warps over this CTA's 128 rows
        constexpr int COLS = BN / 2;                           // columns per warp (of a narrow tile: half of them)
        const int q = warp & 3, ch = (warp - 2) >> 2;          // TMEM lane quarter, half of the columns
        pdl_wait();
        const uint32_t tquarter = tmem_base + ((uint32_t)(q * 32) << 16);
        uint32_t tcount = 0;
        bool ok = true;
        auto drained = [&](uint32_t buf) {                     // this warp has taken the buffer out of TMEM
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(cluster_addr(&bars->tmem_empty[buf], 0));
        };
        auto ready = [&](uint32_t count) -> bool {
            const bool r = __all_sync(0xffffffffu, mbar_wait(&bars->tmem_full[count & 1u], (count >> 1) & 1u, abort_flag, status));
            fence_after();
            return r;
        };
        EpiOut out{smem + STAGES * T::STAGE + (warp - 2) * STG_BYTES, lane, &bars->add_full[warp - 2], abort_flag, status, 0};
        for (int tile = pair; tile < num_tiles && ok; tile += npairs, tcount += NSUB) {
            const TileAt t = tiles.at(tile);
            const int prob = MODE == SUM ? 1 : t.prob, cols = t.narrow ? COLS / 2 : COLS;
            const EpiArgs &pe = epp.p[prob];                   // this tile's problem: its output, scales and addend
            const uint32_t tlane = tquarter + ch * cols;
            const int row0 = t.mb * 2 * BM + (int)rank * BM + q * 32, row = row0 + lane, n0 = t.n0 + ch * cols;
            const bool row_ok = row < M_eff;
            const bool live = row0 < M_eff && n0 < pe.N;       // some of this warp's part of the tile exists
            const float sc = row_ok ? epi_row_scale(pe, row) : 1.f;
            const EpiRow er(pe, row_ok ? row : 0);
            const bool add = MODE != DIRECT && pe.addend && live;
            if ((MODE == TMA || MODE == TMA_HALF) && add) out.add_fetch(io.add, n0, row0);       // the first columns' addend arrives while the products run
            float ss = 0.f;
            auto emit = [&](int c0, const float *v) { out.template emit<MODE == TMA_HALF>(pe, io.c[prob], io.u, n0, c0, row0, row, row_ok, v, ss); };
            if constexpr (MODE == SUM) {
                const EpiArgs &p0 = epp.p[0];
                const float sc0 = row_ok ? epi_row_scale(p0, row) : 1.f;
                float held[COLS];
                if (!(ok = ready(tcount))) break;
#pragma unroll
                for (int c0 = 0; c0 < COLS; c0 += 32) {
                    if (c0 >= cols) break;
                    const bool some = n0 + c0 < pe.N;
                    if (add && some) out.add_fetch(io.add, n0 + c0, row0);
                    uint32_t r[32];
                    tmem_ld_x32(tlane + (tcount & 1u) * BN + c0, r);
                    tmem_wait_ld();
                    float v[32];
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]) * sc0;
                    if (some) epi_pre<false>(p0, er, n0 + c0, v);
                    if (add && some && ok) ok = out.add_take(v);
#pragma unroll
                    for (int j = 0; j < 32; ++j) held[c0 + j] = v[j];
                }
                drained(tcount & 1u);
                if (!ok || !(ok = ready(tcount + 1))) break;
#pragma unroll
                for (int c0 = 0; c0 < COLS; c0 += 32) {
                    if (c0 >= cols) break;
#pragma unroll
                    for (int c1 = c0; c1 < c0 + 32; c1 += 16) {
                        uint32_t r[16];
                        tmem_ld_x16(tlane + ((tcount + 1) & 1u) * BN + c1, r);
                        tmem_wait_ld();
                        if (er.cs_row) {
#pragma unroll
                            for (int j = 0; j < 16; j += 4) {
                                const float4 cs = n0 + c1 + j < pe.N ? __ldg(reinterpret_cast<const float4 *>(er.cs_row + n0 + c1 + j)) : make_float4(0.f, 0.f, 0.f, 0.f);      // N is a multiple of 4
                                held[c1 + j] = fmaf(__uint_as_float(r[j]) * sc, cs.x, held[c1 + j]);
                                held[c1 + j + 1] = fmaf(__uint_as_float(r[j + 1]) * sc, cs.y, held[c1 + j + 1]);
                                held[c1 + j + 2] = fmaf(__uint_as_float(r[j + 2]) * sc, cs.z, held[c1 + j + 2]);
                                held[c1 + j + 3] = fmaf(__uint_as_float(r[j + 3]) * sc, cs.w, held[c1 + j + 3]);
                            }
                        } else {
#pragma unroll
                            for (int j = 0; j < 16; ++j) held[c1 + j] = fmaf(__uint_as_float(r[j]), sc, held[c1 + j]);
                        }
                    }
                    if (c0 == cols - 32) drained((tcount + 1) & 1u);
                    if (live && n0 + c0 < pe.N) emit(c0, held + c0);
                }
            } else {
                if (!(ok = ready(tcount))) break;
#pragma unroll 1
                for (int c0 = 0; c0 < cols; c0 += 32) {
                    uint32_t r[32];
                    tmem_ld_x32(tlane + (tcount & 1u) * BN + c0, r);
                    tmem_wait_ld();
                    if (c0 == cols - 32) drained(tcount & 1u);
                    const int col = n0 + c0;
                    if (!live || col >= pe.N || (MODE == DIRECT && !row_ok)) continue;
                    float v[32];
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]) * sc;
                    epi_pre<true>(pe, er, col, v);
                    if constexpr (MODE == DIRECT) {
                        epi_add_store(pe, er, row, col, v);
                    } else {
                        if (add) {
                            if (c0 > 0) out.add_fetch(io.add, col, row0);
                            if (!(ok = out.add_take(v))) break;
                        }
                        emit(c0, v);
                    }
                }
            }
        }
        if (MODE != DIRECT && lane == 0) {
            bulk_wait_read0();                                 // (what the stores wrote is complete when the launch is)
            if (!ok) sleep_ns(100000000ull);                   // aborting: an addend load in flight gets time to land
        }
    }
    // ---------------------------------------------------------------- teardown: neither CTA leaves while the other may still signal it
    __syncwarp();
    fence_before();
    cluster_sync();
    if (warp == 1) {
        fence_after();
        tmem_dealloc_2cta(tmem_base, T::TMEM_COLS);
    }
}

template <int BN, int MODE>
cudaError_t launch(const GemmArgs &a, const GemmArgs *b, cudaStream_t s) {
    using T = Tile<BN>;
    OpMaps op;
    memset(&op, 0, sizeof(op));
    for (int i = 0; i < (b ? 2 : 1); ++i) {
        const GemmArgs &p = i ? *b : a;
        if (!make_map_2d(&op.a[i], p.A, p.M, p.K, p.lda, BM) || !make_map_2d(&op.b[i], p.B, p.N, p.K, p.ldb, BN / 2)) return cudaErrorInvalidValue;
        if (BN == 256 && !make_map_2d(&op.bn[i], p.B, p.N, p.K, p.ldb, BN / 4)) return cudaErrorInvalidValue;
    }
    constexpr size_t smem = T::STAGES * (size_t)T::STAGE + (MODE == DIRECT ? 0 : 8 * STG_BYTES) + sizeof(Bars) + 1024;
    static_assert(smem <= 232448, "shared memory budget");
    cudaError_t e = cudaFuncSetAttribute(gemm_pair_kernel<BN, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int *status = device_status_ptr();
    if (!status) return cudaErrorUnknown;
    const EpiPair epp = epi_pair_of(a, b);
    IoMaps io;
    memset(&io, 0, sizeof(io));
    if (MODE != DIRECT) {
        for (int i = MODE == SUM ? 1 : 0; i < epp.nprob; ++i) {
            const EpiArgs &p = epp.p[i];
            if (!make_map_out(&io.c[i], p, MODE == TMA_HALF)) return cudaErrorInvalidValue;
        }
        const EpiArgs &p = epp.p[MODE == SUM ? 1 : 0];         // (separate problems in one launch have no addend here: see tma_io)
        if (p.addend && !make_map_f32_2d(&io.add, p.addend, p.M, p.N, p.ld_add, 32)) return cudaErrorInvalidValue;
        if (p.u && !make_map_half(&io.u, p.u, p.M, p.N, p.N)) return cudaErrorInvalidValue;
    }
    const int pairs = sm_count() / 2, tiles = Tiles<BN>(a.M, a.N, MODE == SUM ? 1 : epp.nprob, pairs, epp.n_fast).total, grid = 2 * (tiles < pairs ? tiles : pairs);
    return launch_chain(gemm_pair_kernel<BN, MODE>, grid, NTHREADS, smem, s, 0, op, io, epp, status);
}

bool tma_io(const GemmArgs &a, const GemmArgs *b) { return gemm_tma_io(a) && (!b || (gemm_tma_io(*b) && !a.addend && !b->addend && !a.u && !b->u)); }

}  // namespace

int gemm_pair_cost(bool wide, const GemmArgs &a, int nprob) {
    const int pairs = sm_count() / 2;
    return wide ? Tiles<256>(a.M, a.N, nprob, pairs, 0).cost : Tiles<128>(a.M, a.N, nprob, pairs, 0).cost;
}

cudaError_t gemm_pair_launch(bool wide, const GemmArgs &a, const GemmArgs *b, cudaStream_t s) {
    if (tma_io(a, b)) {
        if (a.addend && a.c_dtype == DM_BF16) return wide ? launch<256, TMA_HALF>(a, b, s) : launch<128, TMA_HALF>(a, b, s);
        return wide ? launch<256, TMA>(a, b, s) : launch<128, TMA>(a, b, s);
    }
    return wide ? launch<256, DIRECT>(a, b, s) : launch<128, DIRECT>(a, b, s);
}

cudaError_t gemm_pair_sum_launch(const GemmArgs &a, const GemmArgs &b, cudaStream_t s) { return launch<256, SUM>(a, &b, s); }

}  // namespace dm
