// The GEMM of gemm_tcgen05.cu for more than 128 rows, on pairs of CTAs (tcgen05 cta_group::2): the two SMs of a pair work on one 256-row
// tile, each holding half of its rows of A and of its accumulators, and each loading half of B -- the tensor cores read the other half
// out of the partner's shared memory.  Per product that is two thirds of the operand traffic (L2 to shared memory) of a single CTA's 128 x 256
// tile.  Bound by the tensor cores under the power limit on large products (about 1.3 GHz in a long run): 16384 x 8512 x 2048 in 438 us =
// 1.30 PFLOP/s, 367 us = 1.56 PFLOP/s after a pause (single-CTA 128 x 256 tiles: 500 and 410 us); by the operand stream from L2, 14 to 15 TB/s over
// all SMs, on small ones (512 x 17024 x 2048: 31 us).
//
// Persistent, one CTA per SM, warp roles per CTA: warp 0 issues this CTA's TMA loads (A: its 128 rows, B: its half of the columns), which
// report to the first CTA's barrier; warp 1 of the first CTA issues the MMAs of the pair; warps 2-9 drain this CTA's accumulators.
// Tile order: the larger operand is streamed from HBM once, the other one stays in L2 (n_fast: consecutive tiles step along N).
//
// Waits and abort as in gemm_tcgen05.cu: every mbarrier wait is bounded, in both CTAs; the CTAs of a pair leave together.
#include "gemm_epi.cuh"

namespace dm {
namespace {

using namespace tc;

constexpr int BM = 128, BK = 64;             // rows of A per CTA and row block, K step
constexpr int NTHREADS = 64 + 8 * 32;
constexpr int MAX_STAGES = 8;

// 256 rows x BN columns per pair.  Stage of one CTA: 128 rows of A and BN / 2 rows of B.
template <int BN> struct Tile {
    static constexpr uint32_t A_BYTES = BM * BK * 2, B_BYTES = BN / 2 * BK * 2, STAGE = A_BYTES + B_BYTES;
    static constexpr int STAGES = BN == 128 ? 8 : 6;
    static constexpr uint32_t TMEM_COLS = 2 * BN;               // two accumulator buffers
};

struct __align__(8) Bars {
    uint64_t full[MAX_STAGES], empty[MAX_STAGES], tmem_full[2], tmem_empty[2];
    uint32_t tmem_base;
    int abort;
};

template <int BN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(NTHREADS, 1)
gemm_pair_kernel(const __grid_constant__ CUtensorMap map_a0, const __grid_constant__ CUtensorMap map_b0,
                 const __grid_constant__ CUtensorMap map_a1, const __grid_constant__ CUtensorMap map_b1,
                 const __grid_constant__ EpiPair epp, int *status) {
    using T = Tile<BN>;
    constexpr int STAGES = T::STAGES;
    const EpiArgs &ep = epp.p[0];              // sizes are common to all problems
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    Bars *bars = reinterpret_cast<Bars *>(smem + STAGES * T::STAGE);
    volatile int *abort_flag = &bars->abort;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
    const int M_eff = ep.m_dev ? min(ep.M, max(0, *ep.m_dev - ep.m_off)) : ep.M;
    const int tiles_m = (M_eff + 2 * BM - 1) / (2 * BM), tiles_n = (ep.N + BN - 1) / BN;
    const int tiles_np = tiles_n * epp.nprob;                  // the problems sit side by side along N
    const int num_tiles = tiles_m * tiles_np;
    auto tile_at = [&](int tile, int &mb, int &cb) {
        mb = epp.n_fast ? tile / tiles_np : tile % tiles_m;
        cb = epp.n_fast ? tile % tiles_np : tile / tiles_m;
    };
    const int kblocks = (ep.K + BK - 1) / BK;

    if (threadIdx.x == 0) {
        for (int i = 0; i < STAGES; ++i) { mbar_init(&bars->full[i], 1); mbar_init(&bars->empty[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&bars->tmem_full[i], 1); mbar_init(&bars->tmem_empty[i], 16); }     // 8 epilogue warps of both CTAs
        bars->abort = 0;
        mbar_fence_init();
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
            for (int tile = pair; tile < num_tiles && ok; tile += npairs) {
                int tm, cb;
                tile_at(tile, tm, cb);
                const int prob = cb / tiles_n;
                const int m0 = tm * 2 * BM + (int)rank * BM, n0 = (cb - prob * tiles_n) * BN + (int)rank * (BN / 2);
                const int prod = epp.ksplit ? prob >> 1 : prob, k_off = epp.p[prob].k_off;
                const CUtensorMap *ma = prod ? &map_a1 : &map_a0, *mb = prod ? &map_b1 : &map_b0;
                for (int kb = 0; kb < kblocks; ++kb, ++it) {
                    const uint32_t s = it % STAGES, ph = (it / STAGES) & 1u;
                    if (!(ok = mbar_wait(&bars->empty[s], ph ^ 1u, abort_flag, status))) break;
                    uint8_t *sa = smem + s * T::STAGE, *sb = sa + T::A_BYTES;
                    const uint32_t full = cluster_addr(&bars->full[s], 0);
                    if (leader) {
                        if (rank == 0) mbar_expect_tx(&bars->full[s], 2 * T::STAGE);        // both CTAs' loads
                        tma_load_2d_pair(sa, ma, k_off + kb * BK, m0, full);
                        tma_load_2d_pair(sb, mb, k_off + kb * BK, n0, full);
                    }
                    __syncwarp();
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
            constexpr uint32_t idesc = idesc_bf16(2 * BM, BN, 0, 0);
            const uint32_t desc_a0 = desc_lo_k(smem_u32(smem));
            uint32_t it = 0, tcount = 0;
            bool ok = true;
            for (int tile = pair; tile < num_tiles && ok; tile += npairs, ++tcount) {
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
    } else {
        // ------------------------------------------------------------ epilogue: 8 warps over this CTA's 128 rows
        constexpr int COLS = BN / 2;                           // columns per warp
        const int q = warp & 3, cfirst = ((warp - 2) >> 2) * COLS;       // TMEM lane quarter, first column
        uint32_t tcount = 0;
        bool ok = true;
        for (int tile = pair; tile < num_tiles && ok; tile += npairs, ++tcount) {
            const uint32_t buf = tcount & 1u, bph = (tcount >> 1) & 1u;
            int tm, cb;
            tile_at(tile, tm, cb);
            const int prob = cb / tiles_n;
            const EpiArgs &pe = epp.p[prob];                   // this tile's problem: its output, scales and addend
            const int row = tm * 2 * BM + (int)rank * BM + q * 32 + lane, n0 = (cb - prob * tiles_n) * BN + cfirst;
            const bool row_ok = row < M_eff;
            const float sc = (pe.row_scale && row_ok) ? pe.row_scale[row] : 1.f;
            const EpiRow er(pe, row);
            ok = mbar_wait(&bars->tmem_full[buf], bph, abort_flag, status);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            fence_after();
#pragma unroll 1
            for (int c0 = 0; c0 < COLS; c0 += 32) {
                uint32_t r[32];
                tmem_ld_x32(tmem_base + ((uint32_t)(q * 32) << 16) + buf * BN + cfirst + c0, r);
                tmem_wait_ld();
                const int col = n0 + c0;
                if (!row_ok || col >= pe.N) continue;
                float v[32];
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]) * sc;
                epi_cols32<true>(pe, er, row, col, v);
            }
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(cluster_addr(&bars->tmem_empty[buf], 0));
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

template <int BN>
cudaError_t launch(const GemmArgs &a, const GemmArgs *b, float *const *hi, cudaStream_t s) {
    using T = Tile<BN>;
    CUtensorMap ma[2], mb[2];
    if (!make_map_2d(&ma[0], a.A, a.M, a.K, a.lda, BM) || !make_map_2d(&mb[0], a.B, a.N, a.K, a.ldb, BN / 2)) return cudaErrorInvalidValue;
    ma[1] = ma[0]; mb[1] = mb[0];
    if (b && (!make_map_2d(&ma[1], b->A, b->M, b->K, b->lda, BM) || !make_map_2d(&mb[1], b->B, b->N, b->K, b->ldb, BN / 2))) return cudaErrorInvalidValue;
    constexpr size_t smem = T::STAGES * (size_t)T::STAGE + sizeof(Bars) + 1024;
    static_assert(smem <= 232448, "shared memory budget");
    cudaError_t e = cudaFuncSetAttribute(gemm_pair_kernel<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int *status = device_status_ptr();
    if (!status) return cudaErrorUnknown;
    const EpiPair epp = epi_pair_of(a, b, hi);
    const int64_t tiles = (int64_t)((a.M + 2 * BM - 1) / (2 * BM)) * ((a.N + BN - 1) / BN) * epp.nprob;
    const int pairs = sm_count() / 2, grid = 2 * (int)(tiles < pairs ? tiles : pairs);
    gemm_pair_kernel<BN><<<grid, NTHREADS, smem, s>>>(ma[0], mb[0], ma[1], mb[1], epp, status);
    count_launch();
    return cudaGetLastError();
}

}  // namespace

cudaError_t gemm_pair_launch(bool wide, const GemmArgs &a, const GemmArgs *b, float *const *hi, cudaStream_t s) {
    return wide ? launch<256>(a, b, hi, s) : launch<128>(a, b, hi, s);
}

}  // namespace dm
