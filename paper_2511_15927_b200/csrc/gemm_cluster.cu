// Sum of two products, s_0 A_0 B_0^T + s_1 A_1 B_1^T + addend (both directions' out_proj), for row counts whose 256 x 256 tiles leave most of the GPU idle (512 rows of 2048
// columns are 16 of them, for 74 pairs of SMs): the 2, or 4, pairs of CTAs of a cluster each take one product, or half of its K, of the same tile, with the operand path of
// gemm_pair.cu (cta_group::2, 256 rows x 256 or 128 columns per pair).  When its products are done, each pair becomes the owner of a 1 / NP share of the tile's columns: every pair sends the
// other shares' accumulators, scaled by its product's row scale, to their owners through distributed shared memory -- into the operand stages, idle by then -- and the
// owner adds them in a fixed order, applies addend and epilogue and stores.  One tile per cluster: the launch is one round.
// Bound by the k-blocks as in gemm_pair.cu, then by the exchange: 1024 rows, 1920 x 3840 (4 CTAs, 256 columns): products done after 20 us, parts sent 3.6 us later (64 KB out of and
// into each SM, the rate of distributed shared memory), stored 2 us later.  512 rows, 2048 x 4096, with the next norm's input: 33 -> 30 us, 1024 rows 42 -> 39 us, against one
// launch of separate (512 rows: K-halved) products into fp32 partials in memory and another to add them; 24 layers of 512 rows 2241 -> 2192 us.
// Roles as in gemm_pair.cu: warp 0 loads, warp 1 of the pair's first CTA issues MMAs, warps 2-9 drain, exchange and store.  Every mbarrier wait is bounded and every role
// reaches every cluster barrier, also after a wait that gave up.
#include <cstring>

#include "gemm_epi.cuh"

namespace dm {
namespace {

using namespace tc;

constexpr int BM = 128, BK = 64;             // rows of A per CTA, K step
constexpr int NTHREADS = 64 + 8 * 32, MAX_STAGES = 8;
constexpr uint32_t A_BYTES = BM * BK * 2;

struct __align__(8) Bars {
    uint64_t full[MAX_STAGES], empty[MAX_STAGES], done, add_full[8];
    uint32_t tmem_base;
    int abort;
};
// 256 rows x BN columns per pair
template <int BN> struct Tile {
    static constexpr uint32_t STAGE = A_BYTES + BN / 2 * BK * 2;
    static constexpr int STAGES = BN == 128 ? 8 : 6;
    static constexpr size_t SMEM = STAGES * (size_t)STAGE + 8 * STG_BYTES + sizeof(Bars) + 1024;
    static_assert(SMEM <= 232448, "shared memory budget");
};

__device__ __forceinline__ void st_cluster_f4(uint32_t addr, float a, float b, float c, float d) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

template <int NP, int BN>
__global__ void __cluster_dims__(2 * NP, 1, 1) __launch_bounds__(NTHREADS, 1)
gemm_cluster_sum_kernel(const __grid_constant__ CUtensorMap map_a0, const __grid_constant__ CUtensorMap map_b0, const __grid_constant__ CUtensorMap map_a1,
                        const __grid_constant__ CUtensorMap map_b1, const __grid_constant__ IoMaps io, const __grid_constant__ EpiPair epp, int *status) {
    constexpr uint32_t STAGE = Tile<BN>::STAGE, TMEM_COLS = BN;
    constexpr int STAGES = Tile<BN>::STAGES;
    constexpr int F = BN / NP, NH = F / 64;    // columns of an owner's share; warps per TMEM lane quarter that finish them (64 columns each)
    constexpr uint32_t SLOT = F / 32 * 4 * STG_BYTES;          // one sender's part: [32-column group][lane quarter][32 rows x 128 bytes, pieces swizzled as in EpiOut]
    static_assert((NP - 1) * SLOT <= STAGES * STAGE, "the parts fit the operand stages");
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    Bars *bars = reinterpret_cast<Bars *>(smem + STAGES * STAGE + 8 * STG_BYTES);
    volatile int *abort_flag = &bars->abort;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank(), lead = rank & ~1u;
    const int share = rank >> 1, dir = share / (NP / 2), part = share % (NP / 2);
    const EpiArgs &pe = epp.p[1];
    const int tiles_m = (pe.M + 2 * BM - 1) / (2 * BM), tile = blockIdx.x / (2 * NP);
    const int m0 = tile % tiles_m * 2 * BM + (int)(rank & 1) * BM, t0 = tile / tiles_m * BN;       // this CTA's rows; the tile's first column
    const int kbt = (pe.K + BK - 1) / BK, kb0 = part * ((kbt + 1) / 2), kblocks = NP == 2 ? kbt : part ? kbt / 2 : (kbt + 1) / 2;
    const CUtensorMap *ma = dir ? &map_a1 : &map_a0, *mb = dir ? &map_b1 : &map_b0;

    if (threadIdx.x == 0) {
        for (int i = 0; i < STAGES; ++i) { mbar_init(&bars->full[i], 1); mbar_init(&bars->empty[i], 1); }
        mbar_init(&bars->done, 1);
        for (int i = 0; i < 8; ++i) mbar_init(&bars->add_full[i], 1);
        bars->abort = 0;
        mbar_fence_init();
    }
    if (threadIdx.x == 64) { prefetch_map(ma); prefetch_map(mb); }
    if (warp == 1) tmem_alloc_2cta(&bars->tmem_base, TMEM_COLS);
    fence_before();
    cluster_sync();                            // barriers are initialised before anyone signals them
    fence_after();
    const uint32_t tmem_base = bars->tmem_base;

    // epilogue role: TMEM lane quarter and half of the columns; rows
    const int q = warp & 3, hf = (warp - 2) >> 2, row0 = m0 + q * 32, row = row0 + lane;
    const bool row_ok = row < pe.M, rows_live = row0 < pe.M;
    const uint32_t tlane = tmem_base + ((uint32_t)(q * 32) << 16);
    const int n0 = t0 + share * F + 64 * hf;   // a finishing warp's first column
    const bool fin = warp >= 2 && hf < NH && rows_live && n0 < pe.N;
    EpiOut out{smem + STAGES * STAGE + (warp - 2) * STG_BYTES, lane, &bars->add_full[warp >= 2 ? warp - 2 : 0], abort_flag, status, 0};
    bool ok = true;
    float sc = 1.f;

    if (warp == 0) {
        const bool leader = elect_one();
        const int nb = t0 + (int)(rank & 1) * (BN / 2);
        // the first stages' share of B (weights) is on its way before the kernel before this one has finished
        const int ahead = min(STAGES, kblocks);
        if (leader) {
            for (int s = 0; s < ahead; ++s) {
                if (rank == lead) mbar_expect_tx(&bars->full[s], 2 * STAGE);
                tma_load_2d_pair(smem + s * STAGE + A_BYTES, mb, (kb0 + s) * BK, nb, cluster_addr(&bars->full[s], lead));
            }
        }
        __syncwarp();
        pdl_wait();
        pdl_trigger();
        for (int kb = 0; kb < kblocks; ++kb) {
            const uint32_t s = kb % STAGES, ph = (kb / STAGES) & 1u;
            if (!(ok = mbar_wait(&bars->empty[s], ph ^ 1u, abort_flag, status))) break;
            const uint32_t full = cluster_addr(&bars->full[s], lead);
            if (leader) {
                if (rank == lead && kb >= ahead) mbar_expect_tx(&bars->full[s], 2 * STAGE);        // both CTAs' loads
                tma_load_2d_pair(smem + s * STAGE, ma, (kb0 + kb) * BK, m0, full);
                if (kb >= ahead) tma_load_2d_pair(smem + s * STAGE + A_BYTES, mb, (kb0 + kb) * BK, nb, full);
            }
            __syncwarp();
        }
        if (!ok) sleep_ns(100000000ull);       // aborting: the loads already issued get time to land before the cluster goes away
    } else if (warp == 1) {
        if (rank == lead) {
            const bool leader = elect_one();
            constexpr uint32_t idesc = idesc_bf16(2 * BM, BN, 0, 0);
            const uint32_t desc_a0 = desc_lo_k(smem_u32(smem));
            pdl_wait();                        // (the limit of the waits below counts from here)
            for (int kb = 0; kb < kblocks; ++kb) {
                const uint32_t s = kb % STAGES, ph = (kb / STAGES) & 1u;
                if (!(ok = mbar_wait(&bars->full[s], ph, abort_flag, status))) break;
                fence_after();
                const uint32_t da = desc_a0 + s * (STAGE >> 4), db = da + (A_BYTES >> 4);
                if (leader) {
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k) umma_ss_2cta(tmem_base, da + 2 * k, db + 2 * k, idesc, (kb | k) != 0);
                    umma_commit_2cta(&bars->empty[s], lead);
                }
                __syncwarp();
            }
            if (ok && leader) umma_commit_2cta(&bars->done, lead);
        }
    } else {
        pdl_wait();
        if (row_ok) sc = epi_row_scale(epp.p[dir], row);
        if (fin && pe.addend) out.add_fetch(io.add, n0, row0);         // the first columns' addend arrives while the products run
        ok = __all_sync(0xffffffffu, mbar_wait(&bars->done, 0, abort_flag, status));
        fence_after();
    }
    __syncwarp();
    cluster_sync();                            // every pair's products are done: nobody reads operand stages any more
    if (warp >= 2 && rows_live) {
        // the other owners' columns, times this product's row scale: the two warps of a quarter take half of each share's groups
#pragma unroll 1
        for (int o = 1; o < NP; ++o) {
            const int to = (share + o) % NP;   // (every pair begins with another owner)
            const uint32_t slot = cluster_addr(smem + (share < to ? share : share - 1) * SLOT, 2 * to + (rank & 1));
#pragma unroll
            for (int g = 0; g < F / 64; ++g) {
                const int grp = hf * (F / 64) + g;
                if (t0 + to * F + grp * 32 >= pe.N) continue;
                uint32_t r[32];
                tmem_ld_x32(tlane + to * F + grp * 32, r);
                tmem_wait_ld();
                const uint32_t dst = slot + (grp * 4 + q) * STG_BYTES + lane * 128;
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    st_cluster_f4(dst + ((j ^ (lane & 7)) << 4), __uint_as_float(r[4 * j]) * sc, __uint_as_float(r[4 * j + 1]) * sc, __uint_as_float(r[4 * j + 2]) * sc, __uint_as_float(r[4 * j + 3]) * sc);
            }
        }
    }
    __syncwarp();
    cluster_sync();                            // all parts have arrived
    if (fin && ok) {
        const EpiRow er(pe, row_ok ? row : 0);
        float ss = 0.f;
#pragma unroll
        for (int c0 = 0; c0 < 64; c0 += 32) {
            const int col = n0 + c0;
            if (col >= pe.N || !ok) break;
            if (pe.addend && c0 > 0) out.add_fetch(io.add, col, row0);
            uint32_t r[32];
            tmem_ld_x32(tlane + share * F + 64 * hf + c0, r);
            tmem_wait_ld();
            float v[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]) * sc;
#pragma unroll
            for (int i = 0; i < NP - 1; ++i) {
                const uint8_t *src = smem + i * SLOT + ((2 * hf + c0 / 32) * 4 + q) * STG_BYTES + lane * 128;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float4 p4 = *reinterpret_cast<const float4 *>(src + ((j ^ (lane & 7)) << 4));
                    v[4 * j] += p4.x; v[4 * j + 1] += p4.y; v[4 * j + 2] += p4.z; v[4 * j + 3] += p4.w;
                }
            }
            epi_pre<false>(pe, er, col, v);
            if (pe.addend) ok = out.add_take(v);
            if (ok) out.emit<false>(pe, io.c[1], io.u, n0, c0, row0, row, row_ok, v, ss);
        }
        if (lane == 0) bulk_wait_read0();      // (what the stores wrote is complete when the launch is)
    }
    if (warp >= 2 && !ok) sleep_ns(100000000ull);      // aborting: an addend load in flight gets time to land
    __syncwarp();
    fence_before();
    cluster_sync();
    if (warp == 1) {
        fence_after();
        tmem_dealloc_2cta(tmem_base, TMEM_COLS);
    }
}

int64_t tiles_of(const GemmArgs &a, int bn) { return (int64_t)((a.M + 2 * BM - 1) / (2 * BM)) * ((a.N + bn - 1) / bn); }

template <int NP, int BN> int resident_clusters() {
    static const int n = [] {
        if (cudaFuncSetAttribute(gemm_cluster_sum_kernel<NP, BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Tile<BN>::SMEM) != cudaSuccess) return 0;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(2 * NP); cfg.blockDim = dim3(NTHREADS); cfg.dynamicSmemBytes = Tile<BN>::SMEM;
        cudaLaunchAttribute at;
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = 2 * NP; at.val.clusterDim.y = 1; at.val.clusterDim.z = 1;
        cfg.attrs = &at; cfg.numAttrs = 1;
        int c = 0;
        return cudaOccupancyMaxActiveClusters(&c, gemm_cluster_sum_kernel<NP, BN>, &cfg) == cudaSuccess ? c : 0;
    }();
    return n;
}

template <int NP, int BN>
cudaError_t launch(const GemmArgs &a, const GemmArgs &b, cudaStream_t s) {
    CUtensorMap ma[2], mb[2];
    if (!make_map_2d(&ma[0], a.A, a.M, a.K, a.lda, BM) || !make_map_2d(&mb[0], a.B, a.N, a.K, a.ldb, BN / 2)) return cudaErrorInvalidValue;
    if (!make_map_2d(&ma[1], b.A, b.M, b.K, b.lda, BM) || !make_map_2d(&mb[1], b.B, b.N, b.K, b.ldb, BN / 2)) return cudaErrorInvalidValue;
    const EpiPair epp = epi_pair_of(a, &b);
    IoMaps io;
    memset(&io, 0, sizeof(io));
    const EpiArgs &p = epp.p[1];
    if (!make_map_out(&io.c[1], p, false)) return cudaErrorInvalidValue;
    if (p.addend && !make_map_f32_2d(&io.add, p.addend, p.M, p.N, p.ld_add, 32)) return cudaErrorInvalidValue;
    if (p.u && !make_map_half(&io.u, p.u, p.M, p.N, p.N)) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(gemm_cluster_sum_kernel<NP, BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Tile<BN>::SMEM);
    if (e != cudaSuccess) return e;
    int *status = device_status_ptr();
    if (!status) return cudaErrorUnknown;
    return launch_chain(gemm_cluster_sum_kernel<NP, BN>, (int)tiles_of(a, BN) * 2 * NP, NTHREADS, Tile<BN>::SMEM, s, 0, ma[0], mb[0], ma[1], mb[1], io, epp, status);
}

// One round of clusters.  A pair's time is that of its k-blocks: 0.31 us at 256 columns, 0.23 us at 128 (see gemm_tcgen05.cu), so the order here is by (k-blocks per pair) x
// (time of one): half of a product at 256 columns, a whole one at 128, a whole one at 256; the first whose clusters are all resident (of eight CTAs: 15 on 148 SMs, of four: 33).
enum Form { NONE, HALF_256, WHOLE_128, WHOLE_256 };
Form form_of(const GemmArgs &a) {
    if (a.N <= 128) return NONE;
    if (a.K > BK && tiles_of(a, 256) <= resident_clusters<4, 256>()) return HALF_256;
    if (tiles_of(a, 128) <= resident_clusters<2, 128>()) return WHOLE_128;
    return tiles_of(a, 256) <= resident_clusters<2, 256>() ? WHOLE_256 : NONE;
}

}  // namespace

bool gemm_cluster_sum_pays(const GemmArgs &a) { return form_of(a) != NONE; }

cudaError_t gemm_cluster_sum_launch(const GemmArgs &a, const GemmArgs &b, cudaStream_t s) {
    switch (form_of(a)) {
        case HALF_256: return launch<4, 256>(a, b, s);
        case WHOLE_128: return launch<2, 128>(a, b, s);
        case WHOLE_256: return launch<2, 256>(a, b, s);
        default: return cudaErrorNotSupported;
    }
}

}  // namespace dm
