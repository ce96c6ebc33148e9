// bf16 x bf16 -> fp32 GEMM on the 5th-generation tensor cores (tcgen05.mma, accumulators in TMEM,
// operands staged by TMA with the 128-byte swizzle, mbarrier pipeline), for the dense projections:
//     C[m, n] = row_scale[m] * sum_k A[m, k] * B[n, k] + addend[m, n]
// This file: the choice of the kernel and its tile, and the kernel for up to 128 rows.  More rows: gemm_pair.cu.
//
// Up to 128 rows: persistent, one CTA per SM, CTA tile 128 x BN, K step 64.  Warp roles: warp 0 issues the TMA
// loads, warp 1 owns TMEM and issues the MMAs, warps 2-5 drain the accumulator (double-buffered in
// TMEM, so the epilogue of one tile overlaps the main loop of the next).
//
// Every wait on an mbarrier is bounded by wall time; when one gives up the CTA raises an abort flag,
// stores DM_ERR_TIMEOUT in the device status word, waits (bounded) for its own TMA loads, frees its
// TMEM and returns.
#include "gemm_epi.cuh"

namespace dm {
namespace {

using namespace tc;

constexpr int BM = 128, BK = 64, NTHREADS = 192;
constexpr int MAX_STAGES = 6;
// pipeline depth: as many (A, B) stages as shared memory holds -- 4 x 48 KB with 256-column tiles, 6 x 32 KB with 128-column tiles (whose
// lower arithmetic intensity needs more bytes in flight per MMA clock)
__host__ __device__ constexpr int stages_for(int bn) { return bn == 128 ? 6 : 4; }

struct __align__(8) PipeBars {
    uint64_t full[MAX_STAGES], empty[MAX_STAGES], tmem_full[2], tmem_empty[2];
    uint32_t tmem_base;
    int abort;
};

template <int BN>
__global__ void __launch_bounds__(NTHREADS, 1)
gemm_tc_kernel(const __grid_constant__ CUtensorMap map_a0, const __grid_constant__ CUtensorMap map_b0,
               const __grid_constant__ CUtensorMap map_a1, const __grid_constant__ CUtensorMap map_b1,
               const __grid_constant__ EpiPair epp, int *status) {
    const EpiArgs &ep = epp.p[0];              // sizes are common to all problems
    extern __shared__ uint8_t smem_raw[];
    // 1024-byte aligned base, derived by offsetting the __shared__ array so that accesses stay shared-space loads and stores
    uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    constexpr int STAGES = stages_for(BN);
    constexpr uint32_t A_BYTES = BM * BK * 2, B_BYTES = BN * BK * 2, STAGE_BYTES = A_BYTES + B_BYTES;
    PipeBars *bars = reinterpret_cast<PipeBars *>(smem + STAGES * STAGE_BYTES);
    volatile int *abort_flag = &bars->abort;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // rows to compute: all of them, or the count another kernel left on the device
    const int M_eff = ep.m_dev ? min(ep.M, max(0, *ep.m_dev - ep.m_off)) : ep.M;
    const int tiles_n = (ep.N + BN - 1) / BN, num_tiles = M_eff > 0 ? tiles_n * epp.nprob : 0;         // the problems sit side by side along N
    const int kblocks = (ep.K + BK - 1) / BK;
    constexpr uint32_t TMEM_COLS = 2 * BN;          // two accumulator buffers

    if (threadIdx.x == 0) {
        for (int i = 0; i < STAGES; ++i) { mbar_init(&bars->full[i], 1); mbar_init(&bars->empty[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&bars->tmem_full[i], 1); mbar_init(&bars->tmem_empty[i], 4); }
        bars->abort = 0;
        mbar_fence_init();
    }
    if (warp == 1) {
        tmem_alloc(&bars->tmem_base, TMEM_COLS);
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem_base = bars->tmem_base;

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer (one lane)
        if (lane == 0) {
            uint32_t it = 0;
            bool ok = true;
            for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
                const int prob = tile / tiles_n, n0 = (tile - prob * tiles_n) * BN;
                const int prod = epp.ksplit ? prob >> 1 : prob, k_off = epp.p[prob].k_off;
                const CUtensorMap *ma = prod ? &map_a1 : &map_a0, *mb = prod ? &map_b1 : &map_b0;
                for (int kb = 0; kb < kblocks; ++kb, ++it) {
                    const uint32_t s = it % STAGES, ph = (it / STAGES) & 1u;
                    if (!(ok = mbar_wait(&bars->empty[s], ph ^ 1u, abort_flag, status))) break;
                    uint8_t *sa = smem + s * STAGE_BYTES, *sb = sa + A_BYTES;
                    mbar_expect_tx(&bars->full[s], STAGE_BYTES);
                    tma_load_2d(sa, ma, k_off + kb * BK, 0, &bars->full[s]);
                    tma_load_2d(sb, mb, k_off + kb * BK, n0, &bars->full[s]);
                }
            }
            if (!ok) {
                // aborting: give the loads already issued a bounded chance to land before the CTA goes away
                const uint32_t first = it > STAGES ? it - STAGES : 0;
                for (uint32_t j = first; j < it; ++j) {
                    mbar_wait_quiet(&bars->full[j % STAGES], (j / STAGES) & 1u, 100000000ull);
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer (one lane)
        if (lane == 0) {
            constexpr uint32_t idesc = idesc_bf16(BM, BN, 0, 0);
            uint32_t it = 0, tcount = 0;
            bool ok = true;
            for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x, ++tcount) {
                const uint32_t buf = tcount & 1u, bph = (tcount >> 1) & 1u;
                if (!(ok = mbar_wait(&bars->tmem_empty[buf], bph ^ 1u, abort_flag, status))) break;
                fence_after();
                const uint32_t d_tmem = tmem_base + buf * BN;
                for (int kb = 0; kb < kblocks; ++kb, ++it) {
                    const uint32_t s = it % STAGES, ph = (it / STAGES) & 1u;
                    if (!(ok = mbar_wait(&bars->full[s], ph, abort_flag, status))) break;
                    fence_after();
                    const uint32_t sa = smem_u32(smem + s * STAGE_BYTES), sb = sa + A_BYTES;
                    const uint64_t da = desc_k_sw128(sa), db = desc_k_sw128(sb);
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k)          // 32 bytes along K per MMA: +2 in 16-byte units
                        umma_bf16(d_tmem, da + 2 * k, db + 2 * k, idesc, (kb | k) != 0);
                    umma_commit(&bars->empty[s]);          // frees the stage when these MMAs have read it
                }
                if (ok) umma_commit(&bars->tmem_full[buf]);
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue: 4 warps, one TMEM lane quarter each
        const int q = warp & 3;                            // warps 2,3,4,5 -> quarters 2,3,0,1
        const int row = q * 32 + lane;
        const bool row_ok = row < M_eff;
        uint32_t tcount = 0;
        bool ok = true;
        for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x, ++tcount) {
            const uint32_t buf = tcount & 1u, bph = (tcount >> 1) & 1u;
            const int prob = tile / tiles_n, n0 = (tile - prob * tiles_n) * BN;
            const EpiArgs &pe = epp.p[prob];               // this tile's problem: its output, scales and addend
            const float sc = row_ok ? epi_row_scale(pe, row) : 1.f;
            const EpiRow er(pe, row);
            ok = mbar_wait(&bars->tmem_full[buf], bph, abort_flag, status);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            fence_after();
#pragma unroll 1
            for (int c0 = 0; c0 < BN; c0 += 32) {
                uint32_t r[32];
                tmem_ld_x32(tmem_base + ((uint32_t)(q * 32) << 16) + buf * BN + c0, r);
                tmem_wait_ld();
                const int col = n0 + c0;
                if (!row_ok || col >= pe.N) continue;
                float v[32];
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]) * sc;
                epi_pre<true>(pe, er, col, v);
                epi_add_store(pe, er, row, col, v);
            }
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->tmem_empty[buf]);
        }
    }
    // ---------------------------------------------------------------- teardown
    fence_before();
    __syncthreads();
    if (warp == 1) {
        fence_after();
        tmem_dealloc(tmem_base, TMEM_COLS);
    }
}

// b == NULL: one product.  hi != NULL (two products, fp32 outputs): each product is cut in two along K; the first half goes to the
// product's own C with its addend and bias, the second half to hi[i] (same pitch), scaled like the first (the scales are linear).
template <int BN>
cudaError_t launch(const GemmArgs &a, const GemmArgs *b, float *const *hi, cudaStream_t s) {
    CUtensorMap ma[2], mb[2];
    if (!make_map_2d(&ma[0], a.A, a.M, a.K, a.lda, BM) || !make_map_2d(&mb[0], a.B, a.N, a.K, a.ldb, BN)) return cudaErrorInvalidValue;
    ma[1] = ma[0]; mb[1] = mb[0];
    if (b && (!make_map_2d(&ma[1], b->A, b->M, b->K, b->lda, BM) || !make_map_2d(&mb[1], b->B, b->N, b->K, b->ldb, BN))) return cudaErrorInvalidValue;
    constexpr size_t smem = stages_for(BN) * (size_t)(BM * BK * 2 + BN * BK * 2) + sizeof(PipeBars) + 1024;
    cudaError_t e = cudaFuncSetAttribute(gemm_tc_kernel<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int *status = device_status_ptr();
    if (!status) return cudaErrorUnknown;
    const EpiPair epp = epi_pair_of(a, b, hi);
    const int tiles = ((a.N + BN - 1) / BN) * epp.nprob;
    const int grid = tiles < sm_count() ? tiles : sm_count();
    gemm_tc_kernel<BN><<<grid, NTHREADS, smem, s>>>(ma[0], mb[0], ma[1], mb[1], epp, status);
    count_launch();
    return cudaGetLastError();
}

int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

// Tile width of the kernel for up to 128 rows, by rounds of CTAs: a 128 x 256 tile costs about 1.6 times a 128 x 128 one (it fetches 1.5
// times the operands for twice the products), so the wide tile wins whenever it saves a round -- also when it leaves a single round partly empty.
bool wide_tile(const GemmArgs &a, int nprob) {
    const int64_t sms = sm_count(), rounds128 = ceil_div(ceil_div(a.N, 128) * nprob, sms), rounds256 = ceil_div(ceil_div(a.N, 256) * nprob, sms);
    return !(a.N <= 128 || 10 * rounds128 <= 16 * rounds256);
}

// Tile width of the pair kernel, by rounds of CTA pairs.  A k-block of a 256 x 256 tile takes 0.31 us, of a 256 x 128 one 0.23 us (its operands, 24 KB
// per CTA, then arrive at 15 TB/s over all SMs: what L2 delivers, while its products take half of that time), so a narrow round counts 0.7.
bool pair_wide_tile(const GemmArgs &a, int nprob) {
    const int64_t pairs = sm_count() / 2, tm = ceil_div(a.M, 256);
    const int64_t r256 = ceil_div(tm * ceil_div(a.N, 256) * nprob, pairs), r128 = ceil_div(tm * ceil_div(a.N, 128) * nprob, pairs);
    return a.N > 128 && 10 * r256 <= 7 * r128;
}

cudaError_t dispatch(const GemmArgs &a, const GemmArgs *b, float *const *hi, cudaStream_t s) {
    const int nprob = hi ? 4 : b ? 2 : 1;
    if (a.M > BM) return gemm_pair_launch(pair_wide_tile(a, nprob), a, b, hi, s);
    return wide_tile(a, nprob) ? launch<256>(a, b, hi, s) : launch<128>(a, b, hi, s);
}

}  // namespace

bool gemm_tcgen05_supports(const GemmArgs &a) {
    if (a.in_dtype != DM_BF16) return false;
    if (a.M <= 0 || a.N <= 0 || a.K <= 0) return false;
    if ((a.lda % 8) || (a.ldb % 8)) return false;                                   // TMA: 16-byte row pitch
    if ((reinterpret_cast<uintptr_t>(a.A) & 15u) || (reinterpret_cast<uintptr_t>(a.B) & 15u)) return false;
    if (reinterpret_cast<uintptr_t>(a.C) & 15u) return false;
    if (a.addend && (reinterpret_cast<uintptr_t>(a.addend) & 15u)) return false;
    if (a.col_bias && (reinterpret_cast<uintptr_t>(a.col_bias) & 15u)) return false;
    if (a.col_scale && ((reinterpret_cast<uintptr_t>(a.col_scale) & 15u) || ((a.ld_cs > 0 ? a.ld_cs : (int64_t)a.N) & 3))) return false;
    if (a.rs_ssq && (reinterpret_cast<uintptr_t>(a.rs_ssq) & 15u)) return false;
    if (a.u && (a.M <= BM || a.c_dtype != DM_F32 || !gemm_pair_tma_io(a) || ((reinterpret_cast<uintptr_t>(a.u) | reinterpret_cast<uintptr_t>(a.u_w)) & 15u) || (a.N % 8))) return false;
    return encode_fn() != nullptr;
}

cudaError_t gemm_tcgen05(const GemmArgs &a, cudaStream_t s) {
    if (!gemm_tcgen05_supports(a)) return cudaErrorNotSupported;
    return dispatch(a, nullptr, nullptr, s);
}

bool gemm_tcgen05_pair_supports(const GemmArgs &a, const GemmArgs &b) {
    return gemm_tcgen05_supports(a) && gemm_tcgen05_supports(b) && a.M == b.M && a.N == b.N && a.K == b.K && !a.m_dev && !b.m_dev &&
           a.c_dtype == b.c_dtype;
}

cudaError_t gemm_tcgen05_pair(const GemmArgs &a, const GemmArgs &b, cudaStream_t s) {
    if (!gemm_tcgen05_pair_supports(a, b)) return cudaErrorNotSupported;
    return dispatch(a, &b, nullptr, s);
}

bool gemm_tcgen05_sum_supports(const GemmArgs &a, const GemmArgs &b) {
    return gemm_tcgen05_supports(b) && gemm_tcgen05_supports(a) && a.M == b.M && a.N == b.N && a.K == b.K && a.M > BM && !a.m_dev && !b.m_dev && gemm_pair_tma_io(b);
}

cudaError_t gemm_tcgen05_sum(const GemmArgs &a, const GemmArgs &b, cudaStream_t s) {
    if (!gemm_tcgen05_sum_supports(a, b)) return cudaErrorNotSupported;
    return gemm_pair_sum_launch(a, b, s);
}

// Few rows and a long K (the out_proj pair of block decoding): whole products fill less than half of the SMs.  Halving K instead doubles
// the number of tiles of the same shape.
bool gemm_tcgen05_pair_splitk_pays(const GemmArgs &a, const GemmArgs &b) {
    if (!gemm_tcgen05_pair_supports(a, b) || a.c_dtype != DM_F32 || a.K % (2 * BK) || a.gelu || b.gelu || a.silu_cols || b.silu_cols) return false;
    const int64_t tiles = ceil_div(a.M, BM) * ceil_div(a.N, 256) * 2;
    return a.N > 128 && 2 * tiles <= sm_count();
}

cudaError_t gemm_tcgen05_pair_splitk(const GemmArgs &a, const GemmArgs &b, float *a_hi, float *b_hi, cudaStream_t s) {
    if (!gemm_tcgen05_pair_splitk_pays(a, b) || !a_hi || !b_hi || ((reinterpret_cast<uintptr_t>(a_hi) | reinterpret_cast<uintptr_t>(b_hi)) & 15u))
        return cudaErrorNotSupported;
    float *const hi[2] = {a_hi, b_hi};
    return dispatch(a, &b, hi, s);
}

}  // namespace dm
