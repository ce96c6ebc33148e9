// bf16 x bf16 -> fp32 GEMM on the 5th-generation tensor cores, for the dense projections:
//     C[m, n] = row_scale[m] * sum_k A[m, k] * B[n, k] + addend[m, n]
// This file chooses the kernel and its tile: gemm_rows.cu for up to 128 rows (reading the weights is nearly all such a product does), gemm_pair.cu for more, and gemm_cluster.cu for
// a sum of two products whose tiles are few.
// All: operands staged by TMA with the 128-byte swizzle, accumulators in TMEM, mbarrier pipelines.
#include "gemm_epi.cuh"

namespace dm {
namespace {

using namespace tc;

constexpr int BM = 128;

// Tile width of the pair kernel, by rounds of CTA pairs.  A k-block of a 256 x 256 tile takes 0.31 us, of a 256 x 128 one 0.23 us (its operands, 24 KB
// per CTA, then arrive at 15 TB/s over all SMs: what L2 delivers, while its products take half of that time), so a narrow round counts 0.74.
bool pair_wide_tile(const GemmArgs &a, int nprob) { return a.N > 128 && gemm_pair_cost(true, a, nprob) <= gemm_pair_cost(false, a, nprob); }

// Which kernel for up to 128 rows.  gemm_rows.cu is the faster reader of weights, but what it does per row -- a row's scale from its sums of squares, one round trip to memory after the other,
// and its stores -- shows where the products are short.  K up to 768, more than 80 rows with such scales or 96 without: few-row kernel / pair kernel 128 x 2000 x 512 12.5 / 10.4 us, 12 decoding
// layers of 96 tokens 344 / 298 us at d_model 512, 377 / 300 at 256; K = 1024: level at 128 rows, 10.4 / 12.5 us at 80.  More tiles than two to an SM go to its looping form at any K
// (128 x 50304 x 512: 18.5 / 22.7 us); so do outputs that the pair kernel cannot store through TMA (100 x 300 x 512, bf16 rows of 600 bytes with an addend: 12.5 / 24 us).
bool few_rows(const GemmArgs &a, int nprob) {
    if (a.M > BM) return false;
    return a.M <= (a.rs_ssq ? 80 : 96) || a.K > 768 || !gemm_tma_io(a) || (int64_t)((a.N + BM - 1) / BM) * nprob > 2 * sm_count();
}

cudaError_t dispatch(const GemmArgs &a, const GemmArgs *b, cudaStream_t s) {
    if (few_rows(a, b ? 2 : 1)) return gemm_rows_launch(a, b, false, s);
    return gemm_pair_launch(pair_wide_tile(a, b ? 2 : 1), a, b, s);
}

}  // namespace

bool gemm_tcgen05_supports(const GemmArgs &a) {
    if (!gemm_tensor_ok(a)) return false;
    if (a.u && (a.c_dtype != DM_F32 || !gemm_tma_io(a) || ((reinterpret_cast<uintptr_t>(a.u) | reinterpret_cast<uintptr_t>(a.u_w)) & 15u) || (a.N % 8))) return false;
    return encode_fn() != nullptr;
}

cudaError_t gemm_tcgen05(const GemmArgs &a, cudaStream_t s) {
    if (!gemm_tcgen05_supports(a)) return cudaErrorNotSupported;
    return dispatch(a, nullptr, s);
}

bool gemm_tcgen05_pair_supports(const GemmArgs &a, const GemmArgs &b) {
    return gemm_tcgen05_supports(a) && gemm_tcgen05_supports(b) && a.M == b.M && a.N == b.N && a.K == b.K && !a.m_dev && !b.m_dev &&
           a.c_dtype == b.c_dtype;
}

cudaError_t gemm_tcgen05_pair(const GemmArgs &a, const GemmArgs &b, cudaStream_t s) {
    if (!gemm_tcgen05_pair_supports(a, b)) return cudaErrorNotSupported;
    return dispatch(a, &b, s);
}

bool gemm_tcgen05_sum_supports(const GemmArgs &a, const GemmArgs &b) { return gemm_sum_ok(a, b) && gemm_tcgen05_supports(a) && gemm_tcgen05_supports(b); }

cudaError_t gemm_tcgen05_sum(const GemmArgs &a, const GemmArgs &b, cudaStream_t s) {
    if (!gemm_tcgen05_sum_supports(a, b)) return cudaErrorNotSupported;
    if (a.M <= BM) return gemm_rows_launch(a, &b, true, s);
    return gemm_cluster_sum_pays(b) ? gemm_cluster_sum_launch(a, b, s) : gemm_pair_sum_launch(a, b, s);
}

}  // namespace dm
