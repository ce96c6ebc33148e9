// Internal declarations shared by the translation units of libdm_bimamba.so (not part of the ABI).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <initializer_list>

#include "dm_bimamba.h"

namespace dm {

// Every kernel launch goes through this counter (dm_kernel_launch_count()).
void count_launch(int n = 1);

// Device status word written by kernels whose bounded waits expire; read and cleared by dm_check().
int *device_status_ptr();

// Programmatic dependent launch along the chain of kernels that one call of the library enqueues: a kernel starts its set-up (and, in the GEMMs, the loads of its
// weights) while the one before it is finishing, and waits for that one's completion before it touches anything a kernel of the chain reads or writes.
//   - Every kernel launched through launch_chain calls pdl_wait() in each thread that accesses such memory, and pdl_trigger() only after it: the next kernel can
//     then rely on everything before this one being complete, and the weights it reads early were not written by this kernel.
//   - The first kernel of a call is launched without the attribute (chain_begin): it follows the caller's work in stream order, completely.
// A decoding pass of 24 layers is 75 to 120 kernels of 4 to 35 us: 1236 -> 974 us for one sequence (hybrid, 2.4 GB of weights), 2449 -> 2302 us for 16; a single
// layer of 1024 tokens 140 -> 136 us.
inline thread_local bool g_chain = false;
inline void chain_begin() { g_chain = false; }
// Before the launch of a kernel of few CTAs that each run long and could share an SM: behind a grid of `ahead` CTAs that covers the GPU it is launched without overlap.  Ahead of time its CTAs
// would be packed onto the SMs that have the most room at that moment and stay there: chunk-32 scan of 1 x 4096 tokens, 32 heads, behind 192 prep CTAs 674 us, 472 us spread out;
// fp32 layer of 1 x 8192 tokens, 8 heads, 830 and 589 us.  Behind a grid that leaves SMs empty the overlap does no harm (1 x 1024: 113 us either way).
inline void chain_spread(int64_t ahead, int64_t ctas, int sms) {
    if (ahead > sms && ctas < 2 * sms) chain_begin();
}
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename... P, typename... A>
inline cudaError_t launch_chain(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, int cluster, A &&...args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s;
    cudaLaunchAttribute at[2];
    int n = 0;
    if (cluster > 0) {                       // (0: the kernel's own cluster size)
        at[n].id = cudaLaunchAttributeClusterDimension;
        at[n].val.clusterDim.x = cluster; at[n].val.clusterDim.y = 1; at[n].val.clusterDim.z = 1;
        ++n;
    }
    if (g_chain) {
        at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    cfg.attrs = at; cfg.numAttrs = n;
    g_chain = true;
    count_launch();
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}
#endif

inline size_t dtype_size(int dtype) { return dtype == DM_BF16 ? 2 : 4; }
inline size_t align_up(size_t v, size_t a = 256) { return (v + a - 1) / a * a; }

// ---------------------------------------------------------------------------------------------
// GEMM:  C[m, n] = row_scale[m] * sum_k A[m, k] * B[n, k]  +  addend[m, n]
// A [M, K] (lda), B [N, K] (ldb): in_dtype.  C [M, N] (ldc): c_dtype.  row_scale [M] fp32 or NULL.
// addend [M, N] (ld_add) fp32 or NULL; it may alias C when c_dtype is DM_F32 and ldc == ld_add.
// ---------------------------------------------------------------------------------------------
struct GemmArgs {
    const void *A; int64_t lda;
    const void *B; int64_t ldb;
    void *C; int64_t ldc;
    int in_dtype, c_dtype;
    int M, N, K;
    const float *row_scale;
    const float *addend; int64_t ld_add;
    int silu_cols;           // output columns [0, silu_cols) get SiLU applied (0 = none)
    // Epilogue order: v = acc * row_scale[r] + col_bias[c];  v = act(v);  v *= col_scale[(r / cs_rows) * ld_cs + c];  v += addend[r, c]
    const float *col_bias;   // [N] or NULL
    int gelu;                // GELU (tanh form) on every output column
    const float *col_scale;  // [ceil(M / cs_rows), ld_cs] or NULL: one scale vector per group of cs_rows consecutive rows
    int cs_rows;
    int64_t ld_cs;           // row pitch of col_scale (0 = N)
    // Row scale from sums of squares instead of row_scale: rsqrt(sum(rs_ssq[r * rs_n .. + rs_n)) * rs_inv + rs_eps); NULL = none
    const float *rs_ssq; int rs_n; float rs_inv, rs_eps;
    // The next RMSNorm's input (fp32 C, tensor-core kernels only): u[r, c] = bf16(C[r, c] * u_w[c]) with row pitch N, and u_ssq[r, j] = sum of
    // C[r, c]^2 over the columns [64 j, 64 j + 64), row pitch ceil(N / 64).  The norm's row scale is left to the product that reads u (rs_ssq); NULL = none
    void *u; const void *u_w; float *u_ssq;
    const int *m_dev;        // device int or NULL: only rows [0, clamp(*m_dev - m_off, 0, M)) are computed (row count known on the device only)
    int m_off;
};
// What the tensor-core kernels take: bf16 operands in 16-byte rows (TMA), and 16-byte alignment of what their epilogues read as vectors.
inline bool gemm_tensor_ok(const GemmArgs &a) {
    auto off16 = [](const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) != 0; };
    if (a.in_dtype != DM_BF16 || a.M <= 0 || a.N <= 0 || a.K <= 0 || a.lda % 8 || a.ldb % 8) return false;
    if (off16(a.A) || off16(a.B) || off16(a.C) || off16(a.addend) || off16(a.col_bias)) return false;
    if (a.col_scale && (off16(a.col_scale) || (a.ld_cs > 0 ? a.ld_cs : (int64_t)a.N) % 4)) return false;
    if (a.rs_ssq && a.rs_n % 4 == 0 && off16(a.rs_ssq)) return false;       // (read as float4 where a row holds whole ones, one by one elsewhere)
    return true;
}
// Output and addend can go through TMA: 16-byte aligned rows.
inline bool gemm_tma_io(const GemmArgs &a) {
    return (a.ldc * (int64_t)dtype_size(a.c_dtype)) % 16 == 0 && (!a.addend || a.ld_add % 4 == 0);
}
// The sum of two products in one launch: its epilogues know scales and, for fp32 outputs, the addend; no bias and no activation.
inline bool gemm_sum_ok(const GemmArgs &a, const GemmArgs &b) {
    for (const GemmArgs *p : {&a, &b})
        if (!gemm_tensor_ok(*p) || p->m_dev || p->col_bias || p->gelu || p->silu_cols) return false;
    return a.M == b.M && a.N == b.N && a.K == b.K && gemm_tma_io(b) && !(b.addend && b.c_dtype == DM_BF16);
}
cudaError_t gemm_simple(const GemmArgs &a, cudaStream_t s);
// fp32 products that do not fill the GPU: n of them (same sizes) in one launch, or both into b's output (sum).
bool gemm_f32_supports(const GemmArgs &a, int n);
cudaError_t gemm_f32(const GemmArgs &a, const GemmArgs *b, bool sum, cudaStream_t s);
// Tensor-core path (tcgen05 + TMEM + TMA).  Returns cudaErrorNotSupported for shapes it does not take.
cudaError_t gemm_tcgen05(const GemmArgs &a, cudaStream_t s);
bool gemm_tcgen05_supports(const GemmArgs &a);
// Two problems of equal M, N, K and output type in one launch (same tile loop, one tail round).  The problems must be independent
// of each other: neither reads what the other writes.
bool gemm_tcgen05_pair_supports(const GemmArgs &a, const GemmArgs &b);
cudaError_t gemm_tcgen05_pair(const GemmArgs &a, const GemmArgs &b, cudaStream_t s);
// C = (s_a A_a) B_a^T + (s_b A_b) B_b^T + addend in one pass (s: each problem's row scale; output, addend, column scale and u from b).
bool gemm_tcgen05_sum_supports(const GemmArgs &a, const GemmArgs &b);
cudaError_t gemm_tcgen05_sum(const GemmArgs &a, const GemmArgs &b, cudaStream_t s);

// ---------------------------------------------------------------------------------------------
// Fused conv + SiLU + discretisation + selective scan + gate, both directions in one launch.
// ---------------------------------------------------------------------------------------------
struct ScanDir {
    const void *conv_w, *conv_b, *norm_w;
    const float *dt_bias, *A_log, *D;
};
struct ScanArgs {
    int B, L, d_inner, H, P, N, k;
    int d_in_proj;           // row pitch of zx in elements (>= 2 d_inner + 2 N + H; the columns beyond are padding)
    int conv_ch;
    int dtype, flags, dir_mask, chunk;
    const void *zx;          // [2][B*L][d_in_proj] dtype: in_proj output of each direction
    int zx_tied;             // both directions read zx[0] (shared in_proj, DM_FLAG_TIED_PROJ)
    int z_gated;             // the z columns of zx already hold SiLU(z) (applied by the in_proj epilogue); the tensor-core scan requires it
    void *g;                 // [2][B*L][d_inner]   dtype: gated output (times norm_w when the norm is on)
    float *ssq;              // [2][B*L][H] per-head sum of squares of the gated output (norm on), or [2][B*L][scan_ssq_parts] of smaller pieces, or NULL
    int ssq_room;            // pieces per row that fit at ssq
    ScanDir dir[2];
    const float *ssm_in;     // [B,H,P,N] or NULL   (left-to-right direction only)
    const void *conv_in;     // [B,k-1,conv_ch] or NULL
    float *ssm_out;          // [B,H,P,N] or NULL
};
size_t scan_seq_workspace_bytes(const ScanArgs &a);
cudaError_t scan_sequential(const ScanArgs &a, void *ws, cudaStream_t s);
bool scan_ssd_supports(const ScanArgs &a);
// chunk values the chunked bf16 path takes (0 = default, 32 = CUDA-core kernel, 128 = tensor-core kernel); other paths take any chunk > 0
bool scan_ssd_chunk_ok(int dtype, int d_state, int chunk);
void scan_ssd_selftest_withhold(int on);
bool scan_selftest_withheld();
// Sums of squares per row that scan_ssd writes: one per head, or (narrow state, with that room) one per 32 channels, whatever the batch
int scan_ssq_parts(const ScanArgs &a);
size_t scan_ssd_workspace_bytes(const ScanArgs &a);
cudaError_t scan_ssd(const ScanArgs &a, void *ws, cudaStream_t s);

// Bidirectional multi-head attention over qkv [B*L, 3 d] (columns [Q | K | V], heads contiguous inside each) -> out [B*L, d];
// bf16, head width 64 or 80.
bool attention_supports(int dtype, int d, int n_heads);
// k_cache != NULL: block mode -- the block's K, V are appended at rows [cache_len, cache_len + L) of the caches [B, cache_cap, d]
// and the queries attend to the first cache_len + L rows.
cudaError_t attention_forward(const void *qkv, void *out, int B, int L, int d, int n_heads, void *k_cache, void *v_cache,
                              int cache_len, int cache_cap, cudaStream_t s);

// The same for few queries (up to ATTN_BLOCK_MAX_Q) and few (head, sequence) pairs: see attention_block.cu; attention_forward chooses.
constexpr int ATTN_BLOCK_MAX_Q = 64;
cudaError_t attention_block(const void *qkv, void *out, int B, int L, int d, int n_heads, void *k_cache, void *v_cache, int cache_len,
                            int cache_cap, cudaStream_t s);

// ---------------------------------------------------------------------------------------------
// Small row-wise kernels
// ---------------------------------------------------------------------------------------------
// rstd[dir][t] = rsqrt(sum_h ssq[dir][t][h] / d_inner + eps)
cudaError_t rstd_from_ssq(const float *ssq, float *rstd, int rows, int H, int d_inner, float eps, cudaStream_t s);
// r[t, :] = embed[tokens[t], :]  (fp32 residual stream)
cudaError_t embed_gather(const void *embed, int dtype, const int32_t *tokens, float *r, int T, int d, int vocab, cudaStream_t s);
// u[t, :] = r[t, :] * rsqrt(mean(r[t]^2) + eps) * w
cudaError_t rmsnorm_rows(const float *r, const void *w, void *u, int dtype, int T, int d, float eps, cudaStream_t s);
// u[t, :] = gamma[t / L, :] * (r[t, :] - mean) / sqrt(var + eps) + beta[t / L, :]   (gamma, beta: rows of pitch ld_mod)
cudaError_t adaln_rows(const float *r, const float *gamma, const float *beta, int64_t ld_mod, void *u, int dtype, int T, int L, int d,
                       float eps, cudaStream_t s);
// mod[b, :] = b_cond + W_cond tau[b, :]   (W_cond [n_out, d_c] dtype, b_cond [n_out] fp32 or NULL, tau [B, d_c] fp32)
cudaError_t modulation_rows(const float *tau, const void *w_cond, const float *b_cond, float *mod, int dtype, int B, int n_out, int d_c,
                            cudaStream_t s);
// Reverse step (Sec. 2, Eq. 3): tokens_out = tokens_in; idx[0..*count) = positions drawn this step (masked and u_keep >= keep_prob)
cudaError_t select_drawn(const int32_t *tokens_in, const float *u_keep, float keep_prob, int mask_id, int32_t *tokens_out, int32_t *idx,
                         int *count, int T, cudaStream_t s);
// dst[j, :] = src[idx[j], :] for j < *count
cudaError_t gather_rows(const void *src, const int32_t *idx, const int *count, void *dst, int dtype, int T, int d, cudaStream_t s);
// tokens_out[idx[row0 + r]] = inverse-CDF draw at u_cat from softmax(logits[r, 0..vocab_real) without mask_id), r < rows, row0 + r < *count
cudaError_t draw_rows(const void *logits, int64_t ld, int dtype, const int32_t *idx, const int *count, int row0, int rows,
                      const float *u_cat, int mask_id, int vocab_real, int32_t *tokens_out, cudaStream_t s);
// out[t] = argmax_v logits[t, v], lowest index on ties
cudaError_t argmax_rows(const void *logits, int dtype, int32_t *out, int T, int V, cudaStream_t s);
// Tied projections: g0[t, :] = s0[t] * g0[t, :] + s1[t] * g1[t, :]  (s = rstd of each direction, or 1 when rstd is NULL), in place over g0
cudaError_t combine_directions(void *g0, const void *g1, const float *rstd0, const float *rstd1, int dtype, int64_t T, int d_inner, cudaStream_t s);
// conv_out[b] = last k-1 rows of concat(conv_in[b] (or zeros), xBC columns of zx[b, 0..L-1])
cudaError_t conv_state_update(const void *zx_fwd, const void *conv_in, void *conv_out, int dtype, int B, int L,
                              int k, int d_inner, int conv_ch, int d_in_proj, cudaStream_t s);

// One CTA whose waits run out by design (see selftest.cu); out: 3 x uint64 on the device
cudaError_t selftest_wait_timeout(unsigned long long limit_ns, unsigned long long *out, cudaStream_t s);

}  // namespace dm
