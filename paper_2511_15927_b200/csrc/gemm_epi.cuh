// Epilogue shared by the tensor-core GEMM kernels: what happens to 32 consecutive accumulator columns of one output row.
#pragma once

#include "dm_internal.h"
#include "tc_ptx.cuh"

namespace dm {
namespace tc {

struct EpiArgs {
    void *C; int64_t ldc; int c_is_f32;
    const float *row_scale; const float *addend; int64_t ld_add;
    int M, N, K;
    int silu_cols;   // SiLU on output columns below this one
    const float *col_bias; int gelu; const float *col_scale; int cs_rows; int64_t ld_cs;   // see GemmArgs
    const int *m_dev; int m_off;
    const float *rs_ssq; int rs_n; float rs_inv, rs_eps;
    __nv_bfloat16 *u; const __nv_bfloat16 *u_w; float *u_ssq;
};

// Up to two products of the same M, N, K in one launch (the two directions' in_proj or out_proj): the tile loop runs over both, so that they share one tail round and
// -- for in_proj, whose A operand is the same x -- the rows of A in L2.
struct EpiPair {
    EpiArgs p[2];
    int nprob;
    int n_fast;      // tile order: consecutive tiles step along N (the A rows are streamed once, B stays in L2) or along M
};

inline EpiArgs epi_of(const GemmArgs &a) {
    return EpiArgs{a.C, a.ldc, a.c_dtype == DM_F32 ? 1 : 0, a.row_scale, a.addend, a.ld_add, a.M, a.N, a.K, a.silu_cols,
                   a.col_bias, a.gelu, a.col_scale, a.cs_rows > 0 ? a.cs_rows : 1, a.ld_cs > 0 ? a.ld_cs : (int64_t)a.N, a.m_dev, a.m_off,
                   a.rs_ssq, a.rs_n, a.rs_inv, a.rs_eps, static_cast<__nv_bfloat16 *>(a.u), static_cast<const __nv_bfloat16 *>(a.u_w), a.u_ssq};
}

inline EpiPair epi_pair_of(const GemmArgs &a, const GemmArgs *b) {
    EpiPair epp{};
    epp.p[0] = epi_of(a);
    epp.p[1] = b ? epi_of(*b) : epp.p[0];
    epp.nprob = b ? 2 : 1;
    epp.n_fast = a.M > a.N ? 1 : 0;
    return epp;
}

// What is the same for every column of a thread's row
struct EpiRow {
    bool wide_c, wide_add;     // 32-byte stores / loads (one full sector per thread): every row of C / of the addend starts on a 32-byte boundary
    const float *add_row, *cs_row;
    __device__ __forceinline__ EpiRow(const EpiArgs &ep, int row) {
        const int c_es = ep.c_is_f32 ? 4 : 2;
        wide_c = (reinterpret_cast<uintptr_t>(ep.C) & 31u) == 0 && ((ep.ldc * c_es) & 31) == 0;
        wide_add = ep.addend && (reinterpret_cast<uintptr_t>(ep.addend) & 31u) == 0 && ((ep.ld_add * 4) & 31) == 0;
        add_row = ep.addend ? ep.addend + (int64_t)row * ep.ld_add : nullptr;
        cs_row = ep.col_scale ? ep.col_scale + (int64_t)(row / ep.cs_rows) * ep.ld_cs : nullptr;
    }
};

// The row's scale: given, or from sums of squares (of the gated output per head, or of the residual stream per 64 channels), added in their order.
__device__ __forceinline__ float epi_row_scale(const EpiArgs &ep, int row) {
    if (ep.row_scale) return ep.row_scale[row];
    if (!ep.rs_ssq) return 1.f;
    const float *q = ep.rs_ssq + (int64_t)row * ep.rs_n;
    float s = 0.f;
    if ((ep.rs_n & 3) == 0) {
#pragma unroll 8
        for (int i = 0; i < ep.rs_n; i += 4) {
            const float4 v = __ldg(reinterpret_cast<const float4 *>(q + i));
            s += (v.x + v.y) + (v.z + v.w);
        }
    } else {
#pragma unroll 8
        for (int i = 0; i < ep.rs_n; ++i) s += __ldg(q + i);
    }
    return rsqrtf(s * ep.rs_inv + ep.rs_eps);
}

// v[j] = accumulator of column col + j, already times the row scale: bias, activation (ACT: they may occur), column scale.
template <bool ACT>
__device__ __forceinline__ void epi_pre(const EpiArgs &ep, const EpiRow &er, int col, float (&v)[32]) {
    const bool full = col + 32 <= ep.N;
    if constexpr (ACT) {
        if (ep.col_bias) {
            if (full) {
#pragma unroll
                for (int j = 0; j < 32; j += 4) {
                    const float4 b4 = *reinterpret_cast<const float4 *>(ep.col_bias + col + j);
                    v[j] += b4.x; v[j + 1] += b4.y; v[j + 2] += b4.z; v[j + 3] += b4.w;
                }
            } else {
#pragma unroll
                for (int j = 0; j < 32; ++j) if (col + j < ep.N) v[j] += ep.col_bias[col + j];
            }
        }
        if (col < ep.silu_cols) {                  // gate columns: SiLU here, where the ALUs idle, not in the scan
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if (col + j < ep.silu_cols) { const float hv = 0.5f * v[j]; v[j] = fmaf(hv, tanh_fast(hv), hv); }   // SiLU(v) = v/2 + v/2 tanh(v/2)
        }
        if (ep.gelu) {
#pragma unroll
            for (int j = 0; j < 32; ++j) {                  // GELU, tanh form
                const float x = v[j], hx = 0.5f * x;
                v[j] = fmaf(hx, tanh_fast(0.7978845608028654f * fmaf(0.044715f * x, x * x, x)), hx);
            }
        }
    }
    if (er.cs_row) {
        const float *cs = er.cs_row + col;
        if (full) {
#pragma unroll
            for (int j = 0; j < 32; j += 4) {
                const float4 c4 = *reinterpret_cast<const float4 *>(cs + j);
                v[j] *= c4.x; v[j + 1] *= c4.y; v[j + 2] *= c4.z; v[j + 3] *= c4.w;
            }
        } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) if (col + j < ep.N) v[j] *= cs[j];
        }
    }
}

// Addend and output by the thread itself, one row per lane.
__device__ __forceinline__ void epi_add_store(const EpiArgs &ep, const EpiRow &er, int row, int col, float (&v)[32]) {
    const bool full = col + 32 <= ep.N;
    if (er.add_row) {
        if (full && er.wide_add) {
#pragma unroll
            for (int j = 0; j < 32; j += 8) {
                uint32_t a8[8];
                ld_global_256(er.add_row + col + j, a8);
#pragma unroll
                for (int e = 0; e < 8; ++e) v[j + e] += __uint_as_float(a8[e]);
            }
        } else if (full && (ep.ld_add & 3) == 0) {
#pragma unroll
            for (int j = 0; j < 32; j += 4) {
                const float4 a4 = *reinterpret_cast<const float4 *>(er.add_row + col + j);
                v[j] += a4.x; v[j + 1] += a4.y; v[j + 2] += a4.z; v[j + 3] += a4.w;
            }
        } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) if (col + j < ep.N) v[j] += er.add_row[col + j];
        }
    }
    if (ep.c_is_f32) {
        float *crow = static_cast<float *>(ep.C) + (int64_t)row * ep.ldc + col;
        if (full && er.wide_c) {
#pragma unroll
            for (int j = 0; j < 32; j += 8) {
                uint32_t o[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) o[e] = __float_as_uint(v[j + e]);
                st_global_256(crow + j, o);
            }
        } else if (full && (ep.ldc & 3) == 0) {
#pragma unroll
            for (int j = 0; j < 32; j += 4) *reinterpret_cast<float4 *>(crow + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
        } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) if (col + j < ep.N) crow[j] = v[j];
        }
    } else {
        __nv_bfloat16 *crow = static_cast<__nv_bfloat16 *>(ep.C) + (int64_t)row * ep.ldc + col;
        if (full && er.wide_c) {
#pragma unroll
            for (int j = 0; j < 32; j += 16) {
                uint32_t o[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) o[e] = pack_bf16(v[j + 2 * e], v[j + 2 * e + 1]);
                st_global_256(crow + j, o);
            }
        } else if (full && (ep.ldc & 7) == 0) {
#pragma unroll
            for (int j = 0; j < 32; j += 8)
                *reinterpret_cast<uint4 *>(crow + j) = make_uint4(pack_bf16(v[j], v[j + 1]), pack_bf16(v[j + 2], v[j + 3]),
                                                                 pack_bf16(v[j + 4], v[j + 5]), pack_bf16(v[j + 6], v[j + 7]));
        } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) if (col + j < ep.N) crow[j] = __float2bfloat16_rn(v[j]);
        }
    }
}

constexpr uint32_t STG_BYTES = 32 * 128;     // staging of one epilogue warp
// Tensor maps of the outputs (boxes of 32 rows x 128 bytes; 64 of a bf16 one stored in halves), the addend and the next norm's input (64 bytes).
struct IoMaps { CUtensorMap c[2], add, u; };

// How one epilogue warp's 32 rows reach memory: 32 rows x 128 bytes at a time through 4 KB of shared memory and TMA.
// Staging: 16-byte piece j of row `lane` sits at lane * 128 + ((j ^ (lane & 7)) << 4), the 128-byte swizzle of the maps.
struct EpiOut {
    uint8_t *stg;
    int lane;
    uint64_t *add_bar;
    volatile int *abort_flag;
    int *status;
    uint32_t add_count;
    __device__ __forceinline__ uint4 *piece(int j) const { return reinterpret_cast<uint4 *>(stg + lane * 128 + ((j ^ (lane & 7)) << 4)); }
    __device__ __forceinline__ uint4 *half_piece(int j) const { return reinterpret_cast<uint4 *>(stg + lane * 64 + ((j ^ ((lane >> 1) & 3)) << 4)); }     // of 32 rows x 64 bytes, the 64-byte swizzle
    __device__ __forceinline__ void free() const {             // the previous store has read the staging bytes
        if (lane == 0) bulk_wait_read0();
        __syncwarp();
    }
    __device__ __forceinline__ void store(const CUtensorMap &map, int x, int y) const {
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) { tma_store_2d(&map, stg, x, y); bulk_commit(); }
    }
    __device__ __forceinline__ void add_fetch(const CUtensorMap &map, int x, int y) const {      // 32 rows x 32 columns of the addend on their way into the staging bytes
        free();
        if (lane == 0) { mbar_expect_tx(add_bar, STG_BYTES); tma_load_2d(stg, &map, x, y, add_bar); }
    }
    __device__ __forceinline__ bool add_take(float *v) {       // v[0..32) += this lane's row
        const bool r = __all_sync(0xffffffffu, mbar_wait(add_bar, add_count++ & 1u, abort_flag, status));
        if (r) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const uint4 a4 = *piece(j);
                v[4 * j] += __uint_as_float(a4.x); v[4 * j + 1] += __uint_as_float(a4.y); v[4 * j + 2] += __uint_as_float(a4.z); v[4 * j + 3] += __uint_as_float(a4.w);
            }
        }
        __syncwarp();
        return r;
    }
    // One 32-column group of results (columns n0 + c0 .., n0 a multiple of 64): to the output, and to the next norm's input where that is asked for.  ss: the row's sum of
    // squares over the current 64 columns.  HALF: a bf16 output 32 columns at a time, because an addend's next columns are fetched into the staging bytes in between.
    template <bool HALF>
    __device__ __forceinline__ void emit(const EpiArgs &pe, const CUtensorMap &map_c, const CUtensorMap &map_u, int n0, int c0, int row0, int row, bool row_ok, const float *v, float &ss) const {
        const int col = n0 + c0;
        if (pe.c_is_f32) {
            free();
#pragma unroll
            for (int j = 0; j < 8; ++j) *piece(j) = make_uint4(__float_as_uint(v[4 * j]), __float_as_uint(v[4 * j + 1]), __float_as_uint(v[4 * j + 2]), __float_as_uint(v[4 * j + 3]));
            store(map_c, col, row0);
        } else if (HALF) {
            free();
#pragma unroll
            for (int j = 0; j < 4; ++j)
                *half_piece(j) = make_uint4(pack_bf16(v[8 * j], v[8 * j + 1]), pack_bf16(v[8 * j + 2], v[8 * j + 3]), pack_bf16(v[8 * j + 4], v[8 * j + 5]), pack_bf16(v[8 * j + 6], v[8 * j + 7]));
            store(map_c, col, row0);
        } else {
            if (!(c0 & 32)) free();
#pragma unroll
            for (int j = 0; j < 4; ++j)
                *piece((c0 & 32) / 8 + j) = make_uint4(pack_bf16(v[8 * j], v[8 * j + 1]), pack_bf16(v[8 * j + 2], v[8 * j + 3]),
                                                      pack_bf16(v[8 * j + 4], v[8 * j + 5]), pack_bf16(v[8 * j + 6], v[8 * j + 7]));
            if ((c0 & 32) || col + 32 >= pe.N) store(map_c, n0 + (c0 & ~63), row0);
        }
        if (pe.u) {
            free();
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const bool in = col + 8 * j < pe.N;            // N is a multiple of 8
                const uint4 w4 = in ? __ldg(reinterpret_cast<const uint4 *>(pe.u_w + col + 8 * j)) : make_uint4(0u, 0u, 0u, 0u);
                const float *x = v + 8 * j;
                *half_piece(j) =
                    make_uint4(pack_bf16(x[0] * bf16_lo(w4.x), x[1] * bf16_hi(w4.x)), pack_bf16(x[2] * bf16_lo(w4.y), x[3] * bf16_hi(w4.y)),
                               pack_bf16(x[4] * bf16_lo(w4.z), x[5] * bf16_hi(w4.z)), pack_bf16(x[6] * bf16_lo(w4.w), x[7] * bf16_hi(w4.w)));
                if (in) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) ss = fmaf(x[e], x[e], ss);
                }
            }
            store(map_u, col, row0);
            if ((c0 & 32) || col + 32 >= pe.N) {
                if (row_ok) pe.u_ssq[(int64_t)row * ((pe.N + 63) / 64) + col / 64] = ss;
                ss = 0.f;
            }
        }
    }
};

// 2-D bf16 tensor [rows, cols] with row pitch ld elements; box = [box_rows, 64 columns], 128-byte swizzle.
inline bool make_map_2d(CUtensorMap *m, const void *base, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
    const uint64_t dims[2] = {(uint64_t)cols, (uint64_t)rows};
    const uint64_t strides[1] = {(uint64_t)ld};
    const uint32_t box[2] = {64, (uint32_t)box_rows};
    return make_map_bf16(m, base, 2, dims, strides, box);
}

// bf16 tensor in boxes of 32 rows x 32 columns, 64-byte swizzle: the next norm's input, a bf16 output with an addend.
inline bool make_map_half(CUtensorMap *m, const void *base, int64_t rows, int64_t cols, int64_t ld) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t d[2] = {(cuuint64_t)cols, (cuuint64_t)rows}, st[1] = {(cuuint64_t)ld * 2};
    const cuuint32_t b[2] = {32, 32}, e[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), d, st, b, e, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The output as EpiOut::emit<half> stores it
inline bool make_map_out(CUtensorMap *m, const EpiArgs &p, bool half) {
    if (p.c_is_f32) return make_map_f32_2d(m, p.C, p.M, p.N, p.ldc, 32);
    return half ? make_map_half(m, p.C, p.M, p.N, p.ldc) : make_map_2d(m, p.C, p.M, p.N, p.ldc, 32);
}

}  // namespace tc

// gemm_pair.cu: the two-CTA kernel.  wide: 256 x 256 tiles, else 256 x 128; b: a second product of the same sizes.  gemm_pair_sum_launch: both products into one output.
int gemm_pair_cost(bool wide, const GemmArgs &a, int nprob);      // of the launch's rounds, for the choice of the tile
cudaError_t gemm_pair_launch(bool wide, const GemmArgs &a, const GemmArgs *b, cudaStream_t s);
cudaError_t gemm_pair_sum_launch(const GemmArgs &a, const GemmArgs &b, cudaStream_t s);
// gemm_cluster.cu: the same with each tile's K spread over a cluster, for few tiles.
bool gemm_cluster_sum_pays(const GemmArgs &a);
cudaError_t gemm_cluster_sum_launch(const GemmArgs &a, const GemmArgs &b, cudaStream_t s);
// gemm_rows.cu: up to 128 rows; sum as in gemm_pair_sum_launch.
cudaError_t gemm_rows_launch(const GemmArgs &a, const GemmArgs *b, bool sum, cudaStream_t s);

}  // namespace dm
