// Internal interface of the projection GEMMs (gemm.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"
#include "dash.h"

namespace dash {

enum GemmEpilogueKind { GEMM_PLAIN = 0, GEMM_ROPE = 1, GEMM_RESID = 2, GEMM_SWIGLU = 3 };

struct GemmEpilogue {
    // ROPE: heads of D columns; columns below n_rot_cols (a multiple of 256) belong to Q and K heads and are rotated with
    // rope_table [n, D/2] = (cos, sin) of every row
    int D = 0, n_rot_cols = 0;
    const float2* rope_table = nullptr;
    // rope_pos null: the table holds one entry per row; else one per position and row t uses entry min(rope_pos[t], rope_len - 1)
    const int32_t* rope_pos = nullptr; int64_t rope_len = 0;
    // ROPE: k_cache / v_cache (null: none): the K and V heads' columns (behind q_cols of Q) once more, rows of ld_cache elements, 8-byte aligned
    // fp32 C: the bf16 copies of the heads, q_copy [n, q_cols] and k_cache / v_cache
    int q_cols = 0;
    void *k_cache = nullptr, *v_cache = nullptr, *q_copy = nullptr; int64_t ld_cache = 0;
    // ROPE, SWIGLU: row_scale (null: none) multiplies the accumulators of a row first -- 1 / rms(row) when the RMSNorm in front of the
    // projection is folded into it (its weight into W, its row factor here)
    const float* row_scale = nullptr;
    // RESID: x_full[tok_index[row]] (tok_index null: row) = H[row] + (A W)[row]; sums [n, N/128] = (sum u^2, sum h^2, sum (h+u)^2, 0)
    // per 128 columns
    const void* H = nullptr; int64_t ldh = 0;
    const int32_t* tok_index = nullptr;
    void* x_full = nullptr; int64_t ldx = 0;
    float4* sums = nullptr;
    // SWIGLU: W = [K, 2m] (gate | up); C [n, m] = silu(A Wg) * (A Wu)
    int m = 0;
};

// Scratch of one GEMM at a time on one stream: part 16-byte aligned, gemm_split_part_bytes() of the GEMM (0: it runs in whole tiles); arrived
// gemm_split_count_bytes(), zero before the first GEMM that uses it (every GEMM leaves it zero again, but for a tile whose parts it waited for in
// vain: DASH_ERR_TIMEOUT); spin_limit: polls of that wait.
struct GemmSplit { float* part = nullptr; unsigned int* arrived = nullptr; uint32_t spin_limit = kSpinLimit; };
size_t gemm_split_part_bytes(int64_t n, int64_t N, int64_t K);
size_t gemm_split_count_bytes();
// The scratch depends on n only through the number of rows of tiles, ceil(n / gemm_tile_rows()), and is 0 above gemm_split_max_rows()
int gemm_tile_rows();
int64_t gemm_split_max_rows();

// true if the kernel takes this problem with this epilogue.  PLAIN: any N % 4 == 0, K % 8 == 0 (rows on 16-byte boundaries); the
// fused epilogues: whole 256-column tiles (SWIGLU: m % 128 == 0) and K in steps of 64 -- otherwise the caller runs the projection
// PLAIN and the element-wise work as passes of their own.
bool gemm_shape_ok(GemmEpilogueKind kind, int64_t n, int64_t N, int64_t K, int64_t lda, int64_t ldw, const GemmEpilogue& e);
// C (or the epilogue's outputs) = A[n, K] W[K, N], A and W bf16; ld* in elements; n_dev: device true row count or null;
// out_f32 (PLAIN, ROPE): C is fp32 instead of bf16; sc: scratch that lets the kernel cut tiles along K (null: whole tiles only);
// w_early: W may be read while the kernel in front of this one still runs.  Only for a W that no kernel of the step writes (a caller's weights),
// behind a kernel of the step that has called pdl_wait() ahead of pdl_launch_dependents() (prologue_kernel): what made W is then
// complete before anything of the step that is launched to start early can start.
int gemm_bf16(GemmEpilogueKind kind, const void* A, int64_t lda, const void* W, int64_t ldw, void* C, int64_t ldc, int64_t n, int64_t N,
              int64_t K, const GemmEpilogue& e, const int32_t* n_dev, cudaStream_t st, bool out_f32 = false, const GemmSplit* sc = nullptr,
              bool w_early = false);
// dst (bf16, row stride ld_dst) = src (fp32, row stride ld_src) rounded to nearest even; cols % 4 == 0
int launch_f32_to_bf16(const float* src, int64_t ld_src, void* dst, int64_t ld_dst, int64_t rows, int64_t cols, cudaStream_t st);
// (cos, sin) of pos * base^(-2i/D) for the positions 0 .. n - 1 into table [n, D/2]
int launch_rope_table(int64_t n, int D, double rope_base, float2* table, cudaStream_t st);

}  // namespace dash
