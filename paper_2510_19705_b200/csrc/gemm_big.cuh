// Matrix products of passes with many token rows (prompt chunks): out[r, n] = sum_k A[r, k] W[n, k] with bf16
// inputs and fp32 accumulation, bound by the tensor cores instead of by the weight stream.
#pragma once
#include <cuda.h>
#include "common.cuh"
#include "forward.cuh"

namespace hsd {

enum BigGemmMode {
  BIG_QKV = 0,        // q rotated -> q; k rotated, v -> their cache pages (bf16)
  BIG_ADD_F32 = 1,    // out_f32[r, n] += acc (residual stream)
  BIG_SWIGLU = 2,     // out_bf16[r, n] = silu(gate) * up
  BIG_LOGITS = 3      // out_bf16[dst[r] or r, n]
};

struct BigGemmArgs {
  CUtensorMap a;                       // activations, box 128 rows x 64 columns, 128-byte swizzle
  CUtensorMap w[3];                    // weights, box 64 rows x 64 columns
  int mode, R, K;
  int seg_n[3];                        // QKV: q, k, v columns (multiples of 128); others: seg_n[0] (SWIGLU: ff)
  int skip_cols;                       // QKV: columns [0, skip_cols) are not needed (a multiple of 256)
  float *out_f32;
  __nv_bfloat16 *out_bf16;
  int ldo;
  const long long *dst;                // LOGITS: destination rows, or null
  // QKV
  const int *row_seq, *row_pos, *page_table;
  const float *cos_tab, *sin_tab;
  __nv_bfloat16 *q, *k_pool, *v_pool;
  int nq, nkv, hd, page, pages_per_seq, n_pages;
  int *status;                         // set non-zero if a bounded wait gave up
  bool chained;                        // part of a chain of kernels (common.cuh)
};

constexpr int kBigBoxRowsA = 128;
int launch_gemm_big(const BigGemmArgs &args, int sm_count, cudaStream_t s);

}  // namespace hsd
