// Weight-streaming skinny GEMM on the 5th-generation tensor cores (tcgen05 + TMEM), operands fed
// by TMA.  out[r, n] = sum_k A[r, k] * W[n, k]: the weight rows sit on the MMA's M side (up to 128 per
// tile), the token rows on its N side (padded to 16..256), so every weight byte is read from HBM
// exactly once per pass whatever the row count.
#pragma once
#include <cuda.h>
#include "common.cuh"
#include "forward.cuh"

namespace hsd {

constexpr int kTcBlockM = 128;     // weight rows per tile
constexpr int kTcBlockK = 64;      // bf16 per k-block (one 128-byte swizzle row)
constexpr int kTcBoxRows = 64;     // weight rows per TMA box

// Encoders obtained from the driver at run time (no link-time dependency on libcuda).
int tc_init();                     // HSD_OK when the tensor-map encoder is available
// 2-D bf16 tensor map over a row-major [rows, cols] matrix, box = [box_rows, 64], 128-byte swizzle.
int tc_make_map(CUtensorMap *map, const void *base, long long rows, long long cols, int box_rows);

int tc_npad(int rows);             // 16, 32, 64, 128 or 256 (rows <= 256)

// Where the q / k / v projection's rows go (GEMM_QKV_T): q rotated -> q; k rotated, v -> their cache pages.
struct TcQkv {
  const int *row_seq, *row_pos, *page_table;
  const float *cos_tab, *sin_tab;
  __nv_bfloat16 *q, *k_pool, *v_pool;
  int nq, hd, page, pages_per_seq, n_pages;
};
struct TcGemmArgs {
  CUtensorMap w[3];                // weight maps
  CUtensorMap a;                   // activation map, covers the whole buffer
  int tile_rows = kTcBlockM, w_box_rows = kTcBoxRows;   // weight rows of a tile (<= 128; SWIGLU: 64 gate + 64 up) and of one box of their maps
  int a_box_rows;                  // rows of one box of the activation map (R .. row padding)
  bool chained = false;            // part of a chain of kernels (common.cuh)
  bool early_weights = false;      // in a chain: the first weights are asked for before the kernel before is over (which must not write them)
  int stream_weights = 0;          // 1: the weights will not be read again soon (evict-first in L2)
  int reset_status = 0;            // 1: the kernel clears the status word first
  TcQkv qkv;
  int seg_n[3], n_segs;
  int K, R, row0;                  // R rows of A starting at buffer row row0
  int mode;                        // GemmMode
  float *out_f32;                  // STORE_F32 / ADD_F32: [.., ldo], written at rows row0..row0+R-1
  __nv_bfloat16 *out_bf16;         // STORE_T_SCATTER: [dst[row], ldo];  SWIGLU_T: [row, ldo]
  const long long *dst;
  int ldo;
  int *status;                     // device word: set non-zero if a bounded wait gave up
};
int tc_tile_rows(int N, int K, int R, int sm_count);
int launch_gemm_tc(const TcGemmArgs &args, int sm_count, cudaStream_t s);

}  // namespace hsd
