// One-launch verifier forward of small fp32 models.
#pragma once
#include "common.cuh"
#include "forward.cuh"

namespace hsd {

struct SmallLayerDev { const float *w[9]; float *k_pool, *v_pool; };   // attn_norm wq wk wv wo mlp_norm wg wu wd; this layer's pools

struct SmallFwdArgs {
  int d, nq, nkv, hd, ff, V, n_run, max_seq, page, pages_per_seq, n_pages;
  float eps;
  const SmallLayerDev *layers;       // global memory [n_layers]
  const float *embed, *final_norm, *lm_head, *cos_tab, *sin_tab;
  int R, L;                          // <= kSmallRows
  const int *tokens, *page_table;
  PassRows rows;
  float *x, *q, *att, *act, *logits;
  unsigned *counter;                 // counts barrier arrivals, never reset: `base` = its value when the launch starts
  unsigned base;
  int *status;                       // set non-zero when a bounded wait gave up
};

constexpr int kSmallRows = 128;          // rows of one launch; longer passes are several, in row order
bool fwd_small_supported(const ModelDims &md);
int fwd_small_grid(const ModelDims &md, int sm_count);
// Barrier arrivals of one launch (added to the counter).
inline unsigned fwd_small_arrivals(int n_run, int L, int grid) { return (unsigned)((5 * n_run - (L > 0 ? 0 : 1)) * grid); }
int launch_forward_small(const SmallFwdArgs &args, int grid, cudaStream_t s);

}  // namespace hsd
