// Causal attention of prompt chunks over the paged cache (bf16 models, head size 64 or 128).
#pragma once
#include <cuda.h>
#include "common.cuh"

namespace hsd {

struct PromptAttnArgs {
  CUtensorMap k, v;                  // one layer's pools as [nkv * n_pages * page, hd], box 64 rows x 64 columns, 128-byte swizzle
  const __nv_bfloat16 *q;            // [R, nq, hd]
  __nv_bfloat16 *att;                // [R, nq, hd]
  const int4 *items;                 // (first packed row, tokens <= 2 * prompt_attn_tokens, sequence, position of the first)
  int n_items;
  const int *page_table;
  int nq, nkv, hd, page_shift, pages_per_seq, n_pages;
  int *status;                       // set non-zero if a bounded wait gave up
  bool chained;                      // part of a chain of kernels (common.cuh)
};

// tokens of one 128-row query tile: the heads of a KV group sit side by side in it
inline int prompt_attn_tokens(int group) { return 128 / group; }
int prompt_attn_map(CUtensorMap *map, const void *pool, long long rows, int hd);
// A 64-key tile is one copy: the pages within it must follow one another in the pool.  (A prompt's do: prompts are read
// from a full free list in ascending order, a sequence's pages in one run.)
bool prompt_attn_pages(const int *pages, int n_pages, int page);
int launch_prompt_attention(const PromptAttnArgs &args, cudaStream_t s);

}  // namespace hsd
