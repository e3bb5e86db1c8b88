// The verification kernels as tests/test_gpu_verify_waits.py builds them: with a wait limit of a millisecond, beside a kernel that
// lets its successor start at once and then takes its time, and with statistics whose data never comes.
#include "../../paper_2510_19705_b200/csrc/sampling.cu"

__global__ void occupy_kernel(unsigned long long ns) {
  chain_next();
  const unsigned long long t0 = hsd::ptx::globaltimer_ns();
  for (int i = 0; i < (1 << 24) && hsd::ptx::globaltimer_ns() - t0 < ns; ++i) {}
}

extern "C" int occupy(unsigned long long ns, void *stream) {
  occupy_kernel<<<1, 32, 0, (cudaStream_t)stream>>>(ns);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// A verification (statistics at the front of `scratch`) whose statistics are computed by grids without their loader warps: the
// computing warps' waits run out, nothing is in flight.
template <typename T, int GROUPS, int WARPS> static int without_loaders(const hsd::RowStatArgs &r, int grid, cudaStream_t s) {
  const auto kernel = hsd::row_stats_kernel<T, GROUPS, WARPS>;
  const int smem = (int)hsd::kRsBytes + 128;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return -1;
  kernel<<<grid, 32 * GROUPS * WARPS, smem, s>>>(r);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}
extern "C" int verify_without_data(const void *p, const void *q, int32_t *tokens, int batch, int t, int vocab, int dtype, int groups, void *scratch,
                                   void *stream, int32_t *out_tokens, int32_t *out_n, int32_t *host_n, int32_t *host_token) {
  hsd::RowStatArgs r = {};
  r.p = p; r.q = q; r.V = vocab; r.t_max = r.regular_t = t; r.batch = batch; r.stats = (hsd::RowStat *)scratch;
  hsd::ClusterArgs a = {};
  a.p = p; a.q = q; a.tokens = tokens; a.V = vocab; a.t_max = a.regular_t = t; a.regular_level = 1; a.seed = 7; a.out_tokens = out_tokens;
  a.out_n = out_n; a.coin24 = hsd::kNoCoin; a.mirror.n = host_n; a.mirror.token = host_token;
  const int rows = batch * (2 * t + 1), grid = rows < 148 ? rows : 148;
  cudaStream_t s = (cudaStream_t)stream;
  const int st = dtype == HSD_F32 ? (groups == 1 ? without_loaders<float, 1, 16>(r, grid, s) : without_loaders<float, 3, 8>(r, grid, s))
                                  : (groups == 1 ? without_loaders<__nv_bfloat16, 1, 16>(r, grid, s) : without_loaders<__nv_bfloat16, 3, 8>(r, grid, s));
  return st ? st : hsd::launch_decisions(a, dtype, batch, r.stats, true, s);
}
