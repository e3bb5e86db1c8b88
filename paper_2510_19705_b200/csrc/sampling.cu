// Sampling kernels of the HSD hot path: level-0 draft sampling (Algorithm 1, base case) and the
// fused softmax-statistics / acceptance / residual-resample step (Algorithm 2; rule of Section 2).
#include "sampling.cuh"
#include "sampling_api.cuh"
#include "tc_ptx.cuh"
#include <algorithm>
#include <atomic>

namespace hsd {

// A call's descriptors: n_inline of them here, or all at `desc`, or (both zero) worked out from the regular layout.
template <typename D> struct DescList {
  const D *desc;
  int n_inline;
  D inl[kInlineDesc];
  __device__ __forceinline__ bool given() const { return n_inline > 0 || desc; }
  __device__ __forceinline__ D at(int i) const { return n_inline > 0 ? inl[i] : desc[i]; }
};
template <typename D> static DescList<D> desc_list(const D *desc, int n, bool on_host) {
  DescList<D> l;
  l.desc = on_host ? nullptr : desc;
  l.n_inline = on_host ? n : 0;
  for (int i = 0; i < l.n_inline; ++i) l.inl[i] = desc[i];
  return l;
}

// ------------------------------------------------------------------------------ draft sampling
// One block per row: token = inverse-CDF sample of softmax(row) with the purpose-0 uniform.  The kernel behind it does not start
// early: its CTAs would take the places that this one's last round frees, two on some SMs and none on others.  200 / 297 / 2000
// fp32 rows of 128256 tokens in a row of calls: 81 / 144 / 744 us; with early starts 115 / 174 / 835, half of that because the
// descriptor was kept in registers through the row.
template <typename T>
__global__ void __launch_bounds__(kSampleThreads)
draft_sample_kernel(const T *__restrict__ logits, int V, const __grid_constant__ DescList<SampleRow> desc,
                    int regular_rows, u32 regular_serial, u64 seed, int32_t *__restrict__ out, const HostMirror mirror) {
  __shared__ float shf[32];
  __shared__ u64 sh64[34];
  chain_wait();
  auto descriptor = [&]() {
    SampleRow d;
    if (desc.given()) return desc.at(blockIdx.x);
    d.logit_row = blockIdx.x;
    d.out_index = blockIdx.x;
    d.j = blockIdx.x % regular_rows;
    d.seq = blockIdx.x / regular_rows;
    d.serial = regular_serial;
    d.level = 0;
    return d;
  };
  const T *row;
  u32 U;
  {
    const SampleRow d = descriptor();
    row = logits + (size_t)d.logit_row * V;
    U = uniform24(seed, d.j, d.serial, d.level, PURPOSE_DRAFT, d.seq);
  }
  int tok;
  if (sizeof(T) == 2 && chunk_layout_ok(row, V, blockDim.x)) {
    const int k0 = threadIdx.x * kChunkTokens;
    const Chunk32 c = chunk_load(reinterpret_cast<const __nv_bfloat16 *>(row), V, k0);
    const float m = block_max(chunk_max(c, V, k0), shf);
    tok = block_inverse_cdf_chunk(V, k0, U, [&](int i) { return (u64)exp_weight(chunk_get(c, i), m); }, sh64, nullptr);
  } else {
    float m = row_max(row, V, shf);
    tok = block_inverse_cdf(V, U, [&](int k) { return (u64)exp_weight(to_f32(row[k]), m); }, sh64, nullptr);
  }
  if (threadIdx.x == 0) {
    const SampleRow d = descriptor();
    out[d.out_index] = tok;
    if (mirror.token) mirror.token[(size_t)d.seq * mirror.stride + d.j] = tok;
  }
}

// 16 bytes of a row
template <typename T> struct StatVec;
template <> struct StatVec<__nv_bfloat16> {
  static constexpr int N = 8;
  __device__ static void unpack(const uint4 &v, float *f) {
    f[0] = __uint_as_float(v.x << 16); f[1] = __uint_as_float(v.x & 0xFFFF0000u);
    f[2] = __uint_as_float(v.y << 16); f[3] = __uint_as_float(v.y & 0xFFFF0000u);
    f[4] = __uint_as_float(v.z << 16); f[5] = __uint_as_float(v.z & 0xFFFF0000u);
    f[6] = __uint_as_float(v.w << 16); f[7] = __uint_as_float(v.w & 0xFFFF0000u);
  }
};
template <> struct StatVec<float> {
  static constexpr int N = 4;
  __device__ static void unpack(const uint4 &v, float *f) {
    f[0] = __uint_as_float(v.x); f[1] = __uint_as_float(v.y); f[2] = __uint_as_float(v.z); f[3] = __uint_as_float(v.w);
  }
};

// ------------------------------------------------------------------------------ decision by a CTA: vocabularies past 131072 tokens, many sequences
// One block per sequence: accept tests for all positions (each with its own counter-addressed
// uniform, so the parallel form equals Algorithm 2's sequential loop with break), n = index of the
// first rejection, then the final draw from the residual of row n (n < t) or from target row t.
// Launched in the ordinary way: started early, beside the streaming statistics' shared memory, it would have no first-level cache to
// read its rows through (16 sequences of 8 drafts, 151936 tokens: 336 us instead of 136).
template <typename T, int CTAS>
__global__ void __launch_bounds__(kSampleThreads, CTAS)
decide_kernel(const T *__restrict__ p_logits, const T *__restrict__ q_logits, int32_t *__restrict__ tokens, int V,
              int t_max, const __grid_constant__ DescList<VerifySeq> desc, int regular_t, u32 regular_serial, u32 regular_level,
              const RowStat *__restrict__ stats, u64 seed, int32_t *__restrict__ out_tokens /*[B, t_max+1] or null*/,
              int32_t *__restrict__ out_n /*[B]*/, int write_in_place, u32 coin24, const HostMirror mirror) {
  __shared__ u64 sh64[34];
  __shared__ int sh_first_reject, sh_none;
  int b = blockIdx.x;
  VerifySeq d;
  if (desc.given()) d = desc.at(b);
  else {
    d.t = regular_t; d.p_row0 = (long long)b * (regular_t + 1); d.q_row0 = (long long)b * regular_t;
    d.tok_off = (long long)b * regular_t; d.serial = regular_serial; d.seq = b; d.level = regular_level;
  }
  const RowStat *st = stats + (size_t)b * (2 * t_max + 1);
  if (threadIdx.x == 0) { sh_first_reject = d.t; sh_none = 0; }
  __syncthreads();
  if ((int)threadIdx.x < d.t) {
    int j = threadIdx.x;
    RowStat sp = st[j], sq = st[t_max + 1 + j];
    if (sp.S == kNoStat || sq.S == kNoStat) sh_none = 1;
    const int tok = tokens[d.tok_off + j];
    const bool in = tok >= 0 && tok < V;
    u64 Pp = fixed_prob(in ? exp_weight(to_f32(p_logits[(size_t)(d.p_row0 + j) * V + tok]), sp.m) : 0u, prob_scale(sp.S));
    u64 Pq = fixed_prob(in ? exp_weight(to_f32(q_logits[(size_t)(d.q_row0 + j) * V + tok]), sq.m) : 0u, prob_scale(sq.S));
    u32 U = uniform24(seed, j, d.serial, d.level, PURPOSE_ACCEPT, d.seq);
    bool ok = (((u64)U * Pq) >> 24) < Pp;                 // u < p(x) / q(x)
    if (coin24 != kNoCoin) ok = U < coin24;               // ablation: IID acceptance with a fixed probability
    if (!ok) atomicMin(&sh_first_reject, j);
  }
  __syncthreads();
  int n = sh_first_reject;
  const bool none = sh_none || st[n].S == kNoStat;             // (what the marks give stays within the row and the buffers)
  u32 U = uniform24(seed, 0, d.serial, d.level, PURPOSE_FINAL, d.seq);
  const T *prow = p_logits + (size_t)(d.p_row0 + n) * V;
  float mp = st[n].m;
  int m_tok = -1;
  if (n < d.t) {
    const T *qrow = q_logits + (size_t)(d.q_row0 + n) * V;
    float mq = st[t_max + 1 + n].m;
    ProbScale psp = prob_scale(st[n].S), psq = prob_scale(st[t_max + 1 + n].S);
    m_tok = block_inverse_cdf(V, U, [&](int k) {
      u64 Pp = fixed_prob(exp_weight(to_f32(prow[k]), mp), psp);
      u64 Pq = fixed_prob(exp_weight(to_f32(qrow[k]), mq), psq);
      return Pp > Pq ? Pp - Pq : 0ull;
    }, sh64, nullptr);
  }
  if (m_tok < 0)   // bonus token, or an all-zero residual: draw from the verifier's own row
    m_tok = block_inverse_cdf(V, U, [&](int k) { return (u64)exp_weight(to_f32(prow[k]), mp); }, sh64, nullptr);
  if (none) m_tok = -1;
  const int n_out = none ? kNoDecision : n;
  if (threadIdx.x == 0) {
    out_n[b] = n_out;
    if (write_in_place) tokens[d.tok_off + n] = m_tok;
    if (mirror.n) { mirror.n[b] = n_out; mirror.token[b] = m_tok; }
    if (mirror.status && b == 0) *mirror.status = __ldcg(mirror.status_src);
  }
  if (out_tokens) {
    for (int j = threadIdx.x; j <= t_max; j += blockDim.x) {
      int v = -1;
      if (j < n_out) v = tokens[d.tok_off + j];
      else if (j == n) v = m_tok;
      out_tokens[(size_t)b * (t_max + 1) + j] = v;
    }
  }
}

// ------------------------------------------------------------------------------ statistics of many rows
// (maximum, integer total) of every row of a verification, rows dealt to a persistent grid of one CTA per SM.  Bound by
// fp32 issue: the unfused exponential is 15 packed multiplies and adds a pair of logits, 14.1 cycles a warp and logit per
// scheduler however it is written (microbenchmark), 1.85 us for 32000 logits on an SM; 64 KB from HBM take 1.4 us.  A warp
// of its own brings the rows into a ring of 32 KB chunks; with a row's first chunk it publishes where the statistics go and
// the elements in front of and behind the row's 16-byte vectors, so that rows may begin on any element.  GROUPS groups of
// WARPS warps take the CTA's rows in turn, each with its own barrier, so that one's reductions and waits (0.7 us a row, as
// much as a row of 2048 logits has of arithmetic) run under the others' exponentials.  A row stays in the ring between its
// maximum and its sum; rows of more chunks than the ring has come through it twice.
constexpr uint32_t kRsPiece = 2048;                        // bytes; a chunk is asked for by its first lanes (a single large copy runs at a fraction of an SM's bandwidth)
constexpr uint32_t kRsChunk = 32768;
constexpr int kRsRing = 7, kRsChunkVecs = kRsChunk / 16;
constexpr uint32_t kRsBytes = kRsRing * kRsChunk;          // of the ring
static_assert(kRsChunk <= 32 * kRsPiece);
constexpr int kRsMaxEdge = 16;

struct RowStatArgs {
  const void *p, *q;
  int V, t_max, batch, regular_t;
  DescList<VerifySeq> desc;
  RowStat *stats;
};
struct RsInfo {
  int stat;                                                // index of the row's statistics, -1: no more rows
  int n_vec, n_edge;
  float edge[kRsMaxEdge];
};

__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
template <typename T> __device__ __forceinline__ uint4 rs_pad();                 // a vector of -inf: weight 0, never the maximum of a row
template <> __device__ __forceinline__ uint4 rs_pad<float>() { return make_uint4(0xFF800000u, 0xFF800000u, 0xFF800000u, 0xFF800000u); }
template <> __device__ __forceinline__ uint4 rs_pad<__nv_bfloat16>() { return make_uint4(0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u); }
// maximum of the vectors' elements so far (bf16: of packed pairs, which is exact)
template <typename T> struct RsMax;
template <> struct RsMax<float> {
  float m = -INFINITY;
  __device__ void take(const uint4 &v) {
    m = fmaxf(fmaxf(fmaxf(m, __uint_as_float(v.x)), __uint_as_float(v.y)), fmaxf(__uint_as_float(v.z), __uint_as_float(v.w)));
  }
  __device__ float get() const { return m; }
};
template <> struct RsMax<__nv_bfloat16> {
  __nv_bfloat162 m = __floats2bfloat162_rn(-INFINITY, -INFINITY);
  __device__ void take(const uint4 &v) {
    const __nv_bfloat162 a = __hmax2(*reinterpret_cast<const __nv_bfloat162 *>(&v.x), *reinterpret_cast<const __nv_bfloat162 *>(&v.y));
    const __nv_bfloat162 b = __hmax2(*reinterpret_cast<const __nv_bfloat162 *>(&v.z), *reinterpret_cast<const __nv_bfloat162 *>(&v.w));
    m = __hmax2(m, __hmax2(a, b));
  }
  __device__ float get() const { return fmaxf(__low2float(m), __high2float(m)); }
};

// A warp's wait gave up: the mark on every row of its CTA (one that gets its statistics all the same may keep either).
__device__ __noinline__ void give_up(RowStat *stats, long long n_items) {
  RowStat st;
  st.m = 0.f; st.S = kNoStat;
  for (long long i = blockIdx.x + (long long)(threadIdx.x & 31) * gridDim.x; i < n_items; i += 32ll * gridDim.x) stats[i] = st;
}

template <typename T, int GROUPS, int WARPS>
__global__ void __launch_bounds__(32 * (GROUPS * WARPS + 1), 1) row_stats_kernel(const __grid_constant__ RowStatArgs a) {
  extern __shared__ uint8_t rs_smem_raw[];
  uint8_t *ring = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(rs_smem_raw) + 127) & ~(uintptr_t)127);
  // full, per group | empty, per slot of the ring | a row's maxima, per group.  A parity wait tells a barrier's phases apart
  // only one phase back, so a barrier's phases all belong to one waiter, which waits for each: chunk y of a group completes
  // barrier y mod kRsRing of that group, and only the producer waits for "empty".
  __shared__ __align__(8) uint64_t bars[kRsRing * (GROUPS + 1) + GROUPS];
  __shared__ RsInfo infos[kRsRing];
  __shared__ int sh_max[GROUPS][2][WARPS];                 // order keys
  __shared__ u64 sh_sum[GROUPS][2][WARPS];
  __shared__ int sh_abort;
  constexpr int ES = (int)sizeof(T), VN = 16 / ES, THREADS = 32 * WARPS;
  const int lane = threadIdx.x & 31, warp = ptx::warp_index();
  const uint32_t full0 = ptx::smem_u32(bars), empty = full0 + 8u * kRsRing * GROUPS, ring0 = ptx::smem_u32(ring);
  if (threadIdx.x == 0) {
    for (int s = 0; s < kRsRing * GROUPS; ++s) ptx::mbar_init(full0 + 8u * s, 1);
    for (int s = 0; s < kRsRing + GROUPS; ++s) ptx::mbar_init(empty + 8u * s, WARPS);
    sh_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  volatile int *abort_flag = &sh_abort;
  // A row is n_chunks chunks (the last may be empty).  In the ring's order row k of the CTA begins at chunk k passes n_chunks.
  const int n_chunks = max(1, (int)(((long long)a.V * ES + kRsChunk - 1) / kRsChunk));
  const bool resident = n_chunks <= kRsRing;
  const int passes = resident ? 1 : 2;
  if (warp == GROUPS * WARPS) {
    // ---- the rows of this CTA, in order
    chain_wait();
    chain_next();
    const int rows_per_seq = 2 * a.t_max + 1, n_items = a.batch * rows_per_seq;
    uint32_t slot = 0, phase = 0;                          // of the next chunk
    auto advance = [&]() { if (++slot == kRsRing) { slot = 0; phase ^= 1u; } };
    uint32_t sent[GROUPS], group = 0;                      // chunks of each group so far (mod kRsRing); the next row's group
#pragma unroll
    for (int g = 0; g < GROUPS; ++g) sent[g] = 0;
    bool ok = true;
    for (int i = blockIdx.x; i < n_items && ok; i += gridDim.x) {
      const int b = i / rows_per_seq, r = i - b * rows_per_seq;
      const bool is_p = r <= a.t_max;
      const int at = is_p ? r : r - a.t_max - 1;
      long long row0;
      if (a.desc.given()) {
        const VerifySeq d = a.desc.at(b);
        if (at >= d.t + (is_p ? 1 : 0)) continue;
        row0 = is_p ? d.p_row0 : d.q_row0;
      } else row0 = (long long)b * (a.regular_t + (is_p ? 1 : 0));
      const T *row = reinterpret_cast<const T *>(is_p ? a.p : a.q) + (size_t)(row0 + at) * a.V;
      const uintptr_t lo = reinterpret_cast<uintptr_t>(row), hi = lo + (size_t)a.V * ES;
      const uintptr_t v0 = min((lo + 15) & ~(uintptr_t)15, hi), v1 = max(hi & ~(uintptr_t)15, v0);   // the whole vectors
      const size_t bytes = v1 - v0;
      const int head = (int)(v0 - lo) / ES, n_edge = head + (int)(hi - v1) / ES;
      uint32_t y = 0;
#pragma unroll
      for (int g = 0; g < GROUPS; ++g)
        if (g == (int)group) y = sent[g];
      for (int ps = 0; ps < passes && ok; ++ps)
        for (int c = 0; c < n_chunks; ++c, advance()) {
          ok = ptx::mbar_wait_warp(empty + 8u * slot, phase ^ 1u, abort_flag);
          if (!ok) break;
          if (c == 0) {
            if (lane == 0) { infos[slot].stat = i; infos[slot].n_vec = (int)(bytes / 16); infos[slot].n_edge = n_edge; }
            if (lane < n_edge) infos[slot].edge[lane] = to_f32(lane < head ? row[lane] : reinterpret_cast<const T *>(v1)[lane - head]);
            __syncwarp();
          }
          const size_t off = (size_t)c * kRsChunk;
          const uint32_t n = off < bytes ? (uint32_t)min((size_t)kRsChunk, bytes - off) : 0u, po = (uint32_t)lane * kRsPiece;
          const uint32_t full = full0 + 8u * (group * kRsRing + y);
          if (++y == kRsRing) y = 0;
          if (lane == 0) { if (n) ptx::mbar_expect_tx(full, n); else ptx::mbar_arrive(full); }
          __syncwarp();
          if (po < n) bulk_load(ring0 + slot * kRsChunk + po, reinterpret_cast<const void *>(v0 + off + po), min(kRsPiece, n - po), full);
        }
#pragma unroll
      for (int g = 0; g < GROUPS; ++g)
        if (g == (int)group) sent[g] = y;
      if (++group == GROUPS) group = 0;
    }
    for (int e = 0; e < GROUPS && ok; ++e) {               // "no more rows", to each group: a row without data, whose other chunks pass by
      uint32_t y = 0;
#pragma unroll
      for (int g = 0; g < GROUPS; ++g)
        if (g == (int)group) y = sent[g];
      for (int c = 0; c < passes * n_chunks; ++c, advance()) {
        ok = ptx::mbar_wait_warp(empty + 8u * slot, phase ^ 1u, abort_flag);
        if (!ok) break;
        if (c == 0 && lane == 0) { infos[slot].stat = -1; ptx::mbar_arrive(full0 + 8u * (group * kRsRing + y)); }
        if (c > 0 && lane < WARPS) ptx::mbar_arrive(empty + 8u * slot);
        __syncwarp();
      }
      if (++group == GROUPS) group = 0;
    }
    if (!ok) {
      // copies already asked for must land before the CTA's shared memory goes away (bounded: 20 us are far longer than one takes)
      const unsigned long long t0 = ptx::globaltimer_ns();
      while (ptx::globaltimer_ns() - t0 < 20000ull) {}
    }
    return;
  }
  // ---- the exponentials
  chain_wait();                                            // (the limit of the waits below is for this kernel's own work)
  const int group = warp / WARPS, gwarp = warp - group * WARPS, gtid = gwarp * 32 + lane;
  const uint32_t maxima = empty + 8u * (kRsRing + group), full = full0 + 8u * kRsRing * group;
  uint32_t slot = (uint32_t)(group * passes * n_chunks) % kRsRing, y = 0, phase = 0;    // the next chunk: its slot, its barrier and phase
  const uint32_t others = (uint32_t)((GROUPS - 1) * passes * n_chunks) % kRsRing;      // slots of the other groups' rows in between
  auto next_slot = [&](uint32_t n) { slot += n; if (slot >= kRsRing) slot -= kRsRing; };
  auto wait_chunk = [&]() {
    const bool there = ptx::mbar_wait_warp(full + 8u * y, phase, abort_flag);
    if (++y == kRsRing) { y = 0; phase ^= 1u; }
    return there;
  };
  auto chunk_done = [&]() {
    __syncwarp();
    if (lane == 0) ptx::mbar_arrive(empty + 8u * slot);
  };
  // f(vector) for the group's vectors of the chunk that is at hand; `left`: vectors of the row from the chunk's first on
  auto vectors = [&](int left, auto &&f) {
    const uint4 *src = reinterpret_cast<const uint4 *>(ring + (size_t)slot * kRsChunk) + gtid;
#pragma unroll 1
    for (int j = 0; j < kRsChunkVecs; j += 4 * THREADS) {
      if (left >= j + 4 * THREADS) {
        uint4 x[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) x[e] = src[j + e * THREADS];
#pragma unroll
        for (int e = 0; e < 4; ++e) f(x[e]);
      } else {
#pragma unroll 1
        for (int e = j; e < min(left, j + 4 * THREADS); e += THREADS) f(e + gtid < left ? src[e] : rs_pad<T>());
        return;
      }
    }
  };
  auto finish = [&](int stat, float m, int k) {            // a warp: the total of the group's row k
    u64 s = lane < WARPS ? sh_sum[group][k & 1][lane] : 0ull;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    if (lane == 0) { RowStat st; st.m = m; st.S = s; a.stats[stat] = st; }
  };
  int last_stat = -1, k = 0;
  float last_m = 0.f;
  for (;; ++k) {
    if (!wait_chunk()) goto gave_up;
    const int stat = infos[slot].stat, n_vec = infos[slot].n_vec, n_edge = infos[slot].n_edge;
    RsMax<T> mx;
    float edge = -INFINITY;
    if (stat >= 0) {
      if (gtid < n_edge) edge = infos[slot].edge[gtid];
      const uint32_t slot0 = slot;
      for (int c = 0; c < n_chunks; ++c) {
        if (c > 0 && !wait_chunk()) goto gave_up;
        vectors(n_vec - c * kRsChunkVecs, [&](const uint4 &x) { mx.take(x); });
        if (!resident) chunk_done();
        next_slot(1);
      }
      if (resident) slot = slot0;
    } else chunk_done();
    // the row's maxima and the last row's totals cross the group
    const int key = __reduce_max_sync(0xFFFFFFFFu, order_key(fmaxf(mx.get(), edge)));
    if (lane == 0) { sh_max[group][k & 1][gwarp] = key; ptx::mbar_arrive(maxima); }
    __syncwarp();
    if (!ptx::mbar_wait_warp(maxima, (uint32_t)k & 1u, abort_flag)) goto gave_up;
    if (last_stat >= 0 && gwarp == k % WARPS) finish(last_stat, last_m, k - 1);
    if (stat < 0) return;
    const float m = order_value(__reduce_max_sync(0xFFFFFFFFu, sh_max[group][k & 1][lane % WARPS]));
    u64 local = 0;
    if (n_edge > 0) local += exp_weight(edge, m);
    for (int c = 0; c < n_chunks; ++c) {
      if (!resident && !wait_chunk()) goto gave_up;
      vectors(n_vec - c * kRsChunkVecs, [&](const uint4 &x) {
        float f[VN];
        StatVec<T>::unpack(x, f);
#pragma unroll
        for (int e = 0; e < VN; e += 2) {
          u32 e0, e1;
          exp_weight2(f[e], f[e + 1], m, e0, e1);
          local += (u64)e0 + (u64)e1;
        }
      });
      chunk_done();
      next_slot(1);
    }
    const u64 s = warp_sum54(local);
    if (lane == 0) sh_sum[group][k & 1][gwarp] = s;
    last_stat = stat; last_m = m;
    next_slot(others);
  }
gave_up:
  give_up(a.stats, (long long)a.batch * (2 * a.t_max + 1));
}

// ------------------------------------------------------------------------------ clusters
// Draws, the statistics of few rows and all decisions: a cluster of C CTAs takes a row (a decision: a row of each side), each CTA
// the same V / C consecutive tokens.  Bound by latency, not by bytes (a row of 32000 bf16 tokens is 64 KB): a CTA's tokens are
// read once into registers, the maximum and then the integer total cross the cluster in one exchange each.  Draws need no
// scratch in global memory; statistics and decisions meet in the RowStats there.
// A warp owns consecutive tokens; lane and unit index are interleaved (unit = 4 bytes: a bf16 pair or an fp32 value;
// 2 bytes when rows of odd length leave bf16 pairs unaligned), so loads are whole lines whatever the row's alignment.
constexpr int kClThreads = 512, kClMaxC = 8;

template <typename T, int PER> struct ClUnit;              // PER tokens of one load
template <> struct ClUnit<float, 1> {
  typedef float raw;
  __device__ static void get(float r, float *f) { f[0] = r; }
  __device__ static raw none() { return -INFINITY; }
};
template <> struct ClUnit<__nv_bfloat16, 1> {
  typedef unsigned short raw;
  __device__ static void get(unsigned short r, float *f) { f[0] = __uint_as_float((u32)r << 16); }
  __device__ static raw none() { return 0xFF80u; }
};
template <> struct ClUnit<__nv_bfloat16, 2> {
  typedef u32 raw;
  __device__ static void get(u32 r, float *f) { f[0] = __uint_as_float(r << 16); f[1] = __uint_as_float(r & 0xFFFF0000u); }
  __device__ static raw none() { return 0xFF80FF80u; }
};

struct ClusterArgs {
  const void *p, *q;
  int32_t *tokens;
  int V, t_max, seg;             // seg: tokens per CTA, a multiple of 64
  DescList<VerifySeq> desc;      // verification: per sequence
  DescList<SampleRow> rows;      // draws: per row
  HostMirror mirror;
  int regular_t;                 // draws: rows per sequence
  u32 regular_serial, regular_level;
  u64 seed;
  int32_t *out_tokens, *out_n;
  int write_in_place;
  u32 coin24;
};

__device__ __forceinline__ u32 cl_rank() { u32 r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ u32 cl_size() { u32 r; asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ u32 cl_id() { u32 r; asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r)); return r; }
__device__ __forceinline__ void cl_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// "This CTA runs": a CTA may touch another's shared memory once every CTA of the cluster has arrived here.
__device__ __forceinline__ void cl_arrive() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cl_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ u32 cl_map(const void *p, u32 rank) {
  u32 r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((u32)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void cl_store(u32 addr, u32 v) { asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }
__device__ __forceinline__ void cl_store(u32 addr, u64 v) { asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory"); }
// Inverse CDF within a CTA whose weights pass the threshold: the warp, then the unit, then the token whose inclusive sum
// does.  w: the thread's weights, sums: the warps' totals, before: the sum of the CTAs in front.
template <int WARPS, int NT, int PER, class W, class Emit>
__device__ __forceinline__ void cl_find_token(const W (&w)[NT], u64 tau, u64 before, const u64 *sums, int k_lane, Emit emit) {
  constexpr int NU = NT / PER;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  u64 mine = lane < WARPS ? sums[lane] : 0ull;                  // every warp finds the owning one for itself
  u64 incl = mine;
  for (int o = 1; o < 32; o <<= 1) {
    const u64 v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += v;
  }
  const int owner = __ffs(__ballot_sync(0xFFFFFFFFu, before + incl > tau)) - 1;
  if (warp != owner) return;
  u64 base = before + __shfl_sync(0xFFFFFFFFu, incl - mine, owner);
  u64 tot[NU];
#pragma unroll
  for (int i = 0; i < NU; ++i) {
    u64 s = 0;
#pragma unroll
    for (int e = 0; e < PER; ++e) s += w[i * PER + e];
    tot[i] = warp_sum54(s);
  }
  bool done = false;
#pragma unroll
  for (int i = 0; i < NU; ++i) {
    if (!done && base + tot[i] > tau) {                            // uniform over the warp
      done = true;
      u64 s = 0;
#pragma unroll
      for (int e = 0; e < PER; ++e) s += w[i * PER + e];
      u64 c = s;
      for (int o = 1; o < 32; o <<= 1) {
        const u64 v = __shfl_up_sync(0xFFFFFFFFu, c, o);
        if (lane >= o) c += v;
      }
      const int l = __ffs(__ballot_sync(0xFFFFFFFFu, base + c > tau)) - 1;
      if (lane == l) {
        u64 run = base + c - s;
        int k = k_lane + 32 * PER * i;
#pragma unroll
        for (int e = 0; e < PER; ++e) {
          run += w[i * PER + e];
          if (run > tau) break;
          ++k;
        }
        emit(k);
      }
    } else if (!done) base += tot[i];
  }
}

// The units of a CTA's part of a row, -inf past its tokens (no weight, never the maximum); their maximum over the cluster; and the
// sum of a u64 a thread over the cluster, in every CTA (ALL) or in the first, whose parts csum holds.
template <typename T, int PER, int NU>
__device__ __forceinline__ void cl_units(const T *row, int k_lane, int tok_end, typename ClUnit<T, PER>::raw (&v)[NU]) {
#pragma unroll
  for (int u = 0; u < NU; ++u) {
    const int k = k_lane + 32 * PER * u;
    v[u] = k < tok_end ? __ldg(reinterpret_cast<const typename ClUnit<T, PER>::raw *>(row + k)) : ClUnit<T, PER>::none();
  }
}
template <int WARPS, int N> __device__ __forceinline__ float cl_max(const float (&f)[N], int *wmax /*[WARPS]*/, int *cmax /*[kClMaxC]*/, u32 rank, u32 C) {
  float m = -INFINITY;
#pragma unroll
  for (int e = 0; e < N; ++e) m = fmaxf(m, f[e]);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, key = __reduce_max_sync(0xFFFFFFFFu, order_key(m));
  if (lane == 0) wmax[warp] = key;
  __syncthreads();
  cl_wait();                                                       // every CTA of the cluster has started
  if (warp == 0) {
    const int all = __reduce_max_sync(0xFFFFFFFFu, wmax[lane & (WARPS - 1)]);
    if (lane < (int)C) cl_store(cl_map(&cmax[rank], (u32)lane), (u32)all);
  }
  cl_sync();
  int top = cmax[0];
  for (u32 c = 1; c < C; ++c) top = max(top, cmax[c]);
  return order_value(top);
}
template <int WARPS, bool ALL> __device__ __forceinline__ void cl_total(u64 local, u64 *wsum /*[WARPS]*/, u64 *csum /*[kClMaxC]*/, u32 rank, u32 C) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const u64 s = warp_sum54(local);
  if (lane == 0) wsum[warp] = s;
  __syncthreads();
  if (warp == 0) {
    u64 t = lane < WARPS ? wsum[lane] : 0ull;
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
    if (lane < (ALL ? (int)C : 1)) cl_store(cl_map(&csum[rank], (u32)lane), t);
  }
  cl_sync();
}

// Level 0's draw: token = inverse-CDF sample of softmax(row) with the purpose-0 uniform.  Two CTAs per SM.
template <typename T, int PER, int NT, int THREADS>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS) cluster_draw_kernel(const __grid_constant__ ClusterArgs a) {
  constexpr int NU = NT / PER, WARPS = THREADS / 32;
  __shared__ int wmax[WARPS], cmax[kClMaxC];                    // order keys
  __shared__ u64 wsum[WARPS], csum[kClMaxC];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const u32 rank = cl_rank(), C = cl_size();
  const int b = (int)cl_id();
  cl_arrive();                                                     // (the wait is in front of the first store to a peer)
  chain_wait();
  chain_next();
  SampleRow d;
  if (a.rows.given()) d = a.rows.at(b);
  else { d.logit_row = b; d.out_index = b; d.j = b % a.regular_t; d.seq = b / a.regular_t; d.serial = a.regular_serial; d.level = 0; }
  const int tok0 = (int)rank * a.seg, tok_end = min(a.V, tok0 + a.seg);
  const int k_lane = tok0 + warp * (32 * NT) + lane * PER;         // first token of unit i: k_lane + 32 PER i
  typename ClUnit<T, PER>::raw v[NU];
  cl_units<T, PER, NU>(reinterpret_cast<const T *>(a.p) + (size_t)d.logit_row * a.V, k_lane, tok_end, v);
  float f[NT];
#pragma unroll
  for (int u = 0; u < NU; ++u) ClUnit<T, PER>::get(v[u], f + u * PER);
  const float m = cl_max<WARPS>(f, wmax, cmax, rank, C);
  u32 w[NT];
  u64 local = 0, total = 0, before = 0;
#pragma unroll
  for (int e = 0; e < NT; e += 2) {
    exp_weight2(f[e], f[e + 1], m, w[e], w[e + 1]);
    local += (u64)w[e] + (u64)w[e + 1];
  }
  cl_total<WARPS, true>(local, wsum, csum, rank, C);
  for (u32 c = 0; c < C; ++c) {
    if (c < rank) before += csum[c];
    total += csum[c];
  }
  const u64 tau = cdf_threshold(uniform24(a.seed, d.j, d.serial, d.level, PURPOSE_DRAFT, d.seq), total);
  auto emit = [&](int k) {
    a.out_tokens[d.out_index] = k;
    if (a.mirror.token) a.mirror.token[(size_t)d.seq * a.mirror.stride + d.j] = k;
  };
  if (total == 0) {                                                // non-finite logits: no token
    if (rank == 0 && tid == 0) emit(-1);
  } else if (tau >= before && tau < before + csum[rank]) {
    cl_find_token<WARPS, NT, PER>(w, tau, before, wsum, k_lane, emit);
  }
}

// The statistics of few rows: a cluster a row, each CTA consecutive tokens of it in registers; the maximum and the total cross the
// cluster in one exchange each.  7 rows of 32000 bf16 tokens: 3.3 us (a CTA a row that takes them through its ring: 5.8).
template <typename T, int PER, int NT, int THREADS>
__global__ void __launch_bounds__(THREADS, (NT == 32 ? 512 : 1024) / THREADS) cluster_stats_kernel(const __grid_constant__ RowStatArgs a, int seg) {
  constexpr int NU = NT / PER, WARPS = THREADS / 32;
  __shared__ int wmax[WARPS], cmax[kClMaxC];                    // order keys
  __shared__ u64 wsum[WARPS], csum[kClMaxC];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const u32 rank = cl_rank(), C = cl_size();
  cl_arrive();                                                     // (the wait is in front of the first store to a peer)
  chain_wait();
  chain_next();
  const int rows_per_seq = 2 * a.t_max + 1, i = (int)cl_id(), b = i / rows_per_seq, r = i - b * rows_per_seq;
  const bool is_p = r <= a.t_max;
  const int at = is_p ? r : r - a.t_max - 1;
  long long row0 = (long long)b * (a.regular_t + (is_p ? 1 : 0));
  if (a.desc.given()) {
    const VerifySeq d = a.desc.at(b);
    if (at >= d.t + (is_p ? 1 : 0)) return;                        // the whole cluster
    row0 = is_p ? d.p_row0 : d.q_row0;
  }
  const T *row = reinterpret_cast<const T *>(is_p ? a.p : a.q) + (size_t)(row0 + at) * a.V;
  const int tok0 = (int)rank * seg, tok_end = min(a.V, tok0 + seg), k_lane = tok0 + warp * (32 * NT) + lane * PER;
  typename ClUnit<T, PER>::raw v[NU];
  cl_units<T, PER, NU>(row, k_lane, tok_end, v);
  float f[NT];
#pragma unroll
  for (int u = 0; u < NU; ++u) ClUnit<T, PER>::get(v[u], f + u * PER);
  const float m = cl_max<WARPS>(f, wmax, cmax, rank, C);
  u64 local = 0;
#pragma unroll
  for (int e = 0; e < NT; e += 2) {
    u32 e0, e1;
    exp_weight2(f[e], f[e + 1], m, e0, e1);
    local += (u64)e0 + (u64)e1;
  }
  cl_total<WARPS, false>(local, wsum, csum, rank, C);
  if (rank == 0 && tid == 0) {
    RowStat st;
    st.m = m; st.S = 0;
    for (u32 c = 0; c < C; ++c) st.S += csum[c];
    a.stats[i] = st;
  }
}

// The decision of a sequence whose rows' statistics are there (row_stats_kernel or cluster_stats_kernel, which this kernel
// follows in a chain): the accept tests by every CTA of the cluster for itself, the residual's weights of the CTA's tokens, one exchange
// of their totals.  Bound by latency: two gathers, a row of each side and an exchange.  Few
// sequences of 32000 tokens: 5.8 us behind the statistics; 64 of them, two CTAs each: 11.  Sums of four tokens instead of weights
// in registers, two CTAs an SM: 11 and 8.4.  The first positions' statistics kept in shared memory: 0.3 us more.
// 32 tokens a thread (calls whose clusters are of one or two CTAs): their 64-bit weights go past 128 registers, 84 to 144 bytes spill.
// MARKS: the statistics may be marks; looking for them costs 0.1 us (one sequence of three drafts: 7.39, with them 7.49), which
// cluster_stats_kernel, without a bounded wait, spares.
template <typename T, int PER, int NT, int THREADS, bool MARKS>
__global__ void __launch_bounds__(THREADS, kClThreads / THREADS) cluster_decide_kernel(const __grid_constant__ ClusterArgs a, const RowStat *stats) {
  typedef typename ClUnit<T, PER>::raw raw_t;
  constexpr int NU = NT / PER, WARPS = THREADS / 32;
  __shared__ u64 wsum[2][WARPS], csum[2][kClMaxC];              // [residual, the verifier's row]
  __shared__ int sh_n, sh_none;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const u32 rank = cl_rank(), C = cl_size();
  const int b = (int)cl_id();
  cl_arrive();                                                     // (the wait is in front of the first store to a peer)
  VerifySeq d;
  if (a.desc.given()) d = a.desc.at(b);
  else {
    d.t = a.regular_t; d.p_row0 = (long long)b * (a.regular_t + 1); d.q_row0 = (long long)b * a.regular_t;
    d.tok_off = (long long)b * a.regular_t; d.serial = a.regular_serial; d.seq = b; d.level = a.regular_level;
  }
  const int t = d.t;
  const T *p = reinterpret_cast<const T *>(a.p) + (size_t)d.p_row0 * a.V, *q = reinterpret_cast<const T *>(a.q) + (size_t)d.q_row0 * a.V;
  const RowStat *sp = stats + (size_t)b * (2 * a.t_max + 1), *sq = sp + a.t_max + 1;
  auto stat = [](const RowStat *s) {
    const float4 v = __ldcg(reinterpret_cast<const float4 *>(s));
    return *reinterpret_cast<const RowStat *>(&v);
  };
  if (tid == 0) { sh_n = t; sh_none = 0; }
  // the call's inputs are complete when the statistics kernel begins: the drafted tokens' logits come ahead of its end
  int tok = -1;
  float lp = 0.f, lq = 0.f;
  auto drafted = [&](int j) {
    tok = a.tokens[d.tok_off + j];
    if (tok >= 0 && tok < a.V) { lp = to_f32(p[(size_t)j * a.V + tok]); lq = to_f32(q[(size_t)j * a.V + tok]); }
  };
  if (tid < t) drafted(tid);
  __syncthreads();
  chain_wait();
  chain_next();
  for (int j = tid; j < t; j += THREADS) {
    if (j != tid) drafted(j);
    const RowStat s = stat(sp + j), r = stat(sq + j);
    if (MARKS && (s.S == kNoStat || r.S == kNoStat)) sh_none = 1;
    const bool in = tok >= 0 && tok < a.V;
    const u64 Pp = fixed_prob(in ? exp_weight(lp, s.m) : 0u, prob_scale(s.S)), Pq = fixed_prob(in ? exp_weight(lq, r.m) : 0u, prob_scale(r.S));
    const u32 U = uniform24(a.seed, j, d.serial, d.level, PURPOSE_ACCEPT, d.seq);
    bool ok = (((u64)U * Pq) >> 24) < Pp;                          // u < p(x) / q(x)
    if (a.coin24 != kNoCoin) ok = U < a.coin24;                    // ablation: IID acceptance with a fixed probability
    if (!ok) atomicMin(&sh_n, j);
  }
  __syncthreads();
  const int n = sh_n, tok0 = (int)rank * a.seg, tok_end = min(a.V, tok0 + a.seg);
  const int k_lane = tok0 + warp * (32 * NT) + lane * PER;         // first token of unit i: k_lane + 32 PER i
  const RowStat spn = stat(sp + n);
  if (MARKS && tid == 0 && spn.S == kNoStat) sh_none = 1;
  raw_t vp[NU];
  auto fetch = [&](const T *row, raw_t *v) {                       // -inf past the CTA's tokens: no weight
#pragma unroll
    for (int i = 0; i < NU; ++i) {
      const int k = k_lane + 32 * PER * i;
      v[i] = k < tok_end ? __ldg(reinterpret_cast<const raw_t *>(row + k)) : ClUnit<T, PER>::none();
    }
  };
  fetch(p + (size_t)n * a.V, vp);
  u64 w[NT], total = 0;
  bool running = false;                                            // every CTA of the cluster has started
  auto exchange = [&](int src, u64 local) {                        // the CTAs' totals -> csum[src], their sum -> total
    const u64 s = warp_sum54(local);
    if (lane == 0) wsum[src][warp] = s;
    __syncthreads();
    if (!running) cl_wait();
    running = true;
    if (warp == 0) {
      u64 c = lane < WARPS ? wsum[src][lane] : 0ull;
      for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xFFFFFFFFu, c, o);
      if (lane < (int)C) cl_store(cl_map(&csum[src][rank], (u32)lane), c);
    }
    cl_sync();
    total = 0;
    for (u32 c = 0; c < C; ++c) total += csum[src][c];
  };
  int src = 0;
  if (n < t) {
    raw_t vq[NU];
    fetch(q + (size_t)n * a.V, vq);
    const RowStat sqn = stat(sq + n);
    const ProbScale psp = prob_scale(spn.S), psq = prob_scale(sqn.S);
    u64 local = 0;
#pragma unroll
    for (int i = 0; i < NU; ++i) {
      float fp[PER], fq[PER];
      ClUnit<T, PER>::get(vp[i], fp);
      ClUnit<T, PER>::get(vq[i], fq);
#pragma unroll
      for (int e = 0; e < PER; ++e) {
        u32 ep, eq;
        exp_weight2m(fp[e], fq[e], spn.m, sqn.m, ep, eq);
        const u64 Pp = fixed_prob(ep, psp), Pq = fixed_prob(eq, psq);
        w[i * PER + e] = Pp > Pq ? Pp - Pq : 0ull;
        local += w[i * PER + e];
      }
    }
    exchange(0, local);
  }
  if (total == 0) {                                                // the bonus token, or an all-zero residual: the verifier's own row
    src = 1;
    u64 local = 0;
    if (n < t) fetch(p + (size_t)n * a.V, vp);                     // (once more, so that the residual need not keep it)
#pragma unroll
    for (int i = 0; i < NU; ++i) {
      float f[PER];
      ClUnit<T, PER>::get(vp[i], f);
#pragma unroll
      for (int e = 0; e < PER; ++e) {
        w[i * PER + e] = exp_weight(f[e], spn.m);
        local += w[i * PER + e];
      }
    }
    exchange(1, local);
  }
  if (MARKS && sh_none) total = 0;                                 // (what the marks gave so far stays within the row and the buffers)
  const u32 U = uniform24(a.seed, 0, d.serial, d.level, PURPOSE_FINAL, d.seq);
  const u64 tau = cdf_threshold(U, total);
  u64 before = 0;
  for (u32 c = 0; c < rank; ++c) before += csum[src][c];
  auto emit = [&](int k) {
    if (a.write_in_place) a.tokens[d.tok_off + n] = k;
    if (a.out_tokens) a.out_tokens[(size_t)b * (a.t_max + 1) + n] = k;
    if (a.mirror.n) a.mirror.token[b] = k;
  };
  if (total == 0) {                                                // non-finite logits or no statistics: no token
    if (rank == 0 && tid == 0) emit(-1);
  } else if (tau >= before && tau < before + csum[src][rank]) {
    cl_find_token<WARPS, NT, PER>(w, tau, before, wsum[src], k_lane, emit);
  }
  if (rank == 0) {
    const int n_out = MARKS && sh_none ? kNoDecision : n;
    if (tid == 0) {
      a.out_n[b] = n_out;
      if (a.mirror.n) a.mirror.n[b] = n_out;
      if (a.mirror.status && b == 0) *a.mirror.status = __ldcg(a.mirror.status_src);
    }
    if (a.out_tokens)
      for (int j = tid; j <= a.t_max; j += THREADS)
        if (j != n) a.out_tokens[(size_t)b * (a.t_max + 1) + j] = j < n_out ? a.tokens[d.tok_off + j] : -1;
  }
}

// Cluster size, tokens a thread, tokens and threads of a CTA of a call with n clusters; false if the rows are too long.  `two`: 1024
// threads' worth of CTAs per SM (decisions: 512).
struct ClusterPlan { int C, NT, per, seg, threads; };
constexpr int kClEights = 14;                     // clusters of eight that run at once (one CTA per SM) on the GPU that was measured: speed only
static bool cluster_plan(const void *p, const void *q, int dtype, int V, int n, bool two, ClusterPlan *pl) {
  pl->per = (dtype == HSD_BF16 && V % 2 == 0 && ((uintptr_t)p & 3) == 0 && ((uintptr_t)q & 3) == 0) ? 2 : 1;
  // as many CTAs as run at once, of at least 4096 tokens (eight a thread) each: clusters of eight do not fit all SMs
  // (16 of them took two rounds), clusters of four and two do
  int C = 1;
  while (C < kClMaxC && V > C * 4096 && 2ll * C * n <= (C == 4 ? 8 * kClEights : two ? 2 * kMeasuredSMs : kMeasuredSMs)) C *= 2;
  const int most = (two ? 16 : 32) * kClThreads;
  while (C < kClMaxC && ceil_div(V, C) > most - 64) C *= 2;
  const int seg = ceil_div(ceil_div(V, C), 64) * 64;
  if (seg > most) return false;
  pl->C = C;
  pl->seg = seg;
  // rows of up to 1024 and 2048 tokens, eight a thread: fewer warps to meet, more rows on an SM
  pl->threads = seg <= 1024 ? 128 : seg <= 2048 ? 256 : kClThreads;
  // decisions of more sequences than SMs: two CTAs a SM, of 16 or 32 tokens a thread (us a verification of 4000 bf16 tokens, 512 / 256
  // threads: 148 x 1 10.3 / 10.8, 200 x 1 15.5 / 12.2, 2000 x 3 151 / 118; 8000: 200 x 1 19.3 / 17.0, 2000 x 3 196 / 165)
  if (!two && n > kMeasuredSMs && seg <= 8192 && pl->threads == kClThreads) pl->threads = 256;
  pl->NT = seg <= 8 * pl->threads ? 8 : seg <= 16 * pl->threads ? 16 : 32;
  return true;
}
// Where clusters are the faster ones (us a call in a row of calls, clusters / other path).  Rows of up to 2048 tokens, in CTAs of 128 or
// 256 threads: always.  Against CTAs of 512 threads and, past two rounds of them, the other path: verifications, bf16, 513 tokens, 1 x 3 8.3 ->
// 7.1, 64 x 8 13.9 -> 9.0, 2000 x 1 103 -> 32; 2048, 64 x 8 12.4 -> 10.5; draws of 513, 1 row 3.5 -> 3.05, 2000 27 -> 8.6, of 2048 3.2 -> 2.8, 24.4 -> 13.3.
//   statistics (the whole verification), while the clusters run in one round: 32000 bf16, 7 rows 8.4 / 10.8, 66 rows 10.1 / 11.5, 88 rows (in
//     two rounds) 12.9 / 11.5; fp32, 7 rows 9.2 / 12.9, 66: 11.1 / 13.3, 88: 13.8 / 13.5; 16000 bf16, 132 rows 10.1 / 10.0, 176 (two) 11.9 / 11.6; 2048:
//     8.0 / 8.0, 176 rows 8.8 / 8.7; 45001 bf16, 33 rows 13.5 / 16.1, 44 (two) 16.4 / 16.2.
//   draws (two CTAs per SM, 16 tokens a thread at most), other path a CTA of 1024 threads a row, which has 32 tokens a thread where bf16 rows
//     allow (`chunked`): while the clusters run in one round, bf16 32000: 1 row 4.0 / 10.2, 64 rows 5.8 / 11.0; 2048: 3.8 / 8.5 to 9.4;
//     fp32 32000: 4.1 / 26, 64 rows 6.6 / 28; 8000: 4.1 / 6.1; 2048: 3.9 / 3.9.  In more rounds, chunked: 32000, 100 rows 9.4 / 11.1, 148: 12.5 / 11.1
//     (a row a CTA then), 200: 14.6 / 20.5, 512: 37 / 40, 16000, 512: 18 / 35; others: fp32 9001, 256: 12 / 9.1, 16000, 256: 11 / 16.9 (two CTAs a row),
//     20000, 148: 13.4 / 10.7, 32000, 100: 10.2 / 28, 512: 41 / 105; 8000, 512: 10.7 / 15.9; bf16 32001, 256: 21 / 38.
//   Rows of more than 65536 tokens (clusters of eight, 32 tokens a thread, one CTA an SM), up to four rounds: 128256 bf16, 1 row 22.4 -> 9, 16 rows
//     26.5 -> 14.6, 48 rows 31.6 -> 21 to 24; 70001, 56 rows as fast, 64 34.6 -> 36.3.
static bool cluster_plan_stats(const RowStatArgs &a, int dtype, int rows, ClusterPlan *pl) {
  if (cluster_plan(a.p, a.q, dtype, a.V, rows, true, pl)) return pl->threads < kClThreads || (long long)pl->C * rows <= 2 * kMeasuredSMs;
  return rows <= 4 * kClEights && cluster_plan(a.p, a.q, dtype, a.V, rows, false, pl);
}
//   decisions of more sequences than SMs by decide_kernel, two CTAs of 1024 threads a SM that read their rows through the first-level
//     cache (the whole verification, clusters / decide_kernel): 12000 bf16 200 x 1 25.0 / 25.5; 16385, 200 x 0 29.7 / 16.9, 2000 x 3 655 / 293;
//     24000, 149 x 3 42.3 / 44.5, 300 x 0 36 / 25, 2000 x 3 472 / 343, fp32 300 x 0 47 / 31, 2000 x 3 581 / 413; 32000 bf16, 300 x 1 60 / 66, fp32 50 / 90.  Up
//     to 8192 tokens against 256 threads: fp32 8000, 200 x 1 20.7 / 22.5, 300 x 0 19.0 / 16.3, 600 x 3 68 / 64, bf16 600 x 3 52.8 / 56.8.
static bool cta_pays_decide(int dtype, int V, int n) {
  return V <= 8192 ? dtype == HSD_F32 && V > 4096 && n > 2 * kMeasuredSMs : V <= 24576 && n > kMeasuredSMs;
}
static bool cluster_pays_draw(const ClusterPlan &pl, int V, int n, bool chunked) {
  if (pl.threads < kClThreads || pl.C * n <= 2 * kMeasuredSMs) return true;
  if (chunked) return n > kMeasuredSMs || pl.C * n <= 3 * kMeasuredSMs;
  return V > 26000 || V <= 8192 || (V > 13500 && pl.C == 2);
}

template <typename T, int PER>
static int launch_cluster_draw_nt(const ClusterArgs &a, const ClusterPlan &pl, int n, cudaStream_t s) {
  const int grid = n * pl.C;
  auto go = [&](auto kernel, int threads) { return hsd_launch(kernel, grid, threads, 0, s, pl.C, true, a); };
  HSD_CUDA_OK(pl.threads == 128   ? go(cluster_draw_kernel<T, PER, 8, 128>, 128)
              : pl.threads == 256 ? go(cluster_draw_kernel<T, PER, 8, 256>, 256)
              : pl.NT == 8        ? go(cluster_draw_kernel<T, PER, 8, kClThreads>, kClThreads)
                                  : go(cluster_draw_kernel<T, PER, 16, kClThreads>, kClThreads));
  hsd_count_launches(1);
  return hsd_launch_status();
}
static int launch_cluster_draw(ClusterArgs a, const ClusterPlan &pl, int dtype, int n, cudaStream_t s) {
  a.seg = pl.seg;
  if (dtype == HSD_F32) return launch_cluster_draw_nt<float, 1>(a, pl, n, s);
  return pl.per == 2 ? launch_cluster_draw_nt<__nv_bfloat16, 2>(a, pl, n, s) : launch_cluster_draw_nt<__nv_bfloat16, 1>(a, pl, n, s);
}

// ------------------------------------------------------------------------------ host launchers
// Scratch of one verification call: a RowStat per logits row, at its front.  (The rest is room that callers' buffers have always had.)
size_t verify_scratch_bytes(int batch, int t_max) {
  return ((size_t)(2 * batch + 2) * 4 + 255) / 256 * 256 + (size_t)batch * (2 * t_max + 1) * sizeof(RowStat);
}

template <typename T>
static int launch_draft_sample_t(const void *logits, int V, const DescList<SampleRow> &desc, int n_rows, int regular_rows,
                                 u32 regular_serial, u64 seed, int32_t *out, cudaStream_t s, const HostMirror &mirror) {
  HSD_CUDA_OK(hsd_launch(draft_sample_kernel<T>, n_rows, kSampleThreads, 0, s, 0, true, (const T *)logits, V, desc, regular_rows, regular_serial, seed, out, mirror));
  hsd_count_launches(1);
  return hsd_launch_status();
}

int launch_draft_sample(const void *logits, int dtype, int V, const SampleRow *desc, int n_rows, int regular_rows,
                        u32 regular_serial, u64 seed, int32_t *out, cudaStream_t s, bool desc_on_host, HostMirror mirror) {
  if (n_rows == 0) return HSD_OK;
  if (desc_on_host && n_rows > kInlineDesc) return HSD_E_INVALID_ARG;
  const DescList<SampleRow> list = desc_list(desc, n_rows, desc_on_host);
  ClusterPlan pl;
  if (cluster_plan(logits, nullptr, dtype, V, n_rows, true, &pl) &&
      cluster_pays_draw(pl, V, n_rows, dtype == HSD_BF16 && V % 8 == 0 && V <= kSampleThreads * kChunkTokens && ((uintptr_t)logits & 15) == 0)) {
    ClusterArgs a = {};
    a.p = logits; a.V = V; a.t_max = 0; a.rows = list; a.mirror = mirror; a.regular_t = regular_rows;
    a.regular_serial = regular_serial; a.seed = seed; a.out_tokens = out; a.coin24 = kNoCoin;
    return launch_cluster_draw(a, pl, dtype, n_rows, s);
  }
  return dtype == HSD_BF16
             ? launch_draft_sample_t<__nv_bfloat16>(logits, V, list, n_rows, regular_rows, regular_serial, seed, out, s, mirror)
             : launch_draft_sample_t<float>(logits, V, list, n_rows, regular_rows, regular_serial, seed, out, s, mirror);
}

static int sm_count() {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) n = 148;
    sms = n;
  }
  return sms;
}

template <typename T, int GROUPS, int WARPS>
static int launch_row_stats_t(const RowStatArgs &a, int grid, cudaStream_t s) {
  constexpr int smem = (int)kRsBytes + 128;
  static std::atomic<u64> limits{0};
  const int limit = hsd_smem_limit((const void *)row_stats_kernel<T, GROUPS, WARPS>, smem, limits);
  if (limit) return limit;
  HSD_CUDA_OK(hsd_launch(row_stats_kernel<T, GROUPS, WARPS>, grid, 32 * (GROUPS * WARPS + 1), smem, s, 0, true, a));
  hsd_count_launches(1);
  return HSD_OK;
}
template <typename T, int PER>
static int launch_cluster_stats(const RowStatArgs &a, const ClusterPlan &pl, int n, cudaStream_t s) {
  const int grid = n * pl.C;
  auto go = [&](auto kernel, int threads) { return hsd_launch(kernel, grid, threads, 0, s, pl.C, true, a, pl.seg); };
  HSD_CUDA_OK(pl.threads == 128   ? go(cluster_stats_kernel<T, PER, 8, 128>, 128)
              : pl.threads == 256 ? go(cluster_stats_kernel<T, PER, 8, 256>, 256)
              : pl.NT == 8        ? go(cluster_stats_kernel<T, PER, 8, kClThreads>, kClThreads)
              : pl.NT == 16       ? go(cluster_stats_kernel<T, PER, 16, kClThreads>, kClThreads)
                                  : go(cluster_stats_kernel<T, PER, 32, kClThreads>, kClThreads));
  hsd_count_launches(1);
  return HSD_OK;
}
// us a call, GROUPS x WARPS = 1 x 16 / 2 x 8 / 3 x 8 (chunks of 32 KB; the middle one and 2 x 12 on chunks of 24 KB, behind it, are not built):
//   a row a CTA, 32000: bf16 5.6 / 5.9 / 6.2, fp32 6.9 / 7.4 / 7.7
//   1088 rows of 32000: bf16 29.7 / 25.3 / 24.6, fp32 35.3 / 32.3 / 32.5; of 2048: bf16 9.6 / 7.0 / 6.9; of 50000, fp32: 57.4 / 57.7 / 58.2
// *marks: the statistics may be marks (kNoStat)
static int launch_row_stats(const RowStatArgs &a, int dtype, cudaStream_t s, bool *marks) {
  const long long n_items = (long long)a.batch * (2 * a.t_max + 1);
  ClusterPlan pl;
  if (n_items <= 0x7FFFFFFFll / kClMaxC && cluster_plan_stats(a, dtype, (int)n_items, &pl)) {
    if (dtype == HSD_F32) return launch_cluster_stats<float, 1>(a, pl, (int)n_items, s);
    return pl.per == 2 ? launch_cluster_stats<__nv_bfloat16, 2>(a, pl, (int)n_items, s) : launch_cluster_stats<__nv_bfloat16, 1>(a, pl, (int)n_items, s);
  }
  *marks = true;
  const int grid = (int)std::min<long long>(sm_count(), n_items);
  if (n_items <= grid)                                     // a row a CTA: all its warps on it
    return dtype == HSD_F32 ? launch_row_stats_t<float, 1, 16>(a, grid, s) : launch_row_stats_t<__nv_bfloat16, 1, 16>(a, grid, s);
  return dtype == HSD_F32 ? launch_row_stats_t<float, 3, 8>(a, grid, s) : launch_row_stats_t<__nv_bfloat16, 3, 8>(a, grid, s);
}

template <typename T, int PER, bool MARKS>
static int launch_decide_nt(const ClusterArgs &a, const ClusterPlan &pl, int n, const RowStat *stats, cudaStream_t s) {
  const int grid = n * pl.C;
  auto go = [&](auto kernel, int threads) { return hsd_launch(kernel, grid, threads, 0, s, pl.C, true, a, stats); };
  cudaError_t e;
  if (!MARKS && pl.threads == 128) e = go(cluster_decide_kernel<T, PER, 8, 128, false>, 128);    // (such rows' statistics are the clusters')
  else if (!MARKS && pl.threads == 256 && pl.NT == 8) e = go(cluster_decide_kernel<T, PER, 8, 256, false>, 256);
  else if (pl.threads == 256 && pl.NT == 16) e = go(cluster_decide_kernel<T, PER, 16, 256, MARKS>, 256);
  else if (pl.threads == 256 && pl.NT == 32) e = go(cluster_decide_kernel<T, PER, 32, 256, MARKS>, 256);
  else if (pl.NT == 8) e = go(cluster_decide_kernel<T, PER, 8, kClThreads, MARKS>, kClThreads);
  else if (pl.NT == 16) e = go(cluster_decide_kernel<T, PER, 16, kClThreads, MARKS>, kClThreads);
  else e = go(cluster_decide_kernel<T, PER, 32, kClThreads, MARKS>, kClThreads);
  HSD_CUDA_OK(e);
  hsd_count_launches(1);
  return hsd_launch_status();
}

template <typename T, int CTAS> static int launch_decide_long(const ClusterArgs &a, int batch, const RowStat *stats, cudaStream_t s) {
  decide_kernel<T, CTAS><<<batch, kSampleThreads, 0, s>>>((const T *)a.p, (const T *)a.q, a.tokens, a.V, a.t_max, a.desc, a.regular_t, a.regular_serial,
                                                    a.regular_level, stats, a.seed, a.out_tokens, a.out_n, a.write_in_place, a.coin24, a.mirror);
  hsd_count_launches(1);
  return hsd_launch_status();
}
template <bool MARKS> static int launch_decide(const ClusterArgs &a, const ClusterPlan &pl, int dtype, int batch, const RowStat *stats, cudaStream_t s) {
  if (dtype == HSD_F32) return launch_decide_nt<float, 1, MARKS>(a, pl, batch, stats, s);
  return pl.per == 2 ? launch_decide_nt<__nv_bfloat16, 2, MARKS>(a, pl, batch, stats, s) : launch_decide_nt<__nv_bfloat16, 1, MARKS>(a, pl, batch, stats, s);
}
static int launch_decisions(ClusterArgs a, int dtype, int batch, const RowStat *stats, bool marks, cudaStream_t s) {
  ClusterPlan pl;
  if (!cluster_plan(a.p, a.q, dtype, a.V, batch, false, &pl))      // rows of more than 131072 tokens
    return dtype == HSD_BF16 ? launch_decide_long<__nv_bfloat16, 1>(a, batch, stats, s) : launch_decide_long<float, 1>(a, batch, stats, s);
  if (cta_pays_decide(dtype, a.V, batch))
    return dtype == HSD_BF16 ? launch_decide_long<__nv_bfloat16, 2>(a, batch, stats, s) : launch_decide_long<float, 2>(a, batch, stats, s);
  a.seg = pl.seg;
  return marks ? launch_decide<true>(a, pl, dtype, batch, stats, s) : launch_decide<false>(a, pl, dtype, batch, stats, s);
}

int launch_verify(const void *p, const void *q, int32_t *tokens, int dtype, int V, int batch, int t_max,
                  const VerifySeq *desc, int regular_t, u32 regular_serial, u32 regular_level, void *scratch,
                  u64 seed, int32_t *out_tokens, int32_t *out_n, int write_in_place, cudaStream_t s,
                  u32 coin24, bool desc_on_host, HostMirror mirror) {
  if (batch == 0) return HSD_OK;
  if (desc_on_host && batch > kInlineDesc) return HSD_E_INVALID_ARG;
  const DescList<VerifySeq> list = desc_list(desc, batch, desc_on_host);
  RowStat *stats = (RowStat *)scratch;
  RowStatArgs r = {};
  r.p = p; r.q = q; r.V = V; r.t_max = t_max; r.batch = batch; r.regular_t = regular_t; r.desc = list; r.stats = stats;
  bool marks = false;
  const int st = launch_row_stats(r, dtype, s, &marks);
  if (st) return st;
  ClusterArgs a = {};
  a.p = p; a.q = q; a.tokens = tokens; a.V = V; a.t_max = t_max; a.desc = list; a.mirror = mirror; a.regular_t = regular_t;
  a.regular_serial = regular_serial; a.regular_level = regular_level; a.seed = seed; a.out_tokens = out_tokens; a.out_n = out_n;
  a.write_in_place = write_in_place; a.coin24 = coin24;
  return launch_decisions(a, dtype, batch, stats, marks, s);
}

// ------------------------------------------------------------------------------ static scratch
// Scratch for hsd_verify_level_static: lives in the library image, so every GPU that loads the
// library holds these bytes until the process exits.  One RowStat per logits row of a call.
constexpr int kStaticStatRows = 4096;
static __device__ RowStat g_static_verify_scratch[kStaticStatRows];

// In host code the array's name is only a stand-in for the symbol, not a device address: the
// address has to be asked for, once per device, with that device current.  The answer is kept per
// device in an atomic (two host threads may make a device's first call at once: both look the
// symbol up and store the same value).  It does not survive cudaDeviceReset(): a process that
// resets a device must not use this entry point on it afterwards.
static std::atomic<void *> g_static_scratch_ptr[64];
static int static_scratch_address(void **out) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return HSD_E_CUDA;
  void *p = g_static_scratch_ptr[dev].load(std::memory_order_acquire);
  if (!p) {
    if (cudaGetSymbolAddress(&p, g_static_verify_scratch) != cudaSuccess || !p) return HSD_E_CUDA;
    g_static_scratch_ptr[dev].store(p, std::memory_order_release);
  }
  *out = p;
  return HSD_OK;
}

}  // namespace hsd

// ------------------------------------------------------------------------------ C ABI
unsigned long long g_hsd_launches = 0;

extern "C" {

uint64_t hsd_kernel_launches(void) { return g_hsd_launches; }

const char *hsd_strerror(int status) {
  switch (status) {
    case HSD_OK: return "ok";
    case HSD_E_INVALID_ARG: return "invalid argument";
    case HSD_E_WORKSPACE_TOO_SMALL: return "workspace too small";
    case HSD_E_OUT_OF_PAGES: return "out of KV pages";
    case HSD_E_CUDA: return "CUDA error";
    case HSD_E_DEVICE_TIMEOUT: return "device-side wait timed out";
    case HSD_E_UNSUPPORTED: return "unsupported configuration";
    case HSD_E_IO: return "I/O error";
    case HSD_E_TOO_LARGE: return "request exceeds the built-in scratch capacity";
    default: return "unknown status";
  }
}

int hsd_draft_sample(const void *logits, int batch, int rows, int vocab, int dtype, uint64_t seed,
                     uint64_t call_serial, void *stream, int32_t *out_tokens) {
  if (!logits || !out_tokens || batch <= 0 || rows <= 0 || vocab <= 0) return HSD_E_INVALID_ARG;
  if (dtype != HSD_F32 && dtype != HSD_BF16) return HSD_E_INVALID_ARG;
  if ((long long)batch * rows > 0x7FFFFFFFll) return HSD_E_INVALID_ARG;
  return hsd::launch_draft_sample(logits, dtype, vocab, nullptr, batch * rows, rows, (u32)call_serial, seed, out_tokens,
                                  (cudaStream_t)stream);
}

size_t hsd_verify_workspace_bytes(int batch, int t) {
  if (batch <= 0 || t < 0) return 0;
  return hsd::verify_scratch_bytes(batch, t);
}

int hsd_verify_level(int level, const void *target_logits, const void *draft_logits, const int32_t *draft_tokens,
                     int batch, int t, int vocab, int dtype, uint64_t seed, uint64_t call_serial, void *workspace,
                     size_t workspace_bytes, void *stream, int32_t *out_tokens, int32_t *out_n_accepted) {
  if (!target_logits || !out_tokens || !out_n_accepted || !workspace) return HSD_E_INVALID_ARG;
  if (batch <= 0 || t < 0 || vocab <= 0 || level < 0 || level > 255) return HSD_E_INVALID_ARG;
  if (t > 0 && (!draft_logits || !draft_tokens)) return HSD_E_INVALID_ARG;
  if (t >= hsd::kSampleThreads || batch > 65535) return HSD_E_INVALID_ARG;
  if (dtype != HSD_F32 && dtype != HSD_BF16) return HSD_E_INVALID_ARG;
  if (((uintptr_t)workspace & 15) != 0) return HSD_E_INVALID_ARG;
  if (workspace_bytes < hsd::verify_scratch_bytes(batch, t)) return HSD_E_WORKSPACE_TOO_SMALL;
  return hsd::launch_verify(target_logits, draft_logits, const_cast<int32_t *>(draft_tokens), dtype, vocab, batch, t,
                            nullptr, t, (u32)call_serial, (u32)level, workspace, seed, out_tokens, out_n_accepted, 0,
                            (cudaStream_t)stream);
}

int hsd_verify_level_static(int level, const void *target_logits, const void *draft_logits, const int32_t *draft_tokens,
                            int batch, int t, int vocab, int dtype, uint64_t seed, uint64_t call_serial, void *stream,
                            int32_t *out_tokens, int32_t *out_n_accepted) {
  if (!target_logits || !out_tokens || !out_n_accepted) return HSD_E_INVALID_ARG;
  if (batch <= 0 || t < 0 || vocab <= 0 || level < 0 || level > 255) return HSD_E_INVALID_ARG;
  if (t > 0 && (!draft_logits || !draft_tokens)) return HSD_E_INVALID_ARG;
  if (t >= hsd::kSampleThreads || batch > 65535) return HSD_E_INVALID_ARG;
  if (dtype != HSD_F32 && dtype != HSD_BF16) return HSD_E_INVALID_ARG;
  if ((long long)batch * (2 * t + 1) > hsd::kStaticStatRows) return HSD_E_TOO_LARGE;
  void *scratch = nullptr;
  int st = hsd::static_scratch_address(&scratch);          // first call on this device looks the symbol up
  if (st) return st;
  // every RowStat the decision reads is written by the same call first
  return hsd::launch_verify(target_logits, draft_logits, const_cast<int32_t *>(draft_tokens), dtype, vocab, batch, t,
                            nullptr, t, (u32)call_serial, (u32)level, scratch, seed, out_tokens, out_n_accepted, 0,
                            (cudaStream_t)stream);
}

}  // extern "C"
