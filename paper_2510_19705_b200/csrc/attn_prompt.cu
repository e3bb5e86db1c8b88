// Prompt attention on tcgen05 with scores, weights and outputs in tensor memory.
//
// One CTA = one KV head and up to 2 x 128 query vectors (two tiles A and B of consecutive tokens x the heads of the
// KV group), over all keys up to the last of them, in tiles of 64 keys.  Per key tile and query tile
//   S[128 x 64]   = Q K^T                      both operands in shared memory
//   P             = exp2((S - m_ref) scale log2 e), thread = query vector, split into bf16 hi + lo halves that overwrite
//                   S (the P V product keeps about 16 bits of P, at every length)
//   O[128 x hd]  += P_hi V + P_lo V            A operand from tensor memory, V as it lies in the cache (MN-major)
// m_ref moves only when a row maximum passes it by a factor 256; then O is rescaled.  Two query tiles share every K
// and V tile.  S has two buffers per query tile: the scores of the next key tile are ready when the weights of this one
// are, so a tile's chain is load - maximum - exponentials - store and the products run beside it.
// Bound by that chain: 2304 rows of the 8B shape behind 4608 cached keys 354 us with one S buffer and 128-key tiles
// (which put the products into the chain; sixteen softmax warps, or the tiles' exponentials in turns, changed nothing),
// 284 us this way with one bf16 per weight, 326 us with hi + lo.
// 320 threads: warps 0-3 / 4-7 = softmax of tile A / B, warp 8 = K / V loader (TMA: a tile per copy and column block;
// the pages of a tile follow one another in the pool), warp 9 = MMA issue (one elected lane).  Items come longest first.
// Every wait is bounded, and no waiter can be passed by (a parity wait sees a completion only until the next one): k_full and
// v_full have their next loads behind k_free / v_free, which the issuer's commits complete; those their next MMAs behind the
// loader's tiles; s_full, pv_done (looked at only before a rescale) and o_done theirs behind p_ready of all four softmax warps;
// p_ready its next weights behind the scores.
#include <algorithm>
#include "attn_prompt.cuh"
#include "gemm_tc.cuh"
#include "tc_ptx.cuh"

namespace hsd {
namespace {

using namespace ptx;

constexpr int kThreads = 320, kLoaderWarp = 8, kMmaWarp = 9;
constexpr int TK = 64;                                   // keys per tile
constexpr int kQBlk = 128 * 128;                         // [128 query vectors][64 bf16] block, 128-byte swizzle
constexpr int kBlk = TK * 128;                           // [64 keys][64 bf16] block
constexpr int kStages = 4;

template <int HD> struct Cfg {
  static constexpr int NB = HD / 64;                     // 64-column blocks
  static constexpr int kQTile = NB * kQBlk, kTile = NB * kBlk;
  static constexpr int kOffK = 2 * kQTile, kOffV = kOffK + kStages * kTile, kOffBar = kOffV + kStages * kTile;
  static constexpr int kSmem = kOffBar + 256 + 1024;
};

// Shared-memory descriptors with the 128-byte swizzle as two words: the low one (address / 16, and between 64-column
// blocks of an MN-major operand their distance / 16) advances by constants from MMA to MMA, the high one (8-row groups
// 1024 bytes apart, descriptor version, swizzle mode) is the same for all.
constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t desc_lo_k(uint32_t addr) { return ((addr & 0x3FFFFu) >> 4) | (1u << 16); }
__device__ __forceinline__ uint32_t desc_lo_mn(uint32_t addr) { return ((addr & 0x3FFFFu) >> 4) | ((uint32_t)(kBlk >> 4) << 16); }
__device__ __forceinline__ void umma_ss(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\tmov.b64 da, {%1, %5};\n\tmov.b64 db, {%2, %5};\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(idesc), "r"(acc), "r"(kDescHi) : "memory");
}
__device__ __forceinline__ void umma_ts(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 db;\n\tmov.b64 db, {%2, %5};\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(idesc), "r"(acc), "r"(kDescHi) : "memory");
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void tmem_st8u(uint32_t taddr, const unsigned *r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]) : "memory");
}

template <int HD>
__global__ void __launch_bounds__(kThreads, 1) prompt_attn_kernel(const __grid_constant__ PromptAttnArgs a) {
  using C = Cfg<HD>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  __shared__ uint32_t tmem_slot;
  __shared__ int sh_abort;
  volatile int *abort_flag = &sh_abort;
  const uint32_t s0 = smem_u32(smem), b0 = s0 + C::kOffBar;
  auto k_full = [&](int b) { return b0 + 8u * b; };
  auto k_free = [&](int b) { return b0 + 8u * (4 + b); };
  auto v_full = [&](int b) { return b0 + 8u * (8 + b); };
  auto v_free = [&](int b) { return b0 + 8u * (12 + b); };
  auto s_full = [&](int x, int b) { return b0 + 8u * (16 + 2 * x + b); };
  auto p_ready = [&](int x, int b) { return b0 + 8u * (20 + 2 * x + b); };   // (per buffer: the softmax may be a tile ahead of the products)
  auto pv_done = [&](int x) { return b0 + 8u * (24 + x); };
  auto o_done = [&](int x) { return b0 + 8u * (26 + x); };           // the last P V (a barrier of its own: the parity wait tells neighbours apart only)
  const uint32_t v_land = b0 + 8u * 28;
  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int kvh = blockIdx.x % a.nkv;
  const int4 it = a.items[blockIdx.x / a.nkv];
  const int row0 = it.x, ntok = it.y, seq = it.z, pos0 = it.w;
  const int group = a.nq / a.nkv, tpt = 128 / group;                 // tokens per query tile
  const int tokA = min(ntok, tpt), tokB = ntok - tokA;
  const int kv_len = pos0 + ntok;
  const int nA = (pos0 + tokA + TK - 1) / TK, nB = tokB > 0 ? (kv_len + TK - 1) / TK : 0;
  const int n = max(nA, nB);

  if (threadIdx.x == 0) {
    for (int b = 0; b < kStages; ++b) { mbar_init(k_full(b), 1); mbar_init(k_free(b), 1); mbar_init(v_full(b), 1); mbar_init(v_free(b), 1); }
    for (int x = 0; x < 2; ++x) { mbar_init(s_full(x, 0), 1); mbar_init(s_full(x, 1), 1); mbar_init(p_ready(x, 0), 4); mbar_init(p_ready(x, 1), 4); mbar_init(pv_done(x), 1); mbar_init(o_done(x), 1); }
    mbar_init(v_land, 1);
    sh_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) tmem_alloc(smem_u32(&tmem_slot), 512);
  chain_next();
  chain_wait();
  if (warp < kLoaderWarp) {
    // Q: thread = query vector; K-major, 128-byte swizzle; vectors past the tile's tokens are zero
    const int x = warp >> 2, row = (warp & 3) * 32 + lane, tok = row / group, g = row - tok * group;
    const bool real = tok < (x ? tokB : tokA) && row < tpt * group;
    const uint4 *src = reinterpret_cast<const uint4 *>(a.q + ((size_t)(row0 + x * tpt + tok) * a.nq + kvh * group + g) * HD);
    uint4 v[HD / 8];
#pragma unroll
    for (int c = 0; c < HD / 8; ++c) v[c] = real ? __ldcg(src + c) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int c = 0; c < HD / 8; ++c)
      *reinterpret_cast<uint4 *>(smem + x * C::kQTile + (c >> 3) * kQBlk + (row >> 3) * 1024 + (row & 7) * 128 + (((c & 7) ^ (row & 7)) << 4)) = v[c];
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  auto tS = [&](int x) { return tmem + (uint32_t)(x * 128); };
  auto tO = [&](int x) { return tmem + 256u + (uint32_t)(x * HD); };

  if (warp == kLoaderWarp) {
    // ------------------------------------------------------------------ loader
    const int *pt = a.page_table + (size_t)seq * a.pages_per_seq;
    const bool issuer = elect_one();
    bool ok = true;
    auto wait = [&](uint32_t bar, uint32_t parity) { ok = mbar_wait_warp(bar, parity, abort_flag); return ok; };
    for (int j = 0; j < n; ++j) {
      const int b = j % kStages, key = j * TK;
      const uint32_t ph = (uint32_t)((j / kStages) & 1);
      // (rows past the last key belong to nobody: their scores are masked, their V rows zeroed below)
      const int row = ((kvh * a.n_pages + pt[key >> a.page_shift]) << a.page_shift) + (key & ((1 << a.page_shift) - 1));
      if (!wait(k_free(b), ph ^ 1u)) break;
      if (issuer) {
        mbar_expect_tx(k_full(b), C::kTile);
#pragma unroll
        for (int i = 0; i < C::NB; ++i) tma_load_2d(s0 + C::kOffK + b * C::kTile + i * kBlk, &a.k, i * 64, row, k_full(b));
      }
      const bool tail = (j + 1) * TK > kv_len;
      if (!wait(v_free(b), ph ^ 1u)) break;
      if (issuer) {
        mbar_expect_tx(tail ? v_land : v_full(b), C::kTile);
#pragma unroll
        for (int i = 0; i < C::NB; ++i) tma_load_2d(s0 + C::kOffV + b * C::kTile + i * kBlk, &a.v, i * 64, row, tail ? v_land : v_full(b));
      }
      if (tail) {                                                    // the last tile: V rows past the last key must be finite (P is 0 there)
        if (!wait(v_land, 0u)) break;
        const int r0 = kv_len - j * TK;
        for (int i = r0 * 8 * C::NB + lane; i < TK * 8 * C::NB; i += 32) {
          const int r = i / (8 * C::NB), c = i % (8 * C::NB);        // whole rows: the swizzle permutes within a row
          *reinterpret_cast<uint4 *>(smem + C::kOffV + b * C::kTile + (c >> 3) * kBlk + r * 128 + ((c & 7) << 4)) = make_uint4(0u, 0u, 0u, 0u);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (issuer) mbar_arrive(v_full(b));
      }
    }
    if (!ok) {                                                       // copies in flight land before the shared memory goes away
      const unsigned long long t0 = globaltimer_ns();
      while (globaltimer_ns() - t0 < 200000ull) {}
    }
  } else if (warp == kMmaWarp) {
    // ------------------------------------------------------------------ MMA issue
    const bool issuer = elect_one();
    const uint32_t id1 = umma_idesc_bf16(TK), id2 = umma_idesc_bf16(HD) | (1u << 16);      // bit 16: B is MN-major
    auto issue_s = [&](int x, int j) {                               // (the issuer only)
      const uint32_t qb = desc_lo_k(s0 + x * C::kQTile), kb = desc_lo_k(s0 + C::kOffK + (j % kStages) * C::kTile), d = tS(x) + (uint32_t)((j & 1) * TK);
#pragma unroll
      for (int ks = 0; ks < HD / 16; ++ks)
        umma_ss(d, qb + (ks >> 2) * (kQBlk / 16) + (ks & 3) * 2, kb + (ks >> 2) * (kBlk / 16) + (ks & 3) * 2, id1, ks > 0 ? 1u : 0u);
      umma_commit(s_full(x, j & 1));
    };
    auto k_wait = [&](int j) { return mbar_wait_warp(k_full(j % kStages), (uint32_t)((j / kStages) & 1), abort_flag); };
    bool ok = true;
    for (int j = 0; j < min(2, n) && ok; ++j) {                      // the first two key tiles' scores
      ok = k_wait(j);
      if (!ok) break;
      tc_fence_after();
      if (issuer) {
        if (j < nA) issue_s(0, j);
        if (j < nB) issue_s(1, j);
        umma_commit(k_free(j % kStages));
      }
    }
    for (int j = 0; j < n && ok; ++j) {
      const uint32_t vb = desc_lo_mn(s0 + C::kOffV + (j % kStages) * C::kTile);
      ok = mbar_wait_warp(v_full(j % kStages), (uint32_t)((j / kStages) & 1), abort_flag);
      if (ok && j + 2 < n) ok = k_wait(j + 2);
      for (int x = 0; x < 2 && ok; ++x) {
        const int nx = x ? nB : nA;
        if (j >= nx) continue;
        ok = mbar_wait_warp(p_ready(x, j & 1), (uint32_t)((j >> 1) & 1), abort_flag);
        if (!ok) break;
        tc_fence_after();
        const uint32_t d = tO(x), p = tS(x) + (uint32_t)((j & 1) * TK);
        if (issuer) {
#pragma unroll
          for (int ks = 0; ks < TK / 16; ++ks) umma_ts(d, p + ks * 16, vb + ks * 128, id2, ks > 0 ? 1u : (j > 0 ? 1u : 0u));
#pragma unroll
          for (int ks = 0; ks < TK / 16; ++ks) umma_ts(d, p + ks * 16 + 8, vb + ks * 128, id2, 1u);
          umma_commit(pv_done(x));
          if (j + 2 < nx) issue_s(x, j + 2);                         // over P(j), after the products that read it
          if (j + 1 == nx) umma_commit(o_done(x));
        }
      }
      if (ok && issuer) {
        umma_commit(v_free(j % kStages));
        if (j + 2 < n) umma_commit(k_free((j + 2) % kStages));
      }
    }
  } else {
    // ------------------------------------------------------------------ softmax of tile x: thread = query vector
    const int x = warp >> 2, row = (warp & 3) * 32 + lane, tok = row / group, g = row - tok * group;
    const int nx = x ? nB : nA, qpos = pos0 + x * tpt + tok;
    const bool real = tok < (x ? tokB : tokA) && row < tpt * group;
    const uint32_t lq = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t O = tO(x) + lq;
    const float sc = rsqrtf((float)HD) * 1.4426950408889634f;        // raw scores -> log2 units
    float m_ref = -INFINITY, l = 0.f;
    bool ok = true;
    auto wait = [&](uint32_t bar, uint32_t parity) {                 // lane 0 waits, the warp takes one decision
      if (lane == 0) ok = mbar_wait(bar, parity, abort_flag);
      ok = __shfl_sync(0xFFFFFFFFu, ok ? 1 : 0, 0) != 0;
      if (ok) tc_fence_after();
      return ok;
    };
    for (int j = 0; j < nx; ++j) {
      const uint32_t S = tS(x) + lq + (uint32_t)((j & 1) * TK);
      if (!wait(s_full(x, j & 1), (uint32_t)((j >> 1) & 1))) break;
      float sv[TK];
#pragma unroll
      for (int c = 0; c < TK; c += 16) tmem_ld16(S + (uint32_t)c, sv + c);
      tmem_ld_wait();
      const int last_ok = real ? qpos - j * TK : TK;                 // keys of this tile up to here count
      if (!real) {
#pragma unroll
        for (int c = 0; c < TK; ++c) sv[c] = 0.f;
      } else if (TK - 1 > last_ok) {
#pragma unroll
        for (int c = 0; c < TK; ++c)
          if (c > last_ok) sv[c] = -INFINITY;
      }
      float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
      for (int c = 0; c < TK; ++c) mx4[c & 3] = fmaxf(mx4[c & 3], sv[c]);
      const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
      // the reference maximum moves only when a row's maximum has passed it by more than 8 in log2 units
      const bool grow = (mx - m_ref) * sc > 8.f;                     // false while both are -inf
      if (j == 0) m_ref = mx;
      else if (__any_sync(0xFFFFFFFFu, grow)) {                      // (a first tile holds key 0: m_ref is finite for real rows)
        // O holds the previous tile's products (those of the tile before that were complete when S(j) was)
        if (!wait(pv_done(x), (uint32_t)((j - 1) & 1))) break;
        const float m_new = grow ? mx : m_ref;
        const float f = (m_new > -INFINITY && m_ref > -INFINITY) ? ex2((m_ref - m_new) * sc) : (m_new > -INFINITY ? 0.f : 1.f);
#pragma unroll 1
        for (int c = 0; c < HD; c += 16) {
          float o[16];
          tmem_ld16(O + (uint32_t)c, o);
          tmem_ld_wait();
          unsigned w[16];
#pragma unroll
          for (int e = 0; e < 16; ++e) w[e] = __float_as_uint(o[e] * f);
          tmem_st16u(O + (uint32_t)c, w);
        }
        l *= f;
        m_ref = m_new;
      }
      const float mneg = m_ref > -INFINITY ? -m_ref * sc : 0.f;
      float2 l2a = make_float2(0.f, 0.f), l2b = l2a;
      const float2 sc2 = make_float2(sc, sc), mneg2 = make_float2(mneg, mneg);
#pragma unroll
      for (int c = 0; c < TK; c += 16) {                             // weights over their own scores: per 16 keys 8 columns of hi, 8 of lo
        unsigned hi[8], lo[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float2 t = __ffma2_rn(make_float2(sv[c + 2 * e], sv[c + 2 * e + 1]), sc2, mneg2);
          const float2 p = make_float2(ex2(t.x), ex2(t.y));
          if (e & 1) l2b = __fadd2_rn(l2b, p);
          else l2a = __fadd2_rn(l2a, p);
          const __nv_bfloat162 h2 = __floats2bfloat162_rn(p.x, p.y);
          hi[e] = *reinterpret_cast<const unsigned *>(&h2);
          const float2 r = __ffma2_rn(make_float2(__uint_as_float(hi[e] << 16), __uint_as_float(hi[e] & 0xFFFF0000u)), make_float2(-1.f, -1.f), p);
          const __nv_bfloat162 lw = __floats2bfloat162_rn(r.x, r.y);
          lo[e] = *reinterpret_cast<const unsigned *>(&lw);
        }
        tmem_st8u(S + (uint32_t)c, hi);
        tmem_st8u(S + (uint32_t)(c + 8), lo);
      }
      l += (l2a.x + l2a.y) + (l2b.x + l2b.y);
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(p_ready(x, j & 1));
    }
    if (ok && nx > 0 && wait(o_done(x), 0u)) {
      const float inv = l > 0.f ? 1.f / l : 0.f;
      __nv_bfloat16 *dst = a.att + ((size_t)(row0 + x * tpt + tok) * a.nq + kvh * group + g) * HD;
#pragma unroll
      for (int c0 = 0; c0 < HD; c0 += 32) {
        float o[32];
        tmem_ld16(O + (uint32_t)c0, o);
        tmem_ld16(O + (uint32_t)(c0 + 16), o + 16);
        tmem_ld_wait();
#pragma unroll
        for (int c = 0; c < 32; c += 8) {
          unsigned w[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const __nv_bfloat162 p = __floats2bfloat162_rn(o[c + 2 * e] * inv, o[c + 2 * e + 1] * inv);
            w[e] = *reinterpret_cast<const unsigned *>(&p);
          }
          if (real) *reinterpret_cast<uint4 *>(dst + c0 + c) = make_uint4(w[0], w[1], w[2], w[3]);
        }
      }
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == kMmaWarp) tmem_dealloc(tmem, 512);
  if (threadIdx.x == 0 && *abort_flag) atomicExch(a.status, 1);
}

template <int HD>
int launch_t(const PromptAttnArgs &a, cudaStream_t s) {
  static std::atomic<u64> limits{0};
  const int limit = hsd_smem_limit((const void *)prompt_attn_kernel<HD>, Cfg<HD>::kSmem, limits);
  if (limit) return limit;
  HSD_CUDA_OK(hsd_launch(prompt_attn_kernel<HD>, a.n_items * a.nkv, kThreads, Cfg<HD>::kSmem, s, 0, a.chained, a));
  hsd_count_launches(1);
  return hsd_launch_status();
}

}  // namespace

int prompt_attn_map(CUtensorMap *map, const void *pool, long long rows, int hd) { return tc_make_map(map, pool, rows, hd, TK); }

bool prompt_attn_pages(const int *pages, int n_pages, int page) {
  for (int i = 1; i < n_pages; ++i)
    if (i * page % TK != 0 && pages[i] != pages[i - 1] + 1) return false;
  return true;
}

int launch_prompt_attention(const PromptAttnArgs &a, cudaStream_t s) {
  if (a.n_items < 1 || a.nq % a.nkv != 0 || a.nq / a.nkv > 8 || a.page_shift < 4) return HSD_E_UNSUPPORTED;
  if (a.hd == 128) return launch_t<128>(a, s);
  if (a.hd == 64) return launch_t<64>(a, s);
  return HSD_E_UNSUPPORTED;
}

}  // namespace hsd
