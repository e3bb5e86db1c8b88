// Prompt attention on tcgen05 with scores, weights and outputs in tensor memory.
//
// One CTA = one KV head and up to 2 x 128 query vectors (two tiles A and B of consecutive tokens x the heads of the
// KV group), over all keys up to the last of them, in tiles of 128 keys.  Per key tile and query tile
//   S[128 x 128]  = Q K^T                      both operands in shared memory
//   P             = exp2((S - m_ref) scale log2 e), thread = query vector, split into bf16 hi + lo halves that
//                   overwrite S (the P V product keeps about 16 bits of P, as in the decode passes' attention)
//   O[128 x hd]  += P_hi V + P_lo V            A operand from tensor memory, V as it lies in the cache (MN-major)
// m_ref moves only when a row maximum passes it by a factor 256; then O is rescaled.  Two query tiles share every K
// and V tile and alternate: the tensor pipe works on one while the softmax warps of the other work on theirs.
// Bound by the tensor pipe (three products per tile pair instead of two because of the hi / lo split: 3 x 512 cycles
// of hd = 128 per 128 x 128 tile; the exponentials take 1024).  A tile's S is complete only after the same tile's previous P V
// (issued before it), so O may be rescaled and P overwritten without further waits.
// 320 threads: warps 0-3 / 4-7 = softmax of tile A / B, warp 8 = K / V loader (TMA, 16 keys of one page per copy),
// warp 9 = MMA issue (one lane).  Items come longest first.  Every wait is bounded.
#include <algorithm>
#include "attn_prompt.cuh"
#include "gemm_tc.cuh"
#include "tc_ptx.cuh"

namespace hsd {
namespace {

using namespace ptx;

constexpr int kThreads = 320;
constexpr int TK = 128;                                  // keys per tile
constexpr int kBlk = 128 * 128;                          // [128 rows][64 bf16] block, 128-byte swizzle
constexpr int kStages = 2;

template <int HD> struct Cfg {
  static constexpr int NB = HD / 64;                     // 64-column blocks
  static constexpr int kTile = NB * kBlk;
  static constexpr int kOffK = 2 * kTile, kOffV = kOffK + kStages * kTile, kOffBar = kOffV + kStages * kTile;
  static constexpr int kSmem = kOffBar + 256 + 1024;
};

__device__ __forceinline__ uint64_t desc_mn(uint32_t smem_addr) {      // MN-major, 128-byte swizzle, 64-column blocks kBlk apart
  uint64_t d = (uint64_t)((smem_addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)(kBlk >> 4) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
__device__ __forceinline__ void umma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void tmem_st16u(uint32_t taddr, const unsigned *r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
               "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

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
  auto k_free = [&](int b) { return b0 + 8u * (2 + b); };
  auto v_full = [&](int b) { return b0 + 8u * (4 + b); };
  auto v_free = [&](int b) { return b0 + 8u * (6 + b); };
  auto s_full = [&](int x) { return b0 + 8u * (8 + x); };
  auto p_ready = [&](int x) { return b0 + 8u * (10 + x); };
  auto o_done = [&](int x) { return b0 + 8u * (12 + x); };
  const uint32_t v_land = b0 + 8u * 14;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kvh = blockIdx.x % a.nkv;
  const int4 it = a.items[blockIdx.x / a.nkv];
  const int row0 = it.x, ntok = it.y, seq = it.z, pos0 = it.w;
  const int group = a.nq / a.nkv, tpt = 128 / group;                 // tokens per query tile
  const int tokA = min(ntok, tpt), tokB = ntok - tokA;
  const int kv_len = pos0 + ntok;
  const int nA = (pos0 + tokA + TK - 1) / TK, nB = tokB > 0 ? (kv_len + TK - 1) / TK : 0;
  const int n = max(nA, nB);

  if (threadIdx.x == 0) {
    for (int b = 0; b < 2; ++b) {
      mbar_init(k_full(b), 1); mbar_init(k_free(b), 1); mbar_init(v_full(b), 1); mbar_init(v_free(b), 1);
      mbar_init(s_full(b), 1); mbar_init(p_ready(b), 4); mbar_init(o_done(b), 1);
    }
    mbar_init(v_land, 1);
    sh_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 9) tmem_alloc(smem_u32(&tmem_slot), 512);
  if (warp < 8) {
    // Q: thread = query vector; K-major, 128-byte swizzle; vectors past the tile's tokens are zero
    const int x = warp >> 2, row = (warp & 3) * 32 + lane, tok = row / group, g = row - tok * group;
    const bool real = tok < (x ? tokB : tokA) && row < tpt * group;
    const uint4 *src = reinterpret_cast<const uint4 *>(a.q + ((size_t)(row0 + x * tpt + tok) * a.nq + kvh * group + g) * HD);
    uint4 v[HD / 8];
#pragma unroll
    for (int c = 0; c < HD / 8; ++c) v[c] = real ? __ldcg(src + c) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int c = 0; c < HD / 8; ++c)
      *reinterpret_cast<uint4 *>(smem + x * C::kTile + (c >> 3) * kBlk + (row >> 3) * 1024 + (row & 7) * 128 + (((c & 7) ^ (row & 7)) << 4)) = v[c];
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  auto tS = [&](int x) { return tmem + (uint32_t)(x * 128); };
  auto tO = [&](int x) { return tmem + 256u + (uint32_t)(x * HD); };

  if (warp == 8) {
    // ------------------------------------------------------------------ loader
    const int *pt = a.page_table + (size_t)seq * a.pages_per_seq;
    constexpr int kCopies = 8 * C::NB;                               // per operand and tile: (16-key group, column block)
    const int grp = lane & 7, blk = lane >> 3;
    const int last_group = (kv_len - 1) >> 4;
    bool ok = true;
    for (int j = 0; j < n && ok; ++j) {
      const int b = j & 1;
      const uint32_t ph = (uint32_t)((j >> 1) & 1);
      // a group past the last key has no page: the last group again (its scores are masked, its V rows zeroed below)
      const int key = min(j * 8 + grp, last_group) * 16;
      int row = 0;
      if (lane < kCopies) {
        const int pg = pt[key >> a.page_shift];
        row = ((kvh * a.n_pages + pg) << a.page_shift) + (key & ((1 << a.page_shift) - 1));
      }
      const uint32_t off = (uint32_t)(blk * kBlk + grp * 2048);
      if (lane == 0) {
        ok = mbar_wait(k_free(b), ph ^ 1u, abort_flag);
        if (ok) mbar_expect_tx(k_full(b), C::kTile);
      }
      ok = __shfl_sync(0xFFFFFFFFu, ok ? 1 : 0, 0) != 0;
      if (!ok) break;
      if (lane < kCopies) tma_load_2d(s0 + C::kOffK + b * C::kTile + off, &a.k, blk * 64, row, k_full(b));
      const bool tail = (j + 1) * TK > kv_len;
      if (lane == 0) {
        ok = mbar_wait(v_free(b), ph ^ 1u, abort_flag);
        if (ok) mbar_expect_tx(tail ? v_land : v_full(b), C::kTile);
      }
      ok = __shfl_sync(0xFFFFFFFFu, ok ? 1 : 0, 0) != 0;
      if (!ok) break;
      if (lane < kCopies) tma_load_2d(s0 + C::kOffV + b * C::kTile + off, &a.v, blk * 64, row, tail ? v_land : v_full(b));
      if (tail) {                                                    // the last tile: V rows past the last key must be finite (P is 0 there)
        if (lane == 0) ok = mbar_wait(v_land, 0u, abort_flag);
        ok = __shfl_sync(0xFFFFFFFFu, ok ? 1 : 0, 0) != 0;
        if (!ok) break;
        const int r0 = kv_len - j * TK;
        for (int i = r0 * 8 * C::NB + lane; i < TK * 8 * C::NB; i += 32) {
          const int r = i / (8 * C::NB), c = i % (8 * C::NB);        // whole rows: the swizzle permutes within a row
          *reinterpret_cast<uint4 *>(smem + C::kOffV + b * C::kTile + (c >> 3) * kBlk + r * 128 + ((c & 7) << 4)) = make_uint4(0u, 0u, 0u, 0u);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(v_full(b));
      }
    }
    if (!ok) {                                                       // copies in flight land before the shared memory goes away
      const unsigned long long t0 = globaltimer_ns();
      while (globaltimer_ns() - t0 < 200000ull) {}
    }
  } else if (warp == 9) {
    // ------------------------------------------------------------------ MMA issue
    if (lane == 0) {
      const uint32_t id1 = umma_idesc_bf16(TK), id2 = umma_idesc_bf16(HD) | (1u << 16);      // bit 16: B is MN-major
      auto issue_s = [&](int x, int j) {
        const uint32_t kb = s0 + C::kOffK + (j & 1) * C::kTile, qb = s0 + x * C::kTile;
#pragma unroll
        for (int ks = 0; ks < HD / 16; ++ks)
          umma_bf16(tS(x), umma_desc(qb + (ks >> 2) * kBlk + (ks & 3) * 32), umma_desc(kb + (ks >> 2) * kBlk + (ks & 3) * 32), id1, ks > 0 ? 1u : 0u);
        umma_commit(s_full(x));
      };
      bool ok = mbar_wait(k_full(0), 0u, abort_flag);
      if (ok) {
        tc_fence_after();
        issue_s(0, 0);
        if (nB > 0) issue_s(1, 0);
        umma_commit(k_free(0));
      }
      for (int j = 0; j < n && ok; ++j) {
        const uint32_t vb = s0 + C::kOffV + (j & 1) * C::kTile;
        ok = mbar_wait(v_full(j & 1), (uint32_t)((j >> 1) & 1), abort_flag);
        if (ok && j + 1 < n) ok = mbar_wait(k_full((j + 1) & 1), (uint32_t)(((j + 1) >> 1) & 1), abort_flag);
        for (int x = 0; x < 2 && ok; ++x) {
          const int nx = x ? nB : nA;
          if (j >= nx) continue;
          ok = mbar_wait(p_ready(x), (uint32_t)(j & 1), abort_flag);
          if (!ok) break;
          tc_fence_after();
#pragma unroll
          for (int half = 0; half < 2; ++half)
#pragma unroll
            for (int ks = 0; ks < TK / 16; ++ks)
              umma_bf16_ts(tO(x), tS(x) + (uint32_t)((ks >> 2) * 64 + half * 32 + (ks & 3) * 8), desc_mn(vb + ks * 2048), id2, (j > 0 || half > 0 || ks > 0) ? 1u : 0u);
          if (j + 1 < nx) issue_s(x, j + 1);
          else umma_commit(o_done(x));
        }
        if (ok) {
          umma_commit(v_free(j & 1));
          if (j + 1 < n) umma_commit(k_free((j + 1) & 1));
        }
      }
    }
  } else {
    // ------------------------------------------------------------------ softmax of tile x: thread = query vector
    const int x = warp >> 2, row = (warp & 3) * 32 + lane, tok = row / group, g = row - tok * group;
    const int nx = x ? nB : nA, qpos = pos0 + x * tpt + tok;
    const bool real = tok < (x ? tokB : tokA) && row < tpt * group;
    const uint32_t lq = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t S = tS(x) + lq, O = tO(x) + lq;
    const float sc = rsqrtf((float)HD) * 1.4426950408889634f;        // raw scores -> log2 units
    float m_ref = -INFINITY, l = 0.f;
    bool ok = true;
    for (int j = 0; j < nx; ++j) {
      if (lane == 0) ok = mbar_wait(s_full(x), (uint32_t)(j & 1), abort_flag);
      ok = __shfl_sync(0xFFFFFFFFu, ok ? 1 : 0, 0) != 0;
      if (!ok) break;
      tc_fence_after();
      // The scores go through registers 64 keys at a time (the whole row would not fit beside the conversion): keys
      // 64..127 last in the maximum pass and first in the conversion, keys 0..63 are read twice.
      const int last_ok = real ? qpos - j * TK : TK;                 // keys of this tile up to here count
      float sv[64];
      auto load_half = [&](int h) {
#pragma unroll
        for (int c = 0; c < 64; c += 16) tmem_ld16(S + (uint32_t)(h * 64 + c), sv + c);
        tmem_ld_wait();
        if (!real) {
#pragma unroll
          for (int c = 0; c < 64; ++c) sv[c] = 0.f;
        } else if (h * 64 + 63 > last_ok) {
#pragma unroll
          for (int c = 0; c < 64; ++c)
            if (h * 64 + c > last_ok) sv[c] = -INFINITY;
        }
      };
      float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        load_half(h);
#pragma unroll
        for (int c = 0; c < 64; ++c) mx4[c & 3] = fmaxf(mx4[c & 3], sv[c]);
      }
      const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
      // the reference maximum moves only when a row's maximum has passed it by more than 8 in log2 units
      const bool grow = (mx - m_ref) * sc > 8.f;                     // false while both are -inf
      if (j == 0) m_ref = mx;
      else if (__any_sync(0xFFFFFFFFu, grow)) {                      // (a first tile holds key 0: m_ref is finite for real rows)
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
      float l4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int h = 1; h >= 0; --h) {                                 // weights of keys 64 h .. over their own scores: hi in 32 columns, lo in the next 32
        if (h == 0) load_half(0);
#pragma unroll
        for (int c = 0; c < 64; c += 32) {
          unsigned hi[16], lo[16];
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            const float p0 = ex2(fmaf(sv[c + 2 * e], sc, mneg)), p1 = ex2(fmaf(sv[c + 2 * e + 1], sc, mneg));
            l4[e & 3] += p0 + p1;
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(p0, p1);
            hi[e] = *reinterpret_cast<const unsigned *>(&h2);
            const __nv_bfloat162 l2 = __floats2bfloat162_rn(p0 - __uint_as_float(hi[e] << 16), p1 - __uint_as_float(hi[e] & 0xFFFF0000u));
            lo[e] = *reinterpret_cast<const unsigned *>(&l2);
          }
          tmem_st16u(S + (uint32_t)(h * 64 + c / 2), hi);
          tmem_st16u(S + (uint32_t)(h * 64 + 32 + c / 2), lo);
        }
      }
      l += (l4[0] + l4[1]) + (l4[2] + l4[3]);
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(p_ready(x));
    }
    if (ok && nx > 0) {
      if (lane == 0) ok = mbar_wait(o_done(x), 0u, abort_flag);
      ok = __shfl_sync(0xFFFFFFFFu, ok ? 1 : 0, 0) != 0;
      if (ok) {
        tc_fence_after();
        const float inv = l > 0.f ? 1.f / l : 0.f;
        __nv_bfloat16 *dst = a.att + ((size_t)(row0 + x * tpt + tok) * a.nq + kvh * group + g) * HD;
#pragma unroll 1
        for (int c = 0; c < HD; c += 16) {
          float o[16];
          tmem_ld16(O + (uint32_t)c, o);
          tmem_ld_wait();
          unsigned w[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const __nv_bfloat162 p = __floats2bfloat162_rn(o[2 * e] * inv, o[2 * e + 1] * inv);
            w[e] = *reinterpret_cast<const unsigned *>(&p);
          }
          if (real) {
            reinterpret_cast<uint4 *>(dst + c)[0] = make_uint4(w[0], w[1], w[2], w[3]);
            reinterpret_cast<uint4 *>(dst + c)[1] = make_uint4(w[4], w[5], w[6], w[7]);
          }
        }
      }
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 9) tmem_dealloc(tmem, 512);
  if (threadIdx.x == 0 && *abort_flag) atomicExch(a.status, 1);
}

template <int HD>
int launch_t(const PromptAttnArgs &a, cudaStream_t s) {
  static bool attr_set = false;
  if (!attr_set) {
    HSD_CUDA_OK(cudaFuncSetAttribute(prompt_attn_kernel<HD>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<HD>::kSmem));
    attr_set = true;
  }
  prompt_attn_kernel<HD><<<a.n_items * a.nkv, kThreads, Cfg<HD>::kSmem, s>>>(a);
  hsd_count_launches(1);
  return hsd_launch_status();
}

}  // namespace

int prompt_attn_map(CUtensorMap *map, const void *pool, long long rows, int hd) { return tc_make_map(map, pool, rows, hd, kPromptBoxRows); }

int launch_prompt_attention(const PromptAttnArgs &a, cudaStream_t s) {
  if (a.n_items < 1 || a.nq % a.nkv != 0 || a.nq / a.nkv > 8 || a.page_shift < 4) return HSD_E_UNSUPPORTED;
  if (a.hd == 128) return launch_t<128>(a, s);
  if (a.hd == 64) return launch_t<64>(a, s);
  return HSD_E_UNSUPPORTED;
}

}  // namespace hsd
