// Prompt-chunk GEMM on CTA pairs (tcgen05 cta_group::2).
//
// Bound by the tensor pipe: a 256 x 256 tile per CTA pair takes about 512 cycles per 64-wide k-block, in which each CTA
// takes 32 KiB of operands from L2 and reads them from shared memory once (its 128 A rows and its 128 of the 256 B
// rows); a 128 x 256 tile per single CTA would take half as much again of both.  One CTA of the pair issues the MMAs;
// both load their own operands and signal the issuing CTA's barrier.  Warp 0 = TMA producer, warp 1 = TMEM owner and
// (leader) MMA issuer, then the epilogue; six stages; two 256-column accumulators (all of tensor memory), so a tile's epilogue
// runs under the next tile's MMAs.  Tiles are dealt round-robin with the token tile fastest: the pairs that work at the same
// time share weight rows, so a weight tile comes from HBM once.  Every wait is bounded, and no waiter can be passed by (a
// parity wait sees a completion only until the next one): full[s] has its next loads behind empty[s], which the issuer's commit
// completes in both CTAs; empty[s] its next MMAs behind the loads of both producers; acc_full its next MMAs behind acc_empty,
// which every epilogue warp of the pair completes; acc_empty its next epilogue behind the MMAs.
// The tensor core's fp32 accumulation loses about as much as its chain is long.  Products for the fp32 residual stream cut K
// into chains (chain_blocks): the accumulators take turns, eight epilogue warps add each chain's sum to their registers under
// the next chain's MMAs and put the whole sum back into tensor memory for the finish (a finish straight from the 128
// registers: 1.5 % of a prompt pass slower; reads of 16 columns instead of 32: O 90 us instead of 86).
//
// Measured on the 8B shape, 2304 rows: gate / up 317 us (1.7 PFLOP/s), down 199 us, O 86 us, QKV 87 us (the last three lose a
// part of their second round of 74 tiles).  A 1023-row prompt pass: 37.3 ms in 128-row chunks of the one-launch forward, 13.0 ms
// this way; eight such prompts 300 -> 99 ms.
#include <algorithm>
#include "gemm_big.cuh"
#include "tc_ptx.cuh"

namespace hsd {
namespace {

using namespace ptx;

constexpr int kBM = 256, kBN = 256, kBK = 64;
constexpr int kStages = 6;
constexpr int kABytes = 128 * kBK * 2, kBBytes = 128 * kBK * 2;      // per CTA and stage
constexpr int kStageBytes = kABytes + kBBytes;
constexpr int kSmemBytes = kStages * kStageBytes + 1024 + 1024;

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Tile load whose completion is counted on a barrier of either CTA of the pair.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar) {
  asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
               ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar) : "memory");
}
__device__ __forceinline__ void umma_bf16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(acc) : "memory");
}
// Arrives on the barrier at this offset in both CTAs once the MMAs issued so far are complete.
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
  const uint16_t mask = 3;
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"(mask) : "memory");
}
__device__ __forceinline__ void remote_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}

// 128 columns of an accumulator row per half (half 0: the first CTA's weight rows, half 1: the second CTA's).
struct Half { int seg, n0; };                       // segment and first column within it; seg < 0: past the end
template <int MODE> __device__ __forceinline__ Half half_of(const BigGemmArgs &a, int nt, int h) {
  Half r;
  if (MODE == BIG_SWIGLU) { r.seg = h; r.n0 = nt * 128; return r; }
  int c = nt * kBN + h * 128 + (MODE == BIG_QKV ? a.skip_cols : 0);
  r.seg = 0;
  if (MODE == BIG_QKV) {
#pragma unroll
    for (int s = 0; s < 2; ++s)
      if (r.seg == s && c >= a.seg_n[s]) { c -= a.seg_n[s]; r.seg = s + 1; }
  }
  r.n0 = c;
  return r;
}

__device__ __forceinline__ void store_bf16x16(__nv_bfloat16 *dst, const float *v) {
  unsigned w[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(v[2 * e], v[2 * e + 1]);
    w[e] = *reinterpret_cast<const unsigned *>(&p);
  }
  reinterpret_cast<uint4 *>(dst)[0] = make_uint4(w[0], w[1], w[2], w[3]);
  reinterpret_cast<uint4 *>(dst)[1] = make_uint4(w[4], w[5], w[6], w[7]);
}

// Threads: a TMA and an MMA warp, four epilogue warps, or eight where the epilogue sums chains (a thread then holds half a row).
template <int MODE> constexpr int threads_of() { return MODE == BIG_ADD_F32 ? 320 : 192; }

template <int MODE, int HD>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(threads_of<MODE>(), 1)
gemm_big_kernel(const __grid_constant__ BigGemmArgs args, int n_tiles, int m_tiles, int KB, int chain) {
  constexpr bool CHAINS = MODE == BIG_ADD_F32;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kStages * kStageBytes);
  // full[STAGES] (used in the leader) | empty[STAGES] | acc_full[2] | acc_empty[2] (used in the leader)
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * kStages + 4);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
  volatile int *wait_ok = reinterpret_cast<volatile int *>(tmem_slot + 2);        // [2], alternating per tile
  const uint32_t bar0 = smem_u32(bars), s0 = smem_u32(smem);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (kStages + s); };
  auto accf_bar = [&](int b) { return bar0 + 8u * (2 * kStages + b); };
  auto acce_bar = [&](int b) { return bar0 + 8u * (2 * kStages + 2 + b); };
  const int warp = warp_index(), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
  chain_next();

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(accf_bar(b), 1); mbar_init(acce_bar(b), CHAINS ? 16 : 8); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512u));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::);
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();                                    // both CTAs' barriers exist, both hold their tensor memory
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer (one lane of each CTA issues)
    const bool issuer = elect_one();
    int s = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int t = pair; t < n_tiles && ok; t += pairs) {
      const int mt = t % m_tiles, nt = t / m_tiles;
      const Half hf = half_of<MODE>(args, nt, (int)rank);
      const int arow = mt * kBM + (int)rank * 128;
      auto load_w = [&](int kb, int slot) {
        const uint32_t dst = s0 + (uint32_t)(slot * kStageBytes) + kABytes, bar = map_to_rank(full_bar(slot), 0);
        if (rank == 0) mbar_expect_tx(full_bar(slot), 2 * kStageBytes);
        tma_load_2d_pair(dst, &args.w[hf.seg], kb * kBK, hf.n0, bar);
        tma_load_2d_pair(dst + kBBytes / 2, &args.w[hf.seg], kb * kBK, hf.n0 + 64, bar);
      };
      auto load_a = [&](int kb, int slot) {
        tma_load_2d_pair(s0 + (uint32_t)(slot * kStageBytes), &args.a, kb * kBK, arow, map_to_rank(full_bar(slot), 0));
      };
      int kb = 0;
      if (t == pair) {                               // the ring's first weights before the wait for the activations
        kb = min(kStages, KB);
        if (issuer)
          for (int i = 0; i < kb; ++i) load_w(i, i);
        chain_wait();
        if (issuer)
          for (int i = 0; i < kb; ++i) load_a(i, i);
        s = kb;
        if (s == kStages) { s = 0; ph ^= 1u; }
      }
      for (; kb < KB; ++kb) {
        if (!mbar_wait_warp(empty_bar(s), ph ^ 1u, abort_flag)) { ok = false; break; }
        if (issuer) { load_a(kb, s); load_w(kb, s); }
        if (++s == kStages) { s = 0; ph ^= 1u; }
      }
    }
    if (!ok) {                                       // copies still in flight must land before the shared memory goes away
      const unsigned long long t0 = globaltimer_ns();
      while (globaltimer_ns() - t0 < 200000ull) {}
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (one lane of the leader issues)
    if (rank == 0) {
      const bool issuer = elect_one();
      chain_wait();                                  // (the limit of the waits below is for this kernel's own work)
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kBN >> 3) << 17) | ((uint32_t)(kBM >> 4) << 24);
      const uint64_t da0 = umma_desc(s0);
      int s = 0, ci = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int t = pair; t < n_tiles && ok; t += pairs) {
        for (int k0 = 0; k0 < KB && ok; k0 += chain, ++ci) {
          const int ab = ci & 1, k1 = min(KB, k0 + chain);
          ok = mbar_wait_warp(acce_bar(ab), (uint32_t)((ci >> 1) & 1) ^ 1u, abort_flag);
          if (!ok) break;
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + (uint32_t)(ab * kBN);
          uint32_t acc = 0u;
          for (int kb = k0; kb < k1; ++kb) {
            if (!mbar_wait_warp(full_bar(s), ph, abort_flag)) { ok = false; break; }
            tc_fence_after();
            const uint64_t da = da0 + (uint64_t)(s * (kStageBytes >> 4)), db = da + (uint64_t)(kABytes >> 4);
            if (issuer) {
              umma_bf16_pair(d_tmem, da, db, idesc, acc);
#pragma unroll
              for (int k = 1; k < kBK / 16; ++k) umma_bf16_pair(d_tmem, da + (uint64_t)(k * 2), db + (uint64_t)(k * 2), idesc, 1u);
              umma_commit_pair(empty_bar(s));
            }
            acc = 1u;
            if (++s == kStages) { s = 0; ph ^= 1u; }
          }
          if (ok && issuer) umma_commit_pair(accf_bar(ab));
        }
      }
    }
  } else if constexpr (CHAINS) {
    // ------------------------------------------------------------------ epilogue (warps 2..9): thread = token row and half
    // of the tile's columns
    const int q = warp & 3, hw = (warp - 2) >> 2;                       // TMEM lane quarter, column half
    chain_wait();
    int ci = 0;
    bool ok = true;
    for (int t = pair; t < n_tiles; t += pairs) {
      uint32_t tb = 0, acce = 0;
      float acc[128];                                                   // sum of the tile's chains so far
#pragma unroll
      for (int i = 0; i < 128; ++i) acc[i] = 0.f;
      for (int k0 = 0; k0 < KB; k0 += chain, ++ci) {
        const int ab = ci & 1;
        if (lane == 0) ok = mbar_wait(accf_bar(ab), (uint32_t)((ci >> 1) & 1), abort_flag);
        ok = __shfl_sync(0xFFFFFFFFu, ok ? 1 : 0, 0) != 0;
        if (!ok) break;
        tc_fence_after();
        tb = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(ab * kBN + hw * 128);
        acce = map_to_rank(acce_bar(ab), 0);
        if (chain >= KB) continue;                                      // one chain: the finish reads it where it lies
#pragma unroll
        for (int c = 0; c < 128; c += 32) {
          float v[32];
          tmem_ld32(tb + c, v);
          tmem_ld_wait();
#pragma unroll
          for (int e = 0; e < 32; ++e) acc[c + e] += v[e];
        }
        if (k0 + chain < KB) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) remote_arrive(acce);
        } else {                                                        // the finish reads the sum where the last chain lay
#pragma unroll
          for (int c = 0; c < 128; c += 16) tmem_st16u(tb + c, reinterpret_cast<const unsigned *>(acc + c));
          tmem_st_wait();
        }
      }
      if (!ok) break;
      const int mt = t % m_tiles, nt = t / m_tiles;
      const int r = mt * kBM + (int)rank * 128 + q * 32 + lane;
      const bool on = r < args.R;
      float *row = args.out_f32 + (size_t)r * args.ldo + nt * kBN + hw * 128;
#pragma unroll 1
      for (int c = 0; c < 128; c += 32) {
        float v[32];
        tmem_ld32(tb + c, v);
        float4 old[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) old[e] = on ? __ldcg(reinterpret_cast<const float4 *>(row + c) + e) : make_float4(0.f, 0.f, 0.f, 0.f);
        tmem_ld_wait();
        if (on) {
#pragma unroll
          for (int e = 0; e < 8; ++e)
            __stcg(reinterpret_cast<float4 *>(row + c) + e, make_float4(old[e].x + v[4 * e], old[e].y + v[4 * e + 1],
                                                                        old[e].z + v[4 * e + 2], old[e].w + v[4 * e + 3]));
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) remote_arrive(acce);
    }
  } else {
    // ------------------------------------------------------------------ epilogue (warps 2..5): thread = token row
    const int q = warp & 3, et = threadIdx.x - 64;
    chain_wait();
    int ti = 0;
    for (int t = pair; t < n_tiles; t += pairs, ++ti) {
      const int ab = ti & 1;
      if (et == 0) wait_ok[ab] = mbar_wait(accf_bar(ab), (uint32_t)((ti >> 1) & 1), abort_flag) ? 1 : 0;
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (!wait_ok[ab]) break;
      tc_fence_after();
      const int mt = t % m_tiles, nt = t / m_tiles;
      const int r = mt * kBM + (int)rank * 128 + q * 32 + lane;
      const bool on = r < args.R;
      const uint32_t tb = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(ab * kBN);
      if (MODE == BIG_SWIGLU) {
        __nv_bfloat16 *row = args.out_bf16 + (size_t)r * args.ldo + nt * 128;
#pragma unroll 1
        for (int c = 0; c < 128; c += 16) {
          float g[16], u[16];
          tmem_ld16(tb + c, g);
          tmem_ld16(tb + 128 + c, u);
          tmem_ld_wait();
#pragma unroll
          for (int e = 0; e < 16; ++e) g[e] = silu_mul(g[e], u[e]);
          if (on && nt * 128 + c < args.seg_n[0]) store_bf16x16(row + c, g);          // ff is a multiple of 64
        }
      } else if (MODE == BIG_LOGITS) {
        const long long dr = on ? (args.dst ? args.dst[r] : (long long)r) : 0;
        __nv_bfloat16 *row = args.out_bf16 + (size_t)dr * args.ldo + nt * kBN;
        const int left = args.seg_n[0] - nt * kBN;
        const bool vec = (args.ldo & 7) == 0 && ((uintptr_t)args.out_bf16 & 15) == 0;     // (the caller's buffer: any element's address)
#pragma unroll 1
        for (int c = 0; c < kBN; c += 16) {
          float v[16];
          tmem_ld16(tb + c, v);
          tmem_ld_wait();
          if (!on) continue;
          if (vec && c + 16 <= left) store_bf16x16(row + c, v);
          else {
#pragma unroll
            for (int e = 0; e < 16; ++e)
              if (c + e < left) row[c + e] = __float2bfloat16_rn(v[e]);
          }
        }
      } else {
        const int seq = on ? args.row_seq[r] : 0, pos = on ? args.row_pos[r] : 0;
        const int pg = on ? args.page_table[(size_t)seq * args.pages_per_seq + pos / args.page] : 0, in_page = pos % args.page;
        constexpr int HALF = HD / 2;
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
          const Half hf = half_of<MODE>(args, nt, h);
          if (hf.seg == 2 && hf.n0 >= args.seg_n[2]) continue;                         // past the last column
#pragma unroll 1
          for (int hd0 = 0; hd0 < 128; hd0 += HD) {                                    // the heads of this half
            const int head = (hf.n0 + hd0) / HD;
            __nv_bfloat16 *dst;
            if (hf.seg == 0) dst = args.q + ((size_t)r * args.nq + head) * HD;
            else dst = (hf.seg == 1 ? args.k_pool : args.v_pool) + (((size_t)head * args.n_pages + pg) * args.page + in_page) * HD;
#pragma unroll 1
            for (int c = 0; c < HALF; c += 16) {
              float lo[16], hi[16];
              tmem_ld16(tb + h * 128 + hd0 + c, lo);
              tmem_ld16(tb + h * 128 + hd0 + HALF + c, hi);
              float cs[16], sn[16];
              if (on && hf.seg < 2) {
                const float4 *ct = reinterpret_cast<const float4 *>(args.cos_tab + (size_t)pos * HALF + c);
                const float4 *st = reinterpret_cast<const float4 *>(args.sin_tab + (size_t)pos * HALF + c);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                  const float4 cv = __ldg(ct + e), sv = __ldg(st + e);
                  cs[4 * e] = cv.x; cs[4 * e + 1] = cv.y; cs[4 * e + 2] = cv.z; cs[4 * e + 3] = cv.w;
                  sn[4 * e] = sv.x; sn[4 * e + 1] = sv.y; sn[4 * e + 2] = sv.z; sn[4 * e + 3] = sv.w;
                }
              } else {
#pragma unroll
                for (int e = 0; e < 16; ++e) { cs[e] = 1.f; sn[e] = 0.f; }
              }
              tmem_ld_wait();
#pragma unroll
              for (int e = 0; e < 16; ++e) {
                const float x = lo[e], y = hi[e];
                if (hf.seg < 2) { lo[e] = x * cs[e] - y * sn[e]; hi[e] = y * cs[e] + x * sn[e]; }
              }
              if (on) { store_bf16x16(dst + c, lo); store_bf16x16(dst + HALF + c, hi); }
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) remote_arrive(map_to_rank(acce_bar(ab), 0));
    }
  }
  // ------------------------------------------------------------------ teardown
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  cluster_sync();                                    // no signal may arrive in a CTA that has left
  tc_fence_after();
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u));
  if (threadIdx.x == 0 && *abort_flag) atomicExch(args.status, 1);
}

// k-blocks of a chain.  Products that go to the fp32 residual stream: as many as a CTA of the one-launch forward (passes of
// up to 128 rows) sums in a row for the same product: a quarter of K while four CTAs to a 128-row tile fit the SMs, and at
// least kMinChain (a shorter chain is over before a tile's finish has given the other accumulator back).  Products whose result
// is rounded to bf16 at once: all of K (4e-6 at 4096 columns against the rounding's 2e-3).  A chain's sum holds the MMAs up
// while it is read; 2304 rows of the 8B shape in one chain / four: O 72 / 86 us, down 190 / 199; chains in QKV and gate / up
// too: 90 / 99 and 322 / 349.
constexpr int kMinChain = 16;
int chain_blocks(const BigGemmArgs &a, int KB, int sm_count) {
  if (a.mode != BIG_ADD_F32) return KB;
  const int tiles = ceil_div(a.seg_n[0], 128);
  const int blocks = tiles * 2 <= sm_count ? ceil_div(KB, std::min(4, sm_count / tiles))
                                           : (int)std::min<long long>(KB, ((long long)tiles * KB + sm_count - 1) / sm_count);
  return std::min(KB, std::max(blocks, kMinChain));
}

template <int MODE, int HD>
int launch_t(const BigGemmArgs &a, int n_tiles, int m_tiles, int sm_count, cudaStream_t s) {
  static std::atomic<u64> limits{0};
  const int limit = hsd_smem_limit((const void *)gemm_big_kernel<MODE, HD>, kSmemBytes, limits);
  if (limit) return limit;
  const int pairs = std::min(sm_count / 2, n_tiles), KB = a.K / kBK;
  HSD_CUDA_OK(hsd_launch(gemm_big_kernel<MODE, HD>, 2 * pairs, threads_of<MODE>(), kSmemBytes, s, 0, a.chained, a, n_tiles, m_tiles, KB, chain_blocks(a, KB, sm_count)));
  hsd_count_launches(1);
  return hsd_launch_status();
}

}  // namespace

int launch_gemm_big(const BigGemmArgs &a, int sm_count, cudaStream_t s) {
  if (a.R < 1 || a.K < kBK || a.K % kBK != 0) return HSD_E_UNSUPPORTED;
  const int m_tiles = ceil_div(a.R, kBM);
  switch (a.mode) {
    case BIG_QKV: {
      if (a.seg_n[0] % 128 || a.seg_n[1] % 128 || a.seg_n[2] % 128 || a.skip_cols % kBN) return HSD_E_UNSUPPORTED;
      const int n_tiles = ceil_div(a.seg_n[0] + a.seg_n[1] + a.seg_n[2] - a.skip_cols, kBN);
      if (a.hd == 128) return launch_t<BIG_QKV, 128>(a, n_tiles * m_tiles, m_tiles, sm_count, s);
      if (a.hd == 64) return launch_t<BIG_QKV, 64>(a, n_tiles * m_tiles, m_tiles, sm_count, s);
      return HSD_E_UNSUPPORTED;
    }
    case BIG_ADD_F32:
      if (a.seg_n[0] % kBN) return HSD_E_UNSUPPORTED;
      return launch_t<BIG_ADD_F32, 128>(a, a.seg_n[0] / kBN * m_tiles, m_tiles, sm_count, s);
    case BIG_SWIGLU:
      if (a.seg_n[0] % 64) return HSD_E_UNSUPPORTED;
      return launch_t<BIG_SWIGLU, 128>(a, ceil_div(a.seg_n[0], 128) * m_tiles, m_tiles, sm_count, s);
    case BIG_LOGITS: return launch_t<BIG_LOGITS, 128>(a, ceil_div(a.seg_n[0], kBN) * m_tiles, m_tiles, sm_count, s);
    default: return HSD_E_INVALID_ARG;
  }
}

}  // namespace hsd
