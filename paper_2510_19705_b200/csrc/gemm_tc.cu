// Weight-streaming GEMM for up to 256 token rows (see gemm_tc.cuh).
//
// Bound by HBM: W is read once.  A tile is up to 128 weight rows on the MMA's M side, the token rows (padded to 16..256)
// on its N side.  With few tiles the k-blocks of a tile are divided over a cluster of CTAs, whose partial sums stay in
// shared memory and are added across the cluster in rank order (bit-reproducible): no pieces in global memory, no
// counters.  With enough tiles to occupy the GPU a CTA takes whole tiles, and the next tile's weights stream in under a tile's finish.
// A stream-K split over all SMs with pieces in global memory took 29.5 us for 14336 x 4096 at 24 rows (117 MB); whole tiles of 104 rows
// on 138 CTAs take 25.6 us (22.5 to 23.2 started early, over five boxes); 4096 x 4096 at 256 rows 49 -> 20 us.
//
// 192 threads: warp 0 = TMA producer, warp 1 = TMEM owner + MMA issuer (one elected lane issues), warps 2..5 = epilogue
// (each reads its own 32-lane quarter of TMEM).  Shared-memory ring of (128 x 64 weight tile + NPAD x 64 activation
// tile), both K-major with the 128-byte swizzle TMA writes and the UMMA descriptors read.  A CTA's k-blocks are summed in
// two halves with a TMEM accumulator each, added in fp32 at the end: the tensor core's fp32 accumulation loses about as
// much as its chain is long (relative error against fp64 at K = 4096: 4.4e-6 in one chain, 2.1e-6 in two).  Every
// wait is bounded by wall time; a wait that gives up raises a flag, every role leaves its loop, TMEM is freed and a
// status word tells the host.  No waiter can be passed by (a parity wait sees a completion only until the next one): full[s]
// has its next loads behind empty[s], which the MMA issuer's commit completes; empty[s] its next MMAs behind the producer's
// loads; acc_full its next MMAs behind acc_empty, which all four epilogue warps complete; acc_empty its next epilogue behind
// the MMAs.
#include <algorithm>
#include "gemm_tc.cuh"
#include "tc_ptx.cuh"

namespace hsd {
namespace {

using namespace ptx;

constexpr int kThreads = 192;
constexpr int kStageWBytes = kTcBlockM * kTcBlockK * 2;       // 16 KiB
constexpr int kSmemTotal = 232448;                            // 227 KiB
constexpr int kLd = kTcBlockM + 4;                            // floats per token row of a staged tile (16-byte rows)

template <int NPAD> struct TcCfg {
  static constexpr int kStageBytes = kStageWBytes + NPAD * kTcBlockK * 2;
  static constexpr int kChunk = NPAD < 32 ? NPAD : 32;        // token rows the epilogue stages at a time (whole tiles)
  static constexpr int kStagingBytes = kChunk * kLd * 4;
  static constexpr int kCtrlBytes = 1024;
  static constexpr int kFit = (kSmemTotal - 1024 - kCtrlBytes - kStagingBytes) / kStageBytes;
  static constexpr int kStages = kFit < 12 ? kFit : 12;       // 12 x 16 KiB of weights in flight per SM cover HBM's latency twice
  static constexpr int kSmemBytes = kStages * kStageBytes + kStagingBytes + kCtrlBytes + 1024;
  static constexpr int kBufs = NPAD == 256 ? 1 : 2;           // tiles whose accumulators exist at a time, two accumulators each
  // one tile at a time: the epilogue adds the first accumulator to the second, and the next tile's first half runs under
  // the finish from there (128256 x 4096 at 256 rows: 322 -> 255 us)
  static constexpr bool kFold = kBufs == 1;
  static constexpr int kTmemCols = 2 * kBufs * NPAD;
  static_assert(NPAD * kLd * 4 <= kStages * kStageBytes, "a cluster's partial sums must fit the ring");
};

struct TileInfo { int seg, row0, col0; };
__device__ __forceinline__ TileInfo tile_info(const TcGemmArgs &a, int tile) {
  TileInfo ti;
  if (a.mode == GEMM_SWIGLU_T) { ti.seg = 0; ti.row0 = tile * kTcBoxRows; ti.col0 = 0; return ti; }
  int t = tile, col0 = 0;
  for (int s = 0; s < a.n_segs; ++s) {
    int nt = (a.seg_n[s] + a.tile_rows - 1) / a.tile_rows;
    if (t < nt || s == a.n_segs - 1) { ti.seg = s; ti.row0 = t * a.tile_rows; ti.col0 = col0; return ti; }
    t -= nt;
    col0 += a.seg_n[s];
  }
  ti.seg = 0; ti.row0 = 0; ti.col0 = 0;
  return ti;
}
__device__ __forceinline__ uint32_t cluster_rank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ float4 ld_cluster4(uint32_t addr, uint32_t rank) {
  uint32_t a;
  float4 v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
  asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ uint2 pack_bf16x4(const float4 &v) {
  const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
  return make_uint2(*reinterpret_cast<const unsigned *>(&a), *reinterpret_cast<const unsigned *>(&b));
}

// Token row r (of the pass), weight rows m .. m + 3 of the tile and, for SWIGLU / QKV, their partners (the up rows; the
// second half of the head) -> the projection's output.
template <int MODE>
__device__ __forceinline__ void finish4(const TcGemmArgs &a, const TileInfo &ti, int r, int m, const float4 &v, const float4 &w) {
  const int n = ti.row0 + m, left = a.seg_n[ti.seg] - n;
  if (left <= 0) return;
  const int row = a.row0 + r;
  if (MODE == GEMM_SWIGLU_T) {                               // ff is a multiple of 64: whole groups of four
    const float4 o = make_float4(silu_mul(v.x, w.x), silu_mul(v.y, w.y), silu_mul(v.z, w.z), silu_mul(v.w, w.w));
    *reinterpret_cast<uint2 *>(a.out_bf16 + (size_t)row * a.ldo + n) = pack_bf16x4(o);
  } else if (MODE == GEMM_QKV_T) {
    const TcQkv &k = a.qkv;
    const int half = k.hd >> 1, head = n / k.hd, c = n - head * k.hd;
    const int pos = k.row_pos[row];
    __nv_bfloat16 *dst;
    if (ti.seg == 0) dst = k.q + ((size_t)row * k.nq + head) * k.hd + c;
    else {
      const int pg = k.page_table[(size_t)k.row_seq[row] * k.pages_per_seq + pos / k.page];
      dst = (ti.seg == 1 ? k.k_pool : k.v_pool) + (((size_t)head * k.n_pages + pg) * k.page + pos % k.page) * k.hd + c;
    }
    float4 lo = v, hi = w;
    if (ti.seg < 2) {
      const float4 cs = __ldg(reinterpret_cast<const float4 *>(k.cos_tab + (size_t)pos * half + c));
      const float4 sn = __ldg(reinterpret_cast<const float4 *>(k.sin_tab + (size_t)pos * half + c));
      lo = make_float4(v.x * cs.x - w.x * sn.x, v.y * cs.y - w.y * sn.y, v.z * cs.z - w.z * sn.z, v.w * cs.w - w.w * sn.w);
      hi = make_float4(w.x * cs.x + v.x * sn.x, w.y * cs.y + v.y * sn.y, w.z * cs.z + v.z * sn.z, w.w * cs.w + v.w * sn.w);
    }
    *reinterpret_cast<uint2 *>(dst) = pack_bf16x4(lo);
    *reinterpret_cast<uint2 *>(dst + half) = pack_bf16x4(hi);
  } else if (MODE == GEMM_STORE_T_SCATTER) {
    __nv_bfloat16 *dst = a.out_bf16 + (size_t)a.dst[row] * a.ldo + ti.col0 + n;
    if (left >= 4 && (a.ldo & 3) == 0 && ((uintptr_t)a.out_bf16 & 7) == 0) *reinterpret_cast<uint2 *>(dst) = pack_bf16x4(v);
    else {
      const float e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (i < left) dst[i] = __float2bfloat16_rn(e[i]);
    }
  } else {
    float *dst = a.out_f32 + (size_t)row * a.ldo + ti.col0 + n;
    float4 o = v;
    if (left >= 4 && (a.ldo & 3) == 0 && ((uintptr_t)a.out_f32 & 15) == 0) {
      if (MODE == GEMM_ADD_F32) {
        const float4 old = __ldcg(reinterpret_cast<const float4 *>(dst));
        o = make_float4(old.x + v.x, old.y + v.y, old.z + v.z, old.w + v.w);
      }
      *reinterpret_cast<float4 *>(dst) = o;
    } else {
      const float e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (i < left) dst[i] = MODE == GEMM_ADD_F32 ? __ldcg(dst + i) + e[i] : e[i];
    }
  }
}

// Items of one staged token row: groups of four weight rows (SWIGLU, QKV: of the first halves only).
template <int MODE> __device__ __forceinline__ int items_of(const TcGemmArgs &a) {
  return (MODE == GEMM_SWIGLU_T || MODE == GEMM_QKV_T) ? kTcBlockM / 8 : (a.tile_rows + 3) / 4;
}
template <int MODE> __device__ __forceinline__ void item_at(const TcGemmArgs &a, int i, int &m, int &partner) {
  m = i * 4; partner = m;
  if (MODE == GEMM_SWIGLU_T) partner = m + kTcBoxRows;
  if (MODE == GEMM_QKV_T) {
    const int half = a.qkv.hd >> 1, head = m / half;
    m += head * half;
    partner = m + half;
  }
}

template <int NPAD, int MODE>
__global__ void __launch_bounds__(kThreads, 1) gemm_tc_kernel(const __grid_constant__ TcGemmArgs args, int n_tiles, int KB, int S) {
  using Cfg = TcCfg<NPAD>;
  constexpr int STAGES = Cfg::kStages;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t *ring = smem;
  float *staging = reinterpret_cast<float *>(smem + STAGES * Cfg::kStageBytes);
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + STAGES * Cfg::kStageBytes + Cfg::kStagingBytes);
  // bars: full[STAGES] | empty[STAGES] | acc_full[2] | acc_empty[2]
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * STAGES + 4);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
  volatile int *wait_ok = reinterpret_cast<volatile int *>(tmem_slot + 2);      // [2], alternating per tile
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (STAGES + s); };
  auto accf_bar = [&](int b) { return bar0 + 8u * (2 * STAGES + b); };
  auto acce_bar = [&](int b) { return bar0 + 8u * (2 * STAGES + 2 + b); };
  const int warp = warp_index(), lane = threadIdx.x & 31;
  chain_next();
  // S > 1: the cluster's CTAs share tile blockIdx.x / S; S = 1: tiles blockIdx.x, + gridDim.x, ...
  const int rank = S > 1 ? (int)cluster_rank() : 0;
  const int tile0 = S > 1 ? (int)blockIdx.x / S : (int)blockIdx.x, step = S > 1 ? n_tiles : (int)gridDim.x;
  const int kb0 = KB * rank / S, kb1 = KB * (rank + 1) / S;
  const int kb_half = kb1 - kb0 > 1 ? (kb0 + kb1) / 2 : kb1;     // the second accumulator's first k-block

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(accf_bar(b), 1); mbar_init(acce_bar(b), 4); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(smem_u32(tmem_slot), Cfg::kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    const bool issuer = elect_one();
    const uint64_t policy = l2_policy_evict_first();
    int s = 0;
    uint32_t ph = 0;
    bool ok = true;
    const uint32_t box_bytes = (uint32_t)args.w_box_rows * kTcBlockK * 2;
    // the ring's first weights before the wait for the activations (128 positions x 32 layers of the 8B shape with all
    // their exits' logits 5.42 -> 5.00 ms, the prompt of a 1B shape 2.45 -> 2.15, eight of 1024 tokens of the 8B shape 97 -> 93)
    const int ahead = tile0 < n_tiles ? min(STAGES, kb1 - kb0) : 0;
    for (int tile = tile0; tile < n_tiles && ok; tile += step) {
      const TileInfo ti = tile_info(args, tile);
      const bool second = MODE == GEMM_SWIGLU_T || (args.w_box_rows < args.tile_rows && ti.row0 + args.w_box_rows < args.seg_n[ti.seg]);
      const CUtensorMap *w0 = &args.w[ti.seg], *w1 = MODE == GEMM_SWIGLU_T ? &args.w[1] : w0;
      const int row1 = MODE == GEMM_SWIGLU_T ? ti.row0 : ti.row0 + args.w_box_rows;
      const uint32_t bytes = (second ? 2 : 1) * box_bytes + (uint32_t)args.a_box_rows * kTcBlockK * 2;
      auto load_w = [&](int kb, int slot) {
        const uint32_t dst = smem_u32(ring) + (uint32_t)(slot * Cfg::kStageBytes);
        mbar_expect_tx(full_bar(slot), bytes);
        if (args.stream_weights) {
          tma_load_2d_hint(dst, w0, kb * kTcBlockK, ti.row0, full_bar(slot), policy);
          if (second) tma_load_2d_hint(dst + box_bytes, w1, kb * kTcBlockK, row1, full_bar(slot), policy);
        } else {
          tma_load_2d(dst, w0, kb * kTcBlockK, ti.row0, full_bar(slot));
          if (second) tma_load_2d(dst + box_bytes, w1, kb * kTcBlockK, row1, full_bar(slot));
        }
      };
      auto load_a = [&](int kb, int slot) {
        tma_load_2d(smem_u32(ring) + (uint32_t)(slot * Cfg::kStageBytes + kStageWBytes), &args.a, kb * kTcBlockK, args.row0, full_bar(slot));
      };
      int kb = kb0;
      if (tile == tile0) {
        if (!args.early_weights) chain_wait();
        // a wait gives up after two seconds, long after every CTA (one per SM) has started
        if (args.reset_status && blockIdx.x == 0 && issuer) *args.status = 0;
        if (issuer)
          for (int i = 0; i < ahead; ++i) {
            load_w(kb0 + i, i);
            if (!args.early_weights) load_a(kb0 + i, i);
          }
        if (args.early_weights) chain_wait();
        if (issuer && args.early_weights)
          for (int i = 0; i < ahead; ++i) load_a(kb0 + i, i);
        kb += ahead; s = ahead;
        if (s == STAGES) { s = 0; ph ^= 1u; }
      }
      for (; kb < kb1; ++kb) {
        if (!mbar_wait_warp(empty_bar(s), ph ^ 1u, abort_flag)) { ok = false; break; }
        if (issuer) { load_w(kb, s); load_a(kb, s); }
        if (++s == STAGES) { s = 0; ph ^= 1u; }
      }
    }
    if (!ok) {                                   // copies in flight land before the shared memory goes away
      const unsigned long long t0 = globaltimer_ns();
      while (globaltimer_ns() - t0 < 200000ull) {}
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    const bool issuer = elect_one();
    chain_wait();                               // (this warp takes part in a cluster's finish)
    const uint32_t idesc = umma_idesc_bf16(NPAD);
    const uint64_t da0 = umma_desc(smem_u32(ring));
    int s = 0, ti = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int tile = tile0; tile < n_tiles && ok; tile += step, ++ti) {
      const int ab = ti % Cfg::kBufs;
      if (!mbar_wait_warp(acce_bar(ab), (uint32_t)((ti / Cfg::kBufs) & 1) ^ 1u, abort_flag)) break;
      tc_fence_after();
      uint32_t d_tmem = tmem_base + (uint32_t)(ab * 2 * NPAD), acc = 0u;
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!mbar_wait_warp(full_bar(s), ph, abort_flag)) { ok = false; break; }
        if (kb == kb_half) {
          if (Cfg::kFold) {
            if (!mbar_wait_warp(acce_bar(1), (uint32_t)(ti & 1) ^ 1u, abort_flag)) { ok = false; break; }
            tc_fence_after();
          }
          d_tmem += NPAD; acc = 0u;
        }
        const uint64_t da = da0 + (uint64_t)(s * (Cfg::kStageBytes >> 4)), db = da + (uint64_t)(kStageWBytes >> 4);
        if (issuer) {
          umma_bf16(d_tmem, da, db, idesc, acc);
#pragma unroll
          for (int k = 1; k < kTcBlockK / 16; ++k) umma_bf16(d_tmem, da + (uint64_t)(k * 2), db + (uint64_t)(k * 2), idesc, 1u);
          umma_commit(empty_bar(s));            // the stage is free once these MMAs have read it
        }
        acc = 1u;
        if (++s == STAGES) { s = 0; ph ^= 1u; }
      }
      if (ok && issuer) umma_commit(accf_bar(ab));      // accumulator complete
    }
  } else {
    // ------------------------------------------------------------------ epilogue (warps 2..5)
    const int q = warp & 3;                     // TMEM lane quarter this warp may read
    const int m = q * 32 + lane;                // weight row of the tile held by this thread
    const int et = threadIdx.x - 64;            // 0..127 among the epilogue threads
    const int n_items = items_of<MODE>(args);
    chain_wait();
    int ti = 0;
    for (int tile = tile0; tile < n_tiles; tile += step, ++ti) {
      const int ab = ti % Cfg::kBufs;
      // one thread waits, all 128 take the same decision (a bail-out must not split the group)
      if (et == 0) wait_ok[ti & 1] = mbar_wait(accf_bar(ab), (uint32_t)((ti / Cfg::kBufs) & 1), abort_flag) ? 1 : 0;
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (!wait_ok[ti & 1]) break;
      tc_fence_after();
      constexpr int CH = Cfg::kChunk;
      const TileInfo info = tile_info(args, tile);
      const uint32_t tbase = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(ab * 2 * NPAD);
      float *part = S > 1 ? reinterpret_cast<float *>(ring) : staging;       // S > 1: every load of the CTA has been consumed
      const bool fold = Cfg::kFold && S == 1 && kb_half < kb1;
      if (fold) {
#pragma unroll 1
        for (int c0 = 0; c0 < NPAD && c0 < args.R; c0 += CH) {
          float v[CH], v2[CH];
#pragma unroll
          for (int j = 0; j < CH / 16; ++j) {
            tmem_ld16(tbase + (uint32_t)(c0 + j * 16), v + j * 16);
            tmem_ld16(tbase + (uint32_t)(NPAD + c0 + j * 16), v2 + j * 16);
          }
          tmem_ld_wait();
#pragma unroll
          for (int r = 0; r < CH; ++r) v[r] += v2[r];
#pragma unroll
          for (int j = 0; j < CH / 16; ++j) tmem_st16u(tbase + (uint32_t)(NPAD + c0 + j * 16), reinterpret_cast<const unsigned *>(v + j * 16));
        }
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acce_bar(0));
      }
#pragma unroll 1
      for (int c0 = 0; c0 < NPAD && c0 < args.R; c0 += CH) {
        float v[CH], v2[CH];
#pragma unroll
        for (int j = 0; j < CH / 16; ++j) tmem_ld16(tbase + (uint32_t)((fold ? NPAD : 0) + c0 + j * 16), v + j * 16);
        if (kb_half < kb1 && !fold) {
#pragma unroll
          for (int j = 0; j < CH / 16; ++j) tmem_ld16(tbase + (uint32_t)(NPAD + c0 + j * 16), v2 + j * 16);
        }
        tmem_ld_wait();
        if (kb_half < kb1 && !fold) {
#pragma unroll
          for (int r = 0; r < CH; ++r) v[r] += v2[r];
        }
        float *to = part + (S > 1 ? c0 * kLd : 0);
#pragma unroll
        for (int r = 0; r < CH; ++r) to[r * kLd + m] = v[r];
        if (S > 1) continue;
        asm volatile("bar.sync 1, 128;" ::: "memory");
        const int rows = min(CH, args.R - c0);
        for (int i = et; i < rows * n_items; i += 128) {
          const int r = i / n_items;
          int mm, pp;
          item_at<MODE>(args, i - r * n_items, mm, pp);
          const float4 a4 = *reinterpret_cast<const float4 *>(to + r * kLd + mm), b4 = *reinterpret_cast<const float4 *>(to + r * kLd + pp);
          finish4<MODE>(args, info, c0 + r, mm, a4, b4);
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acce_bar(fold ? 1 : ab));
    }
  }
  __syncwarp();
  if (S > 1) {
    // ------------------------------------------------------------------ sums across the cluster, in rank order
    __syncthreads();
    cluster_sync();
    const TileInfo info = tile_info(args, tile0);
    const int r0 = args.R * rank / S, r1 = args.R * (rank + 1) / S, n_items = items_of<MODE>(args);
    const uint32_t base = smem_u32(ring);
    const bool ok = !*abort_flag;
    for (int i = threadIdx.x; i < (r1 - r0) * n_items && ok; i += kThreads) {
      const int r = r0 + i / n_items;
      int mm, pp;
      item_at<MODE>(args, i % n_items, mm, pp);
      float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
      for (int p0 = 0; p0 < S; p0 += 4) {                         // up to four ranks' loads in flight
        float4 xs[4], ys[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          if (p0 + p >= S) continue;
          xs[p] = ld_cluster4(base + (uint32_t)(r * kLd + mm) * 4u, (uint32_t)(p0 + p));
          if (MODE == GEMM_SWIGLU_T || MODE == GEMM_QKV_T) ys[p] = ld_cluster4(base + (uint32_t)(r * kLd + pp) * 4u, (uint32_t)(p0 + p));
        }
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          if (p0 + p >= S) continue;
          x.x += xs[p].x; x.y += xs[p].y; x.z += xs[p].z; x.w += xs[p].w;
          if (MODE == GEMM_SWIGLU_T || MODE == GEMM_QKV_T) { y.x += ys[p].x; y.y += ys[p].y; y.z += ys[p].z; y.w += ys[p].w; }
        }
      }
      finish4<MODE>(args, info, r, mm, x, y);
    }
    __syncwarp();
    cluster_sync();                             // nobody leaves while its partial sums are being read
  }
  // ------------------------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem_base, Cfg::kTmemCols);
  if (threadIdx.x == 0 && *abort_flag) atomicExch(args.status, 1);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                  const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn g_encode = nullptr;

template <int NPAD, int MODE>
int launch_t(const TcGemmArgs &args, int n_tiles, int S, int grid, cudaStream_t s) {
  using Cfg = TcCfg<NPAD>;
  static std::atomic<u64> limits{0};
  const int limit = hsd_smem_limit((const void *)gemm_tc_kernel<NPAD, MODE>, Cfg::kSmemBytes, limits);
  if (limit) return limit;
  HSD_CUDA_OK(hsd_launch(gemm_tc_kernel<NPAD, MODE>, grid, kThreads, Cfg::kSmemBytes, s, S, args.chained, args, n_tiles, args.K / kTcBlockK, S));
  hsd_count_launches(1);
  return hsd_launch_status();
}

template <int NPAD>
int launch_mode(const TcGemmArgs &args, int n_tiles, int S, int grid, cudaStream_t s) {
  switch (args.mode) {
    case GEMM_STORE_F32: return launch_t<NPAD, GEMM_STORE_F32>(args, n_tiles, S, grid, s);
    case GEMM_ADD_F32: return launch_t<NPAD, GEMM_ADD_F32>(args, n_tiles, S, grid, s);
    case GEMM_STORE_T_SCATTER: return launch_t<NPAD, GEMM_STORE_T_SCATTER>(args, n_tiles, S, grid, s);
    case GEMM_SWIGLU_T: return launch_t<NPAD, GEMM_SWIGLU_T>(args, n_tiles, S, grid, s);
    case GEMM_QKV_T: return launch_t<NPAD, GEMM_QKV_T>(args, n_tiles, S, grid, s);
    default: return HSD_E_INVALID_ARG;
  }
}

}  // namespace

int tc_init() {
  if (g_encode) return HSD_OK;
  void *fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess || !fn ||
      qres != cudaDriverEntryPointSuccess)
    return HSD_E_UNSUPPORTED;
  g_encode = (EncodeTiledFn)fn;
  return HSD_OK;
}

int tc_make_map(CUtensorMap *map, const void *base, long long rows, long long cols, int box_rows) {
  if (!g_encode) return HSD_E_UNSUPPORTED;
  if (((uintptr_t)base & 15) != 0 || (cols * 2) % 16 != 0 || box_rows < 1 || box_rows > 256) return HSD_E_INVALID_ARG;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
  cuuint32_t box[2] = {(cuuint32_t)kTcBlockK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? HSD_OK : HSD_E_CUDA;
}

int tc_npad(int rows) { return rows <= 16 ? 16 : rows <= 32 ? 32 : rows <= 64 ? 64 : rows <= 128 ? 128 : 256; }

namespace {
// CTAs a tile's k-blocks are divided over: 2, 4 or (few tiles) 8 while full tiles alone leave half the SMs idle.  The division
// does not depend on the number of rows, so neither does a row's result.  48 clusters of three or 16 of eight do not run at
// once (6144 x 4096 at 128 rows: 36 us in threes, 25 us in pairs), 74 of two, 32 of four and 14 of eight do (on the GPU that
// was measured: speed only).
int split_of(int full_tiles, int K, int sm_count) {
  int S = 1;
  while (S < (full_tiles <= 14 ? 8 : 4) && full_tiles * S * 2 <= sm_count && S * 2 <= K / kTcBlockK) S *= 2;
  return S;
}
}  // namespace

// Rows of a tile of one matrix on its own: 128, or as many fewer as spread N evenly over the rounds the SMs need or, with the
// k-blocks divided, over the clusters that run at once (the same sums: a row's result does not change).  Of up to 32 token rows
// full tiles are as fast (5632 x 2048: 8.0 and 8.1 us at 16) and leave SMs on which the next launch starts; of more a CTA's
// activations and finish count: 64 / 128 / 200 rows of 5632 x 2048 11.2 / 14.6 / 19.0 -> 9.3 / 11.4 / 15.8 us, of 2048 x 5632
// 10.2 / 12.3 / 16.9 -> 10.0 / 11.4 / 15.6, of 1024 x 4096 7.9 / 9.6 / 13.0 -> 7.5 / 9.0 / 11.7.
int tc_tile_rows(int N, int K, int R, int sm_count) {
  const int S = split_of(ceil_div(N, kTcBlockM), K, sm_count);
  if (S > 1 && R <= 32) return kTcBlockM;
  const int at_once = S == 2 ? 74 : S == 4 ? 32 : S == 8 ? 14 : sm_count, rounds = ceil_div(N, kTcBlockM * at_once);
  return std::min(kTcBlockM, ceil_div(ceil_div(N, rounds * at_once), 8) * 8);
}

int launch_gemm_tc(const TcGemmArgs &args, int sm_count, cudaStream_t s) {
  if (args.R < 1 || args.R > 256 || args.K < kTcBlockK || args.K % kTcBlockK != 0) return HSD_E_UNSUPPORTED;
  int n_tiles = 0, full_tiles = 0;
  for (int i = 0; i < (args.mode == GEMM_SWIGLU_T ? 1 : args.n_segs); ++i) {
    n_tiles += ceil_div(args.seg_n[i], args.mode == GEMM_SWIGLU_T ? kTcBoxRows : args.tile_rows);
    full_tiles += ceil_div(args.seg_n[i], args.mode == GEMM_SWIGLU_T ? kTcBoxRows : kTcBlockM);
  }
  const int S = split_of(full_tiles, args.K, sm_count);
  const int grid = S > 1 ? n_tiles * S : std::min(n_tiles, sm_count);
  switch (tc_npad(args.R)) {
    case 16: return launch_mode<16>(args, n_tiles, S, grid, s);
    case 32: return launch_mode<32>(args, n_tiles, S, grid, s);
    case 64: return launch_mode<64>(args, n_tiles, S, grid, s);
    case 128: return launch_mode<128>(args, n_tiles, S, grid, s);
    default: return launch_mode<256>(args, n_tiles, S, grid, s);
  }
}

}  // namespace hsd
