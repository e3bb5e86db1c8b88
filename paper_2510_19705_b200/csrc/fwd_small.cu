// One-launch forward of small fp32 models: a cooperative kernel runs every layer of a pass.
//
// Bound by latency: a four-layer pass of width 128 (4.8 rows) moves 4 MB, but as one launch per operation it took 206 us (39
// launches of about 5 us); this way 68 us, 3.3 us a phase.  Here a layer is five phases with a grid barrier after each:
//   q / k / v (RMSNorm of the rows in front, rotary embedding and cache append behind), attention, O + residual,
//   gate / up (RMSNorm in front, SwiGLU behind), down + residual;
// the last phase is the final norm + output head over the logit rows.  In a product a warp owns two weight rows (rotary
// partners in the q / k / v phase, gate and up in the SwiGLU phase) and streams them against the rows staged in shared
// memory, fp32 multiply-adds, sums across lanes at the end.  Attention: a CTA per (row, query head), its warps take
// 32-key tiles in turn and merge at the end.  The grid is as large as the widest phase needs and no larger (the barrier's
// cost grows with it).  Waits are bounded.
#include <algorithm>
#include "fwd_small.cuh"

namespace hsd {
namespace {

constexpr int kThreads = 256, kWarps = kThreads / 32;
constexpr int kChunk = 512;                      // floats of a row staged at a time
constexpr unsigned long long kLimitNs = 2000000000ull;

__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

struct Shared {
  float a[16 * kChunk];                          // rows of the product's left operand
  float inv[kSmallRows];                         // 1 / rms of each row
  int pos[kSmallRows], pg[kSmallRows], tok[kSmallRows];   // position of each row, the page that holds it, its token
  float m[kWarps], l[kWarps];
  __align__(16) float o[kWarps][128];    // attention: the warps' states
  int ok;
};

// All CTAs; false once a wait has given up (every thread of every CTA then leaves).
__device__ __forceinline__ bool barrier(const SmallFwdArgs &a, unsigned &target, Shared &sh) {
  __syncthreads();
  target += gridDim.x;
  if (threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.counter) : "memory");
    int ok = 1;
    unsigned long long t0 = 0;
    for (unsigned it = 1;; ++it) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a.counter) : "memory");
      if ((int)(v - target) >= 0) break;
      if ((it & 63u) == 0u) {
        const unsigned long long t = now_ns();
        if (t0 == 0) t0 = t;
        if (*reinterpret_cast<volatile int *>(a.status) != 0 || t - t0 > kLimitNs) { atomicExch(a.status, 1); ok = 0; break; }
      }
    }
    sh.ok = ok;
  }
  __syncthreads();
  return sh.ok != 0;
}

// acc[0][0 / 1] = row r0 + lane_row(lane) of the operand times weight rows w0 / w1.  The operand's rows: src(r),
// scaled by 1 / rms x gain when gain is given: rows of one chunk are read once, by a warp each, which has the row's scale
// before it stages it; longer ones need their scales in sh.inv (row_scales).
template <int RT, class Src>
__device__ __forceinline__ void product(Shared &sh, const Src &src, const float *gain, float eps, int K, int r0, int rows, bool active, const float *w0,
                                        const float *w1, float (*acc)[2]) {
  const int tid = threadIdx.x, lane = tid & 31;
#pragma unroll
  for (int r = 0; r < RT; ++r) acc[r][0] = acc[r][1] = 0.f;
  for (int kc = 0; kc < K; kc += kChunk) {
    const int n4 = min(kChunk, K - kc) >> 2;     // K is a multiple of 4
    float4 p0 = make_float4(0.f, 0.f, 0.f, 0.f), p1 = p0;
    if (active && lane < n4) {                   // the first weights are on their way while the rows are staged
      p0 = __ldg(reinterpret_cast<const float4 *>(w0 + kc) + lane);
      p1 = __ldg(reinterpret_cast<const float4 *>(w1 + kc) + lane);
    }
    __syncthreads();
    if (gain && K <= kChunk) {
      constexpr int NV = kChunk / 128;
      for (int r = tid >> 5; r < rows; r += kWarps) {
        const float4 *row = reinterpret_cast<const float4 *>(src(r0 + r));
        float4 v[NV], g[NV];
#pragma unroll
        for (int j = 0; j < NV; ++j) {
          const int k = lane + 32 * j;
          v[j] = k < n4 ? __ldcg(row + k) : make_float4(0.f, 0.f, 0.f, 0.f);
          g[j] = k < n4 ? __ldg(reinterpret_cast<const float4 *>(gain) + k) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        float ss = 0.f;
#pragma unroll
        for (int j = 0; j < NV; ++j) ss += (v[j].x * v[j].x + v[j].y * v[j].y) + (v[j].z * v[j].z + v[j].w * v[j].w);
        for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xFFFFFFFFu, ss, o);
        const float s = rsqrtf(ss / (float)K + eps);
#pragma unroll
        for (int j = 0; j < NV; ++j)
          if (lane + 32 * j < n4)
            *reinterpret_cast<float4 *>(sh.a + r * kChunk + 4 * (lane + 32 * j)) =
                make_float4(v[j].x * s * g[j].x, v[j].y * s * g[j].y, v[j].z * s * g[j].z, v[j].w * s * g[j].w);
      }
    } else {
      for (int i = tid; i < rows * n4; i += kThreads) {
        const int r = i / n4, k = i - r * n4;
        float4 v = __ldcg(reinterpret_cast<const float4 *>(src(r0 + r) + kc) + k);
        if (gain) {
          const float4 g = __ldg(reinterpret_cast<const float4 *>(gain + kc) + k);
          const float s = sh.inv[r0 + r];
          v = make_float4(v.x * s * g.x, v.y * s * g.y, v.z * s * g.z, v.w * s * g.w);
        }
        *reinterpret_cast<float4 *>(sh.a + r * kChunk + 4 * k) = v;
      }
    }
    __syncthreads();
    if (!active) continue;
    for (int k = lane; k < n4; k += 32) {
      const float4 u0 = p0, u1 = p1;
      if (k + 32 < n4) {
        p0 = __ldg(reinterpret_cast<const float4 *>(w0 + kc) + k + 32);
        p1 = __ldg(reinterpret_cast<const float4 *>(w1 + kc) + k + 32);
      }
#pragma unroll
      for (int r = 0; r < RT; ++r) {
        if (r >= rows) break;
        const float4 v = *reinterpret_cast<const float4 *>(sh.a + r * kChunk + 4 * k);
        acc[r][0] = fmaf(v.x, u0.x, fmaf(v.y, u0.y, fmaf(v.z, u0.z, fmaf(v.w, u0.w, acc[r][0]))));
        acc[r][1] = fmaf(v.x, u1.x, fmaf(v.y, u1.y, fmaf(v.z, u1.z, fmaf(v.w, u1.w, acc[r][1]))));
      }
    }
  }
  if (active) {
    // sums over the lanes; while there are several rows a lane keeps the half its bit selects and gives the other away
    // (the same additions as a butterfly per value, 12 exchanges instead of 40 for four rows)
    int n = RT;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      if (n > 1) {
        n >>= 1;
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int r = 0; r < RT / 2; ++r) {
          if (r >= n) break;
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const float keep = up ? acc[n + r][e] : acc[r][e], give = up ? acc[r][e] : acc[n + r][e];
            acc[r][e] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, o);
          }
        }
      } else {
        acc[0][0] += __shfl_xor_sync(0xFFFFFFFFu, acc[0][0], o);
        acc[0][1] += __shfl_xor_sync(0xFFFFFFFFu, acc[0][1], o);
      }
    }
  }
}
// The row whose sums product() leaves in acc[0] of a lane (32 / RT neighbours hold the same).
template <int RT> __device__ __forceinline__ int lane_row(int lane) { return lane / (32 / RT); }

// 1 / rms of rows 0 .. n - 1 longer than a chunk, a warp per row (product()'s first barrier comes before the scales are read).
template <class Src> __device__ __forceinline__ void row_scales(Shared &sh, const Src &src, int n, int d, float eps) {
  const int lane = threadIdx.x & 31;
  if (d <= kChunk) return;
  for (int r = threadIdx.x >> 5; r < n; r += kWarps) {
    const float4 *row = reinterpret_cast<const float4 *>(src(r));
    float ss = 0.f;
    for (int k = lane; k < d >> 2; k += 32) {
      const float4 v = __ldcg(row + k);
      ss += (v.x * v.x + v.y * v.y) + (v.z * v.z + v.w * v.w);
    }
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xFFFFFFFFu, ss, o);
    if (lane == 0) sh.inv[r] = rsqrtf(ss / (float)d + eps);
  }
}

// A whole product phase: pairs of weight rows dealt to the grid's warps, row tiles of RT; finish(pair, row, v0, v1) is
// called once per (pair, row), by one lane.
template <int RT, class Src, class Pair, class Finish>
__device__ __forceinline__ void product_phase(Shared &sh, const Src &src, const float *gain, float eps, int K, int n_rows, int n_pairs, const Pair &pair,
                                              const Finish &finish) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int base = blockIdx.x * kWarps; base < n_pairs; base += gridDim.x * kWarps) {      // uniform over the CTA
    const int p = base + warp;
    const bool active = p < n_pairs;
    const float *w0 = nullptr, *w1 = nullptr;
    if (active) pair(p, w0, w1);
    for (int r0 = 0; r0 < n_rows; r0 += RT) {
      const int rows = min(RT, n_rows - r0);
      float acc[RT][2];
      product<RT>(sh, src, gain, eps, K, r0, rows, active, w0, w1, acc);
      // (all rows at once: one lane's finish after the other's is a trip to L2 per row)
      if (active && lane % (32 / RT) == 0 && lane_row<RT>(lane) < rows) finish(p, r0 + lane_row<RT>(lane), acc[0][0], acc[0][1]);
    }
  }
}

// Attention of (row, query head) units, a CTA each: lane = key for the scores, HD / 4 lanes to a key's values for P V (few
// instructions: a warp runs this once a layer, and unrolled code for each key comes from beyond the instruction cache).
// `first`: the thread's cache row in the CTA's first unit, key = thread (the same in every layer: found once).
__device__ __forceinline__ int cache_row(const SmallFwdArgs &a, int u, int key) {
  const int r = u / a.nq, kvh = (u - r * a.nq) / (a.nq / a.nkv);
  return (kvh * a.n_pages + a.page_table[(size_t)a.rows.seq()[r] * a.pages_per_seq + key / a.page]) * a.page + key % a.page;
}
template <int HD> __device__ __forceinline__ void attention_phase(const SmallFwdArgs &a, const SmallLayerDev &ly, Shared &sh, int first) {
  constexpr int LPR = HD / 4, RPI = 32 / LPR, NI = 32 / RPI, PRE = NI < 8 ? NI : 8;   // lanes of a row, rows at a time
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float scale = rsqrtf((float)HD);
  for (int u = blockIdx.x; u < a.R * a.nq; u += gridDim.x) {
    const int r = u / a.nq, h = u - r * a.nq, n_keys = sh.pos[r] + 1;
    __syncthreads();                                                 // the previous unit's merge has been read
    if (tid < HD) sh.a[tid] = __ldcg(a.q + ((size_t)r * a.nq + h) * HD + tid);
    __syncthreads();
    float m = -INFINITY, l = 0.f;
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);                      // four dimensions, of the keys of this lane's group
    for (int k0 = warp * 32; k0 < n_keys; k0 += kWarps * 32) {
      const int key = k0 + lane, nk = min(32, n_keys - k0);
      float s = -INFINITY;
      int row = 0;
      if (lane < nk) {
        row = (u == (int)blockIdx.x && key < kThreads) ? first : cache_row(a, u, key);
        const float4 *kr = reinterpret_cast<const float4 *>(ly.k_pool + (size_t)row * HD);
        float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int c = 0; c < HD / 4; ++c) {
          const float4 kv = __ldcg(kr + c), qv = *reinterpret_cast<const float4 *>(sh.a + 4 * c);
          t = make_float4(fmaf(qv.x, kv.x, t.x), fmaf(qv.y, kv.y, t.y), fmaf(qv.z, kv.z, t.z), fmaf(qv.w, kv.w, t.w));
        }
        s = ((t.x + t.y) + (t.z + t.w)) * scale;
      }
      auto value = [&](int i) {                                      // of key RPI i + lane / LPR of the tile
        const int kk = RPI * i + lane / LPR, vr = __shfl_sync(0xFFFFFFFFu, row, kk);
        return kk < nk ? __ldcg(reinterpret_cast<const float4 *>(ly.v_pool + (size_t)vr * HD) + lane % LPR) : make_float4(0.f, 0.f, 0.f, 0.f);
      };
      auto add = [&](int i, float weight, const float4 &v) {
        const float w = __shfl_sync(0xFFFFFFFFu, weight, RPI * i + lane / LPR);
        o = make_float4(fmaf(w, v.x, o.x), fmaf(w, v.y, o.y), fmaf(w, v.z, o.z), fmaf(w, v.w, o.w));
      };
      float4 pre[PRE];                                               // on their way while the weights are worked out
#pragma unroll
      for (int i = 0; i < PRE; ++i) pre[i] = value(i);
      float mx = s;
#pragma unroll
      for (int x = 16; x > 0; x >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, x));
      // (a tile without a finite score leaves the state as it is)
      const float mn = fmaxf(m, mx), corr = mn > -INFINITY ? __expf(m - mn) : 1.f, p = lane < nk && mn > -INFINITY ? __expf(s - mn) : 0.f;
      float ps = p;
#pragma unroll
      for (int x = 16; x > 0; x >>= 1) ps += __shfl_xor_sync(0xFFFFFFFFu, ps, x);
      l = l * corr + ps;
      m = mn;
      o = make_float4(o.x * corr, o.y * corr, o.z * corr, o.w * corr);
#pragma unroll
      for (int i = 0; i < PRE; ++i) add(i, p, pre[i]);
#pragma unroll 4
      for (int i = PRE; i < NI; ++i) {
        if (RPI * i >= nk) break;
        add(i, p, value(i));
      }
    }
#pragma unroll
    for (int x = LPR; x < 32; x <<= 1)
      o = make_float4(o.x + __shfl_xor_sync(0xFFFFFFFFu, o.x, x), o.y + __shfl_xor_sync(0xFFFFFFFFu, o.y, x),
                      o.z + __shfl_xor_sync(0xFFFFFFFFu, o.z, x), o.w + __shfl_xor_sync(0xFFFFFFFFu, o.w, x));
    if (lane == 0) { sh.m[warp] = m; sh.l[warp] = l; }
    if (lane < LPR) *reinterpret_cast<float4 *>(&sh.o[warp][4 * lane]) = o;
    __syncthreads();
    if (tid < HD) {                                                  // the warps' states in warp order (the first always holds keys)
      float mm = sh.m[0];
      for (int w = 1; w < kWarps; ++w) mm = fmaxf(mm, sh.m[w]);
      float lt = 0.f, ot = 0.f;
      for (int w = 0; w < kWarps; ++w) {
        const float f = sh.m[w] > -INFINITY ? __expf(sh.m[w] - mm) : 0.f;
        lt += f * sh.l[w];
        ot += f * sh.o[w][tid];
      }
      a.att[((size_t)r * a.nq + h) * HD + tid] = ot / lt;
    }
  }
}

template <int RT, int HD>
__global__ void __launch_bounds__(kThreads) fwd_small_kernel(const __grid_constant__ SmallFwdArgs a) {
  __shared__ __align__(16) Shared sh;
  const int tid = threadIdx.x;
  unsigned target = a.base;
  constexpr int HALF = HD / 2;
  if (tid < a.R) {
    const int seq = a.rows.seq()[tid];
    sh.pos[tid] = a.rows.pos()[tid];
    sh.pg[tid] = a.page_table[(size_t)seq * a.pages_per_seq + sh.pos[tid] / a.page];
    // an id outside the vocabulary (only possible after non-finite logits) must not become an address
    sh.tok[tid] = min(max(a.tokens[(size_t)seq * a.max_seq + sh.pos[tid]], 0), a.V - 1);
  }
  __syncthreads();
  // the residual stream starts as the embedding rows (the first phase reads them from the table; they are first needed
  // here by the first residual add, two barriers on)
  for (int r = blockIdx.x; r < a.R; r += gridDim.x) {
    const float *src = a.embed + (size_t)sh.tok[r] * a.d;
    for (int k = tid; k < a.d; k += kThreads) a.x[(size_t)r * a.d + k] = src[k];
  }
  const int nqd = a.nq * HD;
  int first = 0;
  if ((int)blockIdx.x < a.R * a.nq && tid <= sh.pos[blockIdx.x / a.nq]) first = cache_row(a, blockIdx.x, tid);
  for (int l = 0; l < a.n_run; ++l) {
    const SmallLayerDev ly = a.layers[l];
    auto xs = [&](int r) { return l == 0 ? a.embed + (size_t)sh.tok[r] * a.d : (const float *)(a.x + (size_t)r * a.d); };
    auto xr = [&](int r) { return (const float *)(a.x + (size_t)r * a.d); };
    row_scales(sh, xs, a.R, a.d, a.eps);
    product_phase<RT>(sh, xs, ly.w[0], a.eps, a.d, a.R, (a.nq + 2 * a.nkv) * HALF,
                      [&](int p, const float *&w0, const float *&w1) {
                        const int head = p / HALF, c = p - head * HALF;
                        const float *w = head < a.nq ? ly.w[1] + (size_t)head * HD * a.d
                                         : head < a.nq + a.nkv ? ly.w[2] + (size_t)(head - a.nq) * HD * a.d
                                                               : ly.w[3] + (size_t)(head - a.nq - a.nkv) * HD * a.d;
                        w0 = w + (size_t)c * a.d; w1 = w + (size_t)(c + HALF) * a.d;
                      },
                      [&](int p, int r, float v0, float v1) {
                        const int head = p / HALF, c = p - head * HALF, pos = sh.pos[r];
                        if (head < a.nq + a.nkv) {
                          const float cs = __ldg(a.cos_tab + (size_t)pos * HALF + c), sn = __ldg(a.sin_tab + (size_t)pos * HALF + c);
                          const float t = v0 * cs - v1 * sn;
                          v1 = v1 * cs + v0 * sn;
                          v0 = t;
                        }
                        float *dst;
                        if (head < a.nq) dst = a.q + ((size_t)r * a.nq + head) * HD;
                        else {
                          const int kvh = (head - a.nq) % a.nkv;
                          dst = (head < a.nq + a.nkv ? ly.k_pool : ly.v_pool) + (((size_t)kvh * a.n_pages + sh.pg[r]) * a.page + pos % a.page) * HD;
                        }
                        dst[c] = v0;
                        dst[c + HALF] = v1;
                      });
    if (!barrier(a, target, sh)) return;
    attention_phase<HD>(a, ly, sh, first);
    if (!barrier(a, target, sh)) return;
    auto add = [&](int p, int r, float v0, float v1) {
      float2 *dst = reinterpret_cast<float2 *>(a.x + (size_t)r * a.d + 2 * p);
      const float2 old = __ldcg(dst);
      *dst = make_float2(old.x + v0, old.y + v1);
    };
    product_phase<RT>(sh, [&](int r) { return (const float *)(a.att + (size_t)r * nqd); }, nullptr, 0.f, nqd, a.R, a.d / 2,
                      [&](int p, const float *&w0, const float *&w1) { w0 = ly.w[4] + (size_t)2 * p * nqd; w1 = w0 + nqd; }, add);
    if (!barrier(a, target, sh)) return;
    row_scales(sh, xr, a.R, a.d, a.eps);
    product_phase<RT>(sh, xr, ly.w[5], a.eps, a.d, a.R, a.ff,
                      [&](int p, const float *&w0, const float *&w1) { w0 = ly.w[6] + (size_t)p * a.d; w1 = ly.w[7] + (size_t)p * a.d; },
                      [&](int p, int r, float g, float u) { a.act[(size_t)r * a.ff + p] = g / (1.f + __expf(-g)) * u; });
    if (!barrier(a, target, sh)) return;
    product_phase<RT>(sh, [&](int r) { return (const float *)(a.act + (size_t)r * a.ff); }, nullptr, 0.f, a.ff, a.R, a.d / 2,
                      [&](int p, const float *&w0, const float *&w1) { w0 = ly.w[8] + (size_t)2 * p * a.ff; w1 = w0 + a.ff; }, add);
    if (l + 1 < a.n_run || a.L > 0)
      if (!barrier(a, target, sh)) return;
  }
  if (a.L > 0) {
    auto xl = [&](int r) { return (const float *)(a.x + (size_t)a.rows.src()[r] * a.d); };
    row_scales(sh, xl, a.L, a.d, a.eps);
    product_phase<RT>(sh, xl, a.final_norm, a.eps, a.d, a.L, (a.V + 1) / 2,
                      [&](int p, const float *&w0, const float *&w1) {
                        w0 = a.lm_head + (size_t)2 * p * a.d;
                        w1 = 2 * p + 1 < a.V ? w0 + a.d : w0;
                      },
                      [&](int p, int r, float v0, float v1) {
                        float *dst = a.logits + (size_t)a.rows.dst(r) * a.V + 2 * p;
                        dst[0] = v0;
                        if (2 * p + 1 < a.V) dst[1] = v1;
                      });
  }
}

template <int RT, int HD> int launch_t(const SmallFwdArgs &a, int grid, cudaStream_t s) {
  void *params[1] = {const_cast<SmallFwdArgs *>(&a)};
  HSD_CUDA_OK(cudaLaunchCooperativeKernel((const void *)fwd_small_kernel<RT, HD>, dim3(grid), dim3(kThreads), params, 0, s));
  hsd_count_launches(1);
  return HSD_OK;
}
template <int HD> int launch_hd(const SmallFwdArgs &a, int grid, cudaStream_t s) {
  const int rows = std::max(a.R, a.L);
  if (rows <= 4) return launch_t<4, HD>(a, grid, s);
  if (rows <= 8) return launch_t<8, HD>(a, grid, s);
  return launch_t<16, HD>(a, grid, s);
}

}  // namespace

// Small: where launches and not weights take the time.  8 MB of weights a layer are about 2 us of the phases' loads on
// 148 SMs; a much larger model streams its weights better with the many CTAs of one launch per operation.  Passes of models of
// width 512 to 2048 with a vocabulary of 32000 (us, launches per operation / this kernel; 1 row through one layer, about 25
// through two, about 43 through four, a prompt's 128 through four):
//   8.4 MB a layer   81 / 63    384 / 215    1056 / 507     2170 / 815       (just on this kernel's side)
//   16.7             91 / 83    430 / 265    1267 / 679     2700 / 1256
//   25.2            111 / 113   533 / 435    1424 / 1006    3000 / 1764
//   45              129 / 145   577 / 518    1693 / 1336    3720 / 2555
//   180             209 / 295  1203 / 1251   3321 / 3105    7750 / 6680
// So the line lies on the safe side: up to about 25 MB next to nothing would be slower in this kernel.
bool fwd_small_supported(const ModelDims &md) {
  const long long layer = ((long long)md.d * md.hd * (2 * md.nq + 2 * md.nkv) + 3ll * md.d * md.ff) * 4;
  return md.dtype == HSD_F32 && (md.hd == 32 || md.hd == 64 || md.hd == 128) && md.d % 4 == 0 && md.ff % 4 == 0 && (md.nq * md.hd) % 4 == 0 &&
         layer <= (8ll << 20) && (long long)md.V * md.d * 4 <= (64ll << 20);
}
int fwd_small_grid(const ModelDims &md, int sm_count) {
  const int pairs = std::max({(md.nq + 2 * md.nkv) * md.hd / 2, md.ff, md.V / 2});
  return std::max(1, std::min(sm_count, ceil_div(pairs, kWarps)));
}

int launch_forward_small(const SmallFwdArgs &a, int grid, cudaStream_t s) {
  if (a.R < 1 || a.R > kSmallRows || a.L > kSmallRows) return HSD_E_INVALID_ARG;
  switch (a.hd) {
    case 128: return launch_hd<128>(a, grid, s);
    case 64: return launch_hd<64>(a, grid, s);
    case 32: return launch_hd<32>(a, grid, s);
    default: return HSD_E_UNSUPPORTED;
  }
}

}  // namespace hsd
