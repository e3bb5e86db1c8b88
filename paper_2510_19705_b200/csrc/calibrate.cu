// Calibration of the hierarchy search (Section 4.2 needs the acceptance rate alpha_{i,j} of every drafter i
// under every verifier j; Section 2: alpha = 1 - TV(p_i, p_j) = sum_x min(p_i(x), p_j(x))).  Given the logits of
// L models (exit layers) at the same R positions, the kernels below produce the L x L matrix of the rates
// averaged over the positions.
//   1. alpha_stats_kernel:   per (model, position): reference exponent and sum of exp (fp32, fixed order, one read of the row)
//   2. alpha_pairs_kernel:   per (position, <= 4096-token unit): every pair's sum of minima over the unit -> one partial per pair
//   3. alpha_reduce_kernel:  per pair: the partials of all positions and units added in fixed order in fp64
// The three are a chain of launches, early where it pays, which itself starts under the end of what is on the stream: 100 positions
// of 24 models over 2048 tokens 30 us (36 as ordinary launches), 20 of 5 over 17001 17 (18).
// Deterministic (no atomics).  Model pairs are enumerated i < j, pair index = i L - i (i + 1) / 2 + (j - i - 1).
#include <cuda_bf16.h>
#include <math.h>
#include <type_traits>

#include "../../include/hsd.h"
#include "common.cuh"

namespace hsd {
namespace {

constexpr int kAlphaThreads = 256;
constexpr int kAlphaTile = 256;        // units are multiples of this many tokens
constexpr int kAlphaUnit = 4096;       // tokens per partial at most: 128 per lane, all added in fp32
constexpr int kAlphaMaxModels = 32;

template <typename T> struct AlphaVec;         // 16 bytes of logits
template <> struct AlphaVec<__nv_bfloat16> {
  static constexpr int N = 8;
  __device__ static void unpack(const uint4 &v, float *f) {
    f[0] = __uint_as_float(v.x << 16); f[1] = __uint_as_float(v.x & 0xFFFF0000u);
    f[2] = __uint_as_float(v.y << 16); f[3] = __uint_as_float(v.y & 0xFFFF0000u);
    f[4] = __uint_as_float(v.z << 16); f[5] = __uint_as_float(v.z & 0xFFFF0000u);
    f[6] = __uint_as_float(v.w << 16); f[7] = __uint_as_float(v.w & 0xFFFF0000u);
  }
};
template <> struct AlphaVec<float> {
  static constexpr int N = 4;
  __device__ static void unpack(const uint4 &v, float *f) {
    f[0] = __uint_as_float(v.x); f[1] = __uint_as_float(v.y); f[2] = __uint_as_float(v.z); f[3] = __uint_as_float(v.w);
  }
};

constexpr float kLog2e = 1.4426950408889634f;
__device__ __forceinline__ float alpha_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Weight of a logit relative to 2^n, n a whole number: exp(x) 2^-n.  Numerators and sums use the same expression, so
// the approximation's own bias cancels in their quotient.
__device__ __forceinline__ float alpha_weight(float x, float n, float scale = kLog2e) { return alpha_ex2(fmaf(x, scale, -n)); }
// The reference n is off by half its last bit, 2^32 in the weights at |n| = 2^30, which fp32 holds.  Past that (and in a row
// of nothing but its type's lowest value, n = -inf) a logit below the maximum is below it by 32 or more: those rows take
// scale 1 and the maximum itself as n, exactly 1 at the maximum and 2^-32 at most elsewhere.  Their sums carry the sign bit.
constexpr float kAlphaFar = 1073741824.f;

// Online sum of exp of a thread, relative to 2^n with 2^n at or above the largest exp so far: a larger n rescales the
// sum by a power of two, exactly.
struct RefSum {
  float n = -INFINITY, s = 0.f;
  __device__ void raise(float n2) {
    if (n2 > n) {
      s *= n > -INFINITY ? __int_as_float((int)(fmaxf(n - n2, -126.f) + 127.f) << 23) : 0.f;
      n = n2;
    }
  }
  __device__ void merge(float n2, float s2) {
    RefSum o;
    o.n = n2; o.s = s2;
    const float nn = fmaxf(n, n2);
    raise(nn);
    o.raise(nn);
    s += o.s;
  }
};

// Bound by HBM: 16-byte loads when VEC (rows on 16-byte boundaries), four in flight per thread.
template <typename T, bool VEC>
__global__ void __launch_bounds__(kAlphaThreads)
alpha_stats_kernel(const T *__restrict__ logits, long long model_stride, int R, int V, float2 *__restrict__ stats) {
  __shared__ float shm[kAlphaThreads / 32], shs[kAlphaThreads / 32];
  chain_wait();
  chain_next();                                                       // (behind the wait: the pairs' first logits are read ahead of theirs)
  const int r = blockIdx.x, l = blockIdx.y;                           // (positions x models may pass 2^31)
  const T *row = logits + (size_t)l * model_stride + (size_t)r * V;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int N = VEC ? AlphaVec<T>::N : 1, U = 4;
  RefSum ms;
  const int nv = V / N;
  for (int k0 = threadIdx.x; k0 < nv; k0 += kAlphaThreads * U) {
    float f[U][N];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int k = k0 + u * kAlphaThreads;
#pragma unroll
      for (int e = 0; e < N; ++e) f[u][e] = -INFINITY;
      if (k < nv) {
        if constexpr (VEC) AlphaVec<T>::unpack(__ldg(reinterpret_cast<const uint4 *>(row) + k), f[u]);
        else f[u][0] = to_f32(row[k]);
      }
    }
    float mx = -INFINITY;
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int e = 0; e < N; ++e) mx = fmaxf(mx, f[u][e]);
    ms.raise(ceilf(mx * kLog2e));
    if (ms.n > -INFINITY) {
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int e = 0; e < N; ++e) ms.s += alpha_weight(f[u][e], ms.n);
    }
  }
  for (int o = 16; o > 0; o >>= 1) ms.merge(__shfl_xor_sync(0xFFFFFFFFu, ms.n, o), __shfl_xor_sync(0xFFFFFFFFu, ms.s, o));
  if (lane == 0) { shm[warp] = ms.n; shs[warp] = ms.s; }
  __syncthreads();
  RefSum t;
  for (int w = 0; w < kAlphaThreads / 32; ++w) t.merge(shm[w], shs[w]);     // the same in every thread
  if (fabsf(t.n) <= kAlphaFar) {
    if (threadIdx.x == 0) stats[(size_t)l * R + r] = make_float2(t.n, t.s);
    return;
  }
  __syncthreads();
  float m = -INFINITY, s = 0.f;
  for (int k = threadIdx.x; k < V; k += kAlphaThreads) m = fmaxf(m, to_f32(row[k]));
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
  if (lane == 0) shm[warp] = m;
  __syncthreads();
  for (int w = 0; w < kAlphaThreads / 32; ++w) m = fmaxf(m, shm[w]);
  for (int k = threadIdx.x; k < V; k += kAlphaThreads) s += alpha_weight(to_f32(row[k]), m, 1.f);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
  if (lane == 0) shs[warp] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    float tot = 0.f;
    for (int w = 0; w < kAlphaThreads / 32; ++w) tot += shs[w];
    stats[(size_t)l * R + r] = make_float2(m, __int_as_float(__float_as_int(tot) | (int)0x80000000));
  }
}

// Sum over the lanes of 64 values per lane: lane i returns the sums of values 2 i and 2 i + 1 (fixed order).
__device__ __forceinline__ float2 warp_sum64(float *v, int lane) {
  // each step halves the values: a lane keeps the half its bit selects and gives the other to its partner
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < 2 * o; ++i) {
      const float keep = up ? v[2 * o + i] : v[i], give = up ? v[i] : v[2 * o + i];
      v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, o);
    }
  }
  return make_float2(v[0], v[1]);
}
__device__ __forceinline__ int pair_index(int i, int j, int L) { return i * L - i * (i + 1) / 2 + (j - i - 1); }

// Sums of minima of a block of eight models against another (KIND 0), or of the pairs i < j of one block (KIND 1, 2),
// over the lane's tokens of one staged tile.  acc[i][jj] = the pairs (i, 2 jj) and (i, 2 jj + 1).  A diagonal block uses
// the entries i <= 2 jj; a second one (KIND 2) is kept in the other half, entry (i, jj) at [7 - i][3 - jj].
// Bound by instruction issue: a minimum per pair and token, one packed add per two pairs; 16 shared-memory loads feed
// 64 pairs.
template <int KIND, int STRIDE>
__device__ __forceinline__ void alpha_block(const float *pi, const float *pj, int tokens, int step, float2 (*acc)[4]) {
  for (int k = 0; k < tokens; k += step) {
    float a[8], b[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) a[i] = pi[i * STRIDE + k];
#pragma unroll
    for (int j = 0; j < 8; ++j) b[j] = KIND ? a[j] : pj[j * STRIDE + k];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) {
        if (KIND && i > 2 * jj) continue;
        float2 &to = KIND == 2 ? acc[7 - i][3 - jj] : acc[i][jj];
        to = __fadd2_rn(to, make_float2(fminf(a[i], b[2 * jj]), fminf(a[i], b[2 * jj + 1])));
      }
  }
}

// Block r x units + u = unit u of position r (one dimension: any number of positions).  The unit's tokens go through
// shared memory TILE at a time as probabilities [model][token] (double-buffered: the next tile's logits are fetched under
// this tile's minima).  A warp owns one pair of 8-model blocks, or two diagonal blocks (about as much work), and the tokens
// lane + 32 slice, ...; with fewer blocks than warps the warps share a pair and split the tokens.
// 32 models x 256 positions x 32000 tokens: 478 us here + 97 us of statistics, each alone (a call 566 to 571); one pair per lane,
// two shared-memory loads per pair and token, took 5021 + 176 us.
// All 256 threads stage, so TILE x models is constant: 256 tokens of up to 32 models, 512 of 16, 1024 of 8.  (256 tokens of
// two models keep 16 threads busy: 2 x 256 x 32000 in fp32 153 us, this way 70.)
template <typename T, bool VEC, int TILE>
__global__ void __launch_bounds__(kAlphaThreads, TILE == 1024 && VEC && sizeof(T) == 2 ? 3 : 2)
alpha_pairs_kernel(const T *__restrict__ logits, long long model_stride, int L, int R, int V, int unit, int n_units,
                   const float2 *__restrict__ stats, float *__restrict__ partials) {
  constexpr int STRIDE = TILE + 8;                                    // floats between the models of a staged tile
  extern __shared__ float sm[];
  __shared__ float4 st[kAlphaMaxModels];
  const int r = blockIdx.x / n_units, u0 = (blockIdx.x - r * n_units) * unit, nt = min(unit, V - u0);
  const int nb = (L + 7) >> 3, lpad = nb * 8, n_off = nb * (nb - 1) / 2, n_task = n_off + (nb + 1) / 2;
  const int slices = max(1, 8 / n_task);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float *buf[2] = {sm, sm + (size_t)lpad * STRIDE};
  float *wsum = sm + 2 * (size_t)lpad * STRIDE;                 // [slice][task][64]
  const int n_pairs = L * (L - 1) / 2;
  auto load_stats = [&]() {                                           // (scale, reference exponent, 1 / sum)
    chain_wait();
    chain_next();
    if (tid >= lpad) return;
    const float2 v = tid < L ? __ldcg(stats + (size_t)tid * R + r) : make_float2(0.f, 0.f);
    const bool far = __float_as_int(v.y) < 0;
    st[tid] = make_float4(far ? 1.f : kLog2e, v.x, tid < L ? 1.f / fabsf(v.y) : 0.f, 0.f);
  };
  // bf16 in vectors: the first logits are asked for ahead of the statistics' end (24 models x 256 x 32000 434 us instead of 451; fp32,
  // with twice the registers for them, 538 instead of 531; single bf16 logits, 16 x 256 x 13001, 152 instead of 147)
  constexpr bool AHEAD = sizeof(T) == 2 && VEC;
  if constexpr (!AHEAD) { load_stats(); __syncthreads(); }
  // staging: TPM threads per model; vector i of a thread = tokens (TPM i + tid % TPM) N ..
  constexpr int N = VEC ? AlphaVec<T>::N : 1, TPM = TILE / 32, NV = 32 / N;
  const int sm_model = tid / TPM, sv = tid % TPM;
  const bool stager = sm_model < lpad, in_use = sm_model < L;
  const T *row = logits + (size_t)(in_use ? sm_model : 0) * model_stride + (size_t)r * V + u0;
  typename std::conditional<VEC, uint4, T>::type raw[NV];
  auto fetch = [&](int t0) {
    if (!in_use) return;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int k = t0 + (TPM * i + sv) * N;
      if (k < nt) {
        if constexpr (VEC) raw[i] = __ldg(reinterpret_cast<const uint4 *>(row + k));
        else raw[i] = row[k];
      }
    }
  };
  auto convert = [&](int t0, float *dst) {
    if (!stager) return;
    const float4 st4 = st[sm_model];
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int at = (TPM * i + sv) * N;
      float f[N];
#pragma unroll
      for (int e = 0; e < N; ++e) f[e] = 0.f;
      if (in_use && t0 + at < nt) {
        if constexpr (VEC) AlphaVec<T>::unpack(raw[i], f);
        else f[0] = to_f32(raw[i]);
#pragma unroll
        for (int e = 0; e < N; ++e) f[e] = alpha_weight(f[e], st4.y, st4.x) * st4.z;
      }
      float *d = dst + sm_model * STRIDE + at;
      if constexpr (VEC) {
#pragma unroll
        for (int e = 0; e < N; e += 4) *reinterpret_cast<float4 *>(d + e) = make_float4(f[e], f[e + 1], f[e + 2], f[e + 3]);
      } else d[0] = f[0];
    }
  };
  // this warp's task
  const int task = warp % n_task, slice = warp / n_task;
  const bool busy = slice < slices;
  int bi = 0, bj = 0;
  const bool diag = task >= n_off;
  if (diag) { bi = 2 * (task - n_off); bj = bi + 1; }                // two diagonal blocks (the second may not exist)
  else { int t = task; while (t >= nb - 1 - bi) { t -= nb - 1 - bi; ++bi; } bj = bi + 1 + t; }
  const bool two = bj < nb;
  float2 acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
  fetch(0);
  if constexpr (AHEAD) { load_stats(); __syncthreads(); }
  convert(0, buf[0]);
  __syncthreads();
  for (int t0 = 0, b = 0; t0 < nt; t0 += TILE, b ^= 1) {
    const bool more = t0 + TILE < nt;
    if (more) fetch(t0 + TILE);
    if (busy) {
      const float *p = buf[b] + slice * 32 + lane;
      const int tokens = TILE == 1024 ? min(TILE, nt - t0) - slice * 32 : TILE, step = 32 * slices;   // (the tile is zero past the unit's tokens)
      if (TILE == 1024) alpha_block<1, STRIDE>(p, nullptr, tokens, step, acc);    // one block of eight models
      else if (!diag) alpha_block<0, STRIDE>(p + bi * 8 * STRIDE, p + bj * 8 * STRIDE, tokens, step, acc);
      else {
        alpha_block<1, STRIDE>(p + bi * 8 * STRIDE, nullptr, tokens, step, acc);
        if (two) alpha_block<2, STRIDE>(p + bj * 8 * STRIDE, nullptr, tokens, step, acc);
      }
    }
    if (more) convert(t0 + TILE, buf[b ^ 1]);
    __syncthreads();
  }
  // lane sums; the slices of a task are added in slice order
  float *out = partials + (size_t)blockIdx.x * n_pairs;
  float v[64];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) { v[i * 8 + 2 * j] = acc[i][j].x; v[i * 8 + 2 * j + 1] = acc[i][j].y; }
  const float2 lane_sum = warp_sum64(v, lane);
  if (busy) *reinterpret_cast<float2 *>(wsum + (slice * n_task + task) * 64 + 2 * lane) = lane_sum;
  __syncthreads();
  if (!busy || slice != 0) return;
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int ai = lane / 4, ajj = lane % 4;                          // the accumulator entry of values 2 lane, 2 lane + 1
    int ib = bi, jb = bj, i = ai, j = 2 * ajj + e;
    if (diag) {
      if (ai <= 2 * ajj) jb = bi;
      else { if (!two) continue; ib = bj; i = 7 - ai; j = 2 * (3 - ajj) + e; }
    }
    i += ib * 8; j += jb * 8;
    if (i >= j || j >= L) continue;
    float t = 0.f;
    for (int sl = 0; sl < slices; ++sl) t += wsum[(sl * n_task + task) * 64 + 2 * lane + e];
    out[pair_index(i, j, L)] = t;
  }
}

__global__ void __launch_bounds__(kAlphaThreads)
alpha_reduce_kernel(const float *__restrict__ partials, int L, int n_blocks, int R, double *__restrict__ alpha) {
  __shared__ double sh[kAlphaThreads];
  chain_wait();
  chain_next();
  const int n_pairs = L * (L - 1) / 2;
  for (int pr = blockIdx.x; pr < n_pairs; pr += gridDim.x) {
    double s = 0.0;
    for (int b = threadIdx.x; b < n_blocks; b += kAlphaThreads) s += (double)__ldcg(partials + (size_t)b * n_pairs + pr);
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = kAlphaThreads / 2; o > 0; o >>= 1) {
      if ((int)threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
      __syncthreads();
    }
    if (threadIdx.x == 0) {
      int i = 0, rem = pr;
      while (rem >= L - 1 - i) { rem -= L - 1 - i; ++i; }
      const int j = i + 1 + rem;
      const double a = sh[0] / (double)R;
      alpha[(size_t)i * L + j] = a;
      alpha[(size_t)j * L + i] = a;
    }
    __syncthreads();
  }
  if (blockIdx.x == 0 && (int)threadIdx.x < L) alpha[(size_t)threadIdx.x * L + threadIdx.x] = 1.0;
}

struct AlphaPlan { int unit, n_units, n_pairs; size_t stats_off, partials_off, total; };
AlphaPlan alpha_plan(int L, int R, int V) {
  AlphaPlan p;
  // equal units of a multiple of the tile; shorter ones when the positions alone would not fill the SMs
  int n = (V + kAlphaUnit - 1) / kAlphaUnit;
  while ((long long)n * R < 4 * kMeasuredSMs && (V + n - 1) / n > 2 * kAlphaTile) n *= 2;
  p.unit = ((V + n - 1) / n + kAlphaTile - 1) / kAlphaTile * kAlphaTile;
  p.n_units = (V + p.unit - 1) / p.unit;
  p.n_pairs = L * (L - 1) / 2;
  p.stats_off = 0;
  p.partials_off = ((size_t)L * R * sizeof(float2) + 255) / 256 * 256;
  p.total = p.partials_off + (size_t)R * p.n_units * (p.n_pairs > 0 ? p.n_pairs : 1) * sizeof(float);
  return p;
}

template <typename T, bool VEC, int TILE>
int launch_pairs(const T *logits, long long model_stride, int L, int R, int V, const AlphaPlan &p, const float2 *stats, float *partials, bool early, cudaStream_t s) {
  const int lpad = (L + 7) / 8 * 8;
  const size_t smem = (2 * (size_t)lpad * (TILE + 8) + 8 * 64) * sizeof(float);
  static std::atomic<u64> limits{0};
  const int limit = hsd_smem_limit((const void *)alpha_pairs_kernel<T, VEC, TILE>, 100 * 1024, limits);
  if (limit) return limit;
  HSD_CUDA_OK(hsd_launch(alpha_pairs_kernel<T, VEC, TILE>, p.n_units * R, kAlphaThreads, smem, s, 0, early, logits, model_stride, L, R, V, p.unit, p.n_units,
                         stats, partials));
  return HSD_OK;
}

template <typename T, bool VEC>
int launch_alpha_t(const T *logits, long long model_stride, int L, int R, int V, void *ws, double *alpha, cudaStream_t s) {
  const AlphaPlan p = alpha_plan(L, R, V);
  float2 *stats = (float2 *)((char *)ws + p.stats_off);
  float *partials = (float *)((char *)ws + p.partials_off);
  HSD_CUDA_OK(hsd_launch(alpha_stats_kernel<T, VEC>, dim3(R, L), kAlphaThreads, 0, s, 0, true, logits, model_stride, R, V, stats));
  // CTAs that start early are packed on the SMs that the kernel before leaves first.  That costs more than the early start gives where
  // there are no more of them than SMs (a CTA's own time then counts), unless both kernels' fit side by side, and, for more than eight
  // models, in the reduction (us as ordinary launches / all early / this way: 32 models x 8 x 2048 13.2 / 16.6 / 12.6, x 32000 30.0 /
  // 33.4 / 29.2; fp32 32 x 8 x 8192 14.6 / 19.1 / 14.3; 8 x 20 x 2048 8.2 / 8.5 / 7.7; 10 x 1 x 2048 8.1 / 7.0 / 7.0; behind many waves, 32 x
  // 256 x 32000, the reduction takes the last one's places: 571 early, 568 not).
  const long long n_ctas = (long long)p.n_units * R;
  const bool fit = (long long)L * R + n_ctas <= kMeasuredSMs, pairs_early = fit || n_ctas > kMeasuredSMs,
             reduce_early = fit || (pairs_early && L <= 8 && n_ctas <= 6 * kMeasuredSMs);
  int st = HSD_OK;
  if (p.n_pairs > 0)
    st = L <= 8    ? launch_pairs<T, VEC, 1024>(logits, model_stride, L, R, V, p, stats, partials, pairs_early, s)
         : L <= 16 ? launch_pairs<T, VEC, 512>(logits, model_stride, L, R, V, p, stats, partials, pairs_early, s)
                   : launch_pairs<T, VEC, 256>(logits, model_stride, L, R, V, p, stats, partials, pairs_early, s);
  if (st) return st;
  HSD_CUDA_OK(hsd_launch(alpha_reduce_kernel, p.n_pairs > 0 ? min(p.n_pairs, 4 * kMeasuredSMs) : 1, kAlphaThreads, 0, s, 0, reduce_early, partials, L, R * p.n_units, R,
                         alpha));
  hsd_count_launches(p.n_pairs > 0 ? 3 : 2);
  return hsd_launch_status();
}

template <typename T>
int launch_alpha(const void *logits, long long model_stride, int L, int R, int V, void *ws, double *alpha, cudaStream_t s) {
  // 16-byte loads need every row on a 16-byte boundary and no partial vector at a row's end
  constexpr int N = AlphaVec<T>::N;
  const bool vec = V % N == 0 && model_stride % N == 0 && ((uintptr_t)logits & 15) == 0;
  return vec ? launch_alpha_t<T, true>((const T *)logits, model_stride, L, R, V, ws, alpha, s)
             : launch_alpha_t<T, false>((const T *)logits, model_stride, L, R, V, ws, alpha, s);
}

}  // namespace
}  // namespace hsd

extern "C" {

size_t hsd_pairwise_alpha_workspace_bytes(int n_models, int n_rows, int vocab) {
  if (n_models < 1 || n_models > hsd::kAlphaMaxModels || n_rows < 1 || vocab < 1) return 0;
  return hsd::alpha_plan(n_models, n_rows, vocab).total;
}

int hsd_pairwise_alpha(const void *logits, int dtype, int n_models, int n_rows, int vocab, long long model_stride,
                       void *workspace, size_t workspace_bytes, double *alpha, void *stream) {
  if (!logits || !workspace || !alpha) return HSD_E_INVALID_ARG;
  if (dtype != HSD_BF16 && dtype != HSD_F32) return HSD_E_INVALID_ARG;
  if (n_models < 1 || n_models > hsd::kAlphaMaxModels || n_rows < 1 || vocab < 1) return HSD_E_INVALID_ARG;
  if (model_stride < (long long)n_rows * vocab) return HSD_E_INVALID_ARG;
  if (((uintptr_t)workspace & 255) != 0 || workspace_bytes < hsd::alpha_plan(n_models, n_rows, vocab).total) return HSD_E_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  return dtype == HSD_BF16
             ? hsd::launch_alpha<__nv_bfloat16>(logits, model_stride, n_models, n_rows, vocab, workspace, alpha, s)
             : hsd::launch_alpha<float>(logits, model_stride, n_models, n_rows, vocab, workspace, alpha, s);
}

}  // extern "C"
