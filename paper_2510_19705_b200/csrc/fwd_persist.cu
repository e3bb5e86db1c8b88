// Persistent verifier forward (see fwd_persist.cuh).
//
// Warp roles (12 warps): 0 = weight-tile TMA producer, 1 = activation-tile TMA producer, 2 = TMEM
// owner + MMA issuer, 3 = spare, 4..7 = GEMM epilogue (each reads its own TMEM lane quarter) and
// phase workers, 8..11 = phase workers only.  The 256 worker threads walk the phase program
//   embed+norm | QKV(+rope, KV append) | attention | O(+residual) | norm | gate/up(+SwiGLU) |
//   down(+residual) | norm | ... | final norm | output head
// with a grid barrier before each projection that takes its activations by TMA, and behind a q / k / v finish of its own:
// the attention phase reads q and the cache, which are plain stores.  The other phases wait for the words they read
// (kHole).  The weight producer is not tied to the barriers: weights are
// read-only, so it runs ahead into the next GEMM as far as the ring allows; the activation producer
// waits for the barrier that completes its operand.  GEMM work is split evenly over the CTAs in
// (tile, k-block) units; each segment's partial sums go to a piece buffer and the following phase
// (the next RMSNorm for the residual projections, a short finish phase otherwise) adds them up.
// In decode passes two finish phases fold into their consumer: the attention phase finishes the
// q / k / v of its own rows, and with at most four rows the down projection's CTAs build their
// activation tiles from the gate / up pieces in shared memory (warps 5, 7, 9, 11).
// Every wait (mbarrier, grid barrier, words) is bounded by wall time and raises a status word.
//
// A parity wait sees a completion of its barrier only until the next one, so every waiter here is one that the next completion
// cannot do without, and has seen the one before:
//   full[slot]        MMA issuer: the slot's next tiles come behind empty[slot], which its commit completes
//   empty[slot]       weight producer, activation producer or builder: the next MMAs need the tile that each of them brings.
//                     Where the builders bring the activations, the activation producer counts the slots and does not wait:
//                     nothing there would wait for it.  (It finds its next slot's last completion but one behind it: that one
//                     came before the last built stage's weights, and those before the down words its next `ready` rests on.)
//   acc_full[b]       epilogue: the next MMAs come behind acc_empty[b], which its warps complete
//   acc_empty[b]      MMA issuer: the next epilogue needs its MMAs
//   ready[kind]       activation producer, in CTAs with tiles of that kind of projection: the next arrival, a layer later, comes
//                     behind this CTA's epilogue of those tiles.  The other CTAs' producers do not look at it
// In a tensor-memory attention item, per stream:
//   k_full, v_full    MMA issuer: the next loads come behind k_free / v_free, which its commits complete
//   k_free, v_free    loader: the next MMAs need its tile; softmax: they need its P (k_free doubles as "S complete")
//   p_ready           MMA issuer: the next P needs its S
// The weight producer's wait for the end of the attention phase has no such tie in CTAs without tiles: it compares a count.
#include <type_traits>
#include "fwd_persist.cuh"
#include "forward.cuh"
#include "gemm_tc.cuh"
#include "tc_ptx.cuh"

namespace hsd {
namespace {

using namespace ptx;

constexpr int kWBytes = kTcBlockM * kTcBlockK * 2;     // 16 KiB weight tile
constexpr int kBoxBytes = kTcBoxRows * kTcBlockK * 2;  // 8 KiB TMA box
constexpr int kScratchBytes = 78 * 1024;               // union: epilogue staging / attention buffers, + rope cache
constexpr int kCtrlBytes = 4096;                       // barriers, flags, page-id cache, per-row info
constexpr int kSmemTotal = 232448;
constexpr int kMaxLayersSh = 64;                       // layers whose pointer table fits the control area

enum { MODE_QKV = 0, MODE_ADD = 1, MODE_SWIGLU = 2, MODE_LOGITS = 3 };

// Barrier-timeline stamps and cycle laps exist only in a profiling build (-DHSD_PROFILE).
#ifdef HSD_PROFILE
#define HSD_PROF(a) ((a).prof != nullptr)
#else
#define HSD_PROF(a) false
#endif

template <int NPAD> struct PCfg {
  static constexpr int kStageBytes = kWBytes + NPAD * kTcBlockK * 2;
  static constexpr int kStages = (kSmemTotal - 1024 - kCtrlBytes - kScratchBytes) / kStageBytes;
  static constexpr int kSmemBytes = kStages * kStageBytes + kScratchBytes + kCtrlBytes + 1024;
  static constexpr int kTmemCols = (2 * NPAD < 32) ? 32 : 2 * NPAD;
  static constexpr int kChunk = NPAD < 32 ? NPAD : 32;      // accumulator columns handled at a time
};

struct Gemm {
  const CUtensorMap *w[3];
  int seg_n[3];
  int n_segs, K, KB, n_tiles, mode, rows;
};

__device__ __forceinline__ Gemm make_gemm(const FwdArgs &a, int p) {
  Gemm g;
  const int l = p >> 2, j = p & 3;
  g.w[1] = g.w[2] = nullptr;
  g.seg_n[1] = g.seg_n[2] = 0;
  g.n_segs = 1;
  g.rows = a.R;
  if (l >= a.n_run) {                       // output head
    g.w[0] = a.wmaps + a.lm_map; g.seg_n[0] = a.V; g.K = a.d; g.mode = MODE_LOGITS; g.rows = a.L;
  } else if (j == 0) {
    const CUtensorMap *m = a.wmaps + l * 7;
    g.w[0] = m; g.w[1] = m + 1; g.w[2] = m + 2;
    g.seg_n[0] = a.nq * a.hd; g.seg_n[1] = g.seg_n[2] = a.nkv * a.hd;
    g.n_segs = 3; g.K = a.d; g.mode = MODE_QKV;
  } else if (j == 1) {
    g.w[0] = a.wmaps + l * 7 + 3; g.seg_n[0] = a.d; g.K = a.nq * a.hd; g.mode = MODE_ADD;
  } else if (j == 2) {
    g.w[0] = a.wmaps + l * 7 + 4; g.w[1] = a.wmaps + l * 7 + 5; g.seg_n[0] = g.seg_n[1] = a.ff;
    g.n_segs = 2; g.K = a.d; g.mode = MODE_SWIGLU;
  } else {
    g.w[0] = a.wmaps + l * 7 + 6; g.seg_n[0] = a.d; g.K = a.ff; g.mode = MODE_ADD;
  }
  g.KB = g.K / kTcBlockK;
  if (g.mode == MODE_SWIGLU) g.n_tiles = (g.seg_n[0] + kTcBoxRows - 1) / kTcBoxRows;
  else {
    g.n_tiles = 0;
    for (int s = 0; s < g.n_segs; ++s) g.n_tiles += (g.seg_n[s] + kTcBlockM - 1) / kTcBlockM;
  }
  return g;
}

struct Tile { int seg, row0, col0; };
__device__ __forceinline__ Tile tile_of(const Gemm &g, int tile) {
  Tile t;
  if (g.mode == MODE_SWIGLU) { t.seg = 0; t.row0 = tile * kTcBoxRows; t.col0 = 0; return t; }
  int tt = tile, col0 = 0;
  for (int s = 0; s < g.n_segs; ++s) {
    int nt = (g.seg_n[s] + kTcBlockM - 1) / kTcBlockM;
    if (tt < nt || s == g.n_segs - 1) { t.seg = s; t.row0 = tt * kTcBlockM; t.col0 = col0; return t; }
    tt -= nt;
    col0 += g.seg_n[s];
  }
  t.seg = 0; t.row0 = 0; t.col0 = 0;
  return t;
}
// Unit arithmetic in 32 bits (the launcher checks n_tiles * KB * grid < 2^31).
__device__ __forceinline__ int cta_begin(int U, int G, int c) { return (int)(((unsigned)U * (unsigned)c) / (unsigned)G); }
// CTA c owns units [floor(U c / G), floor(U (c + 1) / G)): the owner of unit u is the largest c with
// floor(U c / G) <= u, i.e. c < (u + 1) G / U, i.e. c = floor(((u + 1) G - 1) / U).
__device__ __forceinline__ int unit_owner(int U, int G, int u) {
  return (int)((((unsigned)u + 1u) * (unsigned)G - 1u) / (unsigned)U);
}
// Work of one CTA in one GEMM, a segment (tile, k-block range) at a time.  One SM can pull only its
// share of HBM bandwidth, so every GEMM is split evenly over all CTAs in (tile, k-block) units;
// each segment's partial sums go to a piece buffer and the next phase adds the pieces of a tile in
// fixed piece order (bit-reproducible; no CTA waits for another inside a GEMM).
struct Seg { int tile, kb0, kb1; };
struct SegIter { int tile, kb, left; };        // next k-block (tile, kb) and the k-blocks still to hand out
// regular: every tile is cut into `parts` equal k-ranges (GEMMs with few tiles: at most four pieces per
// tile, residual projections residual_parts(), so the consumer can fetch all of them in one batch);
// otherwise the (tile, k-block) units are dealt out evenly (tiles >= CTAs / 2: a tile then spans at most 3 CTAs).
struct SplitGeom { int U, Gp, pieces_max, parts; };
// The norm after a residual projection holds a row in registers, 16 float4 loads of pieces per thread at a time: 4 pieces
// of up to 4096 columns or 8 of up to 2048.  Width 2048 in 4 parts left 84 of 148 CTAs without a tile of O and down
// and put 22 k-blocks of down on each other one: 1B hierarchy, target pass 0.552 ms in 4 parts, 0.518 in 8.
__host__ __device__ __forceinline__ int residual_parts(int d) { return d <= 2048 ? 8 : 4; }
__host__ __device__ __forceinline__ SplitGeom split_geom(int n_tiles, int KB, int most, int G) {
  SplitGeom sg;
  sg.U = n_tiles * KB;
  if (n_tiles * 2 <= G) {
    const int fit = G / n_tiles < KB ? G / n_tiles : KB;
    sg.parts = most < fit ? most : fit;
    sg.Gp = n_tiles * sg.parts;
    sg.pieces_max = sg.parts;
  } else {
    sg.parts = 0;
    sg.Gp = G < sg.U ? G : sg.U;
    const int per = sg.U / sg.Gp;
    sg.pieces_max = (KB + per - 1) / per + 1;
  }
  return sg;
}
__device__ __forceinline__ SplitGeom split_geom(const Gemm &g, int G) {
  return split_geom(g.n_tiles, g.KB, g.mode == MODE_ADD ? residual_parts(g.seg_n[0]) : 4, G);
}
// What one CTA has to do in one kind of projection (0 QKV, 1 O, 2 gate / up, 3 down, 4 head): the same in every layer, so
// it is worked out once per launch and kept in shared memory (an integer division is ~100 cycles between a phase's barrier
// and its first load).  piece0: the CTA's piece of its first segment's tile; tiles it starts itself: piece 0.
struct PhaseGeom { int tile, kb, left, piece0, KB, pieces_max, parts, U, Gp; };
__device__ __forceinline__ int kind_of(const FwdArgs &a, int p) { return p < 4 * a.n_run ? p & 3 : 4; }
__device__ __forceinline__ SegIter seg_begin(const PhaseGeom &pg) {
  SegIter it;
  it.tile = pg.tile; it.kb = pg.kb; it.left = pg.left;
  return it;
}
__device__ __forceinline__ bool seg_next(const PhaseGeom &pg, SegIter &it, Seg &s) {
  if (it.left <= 0) return false;
  const int n = min(pg.KB - it.kb, it.left);
  s.tile = it.tile; s.kb0 = it.kb; s.kb1 = it.kb + n;
  it.left -= n; it.kb = 0; ++it.tile;
  return true;
}
__device__ __forceinline__ int piece_of(const PhaseGeom &pg, const Seg &s) { return s.kb0 > 0 ? pg.piece0 : 0; }
// Pieces of a tile: they belong to consecutive CTAs.
__device__ __forceinline__ int tile_pieces(const PhaseGeom &pg, int tile) {
  if (pg.parts) return pg.parts;
  return unit_owner(pg.U, pg.Gp, tile * pg.KB + pg.KB - 1) - unit_owner(pg.U, pg.Gp, tile * pg.KB) + 1;
}
__device__ __forceinline__ PhaseGeom phase_geom(const Gemm &g, int G, int c) {
  const SplitGeom sg = split_geom(g, G);
  PhaseGeom pg;
  pg.KB = g.KB; pg.pieces_max = sg.pieces_max; pg.parts = sg.parts; pg.U = sg.U; pg.Gp = sg.Gp;
  pg.tile = pg.kb = pg.left = pg.piece0 = 0;
  if (c < sg.Gp) {
    if (sg.parts) {
      pg.tile = c / sg.parts; pg.piece0 = c - pg.tile * sg.parts;
      pg.kb = cta_begin(g.KB, sg.parts, pg.piece0);
      pg.left = cta_begin(g.KB, sg.parts, pg.piece0 + 1) - pg.kb;
    } else {
      const int cur = cta_begin(sg.U, sg.Gp, c);
      pg.left = cta_begin(sg.U, sg.Gp, c + 1) - cur;
      pg.tile = cur / g.KB;
      pg.kb = cur - pg.tile * g.KB;
      pg.piece0 = c - unit_owner(sg.U, sg.Gp, pg.tile * g.KB);
    }
  }
  return pg;
}
// Phase p is a down projection whose activation tiles are built in place from the gate / up pieces.
__device__ __forceinline__ bool built_down(const FwdArgs &a, int p) { return a.fuse_gu && (p & 3) == 3 && p < 4 * a.n_run; }

// Handing partial sums to the next phase.  A word of the piece and partial buffers that has not been written holds kHole
// (a NaN no sum is stored as), and its reader takes it as soon as it holds something else: the data is its own flag.  A
// counter or barrier in between costs a release that waits until every store of the CTA is in L2 (1 to 1.8 us under the weight
// stream), the flag's way, and then the loads; polling the data costs the loads.  Words are accessed with relaxed
// single-word semantics and depend on no order among themselves.  The words' writer makes them holes again one phase and
// at least one grid barrier after their readers (put_holes), and at least one grid barrier before the next ones, so
// between launches all words are holes.
constexpr unsigned kHole = 0xFFFFFFFFu;
__device__ __forceinline__ void put_word(float *p, float v) {
  const unsigned w = __float_as_uint(v) == kHole ? 0x7FFFFFFFu : __float_as_uint(v);
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(w) : "memory");
}
__device__ __forceinline__ void put_hole(float *p) { asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(kHole) : "memory"); }
__device__ __forceinline__ void put_holes2(float *p) { asm volatile("st.relaxed.gpu.global.v2.u32 [%0], {%1, %1};" ::"l"(p), "r"(kHole) : "memory"); }
__device__ __forceinline__ void put_words2(float *p, float x, float y) {
  const unsigned wx = __float_as_uint(x) == kHole ? 0x7FFFFFFFu : __float_as_uint(x), wy = __float_as_uint(y) == kHole ? 0x7FFFFFFFu : __float_as_uint(y);
  asm volatile("st.relaxed.gpu.global.v2.u32 [%0], {%1, %2};" ::"l"(p), "r"(wx), "r"(wy) : "memory");
}
__device__ __forceinline__ float get_word(const float *p) {
  unsigned w;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(w) : "l"(p) : "memory");
  return __uint_as_float(w);
}
__device__ __forceinline__ float2 get_words2(const float *p) {
  unsigned w[2];
  asm volatile("ld.relaxed.gpu.global.v2.u32 {%0, %1}, [%2];" : "=r"(w[0]), "=r"(w[1]) : "l"(p) : "memory");
  return make_float2(__uint_as_float(w[0]), __uint_as_float(w[1]));
}
__device__ __forceinline__ float4 get_words4(const float *p) {
  unsigned w[4];
  asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "l"(p) : "memory");
  return make_float4(__uint_as_float(w[0]), __uint_as_float(w[1]), __uint_as_float(w[2]), __uint_as_float(w[3]));
}
// A thread's N vectors of words: load(i, v[i]) is asked once for all, then again for those that still hold a hole, for 2 s at
// most or until another CTA has given up (then this one does: what the caller goes on with is never used).  Asking for all of
// them again each time made a look at a row's 64 KB of pieces 1.2 us long; the status word is looked at every 256 rounds, about
// 0.2 ms, because the look costs a trip to L2 of its own.
__device__ __forceinline__ unsigned top(float v) { return __float_as_uint(v); }
__device__ __forceinline__ unsigned top(const float2 &v) { return max(top(v.x), top(v.y)); }
__device__ __forceinline__ unsigned top(const float4 &v) { return max(max(top(v.x), top(v.y)), max(top(v.z), top(v.w))); }
template <int N, class V, class Load>
__device__ __forceinline__ void settle_words(V (&v)[N], const Load &load, volatile int *abort_flag, const int *status) {
  unsigned long long t0 = 0;
  for (unsigned it = 1;; ++it) {
    unsigned seen = 0u;
#pragma unroll
    for (int i = 0; i < N; ++i) seen = max(seen, top(v[i]));
    if (seen != kHole) return;
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (top(v[i]) == kHole) load(i);
    if ((it & 15u) != 0u) continue;
    if (*abort_flag) return;
    const unsigned long long now = globaltimer_ns();
    if (t0 == 0) t0 = now;
    else if (now - t0 > kWaitLimitNs || ((it & 255u) == 0u && *reinterpret_cast<const volatile int *>(status) != 0)) { *abort_flag = 1; return; }
  }
}
template <int N, class V, class Load>
__device__ __forceinline__ void fetch_words(V (&v)[N], const Load &load, volatile int *abort_flag, const int *status) {
#pragma unroll
  for (int i = 0; i < N; ++i) load(i);
  settle_words(v, load, abort_flag, status);
}
__device__ __forceinline__ void worker_sync() { asm volatile("bar.sync 2, 256;" ::: "memory"); }
// The same barrier with a vote: true in every worker thread if `gone` is in any.  Pipeline roles raise the CTA's flag at any
// time, so threads that read it one after the other may differ; a thread that left for that reason alone would be missing at
// the others' next barrier, for good.
__device__ __forceinline__ bool worker_sync_any(bool gone) {
  uint32_t any;
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.or.pred q, 2, 256, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
               : "=r"(any) : "r"(gone ? 1u : 0u) : "memory");
  return any != 0;
}
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, 128;" ::: "memory"); }
// barrier of one 128-thread worker group (id 1 = warps 4..7, the epilogue group; id 3 = warps 8..11)
__device__ __forceinline__ void group_sync(int id) { asm volatile("bar.sync %0, 128;" ::"r"(id) : "memory"); }
__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// A warp's wait for a count in shared memory that only grows.  Looks are 64 ns apart: the softmax warps of the attention phase
// it waits for issue from the same scheduler.
__device__ __forceinline__ bool count_wait_warp(const unsigned *count, unsigned want, volatile int *abort_flag) {
  const unsigned long long t0 = globaltimer_ns();
  for (;;) {
    unsigned v;
    asm volatile("ld.acquire.cta.shared.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(count)) : "memory");
    if (__all_sync(0xFFFFFFFFu, v >= want)) return true;
    if (__any_sync(0xFFFFFFFFu, *abort_flag != 0 || globaltimer_ns() - t0 > kWaitLimitNs)) { *abort_flag = 1; return false; }
    __nanosleep(64);
  }
}

// Grid-wide barrier of the worker threads; false, in all of them, once a wait of the CTA has given up.  `epoch` counts
// barriers; the counter only grows.
// If ready_bar != 0 the spinning thread then releases the activation producer for the next GEMM.
__device__ __forceinline__ bool grid_barrier(const FwdArgs &a, unsigned &epoch, volatile int *abort_flag, int wt,
                                             uint32_t ready_bar) {
  // The CTA's writes of this phase are ordered before the arrival by the CTA barrier plus ONE release at gpu
  // scope by the arriving thread (cumulative over what it has observed through the barrier), instead of a
  // fence in every thread.
  // The activations this phase wrote with plain stores are read by the next GEMM's TMA loads (async proxy):
  // every writer orders its generic-proxy writes before async-proxy accesses here, ahead of the release.
  if (ready_bar) asm volatile("fence.proxy.async.global;" ::: "memory");
  if (worker_sync_any(*abort_flag != 0)) return false;
  ++epoch;
  bool gone = false;
  if (wt == 0) {
    const unsigned target = epoch * gridDim.x;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.grid_counter) : "memory");
    if (HSD_PROF(a) && 2 * epoch + 1 < (unsigned)kFwdProfEvents) a.prof[(size_t)blockIdx.x * kFwdProfEvents + 2 * epoch] = globaltimer_ns();
    unsigned long long t0 = 0;                       // the clock is read only once the wait has lasted a while
    for (uint32_t it = 0; (int)(ld_acquire_u32(a.grid_counter) - target) < 0; ++it) {
      if ((it & 31u) == 31u) {
        const unsigned long long now = globaltimer_ns();
        if (t0 == 0) t0 = now;
        if (*abort_flag || *reinterpret_cast<volatile int *>(a.status) != 0 || now - t0 > kWaitLimitNs) {
          gone = true;
          break;
        }
      }
    }
    if (gone) {
      *abort_flag = 1;
      atomicExch(a.status, 1);
    } else {
      if (HSD_PROF(a) && 2 * epoch + 1 < (unsigned)kFwdProfEvents)
        a.prof[(size_t)blockIdx.x * kFwdProfEvents + 2 * epoch + 1] = globaltimer_ns();
      // the acquire load that left the spin orders everything after it; the CTA barrier below hands that on
      if (ready_bar) {
        mbar_arrive(ready_bar);
      }
    }
  }
  return !worker_sync_any(gone);
}

// ------------------------------------------------------------------------------ RMSNorm phase
// One row per CTA turn, held in registers (all loads issued before their first use).
//   src_embed: the row comes from the embedding table (and is copied to x).
//   pend_pieces: split pieces (np per tile) of the residual-add projection that ran just before; they are added to
//              the row in fixed piece order (x <- x + p_0 + p_1 + ...) and x is written back.
// Requires d % 4 == 0 and d <= 1024 MAXV.
template <int NPAD, int MAXV>                              // MAXV float4 slots per thread: rows of up to 1024 MAXV columns
__device__ __forceinline__ void norm_phase(const FwdArgs &a, int n_rows, const int *row_list, bool src_embed,
                                           const float *pend_pieces, int np, const __nv_bfloat16 *gain, __nv_bfloat16 *dst,
                                           float *red, int wt, volatile int *abort_flag) {
  constexpr int PB = 16 / MAXV;                            // pieces per slot (residual_parts)
  const int d = a.d, nvec = d >> 2;
  // the last CTAs first: some hold no tile of the projection.  The other rows fall to CTAs that do; their epilogue warps
  // write the CTA's words before they come here, so no CTA waits for itself
  const int first = (int)(gridDim.x - 1 - blockIdx.x);
  for (int i = first; i < n_rows; i += gridDim.x) {
    const int row = row_list ? row_list[i] : i;
    float *xrow = a.x + (size_t)row * d;
    float4 v[MAXV];
    if (src_embed) {
      // an id outside the vocabulary (only possible after non-finite logits) must not become an address
      const int tok = min(max(a.tokens[(size_t)a.rows.seq()[row] * a.max_seq + a.rows.pos()[row]], 0), a.V - 1);
      const __nv_bfloat16 *erow = a.embed + (size_t)tok * d;
      uint2 raw[MAXV];
#pragma unroll
      for (int j = 0; j < MAXV; ++j) {
        const int iv = wt + 256 * j;
        raw[j] = iv < nvec ? __ldg(reinterpret_cast<const uint2 *>(erow) + iv) : make_uint2(0u, 0u);
      }
#pragma unroll
      for (int j = 0; j < MAXV; ++j)
        v[j] = make_float4(__uint_as_float(raw[j].x << 16), __uint_as_float(raw[j].x & 0xFFFF0000u),
                           __uint_as_float(raw[j].y << 16), __uint_as_float(raw[j].y & 0xFFFF0000u));
    } else {
#pragma unroll
      for (int j = 0; j < MAXV; ++j) {
        const int iv = wt + 256 * j;
        v[j] = iv < nvec ? __ldcg(reinterpret_cast<const float4 *>(xrow) + iv) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
    uint2 graw[MAXV];
#pragma unroll
    for (int j = 0; j < MAXV; ++j) {
      const int iv = wt + 256 * j;
      graw[j] = iv < nvec ? __ldg(reinterpret_cast<const uint2 *>(gain) + iv) : make_uint2(0u, 0u);
    }
    if (pend_pieces) {
      // every piece of every slot in one batch of loads: the residual projections have at most d / 128
      // = 32 tiles, so they are always cut the regular way (the launcher checks it), np <= PB pieces per
      // tile at a fixed stride
      float4 t[MAXV * PB];
      const float *base[MAXV];
#pragma unroll
      for (int j = 0; j < MAXV; ++j) {
        const int k = (wt + 256 * j) << 2;
        base[j] = pend_pieces + ((size_t)(k >> 7) * np * NPAD + row) * kTcBlockM + (k & 127);
      }
      fetch_words(t, [&](int i) {
        const int j = i / PB, pp = i % PB;
        t[i] = (wt + 256 * j < nvec && pp < np) ? get_words4(base[j] + (size_t)pp * NPAD * kTcBlockM) : make_float4(0.f, 0.f, 0.f, 0.f);
      }, abort_flag, a.status);
#pragma unroll
      for (int j = 0; j < MAXV; ++j)
#pragma unroll
        for (int pp = 0; pp < PB; ++pp) {
          const float4 &e = t[j * PB + pp];
          v[j].x += e.x; v[j].y += e.y; v[j].z += e.z; v[j].w += e.w;
        }
    }
    float ss = 0.f;
#pragma unroll
    for (int j = 0; j < MAXV; ++j) ss += v[j].x * v[j].x + v[j].y * v[j].y + v[j].z * v[j].z + v[j].w * v[j].w;
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xFFFFFFFFu, ss, o);
    worker_sync();
    if ((wt & 31) == 0) red[wt >> 5] = ss;
    worker_sync();
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) tot += red[w];
    const float inv = rsqrtf(tot / (float)d + a.eps);
#pragma unroll
    for (int j = 0; j < MAXV; ++j) {
      const int iv = wt + 256 * j;
      if (iv < nvec) {
        if (src_embed || pend_pieces) reinterpret_cast<float4 *>(xrow)[iv] = v[j];
        const float g0 = __uint_as_float(graw[j].x << 16), g1 = __uint_as_float(graw[j].x & 0xFFFF0000u);
        const float g2 = __uint_as_float(graw[j].y << 16), g3 = __uint_as_float(graw[j].y & 0xFFFF0000u);
        __nv_bfloat162 lo = __floats2bfloat162_rn(v[j].x * inv * g0, v[j].y * inv * g1);
        __nv_bfloat162 hi = __floats2bfloat162_rn(v[j].z * inv * g2, v[j].w * inv * g3);
        uint2 out;
        out.x = *reinterpret_cast<unsigned *>(&lo);
        out.y = *reinterpret_cast<unsigned *>(&hi);
        reinterpret_cast<uint2 *>(dst + (size_t)i * d)[iv] = out;
      }
    }
  }
}

// ------------------------------------------------------------------------------ attention phases
// Under the weight stream every dependent global round trip costs microseconds, so the attention is
// two phases.  Phase A: work item = (attention item, KV head, key split), partial (o, m, l) to global
// memory.  Phase B (after a grid barrier): one (row, head) per 128 threads merges the partials of its
// splits.
constexpr int kRopeCacheRows = 12;                     // rows whose cos / sin values are kept in shared memory
constexpr int kAttnMaxSplits = 20;

__device__ __forceinline__ void cp_async16(void *smem_dst, const void *gsrc) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(smem_dst)), "l"(gsrc) : "memory");
}

struct LayerCache { __nv_bfloat16 *k_pool, *v_pool; };
__device__ __forceinline__ LayerCache cache_of(const FwdArgs &a, int l) {
  LayerCache lc;
  lc.k_pool = reinterpret_cast<__nv_bfloat16 *>(a.k_pool + a.pool_stride * l);
  lc.v_pool = reinterpret_cast<__nv_bfloat16 *>(a.v_pool + a.pool_stride * l);
  return lc;
}
struct PageCache { int tag_item; int pg[128]; };   // pg[warp * 16 + j]: page of the warp's j-th sub-tile

__device__ __forceinline__ void mma_bf16_16x8x16(float *c, const unsigned *a, unsigned b0, unsigned b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// Four 8x8 b16 matrices; lane l gives the address of row l % 8 of matrix l / 8; register i of lane (g, t) holds
// matrix i's elements [g][2t .. 2t + 1] (.trans: [2t .. 2t + 1][g]).
__device__ __forceinline__ void ldmatrix_x4(unsigned *r, const void *row_ptr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_u32(row_ptr)));
}
__device__ __forceinline__ void ldmatrix_x4_trans(unsigned *r, const void *row_ptr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_u32(row_ptr)));
}

// ------------------------------------------------------------------------------ long key ranges on tcgen05
// One work item (attention item, KV head, key split) with a long key range, head size 128, at most 32 query
// vectors.  Keys go through in tiles of 64, dealt to two independent streams (tile j to stream j & 1), each with
// its own running reference maximum, row sums and output accumulator; per tile
//   S[128 x 64]   = Q[128 (<= 32 real rows) x 128] K_tile[64 x 128]^T       tcgen05.mma, both operands K-major
//   P             = exp2((S - m_ref) scale log2 e)  as bf16, row per thread  (m_ref moves only when a row maximum
//                                                                             passes it by a factor 256: then O is rescaled)
//   O[128 x 128] += P[128 x 64] V_tile[64 keys x 128]                        V as the MN-major B operand, as it lies in the cache
// S and O live in tensor memory (S double-buffered per stream: 2 x 2 x 64 columns, O 2 x 128: all 512 columns,
// the GEMM accumulators are idle during this phase).  Rows 32..127 of the A operands are whatever shared memory
// follows the real rows: their results are never read.  The eight worker warps: per stream (warps 0-3 / 4-7) warp
// 0 = softmax (the only one whose TMEM lane quarter holds real rows), warp 1 = K tiles (three buffers: a K buffer
// is free as soon as S is complete), warp 2 = V tiles (two buffers), warp 3 = MMA issue (one elected lane).  Shared memory:
// the weight ring and the attention scratch together (the weight producer does not run ahead over this phase).
constexpr int kTcaTile = 64, kTcaKBufs = 3, kTcaVBufs = 2;
constexpr int kTcaTileBytes = 2 * kTcaTile * 128;                 // two 64-column blocks of [64 keys][128 B]
constexpr int kTcaOffK = 8192, kTcaOffV = kTcaOffK + 2 * kTcaKBufs * kTcaTileBytes, kTcaOffP = kTcaOffV + 2 * kTcaVBufs * kTcaTileBytes;
constexpr int kTcaOffBar = kTcaOffP + 4 * 4096 + 12288, kTcaBytes = kTcaOffBar + 256;
constexpr int kTcaMinKeys = 1920;                                 // shorter key ranges stay on the mma.sync path (the host plans splits of
                                                                  // 2048 keys and more; the last split of a range may fall a little short)
static_assert(kTcaBytes <= 4 * (kWBytes + 128 * kTcBlockK * 2) + kScratchBytes - 2 * 12 * 64 * 4, "tcgen05 attention buffers exceed the ring + scratch");

__device__ __forceinline__ uint64_t umma_desc_mn(uint32_t smem_addr, uint32_t lbo_bytes) {   // MN-major, 128-byte swizzle
  uint64_t d = (uint64_t)((smem_addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)(lbo_bytes >> 4) << 16;                          // between the 64-element blocks along N
  d |= (uint64_t)(1024 >> 4) << 32;                               // between the 8-row groups along K
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float *o) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
               ::"r"(taddr), "r"(__float_as_uint(o[0])), "r"(__float_as_uint(o[1])), "r"(__float_as_uint(o[2])),
               "r"(__float_as_uint(o[3])), "r"(__float_as_uint(o[4])), "r"(__float_as_uint(o[5])), "r"(__float_as_uint(o[6])),
               "r"(__float_as_uint(o[7])), "r"(__float_as_uint(o[8])), "r"(__float_as_uint(o[9])), "r"(__float_as_uint(o[10])),
               "r"(__float_as_uint(o[11])), "r"(__float_as_uint(o[12])), "r"(__float_as_uint(o[13])), "r"(__float_as_uint(o[14])),
               "r"(__float_as_uint(o[15])) : "memory");
}

struct TcaItem { int row0, nrows, seq, pos0, kvh, split, key_lo, key_hi, nqv, group; };

// False, in every thread of the CTA, if a wait gave up.
__device__ __noinline__ bool attn_item_tc(const FwdArgs &a, const __nv_bfloat16 *kpool, const __nv_bfloat16 *vpool, uint8_t *smem,
                                          uint32_t tmem, const TcaItem it, int wt, volatile int *abort_flag, long long *dbg) {
  constexpr int HD = 128, TK = kTcaTile, NKB = kTcaKBufs, NVB = kTcaVBufs;
  const uint32_t s0 = smem_u32(smem), b0 = s0 + kTcaOffBar;
  // per stream s: k_free[3] (= S complete) k_full[3] v_full[2] v_free[2] p_ready[2]
  auto k_full = [&](int s, int b) { return b0 + 8u * (s * 12 + b); };
  auto k_free = [&](int s, int b) { return b0 + 8u * (s * 12 + 3 + b); };
  auto v_full = [&](int s, int b) { return b0 + 8u * (s * 12 + 6 + b); };
  auto v_free = [&](int s, int b) { return b0 + 8u * (s * 12 + 8 + b); };
  auto p_ready = [&](int s, int b) { return b0 + 8u * (s * 12 + 10 + b); };
  const int warp = __shfl_sync(0xFFFFFFFFu, wt >> 5, 0), lane = wt & 31, s = warp >> 2, role = warp & 3;
#ifdef HSD_PROFILE
  // profiling build: CTA 0's first softmax warp laps its set-up [5], waits for S [6], softmax up to P ready [7] and the
  // item's end [8]; [9] counts the items
  long long cyc = clock64();
  auto lap = [&](int k) { if (a.prof && wt == 0 && blockIdx.x == 0) { const long long n_ = clock64(); dbg[k] += n_ - cyc; cyc = n_; } };
  if (a.prof && wt == 0 && blockIdx.x == 0) dbg[9] += 1;
#else
  auto lap = [](int) {};
#endif
  if (wt == 0) {
    for (int ss = 0; ss < 2; ++ss) {
      for (int b = 0; b < NKB; ++b) { mbar_init(k_full(ss, b), 32); mbar_init(k_free(ss, b), 1); }
      for (int b = 0; b < NVB; ++b) { mbar_init(v_full(ss, b), 32); mbar_init(v_free(ss, b), 1); mbar_init(p_ready(ss, b), 1); }
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // Q: K-major, 128-byte swizzle, k-block kb (64 columns) at kb * 4096, rows 0..31 (rows past the item's vectors zero)
  for (int i = wt; i < 32 * 16; i += 256) {
    const int qi = i >> 4, c = i & 15, kb = c >> 3, cc = c & 7;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (qi < it.nqv) {
      const int r = qi / it.group, gq = qi - r * it.group;
      v = __ldcg(reinterpret_cast<const uint4 *>(a.q + ((size_t)(it.row0 + r) * a.nq + it.kvh * it.group + gq) * HD + c * 8));
    }
    *reinterpret_cast<uint4 *>(smem + kb * 4096 + (qi >> 3) * 1024 + (qi & 7) * 128 + ((cc ^ (qi & 7)) << 4)) = v;
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  tc_fence_before();
  worker_sync();
  tc_fence_after();
  lap(5);
  const int n_tiles = (it.key_hi - it.key_lo + TK - 1) / TK;
  const int n_mine = (n_tiles - s + 1) / 2;                      // tiles s, s + 2, ...
  const float sc = rsqrtf((float)HD) * 1.4426950408889634f;      // raw scores -> log2 units
  float m_ref = -INFINITY, l = 0.f;                              // the softmax warps' state (raw score units)
  bool ok = true;
  const uint32_t tS = tmem + (uint32_t)(s * 128), tO = tmem + 256u + (uint32_t)(s * 128);
  if (role == 1 || role == 2) {
    // ---------------- loader warp of one operand: LAG tiles in flight behind the one being issued
    const bool isk = role == 1;
    const int NB = isk ? NKB : NVB, LAG = isk ? 2 : 1;
    const __nv_bfloat16 *pool = isk ? kpool : vpool;
    const uint32_t base = isk ? kTcaOffK + s * NKB * kTcaTileBytes : kTcaOffV + s * NVB * kTcaTileBytes;
    const int *pt = a.page_table + (size_t)it.seq * a.pages_per_seq;
    for (int t = 0; t < n_mine + LAG; ++t) {
      if (t >= LAG) {                                            // tile t - LAG has landed: hand it over before anything can block
        if (isk) asm volatile("cp.async.wait_group 1;" ::: "memory");
        else asm volatile("cp.async.wait_group 0;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        const int tt = t - LAG;
        mbar_arrive(isk ? k_full(s, tt % NKB) : v_full(s, tt % NVB));
      }
      if (t < n_mine) {
        const int b = t % NB;
        if (t >= NB) {
          const int use = t / NB - 1;                            // completion number of the buffer's previous use
          if (lane == 0) mbar_wait(isk ? k_free(s, b) : v_free(s, b), (uint32_t)(use & 1), abort_flag);
          __syncwarp();
        }
        if (__any_sync(0xFFFFFFFFu, *abort_flag != 0)) break;
        const int key0 = it.key_lo + (2 * t + s) * TK;
        // the tile's four 16-key groups lie in one page each (pages hold >= 16 tokens, key ranges start on multiples of 16)
        int pg = 0;
        if (lane < 4 && key0 + lane * 16 < it.key_hi) pg = pt[(key0 + lane * 16) >> a.page_shift];
        const uint32_t tb = base + b * kTcaTileBytes;
        const int c = lane & 15, blk = c >> 3, cc = c & 7, h = lane >> 4;
        if (key0 + TK <= it.key_hi) {
          // a whole tile: per 16-key group one source base (its page) and eight copies per lane, rows 2 i + h; the
          // swizzled destination differs from row to row by compile-time constants only
          const uint32_t dst0 = s0 + tb + blk * (TK * 128) + h * 128;
          const int cch = cc ^ h;
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            const int pgr = __shfl_sync(0xFFFFFFFFu, pg, g);
            const __nv_bfloat16 *src = pool + ((((size_t)it.kvh * a.n_pages + pgr) << a.page_shift) + ((key0 + 16 * g) & (a.page - 1)) + h) * HD + c * 8;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const int r7 = (2 * i) & 7;                         // (row & 7) without h; row = 16 g + 2 i + h
              const uint32_t dst = dst0 + (uint32_t)((2 * g + (i >> 2)) * 1024 + r7 * 128) + (uint32_t)((cch ^ r7) << 4);
              asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src + (size_t)(2 * i) * HD) : "memory");
            }
          }
        } else {
#pragma unroll 4
          for (int i = 0; i < TK / 2; ++i) {
            const int r = 2 * i + h, key = key0 + r;
            const int pgr = __shfl_sync(0xFFFFFFFFu, pg, r >> 4);
            const uint32_t off = tb + blk * (TK * 128) + (r >> 3) * 1024 + (r & 7) * 128 + ((cc ^ (r & 7)) << 4);
            if (key < it.key_hi)
              cp_async16(smem + off, pool + ((((size_t)it.kvh * a.n_pages + pgr) << a.page_shift) + (key & (a.page - 1))) * HD + c * 8);
            else
              *reinterpret_cast<uint4 *>(smem + off) = make_uint4(0u, 0u, 0u, 0u);    // P is 0 there, V must be finite
          }
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
  } else if (role == 3) {
    // ---------------- MMA issue for stream s
    const bool issuer = elect_one();
    const uint32_t id1 = umma_idesc_bf16(TK), id2 = umma_idesc_bf16(HD) | (1u << 16);       // bit 16: B is MN-major
    auto issue_s = [&](int t) {                                   // S[t & 1] = Q K_t^T
      const int b = t % NKB;
      ok = mbar_wait_warp(k_full(s, b), (uint32_t)((t / NKB) & 1), abort_flag);
      if (!ok) return;
      if (issuer) {
#pragma unroll
        for (int ks = 0; ks < HD / 16; ++ks) {
          const uint64_t da = umma_desc(s0 + (ks >> 2) * 4096 + (ks & 3) * 32);
          const uint64_t db = umma_desc(s0 + kTcaOffK + (s * NKB + b) * kTcaTileBytes + (ks >> 2) * (TK * 128) + (ks & 3) * 32);
          umma_bf16(tS + (uint32_t)((t & 1) * 64), da, db, id1, ks > 0 ? 1u : 0u);
        }
        umma_commit(k_free(s, b));                                // S(t) complete = the K buffer is free
      }
    };
    if (n_mine > 0) issue_s(0);
    if (n_mine > 1 && ok) issue_s(1);
    for (int t = 0; t < n_mine && ok; ++t) {
      // P(t) is written (so S(t) has been read as well) and V(t) has landed
      ok = mbar_wait_warp(p_ready(s, t & 1), (uint32_t)((t >> 1) & 1), abort_flag);
      if (!ok) break;
      const int vb = t % NVB;
      ok = mbar_wait_warp(v_full(s, vb), (uint32_t)((t / NVB) & 1), abort_flag);
      if (!ok) break;
      tc_fence_after();
      if (issuer) {
        const uint32_t p_off = kTcaOffP + (s * 2 + (t & 1)) * 4096;
#pragma unroll
        for (int ks = 0; ks < TK / 16; ++ks) {
          const uint64_t da = umma_desc(s0 + p_off + ks * 32);
          const uint64_t db = umma_desc_mn(s0 + kTcaOffV + (s * NVB + vb) * kTcaTileBytes + ks * 2048, TK * 128);
          umma_bf16(tO, da, db, id2, (t > 0 || ks > 0) ? 1u : 0u);
        }
        umma_commit(v_free(s, vb));
      }
      if (t + 2 < n_mine) issue_s(t + 2);                         // its S buffer (t & 1) was read before P(t) was written
    }
  } else {
    // ---------------- stream s: softmax (thread = query vector `lane`)
    auto sync_ok = [&]() { ok = __shfl_sync(0xFFFFFFFFu, ok ? 1 : 0, 0) != 0; };
    const int qpos = it.pos0 + lane / it.group;                   // causal limit of this thread's query vector
    const bool real = lane < it.nqv;
    for (int t = 0; t < n_mine && ok; ++t) {
      if (lane == 0) ok = mbar_wait(k_free(s, t % NKB), (uint32_t)((t / NKB) & 1), abort_flag);
      sync_ok();
      if (!ok) break;
      lap(6);
      tc_fence_after();
      float sv[TK];
#pragma unroll
      for (int c = 0; c < TK; c += 16) tmem_ld16(tS + (uint32_t)((t & 1) * 64 + c), sv + c);
      tmem_ld_wait();
      const int key0 = it.key_lo + (2 * t + s) * TK;
      if (!real) {
#pragma unroll
        for (int c = 0; c < TK; ++c) sv[c] = 0.f;
      } else if (key0 + TK > it.key_hi || key0 + TK - 1 > qpos) {
#pragma unroll
        for (int c = 0; c < TK; ++c)
          if (key0 + c >= it.key_hi || key0 + c > qpos) sv[c] = -INFINITY;
      }
      float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
      for (int c = 0; c < TK; ++c) mx4[c & 3] = fmaxf(mx4[c & 3], sv[c]);
      const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
      // the reference maximum moves only when a row's maximum has passed it by more than 8 in log2 units
      const bool grow = (mx - m_ref) * sc > 8.f;                  // false while both are -inf (no key of the row so far)
      if (t == 0) m_ref = mx;
      else if (__any_sync(0xFFFFFFFFu, grow)) {
        // O of this stream is rescaled: its previous P V must be complete
        if (lane == 0) ok = mbar_wait(v_free(s, (t - 1) % NVB), (uint32_t)(((t - 1) / NVB) & 1), abort_flag);
        sync_ok();
        if (!ok) break;
        tc_fence_after();
        const float m_new = grow ? mx : m_ref;
        const float f = (m_new > -INFINITY && m_ref > -INFINITY) ? ex2_approx((m_ref - m_new) * sc) : (m_new > -INFINITY ? 0.f : 1.f);
#pragma unroll 1
        for (int c = 0; c < HD; c += 16) {
          float o[16];
          tmem_ld16(tO + (uint32_t)c, o);
          tmem_ld_wait();
#pragma unroll
          for (int e = 0; e < 16; ++e) o[e] *= f;
          tmem_st16(tO + (uint32_t)c, o);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        l *= f;
        m_ref = m_new;
      }
      // P buffer t & 1 was read by the P V of tile t - 2
      if (t >= 2) {
        if (lane == 0) ok = mbar_wait(v_free(s, (t - 2) % NVB), (uint32_t)(((t - 2) / NVB) & 1), abort_flag);
        sync_ok();
        if (!ok) break;
      }
      uint8_t *prow = smem + kTcaOffP + (s * 2 + (t & 1)) * 4096 + (lane >> 3) * 1024 + (lane & 7) * 128;
      const float mneg = m_ref > -INFINITY ? -m_ref * sc : 0.f;   // a row without keys so far: exp2(-inf) = 0 everywhere
      float l4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int c8 = 0; c8 < TK / 8; ++c8) {
        unsigned w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float p0 = ex2_approx(fmaf(sv[c8 * 8 + 2 * e], sc, mneg)), p1 = ex2_approx(fmaf(sv[c8 * 8 + 2 * e + 1], sc, mneg));
          l4[e] += p0 + p1;
          const __nv_bfloat162 pb = __floats2bfloat162_rn(p0, p1);
          w[e] = *reinterpret_cast<const unsigned *>(&pb);
        }
        *reinterpret_cast<uint4 *>(prow + ((c8 ^ (lane & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
      }
      l += (l4[0] + l4[1]) + (l4[2] + l4[3]);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(p_ready(s, t & 1));
      lap(7);
    }
    if (ok && n_mine > 0) {                                       // the stream's last P V
      const int tl = n_mine - 1;
      if (lane == 0) ok = mbar_wait(v_free(s, tl % NVB), (uint32_t)((tl / NVB) & 1), abort_flag);
      sync_ok();
    }
    tc_fence_after();
  }
  // ---- all MMAs of the item are complete once both softmax warps are here; stream 1 hands (O, m, l) to stream 0
  //      through shared memory (over the K buffers), stream 0 writes the item's result
  tc_fence_before();
  if (worker_sync_any(*abort_flag != 0)) return false;
  tc_fence_after();
  if (wt == 0)                                                    // nobody waits on the item's barriers any more: their memory
    for (int i = 0; i < 24; ++i)                                  // goes back to the weight ring / the next item
      asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(b0 + 8u * i) : "memory");
  float *xch = reinterpret_cast<float *>(smem + kTcaOffK);       // [32][HD + 2]
  if (role == 0 && s == 1) {
    if (n_mine > 0)
      for (int c = 0; c < HD; c += 16) {
        float o[16];
        tmem_ld16(tO + (uint32_t)c, o);
        tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 16; ++e) xch[lane * (HD + 2) + c + e] = o[e];
      }
    xch[lane * (HD + 2) + HD] = n_mine > 0 ? m_ref : -INFINITY;
    xch[lane * (HD + 2) + HD + 1] = n_mine > 0 ? l : 0.f;
  }
  tc_fence_before();
  worker_sync();
  if (role == 0 && s == 0) {
    const float m1 = xch[lane * (HD + 2) + HD], l1 = xch[lane * (HD + 2) + HD + 1];
    const float mm = fmaxf(m_ref, m1);
    const float f0 = m_ref > -INFINITY ? ex2_approx((m_ref - mm) * sc) : 0.f, f1 = m1 > -INFINITY ? ex2_approx((m1 - mm) * sc) : 0.f;
    const float lt = l * f0 + l1 * f1;
    const bool real = lane < it.nqv, wanted = it.key_lo <= it.pos0 + lane / it.group;   // (the merge phase reads a row's splits up to its own position)
    const int r = it.row0 + lane / it.group, hq = it.kvh * it.group + lane % it.group;
    float *dst = a.attn_partials + (((size_t)r * a.nq + hq) * a.n_splits + it.split) * (HD + 2);
    __nv_bfloat16 *adst = a.att + ((size_t)r * a.nq + hq) * HD;
    const float inv = lt > 0.f ? 1.f / lt : 0.f;
    for (int c = 0; c < HD; c += 16) {
      float o[16];
      tmem_ld16(tO + (uint32_t)c, o);
      tmem_ld_wait();
      if (real) {
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const float o1 = m1 > -INFINITY ? xch[lane * (HD + 2) + c + e] : 0.f;
          o[e] = (f0 > 0.f ? o[e] * f0 : 0.f) + o1 * f1;
        }
        if (a.n_splits == 1) {
#pragma unroll
          for (int e = 0; e < 16; e += 2)
            *reinterpret_cast<__nv_bfloat162 *>(adst + c + e) = __floats2bfloat162_rn(o[e] * inv, o[e + 1] * inv);
        } else if (wanted) {
#pragma unroll
          for (int e = 0; e < 16; e += 2) put_words2(dst + c + e, o[e], o[e + 1]);
        }
      }
    }
    if (real && wanted && a.n_splits > 1) put_words2(dst + HD, mm * rsqrtf((float)HD), lt);   // m in natural-log units, as the merge phase expects
    tc_fence_before();
  }
  lap(8);
  return true;
}

// Phase A: warp-level online softmax.  A work item is (attention item, KV head, key split); its keys
// are cut into 16-key sub-tiles (one KV page or part of one: the launcher requires pages of >= 16
// tokens) that the warps take in turn, each warp with its own running (m, l, O) in registers and its
// own K and V sub-tile buffers, so nothing synchronises the CTA inside the key loop.  S = Q K^T and
// O += P V run on mma.sync m16n8k16 (the S accumulators are re-packed as the A operand of P V; P is
// split into bf16 hi + lo halves, so P V keeps ~16 bits of P); K of the warp's next sub-tile is fetched
// under the softmax and P V of this one, the next V under the next Q K^T.  With up to 16 query vectors
// (rows x group) every warp works on its own sub-tiles; with 17..32 the warps pair up on a sub-tile,
// one 16-row m-tile each.  At the end the warps' states are merged through shared memory and the
// split's partial (o, m, l) goes to global memory.
// False, in every thread, if a wait of a tensor-memory item gave up.
template <int NPAD, int HD, bool TC>
__device__ __forceinline__ bool attn_tiles_phase(const FwdArgs &a, const LayerCache &lay, uint8_t *scratch, PageCache *pc, int wt, long long *dbg,
                                                 const int *first_item, const int *qkv_geom, const int *row_pg_sh, const float *rope_cos_sh,
                                                 const float *rope_sin_sh, uint8_t *tc_smem, uint32_t tmem, volatile int *abort_flag) {
  constexpr int CPR = HD / 8;                      // 16-byte chunks per row
  // Rows of Q, K, V in shared memory: HD >= 64: unpadded, the 16-byte chunk index XORed with the row's low
  // three bits; HD = 32: padded by 16 bytes.  Either way the fragment loads (eight rows, same chunk) and
  // ldmatrix (eight rows of one 8x8 block) touch all banks once.
  constexpr bool SWZ = HD >= 64;
  constexpr int RS = SWZ ? HD : HD + 8;            // row stride (bf16 elements)
  auto swz = [](int row, int chunk) { return SWZ ? (chunk ^ (row & 7)) : chunk; };
  constexpr int KST = HD / 16;                     // k-steps of Q K^T
  constexpr int NT = HD / 8;                       // 8-wide output n-tiles
  constexpr int MS = HD + 8;                       // merge row: o[HD], m, l; stride = 8 mod 32 words: conflict-free float2 stores
  const int group = a.nq / a.nkv;
  const int warp = wt >> 5, lane = wt & 31, g = lane >> 2, t = lane & 3;
  __nv_bfloat16 *shQ = reinterpret_cast<__nv_bfloat16 *>(scratch);                              // [32][RS]
  __nv_bfloat16 *shK = shQ + 32 * RS + warp * (32 * RS);                                        // this warp's [16][RS]
  __nv_bfloat16 *shV = shK + 16 * RS;                                                           // this warp's [16][RS]
  float *shMerge = reinterpret_cast<float *>(scratch);                                          // [8 warps][16][MS], over Q and the K/V buffers
  static_assert(8 * 16 * MS * 4 <= 9 * 32 * RS * 2, "merge area must fit the Q and K/V buffers");
  static_assert(9 * 32 * RS * 2 <= kScratchBytes - 2 * kRopeCacheRows * (HD / 2) * 4, "attention buffers overlap the rope cache");
  const __nv_bfloat16 *kpool = lay.k_pool, *vpool = lay.v_pool;
  const float scale = rsqrtf((float)HD), inv_group = 1.f / (float)group;
  const int n_work = a.n_attn * a.nkv * a.n_splits;
#pragma unroll 1
  for (int wi = blockIdx.x; wi < n_work; wi += gridDim.x) {
#ifdef HSD_PROFILE
    long long cyc = clock64();
    auto lap = [&](int k) { if (a.prof && wt == 0 && blockIdx.x == 0) { const long long n_ = clock64(); dbg[k] += n_ - cyc; cyc = n_; } };
#else
    auto lap = [](int) {};
#endif
    const int split = wi % a.n_splits, kvh = (wi / a.n_splits) % a.nkv, ai = wi / (a.n_splits * a.nkv);
    const int4 it = wi == (int)blockIdx.x ? make_int4(first_item[0], first_item[1], first_item[2], first_item[3])
                                          : a.rows.item(ai);   // the CTA's first item was fetched at kernel start
    const int row0 = it.x, nrows = it.y, seq = it.z, pos0 = it.w;
    const int kv_len = pos0 + nrows;
    const int key_lo = split * a.keys_per_split, key_hi = min(kv_len, key_lo + a.keys_per_split);
    if (key_lo >= kv_len) continue;                              // uniform over the CTA
    const int nqv = nrows * group, n_mt = (nqv + 15) >> 4;
    if (TC && HD == 128 && key_hi - key_lo >= kTcaMinKeys) {     // tensor memory path (uniform over the CTA)
      worker_sync();                                             // the previous item is done with the shared memory
      if (wt == 0) pc->tag_item = -1;
      TcaItem ti;
      ti.row0 = row0; ti.nrows = nrows; ti.seq = seq; ti.pos0 = pos0; ti.kvh = kvh; ti.split = split;
      ti.key_lo = key_lo; ti.key_hi = key_hi; ti.nqv = nqv; ti.group = group;
      if (!attn_item_tc(a, kpool, vpool, tc_smem, tmem, ti, wt, abort_flag, dbg)) return false;
      continue;
    }
    const int n_sub = (key_hi - key_lo + 15) >> 4;
    const int first = n_mt == 2 ? (warp >> 1) : warp, step = n_mt == 2 ? 4 : 8, mt = n_mt == 2 ? (warp & 1) : 0;
    const int n_mine = first < n_sub ? (n_sub - first + step - 1) / step : 0;       // sub-tiles of this warp
    worker_sync();                                               // previous item's merge area fully read
    // ---- q rows of the item (whole CTA) and this warp's page ids: lane j holds the page of the warp's j-th
    //      sub-tile (re-read every 32 sub-tiles); kept in shared memory across layers when the CTA has one item
    if (!a.fuse_qkv) {
      for (int i = wt; i < nqv * CPR; i += 256) {
        const int qi = i / CPR, ch = i % CPR;
        const int r = qi / group, gq = qi % group;
        cp_async16(shQ + qi * RS + swz(qi, ch) * 8, a.q + ((size_t)(row0 + r) * a.nq + kvh * group + gq) * HD + ch * 8);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const bool pages_cached = (pc->tag_item == wi) && n_mine <= 16;
    int pg_reg = 0, pg_base = 0;
    auto load_pages = [&](int j0) {                              // pages of sub-tiles j0 .. j0 + 31 of this warp
      pg_base = j0;
      const int j = j0 + lane;
      if (j < n_mine) {
        if (pages_cached) pg_reg = pc->pg[warp * 16 + j];
        else {
          const int key = key_lo + (first + j * step) * 16;
          pg_reg = a.page_table[(size_t)seq * a.pages_per_seq + (key >> a.page_shift)];
          if (n_mine <= 16) pc->pg[warp * 16 + j] = pg_reg;
        }
      }
    };
    load_pages(0);
    // `key_stop`: keys from there on are not fetched (fused QKV finish: the item's own new keys are written
    // straight into the buffers of a warp's first sub-tile by the threads that compute them)
    auto issue = [&](const __nv_bfloat16 *pool, __nv_bfloat16 *sh, int j, bool zero_pad, int key_stop) {    // one sub-tile, one operand
      const int kt = key_lo + (first + j * step) * 16, nk = min(16, key_hi - kt), nload = min(nk, key_stop - kt);
      const int pg = __shfl_sync(0xFFFFFFFFu, pg_reg, j - pg_base);
      const size_t base = ((((size_t)kvh * a.n_pages + pg) << a.page_shift) + (kt & (a.page - 1))) * HD;
#pragma unroll
      for (int i = 0; i < 16 * CPR / 32; ++i) {
        const int idx = i * 32 + lane, kk = idx / CPR, ch = idx % CPR;
        if (kk < nload) cp_async16(sh + kk * RS + swz(kk, ch) * 8, pool + base + (size_t)kk * HD + ch * 8);
        else if (zero_pad && kk >= nk) *reinterpret_cast<uint4 *>(sh + kk * RS + ch * 8) = make_uint4(0u, 0u, 0u, 0u);   // P is 0 there, V must be finite
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    constexpr int kAllKeys = 0x7FFFFFFF;
    const int first_stop = a.fuse_qkv ? pos0 : kAllKeys;
    if (n_mine > 0) { issue(kpool, shK, 0, false, first_stop); issue(vpool, shV, 0, true, first_stop); }
    else { asm volatile("cp.async.commit_group;\n\tcp.async.commit_group;" ::: "memory"); }
    if (a.fuse_qkv) {
      // ---- QKV finish of the item's own rows: pieces of the projection summed in piece order, rotary embedding,
      //      q -> the Q buffer, k / v of the rows whose position falls into this key split -> their cache page
      //      (and the first sub-tile's buffers, when that is where they belong).  A unit = 8 columns of one
      //      vector plus the 8 columns half a head further on (rotation partners): two 16-byte chunks.
      // geometry of the QKV projection's pieces (the same in every layer; worked out once at kernel start):
      // qg[0..6] = first tile of k, first tile of v, parts, pieces_max, U, Gp, KB
      constexpr int UPV = HD / 16, HALF = HD / 2;
      const int tile_k = qkv_geom[0], tile_v = qkv_geom[1], g_parts = qkv_geom[2], g_pmax = qkv_geom[3];
      const int nr_lo = max(0, key_lo - pos0), n_new = max(0, min(nrows, key_hi - pos0) - nr_lo);
      const int n_units = (nqv + 2 * n_new) * UPV;
      const bool rope_cached = a.R <= kRopeCacheRows;
      const size_t pstride = (size_t)NPAD * kTcBlockM;
#pragma unroll 1
      for (int u = wt; u < n_units; u += 256) {
        const int vec = u / UPV, c8 = u % UPV;
        int kind, rr, n, tile0;
        if (vec < nqv) { kind = 0; rr = (int)(((float)vec + 0.5f) * inv_group); n = (kvh * group + vec - rr * group) * HD; tile0 = 0; }
        else {
          const int v2 = vec - nqv, isv = v2 >= n_new ? 1 : 0;
          kind = 1 + isv; rr = nr_lo + v2 - isv * n_new; n = kvh * HD; tile0 = isv ? tile_v : tile_k;
        }
        n += c8 * 8;
        const int tile = tile0 + n / kTcBlockM, m = n % kTcBlockM;
        int n_pieces = g_parts;
        if (g_parts == 0) {                                      // dealt units: the owners of the tile's first and last k-block
          const int U = qkv_geom[4], Gp = qkv_geom[5], KB = qkv_geom[6];
          n_pieces = unit_owner(U, Gp, tile * KB + KB - 1) - unit_owner(U, Gp, tile * KB) + 1;
        }
        const float *base = a.pieces[0] + ((size_t)(tile * g_pmax) * NPAD + (row0 + rr)) * kTcBlockM + m;
        float4 pc4[16];                                          // [piece][low 0-3, low 4-7, high 0-3, high 4-7]
        fetch_words(pc4, [&](int i) {
          pc4[i] = (i >> 2) < n_pieces ? get_words4(base + (i >> 2) * pstride + (i & 1) * 4 + ((i >> 1) & 1) * HALF) : make_float4(0.f, 0.f, 0.f, 0.f);
        }, abort_flag, a.status);
        float cs[8], sn[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) { cs[e] = 1.f; sn[e] = 0.f; }
        if (kind < 2) {
          const float *ct = rope_cached ? rope_cos_sh + (row0 + rr) * HALF + c8 * 8 : a.cos_tab + (size_t)(pos0 + rr) * HALF + c8 * 8;
          const float *st = rope_cached ? rope_sin_sh + (row0 + rr) * HALF + c8 * 8 : a.sin_tab + (size_t)(pos0 + rr) * HALF + c8 * 8;
#pragma unroll
          for (int e = 0; e < 8; e += 4) {
            const float4 cv = *reinterpret_cast<const float4 *>(ct + e), sv = *reinterpret_cast<const float4 *>(st + e);
            cs[e] = cv.x; cs[e + 1] = cv.y; cs[e + 2] = cv.z; cs[e + 3] = cv.w;
            sn[e] = sv.x; sn[e + 1] = sv.y; sn[e + 2] = sv.z; sn[e + 3] = sv.w;
          }
        }
        float lo[8], hi[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) { lo[e] = 0.f; hi[e] = 0.f; }
#pragma unroll
        for (int pp = 0; pp < 4; ++pp) {
          lo[0] += pc4[4 * pp + 0].x; lo[1] += pc4[4 * pp + 0].y; lo[2] += pc4[4 * pp + 0].z; lo[3] += pc4[4 * pp + 0].w;
          lo[4] += pc4[4 * pp + 1].x; lo[5] += pc4[4 * pp + 1].y; lo[6] += pc4[4 * pp + 1].z; lo[7] += pc4[4 * pp + 1].w;
          hi[0] += pc4[4 * pp + 2].x; hi[1] += pc4[4 * pp + 2].y; hi[2] += pc4[4 * pp + 2].z; hi[3] += pc4[4 * pp + 2].w;
          hi[4] += pc4[4 * pp + 3].x; hi[5] += pc4[4 * pp + 3].y; hi[6] += pc4[4 * pp + 3].z; hi[7] += pc4[4 * pp + 3].w;
        }
        unsigned wl[4], wh[4];
#pragma unroll
        for (int e = 0; e < 8; e += 2) {
          const __nv_bfloat162 l2 = __floats2bfloat162_rn(lo[e] * cs[e] - hi[e] * sn[e], lo[e + 1] * cs[e + 1] - hi[e + 1] * sn[e + 1]);
          const __nv_bfloat162 h2 = __floats2bfloat162_rn(hi[e] * cs[e] + lo[e] * sn[e], hi[e + 1] * cs[e + 1] + lo[e + 1] * sn[e + 1]);
          wl[e >> 1] = *reinterpret_cast<const unsigned *>(&l2);
          wh[e >> 1] = *reinterpret_cast<const unsigned *>(&h2);
        }
        const uint4 vl = make_uint4(wl[0], wl[1], wl[2], wl[3]), vh = make_uint4(wh[0], wh[1], wh[2], wh[3]);
        if (kind == 0) {
          *reinterpret_cast<uint4 *>(shQ + vec * RS + swz(vec, c8) * 8) = vl;
          *reinterpret_cast<uint4 *>(shQ + vec * RS + swz(vec, c8 + CPR / 2) * 8) = vh;
        } else {
          const int pos = pos0 + rr;
          __nv_bfloat16 *pool = kind == 1 ? lay.k_pool : lay.v_pool;
          const size_t off = (((size_t)kvh * a.n_pages + row_pg_sh[row0 + rr]) * a.page + (pos & (a.page - 1))) * HD + c8 * 8;
          *reinterpret_cast<uint4 *>(pool + off) = vl;
          *reinterpret_cast<uint4 *>(pool + off + HALF) = vh;
          const int st = (pos - key_lo) >> 4, kk = (pos - key_lo) & 15;
          if (st < step) {                                       // a first sub-tile: its warp (pair) is waiting for these rows
            const int w0 = n_mt == 2 ? 2 * st : st;
            for (int ww = w0; ww < w0 + (n_mt == 2 ? 2 : 1); ++ww) {
              __nv_bfloat16 *sh = shQ + 32 * RS + ww * (32 * RS) + (kind == 2 ? 16 * RS : 0);
              *reinterpret_cast<uint4 *>(sh + kk * RS + swz(kk, c8) * 8) = vl;
              *reinterpret_cast<uint4 *>(sh + kk * RS + swz(kk, c8 + CPR / 2) * 8) = vh;
            }
          }
        }
      }
    }
    float o[NT][4];
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) o[n][e] = 0.f;
    float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};
    const int qrow[2] = {mt * 16 + g, mt * 16 + g + 8};          // query vectors of this thread's accumulator rows
    const int qpos[2] = {pos0 + qrow[0] / group, pos0 + qrow[1] / group};
    asm volatile("cp.async.wait_group 2;" ::: "memory");         // q rows landed (this thread's copies)
    worker_sync();                                               // ... and everybody's; page ids of the item stored
    if (wt == 0) pc->tag_item = (wi == (int)blockIdx.x && n_work <= (int)gridDim.x) ? wi : -1;
    lap(0);
#pragma unroll 1
    for (int j = 0; j < n_mine; ++j) {
      const int kt = key_lo + (first + j * step) * 16;
      if (j + 1 < n_mine && j + 1 - pg_base >= 32) load_pages(j + 1);
      lap(14);
      asm volatile("cp.async.wait_group 1;" ::: "memory");       // K of this sub-tile landed; V may be in flight
      __syncwarp();
      lap(10);
      // ---- S = Q K^T for 16 query vectors x 16 keys
      float sacc[2][4];
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) sacc[n][e] = 0.f;
      // fragments by ldmatrix: Q as the A operand (matrices: rows 0-7 / 8-15 x k 0-7 / 8-15), K as the B operand
      // of both 8-key n-tiles (keys 0-7 / 8-15 x k 0-7 / 8-15)
      {
        const int mi = lane >> 3, r8 = lane & 7;
        const int qrow_l = (mi & 1) * 8 + r8, krow_l = (mi >> 1) * 8 + r8;
        const __nv_bfloat16 *qbase = shQ + (mt * 16 + qrow_l) * RS, *kbase = shK + krow_l * RS;
#pragma unroll
        for (int ks = 0; ks < KST; ++ks) {
          unsigned af[4], bf4[4];
          ldmatrix_x4(af, qbase + swz(qrow_l, 2 * ks + (mi >> 1)) * 8);
          ldmatrix_x4(bf4, kbase + swz(krow_l, 2 * ks + (mi & 1)) * 8);
          mma_bf16_16x8x16(sacc[0], af, bf4[0], bf4[1]);
          mma_bf16_16x8x16(sacc[1], af, bf4[2], bf4[3]);
        }
      }
      __syncwarp();                                              // every lane is done with the K buffer
      lap(11);
      if (j + 1 < n_mine) issue(kpool, shK, j + 1, false, kAllKeys);
      else asm volatile("cp.async.commit_group;" ::: "memory");  // keep the group count uniform
      // ---- online softmax on the accumulator rows (g and g + 8); P re-packed as the A operand of P V
      unsigned ph[4], pl[4];
      float corr_h[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float sv[4];
        float mx = -INFINITY;
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int key = kt + n * 8 + 2 * t + e;
            float v = sacc[n][h * 2 + e] * scale;
            if (key >= key_hi || key > qpos[h] || qrow[h] >= nqv) v = -INFINITY;
            sv[n * 2 + e] = v;
            mx = fmaxf(mx, v);
          }
        mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 2));
        const float m_new = fmaxf(m_run[h], mx);
        const float corr = (m_new > -INFINITY) ? __expf(m_run[h] - m_new) : 1.f;
        float ps = 0.f, pv[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          pv[i] = (sv[i] > -INFINITY) ? __expf(sv[i] - m_new) : 0.f;
          ps += pv[i];
        }
        m_run[h] = m_new;
        l_run[h] = l_run[h] * corr + ps;                         // this thread's columns only; summed over t at the end
        corr_h[h] = corr;
#pragma unroll
        for (int n = 0; n < 2; ++n) {                            // A fragment: a[h] <- keys 2t.. of n-tile 0, a[2 + h] <- n-tile 1
          const __nv_bfloat162 hi = __floats2bfloat162_rn(pv[n * 2], pv[n * 2 + 1]);
          const float2 hf = __bfloat1622float2(hi);
          const __nv_bfloat162 lo = __floats2bfloat162_rn(pv[n * 2] - hf.x, pv[n * 2 + 1] - hf.y);
          ph[n * 2 + h] = *reinterpret_cast<const unsigned *>(&hi);
          pl[n * 2 + h] = *reinterpret_cast<const unsigned *>(&lo);
        }
      }
      lap(12);
      asm volatile("cp.async.wait_group 1;" ::: "memory");       // V of this sub-tile landed; the next K may be in flight
      __syncwarp();
      lap(13);
      // ---- O = O * corr + P V (the rescale is skipped while no row of the warp has a new maximum)
      if (__any_sync(0xFFFFFFFFu, corr_h[0] != 1.f || corr_h[1] != 1.f)) {
#pragma unroll
        for (int n = 0; n < NT; ++n) { o[n][0] *= corr_h[0]; o[n][1] *= corr_h[0]; o[n][2] *= corr_h[1]; o[n][3] *= corr_h[1]; }
      }
      {
        const int mi = lane >> 3, key_l = (mi & 1) * 8 + (lane & 7);
        const __nv_bfloat16 *vbase = shV + key_l * RS;
#pragma unroll
        for (int n = 0; n < NT; n += 2) {          // two 8-wide slices of the head dimension per ldmatrix
          unsigned bv[4];
          ldmatrix_x4_trans(bv, vbase + swz(key_l, n + (mi >> 1)) * 8);
          mma_bf16_16x8x16(o[n], ph, bv[0], bv[1]);
          mma_bf16_16x8x16(o[n], pl, bv[0], bv[1]);
          mma_bf16_16x8x16(o[n + 1], ph, bv[2], bv[3]);
          mma_bf16_16x8x16(o[n + 1], pl, bv[2], bv[3]);
        }
      }
      __syncwarp();                                              // every lane is done with the V buffer
      if (j + 1 < n_mine) issue(vpool, shV, j + 1, true, kAllKeys);
      else asm volatile("cp.async.commit_group;" ::: "memory");
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    lap(1);
    // ---- merge the warps' states: each warp writes (o, m, l) of its 16 query vectors over the K/V buffers
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      l_run[h] += __shfl_xor_sync(0xFFFFFFFFu, l_run[h], 1);
      l_run[h] += __shfl_xor_sync(0xFFFFFFFFu, l_run[h], 2);
    }
    worker_sync();                                               // all warps are done with their K/V buffers
    lap(2);
    {
      float *mine = shMerge + (size_t)warp * 16 * MS;
      if (n_mine > 0) {
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          if (qrow[0] < nqv) *reinterpret_cast<float2 *>(mine + g * MS + n * 8 + 2 * t) = make_float2(o[n][0], o[n][1]);
          if (qrow[1] < nqv) *reinterpret_cast<float2 *>(mine + (g + 8) * MS + n * 8 + 2 * t) = make_float2(o[n][2], o[n][3]);
        }
      }
      if (t == 0) {                                              // a warp without keys contributes m = -inf only
        mine[g * MS + HD] = m_run[0]; mine[g * MS + HD + 1] = l_run[0];
        mine[(g + 8) * MS + HD] = m_run[1]; mine[(g + 8) * MS + HD + 1] = l_run[1];
      }
    }
    worker_sync();
    lap(3);
#pragma unroll 1
    for (int idx = wt; idx < nqv * (HD / 2); idx += 256) {       // two output dims per thread
      const int qi = idx / (HD / 2), dd = (idx % (HD / 2)) * 2;
      const int w0 = n_mt == 2 ? (qi >> 4) : 0, wstep = n_mt == 2 ? 2 : 1, rr = qi & 15;
      const float *src0 = shMerge + ((size_t)w0 * 16 + rr) * MS;
      const int wstride = wstep * 16 * MS, nw = min(n_mt == 2 ? 4 : 8, n_sub);     // warps (pairs) that had keys
      // one pass, all loads of four warps' states in flight together
      float mm = -INFINITY, l = 0.f, ox = 0.f, oy = 0.f;
#pragma unroll 1
      for (int k0 = 0; k0 < nw; k0 += 4) {
        float mw[4], lw[4];
        float2 ov[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float *src = src0 + (k0 + i) * wstride;
          const bool on = k0 + i < nw;
          mw[i] = on ? src[HD] : -INFINITY;
          lw[i] = on ? src[HD + 1] : 0.f;
          ov[i] = on ? *reinterpret_cast<const float2 *>(src + dd) : make_float2(0.f, 0.f);
        }
        float mn = mm;
#pragma unroll
        for (int i = 0; i < 4; ++i) mn = fmaxf(mn, mw[i]);
        const float c0 = (mn > -INFINITY) ? __expf(mm - mn) : 1.f;
        l *= c0; ox *= c0; oy *= c0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float sc = (mw[i] > -INFINITY) ? __expf(mw[i] - mn) : 0.f;
          l += sc * lw[i]; ox += sc * ov[i].x; oy += sc * ov[i].y;
        }
        mm = mn;
      }
      const int r = row0 + qi / group, hq = kvh * group + qi % group;
      if (a.n_splits == 1) {                                     // the only split: this is the attention output
        *reinterpret_cast<__nv_bfloat162 *>(a.att + ((size_t)r * a.nq + hq) * HD + dd) = __floats2bfloat162_rn(ox / l, oy / l);
      } else if (key_lo <= pos0 + qi / group) {                  // (the merge phase reads a row's splits up to its own position)
        float *dst = a.attn_partials + (((size_t)r * a.nq + hq) * a.n_splits + split) * (HD + 2);
        put_words2(dst + dd, ox, oy);
        if (dd == 0) put_words2(dst + HD, mm, l);
      }
    }
    lap(4);
  }
  return true;
}

// Phase B: merge the split partials of one (row, head) per HD / 2 threads (two output dimensions each); a single
// batch of loads.
template <int HD>
__device__ __forceinline__ void attn_merge_phase(const FwdArgs &a, const int *row_pos_sh, int wt, volatile int *abort_flag) {
  constexpr int TPI = HD / 2, PER = 256 / TPI;                    // threads per item, items per CTA turn
  const int g = wt / TPI, dd = (wt % TPI) * 2;
  const int n_items = a.R * a.nq;
  for (int it = blockIdx.x * PER + g; it < n_items; it += PER * gridDim.x) {
    const int r = it / a.nq;
    const int used = min(a.n_splits, row_pos_sh[r] / a.keys_per_split + 1);   // splits holding keys <= own position
    const float *src = a.attn_partials + (size_t)it * a.n_splits * (HD + 2);
    float2 w[2 * kAttnMaxSplits];                                  // (m, l) and two output dimensions of every split
    fetch_words(w, [&](int i) {
      const int sp = i >> 1;
      w[i] = sp < used ? get_words2(src + sp * (HD + 2) + ((i & 1) ? dd : HD)) : ((i & 1) ? make_float2(0.f, 0.f) : make_float2(-INFINITY, 0.f));
    }, abort_flag, a.status);
    float m = -INFINITY;
#pragma unroll
    for (int s = 0; s < kAttnMaxSplits; ++s) m = fmaxf(m, w[2 * s].x);
    float l = 0.f, ox = 0.f, oy = 0.f;
#pragma unroll
    for (int s = 0; s < kAttnMaxSplits; ++s) {
      const float f = (w[2 * s].x > -INFINITY) ? __expf(w[2 * s].x - m) : 0.f;
      l += f * w[2 * s].y;
      ox += f * w[2 * s + 1].x;
      oy += f * w[2 * s + 1].y;
    }
    *reinterpret_cast<__nv_bfloat162 *>(a.att + (size_t)it * HD + dd) = __floats2bfloat162_rn(ox / l, oy / l);
  }
}

// ------------------------------------------------------------------------------ epilogue stores
// v[i] = final value of output feature (tile row m) for token row c0 + i.
template <int CH>
__device__ __forceinline__ void final_store(const FwdArgs &a, const Gemm &g, const Tile &ti, const LayerCache &lay, int m, int et,
                                            int c0, const float *v, float *staging, const int *rpos, const int *rpg,
                                            const float *cs, const float *sn, int bar_id) {
  const int rows = g.rows;
  if (g.mode == MODE_ADD) {
    // residual-add projections never get here: their pieces are summed by the next norm phase
  } else if (g.mode == MODE_LOGITS) {
    const int n = ti.row0 + m;
    if (n < g.seg_n[0]) {
#pragma unroll
      for (int i = 0; i < CH; ++i) {
        const int r = c0 + i;
        if (r < rows) a.logits[(size_t)a.rows.dst(r) * a.V + n] = __float2bfloat16_rn(v[i]);
      }
    }
  } else if (g.mode == MODE_SWIGLU) {
#pragma unroll
    for (int i = 0; i < CH; ++i) staging[m * (CH + 1) + i] = v[i];
    group_sync(bar_id);
    for (int idx = et; idx < kTcBoxRows * CH; idx += 128) {
      const int cc = idx % kTcBoxRows, i = idx / kTcBoxRows;
      const int r = c0 + i, col = ti.row0 + cc;
      if (r < rows && col < g.seg_n[0]) {
        const float gt = staging[cc * (CH + 1) + i], up = staging[(cc + kTcBoxRows) * (CH + 1) + i];
        a.act[(size_t)r * a.ff + col] = __float2bfloat16_rn(silu_mul(gt, up));
      }
    }
    group_sync(bar_id);
  } else {   // MODE_QKV: rotary embedding on q and k (cos / sin preloaded by the caller), then q -> buffer,
             // k / v -> their cache pages (row position and page id come from the per-launch row table)
#pragma unroll
    for (int i = 0; i < CH; ++i) staging[m * (CH + 1) + i] = v[i];
    group_sync(bar_id);
    const int n = ti.row0 + m;
    if (n < g.seg_n[ti.seg]) {
      const int hd = a.hd, half = hd >> 1;
      const int dd = n % hd, head = n / hd;
      const int mp = dd < half ? m + half : m - half;
#pragma unroll
      for (int i = 0; i < CH; ++i) {
        const int r = c0 + i;
        if (r < rows) {
          float out = v[i];
          if (ti.seg < 2) {
            const float pv = staging[mp * (CH + 1) + i];
            out = dd < half ? v[i] * cs[i] - pv * sn[i] : v[i] * cs[i] + pv * sn[i];
          }
          if (ti.seg == 0) {
            a.q[(size_t)r * g.seg_n[0] + n] = __float2bfloat16_rn(out);
          } else {
            const size_t off = (((size_t)head * a.n_pages + rpg[r]) * a.page + (rpos[r] & (a.page - 1))) * hd + dd;
            (ti.seg == 1 ? lay.k_pool : lay.v_pool)[off] = __float2bfloat16_rn(out);
          }
        }
      }
    }
    group_sync(bar_id);
  }
}

struct WorkerCtx {
  uint32_t tmem_base, accf_bar0, acce_bar0;      // accumulator-full / -empty barrier b = base + 8 b
  volatile int *abort_flag, *wait_ok;
  float *staging;
  const int *row_pos_sh, *row_pg_sh;
  const float *rope_cos_sh, *rope_sin_sh;
  const PhaseGeom *geom;                         // [5], by kind of projection
  int wt, lane, q, G, c;
  int seg_idx;
};

// This CTA's words of a projection become holes again (warps 8..11 while the others are in a later projection).
template <int NPAD>
__device__ __forceinline__ void put_holes(const FwdArgs &a, const WorkerCtx &w, int kind) {
  const PhaseGeom &pg = w.geom[kind];
  SegIter it = seg_begin(pg);
  Seg sg;
#pragma unroll 1
  while (seg_next(pg, it, sg)) {
    float *mine = a.pieces[kind] + ((size_t)sg.tile * pg.pieces_max + piece_of(pg, sg)) * NPAD * kTcBlockM + (w.wt & 127);
    for (int r = 0; r < a.R; ++r) put_hole(mine + r * kTcBlockM);
  }
}
// ... and its attention partials: a warp per query vector.
template <int HD>
__device__ __forceinline__ void put_partial_holes(const FwdArgs &a, int wt, const int *first_item) {
  const int group = a.nq / a.nkv, n_work = a.n_attn * a.nkv * a.n_splits;
  const float inv_group = 1.f / (float)group;
#pragma unroll 1
  for (int wi = blockIdx.x; wi < n_work; wi += gridDim.x) {
    const int unit = wi / a.n_splits, split = wi - unit * a.n_splits, ai = unit / a.nkv, kvh = unit - ai * a.nkv;
    const int4 it = wi == (int)blockIdx.x ? make_int4(first_item[0], first_item[1], first_item[2], first_item[3]) : a.rows.item(ai);
    const int key_lo = split * a.keys_per_split;
    if (key_lo >= it.w + it.y) continue;
    for (int qi = max(0, key_lo - it.w) * group + ((wt >> 5) & 3); qi < it.y * group; qi += 4) {       // rows from key_lo on wrote theirs
      const int r = (int)(((float)qi + 0.5f) * inv_group);
      float *dst = a.attn_partials + (((size_t)(it.x + r) * a.nq + kvh * group + qi - r * group) * a.n_splits + split) * (HD + 2);
      for (int e = wt & 31; e < HD / 2 + 1; e += 32) put_holes2(dst + 2 * e);
    }
  }
}

// GEMM phase p, epilogue side (warps 4..7): accumulator -> this CTA's piece of the tile.  Group-uniform:
// a give-up is decided by one thread and shared.
template <int NPAD>
__device__ __forceinline__ void gemm_epilogue(const FwdArgs &a, WorkerCtx &w, int p) {
  constexpr int CH = PCfg<NPAD>::kChunk;
  const int m = w.q * 32 + w.lane;

  const int kind = kind_of(a, p), rows = kind == 4 ? a.L : a.R;
  const PhaseGeom &pg = w.geom[kind];
  const bool keep = a.L > 0 || p != 4 * a.n_run - 1;            // a pass without logits ends here: nobody reads these pieces
  SegIter it = seg_begin(pg);
  Seg sg;
  for (; seg_next(pg, it, sg); ++w.seg_idx) {
    const int ab = w.seg_idx & 1;
    float *mine = a.pieces[kind] + ((size_t)sg.tile * pg.pieces_max + piece_of(pg, sg)) * NPAD * kTcBlockM;
    if (w.wt == 0) w.wait_ok[w.seg_idx & 1] = mbar_wait((w.accf_bar0 + 8u * ab), (uint32_t)((w.seg_idx >> 1) & 1), w.abort_flag) ? 1 : 0;
    epi_sync();
    if (!w.wait_ok[w.seg_idx & 1]) return;
    tc_fence_after();
    const uint32_t tbase = w.tmem_base + ((uint32_t)(w.q * 32) << 16) + (uint32_t)(ab * NPAD);
#pragma unroll 1
    for (int c0 = 0; c0 < NPAD; c0 += CH) {
      float v[CH];
#pragma unroll
      for (int j = 0; j < CH / 16; ++j) tmem_ld16(tbase + c0 + j * 16, v + j * 16);
      tmem_ld_wait();
      if (c0 + CH >= NPAD) {                   // accumulator fully read: hand it back to the MMA warp
        tc_fence_before();
        __syncwarp();
        if (w.lane == 0) mbar_arrive((w.acce_bar0 + 8u * ab));
      }
      if (c0 < rows && keep) {
#pragma unroll
        for (int i = 0; i < CH; ++i)
          if (c0 + i < rows) put_word(mine + (c0 + i) * kTcBlockM + m, v[i]);
      }
    }
  }
}

// Down projection p of a pass with at most four rows: the worker warps build its activation tiles straight into
// the ring slots (SwiGLU of the gate / up pieces, summed in piece order; k-block kb of the down projection is tile
// kb of gate / up), in the layout the activation TMA box would have had (128-byte rows, 16-byte chunk index XOR
// row & 7).  Builder warp i of four takes the CTA's stages i, i + 4, ...; a lane covers one row x 8 columns.  Under the weight
// stream a load from L2 takes longer than a ring slot's turn-around, so with at most two pieces per tile (PB = 2)
// a warp keeps the loads of its next two stages in flight (DEPTH = 2).
template <int NPAD, int PB, int DEPTH>
__device__ __forceinline__ void build_act_stages(const FwdArgs &a, WorkerCtx &w, int p, uint8_t *ring, uint32_t full_bar0,
                                                 uint32_t empty_bar0, volatile unsigned *ring_pos) {
  constexpr int STAGES = PCfg<NPAD>::kStages;
  // this CTA's k-blocks of the down projection (residual projections: one segment per CTA) and how the gate / up
  // tiles are cut into pieces
  const PhaseGeom &pgu = w.geom[2];
  const SegIter it = seg_begin(w.geom[3]);
  const int g_parts = pgu.parts, g_pmax = pgu.pieces_max, KBg = pgu.KB, Ug = pgu.U, Gpg = pgu.Gp;
  const float inv_U = 1.f / (float)Ug;
  // unit_owner without an integer division (all quantities < 2^24, so the float quotient is off by one at most)
  auto owner = [&](int u) {
    const int x = (u + 1) * Gpg - 1;
    int q = (int)((float)x * inv_U);
    const int rem = x - q * Ug;
    return rem < 0 ? q - 1 : (rem >= Ug ? q + 1 : q);
  };
  // builders: the four worker warps that share no scheduler with the weight producer or the MMA issuer (whose issue rate
  // bounds the phase)
  if (it.left <= 0 || ((w.wt >> 5) & 1) == 0) return;
  // ring position (slot, parity of its empty barrier) of the phase's first stage, published by the weight producer
  ring_pos += (p >> 2) & 15;
  unsigned rp = *ring_pos;
  if (!__all_sync(0xFFFFFFFFu, (int)(rp >> 16) == p)) {
    const unsigned long long t0 = globaltimer_ns();
    while (!__all_sync(0xFFFFFFFFu, (int)((rp = *ring_pos) >> 16) == p))
      if (__any_sync(0xFFFFFFFFu, *w.abort_flag != 0 || globaltimer_ns() - t0 > kWaitLimitNs)) { *w.abort_flag = 1; return; }
  }
  const int s0 = (int)(rp & 0xFFu), warp4 = w.wt >> 6, r = w.lane >> 3, c8 = w.lane & 7;
  const uint32_t par0 = (rp >> 8) & 1u;
  const bool on = r < a.R;
  const size_t pstride = (size_t)NPAD * kTcBlockM;
  const float *lane_base = a.pieces[2] + (size_t)r * kTcBlockM + c8 * 8;
  float4 t[DEPTH][PB * 4];                                     // [stage in flight][piece: gate 0-3, gate 4-7, up 0-3, up 4-7]
  auto load = [&](float4 (&dst)[PB * 4], int i, auto &&take) { // pieces of the CTA's stage i (this lane's row and columns)
    const int kb = it.kb + i;
    int n_pieces = 0;
    if (i < it.left && on) n_pieces = g_parts ? g_parts : owner(kb * KBg + KBg - 1) - owner(kb * KBg) + 1;
    const float *tbase = lane_base + (size_t)kb * g_pmax * pstride;
    take([&](int q) {
      dst[q] = (q >> 2) < n_pieces ? get_words4(tbase + (q >> 2) * pstride + (q & 1) * 4 + ((q >> 1) & 1) * kTcBoxRows) : make_float4(0.f, 0.f, 0.f, 0.f);
    });
  };
  auto ask = [&](auto &&one) {
#pragma unroll
    for (int q = 0; q < PB * 4; ++q) one(q);
  };
#pragma unroll
  for (int dpt = 0; dpt < DEPTH; ++dpt) load(t[dpt], warp4 + 4 * dpt, ask);
#pragma unroll 1
  for (int i0 = warp4; i0 < it.left; i0 += 4 * DEPTH) {
#pragma unroll
    for (int dpt = 0; dpt < DEPTH; ++dpt) {
      const int i = i0 + 4 * dpt;
      if (i >= it.left) break;
      const int pos = s0 + i, s = pos % STAGES;
      const uint32_t par = par0 ^ (uint32_t)((pos / STAGES) & 1);
      load(t[dpt], i, [&](auto &&one) { settle_words(t[dpt], one, w.abort_flag, a.status); });
      __syncwarp();
      bool ok = true;                                          // the slot is free once its previous MMAs have retired
      if (w.lane == 0) ok = mbar_wait(empty_bar0 + 8u * s, par, w.abort_flag);
      if (!__shfl_sync(0xFFFFFFFFu, ok ? 1 : 0, 0)) return;
      float gt[8], up[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) { gt[e] = 0.f; up[e] = 0.f; }
#pragma unroll
      for (int pp = 0; pp < PB; ++pp) {
        gt[0] += t[dpt][4 * pp + 0].x; gt[1] += t[dpt][4 * pp + 0].y; gt[2] += t[dpt][4 * pp + 0].z; gt[3] += t[dpt][4 * pp + 0].w;
        gt[4] += t[dpt][4 * pp + 1].x; gt[5] += t[dpt][4 * pp + 1].y; gt[6] += t[dpt][4 * pp + 1].z; gt[7] += t[dpt][4 * pp + 1].w;
        up[0] += t[dpt][4 * pp + 2].x; up[1] += t[dpt][4 * pp + 2].y; up[2] += t[dpt][4 * pp + 2].z; up[3] += t[dpt][4 * pp + 2].w;
        up[4] += t[dpt][4 * pp + 3].x; up[5] += t[dpt][4 * pp + 3].y; up[6] += t[dpt][4 * pp + 3].z; up[7] += t[dpt][4 * pp + 3].w;
      }
      if (on) {
        unsigned o[4];
#pragma unroll
        for (int e = 0; e < 8; e += 2) {
          const __nv_bfloat162 v2 = __floats2bfloat162_rn(silu_mul(gt[e], up[e]), silu_mul(gt[e + 1], up[e + 1]));
          o[e >> 1] = *reinterpret_cast<const unsigned *>(&v2);
        }
        uint8_t *slot = ring + (size_t)s * PCfg<NPAD>::kStageBytes + kWBytes;
        *reinterpret_cast<uint4 *>(slot + r * 128 + ((c8 ^ (r & 7)) << 4)) = make_uint4(o[0], o[1], o[2], o[3]);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the tensor core reads the tile through the async proxy
      __syncwarp();
      if (w.lane == 0) mbar_arrive(full_bar0 + 8u * s);
      load(t[dpt], i + 4 * DEPTH, ask);                          // this buffer's next stage
    }
  }
}

// Finish phase of GEMM p (QKV, gate/up, output head): units of (tile, block of up to 8 token rows)
// round-robin over the CTAs, two at a time (one per 128-thread group); the pieces of a tile (at most
// four) are added in piece order and the result goes through the projection's own epilogue.  The
// loads of the next four rows (pieces, rope values) are in flight while the current four are stored.
template <int NPAD>
__device__ __forceinline__ void gemm_finish(const FwdArgs &a, WorkerCtx &w, int p) {
  constexpr int RG = 4;                          // token rows per load batch (decode passes have few rows)
  constexpr int PBF = 4;                         // pieces per tile at most (regular: <= 4 parts; dealt units: <= 3)
  constexpr int RB = 8;                          // token rows per unit (two load batches; more units than 2 x CTAs at 24+ rows)
  const Gemm g = make_gemm(a, p);
  const PhaseGeom &pg = w.geom[kind_of(a, p)];
  float *const pieces = a.pieces[kind_of(a, p)];
  const int layer = p >> 2;
  const int gidx = w.wt >> 7, gm = w.wt & 127;   // two groups of 128 threads, one unit each at a time
  float *gstage = w.staging + gidx * (kTcBlockM * (RG + 1));
  const int n_rb = (g.rows + RB - 1) / RB, n_units = g.n_tiles * n_rb;
  const bool rope_cached = a.R <= kRopeCacheRows;
  if (g.mode == MODE_SWIGLU) {
    // gate / up: a thread owns one of the tile's 64 columns (gate in tile row c, up in tile row c + 64) and four of
    // the unit's eight token rows; all its loads are in flight at once, no staging and no barrier
    const int cc = gm & (kTcBoxRows - 1), rh = (gm >> 6) * (RB / 2);
#pragma unroll 1
    for (int u = w.c + gidx * w.G; u < n_units; u += 2 * w.G) {
      const int tile = u / n_rb, r0 = (u - tile * n_rb) * RB + rh, col = tile * kTcBoxRows + cc;
      const int n_pieces = tile_pieces(pg, tile);
      const float *base = pieces + (size_t)tile * pg.pieces_max * NPAD * kTcBlockM + cc;
      float tw[PBF * RB];                        // [piece][row][gate, up]
      fetch_words(tw, [&](int q) {
        const int pp = q / RB, i = (q % RB) >> 1;
        tw[q] = (pp < n_pieces && r0 + i < g.rows) ? get_word(base + ((size_t)pp * NPAD + r0 + i) * kTcBlockM + (q & 1) * kTcBoxRows) : 0.f;
      }, w.abort_flag, a.status);
      if (col < g.seg_n[0]) {
#pragma unroll
        for (int i = 0; i < RB / 2; ++i) {
          float gt = 0.f, up = 0.f;
#pragma unroll
          for (int pp = 0; pp < PBF; ++pp) { gt += tw[pp * RB + 2 * i]; up += tw[pp * RB + 2 * i + 1]; }
          if (r0 + i < g.rows) a.act[(size_t)(r0 + i) * a.ff + col] = __float2bfloat16_rn(silu_mul(gt, up));
        }
      }
    }
    return;
  }
#pragma unroll 1
  for (int u = w.c + gidx * w.G; u < n_units; u += 2 * w.G) {
    const int tile = u / n_rb, r_lo = (u - tile * n_rb) * RB, r_hi = min(g.rows, r_lo + RB);
    const Tile ti = tile_of(g, tile);
    const int n_pieces = tile_pieces(pg, tile);
    float *base = pieces + (size_t)tile * pg.pieces_max * NPAD * kTcBlockM + gm;
    const int half = a.hd >> 1, dh = ((ti.row0 + gm) % a.hd) % half;
    const bool rope = (g.mode == MODE_QKV && ti.seg < 2);
    float tn[PBF * RG], csn[RG], snn[RG];
    auto one = [&](int c0, int q) {
      const int pp = q / RG, i = q % RG;
      tn[q] = (pp < n_pieces && c0 + i < r_hi) ? get_word(base + ((size_t)pp * NPAD + c0 + i) * kTcBlockM) : 0.f;
    };
    auto fetch = [&](int c0) {                   // pieces and rope values of rows c0 .. c0 + RG - 1
#pragma unroll
      for (int q = 0; q < PBF * RG; ++q) one(c0, q);
#pragma unroll
      for (int i = 0; i < RG; ++i) {
        csn[i] = 1.f; snn[i] = 0.f;
        if (rope && c0 + i < r_hi) {
          if (rope_cached) {
            csn[i] = w.rope_cos_sh[(c0 + i) * half + dh];
            snn[i] = w.rope_sin_sh[(c0 + i) * half + dh];
          } else {
            csn[i] = __ldg(a.cos_tab + (size_t)w.row_pos_sh[c0 + i] * half + dh);
            snn[i] = __ldg(a.sin_tab + (size_t)w.row_pos_sh[c0 + i] * half + dh);
          }
        }
      }
    };
    fetch(r_lo);
#pragma unroll 1
    for (int c0 = r_lo; c0 < r_hi; c0 += RG) {
      float v[RG], cs[RG], sn[RG];
      settle_words(tn, [&](int q) { one(c0, q); }, w.abort_flag, a.status);
      if (g.mode == MODE_LOGITS) {               // the pass ends here: the words' one reader makes them holes again
        for (int pp = 0; pp < n_pieces; ++pp)
#pragma unroll
          for (int i = 0; i < RG; ++i)
            if (c0 + i < r_hi) put_hole(base + ((size_t)pp * NPAD + c0 + i) * kTcBlockM);
      }
#pragma unroll
      for (int i = 0; i < RG; ++i) {
        v[i] = 0.f;
#pragma unroll
        for (int pp = 0; pp < PBF; ++pp) v[i] += tn[pp * RG + i];
        cs[i] = csn[i]; sn[i] = snn[i];
      }
      if (c0 + RG < r_hi) fetch(c0 + RG);
      final_store<RG>(a, g, ti, cache_of(a, layer < a.n_run ? layer : 0), gm, gm, c0, v, gstage, w.row_pos_sh,
                      w.row_pg_sh, cs, sn, 1 + 2 * gidx);
    }
  }
}

// TC: the launch's long attention work items run on tensor memory (a.tc_attn; head size 128 only).  A kernel of its
// own, so that the other launches keep their code (and its place in the instruction cache) unchanged.
template <int NPAD, int HD, bool TC>
__global__ void __launch_bounds__(kFwdThreads, 1) fwd_persistent_kernel(const __grid_constant__ FwdArgs a) {
  using Cfg = PCfg<NPAD>;
  constexpr int STAGES = Cfg::kStages;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t *ring = smem;
  uint8_t *scratch = smem + STAGES * Cfg::kStageBytes;
  uint64_t *bars = reinterpret_cast<uint64_t *>(scratch + kScratchBytes);
  // bars: full[STAGES] | empty[STAGES] | acc_full[2] | acc_empty[2] | ready[5] (by kind of projection)
  uint32_t *ctl = reinterpret_cast<uint32_t *>(bars + 2 * STAGES + 9);
  uint32_t *tmem_slot = ctl;
  volatile int *abort_flag = reinterpret_cast<volatile int *>(ctl + 1);
  int *first_item_sh = reinterpret_cast<int *>(ctl + 148);               // [4] this CTA's first attention item
  int *qkv_geom_sh = reinterpret_cast<int *>(ctl + 152);                 // [7] piece geometry of the QKV projection
  // [16] phase << 16 | parity << 8 | slot of the first stage of built down projection number (layer & 15): the
  // weight producer is at most one ring (8 stages) ahead, so never 16 such phases
  volatile unsigned *ring_pos_sh = reinterpret_cast<volatile unsigned *>(ctl + 720);
  PhaseGeom *geom_sh = reinterpret_cast<PhaseGeom *>(ctl + 672);          // [5]
  static_assert(5 * sizeof(PhaseGeom) <= (720 - 672) * 4, "control area overlap");
  static_assert((2 * Cfg::kStages + 9) * 8 + 736 * 4 <= kCtrlBytes - 128, "control area overflow");
  unsigned *attn_done_sh = ctl + 2;                                      // attention phases this CTA is through with (TC)
  volatile int *wait_ok = reinterpret_cast<volatile int *>(ctl + 4);   // [2]
  float *red = reinterpret_cast<float *>(ctl + 8);                      // [8]
  PageCache *pcache = reinterpret_cast<PageCache *>(ctl + 16);          // 130 words
  int *row_pos_sh = reinterpret_cast<int *>(ctl + 160);                 // [128] position of each packed row
  int *row_pg_sh = reinterpret_cast<int *>(ctl + 288);                  // [128] KV page holding that position
  FwdLayerDev *norms_sh = reinterpret_cast<FwdLayerDev *>(ctl + 416);   // [<= kMaxLayersSh] norm gains
  static_assert(kMaxLayersSh * sizeof(FwdLayerDev) <= (672 - 416) * 4, "control area overlap");
  long long *dbg_cy = reinterpret_cast<long long *>(reinterpret_cast<uint8_t *>(bars) + kCtrlBytes - 128);   // debug cycle counters [16]
  // cos / sin of the launch's rows (the tables are touched once per layer, so the weight stream would
  // evict them from L2 between uses): [kRopeCacheRows][hd / 2] each, after the attention / staging area
  float *rope_cos_sh = reinterpret_cast<float *>(scratch + kScratchBytes - 2 * kRopeCacheRows * (HD / 2) * 4);
  float *rope_sin_sh = rope_cos_sh + kRopeCacheRows * (HD / 2);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (STAGES + s); };
  auto accf_bar = [&](int b) { return bar0 + 8u * (2 * STAGES + b); };
  auto acce_bar = [&](int b) { return bar0 + 8u * (2 * STAGES + 2 + b); };
  auto ready_bar = [&](int b) { return bar0 + 8u * (2 * STAGES + 4 + b); };

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int G = gridDim.x, c = blockIdx.x;
  const int n_phases = 4 * a.n_run + (a.L > 0 ? 1 : 0);

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(full_bar(s), 2); mbar_init(empty_bar(s), 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(accf_bar(b), 1); mbar_init(acce_bar(b), 4); }
    for (int k = 0; k < 5; ++k) mbar_init(ready_bar(k), 1);
    *abort_flag = 0;
    for (int i = 0; i < 15; ++i) dbg_cy[i] = 0;
    *attn_done_sh = 0u;
    for (int i = 0; i < 16; ++i) ring_pos_sh[i] = 0xFFFFFFFFu;
    pcache->tag_item = -1;
    if (c == 0) *a.next_counter = 0u;                    // (nobody uses it while this launch runs)
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (threadIdx.x >= 128 && threadIdx.x < 133) {
    const int k = threadIdx.x - 128;
    geom_sh[k] = phase_geom(make_gemm(a, k < 4 ? k : 4 * a.n_run), G, c);
  }
  constexpr uint32_t tmem_cols = TC ? 512u : (uint32_t)Cfg::kTmemCols;      // the attention phase takes all of tensor memory
  if (warp == 2) tmem_alloc(smem_u32(tmem_slot), tmem_cols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // The three pipeline roles below are a warp each, of which one lane issues (elect_one).  They are bound by their own
  // instruction chain wherever the data is there already: the ring's eight stages at the start of every phase, and
  // phases whose CTA streams more than its share.  So they keep wrapped slot counters and parities in registers instead of
  // dividing a stage count, and tcgen05.fence::after_thread_sync (~0.1 us while MMAs are in flight) is issued only where
  // another thread's tcgen05 operations must come first (accumulator reuse), not after the wait on TMA data.
  if (warp == 0) {
    // ------------------------------------------------------------ weight-tile producer (runs ahead)
    const bool issuer = elect_one();
    int s = 0;
    uint32_t par = 1;                                    // parity to wait for on the slot's empty barrier
    const uint64_t w_policy = l2_policy_evict_first();   // weights are read once per pass: first out of L2
    bool ok = true;
    for (int p = 0; p < n_phases && ok; ++p) {
      const Gemm g = make_gemm(a, p);
      const PhaseGeom &pg = geom_sh[kind_of(a, p)];
      SegIter it = seg_begin(pg);
      Seg sg;
      // the tensor-memory attention phase uses the ring's memory: the O projection's tiles wait until it is over
      if (TC && (p & 3) == 1 && p < 4 * a.n_run && !count_wait_warp(attn_done_sh, (unsigned)(p >> 2) + 1u, abort_flag)) { ok = false; break; }
      if (issuer && built_down(a, p)) ring_pos_sh[(p >> 2) & 15] = (unsigned)s | (par << 8) | ((unsigned)p << 16);   // where the builders' tiles go
      while (ok && seg_next(pg, it, sg)) {
        const Tile ti = tile_of(g, sg.tile);
        const bool second = (g.mode == MODE_SWIGLU) || (ti.row0 + kTcBoxRows < g.seg_n[ti.seg]);
        const CUtensorMap *m0 = g.mode == MODE_SWIGLU ? g.w[0] : g.w[ti.seg];
        const CUtensorMap *m1 = g.mode == MODE_SWIGLU ? g.w[1] : m0;
        const int row1 = g.mode == MODE_SWIGLU ? ti.row0 : ti.row0 + kTcBoxRows;
        const uint32_t tx = (second ? 2 : 1) * kBoxBytes;
        for (int kb = sg.kb0; kb < sg.kb1; ++kb) {
          if (!mbar_wait_warp(empty_bar(s), par, abort_flag)) { ok = false; break; }
          if (issuer) {
            const uint32_t dst = smem_u32(ring) + (uint32_t)(s * Cfg::kStageBytes);
            mbar_expect_tx(full_bar(s), tx);
            tma_load_2d_hint(dst, m0, kb * kTcBlockK, ti.row0, full_bar(s), w_policy);
            if (second) tma_load_2d_hint(dst + kBoxBytes, m1, kb * kTcBlockK, row1, full_bar(s), w_policy);
          }
          if (++s == STAGES) { s = 0; par ^= 1u; }
        }
      }
    }
    if (!ok && issuer) atomicExch(a.status, 1);
  } else if (warp == 1) {
    // ------------------------------------------------------------ activation-tile producer
    const bool issuer = elect_one();
    int s = 0;
    uint32_t par = 1;
    bool ok = true;
    const uint32_t a_bytes = (uint32_t)a.a_box_rows * kTcBlockK * 2;
    for (int p = 0; p < n_phases && ok; ++p) {
      const int kind = kind_of(a, p);
      const CUtensorMap *amap = &a.amap[kind == 1 ? 1 : kind == 3 ? 2 : kind == 4 ? 3 : 0];
      const PhaseGeom &pg = geom_sh[kind];
      if (pg.left == 0) continue;
      if (built_down(a, p)) {                            // the workers fill the tiles and arrive
        s += pg.left;
        par ^= (uint32_t)(s / STAGES) & 1u;
        s %= STAGES;
        continue;
      }
      // the operand of phase p is complete once the workers have passed the barrier before it
      if (!mbar_wait_warp(ready_bar(kind), kind == 4 ? 0u : (uint32_t)((p >> 2) & 1), abort_flag)) { ok = false; break; }
      SegIter it = seg_begin(pg);
      Seg sg;
      while (ok && seg_next(pg, it, sg)) {
        for (int kb = sg.kb0; kb < sg.kb1; ++kb) {
          if (!mbar_wait_warp(empty_bar(s), par, abort_flag)) { ok = false; break; }
          if (issuer) {
            mbar_expect_tx(full_bar(s), a_bytes);
            tma_load_2d(smem_u32(ring) + (uint32_t)(s * Cfg::kStageBytes) + kWBytes, amap, kb * kTcBlockK, 0, full_bar(s));
          }
          if (++s == STAGES) { s = 0; par ^= 1u; }
        }
      }
    }
    if (!ok && issuer) atomicExch(a.status, 1);
  } else if (warp == 2) {
    // ------------------------------------------------------------ MMA issuer
    const bool issuer = elect_one();
    const uint32_t idesc = umma_idesc_bf16(NPAD);
    const uint64_t da0 = umma_desc(smem_u32(ring));
    int s = 0, seg_idx = 0;
    uint32_t par = 0;
    bool ok = true;
    for (int p = 0; p < n_phases && ok; ++p) {
      const PhaseGeom &pg = geom_sh[kind_of(a, p)];
      SegIter it = seg_begin(pg);
      Seg sg;
      for (; ok && seg_next(pg, it, sg); ++seg_idx) {
        const int ab = seg_idx & 1;
        if (!mbar_wait_warp(acce_bar(ab), (uint32_t)(((seg_idx >> 1) & 1) ^ 1), abort_flag)) { ok = false; break; }
        tc_fence_after();                                // the epilogue's tcgen05.ld of this accumulator come first
        const uint32_t d_tmem = tmem_base + (uint32_t)(ab * NPAD);
        uint32_t acc = 0u;
        for (int kb = sg.kb0; kb < sg.kb1; ++kb) {
          if (!mbar_wait_warp(full_bar(s), par, abort_flag)) { ok = false; break; }
          const uint64_t da = da0 + (uint64_t)(s * (Cfg::kStageBytes >> 4)), db = da + (uint64_t)(kWBytes >> 4);
          if (issuer) {
            umma_bf16(d_tmem, da, db, idesc, acc);
#pragma unroll
            for (int k = 1; k < kTcBlockK / 16; ++k) umma_bf16(d_tmem, da + (uint64_t)(k * 2), db + (uint64_t)(k * 2), idesc, 1u);
            umma_commit(empty_bar(s));
          }
          acc = 1u;
          if (++s == STAGES) { s = 0; par ^= 1u; }
        }
        if (ok && issuer) umma_commit(accf_bar(ab));
      }
    }
    if (!ok && issuer) atomicExch(a.status, 1);
  } else if (warp >= 4) {
    // ------------------------------------------------------------ workers (+ epilogue: warps 4..7)
    const int wt = threadIdx.x - 128;              // 0..255
    const bool is_epi = warp < 8;
    const int q = warp & 3;
    float *staging = reinterpret_cast<float *>(scratch);
    unsigned epoch = 0;
    bool alive = true;

    WorkerCtx w;
    w.tmem_base = tmem_base; w.accf_bar0 = accf_bar(0); w.acce_bar0 = acce_bar(0);
    w.abort_flag = abort_flag; w.wait_ok = wait_ok; w.staging = staging;
    w.row_pos_sh = row_pos_sh; w.row_pg_sh = row_pg_sh; w.geom = geom_sh;
    w.rope_cos_sh = rope_cos_sh; w.rope_sin_sh = rope_sin_sh;
    w.wt = wt; w.lane = lane; w.q = q; w.G = G; w.c = c; w.seg_idx = 0;

    // ---- phase program
    if (HSD_PROF(a) && wt == 0) a.prof[(size_t)blockIdx.x * kFwdProfEvents] = globaltimer_ns();
    for (int l = wt; l < a.n_run; l += 256) norms_sh[l] = a.layers[l];
    if (a.R <= kRopeCacheRows)
      for (int i = wt; i < a.R * (HD / 2); i += 256) {
        const int r = i / (HD / 2), k = i % (HD / 2);
        rope_cos_sh[i] = a.cos_tab[(size_t)a.rows.pos()[r] * (HD / 2) + k];
        rope_sin_sh[i] = a.sin_tab[(size_t)a.rows.pos()[r] * (HD / 2) + k];
      }
    for (int r = wt; r < a.R; r += 256) {             // per-row facts every layer needs, fetched once
      const int pos = a.rows.pos()[r];
      row_pos_sh[r] = pos;
      row_pg_sh[r] = a.page_table[(size_t)a.rows.seq()[r] * a.pages_per_seq + pos / a.page];
    }
    // descriptor of this CTA's first attention work item, kept in shared memory (the same in every layer; a
    // dependent global load at the start of every attention phase otherwise)
    if (wt == 0) {
      const int n_work = a.n_attn * a.nkv * a.n_splits;
      int4 fi = make_int4(0, 0, 0, 0);
      if ((int)blockIdx.x < n_work) fi = a.rows.item(blockIdx.x / (a.n_splits * a.nkv));
      first_item_sh[0] = fi.x; first_item_sh[1] = fi.y; first_item_sh[2] = fi.z; first_item_sh[3] = fi.w;
      const PhaseGeom &pq = geom_sh[0];
      qkv_geom_sh[0] = (a.nq * a.hd + kTcBlockM - 1) / kTcBlockM;
      qkv_geom_sh[1] = qkv_geom_sh[0] + (a.nkv * a.hd + kTcBlockM - 1) / kTcBlockM;
      qkv_geom_sh[2] = pq.parts; qkv_geom_sh[3] = pq.pieces_max; qkv_geom_sh[4] = pq.U; qkv_geom_sh[5] = pq.Gp; qkv_geom_sh[6] = pq.KB;
    }
    // One step loop, one call site per phase body: the whole per-layer program has to stay resident in
    // the instruction cache (every phase runs once per layer, so code that does not fit is fetched
    // cold through the saturated memory system every single time).
    //   t = 0                embed + norm, barrier                         -> ready(QKV 0)
    //   t = 1 + 10 l + s     s: 0 QKV pieces | 1 QKV finish, barrier | 2 attention tiles | 3 attention merge, barrier -> ready(O)
    //                           4 O pieces | 5 norm (+O pieces), barrier -> ready(gate/up) | 6 gate/up pieces
    //                           7 gate/up finish, barrier -> ready(down) | 8 down pieces | 9 norm (+down pieces), barrier -> ready(next)
    //   t = 1 + 10 n, + 1    output-head pieces | output-head finish
    // Steps 1 and 7 are empty when the finish is folded into the phase after it.  A phase that reads the words of the one
    // before waits for those words, so there is a grid barrier only before a projection that takes its activations by TMA,
    // and behind step 1 (its q and cache rows are plain stores): three per layer, five with both finish phases.  Words become
    // holes again under a later projection, behind a barrier after their last reader and in front of one before their next:
    // QKV, partials and O under gate / up, down under the next QKV or the head, and so gate / up if folded (otherwise under
    // down).
    const int n_steps = 1 + 10 * a.n_run + (a.L > 0 ? 2 : 0);
    enum { K_EPI, K_FIN, K_ATTN_A, K_ATTN_B, K_NORM, K_NONE };
#pragma unroll 1
    for (int t = 0; t < n_steps && alive; ++t) {
      int kind, gp = 0, ready = -1, l = 0;
      bool barrier = true;
      if (t == 0) { kind = K_NORM; ready = 0; }
      else if (t > 10 * a.n_run) { gp = 4 * a.n_run; kind = (t == 1 + 10 * a.n_run) ? K_EPI : K_FIN; barrier = false; }
      else {
        l = (t - 1) / 10;
        const int sstep = (t - 1) % 10, p = 4 * l;
        switch (sstep) {
          case 0: kind = K_EPI; gp = p; barrier = false; break;
          case 1:                                            // folded into the attention phase when every item stands alone
            if (a.fuse_qkv) { kind = K_NONE; barrier = false; }
            else { kind = K_FIN; gp = p; }
            break;
          case 2:
            kind = K_ATTN_A;
            if (a.n_splits == 1) ready = p + 1;                 // a single key split needs no merge phase
            else barrier = false;
            break;
          case 3:
            if (a.n_splits == 1) { kind = K_NONE; barrier = false; }
            else { kind = K_ATTN_B; ready = p + 1; }
            break;
          case 4: kind = K_EPI; gp = p + 1; barrier = !a.early_norm; break;
          case 5: kind = K_NORM; gp = p + 1; ready = p + 2; break;
          case 6: kind = K_EPI; gp = p + 2; barrier = false; break;
          case 7:                                            // folded into the down projection in passes with few rows
            if (a.fuse_gu) { kind = K_NONE; barrier = false; }
            else { kind = K_FIN; gp = p + 2; ready = p + 3; }
            break;
          case 8: kind = K_EPI; gp = p + 3; barrier = (l + 1 < a.n_run || a.L > 0) && !a.early_norm; break;
          default:
            kind = (l + 1 < a.n_run || a.L > 0) ? K_NORM : K_NONE; gp = p + 3; ready = p + 4;
            barrier = (kind == K_NORM);
            break;
        }
      }
      switch (kind) {
        case K_EPI:
          if (built_down(a, gp)) {
            if (a.gu_pieces_max <= 2) build_act_stages<NPAD, 2, 2>(a, w, gp, ring, full_bar(0), empty_bar(0), ring_pos_sh);
            else build_act_stages<NPAD, 4, 1>(a, w, gp, ring, full_bar(0), empty_bar(0), ring_pos_sh);
          }
          if (is_epi) gemm_epilogue<NPAD>(a, w, gp);
          else {
            const int kind = kind_of(a, gp);
            if (kind == 2) {
              put_holes<NPAD>(a, w, 0);
              put_holes<NPAD>(a, w, 1);
              if (a.n_splits > 1) put_partial_holes<HD>(a, wt, first_item_sh);
            } else if (kind == 3 ? !a.fuse_gu : (kind == 0 || kind == 4) && gp > 0) {
              if (kind != 3) put_holes<NPAD>(a, w, 3);
              if (kind == 3 || a.fuse_gu) put_holes<NPAD>(a, w, 2);
            }
          }
          break;
        case K_FIN: gemm_finish<NPAD>(a, w, gp); break;
        case K_ATTN_A:
          alive = attn_tiles_phase<NPAD, HD, TC>(a, cache_of(a, l), scratch, pcache, wt, dbg_cy, first_item_sh, qkv_geom_sh, row_pg_sh, rope_cos_sh,
                                                 rope_sin_sh, ring, tmem_base, abort_flag);
          if (TC && alive) {                                               // the ring's memory is the weight producer's again
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // TMA writes next where these threads wrote
            worker_sync();
            if (wt == 0) asm volatile("st.release.cta.shared.u32 [%0], %1;" ::"r"(smem_u32(attn_done_sh)), "r"((unsigned)l + 1u) : "memory");
          }
          break;
        case K_ATTN_B: attn_merge_phase<HD>(a, row_pos_sh, wt, abort_flag); break;
        case K_NORM: {
          const bool first = (t == 0);
          const bool last = !first && (((t - 1) % 10) == 9) && (l + 1 >= a.n_run);      // final norm over the logit rows
          const bool mid = !first && (((t - 1) % 10) == 5);
          const __nv_bfloat16 *gain = first ? a.layers[0].attn_norm
                                            : (last ? a.final_norm : (mid ? norms_sh[l].mlp_norm : norms_sh[l + 1].attn_norm));
          auto norm = [&](auto slots) {
            norm_phase<NPAD, decltype(slots)::value>(a, last ? a.L : a.R, last ? a.rows.src() : nullptr, first,
                                                     first ? nullptr : a.pieces[gp & 3], geom_sh[gp & 3].pieces_max, gain, last ? a.hf : a.h,
                                                     red, wt, abort_flag);
          };
          if (a.d <= 2048) norm(std::integral_constant<int, 2>{});
          else norm(std::integral_constant<int, 4>{});
          break;
        }
        default: break;
      }
      if (barrier && alive) alive = grid_barrier(a, epoch, abort_flag, wt, ready >= 0 ? ready_bar(kind_of(a, ready)) : 0u);
    }
  }
  if (HSD_PROF(a) && blockIdx.x == 0 && threadIdx.x == 128) for (int i = 0; i < 15; ++i) a.prof[940 + i] = (unsigned long long)dbg_cy[i];
  // ------------------------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (*abort_flag) {                                     // (nobody writes it any more: the same in all threads)
    if (threadIdx.x == 0) atomicExch(a.status, 1);
    const unsigned long long t0 = globaltimer_ns();      // copies and MMAs in flight end before their memory goes away
    while (globaltimer_ns() - t0 < 200000ull) {}
    __syncthreads();
  }
  if (warp == 2) tmem_dealloc(tmem_base, tmem_cols);
}

// The attention tiles phase as a launch of its own (prompt passes with more rows than the persistent forward takes):
// one key split per item, so every work item writes its rows of the attention output itself.  256 threads = the
// phase's eight worker warps; q / k / v of the pass are in place (separate finish kernels).
template <int HD>
__global__ void __launch_bounds__(256, 2) attn_tiles_kernel(const __grid_constant__ FwdArgs a, __nv_bfloat16 *k_pool, __nv_bfloat16 *v_pool) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *scratch = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  __shared__ PageCache pcache;
  __shared__ int first_item_sh[4];
  __shared__ int qkv_geom_sh[8];
  __shared__ long long dbg_cy[16];
  if (threadIdx.x == 0) {
    pcache.tag_item = -1;
    const int n_work = a.n_attn * a.nkv * a.n_splits;
    int4 fi = make_int4(0, 0, 0, 0);
    if ((int)blockIdx.x < n_work) fi = a.rows.item(blockIdx.x / (a.n_splits * a.nkv));
    first_item_sh[0] = fi.x; first_item_sh[1] = fi.y; first_item_sh[2] = fi.z; first_item_sh[3] = fi.w;
  }
  __syncthreads();
  const LayerCache lay = {k_pool, v_pool};
  attn_tiles_phase<128, HD, false>(a, lay, scratch, &pcache, (int)threadIdx.x, dbg_cy, first_item_sh, qkv_geom_sh, nullptr, nullptr, nullptr,
                            nullptr, 0u, nullptr);
}

template <int HD>
int launch_attn_tiles_t(const FwdArgs &a, __nv_bfloat16 *k_pool, __nv_bfloat16 *v_pool, int sm_count, cudaStream_t s) {
  static std::atomic<u64> limits{0};
  const int smem = kScratchBytes + 1024;
  const int limit = hsd_smem_limit((const void *)attn_tiles_kernel<HD>, smem, limits);
  if (limit) return limit;
  const int n_work = a.n_attn * a.nkv * a.n_splits;
  attn_tiles_kernel<HD><<<std::min(n_work, 2 * sm_count), 256, smem, s>>>(a, k_pool, v_pool);
  hsd_count_launches(1);
  return hsd_launch_status();
}

template <int NPAD, int HD, bool TC>
int launch_t(const FwdArgs &args, int sm_count, cudaStream_t s) {
  using Cfg = PCfg<NPAD>;
  static std::atomic<u64> limits{0};
  const int limit = hsd_smem_limit((const void *)fwd_persistent_kernel<NPAD, HD, TC>, Cfg::kSmemBytes, limits);
  if (limit) return limit;
  void *params[1] = {const_cast<FwdArgs *>(&args)};
  HSD_CUDA_OK(cudaLaunchCooperativeKernel((const void *)fwd_persistent_kernel<NPAD, HD, TC>, dim3(sm_count), dim3(kFwdThreads), params,
                                          (size_t)Cfg::kSmemBytes, s));
  hsd_count_launches(1);
  return HSD_OK;
}

template <int HD, bool TC>
int launch_hd(const FwdArgs &args, int npad, int sm_count, cudaStream_t s) {
  switch (npad) {
    case 16: return launch_t<16, HD, TC>(args, sm_count, s);
    case 32: return launch_t<32, HD, TC>(args, sm_count, s);
    case 64: return launch_t<64, HD, TC>(args, sm_count, s);
    case 128: return launch_t<128, HD, TC>(args, sm_count, s);
    default: return HSD_E_INVALID_ARG;
  }
}

}  // namespace

namespace {
// Piece buffers of the five kinds of projections (QKV, O, gate / up, down, head), one after the other; offsets in floats.
struct PieceLayout { size_t off[5], total; int gu_pieces_max; };
PieceLayout piece_layout(int d, int nqd, int nkvd, int ff, int V, int npad, int G) {
  auto tiles = [](int n) { return (n + kTcBlockM - 1) / kTcBlockM; };
  const int n_tiles[5] = {tiles(nqd) + 2 * tiles(nkvd), tiles(d), (ff + kTcBoxRows - 1) / kTcBoxRows, tiles(d), tiles(V)};
  const int K[5] = {d, nqd, d, ff, d};
  PieceLayout pl;
  pl.total = 0;
  for (int g = 0; g < 5; ++g) {
    const SplitGeom sg = split_geom(n_tiles[g], K[g] / kTcBlockK, g == 1 || g == 3 ? residual_parts(d) : 4, G);
    if (g == 2) pl.gu_pieces_max = sg.pieces_max;
    pl.off[g] = pl.total;
    pl.total += (size_t)n_tiles[g] * sg.pieces_max * npad * kTcBlockM;
  }
  return pl;
}
}  // namespace

size_t fwd_pieces_bytes(int d, int nqd, int nkvd, int ff, int V, int sm_count) {
  if (d < kTcBlockK || nqd < kTcBlockK || ff < kTcBlockK) return 0;
  return piece_layout(d, nqd, nkvd, ff, V, 128, sm_count).total * 4;
}

int launch_attention_tiles(const FwdArgs &args, __nv_bfloat16 *k_pool, __nv_bfloat16 *v_pool, int sm_count, cudaStream_t s) {
  if (args.fuse_qkv || args.n_splits != 1 || args.n_attn < 1) return HSD_E_INVALID_ARG;
  switch (args.hd) {
    case 128: return launch_attn_tiles_t<128>(args, k_pool, v_pool, sm_count, s);
    case 64: return launch_attn_tiles_t<64>(args, k_pool, v_pool, sm_count, s);
    case 32: return launch_attn_tiles_t<32>(args, k_pool, v_pool, sm_count, s);
    default: return HSD_E_UNSUPPORTED;
  }
}

bool fwd_persist_supported(int hd, int group) {
  return (hd == 32 || hd == 64 || hd == 128) && group >= 1 && group <= 8 && fwd_attn_rows(group, hd) * group <= 32;
}

int launch_forward_persistent(const FwdArgs &args, int npad, int sm_count, cudaStream_t s) {
  if (args.R < 1 || args.R > npad || args.L > npad) return HSD_E_INVALID_ARG;
  if (args.n_run > kMaxLayersSh) return HSD_E_UNSUPPORTED;
  if (((args.d + kTcBlockM - 1) / kTcBlockM) * 2 > sm_count) return HSD_E_UNSUPPORTED;   // norm phase: regular split only
  {  // unit arithmetic on the device is 32-bit
    long long tiles = std::max<long long>((args.V + 127) / 128, (args.ff + 63) / 64);
    long long kb = std::max(args.ff, std::max(args.d, args.nq * args.hd)) / kTcBlockK;
    if (tiles * kb * sm_count >= (1ll << 31)) return HSD_E_UNSUPPORTED;
  }
  if (args.tc_attn && (args.hd != 128 || args.fuse_qkv)) return HSD_E_INVALID_ARG;
  FwdArgs a = args;
  const PieceLayout pl = piece_layout(a.d, a.nq * a.hd, a.nkv * a.hd, a.ff, a.V, npad, sm_count);
  if (pl.total * 4 > args.pieces_bytes) return HSD_E_WORKSPACE_TOO_SMALL;
  for (int g = 0; g < 5; ++g) a.pieces[g] = args.pieces[0] + pl.off[g];
  a.gu_pieces_max = pl.gu_pieces_max;
  // (a pass without logits ends with the last down projection, after which no phase could make gate / up's words holes)
  if (a.gu_pieces_max > 4 || a.L == 0) a.fuse_gu = 0;
  switch (a.hd) {
    case 128: return a.tc_attn ? launch_hd<128, true>(a, npad, sm_count, s) : launch_hd<128, false>(a, npad, sm_count, s);
    case 64: return launch_hd<64, false>(a, npad, sm_count, s);
    case 32: return launch_hd<32, false>(a, npad, sm_count, s);
    default: return HSD_E_UNSUPPORTED;
  }
}

}  // namespace hsd
