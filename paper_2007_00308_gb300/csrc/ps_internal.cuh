// Internal declarations of the GB300 polar stroking library.
//
// Device-side geometry is FP32; FP64 appears only in the predicated islands of
// the PS_PREC_MIXED variant (GB300 issues FP64 FMAs ~57x slower than FP32).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/polarstroke.h"
#include "ps_df.cuh"

#define PS_PI_F 3.14159265358979323846f
#define PS_TWO_PI_F 6.28318530717958647692f
#define PS_PI_D 3.14159265358979323846
#define PS_TWO_PI_D 6.28318530717958647692

// Bounded spin for inter-CTA waits: after this many polls a wait gives up,
// records PS_ERR_TIMEOUT and proceeds (results of that launch are invalid).
#define PS_SPIN_LIMIT (1 << 22)

// Link kinds stored in LinkRec::meta bits 0-1.
enum { LK_EMPTY = 0, LK_SEG = 1, LK_JOIN = 2, LK_CAP = 3 };

// Per-link interval record written by the setup pass and read by the rib pass.
// 240 bytes; at most 6 intervals (3 curvature-monotone intervals of a cubic,
// each split once at pi -- Sec. 3.3.5), boundaries k = 0..M.  The *_lo fields
// complete psi, p and step to double-float pairs (hi + lo) in PS_PREC_MIXED;
// they are zero in PS_PREC_FP32.
struct __align__(16) LinkRec {
  float2 P[4];        // control points (segment) / P[0] = pivot point (join, cap)
  float w;            // conic weight
  float rN, rP;       // radii of the N and P sides (Eq. 16-17)
  uint32_t meta;      // kind | type<<2 | M<<4 | pivot mask<<8 | style<<16 | flags<<20
  float psi[7];       // Psi_k at interval boundaries (Eq. 5)
  float p[7];         // p_k (Eq. 4)
  float step[6];      // delta_k / Delta_k (Eq. 12, psi(j) of Sec. 4.2.1)
  uint16_t dsum[7];   // Delta_Sigma(k) (Eq. 13)
  uint16_t pad;
  float2 v1, v2;      // miter override vertices for ribs 1 and 2
  float psi_lo[7];
  float p_lo[7];
  float step_lo[6];
};
static_assert(sizeof(LinkRec) == 240, "LinkRec layout");

#define META_KIND(m) ((m) & 3u)
#define META_TYPE(m) (((m) >> 2) & 3u)
#define META_M(m) (((m) >> 4) & 15u)
#define META_PIVOT(m, k) (((m) >> (8 + (k))) & 1u)
#define META_STYLE(m) (((m) >> 16) & 15u)
#define META_FLAG_OVERRIDE (1u << 20)  // ribs 1,2 outer vertex = v1, v2 (miter)
#define META_FLAG_SQUARE (1u << 21)    // square cap: ribs 1,3 outer radius * sqrt(2)
// interior boundary k (1..6) is a split point (Sec. 3.3.5) rather than an inflection
#define META_SPLIT_BIT(k) (1u << (21 + (k)))
#define META_SPLIT(m, k) (((m) >> (21 + (k))) & 1u)

// Profiling slots (one per kernel; the first has lost its own).
enum {
  PK_UNUSED = 0, PK_LINK_SETUP, PK_EMIT, PK_ARCLEN, PK_MIDCHORD, PK_BIN_COUNT, PK_TILE_SCAN,
  PK_BIN_SCATTER, PK_COVERAGE, PK_DASH, PK_COUNT
};
static_assert(PK_COUNT == PS_PROF_SLOTS, "profile slots");

// State of one tile of a single-pass scan (see below).
struct __align__(16) TileState {
  unsigned long long v, flag;
};

// Host-side context.
struct ps_context {
  int prof_on;
  cudaEvent_t prof_ev[PK_COUNT][2];
  int prof_recorded[PK_COUNT];
  int device;
  // CTAs per SM of the kernels launched so far (ps_persistent_grid)
  struct { const void* kernel; int per_sm; } occ[24];
  int n_occ;
  int cov_attr_done[2];  // coverage kernels' shared-memory attribute set on this device
  void* last_stream;
  int captured;             // a call has been captured into a graph
  void** kept;              // blocks outgrown since, [n_kept]
  int n_kept, kept_cap;
  int32_t* d_status;        // first error recorded by a kernel
  // scan tile states (shared by the passes of one call; calls on one context
  // are serialized on the stream they are issued to)
  TileState* d_tile_state;  // [tile_cap]
  int64_t tile_cap;
  int32_t* d_counters;      // ticket counters, 16 ints, right before d_tile_state (one memset)
  LinkRec* d_recs;
  int64_t rec_cap;
  // raster workspace
  int32_t* d_tile_count;    // [n_tile + 1]
  int32_t* d_tile_off;      // [n_tile + 1]
  int32_t* d_tile_cursor;   // [2 (n_tile + 1)]: scatter cursors from the front, then from the back
  int32_t* d_tile_list;     // tiles with bin entries, then their count
  int64_t raster_tile_cap;
  uint32_t* d_bin;          // [pair_cap]
  uint32_t* d_quad_hits;    // [2 quad_hits_cap] per-rib {hits, box} words of the binning passes
  int64_t quad_hits_cap;
  int64_t pair_cap;
  int64_t* d_scratch64;     // 16 int64: the work counts of the last raster call
  int64_t last_n_tile;      // tiles of the most recent raster call
  uint32_t* d_mask_scratch; // per-CTA per-path tile masks beyond shared memory
  size_t d_scratch_words;
  void* d_adj;              // adjoint workspace
  size_t adj_bytes;
  void* d_cap_tasks;        // the dasher's round caps
  size_t cap_bytes;
  int num_sms;
  int tune[PS_TUNE_COUNT];  // launch parameters (ps_set_tuning)
  float pixel_tol;          // pixel tolerance of the per-link step boost (0: off)
};

// ---- status -----------------------------------------------------------------
__device__ __forceinline__ void ps_record_error(int32_t* status, int code) {
  // read first: a launch where many threads fail would otherwise serialize on
  // one atomic per failure
  if (status && *(volatile int32_t*)status == 0) atomicCAS(status, 0, code);
}

// ---- single-pass scans --------------------------------------------------------
// Tile states (decoupled look-back, Merrill & Garland 2016): a value and a flag, 0 = not
// ready, TF_AGG = the tile's aggregate, TF_INCL = its inclusive prefix.  The two are read and
// written as one 128-bit word, so that a reader needs no ordering between them
// and pays one memory latency per round.
#define TF_AGG 1ull
#define TF_INCL 2ull

__device__ __forceinline__ void st_state(TileState* p, unsigned long long v,
                                         unsigned long long flag) {
  asm volatile(
      "{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p),
      "l"(v), "l"(flag)
      : "memory");
}
__device__ __forceinline__ TileState ld_state(const TileState* p) {
  TileState s;
  asm volatile(
      "{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
      : "=l"(s.v), "=l"(s.flag)
      : "l"(p)
      : "memory");
  return s;
}

// Sums of a look-back: int64, or a double-float pair in the state's 64 bits.
struct SumI64 {
  typedef long long T;
  static __device__ __forceinline__ T zero() { return 0; }
  static __device__ __forceinline__ T add(T a, T b) { return a + b; }
  static __device__ __forceinline__ T shfl(T a, int lane) { return __shfl_sync(0xffffffffu, a, lane); }
  static __device__ __forceinline__ T shfl_xor(T a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
  static __device__ __forceinline__ unsigned long long bits(T a) { return (unsigned long long)a; }
  static __device__ __forceinline__ T of(unsigned long long w) { return (T)w; }
};
struct SumDF {
  typedef ps::DF T;
  static __device__ __forceinline__ T zero() { return ps::DF{0.f, 0.f}; }
  static __device__ __forceinline__ T add(T a, T b) { return ps::df_add(a, b); }
  static __device__ __forceinline__ T shfl(T a, int lane) {
    return ps::DF{__shfl_sync(0xffffffffu, a.hi, lane), __shfl_sync(0xffffffffu, a.lo, lane)};
  }
  static __device__ __forceinline__ T shfl_xor(T a, int o) {
    return ps::DF{__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
  }
  static __device__ __forceinline__ unsigned long long bits(T a) {
    return ((unsigned long long)__float_as_uint(a.lo) << 32) | (unsigned long long)__float_as_uint(a.hi);
  }
  static __device__ __forceinline__ T of(unsigned long long w) {
    return ps::DF{__uint_as_float((uint32_t)w), __uint_as_float((uint32_t)(w >> 32))};
  }
};

// Sum of the tiles before tile t, the walk spread over one warp (all 32 lanes
// call it): lane k reads the state of the k-th nearest tile, so one round covers 32
// predecessors.  The walk ends at the nearest tile with an inclusive prefix; that
// tile and every nearer one must have published before the round is summed,
// else the round is read again (bounded by PS_SPIN_LIMIT; PS_ERR_TIMEOUT after it).  The
// lanes add up their own terms and reduce them once at the end.  (With flags
// and values in separate words, read one after the other, the arc-length scan
// took 235 us on 43 M ribs and 997 us on 211 M, and 168 and 731 us with the
// 128-bit states; reading two, four or eight windows of 32 a round cost registers and won
// nothing: 173, 225 and 227 us.)
template <class S>
__device__ __forceinline__ typename S::T lookback_walk(const TileState* state, int64_t t,
                                                       int32_t* status) {
  const int lane = threadIdx.x & 31;
  typename S::T mine = S::zero();
  int spins = 0;
  for (int64_t i = t - 1;;) {
    const int64_t j = i - lane;
    const TileState w = j >= 0 ? ld_state(state + j) : TileState{S::bits(S::zero()), TF_INCL};
    const unsigned stop_m = __ballot_sync(0xffffffffu, w.flag == TF_INCL);
    const unsigned unready = __ballot_sync(0xffffffffu, w.flag == 0ull);
    const int first = stop_m ? __ffs(stop_m) - 1 : 31;
    const unsigned need = first == 31 ? 0xffffffffu : ((2u << first) - 1u);
    if (unready & need) {
      if (++spins > PS_SPIN_LIMIT) {
        if (lane == 0) ps_record_error(status, PS_ERR_TIMEOUT);
        break;
      }
      __nanosleep(32);
      continue;
    }
    // the nearest predecessor holds the whole prefix: nothing to sum
    if (first == 0 && i == t - 1) return S::shfl(S::of(w.v), 0);
    if (lane <= first) mine = S::add(mine, S::of(w.v));
    if (stop_m) break;
    i -= 32;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mine = S::add(mine, S::shfl_xor(mine, o));
  return mine;
}

// Exclusive prefix of tile t for an int64 sum; publishes the tile's own states.
__device__ __forceinline__ long long lookback_sum_warp(TileState* state, long long tile_agg,
                                                       int64_t t, int32_t* status) {
  const int lane = threadIdx.x & 31;
  if (lane == 0) st_state(&state[t], (unsigned long long)tile_agg, t == 0 ? TF_INCL : TF_AGG);
  if (t == 0) return 0;
  const long long prefix = lookback_walk<SumI64>(state, t, status);
  if (lane == 0) st_state(&state[t], (unsigned long long)(prefix + tile_agg), TF_INCL);
  return prefix;
}

// Segmented (by path) sum of the tiles (chunks) before tile t: the carry into
// the tile's elements that precede its first segment head (path start).  A chunk that holds a path
// start publishes its inclusive value at once (it does not depend on the
// carry), so the walk ends at the nearest such chunk.  Sums are double-float
// pairs.
__device__ __forceinline__ ps::DF lookback_segsum_df(TileState* state, ps::DF tile_agg,
                                                     bool tile_head, int64_t t, int32_t* status) {
  const int lane = threadIdx.x & 31;
  if (lane == 0)
    st_state(&state[t], SumDF::bits(tile_agg), t == 0 || tile_head ? TF_INCL : TF_AGG);
  if (t == 0) return ps::DF{0.f, 0.f};
  const ps::DF carry = lookback_walk<SumDF>(state, t, status);
  if (lane == 0 && !tile_head)
    st_state(&state[t], SumDF::bits(ps::df_add(carry, tile_agg)), TF_INCL);
  return carry;
}

// The last link l in [0, n - 1] with off[l] <= r (off non-decreasing, off[0] <= r): a
// warp's 32 probes per round.
__device__ __forceinline__ int64_t find_link_warp(const int32_t* off, int64_t n, int64_t r,
                                                  int lane) {
  int64_t lo = 0, hi = n - 1;  // off[lo] <= r, answer in [lo, hi]
  while (hi - lo > 31) {
    int64_t step = (hi - lo + 31) / 32;
    int64_t cand = lo + lane * step;
    bool ok = cand <= hi && (int64_t)off[cand] <= r;
    uint32_t b = __ballot_sync(0xffffffffu, ok);
    int m = __popc(b);  // lanes 0 .. m-1 ok (lane 0 always)
    int64_t nlo = lo + (int64_t)(m - 1) * step;
    int64_t nhi = m < 32 ? lo + (int64_t)m * step - 1 : hi;
    lo = nlo;
    hi = nhi < hi ? nhi : hi;
  }
  int64_t cand = lo + lane;
  bool ok = cand <= hi && (int64_t)off[cand] <= r;
  uint32_t b = __ballot_sync(0xffffffffu, ok);
  return lo + __popc(b) - 1;
}

// ---- overlapped launches ---------------------------------------------------------
// A kernel that follows another of the same call is launched with programmatic stream
// serialization.  No kernel lets the next one in early (launch_dependents), so the next
// one's CTAs start once the last CTA of the kernel before has ended: what overlaps is the
// launch itself and the end of the kernel before, whose writes may still be on their way.  So
// its CTAs wait here, before any access to memory, until every earlier kernel has finished and
// its writes are visible.  Every such kernel calls dep_wait() first thing, so that a kernel is
// never done before the ones it follows.  One curve on a small canvas: 62 -> 51 us; 64 cubics:
// 99 -> 86; 300 paths: 629 -> 617; a dashed path of 5,031 cubics: 581 -> 565.  (With
// launch_dependents at every kernel's start these took 54, 94, 569 and 573 us, against 52, 92, 566
// and 564 without in the same run.)
//   What the kernels before wrote is read through plain pointers, without __restrict__ or
// __ldg: those say that nobody writes the data while the kernel runs, which is not so before
// the wait, and the wait's memory clobber does not hold back loads of such data.
__device__ __forceinline__ void dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launch of a kernel right after another of the call; overlap = false (event records in
// between, or anything but a kernel before it): an ordinary launch.
template <class... P, class... A>
static inline void ps_launch_after(bool overlap, void (*kernel)(P...), int grid, int block,
                                   size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = overlap ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// ---- host helpers -------------------------------------------------------------
// Notes the stream of a call, and whether it is being captured.  From the first capture on the
// context gives no outgrown block back before it is destroyed: the graph holds its address.
void ps_on_stream(ps_context* ctx, void* stream);
// The capacity to grow to: then at least half as much again, so that the kept blocks of a
// workspace come to less than twice the one in use.
int64_t ps_grown(const ps_context* ctx, int64_t old, int64_t want);
int ps_grow(ps_context* ctx, void** p, size_t bytes);
int ps_ensure_tiles(ps_context* ctx, int64_t n_tile);
int ps_ensure_recs(ps_context* ctx, int64_t n_link);
int ps_ensure_raster(ps_context* ctx, int64_t n_tile, int64_t n_pair);
int ps_ensure_quad_hits(ps_context* ctx, int64_t n_rib);
int ps_cuda_check(cudaError_t e);
// A persistent kernel's CTAs: as many as the device holds at once.  The occupancy is asked for
// once per context and kernel (a query costs about as much as a launch).
int ps_persistent_grid(ps_context* ctx, const void* kernel, int block, size_t smem);
// ... but no more than one per `per` of at most n items.
static inline int ps_grid_for(int grid, int64_t n, int64_t per) {
  const int64_t want = (n + per - 1) / per;
  return want < grid ? (int)(want > 0 ? want : 1) : grid;
}
// Link setup (records in ctx->d_recs, link path indices after them) into the given
// offset arrays; used by the adjoint to rebuild the forward's interval records.
int ps_run_link_setup(ps_context* ctx, const ps_segments* seg, const ps_paths* paths, float dtheta,
                      int precision, int32_t* d_link_off, int32_t* d_path_off, int64_t* d_n_rib,
                      cudaStream_t st);
// Segmented (by path) inclusive prefix of per-rib values, with per-path totals.
int ps_run_segmented_prefix(ps_context* ctx, const float* d_vals, float* d_prefix, const uint32_t* d_tag,
                            const int64_t* d_n_rib, int64_t capacity, float* d_path_tot,
                            int32_t n_path, cudaStream_t st);
void ps_prof_mark(ps_context* ctx, int slot, int end, cudaStream_t st);
struct ProfScope {
  ps_context* c;
  int slot;
  cudaStream_t st;
  ProfScope(ps_context* c_, int s_, cudaStream_t st_) : c(c_), slot(s_), st(st_) {
    ps_prof_mark(c, slot, 0, st);
  }
  ~ProfScope() { ps_prof_mark(c, slot, 1, st); }
};
