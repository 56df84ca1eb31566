// Dashing by cumulative arc length (Sec. 5.2).
//
// On-stretch i of period k covers s in [k*period + cum[2i] - offset,
// k*period + cum[2i+1] - offset).  Each quad [s_{r-1}, s_r] of a rib strip is
// clipped to those stretches by interpolating both rib vertices; every piece is
// an independent 2-rib strip.  A quad of zero length (join, cap, cusp pivot) is
// kept whole iff its s is "on".  Stretch boundaries are evaluated in FP64 with
// explicitly rounded operations (no contraction).
//
// With cap styles (ps_dash_capped), every stretch also gets its path's cap at
// its ends inside the path: a start cap where 0 < a lies in [s_{r-1}, s_r), an
// end cap where b lies in (s_{r-1}, s_r], each the path cap of Sec. 4.3.5
// (pivot through +pi, outer side N, inner radius 0) about the boundary rib --
// centre its midpoint, radius half its length, tangent the rib turned
// clockwise -- as a strip of its own at the boundary's s, written before the
// stretch's first piece or after its last.
#include <cuda_runtime.h>

#include <algorithm>

#include "ps_dash_walk.cuh"
#include "ps_internal.cuh"

namespace {

using namespace ps;

__device__ __forceinline__ int cap_steps(const DashPattern& P, uint32_t path) {
  if (!P.path_cap || (int)path >= P.n_path) return 0;
  switch (P.path_cap[path]) {
    case PS_CAP_TRIANGLE: return 2;
    case PS_CAP_SQUARE: return 4;
    case PS_CAP_ROUND: return P.j_round;
    default: return 0;
  }
}

// A dash cap about boundary rib v (start: pivot from psi + pi, end: from psi; both
// through +pi): its centre, radius and first angle.
struct DashCap {
  float cx, cy, r, psi0;
};
__device__ __forceinline__ DashCap make_cap(float4 v, bool start) {
  const float PI_F = 3.14159265358979323846f;
  DashCap c;
  c.cx = 0.5f * (v.x + v.z);
  c.cy = 0.5f * (v.y + v.w);
  const float vx = v.z - v.x, vy = v.w - v.y;
  c.r = 0.5f * sqrtf(vx * vx + vy * vy);
  const float psi = atan2f(-vx, vy);  // the rib is 2r n(psi), n = (-sin psi, cos psi)
  c.psi0 = start ? psi + PI_F : psi;
  return c;
}

// Ribs k = k0, k0 + dk, .. <= J of a cap whose first rib goes to out[o].
__device__ __forceinline__ void emit_cap(const DashCap& c, int J, bool square, int k0, int dk,
                                         uint32_t tg, float sv, int32_t src, int64_t o,
                                         float4* out_rib, float* out_s, uint32_t* out_tag,
                                         int32_t* out_src) {
  const float PI_F = 3.14159265358979323846f;
  for (int k = k0; k <= J; k += dk) {
    const float ang = k == J ? c.psi0 + PI_F : c.psi0 + PI_F * (float)k / (float)J;
    float sn, cs;
    sincosf(ang, &sn, &cs);
    const float rn = (square && (k == 1 || k == 3)) ? c.r * 1.41421356237309515f : c.r;
    out_rib[o + k] = make_float4(c.cx + rn * sn, c.cy - rn * cs, c.cx, c.cy);
    out_s[o + k] = sv;
    out_tag[o + k] = (tg & ~(PS_TAG_SEGMENT | PS_TAG_LINK_START)) | (k == 0 ? PS_TAG_LINK_START : 0u);
    if (out_src) out_src[o + k] = src;
  }
}

// A round cap to be written by k_dash_caps.
struct CapTask {
  DashCap cap;
  uint32_t tag;
  float s;
  int32_t src, pad;
  int64_t o;
};

constexpr int DASH_NT = 256;
constexpr int DASH_QPT = 4;  // quads per thread
constexpr int DASH_TILE = DASH_NT * DASH_QPT;

// End rib of a whole quad as the FP64 rule computes it (f1 = 1): a0 + (a1 - a0)
// in FP64, which is a1 itself whenever a1 - a0 is exact in FP64 (exponents at
// most 28 apart, or a zero); otherwise the FP64 sum is taken as is.  (That sum is out of
// line: inlined, it was computed for every vertex and discarded, and the FP64
// pipe was 46% busy with it.)
__device__ __noinline__ float4 whole_end64(float4 v0, float4 v1) {
  auto sum = [](float a0, float a1) {
    return (float)__dadd_rn((double)a0, __dsub_rn((double)a1, (double)a0));
  };
  return make_float4(sum(v0.x, v1.x), sum(v0.y, v1.y), sum(v0.z, v1.z), sum(v0.w, v1.w));
}
__device__ __forceinline__ bool is_exact_end(float a0, float a1) {
  const int e0 = (int)((__float_as_uint(a0) >> 23) & 0xffu);
  const int e1 = (int)((__float_as_uint(a1) >> 23) & 0xffu);
  return a0 == 0.f || a1 == 0.f || abs(e0 - e1) <= 28;
}
__device__ __forceinline__ float4 whole_end(float4 v0, float4 v1) {
  if (is_exact_end(v0.x, v1.x) && is_exact_end(v0.y, v1.y) && is_exact_end(v0.z, v1.z) &&
      is_exact_end(v0.w, v1.w))
    return v1;
  return whole_end64(v0, v1);
}

// Where a dash call writes.
struct DashOut {
  float4* rib;
  float* s;
  uint32_t* tag;
  int32_t* src;
  int64_t cap;
};

__device__ __forceinline__ void put_piece(const DashOut& D, int64_t o, float4 p0, float4 p1, float s0,
                                          float s1, uint32_t tg, int32_t r) {
  D.rib[o] = p0;
  D.rib[o + 1] = p1;
  D.s[o] = s0;
  D.s[o + 1] = s1;
  D.tag[o] = tg | PS_TAG_LINK_START;
  D.tag[o + 1] = tg;
  if (D.src) {
    D.src[o] = r;
    D.src[o + 1] = r;
  }
}

// The piece [lo, hi] of a quad by the FP64 rule.
__device__ __noinline__ void piece64(double lo, double hi, double sa, double sb,
                                     const float4* v, float4* p) {
  double f0 = 0.0, f1 = 1.0;
  if (sb > sa) {
    const double d = __dsub_rn(sb, sa);
    f0 = __ddiv_rn(__dsub_rn(lo, sa), d);
    f1 = __ddiv_rn(__dsub_rn(hi, sa), d);
  }
  const float a0[4] = {v[0].x, v[0].y, v[0].z, v[0].w}, a1[4] = {v[1].x, v[1].y, v[1].z, v[1].w};
  float c0[4], c1[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const double dv = __dsub_rn((double)a1[c], (double)a0[c]);
    c0[c] = (float)__dadd_rn((double)a0[c], __dmul_rn(f0, dv));
    c1[c] = (float)__dadd_rn((double)a0[c], __dmul_rn(f1, dv));
  }
  p[0] = make_float4(c0[0], c0[1], c0[2], c0[3]);
  p[1] = make_float4(c1[0], c1[1], c1[2], c1[3]);
}

// Output ribs of a quad by the FP64 walk (out of line, as it is rare).
__device__ __noinline__ int count64(const DashPattern& P, float sa, float sb, int J) {
  DashWalk w;
  w.start(P, sa, sb);
  double lo, hi;
  bool cap0, cap1;
  int n = 0;
  while (w.next(P, J > 0, lo, hi, cap0, cap1)) n += 2 + (cap0 ? J + 1 : 0) + (cap1 ? J + 1 : 0);
  return n;
}

// The same quad's pieces and caps, from out[o] on.
__device__ __noinline__ void quad64(const DashPattern& P, float sa, float sb, int J,
                                    const float4* rib, int64_t r, uint32_t tg, int64_t o,
                                    const DashOut& D, int32_t* status) {
  DashWalk w;
  w.start(P, sa, sb);
  double lo, hi;
  bool cap0, cap1;
  const bool square = J == 4 && P.path_cap[tg >> 2] == PS_CAP_SQUARE;
  while (w.next(P, J > 0, lo, hi, cap0, cap1)) {
    const int64_t o0 = o, op = o + (cap0 ? J + 1 : 0);
    o = op + 2 + (cap1 ? J + 1 : 0);
    if (o > D.cap) {
      ps_record_error(status, PS_ERR_CAPACITY);
      continue;
    }
    const float4 v[2] = {rib[r - 1], rib[r]};
    float4 p[2];
    piece64(lo, hi, w.sa, w.sb, v, p);
    put_piece(D, op, p[0], p[1], (float)lo, (float)hi, tg, (int32_t)r);
    if (cap0)
      emit_cap(make_cap(p[0], true), J, square, 0, 1, tg, (float)lo, (int32_t)r, o0, D.rib, D.s,
               D.tag, D.src);
    if (cap1)
      emit_cap(make_cap(p[1], false), J, square, 0, 1, tg, (float)hi, (int32_t)r, op + 2, D.rib,
               D.s, D.tag, D.src);
  }
}

// Two passes.  The first counts: tiles of 1,024 quads, 128 consecutive ones per
// warp (quad 32 q + lane, so that loads and stores are contiguous over the lanes).
// The FP32 prefilter settles most quads; the others (1.2% of the 5,031-cubic
// path's) are queued per warp and walked densely.  A warp scan of the piece
// counts, the warps' totals through shared memory, and a warp-wide decoupled
// look-back give every quad's output offset, kept with what is to be written as
// one word per quad.  The second pass writes, warps on their own, 256 quads
// each.  A tile's chain (loads, walk, look-back) is all latency: with both passes in
// one kernel, three CTAs an SM for its registers and seven block barriers a tile,
// the 5,031-cubic path took 125 us and 1,000 paths with capped dashes 784 us, and
// 121 and 670 us this way.
enum { DASH_NONE = 0, DASH_WHOLE = 1, DASH_WALK = 2, DASH_WALK64 = 3 };

__global__ void __launch_bounds__(DASH_NT, 5) k_dash_count(
    const float* __restrict__ s, const uint32_t* __restrict__ tag,
    const int64_t* __restrict__ n_rib, int64_t capacity, const __grid_constant__ DashPattern P,
    unsigned long long* __restrict__ word, int64_t* __restrict__ n_out, int64_t out_cap,
    TileState* state, int32_t* counters, int32_t* status) {
  constexpr int WQ = 32 * DASH_QPT;  // quads per warp
  // two copies, used by alternate tiles: a warp may be a tile ahead of another
  __shared__ long long s_total[2][DASH_NT / 32];
  __shared__ long long s_prefix[2];
  __shared__ int64_t s_next[2];
  __shared__ uint8_t s_queue[DASH_NT / 32][WQ];  // a warp's queued quads
  __shared__ uint8_t s_mode[DASH_NT / 32][WQ];
  __shared__ int s_cnt[DASH_NT / 32][WQ];        // their output ribs
  int64_t R = *n_rib;
  if (R > capacity) R = capacity;
  int64_t n_tiles = (R + DASH_TILE - 1) / DASH_TILE;
  if (n_tiles == 0) n_tiles = 1;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (threadIdx.x == 0) s_next[1] = atomicAdd(&counters[3], 1);
  __syncthreads();
  for (int par = 0;; par ^= 1) {
    const int64_t tile = s_next[par ^ 1];
    if (tile >= n_tiles) return;
    const int64_t t0 = tile * DASH_TILE + wid * WQ;
    int cnt[DASH_QPT];  // output ribs; -1: queued
    int qtot = 0;
    {
      float sa[DASH_QPT], sb[DASH_QPT];
      bool quad[DASH_QPT];
#pragma unroll
      for (int q = 0; q < DASH_QPT; ++q) {
        const int64_t r = t0 + 32 * q + lane;
        quad[q] = r >= 1 && r < R;
        sa[q] = sb[q] = 0.f;
        if (quad[q]) {
          quad[q] = !(__ldg(tag + r) & PS_TAG_LINK_START);
          sa[q] = __ldg(s + r - 1);
          sb[q] = __ldg(s + r);
        }
      }
#pragma unroll
      for (int q = 0; q < DASH_QPT; ++q) {
        const int mode = quad[q] ? dash_quick(P, sa[q], sb[q]) : 0;
        cnt[q] = mode < 0 ? -1 : 2 * mode;
        const unsigned qm = __ballot_sync(0xffffffffu, mode < 0);
        if (mode < 0)
          s_queue[wid][qtot + __popc(qm & ((1u << lane) - 1u))] = (uint8_t)(32 * q + lane);
        qtot += __popc(qm);
      }
    }
    __syncwarp();
    for (int i = lane; i < qtot; i += 32) {
      const int lq = s_queue[wid][i];
      const int64_t r = t0 + lq;
      const int J = cap_steps(P, __ldg(tag + r) >> 2);
      DashWalkDF w;
      w.start(P, __ldg(s + r - 1), __ldg(s + r));
      ps::DF a, b;
      bool at_a, at_b, cap0, cap1;
      int n = 0;
      while (w.next(P, J > 0, a, b, at_a, at_b, cap0, cap1))
        n += 2 + (cap0 ? J + 1 : 0) + (cap1 ? J + 1 : 0);
      s_mode[wid][lq] = w.sure ? DASH_WALK : DASH_WALK64;
      s_cnt[wid][lq] = w.sure ? n : count64(P, w.sa, w.sb, J);
    }
    __syncwarp();
    long long off[DASH_QPT];  // of each quad's output in the warp's
    long long wtot = 0;
#pragma unroll
    for (int q = 0; q < DASH_QPT; ++q) {
      const int c = cnt[q] < 0 ? s_cnt[wid][32 * q + lane] : cnt[q];
      long long x = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      off[q] = 4 * (wtot + x - c) +
               (c == 0 ? DASH_NONE : cnt[q] < 0 ? s_mode[wid][32 * q + lane] : DASH_WHOLE);
      wtot += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) s_total[par][wid] = wtot;
    __syncthreads();
    long long total = 0, wpre = 0;
    for (int w = 0; w < DASH_NT / 32; ++w) {
      if (w < wid) wpre += s_total[par][w];
      total += s_total[par][w];
    }
    if (wid == 0) {
      long long pre = lookback_sum_warp(state, total, tile, status);
      if (lane == 0) {
        s_prefix[par] = pre;
        s_next[par] = atomicAdd(&counters[3], 1);  // the tile's prefix is published
        if (tile == n_tiles - 1) {
          *n_out = pre + total;
          if (pre + total > out_cap) ps_record_error(status, PS_ERR_CAPACITY);
        }
      }
    }
    __syncthreads();
    const long long base = 4 * (s_prefix[par] + wpre);
#pragma unroll
    for (int q = 0; q < DASH_QPT; ++q) {
      const int64_t r = t0 + 32 * q + lane;
      if (r < R) word[r] = (unsigned long long)(base + off[q]);
    }
  }
}

constexpr int EMIT_WQ = 256;  // quads per ticket of the writing pass
__global__ void __launch_bounds__(DASH_NT, 3) k_dash(
    const float4* __restrict__ rib, const float* __restrict__ s, const uint32_t* __restrict__ tag,
    const int64_t* __restrict__ n_rib, int64_t capacity, const __grid_constant__ DashPattern P,
    const unsigned long long* word, const __grid_constant__ DashOut D,
    CapTask* __restrict__ tasks, int max_tasks, int32_t* counters, int32_t* status) {
  __shared__ uint8_t s_queue[DASH_NT / 32][EMIT_WQ];  // a warp's queued quads
  dep_wait();
  int64_t R = *n_rib;
  if (R > capacity) R = capacity;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  // warps take the next quads by ticket, as their work differs (caps, long lines
  // with many stretches); a warp's next ticket is drawn while it writes
  int ticket = 0;
  if (lane == 0) ticket = atomicAdd(&counters[7], 1);
  for (;;) {
    const int64_t t0 = (int64_t)__shfl_sync(0xffffffffu, ticket, 0) * EMIT_WQ;
    if (t0 >= R) return;
    if (lane == 0) ticket = atomicAdd(&counters[7], 1);
    int qtot = 0;
#pragma unroll 4
    for (int q = 0; q < EMIT_WQ / 32; ++q) {
      const int64_t r = t0 + 32 * q + lane;
      const unsigned long long wd = r < R ? word[r] : 0ull;
      const int mode = (int)(wd & 3u);
      const int64_t o = (int64_t)(wd >> 2);
      if (mode == DASH_WHOLE) {
        // inside an on-stretch: the quad itself (f0 = 0, f1 = 1 below)
        if (o + 2 <= D.cap) {
          const float4 v0 = __ldg(rib + r - 1), v1 = __ldg(rib + r);
          put_piece(D, o, v0, whole_end(v0, v1), __ldg(s + r - 1), __ldg(s + r), __ldg(tag + r),
                    (int32_t)r);
        } else {
          ps_record_error(status, PS_ERR_CAPACITY);
        }
      }
      const unsigned qm = __ballot_sync(0xffffffffu, mode >= DASH_WALK);
      if (mode >= DASH_WALK)
        s_queue[wid][qtot + __popc(qm & ((1u << lane) - 1u))] = (uint8_t)(32 * q + lane);
      qtot += __popc(qm);
    }
    __syncwarp();
    // queued quads: one per lane, each round one piece of each.  Round caps are left to
    // k_dash_caps, or without its list written by the whole warp (a lane alone
    // would write a cap's 181 ribs at 1 degree in turn: 2.81 ms for 1,000 paths with
    // capped dashes, 24.4 M ribs out, and 1.18 ms by warps; but a line of 200 px
    // has 50 caps, all written by one warp while others had none: 530 us for this
    // kernel, and 290 us and 138 for k_dash_caps with the list)
    for (int i0 = 0; i0 < qtot; i0 += 32) {
      const int lq = i0 + lane < qtot ? s_queue[wid][i0 + lane] : 0;
      bool more = i0 + lane < qtot;
      const int64_t r = t0 + lq;
      int64_t o = 0;
      uint32_t tq = 0u;
      int J = 0;
      float4 v0 = make_float4(0.f, 0.f, 0.f, 0.f), v1 = v0;
      DashWalkDF w{};
      if (more) {
        const unsigned long long wd = word[r];
        o = (int64_t)(wd >> 2);
        tq = __ldg(tag + r);
        J = cap_steps(P, tq >> 2);
        w.start(P, __ldg(s + r - 1), __ldg(s + r));
        if ((wd & 3u) == DASH_WALK) {
          v0 = __ldg(rib + r - 1);
          v1 = __ldg(rib + r);
        } else {
          quad64(P, w.sa, w.sb, J, rib, r, tq, o, D, status);
          more = false;
        }
      }
      const bool square = J == 4 && P.path_cap[tq >> 2] == PS_CAP_SQUARE;
      while (__any_sync(0xffffffffu, more)) {
        bool cap0 = false, cap1 = false, at_a = false, at_b = false;
        ps::DF a{0.f, 0.f}, b{0.f, 0.f};
        if (more) more = w.next(P, J > 0, a, b, at_a, at_b, cap0, cap1);
        float4 p0 = v0, p1 = v1;
        float s0 = w.sa, s1 = w.sb;
        const int64_t o0 = o;                       // a start cap's first rib
        const int64_t op = o + (cap0 ? J + 1 : 0);  // the piece
        if (more) o = op + 2 + (cap1 ? J + 1 : 0);
        if (!more || o > D.cap) {
          if (more) ps_record_error(status, PS_ERR_CAPACITY);
          cap0 = cap1 = false;
        } else {
          // (a vertex that is not finite is left to the FP64 rule)
          bool ok = fabsf(v0.x - v1.x) + fabsf(v0.y - v1.y) + fabsf(v0.z - v1.z) +
                        fabsf(v0.w - v1.w) < INFINITY;
          const ps::DF d = ps::df_diff(w.sb, w.sa);
          const float fe = 2.f * w.err / d.hi;  // (only used when d > 0)
          if (at_a) {
            p0 = cut_rib(v0, v1, ps::df_div(ps::df_add_f(a, -w.sa), d), fe, ok);
            s0 = a.hi;
            ok &= a.hi + (a.lo + w.err) == a.hi && a.hi + (a.lo - w.err) == a.hi;
          }
          if (at_b) {
            p1 = cut_rib(v0, v1, ps::df_div(ps::df_add_f(b, -w.sa), d), fe, ok);
            s1 = b.hi;
            ok &= b.hi + (b.lo + w.err) == b.hi && b.hi + (b.lo - w.err) == b.hi;
          } else {
            p1 = whole_end(v0, v1);
          }
          if (!ok) {  // the stretch's ends in FP64 (k is exact; next() has moved past it)
            const double base = __dmul_rn((double)(w.k0 + (float)w.g), P.period);
            const double lo =
                at_a ? __dsub_rn(__dadd_rn(base, P.cum[w.i - 2]), P.offset) : (double)w.sa;
            const double hi =
                at_b ? __dsub_rn(__dadd_rn(base, P.cum[w.i - 1]), P.offset) : (double)w.sb;
            const float4 v[2] = {v0, v1};
            float4 p[2];
            piece64(lo, hi, (double)w.sa, (double)w.sb, v, p);
            p0 = p[0];
            p1 = p[1];
            s0 = (float)lo;
            s1 = (float)hi;
          }
          put_piece(D, op, p0, p1, s0, s1, tq, (int32_t)r);
        }
#pragma unroll 1
        for (int end = 0; end < 2; ++end) {
          const bool cap = end ? cap1 : cap0;
          if (!__any_sync(0xffffffffu, cap)) continue;
          DashCap C{0.f, 0.f, 0.f, 0.f};
          if (cap) C = make_cap(end ? p1 : p0, end == 0);
          const int64_t oc = end ? op + 2 : o0;
          const float sv = end ? s1 : s0;
          const bool shared = cap && J > 4;
          if (cap && !shared)
            emit_cap(C, J, square, 0, 1, tq, sv, (int32_t)r, oc, D.rib, D.s, D.tag, D.src);
          const unsigned sm = __ballot_sync(0xffffffffu, shared);
          if (tasks) {
            if (!sm) continue;
            const int lead = __ffs(sm) - 1;
            int at = 0;
            if (lane == lead) at = atomicAdd(&counters[8], __popc(sm));
            at = __shfl_sync(0xffffffffu, at, lead) + __popc(sm & ((1u << lane) - 1u));
            // (the list holds a cap for every j_round + 1 output ribs; more come up only when
            // a look-back gave up and output ranges overlap: PS_ERR_TIMEOUT is recorded)
            if (shared && at < max_tasks) tasks[at] = CapTask{C, tq, sv, (int32_t)r, 0, oc};
            continue;
          }
          for (unsigned m = sm; m; m &= m - 1u) {
            const int from = __ffs(m) - 1;
            DashCap B;
            B.cx = __shfl_sync(0xffffffffu, C.cx, from);
            B.cy = __shfl_sync(0xffffffffu, C.cy, from);
            B.r = __shfl_sync(0xffffffffu, C.r, from);
            B.psi0 = __shfl_sync(0xffffffffu, C.psi0, from);
            emit_cap(B, __shfl_sync(0xffffffffu, J, from), false, lane, 32,
                     __shfl_sync(0xffffffffu, tq, from), __shfl_sync(0xffffffffu, sv, from),
                     __shfl_sync(0xffffffffu, (int32_t)r, from),
                     __shfl_sync(0xffffffffu, oc, from), D.rib, D.s, D.tag, D.src);
          }
        }
      }
    }
    __syncwarp();
  }
}

// Round caps, a warp to each.
__global__ void __launch_bounds__(DASH_NT) k_dash_caps(const CapTask* tasks,
                                                       int max_tasks, int J,
                                                       const __grid_constant__ DashOut D,
                                                       const int32_t* counters) {
  dep_wait();
  const int n = min(counters[8], max_tasks), lane = threadIdx.x & 31;
  const int stride = gridDim.x * (DASH_NT / 32);
  for (int i = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; i < n; i += stride) {
    const CapTask T = tasks[i];
    emit_cap(T.cap, J, false, lane, 32, T.tag, T.s, T.src, T.o, D.rib, D.s, D.tag, D.src);
  }
}

}  // namespace

extern "C" int ps_dash_capped(ps_context* ctx, const float* d_rib, const float* d_s,
                              const uint32_t* d_tag, const int64_t* d_n_rib, int64_t capacity,
                              const float* h_pattern, int n_pattern, float offset,
                              const uint8_t* d_path_cap, int32_t n_path, float dtheta,
                              float* d_out_rib, float* d_out_s, uint32_t* d_out_tag,
                              int32_t* d_out_src, int64_t* d_n_out, int64_t out_capacity,
                              void* stream) {
  if (!ctx || !d_rib || !d_s || !d_tag || !d_n_rib || !h_pattern || !d_out_rib || !d_out_s ||
      !d_out_tag || !d_n_out || capacity < 0 || out_capacity < 0)
    return PS_ERR_INVALID;
  if (d_path_cap && (n_path < 0 || !(dtheta >= 1e-4f && dtheta <= 3.14159265f)))
    return PS_ERR_INVALID;
  if (n_pattern < 1 || n_pattern > 32 || !(offset == offset)) return PS_ERR_INVALID;
  DashPattern P;
  if (!dash_pattern(P, h_pattern, n_pattern, offset)) return PS_ERR_INVALID;
  P.path_cap = d_path_cap;
  P.n_path = d_path_cap ? n_path : 0;
  P.j_round = 0;
  if (d_path_cap) {
    // a round cap turns pi in steps of at most q (a ratio within 1e-4 step above
    // an integer takes that integer, as for every turning count)
    double x = 3.14159265358979323846 / (double)dtheta;
    int J = (int)ceil(x - 1e-4);
    P.j_round = J < 1 ? 1 : J;
  }
  cudaStream_t st = (cudaStream_t)stream;
  ps_on_stream(ctx, stream);
  int64_t n_tiles = (capacity + DASH_TILE - 1) / DASH_TILE + 1;
  int rc = ps_ensure_tiles(ctx, n_tiles + 1);
  if (rc != PS_OK) return rc;
  cudaMemsetAsync(ctx->d_counters, 0, 64 + sizeof(TileState) * (n_tiles + 1), st);
  // A word of 8 bytes per quad: the context's, or under a capture that finds too few there,
  // the graph's own (a capture allows no cudaMalloc, and before the words a dash needed none).
  unsigned long long* word = nullptr;
  bool graph_word = false;
  if (capacity > ctx->quad_hits_cap) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    graph_word = cudaStreamIsCapturing(st, &cs) == cudaSuccess && cs == cudaStreamCaptureStatusActive;
  }
  if (graph_word)
    rc = ps_cuda_check(cudaMallocAsync((void**)&word, sizeof(*word) * (size_t)capacity, st));
  else if ((rc = ps_ensure_quad_hits(ctx, capacity)) == PS_OK)
    word = reinterpret_cast<unsigned long long*>(ctx->d_quad_hits);
  if (rc != PS_OK) return rc;
  const DashOut D{reinterpret_cast<float4*>(d_out_rib), d_out_s, d_out_tag, d_out_src, out_capacity};
  const int grid0 =
      ps_grid_for(ps_persistent_grid(ctx, (const void*)k_dash_count, DASH_NT, 0), capacity, DASH_TILE);
  const int grid1 = ps_grid_for(ps_persistent_grid(ctx, (const void*)k_dash, DASH_NT, 0), capacity,
                                DASH_NT / 32 * EMIT_WQ);
  // Room for every round cap (each fills j_round + 1 ribs of the output).  Without it (no
  // memory, or a capture under way and no room from an earlier call) the writing
  // pass writes them itself.
  CapTask* tasks = nullptr;
  const int max_tasks = (int)std::min<int64_t>(out_capacity / (P.j_round + 1) + 1, INT32_MAX);
  if (P.path_cap && P.j_round > 4) {
    const size_t need = sizeof(CapTask) * (size_t)max_tasks;
    if (need > ctx->cap_bytes) {
      cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
      if (cudaStreamIsCapturing(st, &cs) == cudaSuccess && cs == cudaStreamCaptureStatusNone) {
        const size_t room = (size_t)ps_grown(ctx, (int64_t)ctx->cap_bytes, (int64_t)need);
        ctx->cap_bytes = 0;
        if (ps_grow(ctx, &ctx->d_cap_tasks, room) == PS_OK) ctx->cap_bytes = room;  // else carry on without
      }
    }
    if (need <= ctx->cap_bytes) tasks = static_cast<CapTask*>(ctx->d_cap_tasks);
  }
  const int grid2 = ps_grid_for(ps_persistent_grid(ctx, (const void*)k_dash_caps, DASH_NT, 0),
                                max_tasks, 1);
  ProfScope ps_(ctx, PK_DASH, st);
  k_dash_count<<<grid0, DASH_NT, 0, st>>>(d_s, d_tag, d_n_rib, capacity, P, word, d_n_out,
                                                    out_capacity, ctx->d_tile_state, ctx->d_counters,
                                                    ctx->d_status);
  // (one profile slot for all three: no event records in between)
  ps_launch_after(true, &k_dash, grid1, DASH_NT, 0, st, reinterpret_cast<const float4*>(d_rib), d_s,
                  d_tag, d_n_rib, capacity, P, word, D, tasks, max_tasks, ctx->d_counters, ctx->d_status);
  if (tasks)
    ps_launch_after(true, &k_dash_caps, grid2, DASH_NT, 0, st, tasks, max_tasks, P.j_round, D,
                    ctx->d_counters);
  rc = ps_cuda_check(cudaGetLastError());
  if (graph_word && cudaFreeAsync(word, st) != cudaSuccess && rc == PS_OK) rc = PS_ERR_CUDA;
  return rc;
}

extern "C" int ps_dash(ps_context* ctx, const float* d_rib, const float* d_s,
                       const uint32_t* d_tag, const int64_t* d_n_rib, int64_t capacity,
                       const float* h_pattern, int n_pattern, float offset, float* d_out_rib,
                       float* d_out_s, uint32_t* d_out_tag, int32_t* d_out_src, int64_t* d_n_out,
                       int64_t out_capacity, void* stream) {
  return ps_dash_capped(ctx, d_rib, d_s, d_tag, d_n_rib, capacity, h_pattern, n_pattern, offset,
                        nullptr, 0, 1.f, d_out_rib, d_out_s, d_out_tag, d_out_src, d_n_out,
                        out_capacity, stream);
}
