// gf_coop.cuh -- one ray per warp: the warp traverses the ray's tree together
// and shares out its chords.
#pragma once
#include <cstddef>

#include "gf_device.cuh"
#include "gf_trace.cuh"

namespace gf {

struct BlockTables {
  float glx[kGLTotal], glw[kGLTotal];
  float env[8];
};

__device__ __forceinline__ void init_tables(BlockTables& sm, const DevField& F) {
  for (int i = threadIdx.x; i < kGLTotal; i += blockDim.x) {
    sm.glx[i] = F.gl[i];
    sm.glw[i] = F.gl[kGLTotal + i];
  }
  if (threadIdx.x < 8) sm.env[threadIdx.x] = F.env[threadIdx.x];
  __syncthreads();
}

// the next work item of a persistent grid, the same in every lane (unsigned: the
// last warps step past a batch of up to 2^31 - 1 items)
__device__ __forceinline__ uint32_t next_tile(int* counter, uint32_t lane) {
  uint32_t it = 0;
  if (lane == 0) it = (uint32_t)atomicAdd(counter, 1);
  return __shfl_sync(kFull, it, 0);
}

// The rays of a batch, taken by warps up to 32 at a time: lane l looks at the l-th of them,
// and the warp goes through those that meet the scene, while the others are answered by one
// lane.  2,000,000 rays that miss took 1.4 ms at a warp each, 0.1 ms now.  The state lies in
// shared memory, so that nothing of it is live while a ray is in work.
struct WarpItems {
  uint32_t from, todo;        // first of the items in hand, bits of those still to do
  unsigned long long missed;  // rays answered by one lane
};
__device__ __forceinline__ void init_items(WarpItems& S, uint32_t lane) {
  if (lane == 0) {
    S.from = S.todo = 0u;
    S.missed = 0ull;
  }
  __syncwarp();
}
// the next of n items, the same in every lane; kNoItem at the end.  look(item), by one lane: -1
// when it is worth a warp's time, else the number of rays that it has answered.  A warp
// takes a quarter of its even share of what is left, and one by one at the end (those
// unseen), so that the warps finish together.
constexpr uint32_t kNoItem = 0xFFFFFFFFu;
template <class Look>
__device__ __forceinline__ uint32_t next_item(WarpItems& S, int* counter, uint32_t n, uint32_t lane,
                                              Look&& look) {
  uint32_t from = S.from, todo = S.todo;
  while (todo == 0u) {
    const uint32_t k = min(32u, max(1u, (n - from) / (4u * gridDim.x * (blockDim.x >> 5))));
    uint32_t it = 0;
    if (lane == 0) it = (uint32_t)atomicAdd(counter, (int)k);
    from = __shfl_sync(kFull, it, 0);
    if (from >= n) return kNoItem;
    if (k == 1u) {
      todo = 1u;
    } else {
      const int missed = lane < min(k, n - from) ? look(from + lane) : 0;
      todo = __ballot_sync(kFull, missed < 0);
      const int m = __reduce_add_sync(kFull, max(missed, 0));
      if (lane == 0) S.missed += (unsigned long long)m;
    }
  }
  __syncwarp();  // every lane has read
  if (lane == 0) {
    S.from = from;
    S.todo = todo & (todo - 1u);
  }
  __syncwarp();
  return from + (uint32_t)__ffs((int)todo) - 1u;
}
// whether a ray meets the scene's bounds
__device__ __forceinline__ bool meets_scene(const DevField& F, float3 o, float3 v, float tmin, float tmax) {
  float t0, t1;
  return scene_span(F, o, safe_inv(v), tmin, tmax, t0, t1);
}

// The pixels whose rays can meet the scene (PathParams::roi), row by row: pixel i of them.
// The warps take these one by one in order, so that neighbours run at the same time and find
// the same tree nodes in the caches (taken 32 in a row: 13.2 -> 15.4 ms for a 1024x1024
// flight image through 1000 kernels); the background is filled by the launcher.
__device__ __forceinline__ int roi_pixel(const PathParams& P, uint32_t i) {
  return (P.roi_y + (int)(i / (uint32_t)P.roi_w)) * P.cam.W + P.roi_x + (int)(i % (uint32_t)P.roi_w);
}

// Traversal of one ray by a whole warp, from the roots of the trees its mask needs: a
// shared stack of four-wide nodes, up to 32 popped per step (one per lane) and their hit children pushed; the leaves
// reached are queued, and every 32 queued leaves (and the last ones) make a
// round, in which round(j) is called by every lane, j the sorted primitive of the
// lane's leaf or -1.
//
// The ray lives in registers (the same in every lane), so a step has no lane-
// dependent ray data and no branch that parts the lanes.  A step pushes at most
// 128 nodes; above kCoopStack - kCoopMargin entries the warp goes depth first
// (one node per step, at most 3 more entries per tree level, 32 levels), so the
// stack holds a full step plus a whole descent.
constexpr int kCoopStack = 512;
constexpr int kCoopMargin = 200;
constexpr int kCoopLeafQ = 160;  // <= 31 left + 128 new
static_assert(kCoopStack - kCoopMargin + 96 + 3 * 32 <= kCoopStack, "a full step, then a descent");
struct CoopTrav {
  int stk[kCoopStack];
  int lq[kCoopLeafQ];  // directly behind the stack (push_hits)
};
static_assert(offsetof(CoopTrav, lq) == kCoopStack * sizeof(int), "queue behind the stack");

template <class Round>
__device__ __forceinline__ void coop_traverse(const DevField& F, CoopTrav& Q,
                                              unsigned long long mask, float3 o, float3 inv,
                                              float t0, float t1, uint32_t lane, Counters& cnt,
                                              Round&& round) {
  int sp = 0, lq_n = 0;
  {
    unsigned long long cm;
    unsigned bm;
    tree_roots(mask, cm, bm);
    while (cm | bm) {
      const int r = next_root(F, cm, bm);
      if (lane == 0) Q.stk[sp] = r;
      ++sp;
    }
  }
  __syncwarp();
  // every node enters the stack at most once
  const long long max_it = F.n_nodes4 + 64;
  for (long long it = 0;; ++it) {
    if (it > max_it) {
      if (lane == 0) set_err(F, ERR_GUARD);
      break;
    }
    int take = sp < 32 ? sp : 32;
    if (sp > kCoopStack - kCoopMargin) take = 1;  // near capacity: depth first
    const int node = (int)lane < take ? Q.stk[sp - take + (int)lane] : -1;
    __syncwarp();
    sp -= take;
    int ch[4] = {0, 0, 0, 0};
    unsigned hit = 0u;
    if (node >= 0 && (int64_t)node >= F.n_nodes4) {
      set_err(F, ERR_INDEX);  // a node beyond the tree: skipped
    } else if (node >= 0) {
      ++cnt.nodes;
      hit = node4_hits(F.nodes4 + node, o, inv, t0, t1, ch);
    }
    if (!push_hits(Q.stk, kCoopStack, hit, ch, lane, sp, lq_n, [](int, int c) { return c; }) && lane == 0)
      set_err(F, ERR_STACK);
    __syncwarp();
    const bool more = sp > 0;
    while (lq_n >= 32 || (!more && lq_n > 0)) {
      const int tk = lq_n < 32 ? lq_n : 32;
      int j = (int)lane < tk ? Q.lq[lq_n - tk + (int)lane] : -1;
      __syncwarp();
      lq_n -= tk;
      if (j >= 0) ++cnt.leaves;
      if ((int64_t)j >= F.n) {  // a leaf beyond the records
        set_err(F, ERR_INDEX);
        j = -1;
      }
      round(j);
      __syncwarp();
    }
    if (!more && lq_n == 0) break;
  }
}

// inclusive prefix sum over the warp's lanes
__device__ __forceinline__ int warp_incl_sum(int x, uint32_t lane) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int y = __shfl_up_sync(kFull, x, d);
    if ((int)lane >= d) x += y;
  }
  return x;
}

// the lanes' compensated sums combined in a fixed butterfly order: every lane
// receives the total as a pair
__device__ __forceinline__ void warp_sum_pair(float& s, float& c) {
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const float so = __shfl_xor_sync(kFull, s, off), co = __shfl_xor_sync(kFull, c, off);
    float t, e;
    two_sum(s, so, t, e);
    s = t;
    c = __fadd_rn(__fadd_rn(c, co), e);
  }
}

// ---------------------------------------------------------------------------
// Optical depth of one ray (Eq. 2-3).  A round sets up the chords of 32 leaves,
// one per lane.  Gauss-Legendre mode: the nodes of those chords are shared out
// evenly among the lanes (the rule per chord by gl_rule): every chord writes
// its lane number over its stretch of the round's node list, so that node f of the
// round finds its chord with one byte load.  Closed form: each lane integrates its
// own chord.  Every term goes into its lane's compensated sum.
// ---------------------------------------------------------------------------
struct CoopChord {
  float mid, hl, y2, y1, y0, scale, B, delta;
  int off;  // first node of the chord's rule in the tables, less its start in the round
};
struct CoopQ {
  CoopTrav t;
  CoopChord ch[32];  // the round's chords, one per lane
  unsigned char own[32 * gl_n(kNumRules - 1)];  // node of the round -> lane of its chord
};

template <int MODE>  // GF_TR_DETERMINISTIC or GF_TR_CLOSED_FORM
__device__ __forceinline__ void coop_tau(const DevField& F, CoopQ& Q, const Mask& M, float3 o,
                                         float3 v, float tmin, float tmax, const float* glx,
                                         const float* glw, uint32_t lane, float& s_acc,
                                         float& c_acc, Counters& cnt) {
  const float3 inv = safe_inv(v);
  float t0, t1;
  if (M.bits == 0ull || !scene_span(F, o, inv, tmin, tmax, t0, t1)) return;
  if (lane == 0) cnt.windows += 1;
  coop_traverse(F, Q.t, M.bits, o, inv, t0, t1, lane, cnt, [&](int j) {
    int n = 0, off = 0;
    Chord ch;
    float w;
    const bool ok = j >= 0 && prim_chord(F, j, o, v, tmin, tmax,
                                         [&](uint32_t cl) { return mask_weight(M, cl); }, w, ch);
    if (ok) ++cnt.chords;
    if (MODE == GF_TR_CLOSED_FORM) {
      if (ok) neumaier_add(s_acc, c_acc, w * chord_closed(F.wd, ch));
      return;
    }
    const float len = ch.dtout - ch.dtin;
    if (ok) gl_pick(gl_rule(sqrtf(ch.a) * len + 0.5f * fabsf(ch.B) * len), n, off);
    cnt.evals += n;
    const int incl = warp_incl_sum(n, lane);
    const int total = __shfl_sync(kFull, incl, 31);
    if (ok) {
      const int start = incl - n;
      CoopChord C;
      C.mid = 0.5f * (ch.dtin + ch.dtout);
      C.hl = 0.5f * len;
      C.y2 = -0.5f * kLog2e * ch.a;
      C.y1 = -kLog2e * ch.b;
      C.y0 = -0.5f * kLog2e * ch.g;
      C.scale = w * ch.absA * C.hl;
      C.B = ch.B;
      C.delta = ch.delta;
      C.off = off - start;
      Q.ch[lane] = C;
      // rules hold a multiple of 4 nodes, so a stretch is whole 32-bit words
      uint32_t* own4 = reinterpret_cast<uint32_t*>(Q.own) + (start >> 2);
      for (int k = 0; k < (n >> 2); ++k) own4[k] = lane * 0x01010101u;
    }
    __syncwarp();
    for (int f = (int)lane; f < total; f += 32) {
      const CoopChord& C = Q.ch[Q.own[f]];
      const int k = C.off + f;
      const float dt = fmaf(C.hl, glx[k], C.mid);
      const float y = fmaf(fmaf(C.y2, dt, C.y1), dt, C.y0);
      neumaier_add(s_acc, c_acc, C.scale * glw[k] * ex2f(y) * cosf(fmaf(C.B, dt, C.delta)));
    }
  });
}

// ---------------------------------------------------------------------------
// Analytic free flight of one ray (Sec. 3 Eq. 5, Sec. 4.4 distance sampling).  The
// optical depth tau(0, t) is the sum of the closed-form chord integrals up to t; with
// xi the first uniform of the segment's tracking stream, the flight looks for
// tau(0, t) = -ln(1 - xi).
//
// One traversal collects the ray's chords in the warp's list with their full
// integrals; the bisections then work on the list.  A ray with more chords than the
// list holds traverses for each of up to 33 depths.
// ---------------------------------------------------------------------------
constexpr int kFlightList = 4096;  // chords per warp (global scratch)
constexpr int kFlightActive = 512; // chords that a bisection still has to clip
struct FlightRec {
  float tc, dtin, dtout, a, b, g, B, delta, absA, qmin, dts, w;
  float full;  // w times the integral over the whole chord
  float pad[3];
};
static_assert(sizeof(FlightRec) == 64, "chord records of 64 bytes");
struct FlightQ {
  CoopTrav t;
  unsigned short act[kFlightActive];
};
struct Flight {
  FlightRec* list;
  int cap;         // chords the list holds (0: no list)
  int n;           // chords of the ray (may exceed cap)
  float tau, tend; // total optical depth and last chord exit
};

__device__ __forceinline__ Chord flight_chord(const FlightRec& r) {
  Chord c{};
  c.tc = r.tc;
  c.dtin = r.dtin;
  c.dtout = r.dtout;
  c.a = r.a;
  c.b = r.b;
  c.g = r.g;
  c.B = r.B;
  c.delta = r.delta;
  c.absA = r.absA;
  c.qmin = r.qmin;
  c.dts = r.dts;
  return c;
}

__device__ __forceinline__ float warp_max(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(kFull, x, o));
  return x;
}

// chords, total optical depth and last exit of the ray
static __device__ __noinline__ void flight_gather(const DevField& F, FlightQ& Q, const Mask& M, float3 o,
                                           float3 v, uint32_t lane, Flight& L, Counters& cnt) {
  const float3 inv = safe_inv(v);
  float t0, t1, s = 0.f, c = 0.f, tend = -INFINITY;
  L.n = 0;
  L.tau = 0.f;
  L.tend = -INFINITY;
  if (M.bits == 0ull || !scene_span(F, o, inv, 0.f, INFINITY, t0, t1)) return;
  if (lane == 0) cnt.windows += 1;
  int n = 0;
  coop_traverse(F, Q.t, M.bits, o, inv, t0, t1, lane, cnt, [&](int j) {
    Chord ch;
    float w;
    const bool ok = j >= 0 && prim_chord(F, j, o, v, 0.f, INFINITY,
                                         [&](uint32_t cl) { return mask_weight(M, cl); }, w, ch);
    const unsigned b = __ballot_sync(kFull, ok);
    if (ok) {
      ++cnt.chords;
      const float full = w * chord_closed(F.wd, ch);
      neumaier_add(s, c, full);
      tend = fmaxf(tend, ch.tc + ch.dtout);
      const int k = n + __popc(b & ((1u << lane) - 1u));
      if (k < L.cap) {
        float4* d = reinterpret_cast<float4*>(L.list + k);
        d[0] = make_float4(ch.tc, ch.dtin, ch.dtout, ch.a);
        d[1] = make_float4(ch.b, ch.g, ch.B, ch.delta);
        d[2] = make_float4(ch.absA, ch.qmin, ch.dts, w);
        d[3] = make_float4(full, 0.f, 0.f, 0.f);
      }
    }
    n += __popc(b);
  });
  warp_sum_pair(s, c);
  L.n = n;
  L.tau = __fadd_rn(s, c);
  L.tend = warp_max(tend);
  __syncwarp();
}

// the part of chord r in [0, mid] added to (s, c)
__device__ __forceinline__ void flight_part(const DevField& F, const FlightRec& r, float mid, float& s,
                                            float& c) {
  const float hi = fminf(r.dtout, mid - r.tc);
  if (!(r.dtin < hi)) return;
  if (hi == r.dtout) {
    neumaier_add(s, c, r.full);
    return;
  }
  Chord ch = flight_chord(r);
  ch.dtout = hi;
  neumaier_add(s, c, r.w * chord_closed(F.wd, ch));
}

// fn(record) for every chord of the ray, each in some lane
template <class Fn>
__device__ __forceinline__ void flight_each(const DevField& F, FlightQ& Q, const Mask& M, float3 o,
                                            float3 v, float tmax, uint32_t lane, const Flight& L,
                                            Counters& cnt, Fn&& fn) {
  if (L.n <= L.cap) {
    for (int k = (int)lane; k < L.n; k += 32) fn(L.list[k]);
    return;
  }
  const float3 inv = safe_inv(v);
  float t0, t1;
  if (!scene_span(F, o, inv, 0.f, tmax, t0, t1)) return;
  coop_traverse(F, Q.t, M.bits, o, inv, t0, t1, lane, cnt, [&](int j) {
    Chord ch;
    float w;
    if (j < 0 || !prim_chord(F, j, o, v, 0.f, INFINITY,
                             [&](uint32_t cl) { return mask_weight(M, cl); }, w, ch))
      return;
    fn(FlightRec{ch.tc, ch.dtin, ch.dtout, ch.a, ch.b, ch.g, ch.B, ch.delta, ch.absA, ch.qmin, ch.dts,
                 w, w * chord_closed(F.wd, ch), {0.f, 0.f, 0.f}});
  });
}

// CDF inversion: 32 bisections of [0, last chord exit].  Chords that end before the
// bracket keep their full integrals in the lanes' sums, chords that begin behind it
// leave, so that after a few steps a depth takes the chords around the bracket only.
// The first crossing needs a non-negative density along the ray.
static __device__ __noinline__ float cdf_flight(const DevField& F, FlightQ& Q, const Mask& M, float3 o,
                                         float3 v, float target, uint32_t lane, const Flight& L,
                                         Counters& cnt) {
  const unsigned lt = (1u << lane) - 1u;
  const bool listed = L.n <= L.cap;
  float lo = 0.f, hi = L.tend;
  float sb = 0.f, cb = 0.f;  // the lane's chords that end before the bracket
  int na = -1;               // chords in Q.act; -1: every chord is in play
  for (int it = 0; it < 32; ++it) {
    const float mid = 0.5f * (lo + hi);
    float s = sb, c = cb;
    if (na < 0)
      flight_each(F, Q, M, o, v, mid, lane, L, cnt, [&](const FlightRec& r) { flight_part(F, r, mid, s, c); });
    else
      for (int k = (int)lane; k < na; k += 32) flight_part(F, L.list[Q.act[k]], mid, s, c);
    warp_sum_pair(s, c);
    if (__fadd_rn(s, c) < target) lo = mid;
    else hi = mid;
    if (!listed) continue;
    // the chords a depth inside the bracket still clips
    const int m = na >= 0 ? na : L.n;
    int n2 = 0;
    __syncwarp();
    for (int b = 0; b < m && n2 <= kFlightActive; b += 32) {
      const int k = b + (int)lane;
      const int idx = k < m ? (na >= 0 ? (int)Q.act[k] : k) : 0;
      bool keep = false;
      if (k < m) {
        const FlightRec& r = L.list[idx];
        const bool before = r.dtout <= lo - r.tc;
        keep = !before && r.dtin < hi - r.tc;
        if (before && na >= 0) neumaier_add(sb, cb, r.full);
      }
      const unsigned bk = __ballot_sync(kFull, keep);
      const int pos = n2 + __popc(bk & lt);
      if (keep && pos < kFlightActive) Q.act[pos] = (unsigned short)idx;
      n2 += __popc(bk);
      __syncwarp();
    }
    if (na < 0) {
      if (n2 > kFlightActive) continue;  // too many yet: every chord stays in play
      for (int k = (int)lane; k < L.n; k += 32) {
        const FlightRec& r = L.list[k];
        if (r.dtout <= lo - r.tc) neumaier_add(sb, cb, r.full);
      }
    }
    na = n2;
  }
  return 0.5f * (lo + hi);
}

// Uniform sampling within the crossing segment (Sec. 3: the cheap approximation of the
// CDF inversion; Sec. 4.4 distance sampling).  The ray is cut into segments at t = 0 and
// at every chord entry and exit; the segment [e_a, e_b] in which tau(0, t) reaches the
// target holds the collision e_a + u (e_b - e_a).  It is found by bisection on t that
// stops once no chord end lies inside the bracket: every step takes tau(0, mid), the
// chord ends inside both halves of the bracket and the nearest ends around them.
struct SegmentEnds {
  int n_left = 0, n_right = 0;              // chord ends in (lo, mid) and in (mid, hi)
  float below_lo = 0.f, below_mid = 0.f;    // largest end <= lo, <= mid (or 0)
  float above_mid = INFINITY, above_hi = INFINITY;  // smallest end >= mid, >= hi
  __device__ __forceinline__ void add(float e, float lo, float mid, float hi) {
    n_left += (e > lo && e < mid) ? 1 : 0;
    n_right += (e > mid && e < hi) ? 1 : 0;
    if (e <= lo) below_lo = fmaxf(below_lo, e);
    if (e <= mid) below_mid = fmaxf(below_mid, e);
    if (e >= mid) above_mid = fminf(above_mid, e);
    if (e >= hi) above_hi = fminf(above_hi, e);
  }
};
// chord r's ends into E, its part in [0, mid] into (s, c)
__device__ __forceinline__ void segment_part(const DevField& F, const FlightRec& r, float lo, float mid, float hi,
                                             SegmentEnds& E, float& s, float& c) {
  const float tin = r.tc + r.dtin, tout = r.tc + r.dtout;
  E.add(tin, lo, mid, hi);
  E.add(tout, lo, mid, hi);
  if (tin >= mid) return;
  if (!(tout > mid)) {
    neumaier_add(s, c, r.full);
  } else {  // the chord's part in [0, mid]
    Chord ch = flight_chord(r);
    ch.dtout = mid - r.tc;
    neumaier_add(s, c, r.w * chord_closed(F.wd, ch));
  }
}
static __device__ __noinline__ float segment_flight(const DevField& F, FlightQ& Q, const Mask& M, float3 o,
                                             float3 v, float target, float u, uint32_t lane,
                                             const Flight& L, Counters& cnt) {
  float lo = 0.f, hi = L.tend;
  float ea = 0.f, eb = L.tend;
  for (int it = 0; it < 48; ++it) {
    const float mid = 0.5f * (lo + hi);
    float s = 0.f, c = 0.f;
    SegmentEnds E;
    flight_each(F, Q, M, o, v, INFINITY, lane, L, cnt,
                [&](const FlightRec& r) { segment_part(F, r, lo, mid, hi, E, s, c); });
    warp_sum_pair(s, c);
    if (__fadd_rn(s, c) < target) {
      lo = mid;
      ea = warp_max(E.below_mid);
      eb = -warp_max(-E.above_hi);
      if (__reduce_add_sync(kFull, E.n_right) == 0) break;
    } else {
      hi = mid;
      ea = warp_max(E.below_lo);
      eb = -warp_max(-E.above_mid);
      if (__reduce_add_sync(kFull, E.n_left) == 0) break;
    }
    if (!(hi > lo)) break;
  }
  if (!(eb < INFINITY)) eb = L.tend;
  return ea + u * (eb - ea);
}

}  // namespace gf
