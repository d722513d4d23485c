// gf_wavefront.cu -- scattering renderer: lanes traverse, the warp processes.
//
// Every lane of a warp owns one path (one pixel's samples in order).  The
// warp traverses the BVH for all 32 current rays together: one shared stack
// of (node, lane) entries, from which every step pops up to 32 entries, so the
// lanes stay busy while rays of different lengths are in flight.  Leaves that
// are reached go to a per-warp queue in shared memory, and whenever 32 are
// queued the whole warp sets up their chords at once (chord set-up on the
// owning lane's ray).  Each chord that overlaps the owner's window [ta, te)
// is stored (its evaluation record, in a per-warp global store) and queued;
// queued chords are walked 32 at a time, one draw per chord and round, each
// drawing the chord's next tentative point of Sec. 3's per-segment majorant
// from its own Philox stream (chords that may hold more points go back to the
// queue, so the lanes stay busy).  Points land in
// the owner's buffer through shared-memory atomics.  kappa and kappa_bar at
// the points are then summed from the stored records, a lane (or several) per
// point, after which each lane takes its delta-tracking or
// ratio-tracking decision and moves its path on (camera ray -> collision ->
// NEE -> scattering).
//
// The tentative points are a function of the chords and their Philox streams
// only, so results equal a per-ray formulation up to floating-point summation
// order.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstddef>

#include "gf_host.h"
#include "gf_trace.cuh"
#include "gf_window.h"
#include "gf_words.h"

namespace gf {

constexpr int kWWarps = 4;      // warps per block
constexpr int kBlocksPerSM = 4; // resident blocks per SM the kernels are built for
constexpr int kLeafQ = 288;     // queued leaves per warp (<= 31 left + 256 new)
constexpr int kChordQ = 64;     // queued chords per warp (<= 31 left + 32 new)
// A window with more points or chords than its slot holds is halved and traversed
// again.  13 points fill the shared memory of 4 blocks per SM.  Against 8 points and 256
// chords: 1024x1024, 8 samples, 1M kernels, stochastic masks 214 -> 193.5 ms; 512x512, 16
// samples, 100k kernels 93.8 -> 92.0 ms; 120x67, 1 sample, 50k kernels 310 -> 215 us.
constexpr int kPK = 13;         // tentative points per lane and window
constexpr int kSlotCh = 448;    // stored chords per lane and window (global scratch)
constexpr float kFill = 0.7f;     // share of them that a ray's windows aim at (0.5 to 0.9: within 4 %)
constexpr int kHits = 40;         // covering chords a lane collects before it evaluates them
static_assert(kSlotCh % 4 == 0, "spans are read four at a time");
// A warp's stored chords, per slot: entry and exit (8 bytes each, read by themselves
// while points look for the chords that cover them), and the records.
struct ChordStore {
  float2 span[32][kSlotCh];
  float4 rec[32][kSlotCh][2];  // (t*, t_in, t_out, B), (-a log2(e) / 2, log2 h, phase at t*, sqrt(a))
};
static_assert(sizeof(float2) * 32 * kSlotCh % 32 == 0, "records on 32-byte boundaries");

// One slot per lane, 57 words: an odd stride keeps same-field accesses of the
// 32 slots in distinct shared-memory banks.
struct LaneRay {
  float o[3], v[3], inv[3];
  float ta, te;                 // window [ta, te) of the ray (which spans t >= 0)
  uint32_t ray, word;
  uint32_t seed_lo, seed_hi;    // Philox key of the path's render
  int asset;                    // field of the path
  float bw[8];                  // LoD band weights
  uint32_t cx[2];               // per band: one cone with an extra weight factor (Mask::cx)
  uint32_t mask_lo, mask_hi;    // LoD cell bits
  int npts;                     // points emitted in the window (may exceed kPK)
  int nch;                      // chords stored for the window (may exceed kSlotCh)
  int hmax;                     // bits of the largest chord peak h of the window (h >= 0)
  float pt[kPK], pu[kPK];       // the window's tentative points (t, acceptance uniform)
};
static_assert(sizeof(LaneRay) % 8 == 4, "odd word stride");
static_assert(kSlotCh <= 448, "sums of kSlotCh terms below 2^54 (1 + 1e-6) stay below 2^63");
struct ChordItem {
  float tc;
  float dt;           // where the walk stands (relative to tc): the chord's entry, then
                      // the last point drawn
  float dtout, h, sa, dts;
  uint32_t jd;        // majorant pieces per side J (3 bits) | next draw << 3
  uint32_t orig_own;  // original primitive index | owning slot << 26
};
static_assert(sizeof(ChordItem) == 32, "chord items of 32 bytes");
// Shared (node, slot) stack entries per warp: the first roots (32 slots of up to
// kMaxRoots), and a margin of 3 entries per level of a descent (32 four-wide levels).
constexpr int kWStack = 640;
constexpr int kStackMargin = 96;
static_assert(32 * kMaxRoots + 96 <= kWStack - kStackMargin, "full steps on the first roots");
struct TravQ {
  int stk[kWStack];   // index_word(node, slot)
  int lq[kLeafQ];     // index_word(sorted primitive, slot); directly behind the stack
  ChordItem cq[kChordQ];
};
static_assert(offsetof(TravQ, lq) == kWStack * sizeof(int), "queue behind the stack");
// The point evaluation that follows a traversal phase reuses the queues' space.
struct EvalQ {
  float kap[kPK][32], kb[kPK][32];     // kappa and kappa_bar of every slot's points
  unsigned short own[32 * kPK];        // point of the phase -> slot | index << 5
  unsigned short hit[kHits][32];       // per lane: chords that cover its point
};
struct WarpQ {
  LaneRay r[32];
  union {
    TravQ t;  // traversal phase
    EvalQ e;  // point evaluation
  };
};

__device__ __forceinline__ unsigned long long slot_mask(const LaneRay& R) {
  return (unsigned long long)R.mask_lo | ((unsigned long long)R.mask_hi << 32);
}
__device__ __forceinline__ float ray_weight(const LaneRay& R, uint32_t cell) {
  if (!(slot_mask(R) >> cell & 1ull)) return 0.f;
  const int b = cell == 0 ? 0 : (int)((cell - 1u) >> 3) + 1;
  if (b == 0 || (R.cx[0] | R.cx[1]) == 0u) return R.bw[b];
  return R.bw[b] * cone_factor(R.cx, cell, b);
}

__device__ __forceinline__ uint64_t slot_seed(const LaneRay& R) {
  return (uint64_t)R.seed_lo | ((uint64_t)R.seed_hi << 32);
}

// chord of sorted primitive j on the ray of slot R
__device__ __forceinline__ bool slot_chord(const DevField& F, const LaneRay& R, int j, Chord& ch,
                                           float& w) {
  return prim_chord(F, j, make_float3(R.o[0], R.o[1], R.o[2]), make_float3(R.v[0], R.v[1], R.v[2]),
                    0.f, INFINITY, [&](uint32_t c) { return ray_weight(R, c); }, w, ch);
}

// Nodes per lane and traversal step.  Two hide each other's latency where rays visit many
// nodes: with every cone selected, 512x512, 16 samples, 100k kernels take 97.2 ms with
// one and 92.0 with two.  With one-cone masks (100 nodes per ray) a step seldom holds 64
// entries and the longer code costs more: 1M kernels, 1024x1024, 8 samples 193.5 and 212.5 ms.
static int nodes_per_step(const LodDev& a, const LodDev& b) {
  return a.cone_policy == GF_CONE_ALL && b.cone_policy == GF_CONE_ALL && a.freq_policy <= GF_FREQ_CUTOFF &&
                 b.freq_policy <= GF_FREQ_CUTOFF
             ? 2
             : 1;
}

// One draw of a queued chord's walk: the next tentative point of its majorant
// (Sec. 3) from the chord's own Philox stream, recorded for the owner when it
// falls in the window [ta, te).  Returns true when the chord may hold further
// points (c then stands at the point drawn, with the next draw index); false
// when the walk left the chord or the window, or the owner's point buffer is
// full (the owner then halves the window and redoes it).
__device__ __forceinline__ bool walk_step(const DevField& F, WarpQ& Q, ChordItem& c,
                                          const float* env, unsigned long long& npt) {
  LaneRay& R = Q.r[c.orig_own >> 26];
  const uint32_t draw = c.jd >> 3;
  if (draw >= (1u << 16)) {
    set_err(F, ERR_GUARD);
    return false;
  }
  const float invs = 1.0f / c.sa;
  const int J = (int)(c.jd & 7u);
  float dt = c.dt;
  int p = 0;  // the majorant piece holding dt: the pieces ending at or before it
  // (supports up to 3 sigma: without a loop, so that the lanes stay together: 1 % of a
  // 1024x1024 8-sample launch through 1M kernels)
  if (J <= 2) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float bp = q < J ? c.dts - (float)(J - q) * invs : c.dts + (float)(q - J + 1) * invs;
      p += q < 2 * J && bp <= dt && p == q ? 1 : 0;
    }
  } else {
    while (p < 2 * J) {
      const float bp = p < J ? c.dts - (float)(J - p) * invs : c.dts + (float)(p - J + 1) * invs;
      if (bp <= dt) ++p;
      else break;
    }
  }
  const uint4 x = rng4(slot_seed(R), draw, c.orig_own & kOrigMask, R.ray, R.word);
  float z = -__logf(1.0f - u01(x.x));
  bool emit = false;
  for (int q = 0; q < 2 * J + 2; ++q) {
    const float bp = p < J ? c.dts - (float)(J - p) * invs : c.dts + (float)(p - J + 1) * invs;
    const float end = p < 2 * J ? fminf(bp, c.dtout) : c.dtout;
    const int nn = p < J ? J - p : p - J;
    const float lam = c.h * env[nn];
    const float capz = lam * (end - dt);
    if (z < capz) {
      dt += z / lam;
      emit = true;
      break;
    }
    z -= capz;
    dt = end;
    if (dt >= c.dtout) return false;
    ++p;
  }
  if (!emit) return false;
  const float t = c.tc + dt;
  if (t >= R.te) return false;
  if (t >= R.ta) {
    ++npt;
    const int slot = atomicAdd(&R.npts, 1);
    if (slot >= kPK) return false;  // overflow: the owner halves the window and redoes it
    R.pt[slot] = t;
    R.pu[slot] = u01(x.y);
  }
  c.dt = dt;
  c.jd += 8u;
  return true;
}

// One traversal phase for the slots with want = true.  The warp shares one
// stack of (node, slot) entries: every step pops up to 32 entries from the
// frontiers of all its rays, so lanes stay busy while 32 rays are in flight.
// It collects the tentative points of each slot's window and stores the
// window's chords for their evaluation.
template <int kPerStep, class Work>
__device__ void warp_phase(const Work& Wk, WarpQ& Q, bool want, uint32_t lane, const float* env,
                           ChordStore* wch, Counters& cnt) {
  const unsigned lt = (1u << lane) - 1u;
  int sp = 0, lq_n = 0, cq_n = 0;  // warp-uniform sizes
  {
    // the roots of the trees each slot's mask needs, at most 32 kMaxRoots in all
    unsigned long long cm = 0ull;
    unsigned bm = 0u;
    if (want) tree_roots(slot_mask(Q.r[lane]), cm, bm);
    for (;;) {
      const bool has = (cm | bm) != 0ull;
      const unsigned b = __ballot_sync(kFull, has);
      if (b == 0u) break;
      if (has)
        Q.t.stk[sp + __popc(b & lt)] =
            (int)index_word((uint32_t)next_root(Wk.field(Q.r[lane].asset), cm, bm), lane);
      sp += __popc(b);
    }
    __syncwarp();
  }
  const long long max_it = 4 * (Wk.max_n() + 64) + 4096;
  for (long long it = 0;; ++it) {
    if (it > max_it * 32) {
      if (lane == 0) set_err(Wk.err_field(), ERR_GUARD);
      break;
    }
    // ---------------- one traversal step: up to kPerStep (four-wide node, slot) entries
    // per lane
    GF_TIC(t_step);
    int take = min(sp, 32 * kPerStep);
    // near capacity fewer, down to one: a node leaves room for three more entries, and
    // a descent adds at most three per level
    take = min(take, max(1, (kWStack - kStackMargin - sp) / 3));
    uint32_t ent[kPerStep];
#pragma unroll
    for (int u = 0; u < kPerStep; ++u)
      ent[u] = 32 * u + (int)lane < take ? (uint32_t)Q.t.stk[sp - take + 32 * u + (int)lane] : kNoWord;
    __syncwarp();
    sp -= take;
    if (lane == 0) ++cnt.steps;
    int ch[4 * kPerStep];
    unsigned hit = 0u;  // bit k: child k overlaps the window
#pragma unroll
    for (int k = 0; k < 4 * kPerStep; ++k) ch[k] = 0;
#pragma unroll
    for (int u = 0; u < kPerStep; ++u) {
      if (u > 0 && take <= 32 * u) break;  // (the same in every lane)
      if (ent[u] == kNoWord) continue;
      const LaneRay& R = Q.r[word_slot(ent[u])];
      const DevField& F = Wk.field(R.asset);
      if ((int64_t)word_index(ent[u]) >= F.n_nodes4) {
        set_err(Wk.err_field(), ERR_INDEX);  // a node beyond the tree: skipped
        continue;
      }
      const float3 o = make_float3(R.o[0], R.o[1], R.o[2]);
      const float3 inv = make_float3(R.inv[0], R.inv[1], R.inv[2]);
      ++cnt.nodes;
      hit |= node4_hits(F.nodes4 + word_index(ent[u]), o, inv, R.ta, R.te, ch + 4 * u) << (4 * u);
    }
    // ---------------- push internal children, queue leaves
    if (!push_hits(Q.t.stk, kWStack, hit, ch, lane, sp, lq_n,
                   [&](int k, int c) { return (int)index_word((uint32_t)c, word_slot(ent[k >> 2])); }) &&
        lane == 0)
      set_err(Wk.err_field(), ERR_STACK);
    __syncwarp();
    const bool any_trav = sp > 0;
    if (lane == 0) GF_TOC(cnt, 0, t_step);
    // ---------------- leaf rounds: 32 leaves of any slots' rays at a time; once
    // the traversal is over, the last leaves and then the last chords (one
    // walk site, for the instruction cache)
    while (lq_n >= 32 || (!any_trav && (lq_n > 0 || cq_n > 0))) {
      const int tk = lq_n < 32 ? lq_n : 32;
      bool have = (int)lane < tk;
      int j = 0, own = 0;
      if (have) {
        const uint32_t e = (uint32_t)Q.t.lq[lq_n - tk + (int)lane];
        j = (int)word_index(e);
        own = (int)word_slot(e);
        if ((int64_t)j >= Wk.field(Q.r[own].asset).n) {  // a leaf beyond the records
          set_err(Wk.err_field(), ERR_INDEX);
          have = false;
        }
      }
      __syncwarp();
      lq_n -= tk;
      cnt.leaves += have ? 1ull : 0ull;
      GF_TIC(t_leaf);
      bool ok = false;
      ChordItem ci;
      if (have) {
        const LaneRay& R = Q.r[own];
        Chord ch;
        float w;
        if (slot_chord(Wk.field(R.asset), R, j, ch, w)) {
          const float tin = ch.tc + ch.dtin, tout = ch.tc + ch.dtout;
          if (tin < R.te && tout >= R.ta) {
            ok = true;
            const float wa = w * ch.absA;
            const float h = wa * expf(-0.5f * ch.qmin), sa = sqrtf(ch.a);
            // evaluation record for the points of this window
            atomicMax(&Q.r[own].hmax, __float_as_int(h));
            const int k = atomicAdd(&Q.r[own].nch, 1);
            if (k < kSlotCh) {
              // centred on the envelope peak t* = tc + dts: exponent y2 dt^2 + log2 h,
              // phase B dt + delta*, majorant piece floor(|dt| sqrt(a))
              wch->span[own][k] = make_float2(tin, tout);
              float4* dst = wch->rec[own][k];
              dst[0] = make_float4(ch.tc + ch.dts, tin, tout, ch.B);
              dst[1] = make_float4(-0.5f * kLog2e * ch.a, __log2f(h),
                                   reduce_2pi(fmaf(ch.B, ch.dts, ch.delta)), sa);
            }
            ci.tc = ch.tc;
            ci.dt = ch.dtin;
            ci.dtout = ch.dtout;
            ci.h = h;
            ci.sa = sa;
            ci.dts = ch.dts;
            // majorant pieces per side: whitened half-length sa hw rounded up, less one
            int J = (int)ceilf(sa * ch.hw) - 1;
            J = J < 0 ? 0 : (J > 6 ? 6 : J);
            ci.jd = (uint32_t)J;
            ci.orig_own = ch.orig | ((uint32_t)own << 26);
          }
        }
      }
      const unsigned bc = __ballot_sync(kFull, ok);
      if (ok) Q.t.cq[cq_n + __popc(bc & lt)] = ci;
      cq_n += __popc(bc);
      cnt.chords += ok ? 1ull : 0ull;
      __syncwarp();
      if (lane == 0) GF_TOC(cnt, 1, t_leaf);
      GF_TIC(t_walk);
      const bool drain = !any_trav && lq_n == 0;
      while (cq_n >= 32 || (drain && cq_n > 0)) {
        const int tw = cq_n < 32 ? cq_n : 32;
        const bool hv = (int)lane < tw;
        ChordItem cw;
        if (hv) cw = Q.t.cq[cq_n - tw + (int)lane];
        __syncwarp();
        cq_n -= tw;
        // one draw per chord and round; chords that may hold more points go back
        // to the queue, so every round keeps the lanes busy
        const bool again = hv && walk_step(Wk.err_field(), Q, cw, env, cnt.points);
        const unsigned ba = __ballot_sync(kFull, again);
        if (again) Q.t.cq[cq_n + __popc(ba & lt)] = cw;
        cq_n += __popc(ba);
        __syncwarp();
      }
      if (lane == 0) GF_TOC(cnt, 2, t_walk);
    }
    if (!any_trav && lq_n == 0 && cq_n == 0) break;
  }
  __syncwarp();
}

// per-lane path state
struct PathState {
  int rq;         // request of the pixel (0 for a single render)
  int pix;        // -1: no pixel
  int s, b;       // sample, bounce
  int s_end;      // end of the lane's sample range of the pixel
  int kind;       // 0 idle, 1 delta tracking, 2 ratio tracking (NEE)
  long long acc;  // sum of the range's samples in fixed point (2^-32 units)
  float Lsum, thr, T;
  float3 o, v;    // current ray
  float t0, t1;   // scene span of the current ray
  float step;     // window length
  float lim;      // length that holds kFill of a window's chords on average
  unsigned long long allow;  // cells the foveation keeps for the sample's path
};

__device__ __forceinline__ void set_slot(LaneRay& R, float3 o, float3 v, const Mask& m,
                                         uint32_t ray, uint32_t word) {
  R.o[0] = o.x; R.o[1] = o.y; R.o[2] = o.z;
  R.v[0] = v.x; R.v[1] = v.y; R.v[2] = v.z;
  const float3 iv = safe_inv(v);
  R.inv[0] = iv.x; R.inv[1] = iv.y; R.inv[2] = iv.z;
  R.ray = ray;
  R.word = word;
  R.mask_lo = (uint32_t)m.bits;
  R.mask_hi = (uint32_t)(m.bits >> 32);
#pragma unroll
  for (int k = 0; k < 8; ++k) R.bw[k] = m.bw[k];
  R.cx[0] = m.cx[0];
  R.cx[1] = m.cx[1];
}

// chords per unit length that rays with the cell mask `mask` have on average
__device__ __forceinline__ float chords_per_length(const DevField& F, unsigned long long mask) {
  float r = (mask & 1ull) ? F.chords[0] : 0.f;
#pragma unroll
  for (int b = 1; b < 8; ++b)
    r = fmaf(F.chords[b], (float)__popc((unsigned)(mask >> (1 + kCones * (b - 1))) & 0xFFu), r);
  return r;
}

// Start a tracking ray: returns false if it misses the scene (nothing to do).
__device__ __forceinline__ bool start_ray(const DevField& F, LaneRay& R, PathState& S, int kind,
                                          float3 o, float3 v, const Mask& m, uint32_t ray,
                                          uint32_t word) {
  S.kind = kind;
  S.o = o;
  S.v = v;
  set_slot(R, o, v, m, ray, word);
  float t0, t1;
  const bool hit = m.bits != 0ull && scene_span(F, o, safe_inv(v), 0.f, INFINITY, t0, t1);
  S.t0 = t0;
  S.t1 = t1;
  if (!hit) return false;
  S.lim = kFill * (float)kSlotCh / chords_per_length(F, m.bits);
  const Window w = window_first(kind == 1, t0, t1, S.lim);
  R.ta = w.ta;
  R.te = w.te;
  S.step = w.step;
  return true;
}

// kappa and kappa_bar at the points of every slot, from the chords pass 1 stored.
// A lane takes one point of the phase (with few points left, 2, 4, ... 32 lanes share
// one): it runs through the entries and exits of its slot's chords, four per load, and
// notes the chords that cover the point; then it evaluates those, so that the
// evaluations run with the lanes full.  (Adding every covering chord to 64-bit sums in
// shared memory as it was found kept 34 % of the renderer's cycles busy.)
// The sums are exact in 64-bit fixed point: a term is at most the peak h of
// its chord (to ~1e-6), so with H the largest peak of the slot's window and at most
// kSlotCh < 2^9 chords, scaling by 2^(54 - e) (H < 2^e) keeps every partial
// sum below 2^63.  Each term is rounded once (to 2^(e-54), far below FP32
// resolution) and integer addition does not depend on order, so a path's
// decisions do not depend on which other rays shared its warp or on the order
// in which its chords were stored or evaluated.
__device__ __forceinline__ int slot_exp(const LaneRay& R) {
  const int ex = ((R.hmax >> 23) & 0xFF) - 126;  // H < 2^ex
  return ex < -70 ? -70 : ex;
}
__device__ void eval_stored(WarpQ& Q, const ChordStore* wch, const float* env, uint32_t lane,
                            Counters& cnt) {
  EvalQ& E = Q.e;
  int left;  // points of the phase
  {
    const int n = Q.r[lane].npts;  // 0: no points (or an overflowed window)
    int incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(kFull, incl, o);
      if ((int)lane >= o) incl += y;
    }
    left = __shfl_sync(kFull, incl, 31);
    for (int i = 0; i < n; ++i) E.own[incl - n + i] = (unsigned short)(lane | (uint32_t)i << 5);
  }
  __syncwarp();
  for (int q0 = 0; left > 0;) {
    int sh = 0;  // 2^sh lanes per point
    while (sh < 5 && left << (sh + 1) <= 32) ++sh;
    const int pts = min(left, 32 >> sh);
    const bool act = (int)(lane >> sh) < pts;
    const uint32_t own = act ? E.own[q0 + (int)(lane >> sh)] : 0u;
    const int sl = (int)(own & 31u), i = (int)(own >> 5);
    const LaneRay& R = Q.r[sl];
    const float t = R.pt[i];
    const int m = act ? R.nch : 0, ex = slot_exp(R);
    const float S = __int_as_float((127 + 54 - ex) << 23);  // 2^(54 - ex)
    const float2* span = wch->span[sl];
    long long kap = 0, kb = 0;
    int k = 4 * (int)(lane & ((1u << sh) - 1u));
    for (;;) {
      int h = 0;
      for (; k < m && h <= kHits - 4; k += 4 << sh) {
        float4 a, b;
        ld32(span + k, a, b);
        if (t >= a.x && t <= a.y) E.hit[h++][lane] = (unsigned short)k;
        if (t >= a.z && t <= a.w && k + 1 < m) E.hit[h++][lane] = (unsigned short)(k + 1);
        if (t >= b.x && t <= b.y && k + 2 < m) E.hit[h++][lane] = (unsigned short)(k + 2);
        if (t >= b.z && t <= b.w && k + 3 < m) E.hit[h++][lane] = (unsigned short)(k + 3);
      }
      __syncwarp();
      for (int x = 0; x < h; ++x) {
        float4 a, b;
        ld32(wch->rec[sl][E.hit[x][lane]], a, b);
        const float dt = t - a.x;
        kap += __float2ll_rn(ex2f(fmaf(b.x, dt * dt, b.y)) * cosf_fast(fmaf(a.w, dt, b.z)) * S);
        int mm = (int)(fabsf(dt) * b.w);
        mm = mm > 7 ? 7 : mm;
        kb += __float2ll_rn(ex2f(b.y + env[8 + mm]) * S);  // h exp(-m^2/2)
      }
      cnt.evals += (unsigned)h;
      if (!__any_sync(kFull, k < m)) break;
    }
    for (int o = 1; o < 1 << sh; o <<= 1) {
      kap += __shfl_xor_sync(kFull, kap, o);
      kb += __shfl_xor_sync(kFull, kb, o);
    }
    if (act && (lane & ((1u << sh) - 1u)) == 0u) {
      const float u = __int_as_float((127 - 54 + ex) << 23);
      E.kap[i][sl] = __ll2float_rn(kap) * u;
      E.kb[i][sl] = __ll2float_rn(kb) * u;
    }
    q0 += pts;
    left -= pts;
    __syncwarp();
  }
}
// kappa (k = 0) or kappa_bar (k = 1) at point i of the calling lane's slot, as
// eval_stored left them
__device__ __forceinline__ float slot_sum(const WarpQ& Q, uint32_t lane, int i, int k) {
  return k ? Q.e.kb[i][lane] : Q.e.kap[i][lane];
}

// ---------------------------------------------------------------------------
// Work sources.  A lane takes pixels one at a time; a pixel belongs to a
// request (its camera, LoD descriptors, seed and framebuffer) and a request to
// a field.  A single render is one request on one field; the render server
// hands the kernel a batch of items from many requests on several fields.
// ---------------------------------------------------------------------------
// Radiance samples are summed in 64-bit fixed point (2^-32 units): a pixel's
// value then does not depend on how its samples were split between lanes or
// in which order the partial sums arrived.
constexpr float kFixScale = 4294967296.0f;  // 2^32
__device__ __forceinline__ long long fix_sample(float L) { return __float2ll_rn(L * kFixScale); }
__device__ __forceinline__ float fix_mean(long long sum, int spp) {
  return __ll2float_rn(sum) * (1.0f / kFixScale) / (float)spp;
}

// A single render: units of `chunk` consecutive samples of one pixel, so the
// lanes stay busy to the end of the launch; partial sums meet in acc64.
struct ImageWork {
  const DevField* F;
  const PathParams* P;
  unsigned long long* acc64;
  int* counter;
  int npix, chunk, nchunk;
  __device__ const DevField& field(int) const { return *F; }
  __device__ const DevField& err_field() const { return *F; }
  __device__ int64_t max_n() const { return F->n; }
  __device__ const PathParams& params(int) const { return *P; }
  __device__ int asset(int) const { return 0; }
  __device__ bool next(int& rq, int& pix, int& s0, int& s1) const {
    const int u = atomicAdd(counter, 1);
    rq = 0;
    if (u >= npix * nchunk) return false;
    pix = u / nchunk;
    s0 = P->s0 + (u - pix * nchunk) * chunk;
    s1 = min(s0 + chunk, P->s0 + P->spp);
    return true;
  }
  __device__ void finish(int, int pix, long long acc) const {
    atomicAdd(acc64 + pix, (unsigned long long)acc);
  }
};

struct ServerWork {
  const ServerLaunch* L;
  __device__ const DevField& field(int a) const { return L->fields[a]; }
  __device__ const DevField& err_field() const { return L->fields[0]; }
  __device__ int64_t max_n() const { return L->max_n; }
  __device__ const PathParams& params(int rq) const { return L->reqs[rq].P; }
  __device__ int asset(int rq) const { return L->reqs[rq].asset; }
  // the batch's units (chunk consecutive samples of one pixel) are numbered
  // 0..total-1 item after item; a lane takes the next number and finds its
  // item by binary search over the item bases
  __device__ bool next(int& rq, int& pix, int& s0, int& s1) const {
    const int f = atomicAdd(L->counter, 1);
    if (f >= L->total) return false;
    int lo = 0, hi = L->n_items - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (L->items[mid].base <= f) lo = mid;
      else hi = mid - 1;
    }
    const ServerItem it = L->items[lo];
    rq = it.req;
    const ServerReqDev& R = L->reqs[rq];
    const int u = f - it.base, q = u / R.nchunk;
    pix = it.pix0 + q;
    s0 = R.P.s0 + (u - q * R.nchunk) * R.chunk;
    s1 = min(s0 + R.chunk, R.P.s0 + R.P.spp);
    return true;
  }
  // partial sums of a pixel's samples meet in the request's fixed-point sums
  __device__ void finish(int rq, int pix, long long acc) const {
    atomicAdd(L->reqs[rq].acc + pix, (unsigned long long)acc);
  }
};

// The paths of one warp: each lane runs its pixels' samples in order (camera
// ray -> delta tracking -> NEE by ratio tracking -> isotropic scattering), the
// tracking windows of all 32 lanes advancing together through warp_phase.
// Only the first `slots` lanes of a warp take paths: a launch with less work than lanes
// spreads it over every warp of the grid (scatter_slots).
template <int kPerStep, class Work>
__device__ __forceinline__ void render_paths(const Work& Wk, const float* env, WarpQ& Q,
                                             ChordStore* wch, int slots) {
  const uint32_t lane = threadIdx.x & 31u;
  LaneRay& R = Q.r[lane];
  Counters cnt;
  const float inv4pi = 0.25f / 3.14159265358979f;

  PathState S;
  S.rq = 0;
  S.pix = -1;
  S.kind = 0;
  S.acc = 0;
  S.allow = ~0ull;

  // Move the lane's path on from its finished ray (hit: a collision at th on a
  // tracking ray; kind 0: the lane has no path yet) until a new ray starts or
  // no work is left: collision -> NEE, NEE -> isotropic scattering, escape or
  // the last bounce -> the next sample (or pixel).  Every kind of ray is
  // started from one site, which keeps the loop small for the instruction cache.
  auto advance = [&](bool hit, float th) {
    for (int guard = 0; guard < (1 << 20); ++guard) {
      int kind = 0;  // the ray to start: 1 tracking (camera or bounce), 2 NEE
      float3 ro = S.o, rv = S.v;
      bool nee = false;
      if (S.kind == 1 && hit) {
        // collision: next-event estimation towards the light
        const PathParams& P = Wk.params(S.rq);
        ro = make_float3(S.o.x + th * S.v.x, S.o.y + th * S.v.y, S.o.z + th * S.v.z);
        rv = P.light;
        S.thr *= P.albedo;
        S.T = 1.f;
        kind = 2;
        nee = true;
      } else if (S.kind == 2) {
        // NEE finished with transmittance S.T: add it, then scatter isotropically
        const PathParams& P = Wk.params(S.rq);
        S.Lsum += S.thr * P.irradiance * S.T * inv4pi;
        const uint4 y = rng4(P.seed, 0, kNoPrim, (uint32_t)S.pix,
                             stream_word((uint32_t)S.s, (uint32_t)S.b, TAG_SCATTER));
        const float z = 1.0f - 2.0f * u01(y.x);
        const float rr = sqrtf(fmaxf(0.0f, 1.0f - z * z));
        float sn, cs;
        sincosf(2.0f * 3.14159265358979f * u01(y.y), &sn, &cs);
        S.b += 1;
        if (S.b < P.max_bounces) {
          rv = make_float3(rr * cs, rr * sn, z);
          kind = 1;
        }
      }
      if (kind == 0) {
        // the sample is over (escape or last bounce): the next sample, or pixel
        if (S.kind != 0) {
          S.acc += fix_sample(S.Lsum);
          S.s += 1;
        }
        for (;;) {
          if (S.pix < 0) {
            int rq = 0, pix = -1, s0 = 0, s1 = 0;
            if (!Wk.next(rq, pix, s0, s1)) {
              S.pix = -1;
              S.kind = 0;
              return;
            }
            const PathParams& P = Wk.params(rq);
            S.rq = rq;
            S.pix = pix;
            S.s = s0;
            S.s_end = s1;
            S.acc = 0;
            R.asset = Wk.asset(rq);
            R.seed_lo = (uint32_t)P.seed;
            R.seed_hi = (uint32_t)(P.seed >> 32);
          }
          if (S.s < S.s_end) break;
          Wk.finish(S.rq, S.pix, S.acc);
          S.pix = -1;
        }
        const PathParams& P = Wk.params(S.rq);
        camera_ray(P.cam, P.seed, S.pix % P.cam.W, S.pix / P.cam.W, S.s, ro, rv);
        S.b = 0;
        S.thr = 1.f;
        S.Lsum = 0.f;
        S.allow = fov_cells(Wk.field(R.asset), P, rv, (uint32_t)S.pix, (uint32_t)S.s);
        kind = 1;
      }
      const PathParams& P = Wk.params(S.rq);
      const DevField& F = Wk.field(R.asset);
      Mask m = sample_mask(F, nee ? P.lod_nee : P.lod, rv, P.seed, (uint32_t)S.pix, (uint32_t)S.s,
                           (uint32_t)S.b, nee ? TAG_NEE_MASK : TAG_MASK);
      m.bits &= S.allow;
      cnt.rays += 1;
      if (start_ray(F, R, S, kind, ro, rv, m, (uint32_t)S.pix,
                    stream_word((uint32_t)S.s, (uint32_t)S.b, nee ? TAG_NEE : TAG_TRACK)))
        return;
      // the ray misses every primitive: it is over at once (no collision; T = 1 for NEE)
      hit = false;
    }
    set_err(Wk.err_field(), ERR_GUARD);
    S.kind = 0;
  };

  // the first pass takes each lane's first work; every later pass is one window
  bool first = true;
  for (int guard = 0; guard < (1 << 30); ++guard) {
    bool fin = first && (int)lane < slots, fhit = false;
    float fth = 0.f;
    const bool want = S.kind != 0;
    if (!first && !__any_sync(kFull, want)) break;
    if (!first) {
      // ---- pass 1: tentative points of the window
      R.npts = 0;
      R.nch = 0;
      R.hmax = 0;
      __syncwarp();
      warp_phase<kPerStep>(Wk, Q, want, lane, env, wch, cnt);
      // owner: a window whose points overflowed the slots is halved and redone;
      // otherwise its points are sorted by t for the decisions
      int n = 0;
      bool ovf = false;
      if (want) {
        ovf = R.npts > kPK || R.nch > kSlotCh;
        n = ovf ? 0 : R.npts;
        for (int k = 1; k < n; ++k) {
          const float t = R.pt[k], u = R.pu[k];
          int q = k;
          while (q > 0 && R.pt[q - 1] > t) {
            R.pt[q] = R.pt[q - 1];
            R.pu[q] = R.pu[q - 1];
            --q;
          }
          R.pt[q] = t;
          R.pu[q] = u;
        }
        R.npts = n;
      }
      cnt.windows += want ? 1ull : 0ull;
      __syncwarp();
      // ---- kappa and kappa_bar at the points, from the stored chords
      GF_TIC(t_eval);
      if (__any_sync(kFull, want && n > 0)) eval_stored(Q, wch, env, lane, cnt);
      if (lane == 0) GF_TOC(cnt, 3, t_eval);
      // ---- decisions: the window either continues the ray or finishes it
      GF_TIC(t_dec);
      if (want) {
        const bool last = R.te >= S.t1;
        Window w{R.ta, R.te, S.step};
        if (ovf) {
          if (!window_halve(w)) {
            // more points or chords at one t than a window holds: give up on this ray
            set_err(Wk.err_field(), ERR_POINTS);
            fin = true;
          }
        } else {
          if (S.kind == 1) {
            for (int i = 0; i < n && !fhit; ++i) {
              if (R.pu[i] * slot_sum(Q, lane, i, 1) < fmaxf(slot_sum(Q, lane, i, 0), 0.f)) {
                fhit = true;
                fth = R.pt[i];
              }
            }
          } else {
            for (int i = 0; i < n; ++i) {
              const float kb = slot_sum(Q, lane, i, 1);
              if (kb > 0.f) S.T *= 1.f - fmaxf(slot_sum(Q, lane, i, 0), 0.f) / kb;
            }
          }
          fin = fhit || last;
          if (!fin) window_next(w, S.kind == 1, S.lim, S.t1);
        }
        R.ta = w.ta;
        R.te = w.te;
        S.step = w.step;
      }
      if (lane == 0) GF_TOC(cnt, 4, t_dec);
    }
    first = false;
    if (fin) advance(fhit, fth);
    __syncwarp();
  }
  if (S.kind != 0) set_err(Wk.err_field(), ERR_GUARD);  // paths left over
  flush_counters(Wk.err_field(), cnt, lane);
}

__device__ __forceinline__ WarpQ& setup_block(unsigned char* smraw, const float* env_src) {
  // env[0..7] = exp(-n^2/2), env[8..15] = its log2 (-n^2 log2(e) / 2)
  float* env = reinterpret_cast<float*>(smraw);
  WarpQ* Qs = reinterpret_cast<WarpQ*>(smraw + 64);
  if (threadIdx.x < 8) {
    env[threadIdx.x] = env_src[threadIdx.x];
    env[8 + threadIdx.x] = -0.5f * kLog2e * (float)(threadIdx.x * threadIdx.x);
  }
  __syncthreads();
  return Qs[threadIdx.x >> 5];
}

__device__ __forceinline__ ChordStore* warp_store(float4* chord_store) {
  return reinterpret_cast<ChordStore*>(chord_store) + (size_t)blockIdx.x * kWWarps + (threadIdx.x >> 5);
}

template <int kPerStep>
__global__ void __launch_bounds__(kWWarps * 32, kBlocksPerSM)
    k_render_scatter(const __grid_constant__ DevField F, const __grid_constant__ PathParams P,
                     unsigned long long* acc64, int* counter, int chunk, int slots,
                     float4* chord_store) {
  extern __shared__ __align__(16) unsigned char smraw[];
  WarpQ& Q = setup_block(smraw, F.env);
  const ImageWork Wk{&F, &P, acc64, counter, P.cam.W * P.cam.H, chunk, (P.spp + chunk - 1) / chunk};
  render_paths<kPerStep>(Wk, reinterpret_cast<const float*>(smraw), Q, warp_store(chord_store), slots);
}

__global__ void k_fix_to_image(const unsigned long long* acc64, int64_t npix, int spp, float* out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < npix) out[i] = fix_mean((long long)acc64[i], spp);
}

template <int kPerStep>
__global__ void __launch_bounds__(kWWarps * 32, kBlocksPerSM)
    k_render_server(const __grid_constant__ ServerLaunch L, int slots, float4* chord_store) {
  extern __shared__ __align__(16) unsigned char smraw[];
  WarpQ& Q = setup_block(smraw, L.fields[0].env);
  const ServerWork Wk{&L};
  render_paths<kPerStep>(Wk, reinterpret_cast<const float*>(smraw), Q, warp_store(chord_store), slots);
}

size_t scatter_smem_bytes() { return 64 + sizeof(WarpQ) * kWWarps; }
// 228 KB of shared memory per SM, 1 KB of it reserved per resident block
static_assert((64 + sizeof(WarpQ) * kWWarps + 1024) * kBlocksPerSM <= 233472,
              "kBlocksPerSM blocks fit one SM's shared memory");

size_t scatter_store_bytes(int64_t grid) {
  return (size_t)grid * kWWarps * sizeof(ChordStore);
}

// full persistent grid of the scattering kernels
template <class K>
static cudaError_t scatter_grid(K kernel, int sm_count, int64_t& g) {
  const size_t smem = scatter_smem_bytes();
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kWWarps * 32, smem) != cudaSuccess)
    (void)cudaGetLastError();
  if (per_sm < 1) per_sm = 1;
  g = (int64_t)sm_count * per_sm;
  return cudaSuccess;
}

// the grid that both variants of a kernel fit
static cudaError_t render_grid(int sm_count, int64_t& g) {
  int64_t h = 1;
  cudaError_t e = scatter_grid(k_render_scatter<1>, sm_count, g);
  if (e == cudaSuccess) e = scatter_grid(k_render_scatter<2>, sm_count, h);
  g = std::min(g, h);
  return e;
}

// Paths per warp for `units` units of work, and the grid that holds them (g: the full
// grid on entry).  With fewer units than lanes every warp of the grid takes its share
// instead of a few warps taking 32 paths each: a warp works through its paths' windows
// together, so its time grows with their number.  120x67 pixels at 1 sample through 50k
// kernels: 696 us with 251 full warps, 215 us with 2,010 warps of 4 paths; 96x64
// 3-bounce paths through 200k kernels: 9.6 and 1.8 ms.
static int scatter_slots(int64_t units, int64_t& g) {
  const int64_t warps = g * kWWarps;
  const int64_t slots = std::min<int64_t>(32, std::max<int64_t>(1, (units + warps - 1) / warps));
  const int64_t need = (units + slots * kWWarps - 1) / (slots * kWWarps);
  g = std::max<int64_t>(1, std::min(g, need));
  return (int)slots;
}

// pixel sums (8 bytes per pixel) and the per-warp chord store of a full persistent
// grid of g blocks (shared with the analytic flights' lists), grown through the field's
// allocator; g comes back smaller when less memory is to be had
static cudaError_t render_scratch(const Field& F, int64_t npix, int64_t& g, cudaStream_t s) {
  cudaError_t e = render_grid(F.ctx.sm_count, g);
  if (e != cudaSuccess) return e;
  if ((e = grow(F, (void**)&F.acc64, F.acc_bytes, (size_t)npix * 8, s)) != cudaSuccess) return e;
  const size_t share = std::max(scatter_store_bytes(1), (flight_store_bytes(F) + g - 1) / g);
  return grow_shares(F, F.wscratch, share, g, s);
}
cudaError_t ensure_render_scratch(const Field& F, int64_t npix, cudaStream_t s) {
  int64_t g = 1;
  return render_scratch(F, npix, g, s);
}

cudaError_t launch_render_scatter(const Field& F, const PathParams& P, float* out, cudaStream_t s) {
  (void)cudaGetLastError();  // a stale error of an unrelated call is not ours
  cudaError_t e = cudaMemsetAsync(F.counter, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  const int64_t npix = (int64_t)P.cam.W * P.cam.H;
  int64_t g = 1;
  // fixed-point pixel sums and the chord store (allocated ahead by gf_reserve, else here)
  if ((e = render_scratch(F, npix, g, s)) != cudaSuccess) return e;
  // about 16 units per lane: chunk = ceil(npix spp / (16 lanes)), in [1, spp]
  const int64_t lanes = g * kWWarps * 32;
  int64_t chunk = (npix * P.spp + 16 * lanes - 1) / (16 * lanes);
  chunk = chunk < 1 ? 1 : (chunk > P.spp ? P.spp : chunk);
  const int64_t nchunk = (P.spp + chunk - 1) / chunk;
  if (npix * nchunk >= (int64_t)INT_MAX) return cudaErrorInvalidValue;
  if ((e = cudaMemsetAsync(F.acc64, 0, (size_t)npix * 8, s)) != cudaSuccess) return e;
  const int slots = scatter_slots(npix * nchunk, g);
  auto kernel = nodes_per_step(P.lod, P.lod_nee) == 2 ? k_render_scatter<2> : k_render_scatter<1>;
  kernel<<<(unsigned)g, kWWarps * 32, scatter_smem_bytes(), s>>>(F.dev, P, F.acc64, F.counter, (int)chunk,
                                                                 slots, static_cast<float4*>(F.wscratch.p));
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_fix_to_image<<<(unsigned)((npix + 255) / 256), 256, 0, s>>>(F.acc64, npix, P.spp, out);
  return cudaGetLastError();
}

cudaError_t server_grid(int sm_count, int64_t& g) {
  (void)cudaGetLastError();
  int64_t h = 1;
  cudaError_t e = scatter_grid(k_render_server<1>, sm_count, g);
  if (e == cudaSuccess) e = scatter_grid(k_render_server<2>, sm_count, h);
  g = std::min(g, h);
  return e;
}

cudaError_t launch_fix_to_image(const unsigned long long* acc, int64_t npix, int spp, float* out,
                                cudaStream_t s) {
  k_fix_to_image<<<(unsigned)((npix + 255) / 256), 256, 0, s>>>(acc, npix, spp, out);
  return cudaGetLastError();
}

cudaError_t launch_render_server(const ServerLaunch& L, const ServerReqDev* reqs, int64_t grid,
                                 float4* chord_store, cudaStream_t s) {
  (void)cudaGetLastError();
  const int slots = scatter_slots(L.total, grid);
  // two nodes per step when every request of the batch gains by it
  bool two = true;
  for (int i = 0; i < L.n_items; ++i) two = two && nodes_per_step(reqs[i].P.lod, reqs[i].P.lod_nee) == 2;
  auto kernel = two ? k_render_server<2> : k_render_server<1>;
  kernel<<<(unsigned)grid, kWWarps * 32, scatter_smem_bytes(), s>>>(L, slots, chord_store);
  return cudaGetLastError();
}

}  // namespace gf
