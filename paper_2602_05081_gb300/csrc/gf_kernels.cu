// gf_kernels.cu -- render, transmittance and test kernels of the Gabor-field
// renderer.  Persistent warps pull work from a global counter: one ray per warp
// (gf_coop.cuh), or one per lane through a few kernels.
#include <cuda_runtime.h>

#include <algorithm>

#include "gf_coop.cuh"
#include "gf_host.h"
#include "gf_trace.cuh"

namespace gf {

constexpr int kBlock = 128;
constexpr int kCoopBlocks = 5;  // resident blocks per SM of the one-ray-per-warp kernels

struct Ray {
  float3 o, v;
  float tmin, tmax;
};
__device__ __forceinline__ Ray batch_ray(const TrParams& P, int64_t r) {
  return Ray{make_float3(P.o[3 * r], P.o[3 * r + 1], P.o[3 * r + 2]),
             unit_dir(make_float3(P.d[3 * r], P.d[3 * r + 1], P.d[3 * r + 2])),
             P.trange ? P.trange[2 * r] : 0.f, P.trange ? P.trange[2 * r + 1] : INFINITY};
}
// The next ray of a batch for the warp, after ray r (-1: the first); P.n or more at the end.
// A small batch is dealt out (no counter to clear, no atomic per ray); of larger ones, rays
// that miss the scene are answered by one lane.
__device__ __forceinline__ int64_t next_ray(const DevField& F, const TrParams& P, WarpItems& S, uint32_t lane,
                                            int spp, int64_t r) {
  if (P.dealt)
    return r < 0 ? (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)
                 : r + (int64_t)gridDim.x * (blockDim.x >> 5);
  return (int64_t)next_item(S, P.counter, (uint32_t)P.n, lane, [&](uint32_t i) {
    const Ray y = batch_ray(P, i);
    if (meets_scene(F, y.o, y.v, y.tmin, y.tmax)) return -1;
    P.out_T[i] = 1.f;
    if (P.out_tau) P.out_tau[i] = 0.f;
    return spp;
  });
}

// ---------------------------------------------------------------------------
// Optical depth of a batch of rays (Gauss-Legendre quadrature or closed-form
// chord integrals), one ray per warp (coop_tau) at every batch size but for fields of
// a few kernels (lane_work).  Bound by instruction issue.  With one ray per lane the
// lanes part at every leaf: each runs its own tree walk and its own rule of 8 to 64
// nodes.  130,001 rays through 100k kernels (306 chords and 4,092 nodes per ray):
// 65.0 ms with one ray per lane, 3.8 ms with one per warp; 4,096 rays through 256
// kernels: 53.6 us over a binary tree, 19.4 us now.
// ---------------------------------------------------------------------------
template <int MODE>  // GF_TR_DETERMINISTIC or GF_TR_CLOSED_FORM
__global__ void __launch_bounds__(kBlock, kCoopBlocks)
    k_transmittance_coop(const __grid_constant__ DevField F, const __grid_constant__ TrParams P) {
  __shared__ BlockTables sm;
  __shared__ CoopQ qs[kBlock / 32];
  init_tables(sm, F);
  const uint32_t lane = threadIdx.x & 31u;
  __shared__ WarpItems items[kBlock / 32];
  CoopQ& Q = qs[threadIdx.x >> 5];
  init_items(items[threadIdx.x >> 5], lane);
  Counters cnt;
  const int spp = lod_is_deterministic(P.lod) ? 1 : P.spp;
  WarpItems& S = items[threadIdx.x >> 5];
  for (int64_t r = next_ray(F, P, S, lane, spp, -1); r < P.n; r = next_ray(F, P, S, lane, spp, r)) {
    const Ray y = batch_ray(P, r);
    float s_acc = 0.f, c_acc = 0.f;
    for (int s = 0; s < spp; ++s) {
      const Mask m = sample_mask(F, P.lod, y.v, P.seed, (uint32_t)r, (uint32_t)s, 0, TAG_MASK);
      if (lane == 0) cnt.rays += 1;
      coop_tau<MODE>(F, Q, m, y.o, y.v, y.tmin, y.tmax, sm.glx, sm.glw, lane, s_acc, c_acc, cnt);
    }
    warp_sum_pair(s_acc, c_acc);
    if (lane == 0) {
      const float tau = __fadd_rn(s_acc, c_acc) / (float)spp;
      P.out_T[r] = expf(-tau);
      if (P.out_tau) P.out_tau[r] = tau;
    }
  }
  if (lane == 0) cnt.rays += S.missed;
  flush_counters(F, cnt, lane);
}

// ---------------------------------------------------------------------------
// Ratio tracking, one ray per warp, over a window of t, at first all of the ray.  The
// warp traverses the trees together; each round's chords (one per lane) store their
// evaluation records in shared memory and draw their tentative points in the window
// (chord_points: the per-chord streams of the per-thread tracker, so the same points).
// The points are put in t order; then 1, 2, ... 32 lanes per point sum kappa and
// kappa_bar over the window's chords and multiply the factors 1 - kappa / kappa_bar;
// the lanes' products are combined in a fixed butterfly order.  A window with more chords
// than the buffer holds is traversed once more, its chords added to the points' sums a
// buffer at a time; one with more points is halved.  Bound by instruction issue and the
// latency of tree nodes.  30,000 rays through 100k kernels: 38 ms with one ray per lane
// (the per-thread tracker traverses twice per eight points, its lanes parted), 1.9 ms now;
// 4,096 rays through 256 kernels: 24.7 us (rays dealt out).  With 445 kernels over a point
// (14k in all), 130,000 rays: 135 ms with one ray per lane, 742 when windows were halved
// for their chords and the rest left to one lane, 22 now.
//
// Terms come in two forms.  Rays of a small batch that fit one window take records
// centred on the envelope's peak; large batches and other rays take the
// per-thread tracker's own form (`exact`), which differs by up to 2e-4 of T where
// carriers of ~1e3 rad run over a chord (fast cosine of an unreduced phase).  In that
// form the ray's points go in runs of kPts, and a point at the t at which a run ended is
// left out, as in track().  Left to the per-thread tracker (one lane): a window that
// cannot be halved.
// ---------------------------------------------------------------------------
constexpr int kRtRec = 512;    // float4s of chord records of a window in shared memory
constexpr int kRtPts = 128;    // tentative points of a window
struct RtQ {
  CoopTrav t;
  // centred, 2 per chord: (t*, t_in, t_out, B), (-a log2(e) / 2, log2 h, phase at t*,
  // sqrt(a)); exact, 3 per chord: (tc, t_in, t_out, B), exponent's y2, y1, y0 and the phase
  // at tc, (h, t* - tc, sqrt(a), -)
  float4 rec[kRtRec];
  float raw[kRtPts], pt[kRtPts];  // points as drawn (then kappa, with many chords), in t order
  float kb[kRtPts];               // kappa_bar, with many chords
  int npts;
};

// The factors of the sorted points from the stored chords: the lane's share of their
// product; or (add) their sums added to raw and kb.
__device__ __forceinline__ float rt_points(RtQ& Q, int npts, int nch, bool exact, bool add, const float* env,
                                           uint32_t lane, Counters& cnt) {
  float prod = 1.f;
  for (int q0 = 0; q0 < npts;) {
    const int left = npts - q0;
    int sh = 0;  // 2^sh lanes per point
    while (sh < 5 && left << (sh + 1) <= 32) ++sh;
    const int pts = min(left, 32 >> sh), sub = (int)(lane & ((1u << sh) - 1u));
    const bool act = (int)(lane >> sh) < pts;
    const int i = q0 + (int)(lane >> sh);
    const float t = act ? Q.pt[i] : 0.f;
    float kap = 0.f, kb = 0.f;
    for (int c = act ? sub : nch; c < nch; c += 1 << sh) {
      const float4 a = Q.rec[exact ? 3 * c : 2 * c];
      if (!(t >= a.y && t <= a.z)) continue;
      const float dt = t - a.x;
      ++cnt.evals;
      if (exact) {
        const float4 b = Q.rec[3 * c + 1], d = Q.rec[3 * c + 2];
        kap = fmaf(ex2f(fmaf(fmaf(b.x, dt, b.y), dt, b.z)), cosf_fast(fmaf(a.w, dt, b.w)), kap);
        int mm = (int)(fabsf(dt - d.y) * d.z);
        mm = mm > 7 ? 7 : mm;
        kb = fmaf(d.x, env[mm], kb);
      } else {
        const float4 b = Q.rec[2 * c + 1];
        kap = fmaf(ex2f(fmaf(b.x, dt * dt, b.y)), cosf_fast(fmaf(a.w, dt, b.z)), kap);
        int mm = (int)(fabsf(dt) * b.w);
        mm = mm > 7 ? 7 : mm;
        kb = fmaf(ex2f(b.y), env[mm], kb);  // h exp(-m^2/2)
      }
    }
    __syncwarp();
    for (int o2 = 1; o2 < 1 << sh; o2 <<= 1) {
      kap += __shfl_xor_sync(kFull, kap, o2);
      kb += __shfl_xor_sync(kFull, kb, o2);
    }
    if (act && sub == 0) {
      if (add) {
        Q.raw[i] += kap;
        Q.kb[i] += kb;
      } else if (kb > 0.f) {
        prod *= 1.f - kap / kb;
      }
    }
    q0 += pts;
  }
  return prod;
}

// Chords and points of the window [ta, tb), or [ta, t1] when last; returns the chords (those
// beyond the buffer are counted, and draw their points).  With many >= 0 sorted points
// known: their sums instead, the buffer added to them whenever it is nearly full; returns the
// chords left in it.
__device__ __forceinline__ int rt_gather(const DevField& F, RtQ& Q, const Mask& M, float3 o, float3 v,
                                         float3 inv, float tmin, float tmax, float ta, float tb,
                                         bool last, uint64_t seed, uint32_t ray, uint32_t word,
                                         const float* env, uint32_t lane, bool exact, int many, Counters& cnt) {
  const unsigned lt = (1u << lane) - 1u;
  const int cap = exact ? kRtRec / 3 : kRtRec / 2;
  int nch = 0;
  __syncwarp();
  if (lane == 0) Q.npts = 0;
  coop_traverse(F, Q.t, M.bits, o, inv, ta, tb, lane, cnt, [&](int j) {
    Chord ch;
    float w;
    const bool ok = j >= 0 &&
                    prim_chord(F, j, o, v, tmin, tmax,
                               [&](uint32_t cl) { return mask_weight(M, cl); }, w, ch) &&
                    ch.tc + ch.dtin <= tb && ch.tc + ch.dtout >= ta;
    const unsigned bc = __ballot_sync(kFull, ok);
    const int k = nch + __popc(bc & lt);
    if (ok) {
      const float wa = w * ch.absA, h = wa * expf(-0.5f * ch.qmin);
      ++cnt.chords;
      if (k >= cap) {
      } else if (exact) {
        Q.rec[3 * k] = make_float4(ch.tc, ch.tc + ch.dtin, ch.tc + ch.dtout, ch.B);
        Q.rec[3 * k + 1] = make_float4(-0.5f * kLog2e * ch.a, -kLog2e * ch.b,
                                       fmaf(-0.5f * kLog2e, ch.g, log2f(wa)), ch.delta);
        Q.rec[3 * k + 2] = make_float4(h, ch.dts, sqrtf(ch.a), 0.f);
      } else {
        Q.rec[2 * k] = make_float4(ch.tc + ch.dts, ch.tc + ch.dtin, ch.tc + ch.dtout, ch.B);
        Q.rec[2 * k + 1] = make_float4(-0.5f * kLog2e * ch.a, __log2f(h),
                                       reduce_2pi(fmaf(ch.B, ch.dts, ch.delta)), sqrtf(ch.a));
      }
      if (many < 0)
        chord_points(F, ch, h, seed, ray, word, env, [&](float t, float) {
          if (last ? t > tb : t >= tb) return false;
          if (t >= ta) {
            const int q = atomicAdd(&Q.npts, 1);
            if (q >= kRtPts) return false;  // too many: the window is halved
            Q.raw[q] = t;
          }
          return true;
        });
    }
    nch += __popc(bc);
    if (many >= 0 && nch > cap - 32) {
      __syncwarp();
      (void)rt_points(Q, many, nch, true, true, env, lane, cnt);
      nch = 0;
    }
  });
  __syncwarp();
  return nch;
}

__device__ float rt_coop(const DevField& F, RtQ& Q, const Mask& M, float3 o, float3 v, float3 inv,
                         float tmin, float tmax, float t0, float t1, uint64_t seed, uint32_t ray,
                         uint32_t word, const float* env, uint32_t lane, bool exact, Counters& cnt) {
  float prod = 1.f, ta = t0, tb = t1;
  int c8 = 0;           // points since the last multiple of kPts on the ray
  int many = -1;        // points of a window whose chords exceed the buffer
  bool alone = false;   // to the per-thread tracker
  while (!alone) {
    const bool last = tb >= t1;
    const int nch =
        rt_gather(F, Q, M, o, v, inv, tmin, tmax, ta, tb, last, seed, ray, word, env, lane, exact,
                  many, cnt);
    const float w = tb - ta;
    int npts = many;
    if (many < 0) {
      npts = Q.npts;
      __syncwarp();
      if (npts > kRtPts) {
        if (w > 1e-6f * (1.0f + fabsf(ta))) tb = ta + 0.5f * w;
        else alone = true;
        exact = true;
        continue;
      }
      const bool over = nch > (exact ? kRtRec / 3 : kRtRec / 2);
      exact = exact || over;
      // t order (so that the product does not depend on which lane drew first)
      bool tie = false;
      for (int i = (int)lane; i < npts; i += 32) {
        const float t = Q.raw[i];
        int rank = 0;
        for (int k = 0; k < npts; ++k) {
          const float x = Q.raw[k];
          rank += x < t || (x == t && k < i) ? 1 : 0;
          tie = tie || (x == t && k != i);
        }
        Q.pt[rank] = t;
      }
      tie = __any_sync(kFull, exact && tie);
      __syncwarp();
      if (tie) {  // leave out points at the end of a run (every lane writes the same)
        int m = 0;
        float end = -INFINITY;
        for (int i = 0; i < npts; ++i) {
          const float t = Q.pt[i];
          __syncwarp();
          if (t == end) continue;
          Q.pt[m++] = t;
          if (++c8 == kPts) {
            c8 = 0;
            end = t;
          }
        }
        npts = m;
        __syncwarp();
      } else {
        c8 = (c8 + npts) % kPts;
      }
      if (lane == 0) cnt.points += (unsigned long long)npts;
      if (over) {
        for (int i = (int)lane; i < npts; i += 32) Q.raw[i] = Q.kb[i] = 0.f;
        many = npts;
        continue;  // the window again, for the sums
      }
    }
    prod *= rt_points(Q, npts, nch, exact, many >= 0, env, lane, cnt);
    if (many >= 0) {
      __syncwarp();
      for (int i = (int)lane; i < npts; i += 32)
        if (Q.kb[i] > 0.f) prod *= 1.f - Q.raw[i] / Q.kb[i];
      many = -1;
    }
    if (last) break;
    ta = tb;
    tb = fminf(t1, ta + 2.0f * w);
  }
  if (alone) {
    float T = 1.f;
    if (lane == 0) T = track(F, M, o, v, tmin, tmax, seed, ray, word, env, cnt);
    __syncwarp();
    return __shfl_sync(kFull, T, 0);
  }
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) prod *= __shfl_xor_sync(kFull, prod, off);
  return prod;
}

__global__ void __launch_bounds__(kBlock, 4)
    k_transmittance_rt_coop(const __grid_constant__ DevField F, const __grid_constant__ TrParams P) {
  __shared__ BlockTables sm;
  __shared__ RtQ qs[kBlock / 32];
  init_tables(sm, F);
  const uint32_t lane = threadIdx.x & 31u;
  __shared__ WarpItems items[kBlock / 32];
  RtQ& Q = qs[threadIdx.x >> 5];
  init_items(items[threadIdx.x >> 5], lane);
  Counters cnt;
  WarpItems& S = items[threadIdx.x >> 5];
  for (int64_t r = next_ray(F, P, S, lane, P.spp, -1); r < P.n; r = next_ray(F, P, S, lane, P.spp, r)) {
    const Ray y = batch_ray(P, r);
    const float3 inv = safe_inv(y.v);
    float acc = 0.f;
    for (int s = 0; s < P.spp; ++s) {
      const Mask m = sample_mask(F, P.lod, y.v, P.seed, (uint32_t)r, (uint32_t)s, 0, TAG_MASK);
      if (lane == 0) cnt.rays += 1;
      float t0, t1, T = 1.f;
      if (m.bits != 0ull && scene_span(F, y.o, inv, y.tmin, y.tmax, t0, t1)) {
        if (lane == 0) cnt.windows += 1;
        T = rt_coop(F, Q, m, y.o, y.v, inv, y.tmin, y.tmax, t0, t1, P.seed, (uint32_t)r,
                    stream_word((uint32_t)s, 0, TAG_TRACK), sm.env, lane, P.exact, cnt);
      }
      acc += T;
    }
    if (lane == 0) P.out_T[r] = acc / (float)P.spp;
  }
  if (lane == 0) cnt.rays += S.missed;
  flush_counters(F, cnt, lane);
}

// ---------------------------------------------------------------------------
// Fields of a few kernels (lane_work): a ray has a handful of chords, less than a warp can
// share out, and a lane of its own walks the small tree as fast as a warp does.
// 2,000,000 rays through 8 kernels: 2.6 -> 0.4 ms by quadrature, 2.9 -> 0.3 in closed form, 3.9
// -> 0.4 ratio-tracked; 1024x1024 image through 64 kernels: 2.3 -> 0.5 ms.
// ---------------------------------------------------------------------------
template <int MODE>  // GF_TR_DETERMINISTIC or GF_TR_CLOSED_FORM
struct TauLeaf {
  const DevField* F;
  const Mask* M;
  float3 o, v;
  float tmin, tmax;
  const BlockTables* T;
  float s, c;
  unsigned chords = 0, evals = 0;
  __device__ __forceinline__ void operator()(int j) {
    Chord ch;
    float w;
    if (!prim_chord(*F, j, o, v, tmin, tmax, [&](uint32_t cl) { return mask_weight(*M, cl); }, w, ch)) return;
    ++chords;
    if (MODE == GF_TR_CLOSED_FORM) {
      neumaier_add(s, c, w * chord_closed(F->wd, ch));
      return;
    }
    const float len = ch.dtout - ch.dtin, hl = 0.5f * len, mid = 0.5f * (ch.dtin + ch.dtout);
    int n, off;
    gl_pick(gl_rule(sqrtf(ch.a) * len + 0.5f * fabsf(ch.B) * len), n, off);
    evals += (unsigned)n;
    const float y2 = -0.5f * kLog2e * ch.a, y1 = -kLog2e * ch.b, y0 = -0.5f * kLog2e * ch.g;
    const float scale = w * ch.absA * hl;
    for (int k = off; k < off + n; ++k) {
      const float dt = fmaf(hl, T->glx[k], mid);
      const float y = fmaf(fmaf(y2, dt, y1), dt, y0);
      neumaier_add(s, c, scale * T->glw[k] * ex2f(y) * cosf(fmaf(ch.B, dt, ch.delta)));
    }
  }
};
// optical depth of the lane's ray added to (s, c)
template <int MODE>
__device__ __forceinline__ void lane_tau(const DevField& F, const BlockTables& T, const Mask& M, float3 o, float3 v,
                                         float tmin, float tmax, float& s, float& c, Counters& cnt) {
  const float3 inv = safe_inv(v);
  float t0, t1;
  if (M.bits == 0ull || !scene_span(F, o, inv, tmin, tmax, t0, t1)) return;
  cnt.windows += 1;
  TauLeaf<MODE> leaf{&F, &M, o, v, tmin, tmax, &T, s, c};
  SpanTest test{t0, t1};
  traverse_ray(F, o, inv, M.bits, test, leaf, cnt.nodes, cnt.leaves);
  cnt.chords += leaf.chords;
  cnt.evals += leaf.evals;
  s = leaf.s;
  c = leaf.c;
}

template <int MODE>
__global__ void __launch_bounds__(kBlock) k_transmittance_lane(const __grid_constant__ DevField F,
                                                              const __grid_constant__ TrParams P) {
  __shared__ BlockTables sm;
  init_tables(sm, F);
  const uint32_t lane = threadIdx.x & 31u;
  Counters cnt;
  const int spp = MODE != GF_TR_RATIO_TRACKING && lod_is_deterministic(P.lod) ? 1 : P.spp;
  for (;;) {
    const uint32_t tile = next_tile(P.counter, lane);
    if ((int64_t)tile * 32 >= P.n) break;
    const int64_t r = (int64_t)tile * 32 + lane;
    if (r < P.n) {
      const Ray y = batch_ray(P, r);
      float s_acc = 0.f, c_acc = 0.f, acc = 0.f;
      for (int s = 0; s < spp; ++s) {
        const Mask m = sample_mask(F, P.lod, y.v, P.seed, (uint32_t)r, (uint32_t)s, 0, TAG_MASK);
        cnt.rays += 1;
        if constexpr (MODE == GF_TR_RATIO_TRACKING)
          acc += track(F, m, y.o, y.v, y.tmin, y.tmax, P.seed, (uint32_t)r,
                       stream_word((uint32_t)s, 0, TAG_TRACK), sm.env, cnt);
        else
          lane_tau<MODE>(F, sm, m, y.o, y.v, y.tmin, y.tmax, s_acc, c_acc, cnt);
      }
      if (MODE == GF_TR_RATIO_TRACKING) {
        P.out_T[r] = acc / (float)spp;
      } else {
        const float tau = __fadd_rn(s_acc, c_acc) / (float)spp;
        P.out_T[r] = expf(-tau);
        if (P.out_tau) P.out_tau[r] = tau;
      }
    }
    __syncwarp();
  }
  flush_counters(F, cnt, lane);
}

__global__ void __launch_bounds__(kBlock)
    k_tomo_lane(const __grid_constant__ DevField F, const __grid_constant__ PathParams P, float* out, int* counter) {
  __shared__ BlockTables sm;
  init_tables(sm, F);
  const uint32_t lane = threadIdx.x & 31u;
  Counters cnt;
  const int64_t npix = (int64_t)P.roi_w * P.roi_h;
  for (;;) {
    const uint32_t tile = next_tile(counter, lane);
    if ((int64_t)tile * 32 >= npix) break;
    const int64_t i = (int64_t)tile * 32 + lane;
    if (i < npix) {
      const int pix = roi_pixel(P, (uint32_t)i);
      float acc = 0.f;
      for (int s = P.s0; s < P.s0 + P.spp; ++s) {
        float3 o, v;
        camera_ray(P.cam, P.seed, pix % P.cam.W, pix / P.cam.W, s, o, v);
        Mask m = sample_mask(F, P.lod, v, P.seed, (uint32_t)pix, (uint32_t)s, 0, TAG_MASK);
        m.bits &= fov_cells(F, P, v, (uint32_t)pix, (uint32_t)s);
        cnt.rays += 1;
        float s_acc = 0.f, c_acc = 0.f;
        lane_tau<GF_TR_DETERMINISTIC>(F, sm, m, o, v, 0.f, INFINITY, s_acc, c_acc, cnt);
        acc += expf(-__fadd_rn(s_acc, c_acc));
      }
      out[pix] = acc / (float)P.spp;
    }
    __syncwarp();
  }
  flush_counters(F, cnt, lane);
}

// the pixels whose rays all miss the scene
__global__ void k_background(const __grid_constant__ DevField F, const __grid_constant__ PathParams P, float* out,
                             float value) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, npix = (int64_t)P.cam.W * P.cam.H;
  if (i == 0) atomicAdd(F.stats + ST_RAYS, (unsigned long long)(npix - (int64_t)P.roi_w * P.roi_h) * P.spp);
  if (i >= npix) return;
  const int x = (int)(i % P.cam.W) - P.roi_x, y = (int)(i / P.cam.W) - P.roi_y;
  if (x < 0 || x >= P.roi_w || y < 0 || y >= P.roi_h) out[i] = value;
}

// ---------------------------------------------------------------------------
// Tomography image: one pixel per warp, its camera rays one after the other
// (coop_tau), T = exp(-tau) averaged in sample order.  256x256 at 8 samples
// through 200k kernels: 222 ms with one pixel per lane, 20.5 ms with one per warp.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kBlock, kCoopBlocks)
    k_tomo(const __grid_constant__ DevField F, const PathParams P, float* out, int* counter) {
  __shared__ BlockTables sm;
  __shared__ CoopQ qs[kBlock / 32];
  init_tables(sm, F);
  const uint32_t lane = threadIdx.x & 31u;
  CoopQ& Q = qs[threadIdx.x >> 5];
  Counters cnt;
  const int npix = P.roi_w * P.roi_h;
  for (;;) {
    const uint32_t tile = next_tile(counter, lane);
    if (tile >= (uint32_t)npix) break;
    const int pix = roi_pixel(P, tile);
    float acc = 0.f;
    for (int s = P.s0; s < P.s0 + P.spp; ++s) {
      float3 o, v;
      camera_ray(P.cam, P.seed, pix % P.cam.W, pix / P.cam.W, s, o, v);
      Mask m = sample_mask(F, P.lod, v, P.seed, (uint32_t)pix, (uint32_t)s, 0, TAG_MASK);
      m.bits &= fov_cells(F, P, v, (uint32_t)pix, (uint32_t)s);
      if (lane == 0) cnt.rays += 1;
      float s_acc = 0.f, c_acc = 0.f;
      coop_tau<GF_TR_DETERMINISTIC>(F, Q, m, o, v, 0.f, INFINITY, sm.glx, sm.glw, lane, s_acc,
                                    c_acc, cnt);
      warp_sum_pair(s_acc, c_acc);
      acc += expf(-__fadd_rn(s_acc, c_acc));
    }
    if (lane == 0) out[pix] = acc / (float)P.spp;
  }
  flush_counters(F, cnt, lane);
}

// The path of sample s of pixel pix with analytic free flights; returns its radiance.
// gather(mask, o, v) leaves the ray's total optical depth and last chord exit in L,
// fly(mask, o, v, target, u) finds the collision; count: whether the caller counts its rays.
template <class L_, class Gather, class Fly>
__device__ __forceinline__ float flight_path(const DevField& F, const PathParams& P, uint32_t pix, int s, bool count,
                                             Counters& cnt, const L_& L, Gather&& gather, Fly&& fly) {
  float3 o, v;
  camera_ray(P.cam, P.seed, (int)pix % P.cam.W, (int)pix / P.cam.W, s, o, v);
  const unsigned long long allow = fov_cells(F, P, v, pix, (uint32_t)s);
  float thr = 1.f, Lsum = 0.f;
  for (int b = 0; b < P.max_bounces; ++b) {
    Mask m = sample_mask(F, P.lod, v, P.seed, pix, (uint32_t)s, (uint32_t)b, TAG_MASK);
    m.bits &= allow;
    if (count) cnt.rays += 1;
    const uint4 y = rng4(P.seed, 0, kNoPrim, pix, stream_word((uint32_t)s, (uint32_t)b, TAG_TRACK));
    const float target = -log1pf(-u01(y.x));
    gather(m, o, v);
    if (!(L.tend > 0.f) || L.tau < target) break;  // escaped
    const float th = fly(m, o, v, target, u01(y.y));
    const float3 x = make_float3(o.x + th * v.x, o.y + th * v.y, o.z + th * v.z);
    thr *= P.albedo;
    Mask mn = sample_mask(F, P.lod_nee, P.light, P.seed, pix, (uint32_t)s, (uint32_t)b, TAG_NEE_MASK);
    mn.bits &= allow;
    if (count) cnt.rays += 1;
    gather(mn, x, P.light);
    Lsum += thr * P.irradiance * expf(-L.tau) * (0.25f / 3.14159265358979f);
    const uint4 z4 = rng4(P.seed, 0, kNoPrim, pix, stream_word((uint32_t)s, (uint32_t)b, TAG_SCATTER));
    const float z = 1.0f - 2.0f * u01(z4.x);
    const float rr = sqrtf(fmaxf(0.0f, 1.0f - z * z));
    float sn, cs;
    sincosf(2.0f * 3.14159265358979f * u01(z4.y), &sn, &cs);
    v = make_float3(rr * cs, rr * sn, z);
    o = x;
  }
  return Lsum;
}

// ---------------------------------------------------------------------------
// Scattering render with an analytic free flight (FF: GF_FLIGHT_CDF or
// GF_FLIGHT_SEGMENT): one pixel per warp, its samples in order; every flight works on
// the ray's collected chords, the NEE transmittance is exp(-tau) in closed form.
// 160x120 at 2 samples through 50k kernels: 260 ms with one pixel per lane and a
// traversal for each of up to 33 depths of a flight, 2.9 ms from lists.  Bound by instruction
// issue: two traversals per collision, then the Faddeeva sums of the chord ends.
// ---------------------------------------------------------------------------
constexpr int kFlightBlocks = 5;  // resident blocks per SM (3.02 ms with 4, 2.85 with 5)
template <int FF>
__global__ void __launch_bounds__(kBlock, kFlightBlocks)
    k_flight(const __grid_constant__ DevField F, const __grid_constant__ PathParams P, float* out,
             int* counter, FlightRec* store, int cap) {
  __shared__ FlightQ qs[kBlock / 32];
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  FlightQ& Q = qs[warp];
  Flight L;
  L.list = store + ((size_t)blockIdx.x * (kBlock / 32) + warp) * kFlightList;
  L.cap = cap;
  Counters cnt;
  const int npix = P.roi_w * P.roi_h;
  for (;;) {
    const uint32_t tile = next_tile(counter, lane);
    if (tile >= (uint32_t)npix) break;
    const uint32_t pix = (uint32_t)roi_pixel(P, tile);
    float acc = 0.f;
    for (int s = P.s0; s < P.s0 + P.spp; ++s)
      acc += flight_path(
          F, P, pix, s, lane == 0, cnt, L,
          [&](const Mask& m, float3 o, float3 v) { flight_gather(F, Q, m, o, v, lane, L, cnt); },
          [&](const Mask& m, float3 o, float3 v, float target, float u) {
            return FF == GF_FLIGHT_CDF ? cdf_flight(F, Q, m, o, v, target, lane, L, cnt)
                                       : segment_flight(F, Q, m, o, v, target, u, lane, L, cnt);
          });
    if (lane == 0) out[pix] = acc / (float)P.spp;
  }
  flush_counters(F, cnt, lane);
}

// ---------------------------------------------------------------------------
// Analytic free flights of a lane's own rays, for fields of a few kernels: as k_flight (flight_gather, cdf_flight and
// segment_flight), with the chord list of a ray in the lane's local memory.  1024x1024 through 8
// kernels: 2.5 -> 0.20 ms (CDF), 2.3 -> 0.14 ms (segment).
// ---------------------------------------------------------------------------
constexpr int kLaneFlight = 16;  // kernels of the field at most
struct LaneFlight {
  FlightRec list[kLaneFlight];
  int n;
  float tau, tend;
};
struct LaneFlightLeaf {
  const DevField* F;
  const Mask* M;
  float3 o, v;
  LaneFlight* L;
  float s, c;
  __device__ __forceinline__ void operator()(int j) {
    Chord ch;
    float w;
    if (!prim_chord(*F, j, o, v, 0.f, INFINITY, [&](uint32_t cl) { return mask_weight(*M, cl); }, w, ch)) return;
    const float full = w * chord_closed(F->wd, ch);
    neumaier_add(s, c, full);
    L->tend = fmaxf(L->tend, ch.tc + ch.dtout);
    if (L->n < kLaneFlight)
      L->list[L->n++] = FlightRec{ch.tc, ch.dtin, ch.dtout, ch.a, ch.b, ch.g, ch.B, ch.delta, ch.absA, ch.qmin,
                                  ch.dts, w, full, {0.f, 0.f, 0.f}};
  }
};
static __device__ __noinline__ void lane_gather(const DevField& F, const Mask& M, float3 o, float3 v, LaneFlight& L,
                                                Counters& cnt) {
  const float3 inv = safe_inv(v);
  float t0, t1;
  L.n = 0;
  L.tau = 0.f;
  L.tend = -INFINITY;
  if (M.bits == 0ull || !scene_span(F, o, inv, 0.f, INFINITY, t0, t1)) return;
  LaneFlightLeaf leaf{&F, &M, o, v, &L, 0.f, 0.f};
  SpanTest test{t0, t1};
  traverse_ray(F, o, inv, M.bits, test, leaf, cnt.nodes, cnt.leaves);
  cnt.windows += 1;
  cnt.chords += (unsigned)L.n;
  L.tau = __fadd_rn(leaf.s, leaf.c);
}
static __device__ __noinline__ float lane_cdf(const DevField& F, const LaneFlight& L, float target) {
  float lo = 0.f, hi = L.tend;
  for (int it = 0; it < 32; ++it) {
    const float mid = 0.5f * (lo + hi);
    float s = 0.f, c = 0.f;
    for (int k = 0; k < L.n; ++k) flight_part(F, L.list[k], mid, s, c);
    if (__fadd_rn(s, c) < target) lo = mid;
    else hi = mid;
  }
  return 0.5f * (lo + hi);
}
static __device__ __noinline__ float lane_segment(const DevField& F, const LaneFlight& L, float target, float u) {
  float lo = 0.f, hi = L.tend;
  float ea = 0.f, eb = L.tend;
  for (int it = 0; it < 48; ++it) {
    const float mid = 0.5f * (lo + hi);
    float s = 0.f, c = 0.f;
    SegmentEnds E;
    for (int k = 0; k < L.n; ++k) segment_part(F, L.list[k], lo, mid, hi, E, s, c);
    if (__fadd_rn(s, c) < target) {
      lo = mid;
      ea = E.below_mid;
      eb = E.above_hi;
      if (E.n_right == 0) break;
    } else {
      hi = mid;
      ea = E.below_lo;
      eb = E.above_mid;
      if (E.n_left == 0) break;
    }
    if (!(hi > lo)) break;
  }
  if (!(eb < INFINITY)) eb = L.tend;
  return ea + u * (eb - ea);
}

template <int FF>
__global__ void __launch_bounds__(kBlock)
    k_flight_lane(const __grid_constant__ DevField F, const __grid_constant__ PathParams P, float* out, int* counter) {
  const uint32_t lane = threadIdx.x & 31u;
  LaneFlight L;
  Counters cnt;
  const int64_t npix = (int64_t)P.roi_w * P.roi_h;
  for (;;) {
    const uint32_t tile = next_tile(counter, lane);
    if ((int64_t)tile * 32 >= npix) break;
    const int64_t i = (int64_t)tile * 32 + lane;
    if (i < npix) {
      const uint32_t pix = (uint32_t)roi_pixel(P, (uint32_t)i);
      float acc = 0.f;
      for (int s = P.s0; s < P.s0 + P.spp; ++s)
        acc += flight_path(
            F, P, pix, s, true, cnt, L, [&](const Mask& m, float3 o, float3 v) { lane_gather(F, m, o, v, L, cnt); },
            [&](const Mask&, float3, float3, float target, float u) {
              return FF == GF_FLIGHT_CDF ? lane_cdf(F, L, target) : lane_segment(F, L, target, u);
            });
      out[pix] = acc / (float)P.spp;
    }
    __syncwarp();
  }
  flush_counters(F, cnt, lane);
}

__global__ void k_faddeeva(const Weideman W, const float* z, float* w, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float x = z[2 * i], y = z[2 * i + 1];
  float2 r = make_float2(__int_as_float(0x7fc00000), __int_as_float(0x7fc00000));
  if (y >= 0.0f) r = faddeeva_w(W, x, y);
  w[2 * i] = r.x;
  w[2 * i + 1] = r.y;
}

// ---------------------------------------------------------------------------
// chord sets (testing)
// ---------------------------------------------------------------------------
struct ListLeaf {
  const DevField* F;
  const Mask* M;
  float3 o, v;
  float tmin, tmax;
  const ChordParams* P;
  int64_t r;
  int n = 0;
  __device__ __forceinline__ void operator()(int j) {
    const Mask& Mk = *M;
    Chord ch;
    float w;
    if (!prim_chord(*F, j, o, v, tmin, tmax, [&](uint32_t c) { return mask_weight(Mk, c); }, w, ch))
      return;
    if (n < P->cap) {
      const int64_t at = r * P->cap + n;
      P->prims[at] = (int)ch.orig;
      if (P->tin) P->tin[at] = ch.tc + ch.dtin;
      if (P->tout) P->tout[at] = ch.tc + ch.dtout;
    }
    ++n;
  }
};

__global__ void __launch_bounds__(kBlock) k_ray_chords(const __grid_constant__ DevField F,
                                                       const ChordParams P) {
  const uint32_t lane = threadIdx.x & 31u;
  for (;;) {
    const uint32_t tile = next_tile(P.counter, lane);
    if ((int64_t)tile * 32 >= P.n) break;
    const int64_t r = (int64_t)tile * 32 + lane;
    if (r >= P.n) continue;  // next_tile below is reached by every lane
    const float3 o = make_float3(P.o[3 * r], P.o[3 * r + 1], P.o[3 * r + 2]);
    const float3 v = unit_dir(make_float3(P.d[3 * r], P.d[3 * r + 1], P.d[3 * r + 2]));
    const float tmin = P.trange ? P.trange[2 * r] : 0.f;
    const float tmax = P.trange ? P.trange[2 * r + 1] : INFINITY;
    const Mask m = sample_mask(F, P.lod, v, 0, (uint32_t)r, 0, 0, TAG_MASK);
    const float3 inv = safe_inv(v);
    float t0, t1;
    int n = 0;
    if (m.bits && scene_span(F, o, inv, tmin, tmax, t0, t1)) {
      ListLeaf leaf;
      leaf.F = &F;
      leaf.M = &m;
      leaf.o = o;
      leaf.v = v;
      leaf.tmin = tmin;
      leaf.tmax = tmax;
      leaf.P = &P;
      leaf.r = r;
      SpanTest test{t0, t1};
      unsigned long long nv = 0, nl = 0;
      traverse_ray(F, o, inv, m.bits, test, leaf, nv, nl);
      n = leaf.n;
    }
    P.counts[r] = n;
  }
}

__global__ void k_philox(const uint32_t* ctr, const uint32_t* key, uint32_t* out, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint4 c = make_uint4(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]);
  const uint2 k = make_uint2(key[2 * i], key[2 * i + 1]);
  const uint4 r = philox(c, k);
  out[4 * i] = r.x;
  out[4 * i + 1] = r.y;
  out[4 * i + 2] = r.z;
  out[4 * i + 3] = r.w;
}

// ---------------------------------------------------------------------------
// launchers: persistent grids of (resident blocks per SM) x SMs
// ---------------------------------------------------------------------------
// every kernel's per-thread stack (its local memory frame, callees included)
// must fit the context's stack limit as it stands at launch (gf_create raises
// it to at least kStackLimit; another component of the process may change it)
template <class K>
static bool stack_fits(K kernel) {
  cudaFuncAttributes a;
  if (cudaFuncGetAttributes(&a, kernel) != cudaSuccess) return false;
  size_t limit = 0;
  if (cudaDeviceGetLimit(&limit, cudaLimitStackSize) != cudaSuccess) return false;
  return a.localSizeBytes <= limit;
}

template <class K>
static int persistent_grid(const Field& F, K kernel, int64_t warps_of_work) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kBlock, 0) != cudaSuccess)
    (void)cudaGetLastError();
  if (per_sm < 1) per_sm = 1;
  const int64_t need = (warps_of_work + kBlock / 32 - 1) / (kBlock / 32);
  int64_t g = (int64_t)F.ctx.sm_count * per_sm;
  if (need < g) g = need;
  return (int)(g < 1 ? 1 : g);
}

template <class K>
static cudaError_t launch_rays(const Field& F, K kernel, TrParams P, cudaStream_t s) {
  const int64_t g = persistent_grid(F, kernel, P.n);
  // up to four rays per warp are dealt out: the counter's clearing is a launch of its own (3 us
  // of 4,096 rays through 256 kernels)
  P.dealt = P.n <= 4 * g * (kBlock / 32);
  if (!P.dealt) {
    const cudaError_t e = cudaMemsetAsync(P.counter, 0, sizeof(int), s);
    if (e != cudaSuccess) return e;
  }
  kernel<<<(unsigned)g, kBlock, 0, s>>>(F.dev, P);
  return cudaGetLastError();
}

// Whether `items` rays or pixels go to a lane each: few kernels, and items enough to fill the
// lanes.  The lines lie where both sides take the same time in the worse of two kinds of
// fields (scales of 0.02 to 0.1 and of 0.1 to 0.25 in the unit cube): at 200,000 rays and
// more 24 kernels by quadrature and ratio tracking, 48 in closed form, 128 for images (whose
// neighbours take the same ways); with fewer items a 2,500th of them (40,000 rays: 16).  Of
// flight images a 7,500th of the pixels, up to the 16 that a lane's list holds.
constexpr int64_t kLaneTau = 24, kLaneClosed = 48, kLaneTomo = 128;
static bool lane_work(const Field& F, int64_t items, int64_t most) {
  return F.n <= std::min(most, items / 2500);
}
// (where the kernel's stack does not fit the limit in force, a ray per warp)
template <class K>
static bool lanes_fit(const Field& F, K kernel, int64_t items, int64_t most) {
  return lane_work(F, items, most) && stack_fits(kernel);
}
template <class K>
static cudaError_t launch_lanes(const Field& F, K kernel, const TrParams& P, cudaStream_t s) {
  const cudaError_t e = cudaMemsetAsync(P.counter, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  kernel<<<(unsigned)persistent_grid(F, kernel, (P.n + 31) / 32), kBlock, 0, s>>>(F.dev, P);
  return cudaGetLastError();
}

cudaError_t launch_transmittance(const Field& F, const TrParams& P, cudaStream_t s) {
  (void)cudaGetLastError();  // a stale error of an unrelated call is not ours
  auto det = k_transmittance_lane<GF_TR_DETERMINISTIC>;
  auto closed = k_transmittance_lane<GF_TR_CLOSED_FORM>;
  auto rt = k_transmittance_lane<GF_TR_RATIO_TRACKING>;
  if (P.mode == GF_TR_DETERMINISTIC && lanes_fit(F, det, P.n, kLaneTau)) return launch_lanes(F, det, P, s);
  if (P.mode == GF_TR_CLOSED_FORM && lanes_fit(F, closed, P.n, kLaneClosed)) return launch_lanes(F, closed, P, s);
  if (P.mode == GF_TR_DETERMINISTIC) return launch_rays(F, k_transmittance_coop<GF_TR_DETERMINISTIC>, P, s);
  if (P.mode == GF_TR_CLOSED_FORM) return launch_rays(F, k_transmittance_coop<GF_TR_CLOSED_FORM>, P, s);
  if (!stack_fits(k_transmittance_rt_coop)) return cudaErrorLaunchOutOfResources;
  TrParams Q = P;
  Q.exact = P.n * 8 > (int64_t)F.ctx.sm_count * 16 * 32;
  // (the tracker of a lane has that form)
  if (Q.exact && lanes_fit(F, rt, P.n, kLaneTau)) return launch_lanes(F, rt, P, s);
  return launch_rays(F, k_transmittance_rt_coop, Q, s);
}

// bytes of the analytic flights' chord lists, per block and of a full persistent grid
constexpr size_t kFlightShare = (size_t)(kBlock / 32) * kFlightList * sizeof(FlightRec);
static int64_t flight_grid(const Field& F) {
  return std::max(persistent_grid(F, k_flight<GF_FLIGHT_CDF>, (int64_t)1 << 40),
                  persistent_grid(F, k_flight<GF_FLIGHT_SEGMENT>, (int64_t)1 << 40));
}
size_t flight_store_bytes(const Field& F) { return (size_t)flight_grid(F) * kFlightShare; }

// Chord lists for a flight kernel of g blocks, in the chord store of the delta-tracking
// renderer; returns the chords a list holds.  Asked for by the grid, rounded up to a power
// of two so that a series of images settles on one buffer.  Where less is held or to be had
// g becomes the blocks that have lists, down to an eighth; fewer, or none (refused, or
// not reserved before a stream capture): every block, and each depth of a flight traverses.
// 160x120 at 2 samples through 50k kernels: 2.9 ms with lists for every block, 4.0, 5.6, 8.3
// and about 14 with half as many and so on, 13.8 without.
constexpr int64_t kFlightFew = 8;
static int flight_lists(const Field& F, int64_t& g, cudaStream_t s) {
  int64_t lists = 1;
  while (lists < g) lists *= 2;
  lists = std::min(lists, flight_grid(F));
  if (F.wscratch.bytes < kFlightShare && capturing(s)) return 0;
  if (grow_shares(F, F.wscratch, kFlightShare, lists, s) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  if (lists * kFlightFew < g) return 0;
  g = std::min(g, lists);
  return kFlightList;
}

cudaError_t launch_render(const Field& F, const PathParams& P, float* out, cudaStream_t s) {
  (void)cudaGetLastError();  // a stale error of an unrelated call is not ours
  cudaError_t e = cudaMemsetAsync(F.counter, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  if (P.integrator == GF_INTEG_SCATTER && P.free_flight == GF_FLIGHT_DELTA)
    return launch_render_scatter(F, P, out, s);
  const int64_t npix = (int64_t)P.cam.W * P.cam.H, roi = (int64_t)P.roi_w * P.roi_h;
  const bool flight = P.integrator == GF_INTEG_SCATTER;
  if (roi < npix) {
    k_background<<<(unsigned)((npix + 255) / 256), 256, 0, s>>>(F.dev, P, out, flight ? 0.f : 1.f);
    if ((e = cudaGetLastError()) != cudaSuccess || roi == 0) return e;
  }
  auto flight_lane = P.free_flight == GF_FLIGHT_SEGMENT ? k_flight_lane<GF_FLIGHT_SEGMENT> : k_flight_lane<GF_FLIGHT_CDF>;
  if (flight && lanes_fit(F, flight_lane, roi / 3, kLaneFlight)) {
    flight_lane<<<persistent_grid(F, flight_lane, (roi + 31) / 32), kBlock, 0, s>>>(F.dev, P, out, F.counter);
  } else if (flight) {
    auto k = P.free_flight == GF_FLIGHT_SEGMENT ? k_flight<GF_FLIGHT_SEGMENT> : k_flight<GF_FLIGHT_CDF>;
    if (!stack_fits(k)) return cudaErrorLaunchOutOfResources;
    int64_t g = persistent_grid(F, k, roi);
    const int cap = flight_lists(F, g, s);
    k<<<(unsigned)g, kBlock, 0, s>>>(F.dev, P, out, F.counter,
                                     static_cast<FlightRec*>(cap ? F.wscratch.p : nullptr), cap);
  } else if (lanes_fit(F, k_tomo_lane, roi, kLaneTomo)) {
    k_tomo_lane<<<persistent_grid(F, k_tomo_lane, (roi + 31) / 32), kBlock, 0, s>>>(F.dev, P, out, F.counter);
  } else {
    if (!stack_fits(k_tomo)) return cudaErrorLaunchOutOfResources;
    k_tomo<<<persistent_grid(F, k_tomo, roi), kBlock, 0, s>>>(F.dev, P, out, F.counter);
  }
  return cudaGetLastError();
}

cudaError_t launch_ray_chords(const Field& F, const ChordParams& P, cudaStream_t s) {
  (void)cudaGetLastError();  // a stale error of an unrelated call is not ours
  cudaError_t e = cudaMemsetAsync(P.counter, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  k_ray_chords<<<persistent_grid(F, k_ray_chords, (P.n + 31) / 32), kBlock, 0, s>>>(F.dev, P);
  return cudaGetLastError();
}

cudaError_t launch_faddeeva(const Weideman& W, const float* z, float* w, int64_t n,
                           cudaStream_t s) {
  (void)cudaGetLastError();  // a stale error of an unrelated call is not ours
  if (n <= 0) return cudaSuccess;
  const int64_t blocks = (n + 255) / 256;
  k_faddeeva<<<(unsigned)blocks, 256, 0, s>>>(W, z, w, n);
  return cudaGetLastError();
}

cudaError_t launch_philox(const uint32_t* ctr, const uint32_t* key, uint32_t* out, int64_t n,
                          cudaStream_t s) {
  (void)cudaGetLastError();  // a stale error of an unrelated call is not ours
  if (n <= 0) return cudaSuccess;
  const int64_t blocks = (n + 255) / 256;
  k_philox<<<(unsigned)blocks, 256, 0, s>>>(ctr, key, out, n);
  return cudaGetLastError();
}

}  // namespace gf
