// gf_kernels.cu -- render, transmittance and test kernels of the Gabor-field
// renderer.  Persistent warps pull work from a global counter: one ray per warp
// (gf_coop.cuh) for optical depths, analytic free flights and small ratio-tracking
// batches; 32 rays per warp, each lane owning one (gf_trace.cuh), for large
// ratio-tracking batches.
#include <cuda_runtime.h>

#include <algorithm>

#include "gf_coop.cuh"
#include "gf_host.h"
#include "gf_trace.cuh"

namespace gf {

constexpr int kBlock = 128;
constexpr int kCoopBlocks = 5;  // resident blocks per SM of the one-ray-per-warp kernels

// ---------------------------------------------------------------------------
// ratio-tracking transmittance of large batches, one ray per lane
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kBlock, 3)  // at most 168 registers: 12 warps per SM
    k_transmittance_rt(const __grid_constant__ DevField F, const TrParams P) {
  __shared__ BlockTables sm;
  init_tables(sm, F);
  const uint32_t lane = threadIdx.x & 31u;
  Counters cnt;
  for (;;) {
    const uint32_t tile = next_tile(P.counter, lane);
    if ((int64_t)tile * 32 >= P.n) break;
    const int64_t r = (int64_t)tile * 32 + (int)lane;
    if (r < P.n) {
      const float3 o = make_float3(P.o[3 * r], P.o[3 * r + 1], P.o[3 * r + 2]);
      const float3 v = unit_dir(make_float3(P.d[3 * r], P.d[3 * r + 1], P.d[3 * r + 2]));
      const float tmin = P.trange ? P.trange[2 * r] : 0.f;
      const float tmax = P.trange ? P.trange[2 * r + 1] : INFINITY;
      float acc = 0.f;
      for (int s = 0; s < P.spp; ++s) {
        const Mask m = sample_mask(F, P.lod, v, P.seed, (uint32_t)r, (uint32_t)s, 0, TAG_MASK);
        cnt.rays += 1;
        acc += track<false>(F, m, o, v, tmin, tmax, false, P.seed, (uint32_t)r,
                            stream_word((uint32_t)s, 0, TAG_TRACK), sm.env, cnt, nullptr);
      }
      P.out_T[r] = acc / (float)P.spp;
    }
  }
  flush_counters(F, cnt, lane);
}

// ---------------------------------------------------------------------------
// Optical depth of a batch of rays (Gauss-Legendre quadrature or closed-form
// chord integrals), one ray per warp (coop_tau) at every batch size.  Bound by
// instruction issue.  With one ray per lane the lanes part at every leaf: each
// runs its own tree walk and its own rule of 8 to 64 nodes.  130,001 rays
// through 100k kernels (306 chords and 4,092 nodes per ray): 65.0 ms with one
// ray per lane, 5.6 ms with one per warp; 4,096 rays through 256 kernels: 53.6
// us over binary nodes, 35.5 us over four-wide ones with the owner table.
// ---------------------------------------------------------------------------
template <int MODE>  // GF_TR_DETERMINISTIC or GF_TR_CLOSED_FORM
__global__ void __launch_bounds__(kBlock, kCoopBlocks)
    k_transmittance_coop(const __grid_constant__ DevField F, const TrParams P) {
  __shared__ BlockTables sm;
  __shared__ CoopQ qs[kBlock / 32];
  init_tables(sm, F);
  const uint32_t lane = threadIdx.x & 31u;
  CoopQ& Q = qs[threadIdx.x >> 5];
  Counters cnt;
  const int spp = lod_is_deterministic(P.lod) ? 1 : P.spp;
  for (;;) {
    const int64_t r = next_tile(P.counter, lane);
    if (r >= P.n) break;
    const float3 o = make_float3(P.o[3 * r], P.o[3 * r + 1], P.o[3 * r + 2]);
    const float3 v = unit_dir(make_float3(P.d[3 * r], P.d[3 * r + 1], P.d[3 * r + 2]));
    const float tmin = P.trange ? P.trange[2 * r] : 0.f;
    const float tmax = P.trange ? P.trange[2 * r + 1] : INFINITY;
    float s_acc = 0.f, c_acc = 0.f;
    for (int s = 0; s < spp; ++s) {
      const Mask m = sample_mask(F, P.lod, v, P.seed, (uint32_t)r, (uint32_t)s, 0, TAG_MASK);
      if (lane == 0) cnt.rays += 1;
      coop_tau<MODE>(F, Q, m, o, v, tmin, tmax, sm.glx, sm.glw, lane, s_acc, c_acc, cnt);
    }
    warp_sum_pair(s_acc, c_acc);
    if (lane == 0) {
      const float tau = __fadd_rn(s_acc, c_acc) / (float)spp;
      P.out_T[r] = expf(-tau);
      if (P.out_tau) P.out_tau[r] = tau;
    }
  }
  flush_counters(F, cnt, lane);
}

// ---------------------------------------------------------------------------
// Ratio tracking of small batches, one ray per warp.  The warp traverses the
// ray's tree together; each round's chords (one per lane) store their
// evaluation records in shared memory and draw all their tentative points in
// [t0, t1] (chord_points: the per-chord streams of the per-thread tracker, so
// the same points), written in lane order after a counting pass.  Then each
// lane takes points i = lane, lane + 32, ..., sums kappa and kappa_bar at them
// over all stored chords in order, and multiplies its factors 1 - kappa /
// kappa_bar; the lanes' products are combined in a fixed butterfly order.  A
// ray with more chords or points than the buffers hold is tracked by the
// per-thread tracker instead (lane 0).
// ---------------------------------------------------------------------------
constexpr int kRtChords = 256;  // chords of one ray held in shared memory
constexpr int kRtPts = 128;     // tentative points of one ray
struct RtQ {
  CoopTrav t;
  float4 rec[kRtChords][2];  // centred on the envelope peak t*: (t*, t_in, t_out, B),
                             // (-a log2(e) / 2, log2 h, phase at t*, sqrt(a))
  float pt[kRtPts], pu[kRtPts];
};

__device__ float rt_coop(const DevField& F, RtQ& Q, const Mask& M, float3 o, float3 v, float3 inv,
                         float tmin, float tmax, float t0, float t1, uint64_t seed, uint32_t ray,
                         uint32_t word, const float* env, uint32_t lane, Counters& cnt) {
  const unsigned lt = (1u << lane) - 1u;
  int nch = 0, npts = 0;  // warp-uniform
  coop_traverse(F, Q.t, M.bits, o, inv, t0, t1, lane, cnt, [&](int j) {
    Chord ch;
    float w, h = 0.f;
    bool ok = false;
    if (j >= 0 &&
        prim_chord(F, j, o, v, tmin, tmax, [&](uint32_t cl) { return mask_weight(M, cl); }, w, ch) &&
        ch.tc + ch.dtin <= t1 && ch.tc + ch.dtout >= t0) {
      ok = true;
      h = w * ch.absA * expf(-0.5f * ch.qmin);
    }
    const unsigned bc = __ballot_sync(kFull, ok);
    if (ok) {
      ++cnt.chords;
      const int k = nch + __popc(bc & lt);
      if (k < kRtChords) {
        Q.rec[k][0] = make_float4(ch.tc + ch.dts, ch.tc + ch.dtin, ch.tc + ch.dtout, ch.B);
        Q.rec[k][1] = make_float4(-0.5f * kLog2e * ch.a, __log2f(h),
                                  reduce_2pi(fmaf(ch.B, ch.dts, ch.delta)), sqrtf(ch.a));
      }
    }
    nch += __popc(bc);
    // the round's points in lane order: count, then write at the prefix offsets
    int m = 0;
    if (ok)
      chord_points(F, ch, h, seed, ray, word, env, [&](float t, float) {
        if (t > t1) return false;
        if (t >= t0) ++m;
        return true;
      });
    const int incl = warp_incl_sum(m, lane);
    if (ok && m > 0) {
      int q = npts + incl - m;
      chord_points(F, ch, h, seed, ray, word, env, [&](float t, float u) {
        if (t > t1) return false;
        if (t >= t0) {
          if (q < kRtPts) {
            Q.pt[q] = t;
            Q.pu[q] = u;
          }
          ++q;
        }
        return true;
      });
    }
    npts += __shfl_sync(kFull, incl, 31);
  });
  if (lane == 0) cnt.points += (unsigned long long)npts;
  __syncwarp();
  if (nch > kRtChords || npts > kRtPts) {  // too many for the buffers: per-thread tracker
    float T = 1.f;
    if (lane == 0) T = track<false>(F, M, o, v, tmin, tmax, false, seed, ray, word, env, cnt, nullptr);
    return __shfl_sync(kFull, T, 0);
  }
  float prod = 1.f;
  for (int i = (int)lane; i < npts; i += 32) {
    const float t = Q.pt[i];
    float kap = 0.f, kb = 0.f;
    for (int c = 0; c < nch; ++c) {
      const float4 a = Q.rec[c][0];
      if (t >= a.y && t <= a.z) {
        const float4 b = Q.rec[c][1];
        const float dt = t - a.x;
        kap = fmaf(ex2f(fmaf(b.x, dt * dt, b.y)), cosf_fast(fmaf(a.w, dt, b.z)), kap);
        int mm = (int)(fabsf(dt) * b.w);
        mm = mm > 7 ? 7 : mm;
        kb = fmaf(ex2f(b.y), env[mm], kb);  // h exp(-m^2/2)
        ++cnt.evals;
      }
    }
    if (kb > 0.f) prod *= 1.f - kap / kb;
  }
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) prod *= __shfl_xor_sync(kFull, prod, off);
  return prod;
}

__global__ void __launch_bounds__(kBlock, 3)
    k_transmittance_rt_coop(const __grid_constant__ DevField F, const TrParams P) {
  __shared__ BlockTables sm;
  __shared__ RtQ qs[kBlock / 32];
  init_tables(sm, F);
  const uint32_t lane = threadIdx.x & 31u;
  RtQ& Q = qs[threadIdx.x >> 5];
  Counters cnt;
  for (;;) {
    const int64_t r = next_tile(P.counter, lane);  // one ray per warp
    if (r >= P.n) break;
    const float3 o = make_float3(P.o[3 * r], P.o[3 * r + 1], P.o[3 * r + 2]);
    const float3 v = unit_dir(make_float3(P.d[3 * r], P.d[3 * r + 1], P.d[3 * r + 2]));
    const float tmin = P.trange ? P.trange[2 * r] : 0.f;
    const float tmax = P.trange ? P.trange[2 * r + 1] : INFINITY;
    const float3 inv = safe_inv(v);
    float acc = 0.f;
    for (int s = 0; s < P.spp; ++s) {
      const Mask m = sample_mask(F, P.lod, v, P.seed, (uint32_t)r, (uint32_t)s, 0, TAG_MASK);
      if (lane == 0) cnt.rays += 1;
      float t0, t1, T = 1.f;
      if (m.bits != 0ull && scene_span(F, o, inv, tmin, tmax, t0, t1)) {
        if (lane == 0) cnt.windows += 1;
        T = rt_coop(F, Q, m, o, v, inv, tmin, tmax, t0, t1, P.seed, (uint32_t)r,
                    stream_word((uint32_t)s, 0, TAG_TRACK), sm.env, lane, cnt);
      }
      acc += T;
    }
    if (lane == 0) P.out_T[r] = acc / (float)P.spp;
  }
  flush_counters(F, cnt, lane);
}

// ---------------------------------------------------------------------------
// Tomography image: one pixel per warp, its camera rays one after the other
// (coop_tau), T = exp(-tau) averaged in sample order.  256x256 at 8 samples
// through 200k kernels: 222 ms with one pixel per lane, 29 ms with one per warp.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kBlock, kCoopBlocks)
    k_tomo(const __grid_constant__ DevField F, const PathParams P, float* out, int* counter) {
  __shared__ BlockTables sm;
  __shared__ CoopQ qs[kBlock / 32];
  init_tables(sm, F);
  const uint32_t lane = threadIdx.x & 31u;
  CoopQ& Q = qs[threadIdx.x >> 5];
  Counters cnt;
  const int npix = P.cam.W * P.cam.H;
  for (;;) {
    const uint32_t tile = next_tile(counter, lane);
    if (tile >= (uint32_t)npix) break;
    const int pix = (int)tile;
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

// ---------------------------------------------------------------------------
// Scattering render with an analytic free flight (FF: GF_FLIGHT_CDF or
// GF_FLIGHT_SEGMENT): one pixel per warp, its samples in order; every flight works on
// the ray's collected chords, the NEE transmittance is exp(-tau) in closed form.
// 160x120 at 2 samples through 50k kernels: 260 ms with one pixel per lane and a
// traversal for each of up to 33 depths of a flight, 2.9 ms now.  Bound by instruction
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
  const int npix = P.cam.W * P.cam.H;
  for (;;) {
    const uint32_t tile = next_tile(counter, lane);
    if (tile >= (uint32_t)npix) break;
    const uint32_t pix = tile;
    float acc = 0.f;
    for (int s = P.s0; s < P.s0 + P.spp; ++s) {
      float3 o, v;
      camera_ray(P.cam, P.seed, (int)pix % P.cam.W, (int)pix / P.cam.W, s, o, v);
      const unsigned long long allow = fov_cells(F, P, v, pix, (uint32_t)s);
      float thr = 1.f, Lsum = 0.f;
      for (int b = 0; b < P.max_bounces; ++b) {
        Mask m = sample_mask(F, P.lod, v, P.seed, pix, (uint32_t)s, (uint32_t)b, TAG_MASK);
        m.bits &= allow;
        if (lane == 0) cnt.rays += 1;
        const uint4 y = rng4(P.seed, 0, kNoPrim, pix, stream_word((uint32_t)s, (uint32_t)b, TAG_TRACK));
        const float target = -log1pf(-u01(y.x));
        flight_gather(F, Q, m, o, v, lane, L, cnt);
        if (!(L.tend > 0.f) || L.tau < target) break;  // escaped
        const float th = FF == GF_FLIGHT_CDF
                             ? cdf_flight(F, Q, m, o, v, target, lane, L, cnt)
                             : segment_flight(F, Q, m, o, v, target, u01(y.y), lane, L, cnt);
        const float3 x = make_float3(o.x + th * v.x, o.y + th * v.y, o.z + th * v.z);
        thr *= P.albedo;
        Mask mn = sample_mask(F, P.lod_nee, P.light, P.seed, pix, (uint32_t)s, (uint32_t)b,
                              TAG_NEE_MASK);
        mn.bits &= allow;
        if (lane == 0) cnt.rays += 1;
        flight_gather(F, Q, mn, x, P.light, lane, L, cnt);
        Lsum += thr * P.irradiance * expf(-L.tau) * (0.25f / 3.14159265358979f);
        const uint4 z4 = rng4(P.seed, 0, kNoPrim, pix, stream_word((uint32_t)s, (uint32_t)b, TAG_SCATTER));
        const float z = 1.0f - 2.0f * u01(z4.x);
        const float rr = sqrtf(fmaxf(0.0f, 1.0f - z * z));
        float sn, cs;
        sincosf(2.0f * 3.14159265358979f * u01(z4.y), &sn, &cs);
        v = make_float3(rr * cs, rr * sn, z);
        o = x;
      }
      acc += Lsum;
    }
    if (lane == 0) out[pix] = acc / (float)P.spp;
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

cudaError_t launch_transmittance(const Field& F, const TrParams& P, cudaStream_t s) {
  (void)cudaGetLastError();  // a stale error of an unrelated call is not ours
  cudaError_t e = cudaMemsetAsync(P.counter, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  if (P.mode == GF_TR_DETERMINISTIC) {
    auto k = k_transmittance_coop<GF_TR_DETERMINISTIC>;
    k<<<persistent_grid(F, k, P.n), kBlock, 0, s>>>(F.dev, P);
  } else if (P.mode == GF_TR_CLOSED_FORM) {
    auto k = k_transmittance_coop<GF_TR_CLOSED_FORM>;
    k<<<persistent_grid(F, k, P.n), kBlock, 0, s>>>(F.dev, P);
  } else if (P.n * 8 <= (int64_t)F.ctx.sm_count * 16 * 32) {
    // few rays: the whole warp on each ray (k_transmittance_rt_coop)
    auto k = k_transmittance_rt_coop;
    k<<<persistent_grid(F, k, P.n), kBlock, 0, s>>>(F.dev, P);
  } else {
    const int64_t tiles = (P.n + 31) / 32;
    auto k = k_transmittance_rt;
    k<<<persistent_grid(F, k, tiles), kBlock, 0, s>>>(F.dev, P);
  }
  return cudaGetLastError();
}

// bytes of the analytic flights' chord lists of a full persistent grid
size_t flight_store_bytes(const Field& F) {
  const int64_t g = std::max(persistent_grid(F, k_flight<GF_FLIGHT_CDF>, (int64_t)1 << 40),
                             persistent_grid(F, k_flight<GF_FLIGHT_SEGMENT>, (int64_t)1 << 40));
  return (size_t)g * (kBlock / 32) * kFlightList * sizeof(FlightRec);
}

cudaError_t launch_render(const Field& F, const PathParams& P, float* out, cudaStream_t s) {
  (void)cudaGetLastError();  // a stale error of an unrelated call is not ours
  cudaError_t e = cudaMemsetAsync(F.counter, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  if (P.integrator == GF_INTEG_SCATTER && P.free_flight == GF_FLIGHT_DELTA)
    return launch_render_scatter(F, P, out, s);
  const int64_t npix = (int64_t)P.cam.W * P.cam.H;
  if (P.integrator == GF_INTEG_SCATTER) {
    auto k = P.free_flight == GF_FLIGHT_SEGMENT ? k_flight<GF_FLIGHT_SEGMENT> : k_flight<GF_FLIGHT_CDF>;
    if (!stack_fits(k)) return cudaErrorLaunchOutOfResources;
    const int64_t g = persistent_grid(F, k, npix);
    // the chord lists share the chord store of the delta-tracking renderer; without the
    // memory (refused, or not reserved before a stream capture) each depth traverses
    int cap = kFlightList;
    const size_t need = flight_store_bytes(F);
    if (F.wscratch_bytes < need) {
      cudaStreamCaptureStatus cap_st = cudaStreamCaptureStatusNone;
      (void)cudaStreamIsCapturing(s, &cap_st);
      if (cap_st != cudaStreamCaptureStatusNone ||
          grow(F, (void**)&F.wscratch, F.wscratch_bytes, need, s) != cudaSuccess) {
        (void)cudaGetLastError();
        cap = 0;
      }
    }
    k<<<(unsigned)g, kBlock, 0, s>>>(F.dev, P, out, F.counter,
                                     reinterpret_cast<FlightRec*>(cap ? F.wscratch : nullptr), cap);
  } else {
    if (!stack_fits(k_tomo)) return cudaErrorLaunchOutOfResources;
    k_tomo<<<persistent_grid(F, k_tomo, npix), kBlock, 0, s>>>(F.dev, P, out, F.counter);
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
