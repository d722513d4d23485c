// gf_adjoint.cu -- hand-written adjoints of the tomography renderer and (further below)
// of the scattering renderer.
//
// Image I_p = (1/spp) sum_s exp(-tau_s) (Sec. 4.6 tomography), tau_s the
// optical depth of Eq. 2-3 along the jittered camera ray.  Given dL/dI:
//   dL/dtheta_i = sum_{p,s} dL/dI_p (-exp(-tau_s)/spp) dtau_s/dtheta_i,
//   dtau/dtheta = int_chord d(integrand)/dtheta dt
//               + g(t_out) dt_out/dtheta - g(t_in) dt_in/dtheta,
// with the ellipsoid ends moving as dt/dtheta = -(dq/dtheta)/(dq/dt)
// (Leibniz rule for the k-sigma-truncated kernel).  A ray is traversed
// once: its chords' moments are kept until its optical depth is known.  Gradients are
// summed by vector atomics, 16 floats per primitive in BVH order, and copied to the
// caller's layout at the end.
#include <cuda_runtime.h>

#include <algorithm>

#include "gf_coop.cuh"
#include "gf_host.h"
#include "gf_trace.cuh"

namespace gf {

struct BackArgs {
  const float* quat;
  const float* ls;
  const float* om;
  const float* w;
  int frame, wmode;
  int64_t n;
  float* grad;
  // null where the memory is not to be had (tomography): parameters are then read in the
  // caller's order and gradients added to grad itself
  const float4* adj;  // per primitive (BVH order): what PrimDeriv::load needs, 3 float4
  float4* acc;        // gradient sums per primitive (BVH order), 4 float4 each
};

// what the gradient of a primitive needs besides its record
struct AdjPrim {
  float4 q;      // unit quaternion
  float4 is;     // 1 / scales, 1 / |q|
  float4 carry;  // input carrier, dA/dweight
};
// of original primitive i with amplitude A
__device__ __forceinline__ AdjPrim adj_prim(const BackArgs& B, int64_t i, float A) {
  float q[4];
  for (int k = 0; k < 4; ++k) q[k] = B.quat[4 * i + k];
  const float iqn = 1.f / sqrtf(q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
  return AdjPrim{make_float4(q[0] * iqn, q[1] * iqn, q[2] * iqn, q[3] * iqn),
                 make_float4(1.f / expf(B.ls[3 * i]), 1.f / expf(B.ls[3 * i + 1]), 1.f / expf(B.ls[3 * i + 2]), iqn),
                 make_float4(B.om[3 * i], B.om[3 * i + 1], B.om[3 * i + 2],
                             B.wmode == GF_WEIGHT_NORMALIZED ? A / B.w[i] : 1.f)};
}

// Derivatives of one kernel g = A exp(-q/2) cos(theta) with respect to its 15
// raw parameters (mu 3, quaternion 4 through qhat = q/|q|, log scale 3, omega 3
// in the input frame, phase, weight) along a ray, at offsets y = x - mu.
struct PrimDeriv {
  float R[3][3];
  float qh[4], iqn;    // unit quaternion (w, x, y, z) and 1/|q| of the raw one
  float is[3], is2[3], kin[3];  // 1/s, 1/s^2 of the scales s, input carrier
  float A, dAdw;
  float3 om;
  bool local, normalized;

  // from the parameters k_adj_prims gathered for sorted primitive j
  __device__ __forceinline__ void load(const BackArgs& B, float amp, float3 omega, int j) {
    const float4* r = B.adj + 3 * (int64_t)j;
    load(B, amp, omega, AdjPrim{__ldg(r), __ldg(r + 1), __ldg(r + 2)});
  }
  __device__ __forceinline__ void load(const BackArgs& B, float amp, float3 omega, const AdjPrim& p) {
    const float4 a = p.q, b = p.is, c = p.carry;
    qh[0] = a.x; qh[1] = a.y; qh[2] = a.z; qh[3] = a.w;
    is[0] = b.x; is[1] = b.y; is[2] = b.z;
    iqn = b.w;
    kin[0] = c.x; kin[1] = c.y; kin[2] = c.z;
    dAdw = c.w;
    const float qw = qh[0], qx = qh[1], qy = qh[2], qz = qh[3];
    R[0][0] = 1.f - 2.f * (qy * qy + qz * qz); R[0][1] = 2.f * (qx * qy - qw * qz);
    R[0][2] = 2.f * (qx * qz + qw * qy);
    R[1][0] = 2.f * (qx * qy + qw * qz); R[1][1] = 1.f - 2.f * (qx * qx + qz * qz);
    R[1][2] = 2.f * (qy * qz - qw * qx);
    R[2][0] = 2.f * (qx * qz - qw * qy); R[2][1] = 2.f * (qy * qz + qw * qx);
    R[2][2] = 1.f - 2.f * (qx * qx + qy * qy);
#pragma unroll
    for (int k = 0; k < 3; ++k) is2[k] = is[k] * is[k];
    local = B.frame == GF_OMEGA_LOCAL;
    normalized = B.wmode == GF_WEIGHT_NORMALIZED;
    A = amp;
    om = omega;
  }

  // The gradient of sum (weight g) over positions y = p + t v, from the moments of the
  // envelope: C_k of e cos(theta) t^k and S_k of e sin(theta) t^k (e the weighted envelope
  // without the amplitude, theta the phase with the sign of the amplitude folded in).  q
  // is quadratic and theta linear in t.  With z = R^T y and
  //   X = (zp C0 + zv C1) / s^2 + kos S0,  Y = (zp C1 + zv C2) / s^2 + kos S1,
  // kos the local carrier over the scales, every derivative is a contraction of X and Y
  // (the carrier's part of mu apart).  A chord end on the ellipsoid at dt adds one term to
  // both (end), so the contractions run once per chord, the quaternion's through
  // G = p X^T + v Y^T (grad).  Tomography adjoint of 524,288 rays through 200k kernels: 31.3
  // ms with the contractions for p, v and each end apart, 28.7 ms now.
  struct Moments {
    float X[3], Y[3];  // without the carrier's part
    float C0, S0, S1;  // with the amplitude
    float c0;          // C0 without it
    float zp[3], zv[3];
  };
  __device__ __forceinline__ Moments moments(float3 p, float3 v, float C0, float C1, float C2,
                                             float S0, float S1) const {
    Moments m;
    const float aA = fabsf(A);
    m.C0 = aA * C0;
    m.c0 = C0;
    m.S0 = aA * S0;
    m.S1 = aA * S1;
    const float c1 = aA * C1, c2 = aA * C2;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      m.zp[k] = R[0][k] * p.x + R[1][k] * p.y + R[2][k] * p.z;
      m.zv[k] = R[0][k] * v.x + R[1][k] * v.y + R[2][k] * v.z;
      m.X[k] = (m.zp[k] * m.C0 + m.zv[k] * c1) * is2[k];
      m.Y[k] = (m.zp[k] * c1 + m.zv[k] * c2) * is2[k];
    }
    return m;
  }

  // The Leibniz term of a chord end at dt (relative to the chord's tc): the end moves as
  // dt/dtheta = -(dq/dtheta)/(dq/dt), g sgn times that enters the integral.  dq/dt is
  // formed from dq/dmu at the end's position (grazing chords divide by little, so its
  // rounding matters).
  __device__ __forceinline__ void end(const Chord& ch, float3 v, float dt, float sgn,
                                      Moments& m) const {
    const float y[3] = {fmaf(dt, v.x, ch.p.x), fmaf(dt, v.y, ch.p.y), fmaf(dt, v.z, ch.p.z)};
    float z[3], dm[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) z[k] = R[0][k] * y[0] + R[1][k] * y[1] + R[2][k] * y[2];
#pragma unroll
    for (int a = 0; a < 3; ++a)
      dm[a] = -2.f * (R[a][0] * z[0] * is2[0] + R[a][1] * z[1] * is2[1] + R[a][2] * z[2] * is2[2]);
    const float dqdt = -(v.x * dm[0] + v.y * dm[1] + v.z * dm[2]);
    if (dqdt == 0.f) return;
    const float q = fmaf(fmaf(ch.a, dt, 2.f * ch.b), dt, ch.g);
    const float g = ch.absA * ex2f(-0.5f * kLog2e * q) * cosf(fmaf(ch.B, dt, ch.delta));
    const float e = 2.f * sgn * g / dqdt;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float x = e * z[k] * is2[k];
      m.X[k] += x;
      m.Y[k] = fmaf(x, dt, m.Y[k]);
    }
  }

  __device__ __forceinline__ void grad(float3 pp, float3 vv, const Moments& m, float acc[15]) const {
    const float p[3] = {pp.x, pp.y, pp.z}, v[3] = {vv.x, vv.y, vv.z};
    const float om3[3] = {om.x, om.y, om.z};
#pragma unroll
    for (int a = 0; a < 3; ++a)
      acc[a] = R[a][0] * m.X[0] + R[a][1] * m.X[1] + R[a][2] * m.X[2] + om3[a] * m.S0;
    float X[3], Y[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float kos = local ? kin[k] * is[k] : 0.f;
      X[k] = m.X[k] + kos * m.S0;
      Y[k] = m.Y[k] + kos * m.S1;
      const float d = m.zp[k] * X[k] + m.zv[k] * Y[k];
      acc[7 + k] = normalized ? d - m.C0 : d;
      acc[10 + k] = local ? -(m.zp[k] * m.S0 + m.zv[k] * m.S1) * is[k] : -(p[k] * m.S0 + v[k] * m.S1);
    }
    // quaternion: dR/dqhat contracted with G, then through qhat = q/|q|
    float G[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int k = 0; k < 3; ++k) G[a][k] = p[a] * X[k] + v[a] * Y[k];
    const float w = qh[0], x = qh[1], y = qh[2], z = qh[3];
    const float dx = G[2][1] - G[1][2], dy = G[0][2] - G[2][0], dz = G[1][0] - G[0][1];
    const float sx = G[2][1] + G[1][2], sy = G[0][2] + G[2][0], sz = G[1][0] + G[0][1];
    const float h[4] = {x * dx + y * dy + z * dz,
                        w * dx + y * sz + z * sy - 2.f * x * (G[1][1] + G[2][2]),
                        w * dy + x * sz + z * sx - 2.f * y * (G[0][0] + G[2][2]),
                        w * dz + x * sy + y * sx - 2.f * z * (G[0][0] + G[1][1])};
    const float sg = w * h[0] + x * h[1] + y * h[2] + z * h[3];
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[3 + i] = -2.f * (h[i] - qh[i] * sg) * iqn;
    acc[13] = -m.S0;
    acc[14] = (A < 0.f ? -1.f : 1.f) * dAdw * m.c0;
  }
};

// what PrimDeriv::load needs, gathered once per call in BVH order (48 bytes per
// primitive instead of 11 scattered words and their arithmetic per chord).  Scales come
// as reciprocals: nine divisions less per chord took the tomography adjoint of 524,288
// rays through 200k kernels from 37.0 to 31.3 ms.
__global__ void k_adj_prims(const float4* rec, const BackArgs B, float4* adj) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= B.n) return;
  const int64_t i = __float_as_uint(rec[4 * j + 3].w) & kOrigMask;
  const AdjPrim p = adj_prim(B, i, rec[4 * j].w);
  adj[3 * j] = p.q;
  adj[3 * j + 1] = p.is;
  adj[3 * j + 2] = p.carry;
}

// the sums of every primitive to the caller's layout and order
__global__ void k_adj_finish(const float4* rec, const BackArgs B) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= B.n) return;
  const int64_t N = B.n, i = __float_as_uint(rec[4 * j + 3].w) & kOrigMask;
  const float4 a = B.acc[4 * j], b = B.acc[4 * j + 1], c = B.acc[4 * j + 2], d = B.acc[4 * j + 3];
  float* g = B.grad;
  g[3 * i] = a.x; g[3 * i + 1] = a.y; g[3 * i + 2] = a.z;
  g[3 * N + 4 * i] = a.w; g[3 * N + 4 * i + 1] = b.x; g[3 * N + 4 * i + 2] = b.y;
  g[3 * N + 4 * i + 3] = b.z;
  g[7 * N + 3 * i] = b.w; g[7 * N + 3 * i + 1] = c.x; g[7 * N + 3 * i + 2] = c.y;
  g[10 * N + 3 * i] = c.z; g[10 * N + 3 * i + 1] = c.w; g[10 * N + 3 * i + 2] = d.x;
  g[13 * N + i] = d.y;
  g[14 * N + i] = d.z;
}

__device__ __forceinline__ void red_add4(float4* p, float x, float y, float z, float w) {
  asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};"
               ::"l"(p), "f"(x), "f"(y), "f"(z), "f"(w)
               : "memory");
}
__device__ __forceinline__ void add_grad4(const BackArgs& B, int j, const float acc[15], float scale) {
  float4* p = B.acc + 4 * (int64_t)j;
  red_add4(p, scale * acc[0], scale * acc[1], scale * acc[2], scale * acc[3]);
  red_add4(p + 1, scale * acc[4], scale * acc[5], scale * acc[6], scale * acc[7]);
  red_add4(p + 2, scale * acc[8], scale * acc[9], scale * acc[10], scale * acc[11]);
  red_add4(p + 3, scale * acc[12], scale * acc[13], scale * acc[14], 0.f);
}

// straight to the caller's gradient of original primitive i
__device__ __forceinline__ void add_grad(const BackArgs& B, int64_t i, const float acc[15], float scale) {
  const int64_t N = B.n;
  float* g = B.grad;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    atomicAdd(g + 3 * i + k, scale * acc[k]);
    atomicAdd(g + 7 * N + 3 * i + k, scale * acc[7 + k]);
    atomicAdd(g + 10 * N + 3 * i + k, scale * acc[10 + k]);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) atomicAdd(g + 3 * N + 4 * i + k, scale * acc[3 + k]);
  atomicAdd(g + 13 * N + i, scale * acc[13]);
  atomicAdd(g + 14 * N + i, scale * acc[14]);
}

// ---------------------------------------------------------------------------
// Adjoint of the tomography image: one camera ray per warp.
//
// d tau / d theta needs the five moments of the chord's envelope (PrimDeriv) and
// the two chord ends; the first of them, A C0, is the chord's part of tau.  So one
// traversal gives both: chords are queued, so that 32 at a time are integrated, one per
// lane (about half of the leaves reached have none), their moments kept (24 bytes) and
// their integrals added to tau; then the warp goes through the kept chords, 32 at a
// time, and scatters dL/dtau times their gradients.  A ray with more chords than
// kTomoChords is traversed again with its tau known.  Bound by instruction issue.
// With a pixel per lane, 15 derivatives formed at every quadrature node and two
// traversals, forward and adjoint of 524,288 rays through 200k kernels took 882 ms, 51
// now (20.5 and 28).
// ---------------------------------------------------------------------------
constexpr int kBackBlock = 128;
constexpr int kTomoBlocks = 4;     // resident blocks per SM
constexpr int kTomoChords = 1024;  // kept chords per warp (global scratch)
struct TomoChord {
  float C0, C1, C2, S0, S1;
  int j;
};
static_assert(sizeof(TomoChord) == 24, "kept chords of 24 bytes");

// a chord to integrate
struct TomoItem {
  float mid, hl, y2, y1, y0, B, delta, absA;
  int j;
  int rule;  // node count | table offset << 8
};
constexpr int kTomoQ = 64;  // queued chords per warp (<= 31 left + 32 new)
struct TomoQ {
  CoopTrav t;
  float f[8][kTomoQ];
  int j[kTomoQ], rule[kTomoQ];
};
__device__ __forceinline__ TomoItem tomo_item(const Chord& ch, int j) {
  const float len = ch.dtout - ch.dtin;
  int n, off;
  gl_pick(gl_rule(sqrtf(ch.a) * len + 0.5f * fabsf(ch.B) * len), n, off);
  return TomoItem{0.5f * (ch.dtin + ch.dtout), 0.5f * len, -0.5f * kLog2e * ch.a, -kLog2e * ch.b,
                  -0.5f * kLog2e * ch.g, ch.B, ch.delta, ch.absA, j, n | off << 8};
}

// moments of a chord's envelope in t - tc, and its terms of tau into (s, c)
__device__ __forceinline__ TomoChord tomo_moments(const TomoItem& q, const float* glx,
                                                  const float* glw, float& s_acc, float& c_acc,
                                                  Counters& cnt) {
  const int n = q.rule & 0xFF, off = q.rule >> 8;
  cnt.evals += 2 * n;
  const float scale = q.absA * q.hl;
  TomoChord m{0.f, 0.f, 0.f, 0.f, 0.f, q.j};
  for (int k = off; k < off + n; ++k) {
    const float dt = fmaf(q.hl, glx[k], q.mid),
                e = glw[k] * ex2f(fmaf(fmaf(q.y2, dt, q.y1), dt, q.y0));
    float sn, cs;
    sincosf(fmaf(q.B, dt, q.delta), &sn, &cs);
    const float ec = e * cs, es = e * sn, ect = ec * dt;
    neumaier_add(s_acc, c_acc, scale * ec);
    m.C0 += ec;
    m.C1 += ect;
    m.C2 = fmaf(ect, dt, m.C2);
    m.S0 += es;
    m.S1 = fmaf(es, dt, m.S1);
  }
  m.C0 *= q.hl;
  m.C1 *= q.hl;
  m.C2 *= q.hl;
  m.S0 *= q.hl;
  m.S1 *= q.hl;
  return m;
}

// dL/dtau times the gradient of one chord's integral
template <bool SCRATCH>
__device__ __forceinline__ void tomo_scatter(const BackArgs& B, const Prim& P, const Chord& ch,
                                             const TomoChord& m, float3 v, int j, float dLdtau) {
  PrimDeriv D;
  if (SCRATCH) D.load(B, P.A, P.om, j);
  else D.load(B, P.A, P.om, adj_prim(B, P.orig, P.A));
  PrimDeriv::Moments M = D.moments(ch.p, v, m.C0, m.C1, m.C2, m.S0, m.S1);
  // chord ends that lie on the ellipsoid (not on t = 0)
#pragma unroll 1
  for (int e = ch.dts - ch.hw > 0.f - ch.tc ? 0 : 1; e < 2; ++e)
    D.end(ch, v, e ? ch.dtout : ch.dtin, e ? 1.f : -1.f, M);
  float acc[15];
  D.grad(ch.p, v, M, acc);
  if (SCRATCH) add_grad4(B, j, acc, dLdtau);
  else add_grad(B, P.orig, acc, dLdtau);
}

// SCRATCH: with the arrays per primitive and kept chords (store); without, every ray is
// traversed twice
template <bool SCRATCH>
__global__ void __launch_bounds__(kBackBlock, kTomoBlocks)
    k_tomo_backward(const __grid_constant__ DevField F, const PathParams P, const BackArgs Bk,
                    const float* dLdI, int* counter, int chunk, TomoChord* store) {
  __shared__ BlockTables sm;
  __shared__ TomoQ qs[kBackBlock / 32];
  init_tables(sm, F);
  const uint32_t lane = threadIdx.x & 31u;
  TomoQ& Q = qs[threadIdx.x >> 5];
  store += ((size_t)blockIdx.x * (kBackBlock / 32) + (threadIdx.x >> 5)) * kTomoChords;
  Counters cnt;
  const uint32_t nchunk = (uint32_t)((P.spp + chunk - 1) / chunk);
  const uint32_t units = (uint32_t)(P.roi_w * P.roi_h) * nchunk;
  for (;;) {
    const uint32_t u = next_tile(counter, lane);
    if (u >= units) break;
    const int pix = roi_pixel(P, u / nchunk);
    const float gI = dLdI[pix];
    if (gI == 0.f) continue;
    const int sa = P.s0 + (int)(u % nchunk) * chunk, sb = min(sa + chunk, P.s0 + P.spp);
    for (int s = sa; s < sb; ++s) {
      float3 o, v;
      camera_ray(P.cam, P.seed, pix % P.cam.W, pix / P.cam.W, s, o, v);
      if (lane == 0) cnt.rays += 1;
      const float3 inv = safe_inv(v);
      float t0, t1;
      if (!scene_span(F, o, inv, 0.f, INFINITY, t0, t1)) continue;
      if (lane == 0) cnt.windows += 1;
      float s_acc = 0.f, c_acc = 0.f;
      int nch = 0, nq = 0;  // integrated and queued chords
      auto integrate = [&](int tk) {
        const bool have = (int)lane < tk;
        const int at = nq - tk + (int)lane;
        TomoItem q{};
        if (have)
          q = TomoItem{Q.f[0][at], Q.f[1][at], Q.f[2][at], Q.f[3][at], Q.f[4][at],
                       Q.f[5][at], Q.f[6][at], Q.f[7][at], Q.j[at],    Q.rule[at]};
        __syncwarp();
        nq -= tk;
        if (have) {
          ++cnt.chords;
          const TomoChord m = tomo_moments(q, sm.glx, sm.glw, s_acc, c_acc, cnt);
          if (SCRATCH && nch + (int)lane < kTomoChords) store[nch + (int)lane] = m;
        }
        nch += tk;
      };
      coop_traverse(F, Q.t, F.occupied, o, inv, t0, t1, lane, cnt, [&](int j) {
        Chord ch;
        // the support radius is a constant of the differentiation (adaptive extents too)
        bool ok = false;
        if (j >= 0) {
          const Prim Pr = load_prim(F, j);
          ok = chord_setup(Pr, o, v, 0.f, INFINITY, Pr.k2, ch);
        }
        const unsigned b = __ballot_sync(kFull, ok);
        if (ok) {
          const TomoItem q = tomo_item(ch, j);
          const int at = nq + __popc(b & ((1u << lane) - 1u));
          Q.f[0][at] = q.mid;
          Q.f[1][at] = q.hl;
          Q.f[2][at] = q.y2;
          Q.f[3][at] = q.y1;
          Q.f[4][at] = q.y0;
          Q.f[5][at] = q.B;
          Q.f[6][at] = q.delta;
          Q.f[7][at] = q.absA;
          Q.j[at] = q.j;
          Q.rule[at] = q.rule;
        }
        nq += __popc(b);
        __syncwarp();
        if (nq >= 32) integrate(32);
      });
      if (nq > 0) integrate(nq);
      warp_sum_pair(s_acc, c_acc);
      const float dLdtau = -gI * expf(-__fadd_rn(s_acc, c_acc)) / (float)P.spp;
      __syncwarp();  // the kept chords are read by other lanes
      if (SCRATCH && nch <= kTomoChords) {
        for (int k = (int)lane; k < nch; k += 32) {
          const TomoChord m = store[k];
          const Prim Pr = load_prim(F, m.j);
          Chord ch;
          if (chord_setup(Pr, o, v, 0.f, INFINITY, Pr.k2, ch)) tomo_scatter<SCRATCH>(Bk, Pr, ch, m, v, m.j, dLdtau);
        }
      } else {
        coop_traverse(F, Q.t, F.occupied, o, inv, t0, t1, lane, cnt, [&](int j) {
          if (j < 0) return;
          const Prim Pr = load_prim(F, j);
          Chord ch;
          if (!chord_setup(Pr, o, v, 0.f, INFINITY, Pr.k2, ch)) return;
          float s2 = 0.f, c2 = 0.f;
          const TomoChord m = tomo_moments(tomo_item(ch, j), sm.glx, sm.glw, s2, c2, cnt);
          tomo_scatter<SCRATCH>(Bk, Pr, ch, m, v, j, dLdtau);
        });
      }
      __syncwarp();  // before the next ray's chords overwrite the store
    }
  }
  flush_counters(F, cnt, lane);
}

// ---------------------------------------------------------------------------
// Adjoint of the single-scattering radiance.
//
// Per camera sample, the expected-value form of delta tracking over all
// tentative points t_j of the camera ray (Poisson process of rate kappa_bar):
//   I = sum_j W_j G(t_j),   W_j = prod_{i<j} (1 - p_i) p_j,   p = kappa+/kappa_bar,
// has the mean of the delta-tracking estimator (Sec. 3, Eq. 4 majorants; the
// points before t form a Poisson process independent of the point at t).  One
// point js is drawn with probability W_j / sum W by weighted reservoir
// sampling in t order (point j replaces the candidate when u_j S_j < W_j, u_j
// its own second uniform, S_j the running sum), and G(t_js) = albedo E/(4 pi)
// T_light comes from ratio tracking of the NEE ray, so a sample is S G.  The
// derivative holds the points, kappa_bar and the draw probabilities fixed:
//   d/d p_i = S G / (1 - p_i) * (-1)  (i < js),   S G / p_js  (i = js),
//   d/d q_k = -S albedo E/(4 pi) T_light / (1 - q_k)   (NEE points),
// and d p / d theta = 1[kappa > 0] d kappa/d theta / kappa_bar, where
// d kappa/d theta sums the mask-weighted derivatives of the kernels covering
// the point.
// ---------------------------------------------------------------------------

// ---------------------------------------------------------------------------
// Adjoint of the multiple-scattering radiance (max_bounces >= 2).
//
// The delta-tracking path: segment b accepts its first tentative point js_b
// (probability P_b = prod_{i<js} (1 - p_i) p_js) or escapes; the collision
// x_{b+1} adds C_b = thr_b E0 T_b with thr_b = albedo^(b+1), E0 = E/(4 pi) and
// T_b the ratio-tracked NEE product prod_k (1 - q_k).  C_b depends on the
// segments 0..b and on NEE b, so with the points and majorants held fixed
//   d E[L] = E[ sum_b S_b d log P_b + sum_b C_b d log T_b ],  S_b = sum_{b'>=b} C_b',
//   d log P_b = sum_{i<js} -dp_i / (1 - p_i) + dp_js / p_js,
//   C_b d log T_b = -thr_b E0 sum_k dq_k T_b / (1 - q_k),
// dp = 1[kappa > 0] d kappa / kappa_bar.  The path is followed once (the
// renderer's streams and decisions).  NEE points are scattered as soon as T_b is
// known.  A segment's coefficients are linear in S_b, which only the end of the path
// gives: the segment keeps the moments of its chords at S = 1 (32 bytes each), which
// are scattered at the end; a path with more than kRadKeep of them is followed a
// second time with its S_b known.
// ---------------------------------------------------------------------------

// ---------------------------------------------------------------------------
// The radiance adjoints run one path per warp.  Bound by instruction issue and the
// latency of tree nodes.  With one pixel per lane 1.8 of 32 lanes ran, every window
// visited its ray's list three times and paths were followed twice.  Through 200k
// kernels: 305 -> 6.3 ms (128x128, 2 samples, single scattering), 697 -> 2.9 ms (96x64,
// 1 sample, 3 bounces).
//
// A ray is processed over a window of t, at first all of it:
//  gather   the warp traverses the binary tree together; chords go to the warp's list
//           in global scratch, their tentative points to shared memory;
//  sort     the points by t;
//  sums     kappa and kappa_bar of two points at a time: the chords covering a point
//           are collected, their terms computed one per lane and put in the order of a
//           depth-first walk that visits near children first, in which one lane adds
//           them up (FP32).  Decisions therefore do not depend on how the work was
//           shared out: they are those of a single thread walking the tree;
//  scatter  chords covering a point with a coefficient, one per lane: five moments,
//           then the gradient.
// Warps change between these phases every few rounds, so code size counts: 3.5 of 12.3
// cycles per issued instruction were waits for instructions.  Loops are not unrolled, the
// points of a group share one copy of the code, and a gradient takes only the offset of
// its chord (rad_grad) instead of setting it up: 0.3 of 10.1, 8.4 -> 6.8 and 3.6 -> 3.4 ms.
// The order of the walk is a 64-bit key per chord: bit 63 - d is set when the path to
// its leaf takes the second child at depth d.
// A window with more chords or points than the buffers hold is halved; one that cannot
// be halved is worked through eight points at a time by one lane that walks the tree.
// ---------------------------------------------------------------------------
constexpr int kMaxSeg = 15;
constexpr int kRadBlocks = 4;     // resident blocks per SM
constexpr int kRadStack = 256;
constexpr int kRadMargin = 64;    // a descent adds <= 1 entry per level, 64 levels
constexpr int kRadLeafQ = 96;     // <= 31 left + 64 new
// (The buffers are kept small: beside 28 KB of them per warp's block the L1 holds the
// tree's upper nodes.  With 384 stack entries, 128 points and groups of 4 the blocks
// took 215 KB of an SM: 9.7 and 4.4 ms for the cases above, 8.3 and 3.5 with these.)
constexpr int kRadPts = 64;       // tentative points of a window
constexpr int kRadList = 4096;    // chords of a window at most (global scratch; rad_list_cap)
constexpr int kRadKeep = 4096;    // kept segment moments of a path (global scratch)
constexpr int kRadGroup = 2;      // points whose sums are formed together
constexpr int kRadTerms = 128;    // covering chords of a group, 64 per point
static_assert(kStack <= 64, "a key bit per tree level");
static_assert(kPts <= kRadPts && kRadList <= 1 << 16, "point ids");

struct RadKept {  // moments of a segment's chord at S = 1, mask weight included
  float C0, C1, C2, S0, S1;
  int j, seg;
  float tc;
};
static_assert(sizeof(RadKept) == 32, "kept moments of 32 bytes");
// one warp's chords of a window
struct RadList {
  unsigned long long* key;  // order of the depth-first walk
  float2* span;             // entry and exit
  float4* rec;              // 3 per chord: (tc, y2, y1, y0), (h, B, delta, sqrt a),
                            // (peak - tc, exponent at tc without the amplitude, mask
                            // weight, sorted primitive as bits)
};
// a field of fewer kernels needs no longer lists
__host__ __device__ __forceinline__ int rad_list_cap(int64_t n) {
  return (int)(n < kRadList ? (n + 63) / 64 * 64 : kRadList);
}
__host__ __device__ __forceinline__ size_t rad_list_bytes(int cap) { return (size_t)cap * (8 + 8 + 48); }
__host__ __device__ __forceinline__ size_t rad_warp_bytes(int cap) {
  return 2 * rad_list_bytes(cap) + (size_t)kRadKeep * sizeof(RadKept);
}

struct RadTravQ {
  unsigned long long skey[kRadStack];
  unsigned long long lkey[kRadLeafQ];
  int stk[kRadStack];  // node | depth << 26
  int lq[kRadLeafQ];
};
struct RadEvalQ {
  float4 term[kRadTerms];  // envelope, cos, h, majorant factor
  unsigned long long key[kRadTerms];
  int idx[kRadTerms];
};
// tentative points of a window in t order; c: acceptance uniform, then coefficient
struct RadPts {
  float t[kRadPts], c[kRadPts], kap[kRadPts], kb[kRadPts];
};
struct RadRay {  // the ray in work
  Mask M;
  float3 o, v, inv;
  float ta, tb, t1;    // window [ta, tb), or [ta, t1] when tb >= t1
  uint32_t ray, word;
  int nch, npts;       // chords and points of the window
  int c8;              // points since the last multiple of kPts on the ray
  int listed;          // 0: more chords or points than the buffers hold
};
struct RadQ {
  union {
    RadTravQ t;
    RadEvalQ e;
  };
  RadPts pts[2];
  uint32_t id[kRadPts];  // of an unsorted point: chord << 16 | its number on the chord
  RadRay ray;
  float3 so[kMaxSeg], sv[kMaxSeg];  // the path's segments
  float S[kMaxSeg];
};
// what a warp carries through a path
struct RadWarp {
  const DevField& F;
  const PathParams& P;
  const BackArgs& B;
  RadQ& Q;
  unsigned char* scratch;
  const float* env;
  uint32_t lane;
  int cap;      // chords per list
  int nkept;    // kept moments (may exceed kRadKeep)
  bool replay;  // some segment could not be kept
  Counters cnt;
  __device__ __forceinline__ RadList list(int which) const {
    unsigned char* p = scratch + (size_t)which * rad_list_bytes(cap);
    RadList L;
    L.key = reinterpret_cast<unsigned long long*>(p);
    L.span = reinterpret_cast<float2*>(p + (size_t)cap * 8);
    L.rec = reinterpret_cast<float4*>(p + (size_t)cap * 16);
    return L;
  }
  __device__ __forceinline__ RadKept* kept() const {
    return reinterpret_cast<RadKept*>(scratch + 2 * rad_list_bytes(cap));
  }
};

// Chords and tentative points of the window.  The points land unsorted in kap (t),
// kb (acceptance uniform) and id.
__device__ __noinline__ void rad_gather(RadWarp& W, int which) {
  RadQ& Q = W.Q;
  const DevField& F = W.F;
  const uint32_t lane = W.lane;
  const unsigned lt = (1u << lane) - 1u;
  const RadList L = W.list(which);
  RadPts& Pt = Q.pts[which];
  const float3 o = Q.ray.o, v = Q.ray.v, inv = Q.ray.inv;
  const float ta = Q.ray.ta, t1 = Q.ray.t1;
  const bool last = Q.ray.tb >= t1;
  const float tb = last ? t1 : Q.ray.tb;
  const unsigned long long mask = Q.ray.M.bits;
  const SpanTest test{ta, tb};
  const uint32_t ray = Q.ray.ray, word = Q.ray.word;
  const uint64_t seed = W.P.seed;
  unsigned nodes = 0, leaves = 0;
  int nch = 0;
  int sp = F.root >= 0 ? 1 : 0, lq_n = F.root >= 0 ? 0 : 1;
  __syncwarp();
  if (lane == 0) {
    Q.ray.npts = 0;
    if (F.root >= 0) {
      Q.t.stk[0] = F.root;
      Q.t.skey[0] = 0ull;
    } else {  // a one-primitive field has no internal node
      Q.t.lq[0] = 0;
      Q.t.lkey[0] = 0ull;
    }
  }
  __syncwarp();
  const long long max_it = F.n + 64;  // every node enters the stack at most once
  for (long long it = 0;; ++it) {
    if (it > max_it) {
      if (lane == 0) set_err(F, ERR_GUARD);
      break;
    }
    int take = sp < 32 ? sp : 32;
    // near capacity fewer, down to one: a node leaves room for one more entry
    take = min(take, max(1, kRadStack - kRadMargin - sp));
    const bool have = (int)lane < take;
    const int ent = have ? Q.t.stk[sp - take + (int)lane] : 0;
    const unsigned long long key = have ? Q.t.skey[sp - take + (int)lane] : 0ull;
    __syncwarp();
    sp -= take;
    int c[2] = {0, 0};
    bool h[2] = {false, false};
    unsigned long long kk[2] = {key, key};
    const int node = ent & (int)kOrigMask, depth = (int)((unsigned)ent >> 26);
    if (have && (int64_t)node >= F.n - 1) {  // internal nodes 0 .. n-2
      set_err(F, ERR_INDEX);
    } else if (have) {
      const Node* N = F.nodes + node;
      const float4 a = __ldg(&N->a), b = __ldg(&N->b), cc = __ldg(&N->c);
      const int4 d = __ldg(&N->d);
      const uint4 e = __ldg(&N->e);
      ++nodes;
      const unsigned long long m0 = (unsigned long long)e.x | ((unsigned long long)e.y << 32);
      const unsigned long long m1 = (unsigned long long)e.z | ((unsigned long long)e.w << 32);
      float tn0, tf0, tn1, tf1;
      slab_interval(o, inv, a.x, a.y, a.z, a.w, b.x, b.y, tn0, tf0);
      slab_interval(o, inv, b.z, b.w, cc.x, cc.y, cc.z, cc.w, tn1, tf1);
      c[0] = d.x;
      c[1] = d.y;
      h[0] = (m0 & mask) && test(tn0, tf0);
      h[1] = (m1 & mask) && test(tn1, tf1);
      // leaves come before internal nodes, then the nearer internal child
      if (h[0] && h[1]) {
        const bool first0 = c[0] < 0 || (c[1] >= 0 && tn0 <= tn1);
        kk[first0 ? 1 : 0] |= 1ull << (63 - depth);
      }
    }
    int np = 0, nl = 0;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const unsigned bp = __ballot_sync(kFull, h[k] && c[k] >= 0);
      const unsigned bl = __ballot_sync(kFull, h[k] && c[k] < 0);
      if (h[k] && c[k] >= 0) {
        const int pos = sp + np + __popc(bp & lt);
        if (pos < kRadStack) {
          Q.t.stk[pos] = c[k] | (int)((unsigned)(depth + 1) << 26);
          Q.t.skey[pos] = kk[k];
        }
      }
      if (h[k] && c[k] < 0) {
        const int pos = lq_n + nl + __popc(bl & lt);
        Q.t.lq[pos] = ~c[k];
        Q.t.lkey[pos] = kk[k];
      }
      np += __popc(bp);
      nl += __popc(bl);
    }
    if (sp + np > kRadStack) {
      if (lane == 0) set_err(F, ERR_STACK);
      np = kRadStack - sp;
    }
    sp += np;
    lq_n += nl;
    __syncwarp();
    const bool more = sp > 0;
    while (lq_n >= 32 || (!more && lq_n > 0)) {
      const int tk = lq_n < 32 ? lq_n : 32;
      int j = -1;
      unsigned long long lk = 0ull;
      if ((int)lane < tk) {
        j = Q.t.lq[lq_n - tk + (int)lane];
        lk = Q.t.lkey[lq_n - tk + (int)lane];
      }
      __syncwarp();
      lq_n -= tk;
      if (j >= 0) ++leaves;
      if ((int64_t)j >= F.n) {  // a leaf beyond the records
        set_err(F, ERR_INDEX);
        j = -1;
      }
      Chord ch;
      float w;
      const bool ok = j >= 0 &&
                      prim_chord(F, j, o, v, 0.f, INFINITY,
                                 [&](uint32_t cl) { return mask_weight(Q.ray.M, cl); }, w, ch) &&
                      ch.tc + ch.dtin <= tb && ch.tc + ch.dtout >= ta;
      const unsigned bc = __ballot_sync(kFull, ok);
      const int k = nch + __popc(bc & lt);
      if (ok && k < W.cap) {
        const float wa = w * ch.absA;
        const float y2 = -0.5f * kLog2e * ch.a, y1 = -kLog2e * ch.b;
        const float y0 = fmaf(-0.5f * kLog2e, ch.g, log2f(wa));
        const float hh = wa * expf(-0.5f * ch.qmin);
        const float sa = sqrtf(ch.a);
        L.span[k] = make_float2(ch.tc + ch.dtin, ch.tc + ch.dtout);
        L.key[k] = lk;
        L.rec[3 * k] = make_float4(ch.tc, y2, y1, y0);
        L.rec[3 * k + 1] = make_float4(hh, ch.B, ch.delta, sa);
        L.rec[3 * k + 2] = make_float4(ch.dts, -0.5f * kLog2e * ch.g, w, __int_as_float(j));
        uint32_t num = 0;
        chord_points(F, ch, hh, seed, ray, word, W.env, [&](float t, float u) {
          if (t > t1 || (!last && t >= tb)) return false;
          if (t >= ta) {
            const int q = atomicAdd(&Q.ray.npts, 1);
            if (q >= kRadPts) return false;  // too many: the window is halved
            Pt.kap[q] = t;
            Pt.kb[q] = u;
            Q.id[q] = (uint32_t)k << 16 | num;
          }
          ++num;
          return true;
        });
      }
      nch += __popc(bc);
      __syncwarp();
    }
    if (!more && lq_n == 0) break;
  }
  if (lane == 0) Q.ray.nch = nch;
  W.cnt.nodes += nodes;
  W.cnt.leaves += leaves;
  __syncwarp();
}

// The window's points in t order (equal t: in the order of the walk), in t and c.  The
// ray's points go in runs of kPts, and a point at the t at which a run ended is left
// out, as in track().
__device__ __noinline__ void rad_sort(RadWarp& W, int which) {
  RadQ& Q = W.Q;
  RadPts& Pt = Q.pts[which];
  const unsigned long long* keys = W.list(which).key;
  const int n = Q.ray.npts;
  bool tie = false;
  for (int i = (int)W.lane; i < n; i += 32) {
    const float t = Pt.kap[i];
    int rank = 0;
#pragma unroll 1
    for (int k = 0; k < n; ++k) {
      const float tk = Pt.kap[k];
      bool before = tk < t;
      if (tk == t && k != i) {
        const uint32_t a = Q.id[k], b = Q.id[i];
        before = (a >> 16) == (b >> 16) ? a < b : keys[a >> 16] < keys[b >> 16];
        tie = true;
      }
      rank += before ? 1 : 0;
    }
    Pt.t[rank] = t;
    Pt.c[rank] = Pt.kb[i];
  }
  tie = __any_sync(kFull, tie);
  __syncwarp();
  if (W.lane == 0) {
    if (!tie) {
      Q.ray.c8 = (Q.ray.c8 + n) % kPts;
    } else {
      int m = 0, c8 = Q.ray.c8;
      float end = -INFINITY;
      for (int i = 0; i < n; ++i) {
        const float t = Pt.t[i];
        if (t == end) continue;
        Pt.t[m] = t;
        Pt.c[m] = Pt.c[i];
        ++m;
        if (++c8 == kPts) {
          c8 = 0;
          end = t;
        }
      }
      Q.ray.c8 = c8;
      Q.ray.npts = m;
    }
  }
  __syncwarp();
}

// kappa and kappa_bar at `n` points from g on (n = kRadGroup or 1); false when a point
// is covered by more chords than its share of the buffers
__device__ __noinline__ bool rad_sums(RadWarp& W, int which, int g, int n) {
  RadQ& Q = W.Q;
  RadPts& Pt = Q.pts[which];
  const RadList L = W.list(which);
  const uint32_t lane = W.lane;
  const unsigned lt = (1u << lane) - 1u;
  const int nch = Q.ray.nch, cap = kRadTerms / n;
  n = min(n, Q.ray.npts - g);
  __syncwarp();
  float tp[kRadGroup];
  int c[kRadGroup];
#pragma unroll
  for (int p = 0; p < kRadGroup; ++p) {
    tp[p] = p < n ? Pt.t[g + p] : INFINITY;
    c[p] = 0;
  }
#pragma unroll 1
  for (int b = 0; b < nch; b += 32) {
    const int k = b + (int)lane;
    const float2 s = k < nch ? L.span[k] : make_float2(INFINITY, -INFINITY);
#pragma unroll
    for (int p = 0; p < kRadGroup; ++p) {
      const bool in = p < n && tp[p] >= s.x && tp[p] <= s.y;
      const unsigned m = __ballot_sync(kFull, in);
      const int pos = c[p] + __popc(m & lt);
      if (in && pos < cap) Q.e.idx[p * cap + pos] = k;
      c[p] += __popc(m);
    }
  }
#pragma unroll
  for (int p = 0; p < kRadGroup; ++p)
    if (c[p] > cap) return false;
  __syncwarp();
#pragma unroll 1
  for (int p = 0; p < kRadGroup; ++p) {
    const int base = p * cap;
    int cp = c[0];
    float t = tp[0];
#pragma unroll
    for (int q = 1; q < kRadGroup; ++q) {
      cp = p == q ? c[q] : cp;
      t = p == q ? tp[q] : t;
    }
#pragma unroll 1
    for (int i = (int)lane; i < cp; i += 32) Q.e.key[base + i] = L.key[Q.e.idx[base + i]];
    __syncwarp();
#pragma unroll 1
    for (int i = (int)lane; i < cp; i += 32) {
      const unsigned long long key = Q.e.key[base + i];
      const float4* r = L.rec + 3 * Q.e.idx[base + i];
      const float4 a = r[0], b = r[1];
      const float dts = r[2].x;
      int rank = 0;
      for (int k = 0; k < cp; ++k) rank += Q.e.key[base + k] < key ? 1 : 0;
      const float dt = t - a.x;
      const float y = fmaf(fmaf(a.y, dt, a.z), dt, a.w);
      int m = (int)(fabsf(dt - dts) * b.w);
      m = m > 7 ? 7 : m;
      Q.e.term[base + rank] = make_float4(ex2f(y), cosf_fast(fmaf(b.y, dt, b.z)), b.x, W.env[m]);
    }
    W.cnt.evals += (int)lane < cp ? (unsigned)(cp - (int)lane + 31) >> 5 : 0u;
  }
  __syncwarp();
  if ((int)lane < n) {
    int cl = c[0];
#pragma unroll
    for (int p = 1; p < kRadGroup; ++p) cl = (int)lane == p ? c[p] : cl;
    const float4* T = Q.e.term + (int)lane * cap;
    float kap = 0.f, kb = 0.f;
    for (int i = 0; i < cl; ++i) {
      const float4 x = T[i];
      kap = fmaf(x.x, x.y, kap);
      kb = fmaf(x.z, x.w, kb);
    }
    Pt.kap[g + (int)lane] = kap;
    Pt.kb[g + (int)lane] = kb;
  }
  __syncwarp();
  return true;
}

// kappa and kappa_bar at points 0 .. n-1 (n <= kPts) by one lane that walks the tree
__device__ __noinline__ void rad_sums_walk(RadWarp& W, int which, int g, int n) {
  RadQ& Q = W.Q;
  RadPts& Pt = Q.pts[which];
  __syncwarp();
  if (W.lane == 0) {
    PointBuf B;
    AccumLeaf al;
#pragma unroll
    for (int i = 0; i < kPts; ++i) {
      B.t[i] = i < n ? Pt.t[g + i] : INFINITY;
      al.kap[i] = 0.f;
      al.kb[i] = 0.f;
    }
    al.F = &W.F;
    al.M = &Q.ray.M;
    al.o = Q.ray.o;
    al.v = Q.ray.v;
    al.tmin = 0.f;
    al.tmax = INFINITY;
    al.B = &B;
    al.n = n;
    al.env = W.env;
    PointTest pt{&B, n};
    traverse_ray(W.F, Q.ray.o, Q.ray.inv, Q.ray.M.bits, pt, al, W.cnt.nodes, W.cnt.leaves);
#pragma unroll
    for (int i = 0; i < kPts; ++i)
      if (i < n) {
        Pt.kap[g + i] = al.kap[i];
        Pt.kb[g + i] = al.kb[i];
      }
    W.cnt.evals += al.nev;
  }
  __syncwarp();
}

// the next kPts points from ta on by one lane that walks the tree, with their sums
__device__ __noinline__ void rad_collect_walk(RadWarp& W, int which) {
  RadQ& Q = W.Q;
  RadPts& Pt = Q.pts[which];
  __syncwarp();
  if (W.lane == 0) {
    PointBuf B;
#pragma unroll
    for (int i = 0; i < kPts; ++i) {
      B.t[i] = INFINITY;
      B.u[i] = 0.f;
    }
    CollectLeaf cl;
    cl.F = &W.F;
    cl.M = &Q.ray.M;
    cl.o = Q.ray.o;
    cl.v = Q.ray.v;
    cl.tmin = 0.f;
    cl.tmax = INFINITY;
    cl.ta = Q.ray.ta;
    cl.first = true;
    cl.bound = Q.ray.t1;
    cl.B = &B;
    cl.seed = W.P.seed;
    cl.ray = Q.ray.ray;
    cl.word = Q.ray.word;
    cl.env = W.env;
    CollectTest ct{&cl.ta, &cl.bound};
    traverse_ray(W.F, Q.ray.o, Q.ray.inv, Q.ray.M.bits, ct, cl, W.cnt.nodes, W.cnt.leaves);
    int n = 0;
#pragma unroll
    for (int i = 0; i < kPts; ++i)
      if (B.t[i] < INFINITY) {
        Pt.t[i] = B.t[i];
        Pt.c[i] = B.u[i];
        ++n;
      }
    Q.ray.npts = n;
    // the next window begins beyond the last point; fewer points: the ray is over
    Q.ray.tb = n < kPts ? Q.ray.t1 : nextafterf(B.t[kPts - 1], INFINITY);
    Q.ray.listed = 0;
  }
  __syncwarp();
  rad_sums_walk(W, which, 0, Q.ray.npts);
}

// start of a ray: false when it misses every kernel
__device__ __forceinline__ bool rad_begin(RadWarp& W, const Mask& M, float3 o, float3 v, uint32_t ray,
                                          uint32_t word) {
  const float3 inv = safe_inv(v);
  float t0, t1;
  if (M.bits == 0ull || !scene_span(W.F, o, inv, 0.f, INFINITY, t0, t1)) return false;
  __syncwarp();
  if (W.lane == 0) {
    RadRay& R = W.Q.ray;
    R.M = M;
    R.o = o;
    R.v = v;
    R.inv = inv;
    R.ta = t0;
    R.tb = t1;
    R.t1 = t1;
    R.ray = ray;
    R.word = word;
    R.c8 = 0;
  }
  __syncwarp();
  return true;
}

// the window from ta on: its points, sorted; returns their number
__device__ __noinline__ int rad_window(RadWarp& W, int which) {
  RadQ& Q = W.Q;
  for (int it = 0; it < 64; ++it) {
    rad_gather(W, which);
    if (Q.ray.nch <= W.cap && Q.ray.npts <= kRadPts) {
      if (W.lane == 0) Q.ray.listed = 1;
      rad_sort(W, which);
      return Q.ray.npts;
    }
    const float ta = Q.ray.ta, w = fminf(Q.ray.tb, Q.ray.t1) - ta;
    if (w <= 1e-6f * (1.0f + fabsf(ta))) break;
    __syncwarp();
    if (W.lane == 0) Q.ray.tb = ta + 0.5f * w;
    __syncwarp();
  }
  rad_collect_walk(W, which);
  return Q.ray.npts;
}

// on to the next window; false at the end of the ray
__device__ __forceinline__ bool rad_advance(RadWarp& W) {
  RadRay& R = W.Q.ray;
  const float ta = R.ta, tb = R.tb, t1 = R.t1;
  if (tb >= t1) return false;
  __syncwarp();
  if (W.lane == 0) {
    R.ta = tb;
    R.tb = R.listed ? fminf(t1, tb + 2.0f * (tb - ta)) : t1;
  }
  __syncwarp();
  return true;
}

// kappa and kappa_bar at the points of the group from g on
__device__ __forceinline__ void rad_group(RadWarp& W, int which, int g) {
  if (!W.Q.ray.listed) return;  // formed when the points were collected
  if (rad_sums(W, which, g, kRadGroup)) return;
  const int e = min(g + kRadGroup, W.Q.ray.npts);
  for (int i = g; i < e; ++i)
    if (!rad_sums(W, which, i, 1)) rad_sums_walk(W, which, i, 1);
}

// One kernel's gradient from the points with a coefficient, by a lane on its own
struct RadScatterLeaf {
  const RadWarp* W;
  const RadPts* Pt;
  int n;
  float scale;
  __device__ void operator()(int j) {
    const RadRay& R = W->Q.ray;
    const Prim Pr = load_prim(W->F, j);
    Chord ch;
    const float w = mask_weight(R.M, Pr.cell);
    if (w == 0.f || !chord_setup(Pr, R.o, R.v, 0.f, INFINITY, Pr.k2, ch)) return;
    const float tin = ch.tc + ch.dtin, tout = ch.tc + ch.dtout;
    float C0 = 0.f, C1 = 0.f, C2 = 0.f, S0 = 0.f, S1 = 0.f;
    bool any = false;
    for (int i = 0; i < n; ++i) {
      const float t = Pt->t[i], c = Pt->c[i];
      if (c == 0.f || t < tin || t > tout) continue;
      any = true;
      const float dt = t - ch.tc;
      const float e = c * ex2f(-0.5f * kLog2e * fmaf(fmaf(ch.a, dt, 2.f * ch.b), dt, ch.g));
      float sn, cs;
      sincosf(fmaf(ch.B, dt, ch.delta), &sn, &cs);
      C0 += e * cs;
      C1 = fmaf(e * cs, dt, C1);
      C2 = fmaf(e * cs * dt, dt, C2);
      S0 += e * sn;
      S1 = fmaf(e * sn, dt, S1);
    }
    if (!any) return;
    PrimDeriv D;
    D.load(W->B, Pr.A, Pr.om, j);
    float acc[15];
    D.grad(ch.p, R.v, D.moments(ch.p, R.v, C0, C1, C2, S0, S1), acc);
    add_grad4(W->B, j, acc, w * scale);
  }
};

// the gradient of sorted primitive j from the moments of its chord around tc, times
// scale.  The offset at tc is all that it needs of the chord.
__device__ __forceinline__ void rad_grad(const RadWarp& W, int j, float3 o, float3 v, float tc,
                                         float C0, float C1, float C2, float S0, float S1,
                                         float scale) {
  const float4* r = W.F.rec + 4 * (int64_t)j;
  const float4 mu = __ldg(r), om = __ldg(r + 3);
  PrimDeriv D;
  D.load(W.B, mu.w, make_float3(om.x, om.y, om.z), j);
  const float3 p = chord_offset(make_float3(mu.x, mu.y, mu.z), o, v, tc);
  float acc[15];
  D.grad(p, v, D.moments(p, v, C0, C1, C2, S0, S1), acc);
  add_grad4(W.B, j, acc, scale);
}

// gradients of the chords covering points 0 .. n-1 with a coefficient (c), times scale;
// seg >= 0: the moments are kept for the end of the path instead
__device__ __noinline__ void rad_scatter(RadWarp& W, int which, int n, int seg, float scale) {
  RadQ& Q = W.Q;
  RadPts& Pt = Q.pts[which];
  const RadList L = W.list(which);
  const uint32_t lane = W.lane;
  const unsigned lt = (1u << lane) - 1u;
  const int nch = Q.ray.nch;
  if (n <= 0) return;
  __syncwarp();
  if (!Q.ray.listed) {
    if (seg >= 0) {
      W.replay = true;  // scattered when the path is followed again
    } else if (lane == 0) {
      const RadScatterLeaf leaf_c{&W, &Pt, n, scale};
      RadScatterLeaf leaf = leaf_c;
      SpanTest test{Q.ray.ta, fminf(Q.ray.tb, Q.ray.t1)};
      traverse_ray(W.F, Q.ray.o, Q.ray.inv, Q.ray.M.bits, test, leaf, W.cnt.nodes, W.cnt.leaves);
    }
    __syncwarp();
    return;
  }
  int m = 0;  // collected chords
  for (int b = 0; b < nch || m > 0; b += 32) {
    if (b < nch) {
      const int k = b + (int)lane;
      const float2 s = k < nch ? L.span[k] : make_float2(INFINITY, -INFINITY);
      bool in = false;
#pragma unroll 1
      for (int i = 0; i < n; ++i) in |= Pt.c[i] != 0.f && Pt.t[i] >= s.x && Pt.t[i] <= s.y;
      const unsigned bm = __ballot_sync(kFull, in);
      if (in) Q.e.idx[m + __popc(bm & lt)] = k;
      m += __popc(bm);
      __syncwarp();
      if (m < 32 && b + 32 < nch) continue;
    }
    // 32 collected chords (or the last ones)
    const int tk = m < 32 ? m : 32;
    const bool have = (int)lane < tk;
    const int k = have ? Q.e.idx[m - tk + (int)lane] : 0;
    __syncwarp();
    m -= tk;
    const int slot = W.nkept + (int)lane;
    if (have) {
      const float2 s = L.span[k];
      const float4 a = L.rec[3 * k], r1 = L.rec[3 * k + 1], r2 = L.rec[3 * k + 2];
      const int j = __float_as_int(r2.w);
      float C0 = 0.f, C1 = 0.f, C2 = 0.f, S0 = 0.f, S1 = 0.f;
#pragma unroll 1
      for (int i = 0; i < n; ++i) {
        const float t = Pt.t[i], c = Pt.c[i];
        if (c == 0.f || t < s.x || t > s.y) continue;
        const float dt = t - a.x;
        const float e = c * ex2f(fmaf(fmaf(a.y, dt, a.z), dt, r2.y));
        float sn, cs;
        sincosf(fmaf(r1.y, dt, r1.z), &sn, &cs);
        C0 += e * cs;
        C1 = fmaf(e * cs, dt, C1);
        C2 = fmaf(e * cs * dt, dt, C2);
        S0 += e * sn;
        S1 = fmaf(e * sn, dt, S1);
      }
      const float w = r2.z;
      if (seg >= 0) {
        if (slot < kRadKeep) {
          float4* d = reinterpret_cast<float4*>(W.kept() + slot);
          d[0] = make_float4(w * C0, w * C1, w * C2, w * S0);
          d[1] = make_float4(w * S1, __int_as_float(j), __int_as_float(seg), a.x);
        }
      } else {
        rad_grad(W, j, Q.ray.o, Q.ray.v, a.x, C0, C1, C2, S0, S1, w * scale);
      }
    }
    if (seg >= 0) {
      W.nkept += tk;
      if (W.nkept > kRadKeep) W.replay = true;
    }
  }
  __syncwarp();
}

// NEE ray from x: returns T = prod (1 - q_k); windows receives their number.  With one
// window its points stay in pts[which] for nee_scatter.
__device__ __noinline__ float nee_track(RadWarp& W, int which, float3 x, uint32_t pix, uint32_t s,
                                           int b, int& windows) {
  const PathParams& P = W.P;
  const Mask M = sample_mask(W.F, P.lod_nee, P.light, P.seed, pix, s, (uint32_t)b, TAG_NEE_MASK);
  float T = 1.f;
  windows = 0;
  if (!rad_begin(W, M, x, P.light, pix, stream_word(s, (uint32_t)b, TAG_NEE))) return T;
  const RadPts& Pt = W.Q.pts[which];
  do {
    const int n = rad_window(W, which);
    ++windows;
    for (int g = 0; g < n; g += kRadGroup) {
      rad_group(W, which, g);
      for (int i = g; i < min(g + kRadGroup, n); ++i)
        if (Pt.kb[i] > 0.f) T *= 1.f - fmaxf(Pt.kap[i], 0.f) / Pt.kb[i];
    }
  } while (rad_advance(W));
  return T;
}
// coefficients cn / (1 - q_k) / kappa_bar_k of the ray's NEE points, scattered
__device__ __noinline__ void nee_scatter(RadWarp& W, int which, float3 x, uint32_t pix, uint32_t s,
                                            int b, int windows, float cn) {
  const PathParams& P = W.P;
  if (windows == 0 || cn == 0.f) return;
  RadPts& Pt = W.Q.pts[which];
  if (windows > 1) {  // the windows again, each scattered in turn
    const Mask M = sample_mask(W.F, P.lod_nee, P.light, P.seed, pix, s, (uint32_t)b, TAG_NEE_MASK);
    (void)rad_begin(W, M, x, P.light, pix, stream_word(s, (uint32_t)b, TAG_NEE));
  }
  do {
    const int n = windows > 1 ? rad_window(W, which) : W.Q.ray.npts;
    if (windows > 1)
      for (int g = 0; g < n; g += kRadGroup) rad_group(W, which, g);
    __syncwarp();
#pragma unroll 1
    for (int i = (int)W.lane; i < n; i += 32) {
      const float kap = Pt.kap[i], kb = Pt.kb[i];
      float c = 0.f;
      if (kap > 0.f && kb > 0.f) {
        const float q = kap / kb;
        if (1.f - q > 0.f) c = cn / (1.f - q) / kb;
      }
      Pt.c[i] = c;
    }
    rad_scatter(W, which, n, -1, 1.f);
  } while (windows > 1 && rad_advance(W));
}

// One segment of the path from (o, v): delta tracking to the first accepted point
// (returns false on escape, else its t).  Coefficients at S = 1, -1/(1 - p) before the
// accepted point and 1/p at it, are kept for segment b (scale == 0) or scattered with
// scale.
__device__ __noinline__ bool path_segment(RadWarp& W, float3 o, float3 v, uint32_t pix, uint32_t s,
                                             int b, float scale, float& th) {
  const PathParams& P = W.P;
  const Mask M = sample_mask(W.F, P.lod, v, P.seed, pix, s, (uint32_t)b, TAG_MASK);
  if (!rad_begin(W, M, o, v, pix, stream_word(s, (uint32_t)b, TAG_TRACK))) return false;
  RadPts& Pt = W.Q.pts[0];
  const int kept0 = W.nkept;
  const bool replay0 = W.replay;
  do {
    const int n = rad_window(W, 0);
    int acc = -1;
    for (int g = 0; g < n && acc < 0; g += kRadGroup) {
      rad_group(W, 0, g);
      for (int i = g; i < min(g + kRadGroup, n) && acc < 0; ++i) {
        const float kap = Pt.kap[i], kb = Pt.kb[i], u = Pt.c[i];
        const bool take = u * kb < fmaxf(kap, 0.f);
        float c = 0.f;
        if (kap > 0.f && kb > 0.f) {
          const float p = kap / kb;
          c = (take ? 1.f / p : -1.f / (1.f - p)) / kb;
        }
        __syncwarp();
        if (W.lane == 0) Pt.c[i] = c;
        if (take) acc = i;
      }
    }
    rad_scatter(W, 0, acc >= 0 ? acc + 1 : n, scale == 0.f ? b : -1, scale);
    if (acc >= 0) {
      th = Pt.t[acc];
      return true;
    }
  } while (rad_advance(W));
  W.nkept = kept0;  // an escaping segment has no coefficients
  W.replay = replay0;
  return false;
}

__device__ __forceinline__ float3 path_scatter_dir(const PathParams& P, uint32_t pix, uint32_t s,
                                                   int b) {
  const uint4 y = rng4(P.seed, 0, kNoPrim, pix, stream_word(s, (uint32_t)b, TAG_SCATTER));
  const float z = 1.0f - 2.0f * u01(y.x);
  const float rr = sqrtf(fmaxf(0.0f, 1.0f - z * z));
  float sn, cs;
  sincosf(2.0f * 3.14159265358979f * u01(y.y), &sn, &cs);
  return make_float3(rr * cs, rr * sn, z);
}

// multiple scattering: the path of sample s of pixel pix
__device__ __forceinline__ void path_backward(RadWarp& W, float3 o, float3 v, uint32_t pix, uint32_t s,
                                              float base) {
  const PathParams& P = W.P;
  RadQ& Q = W.Q;
  const float E0 = P.irradiance * (0.25f / 3.14159265358979f);
  W.nkept = 0;
  W.replay = false;
  int nseg = 0;
  float thr = 1.f, Ssuf = 0.f;
  for (int b = 0; b < P.max_bounces && b < kMaxSeg; ++b) {
    float th = 0.f;
    if (W.lane == 0) {
      W.cnt.rays += 1;
      Q.so[b] = o;
      Q.sv[b] = v;
    }
    if (!path_segment(W, o, v, pix, s, b, 0.f, th)) break;
    const float3 x = make_float3(fmaf(th, v.x, o.x), fmaf(th, v.y, o.y), fmaf(th, v.z, o.z));
    if (W.lane == 0) W.cnt.rays += 1;
    int windows = 0;
    const float T = nee_track(W, 0, x, pix, s, b, windows);
    thr *= P.albedo;
    const float Cb = thr * E0 * T;
    if (T > 0.f) nee_scatter(W, 0, x, pix, s, b, windows, -base * Cb);
    if (W.lane == 0) Q.S[b] = Cb;
    Ssuf += Cb;
    ++nseg;
    o = x;
    v = path_scatter_dir(P, pix, s, b);
  }
  if (nseg == 0) return;
  // S_b = sum_{b' >= b} C_b'
  __syncwarp();
  if (W.lane == 0) {
    for (int b = 0; b < nseg; ++b) {
      const float Cb = Q.S[b];
      Q.S[b] = Ssuf;
      Ssuf -= Cb;
    }
  }
  __syncwarp();
  if (W.replay) {
    // too many chords to keep: the segments again, with their S_b known
    for (int b = 0; b < nseg; ++b) {
      const float S = base * Q.S[b];
      float th = 0.f;
      if (S == 0.f) continue;
      if (!path_segment(W, Q.so[b], Q.sv[b], pix, s, b, S, th)) break;
    }
    return;
  }
  for (int e = (int)W.lane; e < W.nkept; e += 32) {
    const float4* d = reinterpret_cast<const float4*>(W.kept() + e);
    const float4 a = d[0], c = d[1];
    const int j = __float_as_int(c.y), seg = __float_as_int(c.z);
    const float S = base * Q.S[seg];
    if (S == 0.f) continue;
    const float3 so = Q.so[seg], sv = Q.sv[seg];
    rad_grad(W, j, so, sv, c.w, a.x, a.y, a.z, a.w, c.x, S);
  }
  __syncwarp();
}

// single scattering: the expected-value estimator of sample s of pixel pix
__device__ __forceinline__ void single_backward(RadWarp& W, float3 o, float3 v, uint32_t pix,
                                                uint32_t s, float base) {
  const PathParams& P = W.P;
  RadPts& Pt = W.Q.pts[0];
  const float E = P.albedo * P.irradiance * (0.25f / 3.14159265358979f);
  if (W.lane == 0) W.cnt.rays += 1;
  const Mask M = sample_mask(W.F, P.lod, v, P.seed, pix, s, 0, TAG_MASK);
  const uint32_t wt = stream_word(s, 0, TAG_TRACK);
  if (!rad_begin(W, M, o, v, pix, wt)) return;
  // weights, their sum and the reservoir draw
  float Pr = 1.f, S = 0.f, pjs = 0.f, tjs = 0.f;
  int idx = 0, js = -1, windows = 0;
  do {
    const int n = rad_window(W, 0);
    ++windows;
    for (int g = 0; g < n; g += kRadGroup) {
      rad_group(W, 0, g);
      for (int i = g; i < min(g + kRadGroup, n); ++i) {
        const float kap = Pt.kap[i], kb = Pt.kb[i];
        const float p = kb > 0.f ? fmaxf(kap, 0.f) / kb : 0.f;
        const float Wt = Pr * p;
        S += Wt;
        if (Wt > 0.f && Pt.c[i] * S < Wt) {
          js = idx + i;
          pjs = p;
          tjs = Pt.t[i];
        }
        Pr *= 1.f - p;
      }
    }
    idx += n;
  } while (rad_advance(W));
  if (js < 0 || !(S > 0.f)) return;
  // the camera ray in work, for its scatter after the NEE ray's
  const int nch = W.Q.ray.nch, npts = W.Q.ray.npts, listed = W.Q.ray.listed;
  // NEE from the drawn point by ratio tracking, T = prod (1 - kappa+/kappa_bar)
  const float3 x = make_float3(fmaf(tjs, v.x, o.x), fmaf(tjs, v.y, o.y), fmaf(tjs, v.z, o.z));
  if (W.lane == 0) W.cnt.rays += 1;
  int nwin = 0;
  const float Tl = nee_track(W, 1, x, pix, s, 0, nwin);
  const float G = E * Tl;
  if (Tl > 0.f) nee_scatter(W, 1, x, pix, s, 0, nwin, -base * S * E * Tl);
  // camera points 0 .. js
  (void)rad_begin(W, M, o, v, pix, wt);
  idx = 0;
  do {
    int n;
    if (windows > 1) {
      n = rad_window(W, 0);
      for (int g = 0; g < n; g += kRadGroup) rad_group(W, 0, g);
    } else {
      n = npts;
      if (W.lane == 0) {
        W.Q.ray.nch = nch;
        W.Q.ray.npts = npts;
        W.Q.ray.listed = listed;
      }
    }
    __syncwarp();
    const int m = min(n, js + 1 - idx);
    for (int i = (int)W.lane; i < m; i += 32) {
      const float kap = Pt.kap[i], kb = Pt.kb[i];
      float c = 0.f;
      if (kap > 0.f && kb > 0.f) {
        const float p = kap / kb;
        c = base * (idx + i == js ? S * G / pjs : -S * G / (1.f - p)) / kb;
      }
      Pt.c[i] = c;
    }
    rad_scatter(W, 0, m, -1, 1.f);
    idx += n;
  } while (windows > 1 && idx <= js && rad_advance(W));
}

// PATH = false: single scattering; PATH = true: multiple scattering
template <bool PATH>
__global__ void __launch_bounds__(kBackBlock, kRadBlocks)
    k_radiance_backward(const __grid_constant__ DevField F, const __grid_constant__ PathParams P,
                        const __grid_constant__ BackArgs Bk, const float* dLdI, int* counter,
                        int chunk, unsigned char* scratch) {
  extern __shared__ __align__(16) unsigned char smraw[];
  float* env = reinterpret_cast<float*>(smraw);
  if (threadIdx.x < 8) env[threadIdx.x] = F.env[threadIdx.x];
  __syncthreads();
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  RadWarp W{F, P, Bk, reinterpret_cast<RadQ*>(smraw + 32)[warp],
            scratch + ((size_t)blockIdx.x * (kBackBlock / 32) + warp) * rad_warp_bytes(rad_list_cap(F.n)),
            env, lane, rad_list_cap(F.n), 0, false, Counters()};
  const uint32_t nchunk = (uint32_t)((P.spp + chunk - 1) / chunk);
  const uint32_t units = (uint32_t)(P.roi_w * P.roi_h) * nchunk;
  for (;;) {
    const uint32_t u = next_tile(counter, lane);
    if (u >= units) break;
    const uint32_t pix = (uint32_t)roi_pixel(P, u / nchunk);
    const float gI = dLdI[pix];
    if (gI == 0.f) continue;
    const float base = gI / (float)P.spp;
    const int sa = P.s0 + (int)(u % nchunk) * chunk, sb = min(sa + chunk, P.s0 + P.spp);
    for (int s = sa; s < sb; ++s) {
      float3 o, v;
      camera_ray(P.cam, P.seed, (int)pix % P.cam.W, (int)pix / P.cam.W, s, o, v);
      if constexpr (PATH)
        path_backward(W, o, v, pix, (uint32_t)s, base);
      else
        single_backward(W, o, v, pix, (uint32_t)s, base);
    }
  }
  flush_counters(F, W.cnt, lane);
}

static BackArgs back_args(const Field& F, float* grad) {
  BackArgs B{};
  B.quat = F.p_quat;
  B.ls = F.p_ls;
  B.om = F.p_om;
  B.w = F.p_w;
  B.frame = F.opts.omega_frame;
  B.wmode = F.opts.weight_mode;
  B.n = F.n;
  B.grad = grad;
  return B;
}

static_assert(sizeof(RadQ) % 16 == 0, "aligned per-warp shared memory");
constexpr size_t kRadSmem = 32 + sizeof(RadQ) * (kBackBlock / 32);
static_assert((kRadSmem + 1024) * kRadBlocks <= 233472, "kRadBlocks blocks fit one SM's shared memory");

// blocks of a full persistent grid; the kernel's local frame must fit the context's
// stack limit as it stands
template <class K>
static cudaError_t adjoint_grid(const Field& F, K kernel, size_t smem, int64_t& g) {
  cudaError_t e;
  if (smem && (e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)smem)) != cudaSuccess)
    return e;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kBackBlock, smem) != cudaSuccess)
    (void)cudaGetLastError();
  if (per_sm < 1) per_sm = 1;
  g = (int64_t)F.ctx.sm_count * per_sm;
  return cudaSuccess;
}
template <class K>
static cudaError_t adjoint_stack_fits(K kernel) {
  cudaFuncAttributes fa;
  size_t limit = 0;
  cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
  if (e == cudaSuccess) e = cudaDeviceGetLimit(&limit, cudaLimitStackSize);
  if (e == cudaSuccess && fa.localSizeBytes > limit) e = cudaErrorLaunchOutOfResources;
  return e;
}

// scratch of an adjoint kernel of a full persistent grid of g blocks: the kept chords
// (tomography), or the chord lists and kept moments (radiance), in one buffer
static size_t tomo_scratch(int64_t g) {
  return (size_t)g * (kBackBlock / 32) * kTomoChords * sizeof(TomoChord);
}
static size_t rad_scratch(const Field& F, int64_t g) {
  return (size_t)g * (kBackBlock / 32) * rad_warp_bytes(rad_list_cap(F.n));
}
// the arrays per primitive and `bytes` of scratch for a grid of g blocks, through the
// field's allocator; g comes back smaller when less scratch is to be had
static cudaError_t grow_adjoint(const Field& F, size_t bytes, int64_t& g, cudaStream_t s) {
  const cudaError_t e = grow(F, (void**)&F.adj, F.adj_bytes, (size_t)F.n * 7 * sizeof(float4), s);
  return e != cudaSuccess ? e : grow_shares(F, F.rlist, bytes / g, g, s);
}

// the scratch of every adjoint
cudaError_t ensure_adjoint_lists(const Field& F, cudaStream_t s) {
  int64_t g = 1;
  size_t bytes = 0;
  cudaError_t e;
  if ((e = adjoint_grid(F, k_tomo_backward<true>, 0, g)) != cudaSuccess) return e;
  bytes = tomo_scratch(g);
  if ((e = adjoint_grid(F, k_radiance_backward<false>, kRadSmem, g)) != cudaSuccess) return e;
  bytes = std::max(bytes, rad_scratch(F, g));
  if ((e = adjoint_grid(F, k_radiance_backward<true>, kRadSmem, g)) != cudaSuccess) return e;
  bytes = std::max(bytes, rad_scratch(F, g));
  return grow_adjoint(F, (bytes + g - 1) / g * g, g, s);
}

// An adjoint kernel over units of `chunk` samples of a pixel (about 16 per warp of the
// grid at least), between the per-primitive inputs and the copy of the sums to grad; bare: a
// kernel that goes without scratch, where it is not to be had (null: the call fails)
template <class T>
using AdjointKernel = void (*)(DevField, PathParams, BackArgs, const float*, int*, int, T*);
template <class T>
static cudaError_t launch_adjoint(const Field& F, const PathParams& P, AdjointKernel<T> kernel,
                                  AdjointKernel<T> bare, size_t smem, const float* dLdI, float* grad,
                                  cudaStream_t s) {
  (void)cudaGetLastError();  // a stale error of an unrelated call is not ours
  cudaError_t e = cudaMemsetAsync(F.counter, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  BackArgs B = back_args(F, grad);
  int64_t g = 1;
  if ((e = adjoint_stack_fits(kernel)) != cudaSuccess) return e;
  if ((e = adjoint_grid(F, kernel, smem, g)) != cudaSuccess) return e;
  // (allocated ahead by gf_reserve, else here)
  bool scratch = true;
  if (bare && (!F.adj || !F.rlist.p)) scratch = !capturing(s);
  if (scratch) {
    const int64_t full = g;
    if ((e = grow_adjoint(F, smem ? rad_scratch(F, g) : tomo_scratch(g), g, s)) != cudaSuccess) {
      if (!bare || e != cudaErrorMemoryAllocation) return e;
      (void)cudaGetLastError();
      scratch = false;
    } else if (bare && 2 * g < full) {
      // lists for few blocks: a full grid without them is faster (131,072 rays through 200k
      // kernels: 7.1 ms with all, 11.3 with half, 20.2 with a quarter of them, 15.2 without)
      scratch = false;
    }
  }
  if (!scratch) {
    kernel = bare;
    if ((e = adjoint_stack_fits(kernel)) != cudaSuccess) return e;
    if ((e = adjoint_grid(F, kernel, smem, g)) != cudaSuccess) return e;
  }
  // (pixels whose rays all miss the scene have no part in the gradient)
  const int64_t npix = std::max<int64_t>(1, (int64_t)P.roi_w * P.roi_h), warps = g * (kBackBlock / 32);
  int64_t nchunk = (16 * warps + npix - 1) / npix;
  nchunk = nchunk < 1 ? 1 : (nchunk > P.spp ? P.spp : nchunk);
  const int64_t chunk = (P.spp + nchunk - 1) / nchunk;
  const int64_t units = npix * ((P.spp + chunk - 1) / chunk);
  g = std::min(g, (units + kBackBlock / 32 - 1) / (kBackBlock / 32));
  const unsigned pb = (unsigned)((F.n + 255) / 256);
  if (scratch) {
    B.adj = F.adj;
    B.acc = F.adj + 3 * F.n;
    if ((e = cudaMemsetAsync(B.acc, 0, (size_t)F.n * 4 * sizeof(float4), s)) != cudaSuccess) return e;
    k_adj_prims<<<pb, 256, 0, s>>>(F.dev.rec, B, F.adj);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  } else if ((e = cudaMemsetAsync(grad, 0, (size_t)F.n * 15 * sizeof(float), s)) != cudaSuccess) {
    return e;
  }
  kernel<<<(unsigned)g, kBackBlock, smem, s>>>(F.dev, P, B, dLdI, F.counter, (int)chunk,
                                              scratch ? static_cast<T*>(F.rlist.p) : nullptr);
  if (scratch && (e = cudaGetLastError()) == cudaSuccess) k_adj_finish<<<pb, 256, 0, s>>>(F.dev.rec, B);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_tomo_backward(const Field& F, const PathParams& P, const float* dLdI,
                                 float* grad, cudaStream_t s) {
  return launch_adjoint<TomoChord>(F, P, k_tomo_backward<true>, k_tomo_backward<false>, 0, dLdI, grad, s);
}

cudaError_t launch_radiance_backward(const Field& F, const PathParams& P, const float* dLdI,
                                     float* grad, cudaStream_t s) {
  return launch_adjoint<unsigned char>(
      F, P, P.max_bounces >= 2 ? k_radiance_backward<true> : k_radiance_backward<false>, nullptr, kRadSmem,
      dLdI, grad, s);
}

}  // namespace gf
