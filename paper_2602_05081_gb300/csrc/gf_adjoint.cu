// gf_adjoint.cu -- hand-written adjoint of the tomography renderer.
//
// Image I_p = (1/spp) sum_s exp(-tau_s) (Sec. 4.6 tomography), tau_s the
// optical depth of Eq. 2-3 along the jittered camera ray.  Given dL/dI:
//   dL/dtheta_i = sum_{p,s} dL/dI_p (-exp(-tau_s)/spp) dtau_s/dtheta_i,
//   dtau/dtheta = int_chord d(integrand)/dtheta dt
//               + g(t_out) dt_out/dtheta - g(t_in) dt_in/dtheta,
// with the ellipsoid ends moving as dt/dtheta = -(dq/dtheta)/(dq/dt)
// (Leibniz rule for the k-sigma-truncated kernel).  Each ray is traversed
// twice (forward optical depth, then the adjoint pass): nothing is stored
// per path.  Gradients are accumulated with atomics in SoA layout.
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
  const float4* adj;  // per primitive (BVH order): what PrimDeriv::load needs, 3 float4
  float4* acc;        // gradient sums per primitive (BVH order), 4 float4 each
};

// Derivatives of one kernel g = A exp(-q/2) cos(theta) with respect to its 15
// raw parameters (mu 3, quaternion 4 through qhat = q/|q|, log scale 3, omega 3
// in the input frame, phase, weight), at offsets y = x - mu.
struct PrimDeriv {
  float R[3][3];
  float qh[4], iqn;    // unit quaternion (w, x, y, z) and 1/|q| of the raw one
  float s[3], is2[3], kin[3];
  float A, dAdw;
  float3 om;
  float phi;
  bool local, normalized;

  __device__ void init(const BackArgs& B, const Prim& P, int64_t i) {
    float q[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) q[k] = B.quat[4 * i + k];
    const float qn = sqrtf(q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
    iqn = 1.f / qn;
#pragma unroll
    for (int k = 0; k < 4; ++k) qh[k] = q[k] * iqn;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      s[k] = expf(B.ls[3 * i + k]);
      kin[k] = B.om[3 * i + k];
    }
    dAdw = B.wmode == GF_WEIGHT_NORMALIZED ? P.A / B.w[i] : 1.f;
    derive(B, P);
  }

  // as init, from the parameters k_adj_prims gathered for sorted primitive j
  __device__ __forceinline__ void load(const BackArgs& B, const Prim& P, int j) {
    const float4* r = B.adj + 3 * (int64_t)j;
    const float4 a = __ldg(r), b = __ldg(r + 1), c = __ldg(r + 2);
    qh[0] = a.x; qh[1] = a.y; qh[2] = a.z; qh[3] = a.w;
    s[0] = b.x; s[1] = b.y; s[2] = b.z;
    iqn = b.w;
    kin[0] = c.x; kin[1] = c.y; kin[2] = c.z;
    dAdw = c.w;
    derive(B, P);
  }

  __device__ __forceinline__ void derive(const BackArgs& B, const Prim& P) {
    const float qw = qh[0], qx = qh[1], qy = qh[2], qz = qh[3];
    R[0][0] = 1.f - 2.f * (qy * qy + qz * qz); R[0][1] = 2.f * (qx * qy - qw * qz);
    R[0][2] = 2.f * (qx * qz + qw * qy);
    R[1][0] = 2.f * (qx * qy + qw * qz); R[1][1] = 1.f - 2.f * (qx * qx + qz * qz);
    R[1][2] = 2.f * (qy * qz - qw * qx);
    R[2][0] = 2.f * (qx * qz - qw * qy); R[2][1] = 2.f * (qy * qz + qw * qx);
    R[2][2] = 1.f - 2.f * (qx * qx + qy * qy);
#pragma unroll
    for (int k = 0; k < 3; ++k) is2[k] = 1.f / (s[k] * s[k]);
    local = B.frame == GF_OMEGA_LOCAL;
    normalized = B.wmode == GF_WEIGHT_NORMALIZED;
    A = P.A;
    om = P.om;
    phi = P.phi;
  }

  // dz/dq of the raw quaternion at offset y (linear in y): dz/d(qhat_l) =
  // (dR/d qhat_l)^T y, written out from R(qhat); then through qhat = q/|q|:
  // dz/dq_m = (g_m - qhat_m sum_l qhat_l g_l) / |q|
  __device__ __forceinline__ void dz_dq(const float y[3], float g[4][3]) const {
    const float w = qh[0], x = qh[1], yq = qh[2], zq = qh[3];
    const float y0 = y[0], y1 = y[1], y2 = y[2];
    g[0][0] = 2.f * (zq * y1 - yq * y2);
    g[0][1] = 2.f * (-zq * y0 + x * y2);
    g[0][2] = 2.f * (yq * y0 - x * y1);
    g[1][0] = 2.f * (yq * y1 + zq * y2);
    g[1][1] = 2.f * (yq * y0 - 2.f * x * y1 + w * y2);
    g[1][2] = 2.f * (zq * y0 - w * y1 - 2.f * x * y2);
    g[2][0] = 2.f * (-2.f * yq * y0 + x * y1 - w * y2);
    g[2][1] = 2.f * (x * y0 + zq * y2);
    g[2][2] = 2.f * (w * y0 + zq * y1 - 2.f * yq * y2);
    g[3][0] = 2.f * (-2.f * zq * y0 + w * y1 + x * y2);
    g[3][1] = 2.f * (-w * y0 - 2.f * zq * y1 + yq * y2);
    g[3][2] = 2.f * (x * y0 + yq * y1);
    float sg[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) sg[k] = w * g[0][k] + x * g[1][k] + yq * g[2][k] + zq * g[3][k];
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
      for (int k = 0; k < 3; ++k) g[m][k] = (g[m][k] - qh[m] * sg[k]) * iqn;
  }

  // Sums over positions y = p + t v of weight times dg/dparam, from the moments of
  // the envelope: C_k of e cos(theta) t^k and S_k of e sin(theta) t^k (e the weighted
  // envelope without the amplitude, theta the phase with the sign of the amplitude
  // folded in).  q is quadratic and theta linear in t, so every derivative is a
  // combination of five moments.
  __device__ __forceinline__ void from_moments(float3 pp, float3 vv, float C0, float C1, float C2,
                                               float S0, float S1, float acc[15]) const {
    const float p[3] = {pp.x, pp.y, pp.z}, v[3] = {vv.x, vv.y, vv.z};
    const float aA = fabsf(A), sgn = A < 0.f ? -1.f : 1.f;
    float zp[3], zv[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      zp[k] = R[0][k] * p[0] + R[1][k] * p[1] + R[2][k] * p[2];
      zv[k] = R[0][k] * v[0] + R[1][k] * v[1] + R[2][k] * v[2];
    }
    const float omv[3] = {om.x, om.y, om.z};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float up = R[a][0] * zp[0] * is2[0] + R[a][1] * zp[1] * is2[1] + R[a][2] * zp[2] * is2[2];
      const float uv = R[a][0] * zv[0] * is2[0] + R[a][1] * zv[1] * is2[1] + R[a][2] * zv[2] * is2[2];
      acc[a] = aA * (up * C0 + uv * C1 + omv[a] * S0);
    }
    float gp[4][3], gv[4][3], kos[3];
    dz_dq(p, gp);
    dz_dq(v, gv);
#pragma unroll
    for (int k = 0; k < 3; ++k) kos[k] = local ? kin[k] / s[k] : 0.f;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      float q0 = 0.f, q1 = 0.f, q2 = 0.f, h0 = 0.f, h1 = 0.f;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        q0 += zp[k] * gp[m][k] * is2[k];
        q1 += (zp[k] * gv[m][k] + zv[k] * gp[m][k]) * is2[k];
        q2 += zv[k] * gv[m][k] * is2[k];
        h0 += kos[k] * gp[m][k];
        h1 += kos[k] * gv[m][k];
      }
      acc[3 + m] = -aA * (q0 * C0 + q1 * C1 + q2 * C2 + h0 * S0 + h1 * S1);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float d = (zp[k] * zp[k] * C0 + 2.f * zp[k] * zv[k] * C1 + zv[k] * zv[k] * C2) * is2[k] +
                      kos[k] * (zp[k] * S0 + zv[k] * S1);
      acc[7 + k] = aA * (normalized ? d - C0 : d);
      acc[10 + k] = local ? -aA * (zp[k] * S0 + zv[k] * S1) / s[k] : -aA * (p[k] * S0 + v[k] * S1);
    }
    acc[13] = -aA * S0;
    acc[14] = sgn * dAdw * C0;
  }

  // value g at y; d[15] = dg/dparam; dq[10] = dq/dparam (mu, quaternion, log scale)
  __device__ float at(const float y[3], float d[15], float dq[10]) const {
    float z[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) z[k] = R[0][k] * y[0] + R[1][k] * y[1] + R[2][k] * y[2];
    const float qq = z[0] * z[0] * is2[0] + z[1] * z[1] * is2[1] + z[2] * z[2] * is2[2];
    const float env = expf(-0.5f * qq);
    const float th = om.x * y[0] + om.y * y[1] + om.z * y[2] + phi;
    float sn, cs;
    sincosf(th, &sn, &cs);
    float dth[15], dA[15];
#pragma unroll
    for (int r = 0; r < 15; ++r) {
      dth[r] = 0.f;
      dA[r] = 0.f;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a)
      dq[a] = -2.f * (R[a][0] * z[0] * is2[0] + R[a][1] * z[1] * is2[1] + R[a][2] * z[2] * is2[2]);
    dth[0] = -om.x;
    dth[1] = -om.y;
    dth[2] = -om.z;
    float g[4][3];
    dz_dq(y, g);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      float dqm = 0.f, dthm = 0.f;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        dqm += 2.f * z[k] * g[m][k] * is2[k];
        if (local) dthm += kin[k] / s[k] * g[m][k];
      }
      dq[3 + m] = dqm;
      dth[3 + m] = dthm;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      dq[7 + k] = -2.f * z[k] * z[k] * is2[k];
      if (local) dth[7 + k] = -kin[k] * z[k] / s[k];
      if (normalized) dA[7 + k] = -A;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) dth[10 + k] = local ? z[k] / s[k] : y[k];
    dth[13] = 1.f;
    dA[14] = dAdw;
#pragma unroll
    for (int r = 0; r < 15; ++r) {
      const float dqr = r < 10 ? dq[r] : 0.f;
      d[r] = A * env * (-0.5f * dqr * cs - sn * dth[r]) + dA[r] * env * cs;
    }
    return A * env * cs;
  }
};

__device__ __forceinline__ void add_grad(const BackArgs& B, int64_t i, const float acc[15],
                                         float scale) {
  const int64_t N = B.n;
  float* g = B.grad;
  for (int k = 0; k < 3; ++k) atomicAdd(g + 3 * i + k, scale * acc[k]);
  for (int k = 0; k < 4; ++k) atomicAdd(g + 3 * N + 4 * i + k, scale * acc[3 + k]);
  for (int k = 0; k < 3; ++k) atomicAdd(g + 7 * N + 3 * i + k, scale * acc[7 + k]);
  for (int k = 0; k < 3; ++k) atomicAdd(g + 10 * N + 3 * i + k, scale * acc[10 + k]);
  atomicAdd(g + 13 * N + i, scale * acc[13]);
  atomicAdd(g + 14 * N + i, scale * acc[14]);
}

// what PrimDeriv::load needs, gathered once per call in BVH order (48 bytes per
// primitive instead of 11 scattered words and their arithmetic per chord)
__global__ void k_adj_prims(const float4* rec, const BackArgs B, float4* adj) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= B.n) return;
  const int64_t i = __float_as_uint(rec[4 * j + 3].w) & kOrigMask;
  float q[4];
  for (int k = 0; k < 4; ++k) q[k] = B.quat[4 * i + k];
  const float iqn = 1.f / sqrtf(q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
  const float A = rec[4 * j].w;
  adj[3 * j] = make_float4(q[0] * iqn, q[1] * iqn, q[2] * iqn, q[3] * iqn);
  adj[3 * j + 1] = make_float4(expf(B.ls[3 * i]), expf(B.ls[3 * i + 1]), expf(B.ls[3 * i + 2]), iqn);
  adj[3 * j + 2] = make_float4(B.om[3 * i], B.om[3 * i + 1], B.om[3 * i + 2],
                               B.wmode == GF_WEIGHT_NORMALIZED ? A / B.w[i] : 1.f);
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

// ---------------------------------------------------------------------------
// Adjoint of the tomography image: one camera ray per warp.
//
// d tau / d theta needs the five moments of the chord's envelope (from_moments) and
// the two chord ends; the first of them, A C0, is the chord's part of tau.  So one
// traversal gives both: each lane integrates its own chord, keeps its moments
// (24 bytes) and adds to tau; then the warp goes through the kept chords, 32 at a
// time, and scatters dL/dtau times their gradients.  A ray with more chords than
// kTomoChords is traversed again with its tau known.  Bound by instruction issue.
// Every lane used to carry its own pixel, with 15 derivatives formed at every
// quadrature node and two traversals.
// ---------------------------------------------------------------------------
constexpr int kBackBlock = 128;
constexpr int kTomoBlocks = 4;     // resident blocks per SM
constexpr int kTomoChords = 1024;  // kept chords per warp (global scratch)
struct TomoChord {
  float C0, C1, C2, S0, S1;
  int j;
};
static_assert(sizeof(TomoChord) == 24, "kept chords of 24 bytes");

// moments of a chord's envelope in t - tc, and its terms of tau into (s, c)
__device__ __forceinline__ TomoChord tomo_moments(const Chord& ch, const float* glx,
                                                  const float* glw, float& s_acc, float& c_acc,
                                                  Counters& cnt) {
  const float len = ch.dtout - ch.dtin;
  int n, off;
  gl_pick(gl_rule(sqrtf(ch.a) * len + 0.5f * fabsf(ch.B) * len), n, off);
  cnt.evals += 2 * n;
  const float mid = 0.5f * (ch.dtin + ch.dtout), hl = 0.5f * len;
  const float y2 = -0.5f * kLog2e * ch.a, y1 = -kLog2e * ch.b, y0 = -0.5f * kLog2e * ch.g;
  const float scale = ch.absA * hl;
  TomoChord m{0.f, 0.f, 0.f, 0.f, 0.f, 0};
  for (int k = off; k < off + n; ++k) {
    const float dt = fmaf(hl, glx[k], mid), e = glw[k] * ex2f(fmaf(fmaf(y2, dt, y1), dt, y0));
    float sn, cs;
    sincosf(fmaf(ch.B, dt, ch.delta), &sn, &cs);
    const float ec = e * cs, es = e * sn, ect = ec * dt;
    neumaier_add(s_acc, c_acc, scale * ec);
    m.C0 += ec;
    m.C1 += ect;
    m.C2 = fmaf(ect, dt, m.C2);
    m.S0 += es;
    m.S1 = fmaf(es, dt, m.S1);
  }
  m.C0 *= hl;
  m.C1 *= hl;
  m.C2 *= hl;
  m.S0 *= hl;
  m.S1 *= hl;
  return m;
}

// dL/dtau times the gradient of one chord's integral
__device__ __forceinline__ void tomo_scatter(const BackArgs& B, const Prim& P, const Chord& ch,
                                             const TomoChord& m, float3 v, int j, float dLdtau) {
  PrimDeriv D;
  D.load(B, P, j);
  float acc[15];
  D.from_moments(ch.p, v, m.C0, m.C1, m.C2, m.S0, m.S1, acc);
  // Leibniz terms where a chord end lies on the ellipsoid (not on t = 0): the end
  // moves as dt/dtheta = -(dq/dtheta)/(dq/dt)
  const bool on_in = ch.dts - ch.hw > 0.f - ch.tc;
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    if (e == 0 && !on_in) continue;
    const float dt = e == 0 ? ch.dtin : ch.dtout, sgn = e == 0 ? -1.f : 1.f;
    const float y[3] = {fmaf(dt, v.x, ch.p.x), fmaf(dt, v.y, ch.p.y), fmaf(dt, v.z, ch.p.z)};
    float d[15], dq[10];
    const float g = D.at(y, d, dq);
    const float dqdt = -(v.x * dq[0] + v.y * dq[1] + v.z * dq[2]);
    if (dqdt != 0.f)
      for (int r = 0; r < 10; ++r) acc[r] += sgn * g * (-dq[r] / dqdt);
  }
  add_grad4(B, j, acc, dLdtau);
}

__global__ void __launch_bounds__(kBackBlock, kTomoBlocks)
    k_tomo_backward(const __grid_constant__ DevField F, const PathParams P, const BackArgs Bk,
                    const float* dLdI, int* counter, int chunk, TomoChord* store) {
  __shared__ BlockTables sm;
  __shared__ CoopTrav qs[kBackBlock / 32];
  init_tables(sm, F);
  const uint32_t lane = threadIdx.x & 31u;
  CoopTrav& Q = qs[threadIdx.x >> 5];
  store += ((size_t)blockIdx.x * (kBackBlock / 32) + (threadIdx.x >> 5)) * kTomoChords;
  Counters cnt;
  const uint32_t nchunk = (uint32_t)((P.spp + chunk - 1) / chunk);
  const uint32_t units = (uint32_t)(P.cam.W * P.cam.H) * nchunk;
  for (;;) {
    const uint32_t u = next_tile(counter, lane);
    if (u >= units) break;
    const int pix = (int)(u / nchunk);
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
      int nch = 0;
      coop_traverse(F, Q, F.occupied, o, inv, t0, t1, lane, cnt, [&](int j) {
        Chord ch;
        // the support radius is a constant of the differentiation (adaptive extents too)
        bool ok = false;
        if (j >= 0) {
          const Prim Pr = load_prim(F, j);
          ok = chord_setup(Pr, o, v, 0.f, INFINITY, Pr.k2, ch);
        }
        const unsigned b = __ballot_sync(kFull, ok);
        if (ok) {
          ++cnt.chords;
          TomoChord m = tomo_moments(ch, sm.glx, sm.glw, s_acc, c_acc, cnt);
          m.j = j;
          const int k = nch + __popc(b & ((1u << lane) - 1u));
          if (k < kTomoChords) store[k] = m;
        }
        nch += __popc(b);
      });
      warp_sum_pair(s_acc, c_acc);
      const float dLdtau = -gI * expf(-__fadd_rn(s_acc, c_acc)) / (float)P.spp;
      __syncwarp();  // the kept chords are read by other lanes
      if (nch <= kTomoChords) {
        for (int k = (int)lane; k < nch; k += 32) {
          const TomoChord m = store[k];
          const Prim Pr = load_prim(F, m.j);
          Chord ch;
          if (chord_setup(Pr, o, v, 0.f, INFINITY, Pr.k2, ch)) tomo_scatter(Bk, Pr, ch, m, v, m.j, dLdtau);
        }
      } else {
        coop_traverse(F, Q, F.occupied, o, inv, t0, t1, lane, cnt, [&](int j) {
          if (j < 0) return;
          const Prim Pr = load_prim(F, j);
          Chord ch;
          if (!chord_setup(Pr, o, v, 0.f, INFINITY, Pr.k2, ch)) return;
          float s2 = 0.f, c2 = 0.f;
          const TomoChord m = tomo_moments(ch, sm.glx, sm.glw, s2, c2, cnt);
          tomo_scatter(Bk, Pr, ch, m, v, j, dLdtau);
        });
      }
      __syncwarp();  // before the next ray's chords overwrite the store
    }
  }
  flush_counters(F, cnt, lane);
}

// scratch of the adjoints per primitive: gathered parameters, gradient sums
static cudaError_t ensure_adjoint_prims(const Field& F, cudaStream_t s) {
  return grow(F, (void**)&F.adj, F.adj_bytes, (size_t)F.n * 7 * sizeof(float4), s);
}
static cudaError_t tomo_grid(const Field& F, int64_t& g) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_tomo_backward, kBackBlock, 0) != cudaSuccess)
    (void)cudaGetLastError();
  if (per_sm < 1) per_sm = 1;
  g = (int64_t)F.ctx.sm_count * per_sm;
  return cudaSuccess;
}

// per-primitive inputs gathered and sums cleared, before an adjoint kernel
static cudaError_t adjoint_begin(const Field& F, BackArgs& B, cudaStream_t s) {
  cudaError_t e = ensure_adjoint_prims(F, s);
  if (e != cudaSuccess) return e;
  B.adj = F.adj;
  B.acc = F.adj + 3 * F.n;
  if ((e = cudaMemsetAsync(B.acc, 0, (size_t)F.n * 4 * sizeof(float4), s)) != cudaSuccess) return e;
  k_adj_prims<<<(unsigned)((F.n + 255) / 256), 256, 0, s>>>(F.dev.rec, B, F.adj);
  return cudaGetLastError();
}
static cudaError_t adjoint_end(const Field& F, const BackArgs& B, cudaStream_t s) {
  k_adj_finish<<<(unsigned)((F.n + 255) / 256), 256, 0, s>>>(F.dev.rec, B);
  return cudaGetLastError();
}

// The primitives whose chords cross a ray under its mask, gathered by one
// traversal; the replay passes then visit the list instead of the tree.
constexpr int kRayList = 1024;
struct RayList {
  int* idx;    // this thread's first entry; entry k at idx[k * stride] (a warp's
  int stride;  // lanes hold neighbouring words: coalesced)
  int n;       // listed primitives; > kRayList: overflow, traverse instead
  __device__ bool ok() const { return n <= kRayList; }
  __device__ int at(int k) const { return idx[(int64_t)k * stride]; }
};

struct ListLeaf {
  const DevField* F;
  const Mask* M;
  float3 o, v;
  RayList* L;
  __device__ void operator()(int j) {
    const Mask& Mk = *M;
    Chord ch;
    float w;
    if (!prim_chord(*F, j, o, v, 0.f, INFINITY, [&](uint32_t c) { return mask_weight(Mk, c); }, w, ch))
      return;
    if (L->n < kRayList) L->idx[(int64_t)L->n * L->stride] = j;
    ++L->n;
  }
};

__device__ __forceinline__ void gather_list(const DevField& F, const Mask& M, float3 o, float3 v,
                                            RayList& L, Counters& cnt) {
  L.n = 0;
  const float3 inv = safe_inv(v);
  float t0, t1;
  if (M.bits == 0ull || !scene_span(F, o, inv, 0.f, INFINITY, t0, t1)) return;
  ListLeaf leaf{&F, &M, o, v, &L};
  SpanTest test{t0, t1};
  traverse_ray(F, o, inv, M.bits, test, leaf, cnt.nodes, cnt.leaves);
}

// every primitive of the list, or a traversal with `test` when it overflowed
template <class Test, class Leaf>
__device__ __forceinline__ void visit(const DevField& F, const RayList* L, float3 o, float3 inv,
                                      unsigned long long mask, Test& test, Leaf& leaf,
                                      Counters& cnt) {
  if (L && L->ok()) {
    for (int k = 0; k < L->n; ++k) leaf(L->at(k));
    cnt.leaves += (unsigned long long)L->n;
  } else {
    traverse_ray(F, o, inv, mask, test, leaf, cnt.nodes, cnt.leaves);
  }
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
// the point.  Each ray is re-tracked (same Philox streams, same windows) for
// the derivative passes: nothing per path is stored.
// ---------------------------------------------------------------------------

// Windows of kPts tentative points, in t order, with kappa and kappa_bar
// (the windows of track()); win(B, n, kap, kb) returns false to stop.
template <class Win>
__device__ void for_windows(const DevField& F, const Mask& M, float3 o, float3 v, uint64_t seed,
                            uint32_t ray, uint32_t word, const float* env, Counters& cnt,
                            const RayList* L, Win win) {
  const unsigned am = __activemask();
  const float3 inv = safe_inv(v);
  float t0 = 0.f, t1 = 0.f;
  bool more = M.bits != 0ull && scene_span(F, o, inv, 0.f, INFINITY, t0, t1);
  float ta = t0;
  bool first = true;
  for (int guard = 0; guard < (1 << 16); ++guard) {
    if (!__any_sync(am, more)) break;
    if (!more) continue;
    PointBuf B;
#pragma unroll
    for (int i = 0; i < kPts; ++i) {
      B.t[i] = INFINITY;
      B.u[i] = 0.f;
    }
    CollectLeaf cl;
    cl.F = &F;
    cl.M = &M;
    cl.o = o;
    cl.v = v;
    cl.tmin = 0.f;
    cl.tmax = INFINITY;
    cl.ta = ta;
    cl.first = first;
    cl.bound = t1;
    cl.B = &B;
    cl.seed = seed;
    cl.ray = ray;
    cl.word = word;
    cl.env = env;
    CollectTest ctest{&cl.ta, &cl.bound};
    visit(F, L, o, inv, M.bits, ctest, cl, cnt);
    int n = 0;
#pragma unroll
    for (int i = 0; i < kPts; ++i) n += B.t[i] < INFINITY ? 1 : 0;
    if (n == 0) {
      more = false;
      continue;
    }
    AccumLeaf al;
    al.F = &F;
    al.M = &M;
    al.o = o;
    al.v = v;
    al.tmin = 0.f;
    al.tmax = INFINITY;
    al.B = &B;
    al.n = n;
    al.env = env;
#pragma unroll
    for (int i = 0; i < kPts; ++i) {
      al.kap[i] = 0.f;
      al.kb[i] = 0.f;
    }
    PointTest ptest{&B, n};
    visit(F, L, o, inv, M.bits, ptest, al, cnt);
    cnt.evals += al.nev;
    if (!win(B, n, al.kap, al.kb) || n < kPts) {
      more = false;
      continue;
    }
    ta = B.t[kPts - 1];
    first = false;
  }
}

// coef_i * d kappa(x(t_i)) / d theta, scattered over the kernels at the points
struct RadScatter {
  const DevField* F;
  const BackArgs* B;
  const Mask* M;
  float3 o, v;
  const PointBuf* P;
  const float* coef;
  int n;
  __device__ void operator()(int j) {
    const Prim Pr = load_prim(*F, j);
    Chord ch;
    if (!chord_setup(Pr, o, v, 0.f, INFINITY, Pr.k2, ch)) return;
    const float w = mask_weight(*M, ch.cell);
    if (w == 0.f) return;
    const float tin = ch.tc + ch.dtin, tout = ch.tc + ch.dtout;
    bool any = false;
#pragma unroll
    for (int i = 0; i < kPts; ++i)
      any |= i < n && coef[i] != 0.f && P->t[i] >= tin && P->t[i] <= tout;
    if (!any) return;
    PrimDeriv D;
    D.init(*B, Pr, ch.orig);
    float acc[15];
    for (int r = 0; r < 15; ++r) acc[r] = 0.f;
    for (int i = 0; i < n; ++i) {
      const float t = P->t[i];
      if (coef[i] == 0.f || t < tin || t > tout) continue;
      const float dt = t - ch.tc;
      const float y[3] = {fmaf(dt, v.x, ch.p.x), fmaf(dt, v.y, ch.p.y), fmaf(dt, v.z, ch.p.z)};
      float d[15], dq[10];
      D.at(y, d, dq);
      for (int r = 0; r < 15; ++r) acc[r] = fmaf(coef[i], d[r], acc[r]);
    }
    add_grad(*B, ch.orig, acc, w);
  }
};

__device__ __forceinline__ void scatter_window(const DevField& F, const BackArgs& Bk, const Mask& M,
                                               float3 o, float3 v, const PointBuf& P,
                                               const float* coef, int n, const RayList* L,
                                               Counters& cnt) {
  bool any = false;
#pragma unroll
  for (int i = 0; i < kPts; ++i) any |= i < n && coef[i] != 0.f;
  if (!any) return;
  RadScatter rs{&F, &Bk, &M, o, v, &P, coef, n};
  PointTest ptest{&P, n};
  visit(F, L, o, safe_inv(v), M.bits, ptest, rs, cnt);
}

struct RadSmem {
  float env[8];
};

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
// dp = 1[kappa > 0] d kappa / kappa_bar.  Pass 1 follows the path (the
// renderer's streams and decisions) and keeps only T_b per collision; pass 2
// follows it again, scattering each segment's points up to the accepted one
// and each NEE ray's points with those coefficients.  Nothing per tentative
// point or per segment ray is stored.
// ---------------------------------------------------------------------------
constexpr int kMaxSeg = 15;

// one segment of the path from (o, v): delta tracking to the first accepted
// point (returns false on escape, else t); with coefficients (S != 0), the
// points up to the accepted one are scattered, -S/(1 - p) before it, S/p at it
__device__ __forceinline__ bool path_segment(const DevField& F, const PathParams& P,
                                             const BackArgs& Bk, float3 o, float3 v,
                                             uint32_t pix, uint32_t s, int b, float S,
                                             const float* env, Counters& cnt, RayList& L,
                                             float& th) {
  const Mask M = sample_mask_impl<true>(F, P.lod, v, P.seed, pix, s, (uint32_t)b, TAG_MASK);
  const uint32_t wt = stream_word(s, (uint32_t)b, TAG_TRACK);
  gather_list(F, M, o, v, L, cnt);
  bool hit = false;
  for_windows(F, M, o, v, P.seed, pix, wt, env, cnt, &L,
              [&](const PointBuf& B, int n, const float* kap, const float* kb) {
                float coef[kPts];
                int acc = -1;
#pragma unroll
                for (int i = 0; i < kPts; ++i) {
                  coef[i] = 0.f;
                  if (i < n && acc < 0) {
                    const bool take = B.u[i] * kb[i] < fmaxf(kap[i], 0.f);
                    if (S != 0.f && kap[i] > 0.f && kb[i] > 0.f) {
                      const float p = kap[i] / kb[i];
                      coef[i] = (take ? S / p : -S / (1.f - p)) / kb[i];
                    }
                    if (take) acc = i;
                  }
                }
                if (S != 0.f) scatter_window(F, Bk, M, o, v, B, coef, n, &L, cnt);
                if (acc >= 0) {
                  hit = true;
                  th = B.t[acc];
                  return false;
                }
                return true;
              });
  return hit;
}

// NEE ray of collision b from x: returns T = prod (1 - q_k); with cn != 0 the
// points are scattered with cn / (1 - q_k) / kappa_bar_k
__device__ __forceinline__ float path_nee(const DevField& F, const PathParams& P,
                                          const BackArgs& Bk, float3 x, uint32_t pix,
                                          uint32_t s, int b, float cn, const float* env,
                                          Counters& cnt, RayList& L) {
  const Mask Mn = sample_mask_impl<true>(F, P.lod_nee, P.light, P.seed, pix, s, (uint32_t)b,
                                         TAG_NEE_MASK);
  const uint32_t wn = stream_word(s, (uint32_t)b, TAG_NEE);
  gather_list(F, Mn, x, P.light, L, cnt);
  float Tl = 1.f;
  for_windows(F, Mn, x, P.light, P.seed, pix, wn, env, cnt, &L,
              [&](const PointBuf& B, int n, const float* kap, const float* kb) {
                float coef[kPts];
#pragma unroll
                for (int i = 0; i < kPts; ++i) {
                  coef[i] = 0.f;
                  if (i < n && kb[i] > 0.f) {
                    const float q = fmaxf(kap[i], 0.f) / kb[i];
                    Tl *= 1.f - q;
                    if (cn != 0.f && kap[i] > 0.f && 1.f - q > 0.f) coef[i] = cn / (1.f - q) / kb[i];
                  }
                }
                if (cn != 0.f) scatter_window(F, Bk, Mn, x, P.light, B, coef, n, &L, cnt);
                return true;
              });
  return Tl;
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

__device__ void path_backward(const DevField& F, const PathParams& P, const BackArgs& Bk,
                              float3 o0, float3 v0, uint32_t pix, uint32_t s, float base,
                              const float* env, Counters& cnt, RayList& Lc, RayList& Ln) {
  const float E0 = P.irradiance * (0.25f / 3.14159265358979f);
  float Tb[kMaxSeg];
  int nseg = 0;
  // pass 1: the path, its NEE products
  {
    float3 o = o0, v = v0;
    for (int b = 0; b < P.max_bounces && b < kMaxSeg; ++b) {
      float th = 0.f;
      cnt.rays += 1;
      if (!path_segment(F, P, Bk, o, v, pix, s, b, 0.f, env, cnt, Lc, th)) break;
      const float3 x = make_float3(fmaf(th, v.x, o.x), fmaf(th, v.y, o.y), fmaf(th, v.z, o.z));
      cnt.rays += 1;
      Tb[nseg++] = path_nee(F, P, Bk, x, pix, s, b, 0.f, env, cnt, Ln);
      o = x;
      v = path_scatter_dir(P, pix, s, b);
    }
  }
  if (nseg == 0) return;
  // S_b = sum_{b' >= b} C_b', C_b = albedo^(b+1) E0 T_b
  float Ssuf = 0.f, thr = 1.f;
  for (int b = 0; b < nseg; ++b) {
    thr *= P.albedo;
    Ssuf += thr * E0 * Tb[b];
  }
  // pass 2: the same path again, scattering the coefficients
  float3 o = o0, v = v0;
  thr = 1.f;
  for (int b = 0; b < nseg; ++b) {
    float th = 0.f;
    if (!path_segment(F, P, Bk, o, v, pix, s, b, base * Ssuf, env, cnt, Lc, th)) break;
    const float3 x = make_float3(fmaf(th, v.x, o.x), fmaf(th, v.y, o.y), fmaf(th, v.z, o.z));
    thr *= P.albedo;
    const float Cb = thr * E0 * Tb[b];
    if (Tb[b] > 0.f) (void)path_nee(F, P, Bk, x, pix, s, b, -base * Cb, env, cnt, Ln);
    Ssuf -= Cb;
    o = x;
    v = path_scatter_dir(P, pix, s, b);
  }
}

// PATH = false: single scattering (the expected-value estimator above);
// PATH = true: multiple scattering (path_backward), each with its own frame
template <bool PATH>
__global__ void __launch_bounds__(kBackBlock)
    k_radiance_backward(const __grid_constant__ DevField F, const PathParams P, const BackArgs Bk,
                        const float* dLdI, int* counter, int* lists) {
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int nth = gridDim.x * blockDim.x;
  RayList Lc{lists + tid, nth, 0}, Ln{lists + (int64_t)kRayList * nth + tid, nth, 0};
  __shared__ RadSmem sm;
  if (threadIdx.x < 8) sm.env[threadIdx.x] = F.env[threadIdx.x];
  __syncthreads();
  const uint32_t lane = threadIdx.x & 31u;
  Counters cnt;
  const float E = P.albedo * P.irradiance * (0.25f / 3.14159265358979f);
  const int tiles_x = (P.cam.W + 7) / 8, tiles_y = (P.cam.H + 3) / 4;
  for (;;) {
    int tile = 0;
    if (lane == 0) tile = atomicAdd(counter, 1);
    tile = __shfl_sync(kFull, tile, 0);
    if (tile >= tiles_x * tiles_y) break;
    const int px = (tile % tiles_x) * 8 + (int)(lane % 8);
    const int py = (tile / tiles_x) * 4 + (int)(lane / 8);
    if (px >= P.cam.W || py >= P.cam.H) continue;  // every lane returns to the tile fetch
    const uint32_t pix = (uint32_t)(py * P.cam.W + px);
    const float gI = dLdI[pix];
    if (gI == 0.f) continue;
    const float base = gI / (float)P.spp;
    for (int s = P.s0; s < P.s0 + P.spp; ++s) {
      float3 o, v;
      camera_ray(P.cam, P.seed, px, py, s, o, v);
      if constexpr (PATH) {
        path_backward(F, P, Bk, o, v, pix, (uint32_t)s, base, sm.env, cnt, Lc, Ln);
        continue;
      }
      cnt.rays += 1;
      const Mask M = sample_mask_impl<true>(F, P.lod, v, P.seed, pix, (uint32_t)s, 0, TAG_MASK);
      const uint32_t wt = stream_word((uint32_t)s, 0, TAG_TRACK);
      gather_list(F, M, o, v, Lc, cnt);
      // pass 1: weights, their sum and the reservoir draw
      float Pr = 1.f, S = 0.f, pjs = 0.f, tjs = 0.f;
      int idx = 0, js = -1;
      for_windows(F, M, o, v, P.seed, pix, wt, sm.env, cnt, &Lc,
                  [&](const PointBuf& B, int n, const float* kap, const float* kb) {
                    for (int i = 0; i < n; ++i) {
                      const float p = kb[i] > 0.f ? fmaxf(kap[i], 0.f) / kb[i] : 0.f;
                      const float W = Pr * p;
                      S += W;
                      if (W > 0.f && B.u[i] * S < W) {
                        js = idx + i;
                        pjs = p;
                        tjs = B.t[i];
                      }
                      Pr *= 1.f - p;
                    }
                    idx += n;
                    return true;
                  });
      if (js < 0 || !(S > 0.f)) continue;
      // NEE from the drawn point by ratio tracking
      const float3 x = make_float3(fmaf(tjs, v.x, o.x), fmaf(tjs, v.y, o.y), fmaf(tjs, v.z, o.z));
      const Mask Mn = sample_mask_impl<true>(F, P.lod_nee, P.light, P.seed, pix, (uint32_t)s, 0, TAG_NEE_MASK);
      const uint32_t wn = stream_word((uint32_t)s, 0, TAG_NEE);
      cnt.rays += 1;
      gather_list(F, Mn, x, P.light, Ln, cnt);
      // ratio tracking of the NEE ray, T = prod (1 - kappa+/kappa_bar)
      float Tl = 1.f;
      for_windows(F, Mn, x, P.light, P.seed, pix, wn, sm.env, cnt, &Ln,
                  [&](const PointBuf& B, int n, const float* kap, const float* kb) {
                    for (int i = 0; i < n; ++i)
                      if (kb[i] > 0.f) Tl *= 1.f - fmaxf(kap[i], 0.f) / kb[i];
                    return true;
                  });
      const float G = E * Tl;
      // pass 2: camera points 0..js
      idx = 0;
      for_windows(F, M, o, v, P.seed, pix, wt, sm.env, cnt, &Lc,
                  [&](const PointBuf& B, int n, const float* kap, const float* kb) {
                    float coef[kPts];
#pragma unroll
                    for (int i = 0; i < kPts; ++i) {
                      coef[i] = 0.f;
                      const int gi = idx + i;
                      if (i < n && gi <= js && kap[i] > 0.f && kb[i] > 0.f) {
                        const float p = kap[i] / kb[i];
                        const float c = gi == js ? S * G / pjs : -S * G / (1.f - p);
                        coef[i] = base * c / kb[i];
                      }
                    }
                    scatter_window(F, Bk, M, o, v, B, coef, n, &Lc, cnt);
                    idx += n;
                    return idx <= js;
                  });
      // pass 3: NEE points
      if (Tl > 0.f) {
        for_windows(F, Mn, x, P.light, P.seed, pix, wn, sm.env, cnt, &Ln,
                    [&](const PointBuf& B, int n, const float* kap, const float* kb) {
                      float coef[kPts];
#pragma unroll
                      for (int i = 0; i < kPts; ++i) {
                        coef[i] = 0.f;
                        if (i < n && kap[i] > 0.f && kb[i] > 0.f) {
                          const float q = kap[i] / kb[i];
                          if (1.f - q > 0.f) coef[i] = -base * S * E * Tl / (1.f - q) / kb[i];
                        }
                      }
                      scatter_window(F, Bk, Mn, x, P.light, B, coef, n, &Ln, cnt);
                      return true;
                    });
      }
    }
  }
  flush_counters(F, cnt, lane);
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

cudaError_t launch_tomo_backward(const Field& F, const PathParams& P, const float* dLdI,
                                 float* grad, cudaStream_t s) {
  (void)cudaGetLastError();  // a stale error of an unrelated call is not ours
  cudaError_t e = cudaMemsetAsync(F.counter, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  BackArgs B = back_args(F, grad);
  cudaFuncAttributes fa;
  size_t limit = 0;
  if ((e = cudaFuncGetAttributes(&fa, k_tomo_backward)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetLimit(&limit, cudaLimitStackSize)) != cudaSuccess) return e;
  if (fa.localSizeBytes > limit) return cudaErrorLaunchOutOfResources;
  int64_t g = 1;
  if ((e = tomo_grid(F, g)) != cudaSuccess) return e;
  // scratch for a full grid (allocated ahead by gf_reserve, else here)
  if ((e = ensure_adjoint_lists(F, s)) != cudaSuccess) return e;
  // units of `chunk` samples of a pixel, about 16 per warp of the grid at least
  const int64_t npix = (int64_t)P.cam.W * P.cam.H, warps = g * (kBackBlock / 32);
  int64_t nchunk = (16 * warps + npix - 1) / npix;
  nchunk = nchunk < 1 ? 1 : (nchunk > P.spp ? P.spp : nchunk);
  const int64_t chunk = (P.spp + nchunk - 1) / nchunk;
  const int64_t units = npix * ((P.spp + chunk - 1) / chunk);
  const int64_t need = (units + kBackBlock / 32 - 1) / (kBackBlock / 32);
  if (need < g) g = need;
  if ((e = adjoint_begin(F, B, s)) != cudaSuccess) return e;
  k_tomo_backward<<<(unsigned)g, kBackBlock, 0, s>>>(F.dev, P, B, dLdI, F.counter, (int)chunk,
                                                     reinterpret_cast<TomoChord*>(F.rlist));
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  return adjoint_end(F, B, s);
}

// scratch of the adjoints, grown through the field's allocator: the radiance adjoint's
// primitive lists (2 per thread of a full persistent grid) or the tomography adjoint's
// kept chords in the same buffer, and the arrays per primitive
cudaError_t ensure_adjoint_lists(const Field& F, cudaStream_t s) {
  int per_sm = 0;
  for (auto k : {k_radiance_backward<false>, k_radiance_backward<true>}) {
    int q = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&q, k, kBackBlock, 0) != cudaSuccess)
      (void)cudaGetLastError();
    per_sm = q > per_sm ? q : per_sm;
  }
  if (per_sm < 1) per_sm = 1;
  const int64_t threads = (int64_t)F.ctx.sm_count * per_sm * kBackBlock;
  size_t bytes = (size_t)threads * 2 * kRayList * sizeof(int);
  int64_t g = 1;
  cudaError_t e = tomo_grid(F, g);
  if (e != cudaSuccess) return e;
  bytes = std::max(bytes, (size_t)g * (kBackBlock / 32) * kTomoChords * sizeof(TomoChord));
  if ((e = ensure_adjoint_prims(F, s)) != cudaSuccess) return e;
  return grow(F, (void**)&F.rlist, F.rlist_bytes, bytes, s);
}

cudaError_t launch_radiance_backward(const Field& F, const PathParams& P, const float* dLdI,
                                     float* grad, cudaStream_t s) {
  (void)cudaGetLastError();  // a stale error of an unrelated call is not ours
  cudaError_t e = cudaMemsetAsync(F.counter, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  const BackArgs B = back_args(F, grad);
  auto kernel = P.max_bounces >= 2 ? k_radiance_backward<true> : k_radiance_backward<false>;
  // the kernel's local frame must fit the context's stack limit as it stands
  cudaFuncAttributes fa;
  size_t limit = 0;
  if ((e = cudaFuncGetAttributes(&fa, kernel)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetLimit(&limit, cudaLimitStackSize)) != cudaSuccess) return e;
  if (fa.localSizeBytes > limit) return cudaErrorLaunchOutOfResources;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kBackBlock, 0) != cudaSuccess)
    (void)cudaGetLastError();
  if (per_sm < 1) per_sm = 1;
  const int64_t tiles = (int64_t)((P.cam.W + 7) / 8) * ((P.cam.H + 3) / 4);
  const int64_t need = (tiles + kBackBlock / 32 - 1) / (kBackBlock / 32);
  int64_t g = (int64_t)F.ctx.sm_count * per_sm;
  if (need < g) g = need;
  if (g < 1) g = 1;
  // lists sized for a full grid (allocated ahead by gf_reserve, else here)
  if ((e = ensure_adjoint_lists(F, s)) != cudaSuccess) return e;
  kernel<<<(unsigned)g, kBackBlock, 0, s>>>(F.dev, P, B, dLdI, F.counter, F.rlist);
  return cudaGetLastError();
}

}  // namespace gf
