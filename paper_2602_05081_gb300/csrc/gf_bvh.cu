// gf_bvh.cu -- primitive packing (load-time binning of Sec. 4.6) and the BVH
// over the k-sigma ellipsoid bounds (Sec. 3): Morton codes under a cell
// prefix, radix sort, Karras's binary radix tree, bottom-up box/mask refit.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <type_traits>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <cub/device/device_radix_sort.cuh>
#include <cub/device/device_scan.cuh>

#include "gf_host.h"

namespace gf {

// ---------------------------------------------------------------------------
// pack: parameters -> Sigma^-1, world carrier, amplitude, labels, boxes
// ---------------------------------------------------------------------------
struct PackArgs {
  gf_params p;
  int weight_mode, omega_frame, precision;
  float ksig;
  float clamp_eps;  // adaptive clamping threshold (0: off)
  float axes[kCones][3];
  float4* rec;
  float* box;
  float* kw;
  float* ext2;      // support radius squared per primitive (k^2 or adaptive)
  uint8_t* labels;  // band[N], cone[N], cell[N]
  CellAcc* cell_acc;
  int* err;
};

__global__ void k_pack(const __grid_constant__ PackArgs A) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= A.p.n) return;
  float mu[3], q[4], ls[3], om_in[3];
  for (int j = 0; j < 3; ++j) {
    mu[j] = A.p.mu[3 * i + j];
    ls[j] = A.p.log_scale[3 * i + j];
    om_in[j] = A.p.omega[3 * i + j];
  }
  for (int j = 0; j < 4; ++j) q[j] = A.p.quat[4 * i + j];
  float phi = A.p.phase[i], wt = A.p.weight[i];
  bool finite = isfinite(phi) && isfinite(wt);
  for (int j = 0; j < 3; ++j) finite = finite && isfinite(mu[j]) && isfinite(ls[j]) && isfinite(om_in[j]);
  for (int j = 0; j < 4; ++j) finite = finite && isfinite(q[j]);
  float qn = sqrtf(q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
  if (!finite || !(qn > 0.f)) {
    atomicOr(A.err, ERR_INPUT);
    qn = 1.f;
    q[0] = 1.f; q[1] = q[2] = q[3] = 0.f;
  }
  float w = q[0] / qn, x = q[1] / qn, y = q[2] / qn, z = q[3] / qn;
  float R[3][3] = {{1.f - 2.f * (y * y + z * z), 2.f * (x * y - w * z), 2.f * (x * z + w * y)},
                   {2.f * (x * y + w * z), 1.f - 2.f * (x * x + z * z), 2.f * (y * z - w * x)},
                   {2.f * (x * z - w * y), 2.f * (y * z + w * x), 1.f - 2.f * (x * x + y * y)}};
  float s[3] = {expf(ls[0]), expf(ls[1]), expf(ls[2])};
  float is2[3] = {1.f / (s[0] * s[0]), 1.f / (s[1] * s[1]), 1.f / (s[2] * s[2])};
  float P[3][3];
  for (int a = 0; a < 3; ++a)
    for (int b = 0; b < 3; ++b)
      P[a][b] = R[a][0] * R[b][0] * is2[0] + R[a][1] * R[b][1] * is2[1] + R[a][2] * R[b][2] * is2[2];
  float om[3], kw[3];
  if (A.omega_frame == GF_OMEGA_LOCAL) {
    for (int a = 0; a < 3; ++a)
      om[a] = R[a][0] * om_in[0] / s[0] + R[a][1] * om_in[1] / s[1] + R[a][2] * om_in[2] / s[2];
    for (int j = 0; j < 3; ++j) kw[j] = om_in[j];
  } else {
    for (int a = 0; a < 3; ++a) om[a] = om_in[a];
    for (int j = 0; j < 3; ++j) kw[j] = s[j] * (R[0][j] * om[0] + R[1][j] * om[1] + R[2][j] * om[2]);
  }
  float amp = wt;
  if (A.weight_mode == GF_WEIGHT_NORMALIZED) amp = wt / (15.749609945722419f * s[0] * s[1] * s[2]);
  // band: caller's octave label, else floor(log2(1 + |omega|/(2 pi))) decided in FP32
  int band;
  if (A.p.band) {
    band = A.p.band[i];
    if (band > 7) {
      atomicOr(A.err, ERR_INPUT);
      band = 7;
    }
  } else {
    float n2 = __fadd_rn(__fadd_rn(__fmul_rn(om[0], om[0]), __fmul_rn(om[1], om[1])), __fmul_rn(om[2], om[2]));
    float onef = __fadd_rn(1.0f, __fdiv_rn(__fsqrt_rn(n2), 6.28318530717958647692f));
    band = 0;
    for (int j = 1; j <= 7; ++j)
      if (onef >= (float)(1 << j)) band = j;
  }
  // orientation bin: argmax |omega . o_k| in FP32, ties to the lowest k
  int cone = 0;
  if (band > 0) {
    float bv = -1.f;
    for (int k = 0; k < kCones; ++k) {
      float d = fabsf(__fadd_rn(__fadd_rn(__fmul_rn(om[0], A.axes[k][0]), __fmul_rn(om[1], A.axes[k][1])),
                                __fmul_rn(om[2], A.axes[k][2])));
      if (d > bv) {
        bv = d;
        cone = k;
      }
    }
  }
  int cell = band == 0 ? 0 : 1 + kCones * (band - 1) + cone;
  float kn = sqrtf(kw[0] * kw[0] + kw[1] * kw[1] + kw[2] * kw[2]);
  // support radius: k, or the adaptive extent of Sec. 4.4 (Eqs. 14-15) where the
  // kernel's largest line integral rho = |A| sqrt(2 pi) s_max, attenuated by
  // exp(-(E^2 + |k_W|^2)/2), falls to clamp_eps
  float k2i = A.ksig * A.ksig;
  if (A.clamp_eps > 0.0f) {
    const float rho = fabsf(amp) * 2.5066282746310002f * fmaxf(fmaxf(s[0], s[1]), s[2]);
    const float e2 = 2.0f * logf(rho / A.clamp_eps) - kn * kn;
    k2i = e2 > 0.0f ? fminf(k2i, e2) : -1.0f;  // -1: dropped, no ray finds a chord
  }
  A.ext2[i] = k2i;
  const float kext = sqrtf(fmaxf(k2i, 0.0f));
  float4* r = A.rec + 4 * i;
  r[0] = make_float4(mu[0], mu[1], mu[2], amp);
  r[1] = make_float4(P[0][0], P[0][1], P[0][2], P[1][1]);
  r[2] = make_float4(P[1][2], P[2][2], phi, k2i);
  r[3] = make_float4(om[0], om[1], om[2], __uint_as_float((uint32_t)i | ((uint32_t)cell << 26)));
  // box of the k-sigma ellipsoid: half-extent k sqrt(Sigma_jj), padded.
  // Reduced-precision records store the whitening factor T (upper triangular,
  // T^T T = Sigma^-1) with every entry rounded by u = 2^-11 (FP16) or 2^-8
  // (BF16) of itself: with dT that rounding, |dT z| <= u ||T||_F |z| and
  // |z| <= ||T^-1||_2 |T z|, so the decoded ellipsoid lies within the exact one
  // grown by eps = u ||T||_F ||T^-1||_2 = u s_max sqrt(sum 1/s_i^2) of itself
  // (2e-7 more covers entries that round as FP16 subnormals); pad with a 1.5x
  // margin (the mean's u16 step is added once the means' box is known, in
  // build_bvh)
  const float urel = A.precision == GF_PREC_BF16 ? 3.90625e-3f
                   : A.precision == GF_PREC_FP16 ? 4.8828125e-4f : 0.f;
  const float tcond = fmaxf(fmaxf(s[0], s[1]), s[2]) * sqrtf(is2[0] + is2[1] + is2[2]);
  const float rel = urel > 0.f ? 1.5f * (urel + 2e-7f) * tcond : 1e-5f;
  for (int a = 0; a < 3; ++a) {
    float sjj = R[a][0] * R[a][0] * s[0] * s[0] + R[a][1] * R[a][1] * s[1] * s[1] +
                R[a][2] * R[a][2] * s[2] * s[2];
    float hw = kext * sqrtf(sjj);
    float pad = rel * hw + 1e-6f * (1.f + fabsf(mu[a]));
    A.box[6 * i + a] = mu[a] - hw - pad;
    A.box[6 * i + 3 + a] = mu[a] + hw + pad;
  }
  A.kw[i] = kn;
  A.labels[i] = (uint8_t)band;
  A.labels[A.p.n + i] = (uint8_t)cone;
  A.labels[2 * A.p.n + i] = (uint8_t)cell;
  // largest |k_W| and largest world carrier |omega| per band (the per-cell sums
  // follow in k_cell_sums, on the scale the first one sets)
  // one atomic per warp (and band): 200k atomics on one word took most of this kernel's
  // 78 us
  const unsigned am = __activemask();
  const int me = (int)(threadIdx.x & 31u);
  const unsigned km = __reduce_max_sync(am, __float_as_uint(kn));
  if (me == __ffs((int)am) - 1) atomicMax(&A.cell_acc->kw_max, km);
  const unsigned same = __match_any_sync(am, band);
  const unsigned wm = __reduce_max_sync(
      same, __float_as_uint(sqrtf(om[0] * om[0] + om[1] * om[1] + om[2] * om[2])));
  if (me == __ffs((int)same) - 1) atomicMax(&A.cell_acc->band_wmax[band], wm);
}

// per cell: the sum of |k_W| in exact fixed point and the member count.  A block sums
// kCellBlock kernels in shared memory first, each term (at most 2^36) as a low and a high
// part of 18 bits (400k 64-bit atomics on a few dozen words took 50 to 98 us).
constexpr int kCellBlock = 1024;
__global__ void __launch_bounds__(256) k_cell_sums(const float* kw, const uint8_t* cell, int64_t n,
                                                   CellAcc* acc) {
  __shared__ unsigned lo[64], hi[64], cnt[64];
  if (threadIdx.x < 64) lo[threadIdx.x] = hi[threadIdx.x] = cnt[threadIdx.x] = 0u;
  __syncthreads();
  const int e = cell_fix_exp(acc->kw_max);
  const float sc = __int_as_float((127 + 36 - e) << 23);  // 2^(36 - e)
  const int64_t i0 = (int64_t)blockIdx.x * kCellBlock;
  for (int k = (int)threadIdx.x; k < kCellBlock && i0 + k < n; k += 256) {
    const unsigned c = cell[i0 + k] & 63u;
    const unsigned long long v = (unsigned long long)__float2ull_rn(kw[i0 + k] * sc);
    atomicAdd(&lo[c], (unsigned)(v & 0x3FFFFull));
    atomicAdd(&hi[c], (unsigned)(v >> 18));
    atomicAdd(&cnt[c], 1u);
  }
  __syncthreads();
  if (threadIdx.x < 64 && cnt[threadIdx.x]) {
    const unsigned c = threadIdx.x;
    atomicAdd(&acc->kw_fix[c], ((unsigned long long)hi[c] << 18) + lo[c]);
    atomicAdd(&acc->count[c], (unsigned long long)cnt[c]);
  }
}

cudaError_t launch_pack(Field& F, const gf_params& P, cudaStream_t s) {
  (void)cudaGetLastError();  // a stale error of an unrelated call is not ours
  PackArgs A;
  A.p = P;
  A.weight_mode = F.opts.weight_mode;
  A.omega_frame = F.opts.omega_frame;
  A.precision = F.opts.precision;
  A.ksig = F.opts.k_sigma;
  A.clamp_eps = F.opts.clamp_eps;
  A.ext2 = F.ext2_orig;
  for (int k = 0; k < kCones; ++k)
    for (int j = 0; j < 3; ++j) A.axes[k][j] = F.dev.axes[k][j];
  A.rec = F.rec_orig;
  A.box = F.box_orig;
  A.kw = F.kw_orig;
  A.labels = F.labels;
  A.cell_acc = F.cell_acc;
  A.err = F.err;
  int64_t blocks = (P.n + 127) / 128;
  k_pack<<<(unsigned)blocks, 128, 0, s>>>(A);
  k_cell_sums<<<(unsigned)((P.n + kCellBlock - 1) / kCellBlock), 256, 0, s>>>(A.kw, A.labels + 2 * P.n,
                                                                             P.n, A.cell_acc);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// BVH build
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned int ord_enc(float f) {
  unsigned int u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ord_dec(unsigned int u) {
  return __uint_as_float((u & 0x80000000u) ? (u & 0x7FFFFFFFu) : ~u);
}

// bounds[0..2] box min, [3..5] box max, [6..8] centre min, [9..11] centre max (ordered ints)
__global__ void k_bounds(const float* box, const float4* rec, int64_t n, unsigned int* bounds) {
  float v[12];
  for (int j = 0; j < 3; ++j) {
    v[j] = INFINITY; v[3 + j] = -INFINITY; v[6 + j] = INFINITY; v[9 + j] = -INFINITY;
  }
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    float4 r0 = rec[4 * i];
    float m[3] = {r0.x, r0.y, r0.z};
    for (int j = 0; j < 3; ++j) {
      v[j] = fminf(v[j], box[6 * i + j]);
      v[3 + j] = fmaxf(v[3 + j], box[6 * i + 3 + j]);
      v[6 + j] = fminf(v[6 + j], m[j]);
      v[9 + j] = fmaxf(v[9 + j], m[j]);
    }
  }
  // warp, block, then one atomic per block and bound
  __shared__ unsigned int part[12][8];
  for (int j = 0; j < 12; ++j) {
    const bool mn = (j < 3) || (j >= 6 && j < 9);
    const unsigned x = ord_enc(v[j]);
    const unsigned r = mn ? __reduce_min_sync(kFull, x) : __reduce_max_sync(kFull, x);
    if ((threadIdx.x & 31) == 0) part[j][threadIdx.x >> 5] = r;
  }
  __syncthreads();
  if (threadIdx.x < 12) {
    const int j = (int)threadIdx.x;
    const bool mn = (j < 3) || (j >= 6 && j < 9);
    unsigned r = part[j][0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) r = mn ? min(r, part[j][w]) : max(r, part[j][w]);
    if (mn) atomicMin(bounds + j, r);
    else atomicMax(bounds + j, r);
  }
}

__device__ __forceinline__ unsigned int spread10(unsigned int x) {
  x &= 1023u;
  x = (x | (x << 16)) & 0x030000FFu;
  x = (x | (x << 8)) & 0x0300F00Fu;
  x = (x | (x << 4)) & 0x030C30C3u;
  x = (x | (x << 2)) & 0x09249249u;
  return x;
}

// sort keys of both trees: the cell, or its band, above 30 Morton bits of the mean; the
// second tree's n entries follow the first's, with bit 36 set, so that one sort orders
// both
__device__ __forceinline__ uint32_t cell_band(uint32_t cell) { return cell == 0 ? 0u : ((cell - 1u) >> 3) + 1u; }
// face areas of a box, summed over the three axes
__host__ __device__ __forceinline__ float face_areas(float x, float y, float z) { return x * y + y * z + z * x; }
// unit of the summed shares of the scene's face areas that the kernels' boxes take: a
// share is at most 1, so 256 of them stay below 2^32
constexpr float kAreaUnit = 1.0f / 2097152.0f;

__global__ void __launch_bounds__(256) k_morton(const float4* rec, const float* box, int64_t n,
                                                const unsigned int* bounds, unsigned long long* keys,
                                                int* idx, unsigned long long* area) {
  // per band: the boxes' shares of the scene's face areas (sums of integers, the same in
  // any order)
  __shared__ unsigned int part[8];
  if (threadIdx.x < 8) part[threadIdx.x] = 0u;
  __syncthreads();
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    const float* b = box + 6 * i;
    const float s = face_areas(ord_dec(bounds[3]) - ord_dec(bounds[0]), ord_dec(bounds[4]) - ord_dec(bounds[1]),
                               ord_dec(bounds[5]) - ord_dec(bounds[2]));
    const float q = face_areas(b[3] - b[0], b[4] - b[1], b[5] - b[2]) / s;
    if (q > 0.f)  // (not for boxes without faces)
      atomicAdd(&part[cell_band(__float_as_uint(rec[4 * i + 3].w) >> 26)],
                (unsigned)__float2uint_rn(fminf(q, 1.0f) * (1.0f / kAreaUnit)));
  }
  __syncthreads();
  if (threadIdx.x < 8 && part[threadIdx.x]) atomicAdd(area + threadIdx.x, (unsigned long long)part[threadIdx.x]);
  if (i >= n) return;
  float lo[3], hi[3];
  for (int j = 0; j < 3; ++j) {
    lo[j] = ord_dec(bounds[6 + j]);
    hi[j] = ord_dec(bounds[9 + j]);
  }
  float4 r0 = rec[4 * i];
  uint32_t cell = __float_as_uint(rec[4 * i + 3].w) >> 26;
  float m[3] = {r0.x, r0.y, r0.z};
  unsigned int c[3];
  for (int j = 0; j < 3; ++j) {
    float ext = hi[j] - lo[j];
    float u = ext > 0.f ? (m[j] - lo[j]) / ext : 0.5f;
    u = fminf(fmaxf(u, 0.f), 1.f);
    c[j] = (unsigned int)fminf(u * 1024.f, 1023.f);
  }
  unsigned int mc = (spread10(c[0]) << 2) | (spread10(c[1]) << 1) | spread10(c[2]);
  keys[i] = ((unsigned long long)cell << 30) | mc;
  keys[n + i] = 1ull << 36 | ((unsigned long long)cell_band(cell) << 30) | mc;
  idx[i] = (int)i;
  idx[n + i] = (int)i;
}

__global__ void k_gather(const float4* rec_in, const float* box_in, const float* ext2_in,
                         const int* idx, int64_t n, float4* rec_out, float* box_out,
                         float* ext2_out, float4* muw_out, int* sorted_orig, int* pos) {
  int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  int i = idx[j];
  for (int k = 0; k < 4; ++k) rec_out[4 * j + k] = rec_in[4 * (int64_t)i + k];
  for (int k = 0; k < 6; ++k) box_out[6 * j + k] = box_in[6 * (int64_t)i + k];
  ext2_out[j] = ext2_in[i];
  // mean and |omega| (FP32, no contraction) for the camera LoD selection
  const float4 r0 = rec_in[4 * (int64_t)i], r3 = rec_in[4 * (int64_t)i + 3];
  const float wn = __fsqrt_rn(__fadd_rn(__fadd_rn(__fmul_rn(r3.x, r3.x), __fmul_rn(r3.y, r3.y)),
                                        __fmul_rn(r3.z, r3.z)));
  muw_out[j] = make_float4(r0.x, r0.y, r0.z, wn);
  sorted_orig[j] = i;
  pos[i] = (int)j;
}

// leaves of the tree by bands: the sorted primitive of each
__global__ void k_band_leaves(const int* idx, const int* pos, int64_t n, int* of) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p < n) of[p] = pos[idx[n + p]];
}

// One of the two binary trees in the making (by cells, by bands).  The kernels below
// build both in one launch (blockIdx.y): each is bound by the latency of its chains, not
// by its size.
struct TreeBuild {
  const unsigned long long* keys;
  Node* nodes;
  int* above;               // node above each leaf
  int* flags;               // refit counters, then marks of four-wide nodes
  const int* of;            // sorted primitive of each leaf (null: the leaf itself)
  unsigned int* max_depth;
  bool band;
};
struct TreePair {
  TreeBuild t[2];
};

// camera LoD selection (Supp. A): primitive j stays in the mixture iff
// |omega| d <= c, d the distance from the eye to its mean, c = pi H / (2 tan(phi/2))
// (c = +inf restores every primitive).  A removed primitive gets the support
// radius squared -1, so no ray finds a chord of it; the cells still holding a
// primitive are OR-ed into *cells.
__global__ void k_camera_lod(const float4* muw, const float* k2own, const uint8_t* cell_of_orig,
                             const int* sorted_orig, int64_t n, float3 eye, float c, float4* rec,
                             float* k2eff, unsigned long long* cells) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long cb = 0ull;
  if (j < n) {
    const float4 m = muw[j];
    const float dx = __fsub_rn(m.x, eye.x), dy = __fsub_rn(m.y, eye.y), dz = __fsub_rn(m.z, eye.z);
    const float d = __fsqrt_rn(__fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)),
                                         __fmul_rn(dz, dz)));
    const bool k = __fmul_rn(m.w, d) <= c;
    const float v = k ? k2own[j] : -1.0f;
    if (rec) rec[4 * j + 2].w = v;
    if (k2eff) k2eff[j] = v;
    if (k) cb = 1ull << (cell_of_orig[sorted_orig[j]] & 63u);
  }
  const unsigned lo = __reduce_or_sync(kFull, (unsigned)cb);
  const unsigned hi = __reduce_or_sync(kFull, (unsigned)(cb >> 32));
  if ((threadIdx.x & 31u) == 0 && (lo | hi)) atomicOr(cells, ((unsigned long long)hi << 32) | lo);
}

cudaError_t launch_camera_lod(Field& F, float3 eye, float c, cudaStream_t s) {
  (void)cudaGetLastError();  // a stale error of an unrelated call is not ours
  cudaError_t e = cudaMemsetAsync(F.cells_dev, 0, sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  k_camera_lod<<<(unsigned)((F.n + 255) / 256), 256, 0, s>>>(
      F.muw, F.ext2, F.labels + 2 * F.n, F.sorted_orig, F.n, eye, c, F.rec, F.keff2, F.cells_dev);
  return cudaGetLastError();
}

__device__ __forceinline__ int delta_key(const unsigned long long* k, int64_t n, int64_t i, int64_t j) {
  if (j < 0 || j >= n) return -1;
  unsigned long long a = k[i], b = k[j];
  if (a == b) return 64 + __clz((unsigned int)(i ^ j));
  return __clzll(a ^ b);
}

// Karras (HPG 2012): internal node i covers [min(i,j), max(i,j)], split at gamma
__global__ void k_karras(const __grid_constant__ TreePair T, int64_t n) {
  const unsigned long long* keys = T.t[blockIdx.y].keys;
  Node* nodes = T.t[blockIdx.y].nodes;
  int* leaf_parent = T.t[blockIdx.y].above;
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n - 1) return;
  int d = (delta_key(keys, n, i, i + 1) - delta_key(keys, n, i, i - 1)) >= 0 ? 1 : -1;
  int dmin = delta_key(keys, n, i, i - d);
  int64_t lmax = 2;
  while (delta_key(keys, n, i, i + lmax * d) > dmin) lmax *= 2;
  int64_t l = 0;
  for (int64_t t = lmax / 2; t >= 1; t /= 2)
    if (delta_key(keys, n, i, i + (l + t) * d) > dmin) l += t;
  int64_t j = i + l * d;
  int dnode = delta_key(keys, n, i, j);
  int64_t s = 0;
  int64_t t = l;
  do {
    t = (t + 1) / 2;
    if (delta_key(keys, n, i, i + (s + t) * d) > dnode) s += t;
  } while (t > 1);
  int64_t gamma = i + s * d + (d < 0 ? -1 : 0);
  int64_t lo = i < j ? i : j, hi = i < j ? j : i;
  int left = (lo == gamma) ? ~(int)gamma : (int)gamma;
  int right = (hi == gamma + 1) ? ~(int)(gamma + 1) : (int)(gamma + 1);
  nodes[i].d.x = left;
  nodes[i].d.y = right;
  if (left >= 0) nodes[left].d.z = (int)i; else leaf_parent[gamma] = (int)i;
  if (right >= 0) nodes[right].d.z = (int)i; else leaf_parent[gamma + 1] = (int)i;
  if (i == 0) nodes[0].d.z = -1;
}

__device__ __forceinline__ void write_slot(Node* nd, int slot, const float* b, unsigned long long m) {
  volatile float* a = reinterpret_cast<volatile float*>(&nd->a);
  volatile unsigned int* e = reinterpret_cast<volatile unsigned int*>(&nd->e);
  if (slot == 0) {
    a[0] = b[0]; a[1] = b[1]; a[2] = b[2]; a[3] = b[3]; a[4] = b[4]; a[5] = b[5];
    e[0] = (unsigned int)m; e[1] = (unsigned int)(m >> 32);
  } else {
    a[6] = b[0]; a[7] = b[1]; a[8] = b[2]; a[9] = b[3]; a[10] = b[4]; a[11] = b[5];
    e[2] = (unsigned int)m; e[3] = (unsigned int)(m >> 32);
  }
}

// bottom-up refit: the second child to arrive at a node merges both slots.  Leaf j of
// the tree is the sorted primitive of[j] (j itself without of); masks hold cells, or
// bands when by_band.
__global__ void k_refit(const float* box, const float4* rec, const __grid_constant__ TreePair T,
                        int64_t n) {
  const TreeBuild& B = T.t[blockIdx.y];
  const int* of = B.of;
  const bool by_band = B.band;
  Node* nodes = B.nodes;
  const int* leaf_parent = B.above;
  int* flags = B.flags;
  int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const int64_t pj = of ? of[j] : j;
  float b[6];
  for (int k = 0; k < 6; ++k) b[k] = box[6 * pj + k];
  const uint32_t cell = __float_as_uint(rec[4 * pj + 3].w) >> 26;
  unsigned long long m = 1ull << (by_band ? cell_band(cell) : cell);
  int child = ~(int)j;
  int node = leaf_parent[j];
  for (int guard = 0; node >= 0 && guard < 4096; ++guard) {
    Node* nd = nodes + node;
    int slot = (nd->d.x == child) ? 0 : 1;
    write_slot(nd, slot, b, m);
    __threadfence();
    if (atomicAdd(flags + node, 1) == 0) return;
    __threadfence();
    volatile float* a = reinterpret_cast<volatile float*>(&nd->a);
    volatile unsigned int* e = reinterpret_cast<volatile unsigned int*>(&nd->e);
    b[0] = fminf(a[0], a[6]); b[1] = fminf(a[1], a[7]); b[2] = fminf(a[2], a[8]);
    b[3] = fmaxf(a[3], a[9]); b[4] = fmaxf(a[4], a[10]); b[5] = fmaxf(a[5], a[11]);
    m = ((unsigned long long)e[0] | ((unsigned long long)e[1] << 32)) |
        ((unsigned long long)e[2] | ((unsigned long long)e[3] << 32));
    child = node;
    node = nd->d.z;
  }
}

// ---------------------------------------------------------------------------
// Four-wide trees.  Keys begin with the class (cell, or band), so the primitives of a
// class are one subtree of the binary tree (or one leaf).  Within it, binary nodes at
// even depth below its root become Node4s whose children are their children's children
// (a leaf child stays a leaf).
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long node_mask(const Node& N) {
  return (unsigned long long)(N.e.x | N.e.z) | ((unsigned long long)(N.e.y | N.e.w) << 32);
}
__device__ __forceinline__ bool one_class(unsigned long long m) { return (m & (m - 1ull)) == 0ull; }

__global__ void k_depth_parity(const __grid_constant__ TreePair T, int64_t m) {
  const Node* nodes = T.t[blockIdx.y].nodes;
  int* even = T.t[blockIdx.y].flags;
  unsigned int* max_depth = T.t[blockIdx.y].max_depth;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  int d = 0, dc = 0;  // depth, depth below the class's root
  bool in = one_class(node_mask(nodes[i]));
  even[i] = in ? 1 : 0;
  int v = (int)i;
  for (int g = 0; g < 4096 && v > 0; ++g) {  // node 0 is the root
    v = nodes[v].d.z;
    ++d;
    in = in && one_class(node_mask(nodes[v]));
    dc += in ? 1 : 0;
  }
  if (dc & 1) even[i] = 0;
  const unsigned am = __activemask();
  const unsigned dm = __reduce_max_sync(am, (unsigned)d);
  if ((int)(threadIdx.x & 31u) == __ffs((int)am) - 1) atomicMax(max_depth, dm);
}

__device__ __forceinline__ void node_slot(const Node& N, int slot, float* b, unsigned long long& m,
                                          int& child) {
  const float* a = reinterpret_cast<const float*>(&N.a);
  const int o = slot == 0 ? 0 : 6;
  for (int k = 0; k < 6; ++k) b[k] = a[o + k];
  m = slot == 0 ? ((unsigned long long)N.e.x | ((unsigned long long)N.e.y << 32))
                : ((unsigned long long)N.e.z | ((unsigned long long)N.e.w << 32));
  child = slot == 0 ? N.d.x : N.d.y;
}

__device__ __forceinline__ Node4 emit_node4(int nc, const float box[4][6], const int ch[4]) {
  float lo[3], hi[3], sc[3];
  for (int a = 0; a < 3; ++a) {
    lo[a] = box[0][a];
    hi[a] = box[0][3 + a];
    for (int k = 1; k < nc; ++k) {
      lo[a] = fminf(lo[a], box[k][a]);
      hi[a] = fmaxf(hi[a], box[k][3 + a]);
    }
    // grid step s, never zero, and origin lo - s/64: every child keeps a margin of s/128
    // between its box and its decoded planes (254.9 s + s/64 + s/128 <= 255 s), which
    // covers the rounding of the codes' part of a plane in the traversal (s/512)
    sc[a] = __fdiv_ru(__fsub_ru(hi[a], lo[a]), 254.9f);
    const float floor_s = fmaxf(fabsf(lo[a]), fabsf(hi[a])) * 1e-7f + 1e-30f;
    sc[a] = fmaxf(sc[a], floor_s);
    lo[a] = __fsub_rd(lo[a], 0.015625f * sc[a]);
  }
  uint32_t ql[3] = {0, 0, 0}, qh[3] = {0, 0, 0};
  for (int k = 0; k < nc; ++k) {
    for (int a = 0; a < 3; ++a) {
      // conservative codes with the margin
      const float m = 0.0078125f * sc[a];
      const float bl = __fsub_rd(box[k][a], m), bh = __fadd_ru(box[k][3 + a], m);
      float fl = floorf((bl - lo[a]) / sc[a]);
      int cl = (int)fminf(fmaxf(fl, 0.f), 255.f);
      while (cl > 0 && fmaf((float)cl, sc[a], lo[a]) > bl) --cl;
      float fh = ceilf((bh - lo[a]) / sc[a]);
      int chh = (int)fminf(fmaxf(fh, 0.f), 255.f);
      while (chh < 255 && fmaf((float)chh, sc[a], lo[a]) < bh) ++chh;
      ql[a] |= (uint32_t)cl << (8 * k);
      qh[a] |= (uint32_t)chh << (8 * k);
    }
  }
  Node4 o;
  o.v0 = make_float4(lo[0], lo[1], lo[2], 32768.0f * sc[0]);
  o.v1 = make_float4(32768.0f * sc[1], 32768.0f * sc[2], __uint_as_float(ql[0]), __uint_as_float(ql[1]));
  o.q = make_uint4(ql[2], qh[0], qh[1], qh[2]);
  o.child = make_int4(ch[0], nc > 1 ? ch[1] : kNoChild, nc > 2 ? ch[2] : kNoChild,
                      nc > 3 ? ch[3] : kNoChild);
  return o;
}

// out[base + map[i]]: Node4 of the marked binary node i; out[single + class]: the root of
// a class with one primitive.  roots[class] receives the class's root.
struct CollapseArgs {
  const Node* nodes;
  int64_t m;
  const int *even, *map, *of;
  Node4* out;
  int base, single;  // out index of map 0, and of class 0's one-primitive root
  int* roots;
};
struct CollapsePair {
  CollapseArgs a[2];
};
__global__ void k_collapse4(const __grid_constant__ CollapsePair C2) {
  const CollapseArgs& A = C2.a[blockIdx.y];
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= A.m) return;
  auto leaf = [&](int c) { return A.of ? ~A.of[~c] : c; };
  const Node& N = A.nodes[i];
  const unsigned long long mi = node_mask(N);
  float box[4][6];
  unsigned long long mm;
  int ch[4] = {kNoChild, kNoChild, kNoChild, kNoChild};
  if (!one_class(mi)) {
    // a class of one primitive hangs below as a leaf
    for (int s = 0; s < 2; ++s) {
      int c;
      node_slot(N, s, box[0], mm, c);
      if (c >= 0) continue;
      const int cls = __ffsll((long long)mm) - 1, at = A.single + cls;
      ch[0] = leaf(c);
      A.out[at] = emit_node4(1, box, ch);
      A.roots[cls] = at;
    }
    return;
  }
  if (!A.even[i]) return;
  int nc = 0;
  for (int s = 0; s < 2; ++s) {
    float b[6];
    int c;
    node_slot(N, s, b, mm, c);
    if (c < 0) {
      for (int k = 0; k < 6; ++k) box[nc][k] = b[k];
      ch[nc++] = leaf(c);
      continue;
    }
    const Node& C = A.nodes[c];
    for (int t = 0; t < 2; ++t) {
      int cc;
      node_slot(C, t, box[nc], mm, cc);
      ch[nc++] = cc < 0 ? leaf(cc) : A.base + A.map[cc];
    }
  }
  const int at = A.base + A.map[i];
  A.out[at] = emit_node4(nc, box, ch);
  if (i == 0 || !one_class(node_mask(A.nodes[N.d.z]))) A.roots[__ffsll((long long)mi) - 1] = at;
}

// the tree of a one-primitive field
__global__ void k_single4(const float* box, const float4* rec, bool by_band, Node4* out, int base,
                          int* roots) {
  float b[4][6];
  for (int k = 0; k < 6; ++k) b[0][k] = box[k];
  const int ch[4] = {~0, kNoChild, kNoChild, kNoChild};
  const uint32_t cell = __float_as_uint(rec[3].w) >> 26;
  const int cls = (int)(by_band ? cell_band(cell) : cell);
  out[base + cls] = emit_node4(1, b, ch);
  roots[cls] = base + cls;
}

// reduced-precision records: the decoded mean moves by up to half a u16 step of
// the means' box on each axis; grow every box by that (with 2 % margin)
__global__ void k_pad_mean_step(float* box, int64_t n, const unsigned int* bounds) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  for (int a = 0; a < 3; ++a) {
    const float ext = ord_dec(bounds[9 + a]) - ord_dec(bounds[6 + a]);
    const float pad = ext > 0.f ? 0.51f * ext / 65535.f : 0.f;
    box[6 * i + a] -= pad;
    box[6 * i + 3 + a] += pad;
  }
}


// results of the build that the host reads
struct BuildHead {
  unsigned int bounds[16];     // boxes (12), the two trees' depths
  unsigned long long area[8];  // per band: summed face areas (k_morton)
};

cudaError_t build_bvh(Field& F, cudaStream_t s) {
  (void)cudaGetLastError();  // a stale error of an unrelated call is not ours
  const int64_t n = F.n;
  cudaError_t e = cudaSuccess;
  // temporaries, in one block
  BuildHead* head = nullptr;
  unsigned int* bounds = nullptr;  // boxes (12), the two trees' depths
  int* roots = nullptr;            // of cells, then of bands
  unsigned long long *keys = nullptr, *keys2 = nullptr;
  int *idx = nullptr, *idx2 = nullptr, *above = nullptr, *above_b = nullptr, *flags = nullptr, *map = nullptr,
      *pos = nullptr, *of = nullptr;
  float* box_sorted = nullptr;
  Node* nodes_b = nullptr;  // binary tree by bands
  void *tmp = nullptr, *block = nullptr;
  size_t tmp_bytes = 0, sort_bytes = 0;
  const int64_t m = n - 1;
  const unsigned pn = (unsigned)((n + 255) / 256), pm = (unsigned)((m + 255) / 256);
  BuildHead hh;
  const unsigned int* hb = hh.bounds;
  int hroots[kMaxCells + 8];
#define GF_TRY(x) do { e = (x); if (e != cudaSuccess) goto done; } while (0)
  GF_TRY(cub::DeviceRadixSort::SortPairs(nullptr, sort_bytes, keys, keys2, idx, idx2, (int)(2 * n), 0, 37, s));
  GF_TRY(cub::DeviceScan::ExclusiveSum(nullptr, tmp_bytes, flags, map, (int)(2 * n), s));
  if (sort_bytes > tmp_bytes) tmp_bytes = sort_bytes;
  for (int pass = 0; pass < 2; ++pass) {  // sizes, then places
    uintptr_t at = reinterpret_cast<uintptr_t>(block);
    auto take = [&](auto*& p, size_t bytes) {
      p = reinterpret_cast<std::remove_reference_t<decltype(p)>>(at);
      at += (bytes + 255) & ~size_t(255);
    };
    char* tp = nullptr;
    take(head, sizeof(BuildHead));
    take(roots, sizeof(hroots));
    take(keys, 2 * n * sizeof(unsigned long long));
    take(keys2, 2 * n * sizeof(unsigned long long));
    take(idx, 2 * n * sizeof(int));
    take(idx2, 2 * n * sizeof(int));
    take(above, n * sizeof(int));
    take(above_b, n * sizeof(int));
    take(flags, 2 * n * sizeof(int));  // marks of both trees, m each
    take(map, 2 * n * sizeof(int));    // their scan
    take(pos, n * sizeof(int));
    take(of, n * sizeof(int));
    take(box_sorted, n * 6 * sizeof(float));
    take(nodes_b, n * sizeof(Node));
    take(tp, tmp_bytes);
    tmp = tp;
    if (pass == 0) GF_TRY(F.mem.alloc(&block, (size_t)at, s));
  }
  bounds = head->bounds;
  GF_TRY(cudaMemsetAsync(bounds + 12, 0, sizeof(BuildHead) - 12 * sizeof(unsigned int), s));
  GF_TRY(cudaMemsetAsync(roots, 0xFF, sizeof(hroots), s));
  {
    unsigned int init[12];
    for (int j = 0; j < 12; ++j) {
      bool mn = (j < 3) || (j >= 6 && j < 9);
      init[j] = mn ? 0xFFFFFFFFu : 0u;
    }
    GF_TRY(cudaMemcpyAsync(bounds, init, sizeof(init), cudaMemcpyHostToDevice, s));
  }
  {
    const int blocks = (int)std::min<int64_t>((n + 255) / 256, 2 * F.ctx.sm_count);
    k_bounds<<<blocks, 256, 0, s>>>(F.box_orig, F.rec_orig, n, bounds);
    GF_TRY(cudaGetLastError());
    if (F.opts.precision != GF_PREC_FP32) {
      // grow the boxes by the mean's quantisation step, then take the bounds again
      k_pad_mean_step<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(F.box_orig, n, bounds);
      GF_TRY(cudaGetLastError());
      unsigned int init[12];
      for (int j = 0; j < 12; ++j) init[j] = ((j < 3) || (j >= 6 && j < 9)) ? 0xFFFFFFFFu : 0u;
      GF_TRY(cudaMemcpyAsync(bounds, init, sizeof(init), cudaMemcpyHostToDevice, s));
      k_bounds<<<blocks, 256, 0, s>>>(F.box_orig, F.rec_orig, n, bounds);
      GF_TRY(cudaGetLastError());
    }
    k_morton<<<pn, 256, 0, s>>>(F.rec_orig, F.box_orig, n, bounds, keys, idx, head->area);
    GF_TRY(cudaGetLastError());
  }
  GF_TRY(cub::DeviceRadixSort::SortPairs(tmp, tmp_bytes, keys, keys2, idx, idx2, (int)(2 * n), 0, 37, s));
  k_gather<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(F.rec_orig, F.box_orig, F.ext2_orig, idx2,
                                                      n, F.rec, box_sorted, F.ext2, F.muw,
                                                      F.sorted_orig, pos);
  GF_TRY(cudaGetLastError());
  {
    // the binary trees by cells (kept) and by bands with their boxes, the marks of their
    // four-wide nodes (flags) and the marks' scan (map)
    int last[3] = {0, 0, 0};  // marks before the second tree's; of the last node, scan and mark
    const dim3 gn(pn, 2), gm(pm, 2);
    if (n >= 2) {
      k_band_leaves<<<pn, 256, 0, s>>>(idx2, pos, n, of);
      GF_TRY(cudaGetLastError());
      const TreePair T{{{keys2, F.nodes, above, flags, nullptr, bounds + 12, false},
                        {keys2 + n, nodes_b, above_b, flags + m, of, bounds + 13, true}}};
      GF_TRY(cudaMemsetAsync(flags, 0, 2 * m * sizeof(int), s));
      k_karras<<<gm, 256, 0, s>>>(T, n);
      GF_TRY(cudaGetLastError());
      k_refit<<<gn, 256, 0, s>>>(box_sorted, F.rec, T, n);
      GF_TRY(cudaGetLastError());
      k_depth_parity<<<gm, 256, 0, s>>>(T, m);
      GF_TRY(cudaGetLastError());
      GF_TRY(cub::DeviceScan::ExclusiveSum(tmp, tmp_bytes, flags, map, (int)(2 * m), s));
      GF_TRY(cudaMemcpyAsync(&last[0], map + m, sizeof(int), cudaMemcpyDeviceToHost, s));
      GF_TRY(cudaMemcpyAsync(&last[1], map + 2 * m - 1, sizeof(int), cudaMemcpyDeviceToHost, s));
      GF_TRY(cudaMemcpyAsync(&last[2], flags + 2 * m - 1, sizeof(int), cudaMemcpyDeviceToHost, s));
    }
    GF_TRY(cudaStreamSynchronize(s));
    // nodes4: the cells' trees, the cells' one-primitive roots, then the same of the bands
    const int ma = last[0], mb = last[1] + last[2] - last[0];
    const int single_b = ma + kMaxCells + mb;
    F.n_nodes4 = (int64_t)single_b + 8;
    F.mem.release(F.nodes4, s);  // a rebuild (the stream was synchronised above)
    F.nodes4 = nullptr;
    GF_TRY(F.mem.alloc((void**)&F.nodes4, (size_t)F.n_nodes4 * sizeof(Node4), s));
    if (n >= 2) {
      k_collapse4<<<gm, 256, 0, s>>>(
          CollapsePair{{{F.nodes, m, flags, map, nullptr, F.nodes4, 0, ma, roots},
                        {nodes_b, m, flags + m, map + m, of, F.nodes4, kMaxCells, single_b, roots + kMaxCells}}});
    } else {
      k_single4<<<1, 1, 0, s>>>(box_sorted, F.rec, false, F.nodes4, 0, roots);
      k_single4<<<1, 1, 0, s>>>(box_sorted, F.rec, true, F.nodes4, single_b, roots + kMaxCells);
    }
    GF_TRY(cudaGetLastError());
  }
  GF_TRY(cudaMemcpyAsync(hroots, roots, sizeof(hroots), cudaMemcpyDeviceToHost, s));
  GF_TRY(cudaMemcpyAsync(&hh, head, sizeof(hh), cudaMemcpyDeviceToHost, s));
  GF_TRY(cudaStreamSynchronize(s));
  {
    auto dec = [](unsigned int u) {
      unsigned int b = (u & 0x80000000u) ? (u & 0x7FFFFFFFu) : ~u;
      float f;
      memcpy(&f, &b, 4);
      return f;
    };
    // levels of internal nodes (0 for a single primitive) of the deeper tree.  (By bands
    // the keys are 3 bits shorter and runs of equal keys below 2^26 primitives.)
    F.depth = (int)std::max(hb[12], hb[13]) + 1;
    if (n < 2) F.depth = 0;
    F.dev.lo = make_float3(dec(hb[0]), dec(hb[1]), dec(hb[2]));
    F.dev.hi = make_float3(dec(hb[3]), dec(hb[4]), dec(hb[5]));
    // a convex body of mean projected area a in a volume V is crossed a / V times per unit
    // length; an ellipsoid's is about pi / 12 of its box's face areas.  V: the box of the
    // means, which holds the bodies but for the margins around it
    const float x = F.dev.hi.x - F.dev.lo.x, y = F.dev.hi.y - F.dev.lo.y, z = F.dev.hi.z - F.dev.lo.z;
    const double V = (double)fmaxf(dec(hb[9]) - dec(hb[6]), 0.5f * x) * fmaxf(dec(hb[10]) - dec(hb[7]), 0.5f * y) *
                     fmaxf(dec(hb[11]) - dec(hb[8]), 0.5f * z);
    const double per = 3.14159265358979323846 / 12.0 * kAreaUnit * face_areas(x, y, z) / V;
    for (int b = 0; b < 8; ++b) {
      const unsigned long long cones = b == 0 ? F.dev.occupied & 1ull : F.dev.occupied >> (1 + kCones * (b - 1)) & 0xFFull;
      const int k = __builtin_popcountll(cones);
      F.dev.chords[b] = k && hh.area[b] ? (float)(per * (double)hh.area[b] / k) : 0.f;
    }
    for (int k = 0; k < 3; ++k) {
      F.mu_lo[k] = dec(hb[6 + k]);
      F.mu_hi[k] = dec(hb[9 + k]);
    }
  }
  F.dev.rec = F.rec;
  // read by the reduced-precision path (FP32 records carry their own); without
  // adaptive clamping every support radius is k_sigma and none is read
  F.dev.ext2 = F.opts.clamp_eps > 0.f ? F.ext2 : nullptr;
  F.dev.nodes = F.nodes;
  F.dev.nodes4 = F.nodes4;
  F.dev.n_nodes4 = F.n_nodes4;
  // an empty class's root is never started from; node 0 stands in
  for (int c = 0; c < kMaxCells; ++c) F.dev.croot[c] = std::max(0, hroots[c]);
  for (int b = 0; b < 8; ++b) F.dev.broot[b] = std::max(0, hroots[kMaxCells + b]);
  F.dev.root = n >= 2 ? 0 : -1;
done:
#undef GF_TRY
  cudaStreamSynchronize(s);  // the temporaries are no longer read
  F.mem.release(block, s);
  return e;
}

// ---------------------------------------------------------------------------
// reduced-precision records (layout in gf_device.cuh), BVH order
// ---------------------------------------------------------------------------
struct Pack16Args {
  const float *mu, *quat, *ls, *om, *ph, *w;
  const uint8_t* cell;  // per original index
  const int* sorted_orig;
  int64_t n;
  int prec, omega_frame, weight_mode;
  float3 lo, scale;
  uint4* out;
  int* err;
};

__device__ __forceinline__ uint32_t to_half_bits(float x, int prec) {
  return prec == GF_PREC_BF16 ? (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(x))
                              : (uint32_t)__half_as_ushort(__float2half_rn(x));
}

__global__ void k_pack16(const __grid_constant__ Pack16Args A) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= A.n) return;
  const int64_t i = A.sorted_orig[j];
  uint32_t mc[3];
  const float lo[3] = {A.lo.x, A.lo.y, A.lo.z}, sc[3] = {A.scale.x, A.scale.y, A.scale.z};
  for (int k = 0; k < 3; ++k) {
    const float c = rintf((A.mu[3 * i + k] - lo[k]) / sc[k]);
    mc[k] = (uint32_t)fminf(fmaxf(c, 0.f), 65535.f);
  }
  float q[4];
  float qn = 0.f;
  for (int k = 0; k < 4; ++k) {
    q[k] = A.quat[4 * i + k];
    qn += q[k] * q[k];
  }
  qn = rsqrtf(qn);
  float s[3];
  for (int k = 0; k < 3; ++k) s[k] = expf(A.ls[3 * i + k]);
  const float w = q[0] * qn, x = q[1] * qn, y = q[2] * qn, z = q[3] * qn;
  const float R[3][3] = {{1.f - 2.f * (y * y + z * z), 2.f * (x * y - w * z), 2.f * (x * z + w * y)},
                         {2.f * (x * y + w * z), 1.f - 2.f * (x * x + z * z), 2.f * (y * z - w * x)},
                         {2.f * (x * z - w * y), 2.f * (y * z + w * x), 1.f - 2.f * (x * x + y * y)}};
  // whitened carrier in the frame of W = S^-1 R^T
  float kl[3];
  for (int k = 0; k < 3; ++k) {
    if (A.omega_frame == GF_OMEGA_LOCAL) {
      kl[k] = A.om[3 * i + k];
    } else {
      kl[k] = s[k] * (R[0][k] * A.om[3 * i] + R[1][k] * A.om[3 * i + 1] + R[2][k] * A.om[3 * i + 2]);
    }
  }
  // W = Q T (modified Gram-Schmidt on W's columns, W_kj = R_jk / s_k): then
  // T^T T = W^T W = Sigma^-1, T is upper triangular with T_kk > 0, and the
  // carrier in T's frame is Q^T times the one in W's frame (omega . z =
  // k_W . W z = (Q^T k_W) . T z)
  float c[3][3];  // c[j]: column j of W
  for (int j = 0; j < 3; ++j)
    for (int k = 0; k < 3; ++k) c[j][k] = R[j][k] / s[k];
  float T[3][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
  for (int j = 0; j < 3; ++j) {
    for (int r = 0; r < j; ++r) {
      const float d = c[r][0] * c[j][0] + c[r][1] * c[j][1] + c[r][2] * c[j][2];
      T[r][j] = d;
      for (int k = 0; k < 3; ++k) c[j][k] -= d * c[r][k];
    }
    const float nrm = sqrtf(c[j][0] * c[j][0] + c[j][1] * c[j][1] + c[j][2] * c[j][2]);
    T[j][j] = nrm;
    for (int k = 0; k < 3; ++k) c[j][k] /= nrm;  // c[j] is now q_j
  }
  float kw[3];
  for (int j = 0; j < 3; ++j) kw[j] = c[j][0] * kl[0] + c[j][1] * kl[1] + c[j][2] * kl[2];
  // one power of two for T: its largest entry scaled into [0.5, 1)
  const float tmax = fmaxf(fmaxf(fmaxf(T[0][0], fabsf(T[0][1])), fmaxf(fabsf(T[0][2]), T[1][1])),
                           fmaxf(fabsf(T[1][2]), T[2][2]));
  int E = 0;
  (void)frexpf(tmax, &E);
  if (E < -126 || E > 127) atomicOr(A.err, ERR_INPUT);
  E = E < -126 ? -126 : (E > 127 ? 127 : E);
  float amp = A.w[i];
  if (A.weight_mode == GF_WEIGHT_NORMALIZED) amp = amp / (15.749609945722419f * s[0] * s[1] * s[2]);
  if (A.prec == GF_PREC_FP16 && !(fabsf(amp) <= 65504.f && fabsf(kw[0]) <= 65504.f &&
                                  fabsf(kw[1]) <= 65504.f && fabsf(kw[2]) <= 65504.f))
    atomicOr(A.err, ERR_INPUT);
  float ph = fmodf(A.ph[i], 6.28318530717958647692f);
  if (ph < 0.f) ph += 6.28318530717958647692f;
  const uint32_t pc = (uint32_t)rintf(ph * (65536.0f / 6.28318530717958647692f)) & 0xFFFFu;
  const uint32_t cell = A.cell[i];
  auto th = [&](float v) { return to_half_bits(ldexpf(v, -E), A.prec); };
  uint4 r0, r1;
  r0.x = mc[0] | (mc[1] << 16);
  r0.y = mc[2] | (th(T[0][0]) << 16);
  r0.z = th(T[0][1]) | (th(T[0][2]) << 16);
  r0.w = th(T[1][1]) | (th(T[1][2]) << 16);
  r1.x = th(T[2][2]) | (to_half_bits(kw[0], A.prec) << 16);
  r1.y = to_half_bits(kw[1], A.prec) | (to_half_bits(kw[2], A.prec) << 16);
  r1.z = to_half_bits(amp, A.prec) | (pc << 16);
  r1.w = (cell & 63u) | ((uint32_t)(E + 127) << 8);
  A.out[2 * j] = r0;
  A.out[2 * j + 1] = r1;
}

cudaError_t launch_pack16(Field& F, cudaStream_t s) {
  (void)cudaGetLastError();  // a stale error of an unrelated call is not ours
  Pack16Args A;
  A.mu = F.p_mu;
  A.quat = F.p_quat;
  A.ls = F.p_ls;
  A.om = F.p_om;
  A.ph = F.p_ph;
  A.w = F.p_w;
  A.cell = F.labels + 2 * F.n;
  A.sorted_orig = F.sorted_orig;
  A.n = F.n;
  A.prec = F.opts.precision;
  A.omega_frame = F.opts.omega_frame;
  A.weight_mode = F.opts.weight_mode;
  float sc[3];
  for (int k = 0; k < 3; ++k) {
    const float ext = F.mu_hi[k] - F.mu_lo[k];
    sc[k] = ext > 0.f ? ext / 65535.f : 1.f;
  }
  A.lo = make_float3(F.mu_lo[0], F.mu_lo[1], F.mu_lo[2]);
  A.scale = make_float3(sc[0], sc[1], sc[2]);
  A.out = F.rec16;
  A.err = F.err;
  F.dev.qlo = A.lo;
  F.dev.qscale = A.scale;
  k_pack16<<<(unsigned)((F.n + 255) / 256), 256, 0, s>>>(A);
  return cudaGetLastError();
}

}  // namespace gf
