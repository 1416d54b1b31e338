// Depth-image integration and the TSDF adjoint.
//
// ohm_integrate_depth back-projects a z-depth image into rays on the device
// and integrates them (every layer of the map, Sec. II-F for TSDF).
//
// ohm_tsdf_backward gives the gradient of L = sum_q g_q D(v_q), D the TSDF
// distance right after the frame was integrated, with respect to the frame's
// per-pixel depths and its pose (a left twist xi = (rho, phi) moving every
// world point p to p + rho + phi x p), with the voxel sets of the band walks
// and the per-voxel counts held fixed.  It recomputes each pixel's band walk
// instead of storing traces.  For an unclamped s = (e - c).u:
//   ds/de = u + r_perp / d,  ds/do = -r_perp / d,  r = e - c,
//   r_perp = r - (r.u) u,  dD/ds = 1 / W   (W = the weight after the frame),
// so per ray, with w_v = G(v) / W(v) summed over its unclamped band voxels,
//   dL/de = (sum w) u + (sum w r_perp) / d,  dL/do = -(sum w r_perp) / d,
//   dL/dz = dL/de . R p~,  p~ = ((u - cx) / fx, (v - cy) / fy, 1),
//   dL/drho += dL/de + dL/do,  dL/dphi += e x dL/de + o x dL/do.
//
// ohm_integrate_posed moves sensor-frame rays to the world by a pose and
// integrates them; ohm_ndt_backward gives the gradient of
// L = sum_q gm_q . mean(v_q) + gc_q . packed C(v_q), mean and C the NDT-OM
// sample statistics (Sec. II-D, III-C) right after that frame, with respect to
// the frame's sensor-frame endpoints and its pose twist, the voxel of every
// sample held fixed.  With n, S the voxel's count and sum of sample positions
// p (relative to its corner) and d = p_j - S / n,
//   dL/dp_j = (1 / n) [ gm + (G + G^T) d ],  G = upper-triangular(gc),
// then dL/de_sensor = R^T dL/dp_j and the twist as for the TSDF.
#include <algorithm>
#include <cstring>
#include <string>
#include <vector>

#include "ohm_kernels.cuh"

namespace ohm {
namespace {

struct DepthFrame {
  const float* depth;
  int32_t width, height;
  double fx, fy, cx, cy;
  double R[9];
  double t[3];
  double z_min, z_max;
  float z_lo, z_hi;   // the largest floats up to z_min and z_max: a float z has z > z_min iff z > z_lo
  FF Rf[9], tf[3], zf_max;  // R, t and z_max as float-float
  const double* pxy;  // (u - cx) / fx for u < width, then (v - cy) / fy for v < height
  const float2* pxyf; // the same as float-float (hi, lo)
};

// Pixel of the i-th thread of a frame, so that a warp holds an 8 x 4 tile: its
// rays stay within a voxel or two of one another, where 32 pixels of a row
// spread over several (the TSDF walk then has more voxels per step to update).
// Rows in bands of 4 (the last may be lower), columns in tiles of 8, the
// columns left over behind them.
__device__ __forceinline__ long long tile_pixel(long long p, int width, int height) {
  if ((long long)width * height >= (1LL << 31) || width >= (1 << 28)) return p;  // row by row (32-bit indices)
  const int i = (int)p;
  const int band = i / (4 * width), rows = height - 4 * band < 4 ? height - 4 * band : 4;
  const int t = i - band * 4 * width, tiles = width / 8, in_tiles = tiles * 8 * rows;
  int row, col;
  if (t < in_tiles) {
    const int tile = t / (8 * rows), r = t - tile * 8 * rows;
    row = r / 8;
    col = tile * 8 + (r & 7);
  } else {
    const int rest = width - 8 * tiles, r = t - in_tiles;
    row = r / rest;
    col = 8 * tiles + r - row * rest;
  }
  return (long long)(4 * band + row) * width + col;
}

// Back-projection of one pixel, one rounding per double operation:
// x = ((u - cx) / fx) z, y = ((v - cy) / fy) z, e_k = ((R_k0 x + R_k1 y) + R_k2 z) + t_k,
// rounded to float.  A depth outside (z_min, z_max] gives a NO_RETURN ray at z_max.
// The quotients depend on the column or the row only: they come from the
// frame's table, formed on the host by the same double operations.
//
// Evaluated in float-float first: with S_k = |R_k0 x| + |R_k1 y| + |R_k2 z| +
// |t_k|, x and y are good to 6 u^2 (their quotient's 48 bits and one product),
// the products by R to 13 u^2, and the three additions and t add 10 u^2 S_k; the
// double evaluation is within 2^-50 S_k. The float is taken when no midpoint
// between floats lies within 2^-41 S_k = 128 u^2 S_k; else the pixel is
// evaluated in double (20 double instructions, 64 scheduler cycles each).
__device__ __noinline__ void depth_ray_double(const DepthFrame& f, double px, double py, double zz, float e[3]) {
  const double x = __dmul_rn(px, zz), y = __dmul_rn(py, zz);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    double a = __dmul_rn(f.R[3 * k], x);
    a = __dadd_rn(a, __dmul_rn(f.R[3 * k + 1], y));
    a = __dadd_rn(a, __dmul_rn(f.R[3 * k + 2], zz));
    a = __dadd_rn(a, f.t[k]);
    e[k] = __double2float_rn(a);
  }
}
__device__ __forceinline__ bool depth_ray(const DepthFrame& f, long long pix, float e[3], float* px, float* py) {
  const int v = pix < (1LL << 31) ? (int)pix / f.width : (int)(pix / f.width);
  const int u = (int)(pix - (long long)v * f.width);
  const float z = f.depth[pix];
  const bool valid = z > f.z_lo && z <= f.z_hi;
  const float2 qx = f.pxyf[u], qy = f.pxyf[f.width + v];
  const FF X = {qx.x, qx.y}, Y = {qy.x, qy.y}, Z = valid ? FF{z, 0.0f} : f.zf_max;
  const FF x = ff_mul(X, Z), y = ff_mul(Y, Z);
  bool settled = true;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const FF a = ff_mul(f.Rf[3 * k], x), b = ff_mul(f.Rf[3 * k + 1], y), c = ff_mul(f.Rf[3 * k + 2], Z);
    const FF s = ff_add(ff_add(ff_add(a, b), c), f.tf[k]);
    const float S = fabsf(a.hi) + fabsf(b.hi) + fabsf(c.hi) + fabsf(f.tf[k].hi);
    settled = ff_to_float(s, 4.547474e-13f * S, &e[k]) && S < 1e18f && settled;
  }
  if (!settled) depth_ray_double(f, f.pxy[u], f.pxy[f.width + v], valid ? (double)z : f.z_max, e);
  *px = qx.x;
  *py = qy.x;
  return valid;
}

__global__ void __launch_bounds__(kBlock) k_depth_rays(DepthFrame f, float* origins, float* endpoints, uint8_t* flags) {
  const long long n = (long long)f.width * f.height;
  if (blockIdx.x == 0 && threadIdx.x < 3) origins[threadIdx.x] = __double2float_rn(f.t[threadIdx.x]);
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += (long long)gridDim.x * blockDim.x) {
    float e[3], px, py;
    const bool valid = depth_ray(f, tile_pixel(p, f.width, f.height), e, &px, &py);
    endpoints[3 * p + 0] = e[0];
    endpoints[3 * p + 1] = e[1];
    endpoints[3 * p + 2] = e[2];
    flags[p] = valid ? 0 : kFlagNoReturn;
  }
}

__device__ __forceinline__ long long point_offset(const DeviceMap& m, const float* p) {
  long long q[3];
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 3; ++k) ok = quantise_coord(m, p[k], k, &q[k]) && ok;
  ok = ok && in_extent(q, m.frac_bits);
  if (!ok) return -1;
  const int F = m.frac_bits;
  const int32_t vx = (int32_t)(q[0] >> F), vy = (int32_t)(q[1] >> F), vz = (int32_t)(q[2] >> F);
  const int32_t slot = region_slot_of(m, vx, vy, vz);
  return slot < 0 ? -1 : voxel_offset(slot, local_morton(vx, vy, vz));
}

// Rows of upstream weights.  The queries that fall into one voxel share a row
// of doubles, claimed by the first of them to arrive; `plane` holds the row
// plus one of every voxel, 0 for none and between calls.  The sums are double
// because the order in which queries arrive differs from run to run: in float
// that moved a weight by 6e-8 of itself, which the double twist shows; in double
// it is 1e-16.  A row per query, or per voxel where there are fewer of those.
__device__ __forceinline__ long long claim_row(uint32_t* plane, long long off, long long row) {
  uint32_t r = plane[off];
  if (r == 0u) {
    r = atomicCAS(plane + off, 0u, (uint32_t)row + 1u);
    if (r == 0u) r = (uint32_t)row + 1u;
  }
  return (long long)r - 1;
}

// The upstream weight G(v) of a voxel, the sum of g_q over the queries it
// holds, in three passes over the queries: add them up in rows of one double
// (row[q]: the row of query q; by_voxel: the voxel's own), put each voxel's sum
// into its word as a float, and, after the backward pass, zero everything.
// The backward pass reads a float per band voxel: with the row in the word and the
// sum behind it, the call took 102 us for a 640 x 480 frame at 5 cm and 130 at
// 2 cm; with the second pass 101 and 122, with the four kernels chained 99 and 118
// (float atomics straight into the words: 94 and 115).
enum GradPass { kGradAdd, kGradSettle, kGradClear };
template <GradPass kPass>
__global__ void __launch_bounds__(kBlock) k_grad_scatter(DeviceMap m, const float* pts, const float* g, long long n,
                                                         double* rows, uint32_t* row, int by_voxel) {
  chain_enter();
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
    const long long off = point_offset(m, pts + 3 * q);
    if (off < 0) continue;
    long long r = off;
    if (kPass == kGradAdd) {
      if (!by_voxel) row[q] = (uint32_t)(r = claim_row(m.grad, off, q));
      atomicAdd(rows + r, (double)g[q]);
      continue;
    }
    if (!by_voxel) r = row[q];
    if (kPass == kGradSettle) {
      m.grad[off] = __float_as_uint((float)rows[r]);
    } else {
      if (!by_voxel) row[q] = 0u;
      rows[r] = 0.0;
      m.grad[off] = 0u;
    }
  }
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Compiled for 2 blocks per SM (128 registers; 184 unbounded, which fits one;
// 3 and 4 blocks: no difference).  Bound by instruction issue.  The whole call for
// a 640 x 480 frame with 20,000 queries: 121 us with the double back-projection and
// the 64-bit walker, row by row; 99 us now.
__global__ void __launch_bounds__(kBlock, 2) k_tsdf_backward(DeviceMap m, DepthFrame f, float* grad_depth,
                                                          double* grad_twist) {
  chain_enter();
  __shared__ double red[kBlock / 32][6];
  __shared__ uint32_t tabs[8 * kBlock];
  uint32_t* const tab = tabs + threadIdx.x;
  const long long n = (long long)f.width * f.height;
  const int F = m.frac_bits;
  const float to_m = (float)(m.voxel_size / (double)(1LL << F));
  const float O[3] = {(float)f.t[0], (float)f.t[1], (float)f.t[2]};
  double acc[6] = {0, 0, 0, 0, 0, 0};
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += (long long)gridDim.x * blockDim.x) {
    const long long pix = tile_pixel(p, f.width, f.height);
    float gz = 0.f;
    float e[3], px, py;
    bool ok = depth_ray(f, pix, e, &px, &py);
    long long qo[3], qe[3], a[3], b[3];
    float u[3], lenf = 0.f;
    // the band of the forward pass, recomputed the same way
    ok = ok && quantise_ray(m, O, e, qo, qe) && tsdf_ray_band(m, qo, qe, a, b, u, &lenf);
    if (ok) {
      const float dm = lenf * to_m;  // ray length in metres (chain rule only)
      TsdfRec t;
      tsdf_record(a, b, qe, F, &t);
      const int M = (t.r.flags >> kRayAxisShift) & 3;
      const int32_t nmaj = M == 0 ? t.r.n[0] : (M == 1 ? t.r.n[1] : t.r.n[2]);
      float A = 0.f, B[3] = {0.f, 0.f, 0.f};
      // up to the first voxel whose region the map does not hold (moved to the
      // host since the frame, or the frame was never integrated)
      int32_t left = 0;
      for (int32_t K = 0; K <= nmaj && left != kWalkEnded; K += kPieceSlots) {
        const int32_t Ke = K + kPieceSlots < nmaj + 1 ? K + kPieceSlots : nmaj + 1;
        PieceStart ps;
        LWalker w;
        uint32_t mo;
        piece_start(t.r, F, K, Ke, Ke == nmaj + 1, &ps, &w);
        if (!piece_regions<true>(m, ps, w, t.r.flags, tab, &mo)) break;
        int32_t rel[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) rel[k] = t.e[k] - ((ps.v[k] - t.r.v0[k]) << F);
        for (left = ps.visits; left > 0;) {
          uint32_t at[kFastBatch], off[kFastBatch], valid;
          float G[kFastBatch];
          piece_fill<true>(m, &t.r, K, tab, w, mo, left, at, off, valid);
#pragma unroll
          for (int j = 0; j < kFastBatch; ++j) G[j] = ((valid >> j) & 1u) ? __uint_as_float(m.grad[off[j]]) : 0.f;
#pragma unroll
          for (int j = 0; j < kFastBatch; ++j) {
            if (G[j] != 0.f) {
              const float ex = (float)rel[0], ey = (float)rel[1], ez = (float)rel[2];
              const float s = (ex * u[0] + ey * u[1] + ez * u[2]) * to_m;  // as in the forward pass
              if (s > -m.tau_m && s < m.tau_m) {
                const float wv = G[j] / m.tsdf[off[j]].y;
                const float r[3] = {ex * to_m, ey * to_m, ez * to_m};
                A += wv;
#pragma unroll
                for (int k = 0; k < 3; ++k) B[k] += wv * (r[k] - s * u[k]);
              }
            }
            const uint32_t moved = at[j] ^ (j + 1 < kFastBatch ? at[j + 1] : mo);
            const int k = (moved & 0x9249u) ? 0 : ((moved & 0x12492u) ? 1 : 2);
            const int32_t d = ((t.r.flags >> (kRaySignShift + k)) & 1) ? 1 << F : -(1 << F);
            rel[0] += k == 0 ? d : 0;
            rel[1] += k == 1 ? d : 0;
            rel[2] += k == 2 ? d : 0;
          }
        }
      }
      // The chain rule from here on is plain float arithmetic (its inputs
      // are floats; the gradients are checked to 1e-3 relative), summed
      // over pixels in double.  The band above is recomputed exactly as
      // the forward pass forms it, since it decides the voxel set.
      const float rdm = 1.0f / dm;
      float ge[3], go[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        go[k] = -B[k] * rdm;
        ge[k] = A * u[k] - go[k];
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) gz += ge[k] * (f.Rf[3 * k].hi * px + f.Rf[3 * k + 1].hi * py + f.Rf[3 * k + 2].hi);
#pragma unroll
      for (int k = 0; k < 3; ++k) acc[k] += (double)(ge[k] + go[k]);
      acc[3] += (double)(e[1] * ge[2] - e[2] * ge[1] + O[1] * go[2] - O[2] * go[1]);
      acc[4] += (double)(e[2] * ge[0] - e[0] * ge[2] + O[2] * go[0] - O[0] * go[2]);
      acc[5] += (double)(e[0] * ge[1] - e[1] * ge[0] + O[0] * go[1] - O[1] * go[0]);
    }
    grad_depth[pix] = gz;
  }
  // block reduction of the twist gradient, one double atomic per component
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const double v = warp_sum(acc[k]);
    if (lane == 0) red[wid][k] = v;
  }
  __syncthreads();
  if (threadIdx.x < 6) {
    double v = 0.0;
    for (int i = 0; i < kBlock / 32; ++i) v += red[i][threadIdx.x];
    atomicAdd(grad_twist + threadIdx.x, v);
  }
}

// A camera-to-world pose [R | t], row major.
struct Pose34 {
  double m[12];
};

// p_k = ((R_k0 x + R_k1 y) + R_k2 z) + t_k in double, one rounding per
// operation, rounded to float (the depth back-projection's order).
__device__ __forceinline__ void pose_point(const Pose34& P, const float* in, float* out) {
  const double x = in[0], y = in[1], z = in[2];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    double a = __dmul_rn(P.m[4 * k], x);
    a = __dadd_rn(a, __dmul_rn(P.m[4 * k + 1], y));
    a = __dadd_rn(a, __dmul_rn(P.m[4 * k + 2], z));
    out[k] = __double2float_rn(__dadd_rn(a, P.m[4 * k + 3]));
  }
}

__global__ void __launch_bounds__(kBlock) k_pose_rays(Pose34 P, CallArgs in, float* origins, float* endpoints,
                                                      uint8_t* flags) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < in.n; i += (long long)gridDim.x * blockDim.x) {
    pose_point(P, in.endpoints + 3 * i, endpoints + 3 * i);
    if (i < in.n_origins) pose_point(P, in.origins + 3 * i, origins + 3 * i);
    flags[i] = in.flags ? in.flags[i] : 0;
  }
}

// Index of the NDT voxel holding a point (block * 32768 + Morton index), -1:
// outside the map or in a region without samples (nothing to differentiate).
__device__ __forceinline__ long long ndt_point_offset(const DeviceMap& m, const float* p) {
  long long q[3];
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 3; ++k) ok = quantise_coord(m, p[k], k, &q[k]) && ok;
  ok = ok && in_extent(q, m.frac_bits);
  if (!ok) return -1;
  const int F = m.frac_bits;
  const int32_t vx = (int32_t)(q[0] >> F), vy = (int32_t)(q[1] >> F), vz = (int32_t)(q[2] >> F);
  const int32_t slot = region_slot_of(m, vx, vy, vz);
  const int32_t ns = slot < 0 ? -1 : m.ndt_slot[slot];
  return ns < 0 ? -1 : voxel_offset(ns, local_morton(vx, vy, vz));
}

// The upstream weights of a voxel (mean x y z, covariance xx xy xz yy yz zz),
// summed over the queries it holds: a row of 9 doubles, added to for each
// query point, or (clear) zeroed and forgotten.
__global__ void __launch_bounds__(kBlock) k_ndt_grad_scatter(DeviceMap m, const float* pts, const float* gmean,
                                                             const float* gcov, long long n, double* rows,
                                                             int by_voxel, int clear) {
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
    const long long off = ndt_point_offset(m, pts + 3 * q);
    if (off < 0) continue;
    if (clear) {
      const uint32_t row = m.ndt_grad_row[off];  // 0: another query of the voxel was here
#pragma unroll
      for (int k = 0; k < 9; ++k)
        if (row) rows[9LL * (row - 1u) + k] = 0.0;
      m.ndt_grad_row[off] = 0u;
      continue;
    }
    double* g = rows + 9 * claim_row(m.ndt_grad_row, off, by_voxel ? off : q);
#pragma unroll
    for (int k = 0; k < 9; ++k) atomicAdd(g + k, (double)(k < 3 ? gmean[3 * q + k] : gcov[6 * q + k - 3]));
  }
}

// Per ray of the frame (world rays in `a`, as integrated): the sample's voxel
// by the quantisation and truncation of the forward pass, then dL/dp from the
// voxel's moments and weights.
__global__ void __launch_bounds__(kBlock) k_ndt_backward(DeviceMap m, CallArgs a, Pose34 P, const double* rows,
                                                         float* grad_e, double* grad_twist) {
  __shared__ double red[kBlock / 32][6];
  const int F = m.frac_bits;
  const long long U = 1LL << F;
  const double cell = m.voxel_size / (double)U;
  double acc[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  const long long n = a.n;
  const long long nb = ((n + kBlock - 1) / kBlock) * kBlock;  // every thread of a block reaches the reduction
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nb; i += (long long)gridDim.x * blockDim.x) {
    if (i >= n) continue;
    double gp[3] = {0.0, 0.0, 0.0};
    float o[3], e[3];
    uint8_t flag;
    load_ray(a, i, o, e, &flag);
    long long qo[3], qe[3];
    bool ok = (flag & kFlagNoReturn) == 0 && quantise_ray(m, o, e, qo, qe);
    if (ok) {
      double d[3];
      ok = ray_length(qo, qe, d) <= m.rmax_q && in_extent(qo, F) && in_extent(qe, F);
    }
    if (ok) {
      const int32_t v[3] = {(int32_t)(qe[0] >> F), (int32_t)(qe[1] >> F), (int32_t)(qe[2] >> F)};
      const int32_t slot = region_slot_of(m, v[0], v[1], v[2]);
      const int32_t ns = slot < 0 ? -1 : m.ndt_slot[slot];
      if (ns < 0) {
        // no end kernel follows: the host's word is written here
        const int32_t status = atomicOr(m.status, kStatusMissing);
        if (!(status & kStatusMissing)) *(volatile int32_t*)m.host_status = status | kStatusMissing;
      } else {
        const uint32_t mo = local_morton(v[0], v[1], v[2]);
        const uint32_t row = m.ndt_grad_row[voxel_offset(ns, mo)];  // 0: no query fell into the voxel
        double w[9];
        bool any = false;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
          w[k] = row ? rows[9LL * (row - 1u) + k] : 0.0;
          any = any || w[k] != 0.0;
        }
        const long long* mom = ndt_moments(m, ns, mo);
        const double cnt = (double)mom[0];
        if (any && cnt > 0.0) {
          double dv[3];
#pragma unroll
          for (int k = 0; k < 3; ++k)
            dv[k] = (double)(qe[k] - (long long)v[k] * U) * cell - (double)mom[1 + k] * cell / cnt;
          // (G + G^T) d with G upper triangular from the packed xx xy xz yy yz zz
          const double Gs[3][3] = {{2.0 * w[3], w[4], w[5]}, {w[4], 2.0 * w[6], w[7]}, {w[5], w[7], 2.0 * w[8]}};
#pragma unroll
          for (int k = 0; k < 3; ++k) gp[k] = (w[k] + Gs[k][0] * dv[0] + Gs[k][1] * dv[1] + Gs[k][2] * dv[2]) / cnt;
        }
      }
    }
    // sensor frame: dL/de = R^T dL/dp
#pragma unroll
    for (int c = 0; c < 3; ++c)
      grad_e[3 * i + c] = (float)(P.m[c] * gp[0] + P.m[4 + c] * gp[1] + P.m[8 + c] * gp[2]);
    const double E[3] = {e[0], e[1], e[2]};
#pragma unroll
    for (int k = 0; k < 3; ++k) acc[k] += gp[k];
    acc[3] += E[1] * gp[2] - E[2] * gp[1];
    acc[4] += E[2] * gp[0] - E[0] * gp[2];
    acc[5] += E[0] * gp[1] - E[1] * gp[0];
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const double v = warp_sum(acc[k]);
    if (lane == 0) red[wid][k] = v;
  }
  __syncthreads();
  if (threadIdx.x < 6) {
    double v = 0.0;
    for (int i = 0; i < kBlock / 32; ++i) v += red[i][threadIdx.x];
    atomicAdd(grad_twist + threadIdx.x, v);
  }
}

bool frame_from(const float* depth, int32_t width, int32_t height, const double* K, const double* pose, double z_min,
                double z_max, DepthFrame* f) {
  if (!depth || width < 1 || height < 1 || !K || !pose || !(z_max > z_min)) return false;
  f->depth = depth;
  f->width = width;
  f->height = height;
  f->fx = K[0];
  f->fy = K[1];
  f->cx = K[2];
  f->cy = K[3];
  for (int r = 0; r < 3; ++r) {
    for (int c = 0; c < 3; ++c) f->R[3 * r + c] = pose[4 * r + c];
    f->t[r] = pose[4 * r + 3];
  }
  f->z_min = z_min;
  f->z_max = z_max;
  auto below = [](double z) {  // the largest float not above z
    float r = (float)z;
    return (double)r > z ? std::nextafter(r, -INFINITY) : r;
  };
  f->z_lo = below(z_min);
  f->z_hi = below(z_max);
  for (int k = 0; k < 9; ++k) f->Rf[k] = ff_of_double(f->R[k]);
  for (int k = 0; k < 3; ++k) f->tf[k] = ff_of_double(f->t[k]);
  f->zf_max = ff_of_double(z_max);
  f->pxy = nullptr;
  f->pxyf = nullptr;
  return f->fx != 0.0 && f->fy != 0.0;
}

// The frame's per-column and per-row quotients, kept on the device for the
// last image size and intrinsics (rebuilt when they change).
cudaError_t frame_tables(ohm_map* map, DepthFrame* f, cudaStream_t s) {
  const double key[6] = {(double)f->width, (double)f->height, f->fx, f->fy, f->cx, f->cy};
  const long long n = (long long)f->width + f->height;  // doubles, then as many float pairs
  if (map->pxy && std::memcmp(key, map->pxy_key, sizeof(key)) == 0) {
    f->pxy = map->pxy;
    f->pxyf = reinterpret_cast<const float2*>(map->pxy + n);
    return cudaSuccess;
  }
  // earlier work of the map may still read the old table
  cudaError_t e = map->work_done ? cudaStreamWaitEvent(s, map->work_done, 0) : cudaSuccess;
  if (e == cudaSuccess && 2 * n > map->pxy_cap) {
    if (map->pxy) {
      e = cudaStreamSynchronize(s);
      if (e == cudaSuccess) e = cudaFree(map->pxy);
      map->pxy = nullptr;
      map->pxy_cap = 0;
    }
    const long long cap = 2 * n > 8192 ? 2 * n : 8192;
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&map->pxy), sizeof(double) * cap);
    if (e != cudaSuccess) return e;
    map->pxy_cap = cap;
  }
  if (e != cudaSuccess) return e;
  std::vector<double> t((size_t)(2 * n));
  for (int u = 0; u < f->width; ++u) t[u] = ((double)u - f->cx) / f->fx;
  for (int v = 0; v < f->height; ++v) t[f->width + v] = ((double)v - f->cy) / f->fy;
  for (long long k = 0; k < n; ++k) {
    const FF q = ff_of_double(t[(size_t)k]);
    const float pair[2] = {q.hi, q.lo};
    std::memcpy(&t[(size_t)(n + k)], pair, sizeof(pair));
  }
  e = cudaMemcpyAsync(map->pxy, t.data(), sizeof(double) * 2 * n, cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return e;
  std::memcpy(map->pxy_key, key, sizeof(key));
  f->pxy = map->pxy;
  f->pxyf = reinterpret_cast<const float2*>(map->pxy + n);
  return cudaSuccess;
}

// Zeroed rows of `width` doubles for a backward call's queries (claim_row), one
// per query (and `extra` doubles behind them) or, where there are fewer, per
// voxel of the layer.  The buffer stays with the map and the clearing pass zeroes
// what the call used, so that a call costs no allocation and no fill (a pool
// allocation and a fill for each call took 12 to 30 us of 510).  It grows by
// doubling; a captured call that finds it too small takes memory that its graph
// then holds (`own`).
struct Rows {
  double* p = nullptr;
  int by_voxel = 0;
  bool own = false;
};
cudaError_t take_rows(RowBuffers& kept, long long n_query, long long voxels, int width, long long extra, cudaStream_t s,
                      Rows* r) {
  r->by_voxel = n_query > voxels ? 1 : 0;
  const long long need = r->by_voxel ? width * voxels : width * n_query + extra;
  if (need <= kept.cap) {
    r->p = kept.all.back();
    return cudaSuccess;
  }
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  cudaError_t e = cudaStreamIsCapturing(s, &capture);
  if (e != cudaSuccess) return e;
  double* p = nullptr;
  long long cap = need;
  if (capture != cudaStreamCaptureStatusNone) {
    e = cudaMallocAsync(reinterpret_cast<void**>(&p), sizeof(double) * (size_t)need, s);
    r->own = e == cudaSuccess;
  } else {
    cap = std::max(need, std::max(2 * kept.cap, 1LL << 16));
    e = cudaMalloc(reinterpret_cast<void**>(&p), sizeof(double) * (size_t)cap);
    if (e == cudaErrorMemoryAllocation && cap > need) {  // no room to grow ahead
      cudaGetLastError();
      cap = need;
      e = cudaMalloc(reinterpret_cast<void**>(&p), sizeof(double) * (size_t)cap);
    }
  }
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(p, 0, sizeof(double) * (size_t)cap, s);
  if (!r->own) {
    if (e != cudaSuccess) {
      cudaFree(p);
      return e;
    }
    kept.all.push_back(p);
    kept.cap = cap;
  }
  r->p = p;
  return e;
}
cudaError_t give_rows(const Rows& r, cudaStream_t s) { return r.own ? cudaFreeAsync(r.p, s) : cudaSuccess; }

ohm_status afail(ohm_status code, const std::string& msg) {
  set_last_error(msg);
  return code;
}

bool is_device(const void* p) {
  cudaPointerAttributes a;
  if (!p || cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace
}  // namespace ohm

extern "C" {

ohm_status ohm_integrate_depth(ohm_map* map, const float* depth, int32_t width, int32_t height,
                               const double* intrinsics, const double* pose, double z_min, double z_max,
                               void* stream) {
  using namespace ohm;
  if (!map) return afail(OHM_ERR_INVALID, "integrate_depth: map is NULL");
  DepthFrame f;
  if (!frame_from(depth, width, height, intrinsics, pose, z_min, z_max, &f))
    return afail(OHM_ERR_INVALID, "integrate_depth: bad image, intrinsics, pose or depth range");
  const long long n = (long long)width * height;
  if (n > map->p.max_rays) return afail(OHM_ERR_INVALID, "integrate_depth: width * height exceeds max_rays");
  if (!is_device(depth)) return afail(OHM_ERR_INVALID, "integrate_depth: depth must be device memory");
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != map->device) cudaSetDevice(map->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int blocks = (int)((n + kBlock - 1) / kBlock < 4096 ? (n + kBlock - 1) / kBlock : 4096);
  cudaError_t et = frame_tables(map, &f, s);
  if (et != cudaSuccess) {
    if (prev >= 0 && prev != map->device) cudaSetDevice(prev);
    return afail(OHM_ERR_CUDA, std::string("integrate_depth: ") + cudaGetErrorString(et));
  }
  k_depth_rays<<<blocks, kBlock, 0, s>>>(f, map->stage_origins, map->stage_endpoints, map->stage_flags);
  map->launches += 1;
  CallArgs a;
  a.origins = map->stage_origins;
  a.endpoints = map->stage_endpoints;
  a.flags = map->stage_flags;
  a.n = n;
  a.n_origins = 1;
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = launch_integrate(map, a, s);
  if (e == cudaSuccess) note_work(map, s);
  if (prev >= 0 && prev != map->device) cudaSetDevice(prev);
  if (e != cudaSuccess) return afail(OHM_ERR_CUDA, std::string("integrate_depth: ") + cudaGetErrorString(e));
  return OHM_OK;
}

ohm_status ohm_tsdf_backward(ohm_map* map, const float* depth, int32_t width, int32_t height,
                             const double* intrinsics, const double* pose, double z_min, double z_max,
                             const float* query_points, const float* grad_query, int64_t n_query, float* grad_depth,
                             double* grad_twist, void* stream) {
  using namespace ohm;
  if (!map) return afail(OHM_ERR_INVALID, "tsdf_backward: map is NULL");
  if (!(map->p.layers & OHM_LAYER_TSDF)) return afail(OHM_ERR_UNSUPPORTED, "tsdf_backward: map has no TSDF layer");
  DepthFrame f;
  if (!frame_from(depth, width, height, intrinsics, pose, z_min, z_max, &f))
    return afail(OHM_ERR_INVALID, "tsdf_backward: bad image, intrinsics, pose or depth range");
  if (n_query < 0 || (n_query > 0 && (!query_points || !grad_query)) || !grad_depth || !grad_twist)
    return afail(OHM_ERR_INVALID, "tsdf_backward: NULL buffer");
  const void* bufs[] = {depth, grad_depth, grad_twist};
  for (const void* b : bufs)
    if (!is_device(b)) return afail(OHM_ERR_INVALID, "tsdf_backward: buffers must be device memory");
  if (n_query > 0 && (!is_device(query_points) || !is_device(grad_query)))
    return afail(OHM_ERR_INVALID, "tsdf_backward: buffers must be device memory");
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != map->device) cudaSetDevice(map->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaSuccess;
  const long long voxels = (long long)map->p.max_regions * kRegionVoxels;
  if (!map->d.grad) {
    // upstream weights per voxel, allocated on the first backward call
    e = cudaMalloc(reinterpret_cast<void**>(&map->d.grad), sizeof(uint32_t) * (size_t)voxels);
    if (e == cudaSuccess) e = cudaMemsetAsync(map->d.grad, 0, sizeof(uint32_t) * (size_t)voxels, s);
  }
  const long long n = (long long)width * height;
  const int qb = (int)(n_query > 0 ? ((n_query + kBlock - 1) / kBlock < 4096 ? (n_query + kBlock - 1) / kBlock : 4096) : 0);
  const int pb = (int)((n + kBlock - 1) / kBlock < 4096 ? (n + kBlock - 1) / kBlock : 4096);
  if (e == cudaSuccess) e = frame_tables(map, &f, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(grad_twist, 0, 6 * sizeof(double), s);
  Rows rows;
  if (e == cudaSuccess && qb) e = take_rows(map->tsdf_rows, n_query, voxels, 1, (n_query + 1) / 2, s, &rows);
  uint32_t* const row = rows.p && !rows.by_voxel ? reinterpret_cast<uint32_t*>(rows.p + n_query) : nullptr;
  if (e == cudaSuccess && qb) {
    launch_chained(k_grad_scatter<kGradAdd>, qb, s, map->d, query_points, grad_query, n_query, rows.p, row, rows.by_voxel);
    launch_chained(k_grad_scatter<kGradSettle>, qb, s, map->d, query_points, grad_query, n_query, rows.p, row, rows.by_voxel);
    map->launches += 2;
  }
  if (e == cudaSuccess) {
    launch_chained(k_tsdf_backward, pb, s, map->d, f, grad_depth, grad_twist);
    map->launches += 1;
  }
  if (rows.p) {
    // whatever else failed: no row may outlive its call in the plane
    launch_chained(k_grad_scatter<kGradClear>, qb, s, map->d, query_points, grad_query, n_query, rows.p, row, rows.by_voxel);
    map->launches += 1;
    const cudaError_t ef = give_rows(rows, s);
    if (e == cudaSuccess) e = ef;
  }
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e == cudaSuccess) note_work(map, s);
  if (prev >= 0 && prev != map->device) cudaSetDevice(prev);
  if (e != cudaSuccess) return afail(OHM_ERR_CUDA, std::string("tsdf_backward: ") + cudaGetErrorString(e));
  return OHM_OK;
}

static ohm_status posed_args(ohm_map* map, const double* pose, const float* origins, int64_t n_origins,
                             const float* endpoints, const uint8_t* flags, int64_t n, const char* who,
                             ohm::Pose34* P) {
  using namespace ohm;
  if (!map || !pose) return afail(OHM_ERR_INVALID, std::string(who) + ": NULL map or pose");
  if (n < 0 || n > map->p.max_rays) return afail(OHM_ERR_INVALID, std::string(who) + ": n outside [0, max_rays]");
  if (n > 0 && (!origins || !endpoints || (n_origins != 1 && n_origins != n)))
    return afail(OHM_ERR_INVALID, std::string(who) + ": bad origins / endpoints");
  if (n > 0 && (!is_device(origins) || !is_device(endpoints) || (flags && !is_device(flags))))
    return afail(OHM_ERR_INVALID, std::string(who) + ": rays must be device memory");
  for (int k = 0; k < 12; ++k) {
    if (!std::isfinite(pose[k])) return afail(OHM_ERR_INVALID, std::string(who) + ": pose not finite");
    P->m[k] = pose[k];
  }
  return OHM_OK;
}

// Transform into the map's staging buffers; returns the call arguments.
static cudaError_t stage_posed(ohm_map* map, const ohm::Pose34& P, const float* origins, int64_t n_origins,
                               const float* endpoints, const uint8_t* flags, int64_t n, cudaStream_t s,
                               ohm::CallArgs* a) {
  using namespace ohm;
  CallArgs in;
  in.origins = origins;
  in.endpoints = endpoints;
  in.flags = flags;
  in.n = n;
  in.n_origins = n_origins;
  const int blocks = (int)((n + kBlock - 1) / kBlock < 4096 ? (n + kBlock - 1) / kBlock : 4096);
  k_pose_rays<<<blocks > 0 ? blocks : 1, kBlock, 0, s>>>(P, in, map->stage_origins, map->stage_endpoints,
                                                         map->stage_flags);
  map->launches += 1;
  a->origins = map->stage_origins;
  a->endpoints = map->stage_endpoints;
  a->flags = map->stage_flags;
  a->n = n;
  a->n_origins = n_origins;
  return cudaGetLastError();
}

ohm_status ohm_integrate_posed(ohm_map* map, const double* pose, const float* origins, int64_t n_origins,
                               const float* endpoints, const uint8_t* flags, int64_t n, void* stream) {
  using namespace ohm;
  Pose34 P;
  const ohm_status st = posed_args(map, pose, origins, n_origins, endpoints, flags, n, "integrate_posed", &P);
  if (st != OHM_OK || n == 0) return st;
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != map->device) cudaSetDevice(map->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  CallArgs a;
  cudaError_t e = stage_posed(map, P, origins, n_origins, endpoints, flags, n, s, &a);
  if (e == cudaSuccess) e = launch_integrate(map, a, s);
  if (e == cudaSuccess) note_work(map, s);
  if (prev >= 0 && prev != map->device) cudaSetDevice(prev);
  if (e != cudaSuccess) return afail(OHM_ERR_CUDA, std::string("integrate_posed: ") + cudaGetErrorString(e));
  return OHM_OK;
}

ohm_status ohm_ndt_backward(ohm_map* map, const double* pose, const float* origins, int64_t n_origins,
                            const float* endpoints, const uint8_t* flags, int64_t n, const float* query_points,
                            const float* grad_mean, const float* grad_cov, int64_t n_query, float* grad_endpoints,
                            double* grad_twist, void* stream) {
  using namespace ohm;
  Pose34 P;
  ohm_status st = posed_args(map, pose, origins, n_origins, endpoints, flags, n, "ndt_backward", &P);
  if (st != OHM_OK) return st;
  if (!(map->p.layers & OHM_LAYER_NDT)) return afail(OHM_ERR_UNSUPPORTED, "ndt_backward: map has no NDT layer");
  if (map->p.ndt_clear_below > -INFINITY)
    return afail(OHM_ERR_UNSUPPORTED, "ndt_backward: sample clearing changes the statistics discontinuously; "
                                      "the adjoint needs ndt_clear_below = -inf");
  if (n_query < 0 || (n_query > 0 && (!query_points || !grad_mean || !grad_cov)) || (n > 0 && !grad_endpoints) ||
      !grad_twist)
    return afail(OHM_ERR_INVALID, "ndt_backward: NULL buffer");
  if ((n > 0 && !is_device(grad_endpoints)) || !is_device(grad_twist) ||
      (n_query > 0 && (!is_device(query_points) || !is_device(grad_mean) || !is_device(grad_cov))))
    return afail(OHM_ERR_INVALID, "ndt_backward: buffers must be device memory");
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != map->device) cudaSetDevice(map->device);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaSuccess;
  const long long voxels = (long long)map->d.max_ndt * kRegionVoxels;
  if (!map->d.ndt_grad_row) {
    // rows of upstream weights per NDT voxel, allocated on the first backward call
    const size_t bytes = sizeof(uint32_t) * (size_t)voxels;
    e = cudaMalloc(reinterpret_cast<void**>(&map->d.ndt_grad_row), bytes);
    if (e == cudaSuccess) e = cudaMemsetAsync(map->d.ndt_grad_row, 0, bytes, s);
  }
  if (e == cudaSuccess) e = cudaMemsetAsync(grad_twist, 0, 6 * sizeof(double), s);
  const int qb = (int)(n_query > 0 ? ((n_query + kBlock - 1) / kBlock < 4096 ? (n_query + kBlock - 1) / kBlock : 4096) : 0);
  Rows rows;
  if (e == cudaSuccess && qb) e = take_rows(map->ndt_rows, n_query, voxels, 9, 0, s, &rows);
  if (e == cudaSuccess && qb) {
    k_ndt_grad_scatter<<<qb, kBlock, 0, s>>>(map->d, query_points, grad_mean, grad_cov, n_query, rows.p, rows.by_voxel, 0);
    map->launches += 1;
  }
  if (e == cudaSuccess && n > 0) {
    CallArgs a;
    e = stage_posed(map, P, origins, n_origins, endpoints, flags, n, s, &a);
    const int pb = (int)((n + kBlock - 1) / kBlock < 4096 ? (n + kBlock - 1) / kBlock : 4096);
    if (e == cudaSuccess) {
      k_ndt_backward<<<pb, kBlock, 0, s>>>(map->d, a, P, rows.p, grad_endpoints, grad_twist);
      map->launches += 1;
    }
  }
  if (rows.p) {
    // whatever else failed: no row may outlive its call in the plane
    k_ndt_grad_scatter<<<qb, kBlock, 0, s>>>(map->d, query_points, grad_mean, grad_cov, n_query, rows.p, rows.by_voxel, 1);
    map->launches += 1;
    const cudaError_t ef = give_rows(rows, s);
    if (e == cudaSuccess) e = ef;
  }
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e == cudaSuccess) note_work(map, s);
  if (prev >= 0 && prev != map->device) cudaSetDevice(prev);
  if (e != cudaSuccess) return afail(OHM_ERR_CUDA, std::string("ndt_backward: ") + cudaGetErrorString(e));
  return OHM_OK;
}

ohm_status ohm_twist_pose(const double* xi, const double* pose0, double* pose) {
  if (!xi || !pose0 || !pose) return ohm::afail(OHM_ERR_INVALID, "twist_pose: NULL argument");
  // T = exp(xi) as a rigid motion (Rodrigues' formula for the rotation R and
  // V rho for the translation, V the left Jacobian of SO(3)); pose = T pose0.
  const double rho[3] = {xi[0], xi[1], xi[2]}, phi[3] = {xi[3], xi[4], xi[5]};
  const double th = std::sqrt(phi[0] * phi[0] + phi[1] * phi[1] + phi[2] * phi[2]);
  const double Kx[3][3] = {{0.0, -phi[2], phi[1]}, {phi[2], 0.0, -phi[0]}, {-phi[1], phi[0], 0.0}};
  double K2[3][3];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) K2[i][j] = Kx[i][0] * Kx[0][j] + Kx[i][1] * Kx[1][j] + Kx[i][2] * Kx[2][j];
  // small angles: the series to first order, as an exact rotation is not needed there
  const double a = th < 1e-12 ? 1.0 : std::sin(th) / th;
  const double b = th < 1e-12 ? 0.0 : (1.0 - std::cos(th)) / (th * th);
  const double bv = th < 1e-12 ? 0.5 : b;
  const double cv = th < 1e-12 ? 0.0 : (th - std::sin(th)) / (th * th * th);
  double R[3][3], V[3][3];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      const double I = i == j ? 1.0 : 0.0;
      R[i][j] = I + a * Kx[i][j] + b * K2[i][j];
      V[i][j] = I + bv * Kx[i][j] + cv * K2[i][j];
    }
  for (int i = 0; i < 3; ++i) {
    for (int j = 0; j < 3; ++j)
      pose[4 * i + j] = R[i][0] * pose0[0 + j] + R[i][1] * pose0[4 + j] + R[i][2] * pose0[8 + j];
    pose[4 * i + 3] = R[i][0] * pose0[3] + R[i][1] * pose0[7] + R[i][2] * pose0[11] +
                      (V[i][0] * rho[0] + V[i][1] * rho[1] + V[i][2] * rho[2]);
  }
  return OHM_OK;
}

}  // extern "C"
