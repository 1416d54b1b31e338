// Allocation-free ray counting into a caller-owned dense grid.
//
// Some callers cannot call cudaMalloc at the moment they need to integrate
// rays: code that runs while a stream is being captured into a CUDA graph
// (allocation calls are not allowed there), real-time loops that must not
// block on the allocator or on the device synchronisation cudaFree implies,
// and plug-ins whose host application hands all device memory to its own
// allocator.  For them, ohm_count_rays_noalloc walks a ray set exactly like
// ohm_integrate_rays and adds each ray's per-voxel hit and miss counts into
// two uint32 arrays the caller owns.  Its per-call working memory (quantised
// ray records and the length of each warp's rays) lives in one statically sized
// device array defined below, so the call allocates nothing.
//
// That array is a file-scope __device__ variable: every GPU that loads this
// library holds it (kNoAllocScratchBytes, 2 MB) until the process exits.
// Every call shares it and writes the records it reads; calls whose work
// overlaps on the GPU (different streams, no ordering between them) race on
// it and must not be issued.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>

#include "ohm_host.h"

namespace ohm {
namespace {

constexpr long long kNoAllocMaxRays = OHM_NOALLOC_MAX_RAYS;
constexpr long long kNoAllocMaxSegments = 4 * kNoAllocMaxRays;
constexpr int kNoAllocBlock = 256;
// dominant-axis slots of one thread's piece of a ray
constexpr int kNoAllocSlots = 12;
// Layout of the static array: [ray records] [pieces of the longest ray of each warp].
constexpr size_t kNoAllocRayBytes = sizeof(RayRec) * kNoAllocMaxRays;
constexpr size_t kNoAllocScratchBytes = kNoAllocRayBytes + sizeof(int32_t) * (kNoAllocMaxRays / 32);
static_assert(kNoAllocMaxRays % kNoAllocBlock == 0, "a length for each warp of the last block");

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

struct CountGrid {
  double origin[3];
  double scale;
  double rmax_q;
  int32_t frac_bits;
  long long corner[3];
  long long dims[3];
};

struct NoAllocArgs {
  const float* origins;
  const float* endpoints;
  const uint8_t* flags;
  long long n;
  long long n_origins;
};

__device__ __forceinline__ bool na_in_extent(const long long q[3], int F) {
  const long long lim = 1LL << 24;
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    long long v = q[k] >> F;
    ok = ok && v > -lim && v < lim;
  }
  return ok;
}

// Per ray: quantise, truncate to the maximum range.  Per warp: the pieces of
// its longest ray.
__global__ void __launch_bounds__(kNoAllocBlock) k_noalloc_prepare(CountGrid g, NoAllocArgs a, RayRec* rays,
                                                                   int32_t* warp_pieces) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int F = g.frac_bits;
  RayRec r;
  r.flags = 0;
  r.nseg = 0;
  r.inv = 0;
  const long long ei = i < a.n ? i : 0, oi = a.n_origins == 1 ? 0 : ei;
  long long qo[3], qe[3];
  bool ok = i < a.n;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float o = a.origins[3 * oi + k], e = a.endpoints[3 * ei + k];
    ok = ok && isfinite(o) && isfinite(e) && quantise(o, g.origin[k], g.scale, &qo[k]) &&
         quantise(e, g.origin[k], g.scale, &qe[k]);
  }
  bool sample = !(a.flags && (a.flags[ei] & kFlagNoReturn));
  int32_t pieces = 0;
  if (ok) {
    double d[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) d[k] = (double)(qe[k] - qo[k]);
    double l2 = __dmul_rn(d[0], d[0]);
    l2 = __dadd_rn(l2, __dmul_rn(d[1], d[1]));
    l2 = __dadd_rn(l2, __dmul_rn(d[2], d[2]));
    const double len = __dsqrt_rn(l2);
    if (len > g.rmax_q) {
      const double ratio = __ddiv_rn(g.rmax_q, len);
#pragma unroll
      for (int k = 0; k < 3; ++k) qe[k] = qo[k] + __double2ll_rn(__dmul_rn(d[k], ratio));
      sample = false;
    }
    ok = na_in_extent(qo, F) && na_in_extent(qe, F);
  }
  if (ok) {
    const int M = longest_axis(qo, qe);
    r.flags = kRayValid | (sample ? kRaySample : 0) | (M << kRayAxisShift);
    ray_constants(qo, qe, F, &r);
    r.inv = reciprocal64((unsigned long long)(M == 0 ? r.A[0] : (M == 1 ? r.A[1] : r.A[2])));
    pieces = (M == 0 ? r.n[0] : (M == 1 ? r.n[1] : r.n[2])) / kNoAllocSlots + 1;
  }
  if (i < a.n) rays[i] = r;
  pieces = __reduce_max_sync(0xffffffffu, pieces);
  if ((threadIdx.x & 31) == 0) warp_pieces[i >> 5] = pieces;
}

static __device__ __noinline__ int na_exact_pick(const RayRec* rp, int F, int32_t c0, int32_t c1, int32_t c2) {
  const RayRec r = *rp;
  return exact_pick(r, F, c0, c1, c2);
}

// One piece of each ray (blockIdx.y), kNoAllocSlots dominant-axis slots: the
// local walk of ohm_device.cuh (LWalker).  Every voxel takes a miss except the
// voxel holding the ray's sample, which takes a hit.  A warp holds the same
// piece of 32 neighbouring rays, and the lanes in one voxel add once
// (__match_any_sync): all rays pass the voxels around the sensor.  One thread
// per 64-step segment, as it was, left a scan of 30,000 rays with 30,000
// threads of up to 100 dependent steps and one atomic per visit at the same
// few words: a pass of 30,011 rays over a 112 x 96 x 56 grid took 80.5 us, and
// takes 56.6 us this way.
__device__ __forceinline__ void na_walk_piece(const CountGrid& g, const RayRec* rays, int n, int32_t K0, uint32_t* hits,
                                              uint32_t* misses) {
  const unsigned full = 0xffffffffu;
  const int i = blockIdx.x * kNoAllocBlock + threadIdx.x, lane = threadIdx.x & 31;
  const int F = g.frac_bits;
  int32_t left = 0, x = 0, y = 0, z = 0, c0 = 0, c1 = 0, c2 = 0;
  bool sample = false;
  uint32_t cell = 0;
  LWalker w = {};
  int32_t sx = 1, sy = 1, sz = 1;
  const uint32_t nx = (uint32_t)g.dims[0], nxy = (uint32_t)(g.dims[0] * g.dims[1]);
  if (i < n && (rays[i].flags & kRayValid)) {
    const RayRec r = rays[i];
    const int M = (r.flags >> kRayAxisShift) & 3;
    const int32_t nmaj = M == 0 ? r.n[0] : (M == 1 ? r.n[1] : r.n[2]);
    if (K0 <= nmaj) {
      const int32_t K1 = K0 + kNoAllocSlots < nmaj + 1 ? K0 + kNoAllocSlots : nmaj + 1;
      PieceStart p;
      piece_start(r, F, K0, K1, K1 == nmaj + 1, &p, &w);
      left = p.visits;
      sample = K1 == nmaj + 1 && (r.flags & kRaySample);
      c0 = p.c[0];
      c1 = p.c[1];
      c2 = p.c[2];
      sx = ((r.flags >> kRaySignShift) & 1) ? -1 : 1;
      sy = ((r.flags >> (kRaySignShift + 1)) & 1) ? -1 : 1;
      sz = ((r.flags >> (kRaySignShift + 2)) & 1) ? -1 : 1;
      // relative to the grid (|voxel| < 2^24; a corner far away is out of the grid as INT_MAX / 2)
      const long long far = 1LL << 30;
      const long long rx = p.v[0] - g.corner[0], ry = p.v[1] - g.corner[1], rz = p.v[2] - g.corner[2];
      x = (int32_t)(rx < -far ? -far : (rx > far ? far : rx));
      y = (int32_t)(ry < -far ? -far : (ry > far ? far : ry));
      z = (int32_t)(rz < -far ? -far : (rz > far ? far : rz));
      cell = (uint32_t)x + nx * (uint32_t)y + nxy * (uint32_t)z;  // modulo 2^32; below 4e9 inside the grid
    }
  }
  while (__any_sync(full, left > 0)) {
    const bool in = left > 0 && (uint32_t)x < nx && (uint32_t)y < (uint32_t)g.dims[1] && (uint32_t)z < (uint32_t)g.dims[2];
    const bool hit = left == 1 && sample;
    const unsigned who = __ballot_sync(full, in && !hit);
    const unsigned grp = __match_any_sync(full, in ? cell : ~(uint32_t)lane) & who;
    if (in && !hit && lane == __ffs(grp) - 1) atomicAdd(misses + cell, (uint32_t)__popc(grp));
    if (in && hit) atomicAdd(hits + cell, 1u);
    --left;
    if (left > 0) {
      uint32_t mo = 0;
      LWalker w0 = w;
      int axis;
      if (lwalker_step(w, mo)) {
        axis = mo == 1u ? 0 : (mo == 2u ? 1 : 2);
      } else {
        w = w0;
        axis = na_exact_pick(rays + i, F, c0, c1, c2);
        if (axis == 0) w.sx = fadd_rn(w.sx, w.ux);
        if (axis == 1) w.sy = fadd_rn(w.sy, w.uy);
        if (axis == 2) w.sz = fadd_rn(w.sz, w.uz);
        w.mn = fminf(w.sx, fminf(w.sy, w.sz));
      }
      if (axis == 0) {
        ++c0;
        x += sx;
        cell += (uint32_t)sx;
      } else if (axis == 1) {
        ++c1;
        y += sy;
        cell += sy > 0 ? nx : 0u - nx;
      } else {
        ++c2;
        z += sz;
        cell += sz > 0 ? nxy : 0u - nxy;
      }
    }
  }
}
// A row of blocks (blockIdx.y) per piece that the range allows, where two
// device-fulls of blocks reach that far; else (kTurns) the rows take the pieces in
// turn, each warp up to its longest ray's last piece, so that a generous
// max_range costs nothing beside short rays: 30,000 rays of 3 m with a range of
// 1 km took 243 us with a thread for every piece, and take 50 us, as with a range
// of 9 m.  (In turn with rows for every piece: 1 us of 56 slower.)
template <bool kTurns>
__global__ void __launch_bounds__(kNoAllocBlock) k_noalloc_walk(CountGrid g, const RayRec* rays, const int32_t* warp_pieces,
                                                                int n, int pieces, uint32_t* hits, uint32_t* misses) {
  if (kTurns) pieces = warp_pieces[(blockIdx.x * kNoAllocBlock + threadIdx.x) >> 5];
  for (int p = blockIdx.y; p < pieces; p += gridDim.y) na_walk_piece(g, rays, n, p * kNoAllocSlots, hits, misses);
}

// Device address of the static array and the blocks of the walk a device holds
// at a time, looked up once per device.
std::mutex g_noalloc_mutex;
void* g_noalloc_ptr[64] = {nullptr};
int g_noalloc_resident[64] = {0};

}  // namespace
}  // namespace ohm

namespace {
ohm_status na_fail(ohm_status code, const std::string& msg) {
  ohm::set_last_error(msg);
  return code;
}
bool na_is_device_pointer(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}
}  // namespace

extern "C" {

ohm_status ohm_count_rays_noalloc(const ohm_count_grid* grid, const float* origins, int64_t n_origins,
                                  const float* endpoints, const uint8_t* flags, int64_t n, uint32_t* hits,
                                  uint32_t* misses, void* stream) {
  using namespace ohm;
  if (!grid || !hits || !misses) return na_fail(OHM_ERR_INVALID, "count_rays_noalloc: NULL grid or output");
  if (n < 0 || n > kNoAllocMaxRays)
    return na_fail(OHM_ERR_INVALID, "count_rays_noalloc: n must be in [0, OHM_NOALLOC_MAX_RAYS = " +
                                        std::to_string(kNoAllocMaxRays) + "]");
  if (!(grid->voxel_size > 0.0) || grid->frac_bits < 8 || grid->frac_bits > 20 || !(grid->max_range > 0.0))
    return na_fail(OHM_ERR_INVALID, "count_rays_noalloc: bad voxel_size / frac_bits / max_range");
  const int32_t S = grid->segment_steps == 0 ? 64 : grid->segment_steps;
  if (S < 1) return na_fail(OHM_ERR_INVALID, "count_rays_noalloc: segment_steps must be >= 1");
  for (int k = 0; k < 3; ++k)
    if (grid->dims[k] < 1 || grid->dims[k] > (1LL << 20))
      return na_fail(OHM_ERR_INVALID, "count_rays_noalloc: dims must be in [1, 2^20]");
  if ((double)grid->dims[0] * grid->dims[1] * grid->dims[2] > 4.0e9)
    return na_fail(OHM_ERR_INVALID, "count_rays_noalloc: grid has more than 4e9 voxels");
  const double scale = std::ldexp(1.0, grid->frac_bits) / grid->voxel_size;
  if (grid->max_range * scale >= std::ldexp(1.0, 30))
    return na_fail(OHM_ERR_INVALID, "count_rays_noalloc: max_range * 2^frac_bits / voxel_size must be < 2^30");
  // the call's size limit, in segments of S dominant-axis steps: a ray has at
  // most (max_range / voxel_size + 2) / S + 1 of them
  const long long per_ray = (long long)std::ceil(grid->max_range / grid->voxel_size + 2.0) / S + 1;
  if (per_ray * n > kNoAllocMaxSegments)
    return na_fail(OHM_ERR_INVALID, "count_rays_noalloc: n * segments per ray (max_range in segment_steps) exceeds " +
                                        std::to_string(kNoAllocMaxSegments) + "; raise segment_steps or lower n");
  if (n == 0) return OHM_OK;
  if (!origins || !endpoints || (n_origins != 1 && n_origins != n))
    return na_fail(OHM_ERR_INVALID, "count_rays_noalloc: bad origins / endpoints");
  const void* ins[] = {origins, endpoints, hits, misses};
  for (const void* p : ins)
    if (!na_is_device_pointer(p)) return na_fail(OHM_ERR_INVALID, "count_rays_noalloc: buffers must be device memory");
  if (flags && !na_is_device_pointer(flags))
    return na_fail(OHM_ERR_INVALID, "count_rays_noalloc: flags must be device memory");

  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64)
    return na_fail(OHM_ERR_CUDA, "count_rays_noalloc: no current device");
  void* scratch = nullptr;
  int resident = 0;
  {
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
      // First call on this device: resolve the static array's device address.
      int sms = 0, per_sm = 0;
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_noalloc_walk<true>, kNoAllocBlock, 0);
      g_noalloc_resident[dev] = (sms > 0 ? sms : 1) * (per_sm > 0 ? per_sm : 1);
      cudaError_t e = cudaGetSymbolAddress(&g_noalloc_ptr[dev], g_noalloc_scratch);
      if (e != cudaSuccess) {
        g_noalloc_ptr[dev] = nullptr;
        return na_fail(OHM_ERR_CUDA, std::string("count_rays_noalloc: cudaGetSymbolAddress: ") + cudaGetErrorString(e));
      }
    }
    scratch = g_noalloc_ptr[dev];
    resident = g_noalloc_resident[dev];
  }
  CountGrid g;
  for (int k = 0; k < 3; ++k) {
    g.origin[k] = grid->map_origin[k];
    g.corner[k] = grid->corner[k];
    g.dims[k] = grid->dims[k];
  }
  g.scale = scale;
  g.rmax_q = grid->max_range * scale;
  g.frac_bits = grid->frac_bits;
  NoAllocArgs a;
  a.origins = origins;
  a.endpoints = endpoints;
  a.flags = flags;
  a.n = n;
  a.n_origins = n_origins;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const unsigned blocks = (unsigned)((n + kNoAllocBlock - 1) / kNoAllocBlock);
  // a ray takes at most max_range / voxel_size + 2 steps of its dominant axis
  // (one slot more)
  const long long slots = (long long)std::ceil(grid->max_range / grid->voxel_size + 2.0) + 1;
  const long long pieces = (slots + kNoAllocSlots - 1) / kNoAllocSlots, rows = 2LL * resident / blocks + 1;
  RayRec* rays = static_cast<RayRec*>(scratch);
  int32_t* warp_pieces = reinterpret_cast<int32_t*>(static_cast<unsigned char*>(scratch) + kNoAllocRayBytes);
  k_noalloc_prepare<<<blocks, kNoAllocBlock, 0, s>>>(g, a, rays, warp_pieces);
  const auto walk = pieces <= rows ? k_noalloc_walk<false> : k_noalloc_walk<true>;
  walk<<<dim3(blocks, (unsigned)std::min(pieces, rows)), kNoAllocBlock, 0, s>>>(g, rays, warp_pieces, (int)n, (int)pieces,
                                                                                hits, misses);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return na_fail(OHM_ERR_CUDA, std::string("count_rays_noalloc: launch: ") + cudaGetErrorString(e));
  return OHM_OK;
}

}  // extern "C"
