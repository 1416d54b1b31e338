// Per-item device functions of the ray-integration kernels (Sec. III-B,
// III-C of arxiv 2206.06079, re-designed for sm_103a).  The single-map
// kernels (ohm_integrate.cu) and the multi-map batch kernels (ohm_batch.cu)
// are thin loops around these.
#pragma once

#include <climits>

#include "ohm_host.h"

namespace ohm {

constexpr int kBlock = 256;
// regions whose first hash probes one thread of the prepare walk loads together
#ifndef OHM_REGION_BATCH
#define OHM_REGION_BATCH 4
#endif
constexpr int kRegionBatch = OHM_REGION_BATCH;

__device__ __forceinline__ bool latched(const DeviceMap& m) { return *(volatile int32_t*)m.status != 0; }

// Programmatic dependent launch (sm_90 and later).  A kernel launched with
// programmatic stream serialisation may be scheduled while the kernel before
// it in the stream is still draining.  chain_enter() first waits until that
// kernel has completed and its writes are visible (griddepcontrol.wait; a
// no-op for an ordinary launch), then allows the next kernel of the stream to
// be scheduled.  Called first thing by every kernel of an integrate chain
// (single map or batched), so each body still runs strictly after its
// predecessor; only the launch latency and the block scheduling overlap.
__device__ __forceinline__ void chain_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Host side: launch one kernel of a chain with programmatic stream
// serialisation: its blocks may be scheduled while the previous kernel of the
// stream drains, and wait in chain_enter() until that kernel has completed.
// Where the attribute is refused the kernel is launched the ordinary way.
template <typename... K, typename... A>
inline void launch_chained_of(unsigned block, void (*kernel)(K...), unsigned grid, cudaStream_t stream, A... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, kernel, args...) != cudaSuccess) {
    (void)cudaGetLastError();
    cfg.numAttrs = 0;
    (void)cudaLaunchKernelEx(&cfg, kernel, args...);
  }
}

template <typename... K, typename... A>
inline void launch_chained(void (*kernel)(K...), unsigned grid, cudaStream_t stream, A... args) {
  launch_chained_of(kBlock, kernel, grid, stream, args...);
}

// Tells the compiler that a pointer read from a DeviceMap outside constant
// memory (by reference, or from the batch kernels' shared copy) is global: its
// loads are global ones and an atomic whose result is unused goes out as a
// reduction instead of a generic atomic that returns a value.
template <typename T>
__device__ __forceinline__ T* global_ptr(T* p) {
  __builtin_assume(__isGlobal(p));
  return p;
}

// Log-odds of a stored occupancy word for an update: an unknown voxel (NaN)
// starts from the prior 0, and a value stored below l_min stands for l_min
// (the miss walk may leave it there, see walk_segments).
__device__ __forceinline__ float logodds_value(float s, float l_min) { return s != s ? 0.0f : fmaxf(s, l_min); }

// Log-odds a stored occupancy word reports: NaN stays unknown, a value stored
// below l_min reads as l_min.
__device__ __forceinline__ float logodds_read(float s, float l_min) { return s < l_min ? l_min : s; }

// One coordinate of a point: quantise(), in float-float where that settles it.
// Returns false for a non-finite coordinate too.
__device__ __forceinline__ bool quantise_coord(const DeviceMap& m, float x, int k, long long* q) {
  if (quantise_ff(x, m.origin_ff[k], m.scale_ff, q)) return true;
  return isfinite(x) && quantise(x, m.origin[k], m.scale, q);
}

// Quantise a ray, returns false when it is skipped (non-finite coordinate or
// a point beyond the fixed-point range).
__device__ __forceinline__ bool quantise_ray(const DeviceMap& m, const float o[3], const float e[3], long long qo[3],
                                             long long qe[3]) {
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    ok = quantise_coord(m, o[k], k, &qo[k]) && ok;
    ok = quantise_coord(m, e[k], k, &qe[k]) && ok;
  }
  return ok;
}

// |qe - qo| in fixed-point units, double, fixed evaluation order.
__device__ __forceinline__ double ray_length(const long long qo[3], const long long qe[3], double d[3]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) d[k] = (double)(qe[k] - qo[k]);
  double l2 = __dmul_rn(d[0], d[0]);
  l2 = __dadd_rn(l2, __dmul_rn(d[1], d[1]));
  l2 = __dadd_rn(l2, __dmul_rn(d[2], d[2]));
  return __dsqrt_rn(l2);
}

__device__ __forceinline__ bool in_extent(const long long q[3], int F) {
  const long long lim = 1LL << 24;
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    long long v = q[k] >> F;
    ok = ok && v > -lim && v < lim;
  }
  return ok;
}

__device__ __forceinline__ void load_ray(const CallArgs& a, long long i, float o[3], float e[3], uint8_t* flag) {
  const long long oi = a.n_origins == 1 ? 0 : i;
  o[0] = a.origins[3 * oi + 0];
  o[1] = a.origins[3 * oi + 1];
  o[2] = a.origins[3 * oi + 2];
  e[0] = a.endpoints[3 * i + 0];
  e[1] = a.endpoints[3 * i + 1];
  e[2] = a.endpoints[3 * i + 2];
  *flag = a.flags ? a.flags[i] : 0;
}

// Walk the regions (32^3 voxel blocks) a ray passes through, inserting each
// into the hash table.  The same exact walk at region resolution visits
// exactly the regions of the voxels the voxel walk visits: region boundaries
// are voxel boundaries, crossed at the same t in the same tie order.
//
// The lookups of successive regions do not depend on one another, and a
// 131,072-ray scan runs as one wave, so the kernel lasts as long as its
// longest chain of dependent loads (a ray to the range limit crosses dozens
// of regions).  So the walk goes kRegionBatch regions ahead and loads their
// first probe entries together.  A first entry holding the key with a slot
// is the common case (the region exists): it is stamped as insert_region
// would.  Every other case goes through insert_region.  A ray visits a
// region once, so a batch holds distinct keys.
//
// Returns the slot of the last region (the one holding the end point) where
// this thread learnt it, else -1 (see insert_region).
__device__ __forceinline__ int32_t insert_ray_regions(const DeviceMap& m, const long long a[3], const long long b[3]) {
  const int S = m.frac_bits + kRegionShift;
  if ((a[0] >> S) == (b[0] >> S) && (a[1] >> S) == (b[1] >> S) && (a[2] >> S) == (b[2] >> S))
    return insert_region(m, (int)(b[0] >> S), (int)(b[1] >> S), (int)(b[2] >> S));  // without setting up a walk
  Walker w;
  walker_init(w, a, b, m.frac_bits + kRegionShift, 0, 0);
  const int32_t seq = m.calls->seq;
  int32_t last = -1;
  bool more = true;
  while (more) {
    long long key[kRegionBatch];
    uint32_t h[kRegionBatch];
    unsigned n = 0;
#pragma unroll
    for (int j = 0; j < kRegionBatch; ++j) {
      key[j] = kEmptyKey;
      h[j] = 0;
      if (more) {
        key[j] = pack_region(w.vx, w.vy, w.vz);
        h[j] = hash_key(key[j]) & m.hmask;
        n = j + 1;
        if (w.total > 0) {
          int32_t c, s;
          walker_step(w, walker_choose(w), &c, &s);
        } else {
          more = false;
        }
      }
    }
    longlong2 e[kRegionBatch];
#pragma unroll
    for (int j = 0; j < kRegionBatch; ++j)
      if (j < (int)n) e[j] = m.htab[h[j]];
#pragma unroll
    for (int j = 0; j < kRegionBatch; ++j) {
      if (j < (int)n) {
        if (e[j].x == key[j] && e[j].y >= 0) {
          m.stamp[e[j].y] = seq;
          last = (int32_t)e[j].y;
        } else {
          const unsigned long long k = (unsigned long long)key[j];
          const int32_t mask = (1 << 21) - 1;
          // sign-extend the 21-bit fields of the packed key
          const int rx = (int32_t)((uint32_t)((k >> 42) & mask) << 11) >> 11;
          const int ry = (int32_t)((uint32_t)((k >> 21) & mask) << 11) >> 11;
          const int rz = (int32_t)((uint32_t)(k & mask) << 11) >> 11;
          last = insert_region(m, rx, ry, rz);
        }
      }
    }
  }
  return last;
}

// Give region `slot` an NDT block if it has none: one thread wins the claim
// (-1 -> -2) and takes a block from the pool.
__device__ __forceinline__ void ndt_claim(const DeviceMap& m, int32_t slot) {
  if (*(volatile int32_t*)&m.ndt_slot[slot] != -1) return;
  if (atomicCAS(&m.ndt_slot[slot], -1, -2) == -1) {
    const int32_t id = alloc_ndt_block(m);
    if (id >= 0) {
      m.ndt_born[slot] = m.calls->seq;
      m.ndt_slot[slot] = id;
    } else {
      atomicOr(m.status, kStatusCapacity);
    }
  }
}

__device__ __forceinline__ long long voxel_offset(int32_t slot, uint32_t mo) {
  return (long long)slot * kRegionVoxels + mo;
}

__device__ __forceinline__ int32_t region_slot_of(const DeviceMap& m, int32_t vx, int32_t vy, int32_t vz) {
  return find_region(m, pack_region(vx >> kRegionShift, vy >> kRegionShift, vz >> kRegionShift));
}

__device__ __forceinline__ uint32_t local_morton(int32_t vx, int32_t vy, int32_t vz) { return region_morton(vx, vy, vz); }

// The 10 moments (n, Sx, Sy, Sz, Sxx, Sxy, Sxz, Syy, Syz, Szz) of a voxel of
// NDT block ns.  They lie side by side, 80 bytes on a 16-byte boundary: a
// sample, a query or an exported voxel touches 3 sectors instead of one in
// each of 10 planes.
__device__ __forceinline__ long long* ndt_moments(const DeviceMap& m, int32_t ns, uint32_t mo) {
  return m.ndt + ((long long)ns * kRegionVoxels + mo) * 10;
}

// Sample clearing (Sec. II-D): a miss that took voxel `off` from at or above
// the threshold (or from unknown) to below it clears the voxel's NDT samples.
// Misses only lower a voxel within the miss phase, so exactly one successful
// CAS per voxel and call can make this crossing.
__device__ __forceinline__ void after_miss(const DeviceMap& m, long long off, unsigned int old_bits, unsigned int new_bits) {
  const float lo = __uint_as_float(old_bits), ln = __uint_as_float(new_bits);
  if (!(ln < m.ndt_clear) || (lo < m.ndt_clear)) return;  // NaN (unknown) compares false: counts as above
  if (!(m.layers & kLayerNdt)) return;
  const int32_t ns = m.ndt_slot[off >> (3 * kRegionShift)];
  if (ns < 0) return;
  long long* base = ndt_moments(m, ns, (uint32_t)off & (kRegionVoxels - 1));
#pragma unroll
  for (int k = 0; k < 10; ++k) base[k] = 0;
}

// Retry a clamped log-odds CAS whose first attempt found `cur` instead of
// the value it expected (see logodds_update_n).
static __device__ __noinline__ void logodds_retry(const DeviceMap& m, unsigned int* u, unsigned int cur, float delta) {
  for (int it = 0; it < 256; ++it) {
    const float l0 = logodds_value(__uint_as_float(cur), m.l_min);
    const unsigned int nb = __float_as_uint(fminf(fmaxf(__fadd_rn(l0, delta), m.l_min), m.l_max));
    if (nb == cur) return;
    const unsigned int prev = atomicCAS(u, cur, nb);
    if (prev == cur) {
      if (delta < 0.f) after_miss(m, u - reinterpret_cast<unsigned int*>(m.occ), cur, nb);
      return;
    }
    cur = prev;
  }
  atomicOr(m.status, kStatusCasLimit);
}

// Clamped compare-and-swap miss of one voxel whose word was read as `old`
// (with NDT sample clearing: clears its samples if the miss crosses the
// threshold).
__device__ __forceinline__ void miss_cas(const DeviceMap& m, unsigned int* u, unsigned int old, unsigned int& ops) {
  const float l0 = logodds_value(__uint_as_float(old), m.l_min);
  const unsigned int nb = __float_as_uint(fminf(fmaxf(__fadd_rn(l0, m.miss), m.l_min), m.l_max));
  if (nb == old) return;
  ++ops;
  const unsigned int prev = atomicCAS(u, old, nb);
  if (prev != old)
    logodds_retry(m, u, prev, m.miss);
  else
    after_miss(m, u - reinterpret_cast<unsigned int*>(m.occ), old, nb);
}

// Launch shapes (measured on GB300, tunnel scans of 131,072 rays):
//  OHM_WALK_OVERSUBSCRIBE  the walk's grid-stride launch covers this many
//                          times the resident blocks (2, 4, 6, 8: 73.0, 72.4,
//                          74.3, 75.4 us mapped, 179, 154, 156, 160 us unknown)
//  OHM_PREPARE_MIN_BLOCKS  blocks per SM of the prepare kernels (4: a
//                          131,072-ray scan fits one wave on 152 SMs)
#ifndef OHM_WALK_OVERSUBSCRIBE
#define OHM_WALK_OVERSUBSCRIBE 4
#endif
#ifndef OHM_PREPARE_MIN_BLOCKS
#define OHM_PREPARE_MIN_BLOCKS 4
#endif

// The rollback point of the next call: the pool counters as they stand.
__device__ __forceinline__ void snapshot_pool(const DeviceMap& m) {
  m.calls->region_start = *m.region_count;
  m.calls->ndt_start = *m.ndt_count;
  m.calls->free_used_start = m.free_info[1];
  m.calls->ndt_free_used_start = m.free_info[3];
}

// End of a call, one thread of its last kernel: its counters become `last`
// and stand ready for the next call.  A failed call keeps its sequence number
// and its rollback point, which the rollback (running beside this) reads.
// Doing this here saves a kernel at the start of every call, about 3 us of a
// small scan and one launch.  One thread's latency bounds it, so every load
// goes out before the first store, and the host's word, which ohm_map_sync
// reads (and zeroes) without a copy of its own, is written after a failure
// only.
__device__ __forceinline__ void finish_call(const DeviceMap& m, long long rays) {
  CallCounters* c = m.calls;
  const auto segments = c->segments;
  const auto visits = c->visits;
  const auto touched = c->touched;
  const auto atomics = c->atomics;
  const auto restores = c->restores;
  const auto total = c->total_visits;
  const auto seq = c->seq;
  const auto regions = *m.region_count;
  const auto ndt_blocks = *m.ndt_count;
  const auto free_used = m.free_info[1];
  const auto ndt_free_used = m.free_info[3];
  const int32_t status = *(volatile int32_t*)m.status;
  c->last.rays = (unsigned long long)rays;
  c->last.segments = segments;
  c->last.visits = visits;
  c->last.touched = touched;
  c->last.atomics = atomics;
  c->last.restores = restores;
  c->total_visits = total + visits;
  c->segments = 0;
  c->visits = 0;
  c->touched = 0;
  c->atomics = 0;
  c->restores = 0;
  c->ndt_pending = 0;
  c->mean_touched = 0;
  if (status == 0) {
    c->seq = seq + 1;
    c->region_start = regions;
    c->ndt_start = ndt_blocks;
    c->free_used_start = free_used;
    c->ndt_free_used_start = ndt_free_used;
  } else {
    *(volatile int32_t*)m.host_status = status;
  }
}

// Fixed-point origin of the current call's rays where they share one: the
// first three lanes quantise a coordinate each.  Whole warps.
struct CallOrigin {
  long long q[3];
  bool ok;
};
__device__ __forceinline__ CallOrigin call_origin(const DeviceMap& m, const CallArgs& a) {
  const unsigned full = 0xffffffffu;
  CallOrigin r = {{0, 0, 0}, false};
  if (a.n_origins != 1 || a.n <= 0) return r;
  const int lane = threadIdx.x & 31, k = lane < 3 ? lane : 2;
  const float o = a.origins[k];
  long long q = 0;
  bool ok = quantise_ff(o, k == 0 ? m.origin_ff[0] : (k == 1 ? m.origin_ff[1] : m.origin_ff[2]), m.scale_ff, &q);
  if (!ok) ok = isfinite(o) && quantise(o, k == 0 ? m.origin[0] : (k == 1 ? m.origin[1] : m.origin[2]), m.scale, &q);
#pragma unroll
  for (int i = 0; i < 3; ++i) r.q[i] = __shfl_sync(full, q, i);
  r.ok = __all_sync(full, ok);
  return r;
}

// quantise_ray for the rays of the current call: a shared origin comes
// quantised from call_origin.
__device__ __forceinline__ bool quantise_call_ray(const DeviceMap& m, const CallArgs& a, const CallOrigin& origin,
                                                  const float o[3], const float e[3], long long qo[3],
                                                  long long qe[3]) {
  if (a.n_origins != 1) return quantise_ray(m, o, e, qo, qe);
  bool ok = origin.ok;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    qo[k] = origin.q[k];
    ok = quantise_coord(m, e[k], k, &qe[k]) && ok;
  }
  return ok;
}

// Segment table entries (ray i, segment j) of the rays of a full warp, in
// (j, lane) order: the first segments of the warp's 32 rays, then their second
// segments, and so on.  Neighbouring rays' j-th segments lie close together in
// space, so the walk's warps (which take consecutive entries) touch compact
// patches of the map; the stores of each j are coalesced.  Every lane calls
// this together with its ray's segment count (0 for none).
__device__ __forceinline__ void write_segments(const DeviceMap& m, long long i, unsigned int nseg) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const unsigned int total = __reduce_add_sync(full, nseg);
  unsigned long long base = 0;
  if (lane == 0 && total) base = atomicAdd(&m.calls->segments, (unsigned long long)total);
  base = __shfl_sync(full, base, 0);
  if (total == 0) return;
  if (base + total > (unsigned long long)m.max_segs) {
    if (lane == 0) atomicOr(m.status, kStatusScratch);
    return;
  }
  const unsigned int rounds = __reduce_max_sync(full, nseg);
  const unsigned int below = (1u << lane) - 1u;
  unsigned long long pos = base;
  for (unsigned int j = 0; j < rounds; ++j) {
    const unsigned int has = __ballot_sync(full, nseg > j);
    if (nseg > j) m.segs[pos + __popc(has & below)] = make_int2((int)i, (int)j);
    pos += __popc(has);
  }
}

// Per ray: fixed-point quantisation, max-range truncation, region walk with
// hash insertion, segment table.  Every lane of the warp must call this
// together with the same map (the segment reservation is warp-aggregated);
// lanes without a ray pass active = false.
__device__ __forceinline__ void prepare_occ_ray(const DeviceMap& m, const CallArgs& args, long long i, bool active) {
  active = active && !latched(m);
  const CallOrigin origin = call_origin(m, args);
  const int F = m.frac_bits;
  unsigned int nseg = 0, nvisit = 0;
  bool ndt_listed = false;
  RayRec r;
  r.flags = 0;
  r.nseg = 0;
  r.inv = 0;
  if (active) {
    float o[3], e[3];
    uint8_t flag;
    load_ray(args, i, o, e, &flag);
    long long qo[3], qe[3];
    bool ok = quantise_call_ray(m, args, origin, o, e, qo, qe);
    bool sample = (flag & kFlagNoReturn) == 0;
    if (ok) {
      // Truncation test len > rmax_q with len the double length.  Up to 2^53
      // the squared length is exact in double as in integers, so the test is
      // one on integers; the truncated end point is formed in float-float
      // where that settles it.  A missing return lies within rounding of the
      // range limit, so half of them come here, and a warp that holds one ran
      // a double square root and division for all its lanes.
      bool done = false;
      const long long dx = qe[0] - qo[0], dy = qe[1] - qo[1], dz = qe[2] - qo[2];
      const long long lim = 1LL << 30;
      if (dx > -lim && dx < lim && dy > -lim && dy < lim && dz > -lim && dz < lim) {
        const unsigned long long l2 = (unsigned long long)(dx * dx) + (unsigned long long)(dy * dy) +
                                      (unsigned long long)(dz * dz);
        if (l2 <= m.rmax_safe2) {
          done = true;
        } else if (l2 < (1ULL << 53)) {  // every difference below 2^27
          if (l2 <= m.rmax_in2) {
            done = true;
          } else {
            const int32_t d[3] = {(int32_t)dx, (int32_t)dy, (int32_t)dz};
            int32_t cut[3];
            if (truncate_ff(d, l2, m.band.rmax, cut)) {
#pragma unroll
              for (int k = 0; k < 3; ++k) qe[k] = qo[k] + cut[k];
              sample = false;
              done = true;
            }
          }
        }
      }
      if (!done) {
        double d[3];
        const double len = ray_length(qo, qe, d);
        if (len > m.rmax_q) {
          const double ratio = __ddiv_rn(m.rmax_q, len);
#pragma unroll
          for (int k = 0; k < 3; ++k) qe[k] = qo[k] + __double2ll_rn(__dmul_rn(d[k], ratio));
          sample = false;
        }
      }
      ok = in_extent(qo, F) && in_extent(qe, F);
    }
    if (ok) {
      const int M = longest_axis(qo, qe);
      long long nmaj = 0;
      long long l1 = 0;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        long long dv = (qe[k] >> F) - (qo[k] >> F);
        dv = dv < 0 ? -dv : dv;
        l1 += dv;
        if (k == M) nmaj = dv;
      }
      const SegSplit sp = ray_segment_split((int32_t)nmaj, l1, m.seg_steps);
      nseg = (unsigned int)sp.nseg;
      const long long am = sel3(M, qe[0] - qo[0], qe[1] - qo[1], qe[2] - qo[2]);
      r.inv = reciprocal64((unsigned long long)(am < 0 ? -am : am));
      r.flags = kRayValid | (sample ? kRaySample : 0) | (M << kRayAxisShift) | (int32_t)((uint32_t)sp.q << kRaySegShift);
      ray_constants(qo, qe, F, &r);
      r.nseg = (int32_t)nseg;
      if (m.layers & kLayerDecay) {
        DecayRec dr;
#pragma unroll
        for (int k = 0; k < 3; ++k) dr.inv[k] = reciprocal64((unsigned long long)r.A[k]);
        dr.length = walk_length_units(qo, qe, m.voxel_size, F);
        m.decay_rays[i] = dr;
      }
      nvisit = (unsigned int)(1 + l1);
      const int32_t last = insert_ray_regions(m, qo, qe);
      // NDT-OM: the sample's region (the ray's last) gets its NDT block here
      // when this thread learnt the region's slot; otherwise the ray is
      // listed for the NDT pass after this kernel
      if (sample && (m.layers & kLayerNdt)) {
        if (last >= 0)
          ndt_claim(m, last);
        else
          ndt_listed = true;
      }
    }
    m.rays[i] = r;
  }
  if (m.layers & kLayerNdt) {
    const unsigned full = 0xffffffffu;
    const unsigned listed = __ballot_sync(full, ndt_listed);
    if (listed) {
      const int lane = threadIdx.x & 31;
      unsigned long long base = 0;
      if (lane == 0) base = atomicAdd(&m.calls->ndt_pending, (unsigned long long)__popc(listed));
      base = __shfl_sync(full, base, 0);
      if (ndt_listed) m.ndt_pending[base + __popc(listed & ((1u << lane) - 1u))] = (int32_t)i;
    }
  }
  write_segments(m, i, nseg);
  warp_add(&m.calls->visits, nvisit);
}

// Per sample: give the sample's region an NDT layer.
__device__ __forceinline__ void ndt_alloc_ray(const DeviceMap& m, long long i) {
  const RayRec r = m.rays[i];
  if (!(r.flags & kRaySample)) return;
  const int32_t vx = r.v0[0] + (((r.flags >> kRaySignShift) & 1) ? -r.n[0] : r.n[0]);
  const int32_t vy = r.v0[1] + (((r.flags >> (kRaySignShift + 1)) & 1) ? -r.n[1] : r.n[1]);
  const int32_t vz = r.v0[2] + (((r.flags >> (kRaySignShift + 2)) & 1) ? -r.n[2] : r.n[2]);
  const int32_t slot = region_slot_of(m, vx, vy, vz);
  if (slot < 0) {
    atomicOr(m.status, kStatusMissing);
    return;
  }
  ndt_claim(m, slot);
}

// Decay layer: distance along the ray, in 2^-20 m, at which the walk crosses
// a boundary of an axis that has taken `done` steps.  The crossing happens at
// t = dist / A with dist = d0 + done U; t is taken as floor(2^32 dist / A) /
// 2^32 (exact, by the reciprocal inv = reciprocal64(A); 2^32 dist < 2^62) and
// the distance as rint(t L).  Monotone in t, so per-voxel differences are
// never negative, and they add up to L over the ray.
//
// dist is below 2^31 (a ray is shorter than 2^30 units and U at most 2^20), so
// the quotient's estimate floor(2^32 dist inv / 2^64) = floor(dist inv / 2^32)
// takes two 32-bit multiplies; one remainder test makes it exact (div_by_inv).
__device__ __forceinline__ unsigned long long decay_position(uint32_t dist, uint32_t A, unsigned long long inv,
                                                             unsigned long long length) {
  unsigned long long tq = (unsigned long long)dist * (uint32_t)(inv >> 32) +
                          (((unsigned long long)dist * (uint32_t)inv) >> 32);
  if (((unsigned long long)dist << 32) - tq * A >= A) tq += 1;
  const unsigned long long lo = tq * length, hi = __umul64hi(tq, length);
  const unsigned long long lo2 = lo + (1ULL << 31);
  return ((hi + (lo2 < lo ? 1ULL : 0ULL)) << 32) | (lo2 >> 32);
}

// Pool slots of two regions (or -1), their first probes issued together.
__device__ __forceinline__ void find_region2(const DeviceMap& m, long long k1, long long k2, int32_t* s1, int32_t* s2) {
  const longlong2 e1 = m.htab[hash_key(k1) & m.hmask];
  const longlong2 e2 = m.htab[hash_key(k2) & m.hmask];
  *s1 = e1.x == k1 ? (int32_t)e1.y : (e1.x == kEmptyKey ? -1 : find_region(m, k1));
  *s2 = e2.x == k2 ? (int32_t)e2.y : (e2.x == kEmptyKey ? -1 : find_region(m, k2));
}

// Out of line: the rare paths of the miss walk (a batch with a near-tie,
// stepped exactly from the ray record; a region the piece's set-up did not
// foresee), so that neither the record nor the hash loop takes registers in
// the walk.
struct ExactBatch {
  LWalker w;
  uint32_t mo;
  uint32_t at[8];
};
static __device__ __noinline__ void exact_batch(const RayRec* rp, int F, int32_t K0, int n, ExactBatch* b) {
  const RayRec r = *rp;
  piece_exact_steps(r, F, K0, b->w, b->mo, n, b->at);
}

// The key of the region reached from region `key` by one step along each
// axis whose bit is set in idx, in the direction of the ray's signs.
__device__ __forceinline__ long long neighbour_key(long long key, uint32_t idx, int32_t signs) {
  const unsigned long long k = (unsigned long long)key;
  const int32_t mask = (1 << 21) - 1;
  int32_t c[3] = {(int32_t)((k >> 42) & mask), (int32_t)((k >> 21) & mask), (int32_t)(k & mask)};
#pragma unroll
  for (int a = 0; a < 3; ++a)
    if ((idx >> a) & 1u) c[a] += ((signs >> a) & 1) ? -1 : 1;
  return pack_region(c[0], c[1], c[2]);
}
static __device__ __noinline__ int32_t find_neighbour_rare(const DeviceMap& m, const RayRec* rp, int32_t K0, uint32_t idx) {
  const RayRec r = *rp;
  PieceStart p;
  LWalker w;
  piece_start(r, m.frac_bits, K0, K0 + 1, false, &p, &w);
  return find_region(m, neighbour_key(pack_region(p.v[0] >> kRegionShift, p.v[1] >> kRegionShift, p.v[2] >> kRegionShift),
                                      idx, (r.flags >> kRaySignShift) & 7));
}

// Voxels per batch of the miss walk, and the blocks per SM it is compiled for
// (batches of 3 / 4 / 5 / 6 on a mapped 131,072-ray tunnel scan: 73.6 / 73.0 / 69.7 /
// 77 us: a segment of about 24 voxels takes five batches of 5 with the least left
// over; 6 spills).
#ifndef OHM_FAST_BATCH
#define OHM_FAST_BATCH 5
#endif
#ifndef OHM_FAST_MIN_BLOCKS
#define OHM_FAST_MIN_BLOCKS 4
#endif
constexpr int kFastBatch = OHM_FAST_BATCH;

// Shared memory of a walk block.
//
// Region bases of a piece, one column of `tab` per thread.  Entry idx (bit k:
// the walk has left its first region along axis k) at idx * kBlock is
// base ^ neg ^ (idx << 15) with base the region's first voxel offset, so that
// its exclusive or with the sign-normalised Morton index mo (idx = mo >> 15)
// is the voxel's offset base | ((mo ^ neg) & 0x7fff).  kNoRegion: not looked up.
//
// `open`: per warp, offsets of voxels whose saturation bit was clear, waiting
// to be looked at; less than a round between batches.  They are
// looked at kOpenEach per lane (2 and 8 were slower: 73 / 72 / 86 us for 2, 4
// and 8 on a mapped tunnel scan, 170 / 154 / 161 us in unknown space).
#ifndef OHM_OPEN_EACH
#define OHM_OPEN_EACH 4
#endif
constexpr uint32_t kOpenEach = OHM_OPEN_EACH;
constexpr uint32_t kOpenRound = 32 * kOpenEach;
constexpr int kOpenCap = kOpenRound + 32 * kFastBatch;
struct WalkShared {
  uint32_t tab[8 * kBlock];
  uint32_t open[kBlock / 32][kOpenCap];
  uint32_t n_open[kBlock / 32];
  uint32_t sum[kBlock];  // decay layer: path length of the lanes in one voxel, at its lowest lane; zero between steps
};
__device__ __forceinline__ void walk_shared_init(WalkShared& sh) {
  if ((threadIdx.x & 31) == 0) sh.n_open[threadIdx.x >> 5] = 0;
  sh.sum[threadIdx.x] = 0;
  __syncwarp();
}
constexpr uint32_t kNoRegion = 0x80000000u;
__device__ __forceinline__ uint32_t region_entry(int32_t slot, uint32_t neg, uint32_t idx) {
  return ((uint32_t)slot << (3 * kRegionShift)) ^ neg ^ (idx << (3 * kRegionShift));
}

// One miss of voxel `off`, whose word was read as `word` (add form, see
// walk_segments).  Returns true if the voxel was unknown and the
// compare-and-swap went out: its result is in `word` then.
__device__ __forceinline__ bool miss_add(float* occ, uint32_t off, uint32_t& word, float miss, float l_min,
                                         unsigned int& ops) {
  const float l = __uint_as_float(word);
  if (l > l_min) {
    atomicAdd(occ + off, miss);
    ++ops;
  } else if (l != l) {
    // an unknown voxel's first miss
    word = atomicCAS(reinterpret_cast<unsigned int*>(occ) + off, word, __float_as_uint(__fadd_rn(0.0f, miss)));
    ++ops;
    return true;
  }
  return false;
}

// Look at the warp's waiting voxels and give them their misses, until fewer
// than `keep` wait; four per lane at a time.  Returns the log-odds atomics
// this lane issued.  Whole warps; out of line: a well observed map comes here
// about once per six rounds of segments.
static __device__ __noinline__ unsigned int drain_open(float* occ_any, uint32_t* sat_any, float miss, float l_min,
                                                       WalkShared& sh, uint32_t keep) {
  constexpr int kEach = (int)kOpenEach;
  float* const occ = global_ptr(occ_any);
  uint32_t* const sat = global_ptr(sat_any);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  unsigned int ops = 0;
  __syncwarp();
  uint32_t n = sh.n_open[wid];
  while (n >= keep) {
    const uint32_t first = n > kOpenRound ? n - kOpenRound : 0u;
    uint32_t off[kEach], word[kEach], bits[kEach];
    bool cas[kEach];
#pragma unroll
    for (int j = 0; j < kEach; ++j) {
      const uint32_t i = first + (uint32_t)(32 * j + lane);
      off[j] = i < n ? sh.open[wid][i] : kNoRegion;
      if (off[j] != kNoRegion) word[j] = __float_as_uint(occ[off[j]]);
    }
    // voxels found at or below l_min get their bit.  Its word is looked at in
    // L2 first: many rays find the voxels around the sensor saturated in the
    // same call, and repeated ORs of one word would queue
#pragma unroll
    for (int j = 0; j < kEach; ++j) {
      bits[j] = ~0u;
      if (off[j] != kNoRegion && __uint_as_float(word[j]) <= l_min) bits[j] = __ldcg(sat + (off[j] >> 5));
      cas[j] = off[j] != kNoRegion && miss_add(occ, off[j], word[j], miss, l_min, ops);
    }
#pragma unroll
    for (int j = 0; j < kEach; ++j) {
      if (!((bits[j] >> (off[j] & 31u)) & 1u)) atomicOr(sat + (off[j] >> 5), 1u << (off[j] & 31u));
      if (cas[j] && __uint_as_float(word[j]) > l_min) {
        atomicAdd(occ + off[j], miss);
        ++ops;
      }
    }
    n = first;
  }
  __syncwarp();
  if (lane == 0) sh.n_open[wid] = n;
  __syncwarp();
  return ops;
}
__device__ __forceinline__ unsigned int drain_open(const DeviceMap& m, WalkShared& sh, uint32_t keep) {
  return drain_open(m.occ, m.sat, m.miss, m.l_min, sh, keep);
}

// Look up the regions of a piece and fill its column of the table; *mo becomes
// the sign-normalised index of its first voxel.  False if its first or last
// region is not in the map (kPartial: its first only).
template <bool kPartial = false>
__device__ __forceinline__ bool piece_regions(const DeviceMap& m, const PieceStart& p, const LWalker& w, int32_t flags,
                                              uint32_t* tab, uint32_t* mo) {
  const uint32_t neg = morton_neg(flags);
  const int32_t signs = (flags >> kRaySignShift) & 7;
  *mo = local_morton(p.v[0], p.v[1], p.v[2]) ^ neg;
  const int32_t a0 = p.v[0] >> kRegionShift, a1 = p.v[1] >> kRegionShift, a2 = p.v[2] >> kRegionShift;
  const int32_t b0 = p.ve[0] >> kRegionShift, b1 = p.ve[1] >> kRegionShift, b2 = p.ve[2] >> kRegionShift;
  const uint32_t idx = (a0 != b0 ? 1u : 0u) | (a1 != b1 ? 2u : 0u) | (a2 != b2 ? 4u : 0u);
  int32_t slot, slotE;
  find_region2(m, pack_region(a0, a1, a2), pack_region(b0, b1, b2), &slot, &slotE);
#pragma unroll
  for (int i = 1; i < 8; ++i) tab[i * kBlock] = kNoRegion;
  tab[0] = region_entry(slot, neg, 0);
  tab[idx * kBlock] = kPartial && slotE < 0 ? kNoRegion : region_entry(slotE, neg, idx);
  if (slot < 0 || (!kPartial && slotE < 0)) return false;
  if (idx & (idx - 1u)) {  // two or three boundaries: the regions between
    // the parameter at which the piece leaves its first region, per axis it does
    const float o0 = (idx & 1u) ? w.sx + (float)((signs & 1) ? p.v[0] & 31 : ~p.v[0] & 31) * w.ux : INFINITY;
    const float o1 = (idx & 2u) ? w.sy + (float)((signs & 2) ? p.v[1] & 31 : ~p.v[1] & 31) * w.uy : INFINITY;
    const float o2 = (idx & 4u) ? w.sz + (float)((signs & 4) ? p.v[2] & 31 : ~p.v[2] & 31) * w.uz : INFINITY;
    const uint32_t i1 = o0 <= o1 ? (o0 <= o2 ? 1u : 4u) : (o1 <= o2 ? 2u : 4u);
    const uint32_t i3 = o0 > o1 ? (o0 > o2 ? 1u : 4u) : (o1 > o2 ? 2u : 4u);
    const uint32_t i2 = idx == 7u ? 7u & ~i3 : i1;
    int32_t s1, s2;
    find_region2(m, pack_region((i1 & 1u) ? b0 : a0, (i1 & 2u) ? b1 : a1, (i1 & 4u) ? b2 : a2),
                 pack_region((i2 & 1u) ? b0 : a0, (i2 & 2u) ? b1 : a1, (i2 & 4u) ? b2 : a2), &s1, &s2);
    if (s1 >= 0) tab[i1 * kBlock] = region_entry(s1, neg, i1);
    if (s2 >= 0) tab[i2 * kBlock] = region_entry(s2, neg, i2);
  }
  return true;
}

// kFastBatch steps of the local walk from `mo` (left: voxels of the piece not
// yet stepped): sign-normalised Morton indices `at`, voxel offsets, and which of
// them exist (`valid`).  rp, K: the ray and the piece's first dominant-axis step.
// A voxel whose region is not in the map fails the call, which inserted every
// region that it walks; kPartial (a map that may lack some): it ends the walk,
// left = kWalkEnded.
constexpr int32_t kWalkEnded = INT_MIN;
template <bool kPartial = false>
__device__ __forceinline__ void piece_fill(const DeviceMap& m, const RayRec* rp, int32_t K, uint32_t* tab, LWalker& w,
                                           uint32_t& mo, int32_t& left, uint32_t (&at)[kFastBatch],
                                           uint32_t (&off)[kFastBatch], uint32_t& valid) {
  bool sure = true;
#pragma unroll
  for (int j = 0; j < kFastBatch; ++j) {
    at[j] = mo;
    sure = lwalker_step(w, mo) && sure;
  }
  valid = left >= kFastBatch ? (1u << kFastBatch) - 1u : (left > 0 ? (1u << left) - 1u : 0u);
  if (!sure && valid) {
    ExactBatch b;
    b.mo = at[0];
    exact_batch(rp, m.frac_bits, K, kFastBatch, &b);
    w = b.w;
    mo = b.mo;
#pragma unroll
    for (int j = 1; j < kFastBatch; ++j) at[j] = b.at[j - 1];
  }
  left -= kFastBatch;
  uint32_t any = 0;
#pragma unroll
  for (int j = 0; j < kFastBatch; ++j) {
    off[j] = tab[(at[j] >> 15) * kBlock] ^ at[j];  // voxel offset (< 2^31: at most 2^16 regions of 2^15 voxels)
    any |= off[j];
  }
  if ((any & kNoRegion) && valid) {
#pragma unroll
    for (int j = 0; j < kFastBatch; ++j) {
      if (((valid >> j) & 1u) && (off[j] & kNoRegion)) {
        const uint32_t idx = at[j] >> 15;
        uint32_t e = tab[idx * kBlock];
        if (e == kNoRegion) {
          const int32_t s = find_neighbour_rare(m, rp, K, idx);
          if (s < 0) {
            if (kPartial) {
              valid &= (1u << j) - 1u;
              left = kWalkEnded;
              return;
            }
            atomicOr(m.status, kStatusMissing);
            valid &= ~(1u << j);
            continue;
          }
          e = region_entry(s, morton_neg(rp->flags), idx);
          tab[idx * kBlock] = e;
        }
        off[j] = e ^ at[j];
      }
    }
  }
}

// Miss phase (Sec. III-C phase one) of one segment per lane (has = false: no
// segment): every voxel a ray passes through, except the voxel holding its
// sample, takes one miss.  Whole warps.  The walk is the exact local walk of
// ohm_device.cuh (LWalker), piece by piece (a segment of the default length is
// one piece).  The regions a piece passes through are looked up before it is
// walked, with the order of the boundary crossings taken from the estimates;
// one the estimates mistook is looked up when met.
//
// Occupancy update.  With kCas false (the miss increment is negative and the
// map does not clear NDT samples) a miss is a fire-and-forget float atomic add
// of the increment, and the lower clamp is applied where log-odds are read:
// a voxel's log-odds is max(stored, l_min).  Within a call every miss of a
// voxel adds the same delta < 0, so whatever the order the adds produce the
// floats l, fl(l + delta), fl(fl(l + delta) + delta), ...  While they stay at or
// above l_min these are the values of the clamped one-at-a-time updates
// l <- min(max(l + delta, l_min), l_max) (Eq. 2 with the clamp of Sec. II-B);
// once one drops below l_min the clamped sequence stays at l_min (fl(l_min +
// delta) <= l_min), which is what max(stored, l_min) reads, however far below
// the later adds take the stored value.  So the result is bit for bit that of
// the sequential updates.  A voxel already at or below l_min takes no add (a
// miss leaves it at l_min), and an unknown voxel (NaN) is first set to
// fl(0 + delta) by compare-and-swap; a thread that loses that race adds its
// miss to the value it found.  No value comes near the float subnormal range
// (create rejects increments and bounds below 2^-100 in magnitude), where the
// atomic add would flush to zero.  With kCas (NDT sample clearing, which must
// see the update that crosses its threshold, or a miss increment >= 0) every
// miss is a clamped compare-and-swap.
//
// Saturated voxels.  Most voxels a ray passes are free space that is at l_min
// already (99 % of the visits of a scan in a mapped tunnel).  Their bit in
// DeviceMap::sat says so: 32 bits, a 4 x 4 x 2 brick of voxels, per load instead
// of one float per voxel, read once per brick the ray enters, from a plane 1/32
// the size of the floats.  Voxels whose bit is clear are collected per warp
// and looked at kOpenRound at a time (drain_open), so the few of a well
// observed map neither stop the warp nor run its update code for one lane,
// and the many of unknown space go out kOpenEach per lane.  A voxel found at
// l_min gets its bit there; the hits clear it; a stale clear bit only costs
// the look.
//
// Counts and path lengths (kCounts, kDecay).  Every visit adds to these, and
// all rays of a scan pass the voxels around the sensor: one 64-bit atomic per
// visit queued at the few words there (a 65,344-ray scan with both layers took
// 409 us, 106 us in this form).  The lanes of a warp that stand in the same voxel (neighbouring rays
// at the same depth) form a group (__match_any_sync) whose lowest lane adds for
// all of them; their path lengths are summed in shared memory.  The sums are
// of integers, so grouping changes nothing.  kDecay: the voxel holding a
// sample takes path length too.
//
// A batch is stepped without a branch; one that met a near-tie is stepped
// again exactly.  What bounds the walk is instruction issue (46 M warp
// instructions for 19.3 M visits of a 131,072-ray tunnel scan, 83 M before)
// and the code is kept small, one copy of the stepping: a software pipeline
// of two batches and a second form that reads the floats directly were slower
// by what they add to the instruction cache and the registers.
// Measured (131,072-ray tunnel scan, 0.1 m, 865 k segments): 123.5 -> 69.7 us in
// a mapped tunnel, 164 -> 148 us in unknown space; 262,144 rays at 0.05 m
// 308 -> 157 us; outdoor scans into half-known space 144 -> 101 us.
template <bool kOcc, bool kCounts, bool kCas, bool kDecay>
__device__ __forceinline__ void walk_segments(const DeviceMap& m, bool has, int2 sg, WalkShared& sh,
                                              unsigned int& ops, const RayRec* prefetch = nullptr) {
  static_assert(kFastBatch <= 8, "ExactBatch holds 8 indices");
  const unsigned full = 0xffffffffu;
  const int F = m.frac_bits;
  uint32_t* const tab = sh.tab + threadIdx.x;
  const RayRec* rp = global_ptr(m.rays) + (has ? sg.x : 0);
  unsigned int* const occ = reinterpret_cast<unsigned int*>(global_ptr(m.occ));
  const uint32_t* const sat = global_ptr(m.sat);
  unsigned long long* const counts = global_ptr(m.counts);
  unsigned long long* const decay = global_ptr(m.decay);
  // 32 lanes' path lengths through one voxel (at most sqrt(3) voxels each) add up in 32 bits
  const bool small = m.voxel_size < 70.0;
  int32_t K = 0, K1 = -1;  // the piece's first dominant-axis step, the segment's end (not yet known)
  bool more = has;
  while (__any_sync(full, more)) {
    LWalker w = {};
    uint32_t mo = 0;
    int32_t left = 0;
    bool to_end = false, sample = false;   // (decay) the piece ends the ray, at a sample
    uint32_t c0 = 0, c1 = 0, c2 = 0;       // (decay) crossings taken per axis
    unsigned long long pos = 0, len = 0;   // (decay) where the walk entered the voxel, the ray's length
    if (more) {
      const RayRec r = *rp;
      const int M = (r.flags >> kRayAxisShift) & 3;
      const int32_t nmaj = M == 0 ? r.n[0] : (M == 1 ? r.n[1] : r.n[2]);
      if (K1 < 0) {
        // segment_bounds in 32 bits (at most 2^25 slots per ray)
        const int32_t q = (int32_t)((uint32_t)r.flags >> kRaySegShift), extra = nmaj + 1 - r.nseg * q;
        K = sg.y * q + (sg.y < extra ? sg.y : extra);
        K1 = K + q + (sg.y < extra ? 1 : 0);
        // the record of the thread's next segment, into L2 while this one walks
        if (prefetch) asm volatile("prefetch.global.L2 [%0];" ::"l"(prefetch));
      }
      const int32_t K0 = K, Ke = K + kPieceSlots < K1 ? K + kPieceSlots : K1;
      PieceStart p;
      piece_start(r, F, K0, Ke, Ke == nmaj + 1, &p, &w);
      to_end = Ke == nmaj + 1;
      sample = to_end && (r.flags & kRaySample);
      left = p.visits - ((sample && !kDecay) ? 1 : 0);
      if (kDecay) {
        c0 = (uint32_t)p.c[0];
        c1 = (uint32_t)p.c[1];
        c2 = (uint32_t)p.c[2];
        len = m.decay_rays[sg.x].length;
        if (K0 > 0)
          pos = decay_position((uint32_t)(M == 0 ? r.d0[0] : (M == 1 ? r.d0[1] : r.d0[2])) + ((uint32_t)(K0 - 1) << F),
                               (uint32_t)(M == 0 ? r.A[0] : (M == 1 ? r.A[1] : r.A[2])), r.inv, len);
      }
      if (!piece_regions(m, p, w, r.flags, tab, &mo)) {
        if (left > 0) atomicOr(m.status, kStatusMissing);
        left = 0;
      }
    }
    // batches of the warp's longest piece
    int rounds = __reduce_max_sync(full, left > 0 ? left + kFastBatch - 1 : 0) / kFastBatch;
    uint32_t brick = ~mo, word = 0;  // the last voxel stepped; the word of the last brick
    for (; rounds > 0; --rounds) {
      uint32_t at[kFastBatch], off[kFastBatch], v[kFastBatch] = {}, valid;
      piece_fill(m, rp, K, tab, w, mo, left, at, off, valid);
      if (kCounts || kDecay) {
        const int lane = threadIdx.x & 31;
        uint32_t missed = valid;  // the voxels that take a miss
        if (kDecay && sample && left <= 0 && valid) missed &= ~(1u << (31 - __clz(valid)));
#pragma unroll
        for (int j = 0; j < kFastBatch; ++j) {
          const bool in = (valid >> j) & 1u;
          uint32_t d = 0;
          unsigned long long wide = 0;
          if (kDecay && in) {
            // leave the voxel across the next boundary, or end in it
            const uint32_t moved = at[j] ^ (j + 1 < kFastBatch ? at[j + 1] : mo);
            const int axis = (moved & 0x9249u) ? 0 : ((moved & 0x12492u) ? 1 : 2);
            unsigned long long out = len;
            if (!(to_end && left <= 0 && !(valid >> (j + 1)))) {
              const uint32_t c = axis == 0 ? c0 : (axis == 1 ? c1 : c2);
              out = decay_position((uint32_t)rp->d0[axis] + (c << F), (uint32_t)rp->A[axis],
                                   global_ptr(m.decay_rays)[sg.x].inv[axis], len);
              c0 += axis == 0;
              c1 += axis == 1;
              c2 += axis == 2;
            }
            wide = out - pos;
            d = (uint32_t)wide;
            pos = out;
          }
          const unsigned grp = __match_any_sync(full, in ? off[j] : (kNoRegion | (uint32_t)lane));
          const int lead = __ffs(grp) - 1;
          if (kCounts) {
            const unsigned n = __popc(grp & __ballot_sync(full, (missed >> j) & 1u));
            if (in && lane == lead && n) atomicAdd(counts + off[j], (unsigned long long)n);
          }
          if (kDecay) {
            if (small) {
              uint32_t* const sum = sh.sum + (threadIdx.x & ~31u) + lead;
              if (in && d) atomicAdd(sum, d);
              __syncwarp();
              if (in && lane == lead) {
                if (*sum) atomicAdd(decay + off[j], (unsigned long long)*sum);
                *sum = 0;
              }
              __syncwarp();
            } else if (in && wide) {
              atomicAdd(decay + off[j], wide);
            }
          }
        }
        if (kDecay) valid = missed;
      }
      if (!kOcc) continue;
      if (kCas) {
#pragma unroll
        for (int j = 0; j < kFastBatch; ++j)
          if ((valid >> j) & 1u) v[j] = occ[off[j]];
#pragma unroll
        for (int j = 0; j < kFastBatch; ++j)
          if ((valid >> j) & 1u) miss_cas(m, occ + off[j], v[j], ops);
        continue;
      }
      // the words of the bricks entered, then the voxels not known to be saturated
      const uint32_t before = brick;
      brick = at[kFastBatch - 1];
#pragma unroll
      for (int j = 0; j < kFastBatch; ++j)
        if (((at[j] ^ (j ? at[j - 1] : before)) & ~31u) && ((valid >> j) & 1u)) v[j] = sat[off[j] >> 5];
      bool open[kFastBatch], some = false;
#pragma unroll
      for (int j = 0; j < kFastBatch; ++j) {
        if ((at[j] ^ (j ? at[j - 1] : before)) & ~31u) word = v[j];
        open[j] = ((valid >> j) & 1u) && !((word >> (off[j] & 31u)) & 1u);
        some = some || open[j];
      }
      if (__any_sync(full, some)) {
        const int wid = threadIdx.x >> 5;
        if (some) {
          uint32_t n = 0;
#pragma unroll
          for (int j = 0; j < kFastBatch; ++j) n += open[j] ? 1u : 0u;
          uint32_t i = atomicAdd(&sh.n_open[wid], n);
#pragma unroll
          for (int j = 0; j < kFastBatch; ++j)
            if (open[j]) sh.open[wid][i++] = off[j];
        }
        __syncwarp();
        if (sh.n_open[wid] >= kOpenRound) ops += drain_open(m, sh, kOpenRound);
      }
    }
    K += kPieceSlots;
    more = more && K < K1;
  }
}

// Whether a map's misses need the compare-and-swap form of walk_segments.
__device__ __host__ __forceinline__ bool walk_needs_cas(uint32_t layers, float miss, float ndt_clear) {
  return !(miss < 0.0f) || ((layers & kLayerNdt) && ndt_clear > -INFINITY);
}

// Which miss walk a map takes: walk_segments' template arguments as bits (8:
// decay, 4: occupancy, 2: counts, 1: every miss a compare-and-swap), or
// kWalkNone (no layer the walk updates).
constexpr int kWalkNone = -1;
constexpr int kWalkDecay = 8;
#define OHM_WALK_VARIANTS(X) X(2) X(4) X(5) X(6) X(7) X(8) X(10) X(12) X(13) X(14) X(15)
__device__ __host__ __forceinline__ int walk_variant(uint32_t layers, float miss, float ndt_clear) {
  const bool occ = (layers & kLayerOcc) != 0, cnt = (layers & kLayerCounts) != 0;
  const bool decay = (layers & kLayerDecay) != 0;
  if (!occ && !cnt && !decay) return kWalkNone;
  return (decay ? kWalkDecay : 0) | (occ ? 4 : 0) | (cnt ? 2 : 0) | ((occ && walk_needs_cas(layers, miss, ndt_clear)) ? 1 : 0);
}

// Position of a sample inside its voxel (fixed-point offset 0 .. 2^F - 1) in
// 1/1024 of the voxel, rounded down: the voxel-mean layer's 10-bit field.
__device__ __forceinline__ unsigned long long sub_voxel10(long long offset, int F) {
  return F >= 10 ? (unsigned long long)(offset >> (F - 10)) : (unsigned long long)(offset << (10 - F));
}

// Clamped log-odds update of a voxel by n hits of the same delta (Eq. 2 with
// the clamp of Sec. II-B): n steps l <- min(max(l + delta, l_min), l_max)
// from the stored value (0 for an unknown voxel), written with one
// compare-and-swap.  Within a kernel all updates of a voxel use the same
// delta and the step map composes, so the result depends neither on their
// order nor on how they are grouped.  The loop is bounded: every failed CAS
// means another thread advanced the value toward its clamp.
__device__ __forceinline__ void logodds_update_n(const DeviceMap& m, float* p, float delta, unsigned int n) {
  unsigned int* u = reinterpret_cast<unsigned int*>(p);
  unsigned int old = *u;
  for (int it = 0; it < 256; ++it) {
    float v = logodds_value(__uint_as_float(old), m.l_min);
    for (unsigned int t = 0; t < n; ++t) {
      const float nv = fminf(fmaxf(__fadd_rn(v, delta), m.l_min), m.l_max);
      if (nv == v) break;  // at a clamp: later steps change nothing
      v = nv;
    }
    const unsigned int nb = __float_as_uint(v);
    if (nb == old) return;
    const unsigned int prev = atomicCAS(u, old, nb);
    if (prev == old) {
      // a voxel stored at or below l_min may have its bit set
      if (__uint_as_float(old) <= m.l_min) {
        const long long off = p - m.occ;
        atomicAnd(global_ptr(m.sat) + (off >> 5), ~(1u << (off & 31)));
      }
      return;
    }
    old = prev;
  }
  atomicOr(m.status, kStatusCasLimit);
}

// Sample phase (Sec. III-C phase two) for one ray: the voxel holding its
// sample takes a hit; with the NDT layer it also accumulates the sample's
// exact integer moments (count, sum, outer-product sum of the position inside
// the voxel), from which mean and covariance are formed when queried.
//
// Every lane of the warp calls this together (active = false for a lane
// without a ray of this map).  Neighbouring rays often end in the same voxel,
// and concurrent compare-and-swaps on one word retry, so the lanes holding the
// same voxel (__match_any_sync) form a group whose lowest lane applies all of
// the group's occupancy hits, n clamped steps in one compare-and-swap, and
// adds the group's hit count.  The voxel-mean fields and NDT moments are
// fire-and-forget integer adds (summing them across the group first was
// measured slower).  The moments of the warp's samples pass through shared
// memory (sh), so that neighbouring lanes add neighbouring words: a warp's 320
// adds go out as about 100 sectors; with each lane adding its own sample's 10
// they were 320 (hits of a 131,072-ray tunnel scan: 16.6 -> 13.8 us; of
// outdoor scans into unknown space 20.3 -> 15.0 us).
struct HitShared {
  unsigned long long val[kBlock * 10];
  long long base[kBlock];  // first moment word of the sample's voxel, -1: none
};
template <bool kOcc, bool kCounts, bool kNdt>
__device__ __forceinline__ void hit_ray(const DeviceMap& m, long long i, bool active, HitShared* sh) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int F = m.frac_bits;
  const long long U = 1LL << F;
  bool ok = false;
  long long b[3] = {0, 0, 0};
  int32_t vx = 0, vy = 0, vz = 0, slot = 0;
  uint32_t mo = 0;
  if (active) {
    const RayRec r = m.rays[i];
    if (r.flags & kRaySample) {
      ray_end(r, F, b);
      vx = (int32_t)(b[0] >> F);
      vy = (int32_t)(b[1] >> F);
      vz = (int32_t)(b[2] >> F);
      slot = region_slot_of(m, vx, vy, vz);
      if (slot < 0) {
        atomicOr(m.status, kStatusMissing);
      } else {
        ok = true;
        mo = local_morton(vx, vy, vz);
      }
    }
  }
  // the NDT block is looked up before the occupancy update, so that the two
  // loads are in flight together
  int32_t ns = -1;
  if (kNdt && ok) ns = m.ndt_slot[slot];
  const long long off = ok ? voxel_offset(slot, mo) : 0;
  const unsigned grp = __match_any_sync(full, ok ? (uint32_t)off : 0xffffffffu);  // offsets are < 2^31
  const bool lead = ok && lane == __ffs(grp) - 1;
  const unsigned int n = __popc(grp);
  if (kOcc && lead) logodds_update_n(m, m.occ + off, m.hit, n);
  if (kCounts && lead) atomicAdd(global_ptr(m.counts) + off, (unsigned long long)n << 32);
  if (ok && (m.layers & kLayerMean)) {
    // 10-bit position inside the voxel per axis; per-call sums (x | y << 32, z | count << 32)
    unsigned long long* const acc = global_ptr(m.vmean_acc) + 2 * off;
    const unsigned long long p0 =
        sub_voxel10(b[0] - (long long)vx * U, F) | (sub_voxel10(b[1] - (long long)vy * U, F) << 32);
    const unsigned long long p1 = sub_voxel10(b[2] - (long long)vz * U, F) | (1ULL << 32);
    atomicAdd(acc, p0);
    const unsigned long long prev = atomicAdd(acc + 1, p1);
    if ((prev >> 32) == 0) m.mean_list[atomicAdd(&m.calls->mean_touched, 1)] = (int32_t)off;
  }
  if (kNdt && __any_sync(full, ok)) {
    if (ok && ns < 0) atomicOr(m.status, kStatusMissing);
    unsigned long long* const val = sh->val + 10 * (threadIdx.x & ~31u);
    long long* const base = sh->base + (threadIdx.x & ~31u);
    const unsigned long long px = (unsigned long long)(b[0] - (long long)vx * U);
    const unsigned long long py = (unsigned long long)(b[1] - (long long)vy * U);
    const unsigned long long pz = (unsigned long long)(b[2] - (long long)vz * U);
    const unsigned long long vals[10] = {1, px, py, pz, px * px, px * py, px * pz, py * py, py * pz, pz * pz};
    base[lane] = ok && ns >= 0 ? ndt_moments(m, ns, mo) - m.ndt : -1;
#pragma unroll
    for (int k = 0; k < 10; ++k) val[10 * lane + k] = vals[k];
    __syncwarp();
    unsigned long long* const ndt = reinterpret_cast<unsigned long long*>(global_ptr(m.ndt));
#pragma unroll
    for (int k = 0; k < 10; ++k) {
      const int j = 32 * k + lane, of = j / 10;
      if (base[of] >= 0) atomicAdd(ndt + base[of] + (j - 10 * of), val[j]);
    }
    __syncwarp();
  }
}

// The fixed-point TSDF band [a, b] and direction of a ray, and its float length
// (Sec. II-F): from range max(0, d - tau) to d + tau, quantised like a
// truncated endpoint.  In float-float where that settles the range test and
// the band, else in double.  False: out of range or extent.
__device__ __forceinline__ bool tsdf_ray_band(const DeviceMap& m, const long long qo[3], const long long qe[3],
                                              long long a[3], long long b[3], float u[3], float* len_out) {
  const int F = m.frac_bits;
  bool in_range = false;
  if (!tsdf_band_ff(qo, qe, m.band, &in_range, a, b, u, len_out)) {
    double d[3];
    const double len = ray_length(qo, qe, d);
    in_range = len > m.rmin_q && len <= m.rmax_q;
    if (in_range && in_extent(qo, F) && in_extent(qe, F)) tsdf_band(qo, d, len, m.tau_q, a, b, u);
    *len_out = (float)len;
  }
  return in_range && in_extent(qo, F) && in_extent(qe, F);
}

// The record of a TSDF band's walk; returns the voxels it visits.
__device__ __forceinline__ int32_t tsdf_record(const long long a[3], const long long b[3], const long long qe[3], int F,
                                               TsdfRec* t) {
  const int M = longest_axis(a, b);
  t->r.flags = kRayValid | (M << kRayAxisShift);
  t->r.nseg = 1;
  ray_constants(a, b, F, &t->r);
  const int32_t nmaj = M == 0 ? t->r.n[0] : (M == 1 ? t->r.n[1] : t->r.n[2]);
  t->r.inv = nmaj < kPieceSlots ? 0 : reciprocal64((unsigned long long)(M == 0 ? t->r.A[0] : (M == 1 ? t->r.A[1] : t->r.A[2])));
#pragma unroll
  for (int k = 0; k < 3; ++k) t->e[k] = (int32_t)(qe[k] - (((long long)t->r.v0[k] << F) + (1LL << (F - 1))));
  return t->r.n[0] + t->r.n[1] + t->r.n[2] + 1;
}

// TSDF band of one ray: its record, and its regions inserted.  Full warp, like
// prepare_occ_ray.  The lanes whose band lies in one region (neighbouring
// pixels: most of a warp) insert it once.
__device__ __forceinline__ void prepare_tsdf_ray(const DeviceMap& m, const CallArgs& args, long long i, bool active) {
  active = active && !latched(m);
  const CallOrigin origin = call_origin(m, args);
  const int F = m.frac_bits;
  unsigned int nvisit = 0;
  TsdfRec r;
  r.r.flags = 0;
  long long a[3], b[3];
  bool ok = false, one = false;
  long long key = -1;
  if (active) {
    float o[3], e[3];
    uint8_t flag;
    load_ray(args, i, o, e, &flag);
    long long qo[3], qe[3];
    float len;
    ok = quantise_call_ray(m, args, origin, o, e, qo, qe) && (flag & kFlagNoReturn) == 0 &&
         tsdf_ray_band(m, qo, qe, a, b, r.u, &len);
    if (ok) {
      nvisit = (unsigned int)tsdf_record(a, b, qe, F, &r);
      const int S = F + kRegionShift;
      one = (a[0] >> S) == (b[0] >> S) && (a[1] >> S) == (b[1] >> S) && (a[2] >> S) == (b[2] >> S);
      if (one) key = pack_region((int)(a[0] >> S), (int)(a[1] >> S), (int)(a[2] >> S));
      m.trays[i] = r;
    } else {
      m.trays[i].r.flags = 0;
    }
  }
  const unsigned grp = __match_any_sync(0xffffffffu, one ? key : -1LL - (long long)(threadIdx.x & 31));
  if (ok && (!one || (int)(threadIdx.x & 31) == __ffs(grp) - 1)) insert_ray_regions(m, a, b);
  warp_add(&m.calls->visits, nvisit);
}

// TSDF band walk of one ray: per visited voxel c, s = (e - c).u (equal to
// d - (c - o).u), truncated to [-tau, tau], summed in 2^-32 m fixed point
// with a count.  The first visitor of a voxel in this call records it for the
// apply pass.
//
// Every lane of the warp calls this together (active = false for a lane
// without a ray of this map); blocks have kBlock threads, tab is the thread's
// column of region bases (WalkShared::tab), acc 64 words of the warp that stand
// at zero.  The walk is the local walk of the miss phase.  Neighbouring
// pixels' rays cross the same band voxels (a 5 cm voxel at 1-2 m is crossed by
// hundreds of them per frame), so the updates are aggregated per warp: where
// kTsdfReduce lanes or more stand in the voxel of the lowest lane, one warp
// reduction adds them up (the sum in two halves of 32 bits); the other lanes
// are grouped by __match_any_sync and summed in shared memory.  Each group
// adds its count and sum with one atomic each.  The sums are of integers, so
// the result does not depend on the grouping.  The first visitors the counts
// reveal are appended to the touched list with one atomic per warp and batch.
// Measured on 640 x 480 frames at 5 cm: 72 us with the 64-bit walker, rows of 32
// pixels per warp and each group's leader adding up its lanes; with the local
// walk and 8 x 4 pixel tiles 106 us in that form, 80 / 96 / 209 us reducing up to 3 /
// 6 / 12 groups, 56 us with shared sums alone, 41 us compiled for 4 blocks per SM
// (the launch's two full waves), 40 us in this form.
constexpr int kTsdfReduce = 8;
__device__ __forceinline__ void tsdf_walk_ray(const DeviceMap& m, long long i, bool active, uint32_t* tab,
                                              uint32_t* acc) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int F = m.frac_bits;
  const float to_m = (float)(m.voxel_size / (double)(1LL << F));
  unsigned int* const cnt = global_ptr(m.tsdf_cnt);
  unsigned long long* const sum = reinterpret_cast<unsigned long long*>(global_ptr(m.tsdf_sum));
  const TsdfRec* rec = global_ptr(m.trays) + (active ? i : 0);
  const bool small = m.tau_m < 1000.0f;  // |s| 2^32 < 2^42: the high halves of 32 lanes add up in 32 bits
  bool more = active && (rec->r.flags & kRayValid);
  float u[3] = {0.f, 0.f, 0.f};
  if (more) {
#pragma unroll
    for (int k = 0; k < 3; ++k) u[k] = rec->u[k];
  }
  for (int32_t K = 0; __any_sync(full, more); K += kPieceSlots) {
    LWalker w = {};
    uint32_t mo = 0;
    int32_t left = 0, rel[3] = {0, 0, 0}, d[3] = {0, 0, 0};
    if (more) {
      const RayRec r = rec->r;
      const int M = (r.flags >> kRayAxisShift) & 3;
      const int32_t nmaj = M == 0 ? r.n[0] : (M == 1 ? r.n[1] : r.n[2]);
      const int32_t Ke = K + kPieceSlots < nmaj + 1 ? K + kPieceSlots : nmaj + 1;
      PieceStart p;
      piece_start(r, F, K, Ke, Ke == nmaj + 1, &p, &w);
      left = p.visits;
      more = Ke < nmaj + 1;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        rel[k] = rec->e[k] - ((p.v[k] - r.v0[k]) << F);
        d[k] = ((r.flags >> (kRaySignShift + k)) & 1) ? 1 << F : -(1 << F);
      }
      if (!piece_regions(m, p, w, r.flags, tab, &mo)) {
        atomicOr(m.status, kStatusMissing);
        left = 0;
      }
    }
    for (int rounds = __reduce_max_sync(full, left > 0 ? left + kFastBatch - 1 : 0) / kFastBatch; rounds > 0; --rounds) {
      uint32_t at[kFastBatch], off[kFastBatch], valid;
      piece_fill(m, &rec->r, K, tab, w, mo, left, at, off, valid);
      unsigned int prev[kFastBatch];
#pragma unroll
      for (int j = 0; j < kFastBatch; ++j) {
        float sv = ((float)rel[0] * u[0] + (float)rel[1] * u[1] + (float)rel[2] * u[2]) * to_m;
        sv = fminf(fmaxf(sv, -m.tau_m), m.tau_m);
        const long long sq = __float2ll_rn(sv * 4294967296.0f);
        const uint32_t moved = at[j] ^ (j + 1 < kFastBatch ? at[j + 1] : mo);
        if (moved & 0x9249u)
          rel[0] += d[0];
        else if (moved & 0x12492u)
          rel[1] += d[1];
        else
          rel[2] += d[2];
        const bool in = (valid >> j) & 1u;
        prev[j] = 1u;
        unsigned todo = __ballot_sync(full, in);
        if (!small) {
          if (in) {
            prev[j] = atomicAdd(cnt + off[j], 1u);
            atomicAdd(sum + off[j], (unsigned long long)sq);
          }
          continue;
        }
        if (!todo) continue;
        // the voxel of the lowest lane, where it holds a good part of the warp
        const uint32_t lo = (uint32_t)sq & 0xffffu;
        const int32_t hi = (int32_t)(sq >> 16);
        const int lead0 = __ffs(todo) - 1;
        const uint32_t voxel = __shfl_sync(full, off[j], lead0);
        bool rest = in;
        const bool mine = in && off[j] == voxel;
        const unsigned grp0 = __ballot_sync(full, mine);
        if (__popc(grp0) >= kTsdfReduce) {
          const uint32_t slo = __reduce_add_sync(full, mine ? lo : 0u);
          const int32_t shi = __reduce_add_sync(full, mine ? hi : 0);
          if (lane == lead0) {
            prev[j] = atomicAdd(cnt + off[j], (unsigned int)__popc(grp0));
            atomicAdd(sum + off[j], (unsigned long long)(((long long)shi << 16) + (long long)slo));
          }
          rest = in && !mine;
          todo &= ~grp0;
          if (!todo) continue;
        }
        // the others: sums of each voxel's lanes in shared memory, at its lowest lane
        const unsigned grp = __match_any_sync(full, rest ? off[j] : (kNoRegion | (uint32_t)lane));
        const int lead = __ffs(grp) - 1;
        if (rest) {
          atomicAdd(acc + lead, lo);
          atomicAdd(acc + 32 + lead, (uint32_t)hi);
        }
        __syncwarp();
        if (rest && lane == lead) {
          const long long tot = ((long long)(int32_t)acc[32 + lead] << 16) + acc[lead];
          acc[lead] = 0;
          acc[32 + lead] = 0;
          prev[j] = atomicAdd(cnt + off[j], (unsigned int)__popc(grp));
          atomicAdd(sum + off[j], (unsigned long long)tot);
        }
        __syncwarp();
      }
      uint32_t first = 0;
#pragma unroll
      for (int j = 0; j < kFastBatch; ++j)
        if (prev[j] == 0) first |= 1u << j;
      // first visitors of a voxel in this call: one table range per warp
      if (!__any_sync(full, first != 0)) continue;
      const unsigned int nf = __popc(first);
      unsigned int incl = nf;
#pragma unroll
      for (int s = 1; s < 32; s <<= 1) {
        const unsigned int t = __shfl_up_sync(full, incl, s);
        if (lane >= s) incl += t;
      }
      unsigned long long base = 0;
      if (lane == 31) base = atomicAdd(&m.calls->touched, (unsigned long long)incl);
      base = __shfl_sync(full, base, 31);
      unsigned long long pos = base + (incl - nf);
#pragma unroll
      for (int j = 0; j < kFastBatch; ++j) {
        if ((first >> j) & 1u) {
          if (pos < (unsigned long long)m.max_touched)
            m.touched[pos] = (int32_t)off[j];
          else
            atomicOr(m.status, kStatusScratch);
          ++pos;
        }
      }
    }
  }
}

// Weighted average of one touched voxel: D <- (W D + sum s) / (W + c),
// W <- min(W + c, W_max); the per-call sums are cleared for the next call.
__device__ __forceinline__ void tsdf_apply_one(const DeviceMap& m, long long t) {
  const int32_t off = m.touched[t];
  const unsigned int c = m.tsdf_cnt[off];
  const long long sum = m.tsdf_sum[off];
  m.tsdf_cnt[off] = 0;
  m.tsdf_sum[off] = 0;
  // in float (D and W are stored as floats; W and W + c are integers below
  // 2^24, exact): the rounding of D is far below the layer's 1e-5 m
  // tolerance, and the device's double division is slow
  const float2 dw = m.tsdf[off];
  const float S = (float)sum * 2.3283064365386962890625e-10f;  // 2^-32
  const float Wn = dw.y + (float)c;
  const float Dn = (dw.y * dw.x + S) / Wn;
  m.tsdf[off] = make_float2(Dn, fminf(Wn, m.wmax));
}

// Voxel-mean update of one voxel given samples by the call: per axis
// m <- floor((m n + S + floor((n + c) / 2)) / (n + c)), n <- min(n + c, 2^32 - 1);
// the per-call sums are cleared.  apply = false (a failed call) only clears.
__device__ __forceinline__ void mean_apply_one(const DeviceMap& m, long long t, bool apply) {
  const int32_t off = m.mean_list[t];
  const unsigned long long a0 = m.vmean_acc[2LL * off], a1 = m.vmean_acc[2LL * off + 1];
  m.vmean_acc[2LL * off] = 0;
  m.vmean_acc[2LL * off + 1] = 0;
  if (!apply) return;
  const unsigned long long S[3] = {a0 & 0xffffffffULL, a0 >> 32, a1 & 0xffffffffULL};
  const unsigned long long c = a1 >> 32;
  const unsigned long long w = m.vmean[off];
  const unsigned long long n0 = w >> 32, nt = n0 + c;
  unsigned long long packed = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const unsigned long long mk = (w >> (10 * k)) & 1023ULL;
    packed |= ((mk * n0 + S[k] + nt / 2) / nt) << (10 * k);
  }
  m.vmean[off] = ((nt < 0xffffffffULL ? nt : 0xffffffffULL) << 32) | packed;
}

__device__ __forceinline__ long long mean_touched_count(const DeviceMap& m) { return (long long)m.calls->mean_touched; }

__device__ __forceinline__ long long touched_count(const DeviceMap& m) {
  unsigned long long nt = m.calls->touched;
  return (long long)(nt > (unsigned long long)m.max_touched ? (unsigned long long)m.max_touched : nt);
}

// Undo the allocations of a failed call (threads t0, t0 + stride, ...): keys
// inserted by it become tombstones, keys it asked to restore go back to
// "evicted", its NDT blocks are released, and the pool counters and free-list
// positions are restored.  Stamps stay: regions the call touched count as
// recently used.
__device__ __forceinline__ void rollback_call(const DeviceMap& m, long long t0, long long stride) {
  const int32_t seq = m.calls->seq;
  for (long long h = t0; h <= (long long)m.hmask; h += stride) {
    const longlong2 e = m.htab[h];
    if (e.x == kEmptyKey || e.x == kTombKey) continue;
    if (e.y == kSlotRestoring)
      m.htab[h].y = kSlotEvicted;
    else if (e.y == kSlotPending || (e.y >= 0 && m.born[e.y] == seq))
      m.htab[h] = make_longlong2(kTombKey, -1);
  }
  for (long long s = t0; s < m.max_regions; s += stride) {
    const int32_t v = m.ndt_slot[s];
    if (v == -2 || (v >= 0 && (m.ndt_born[s] == seq || m.born[s] == seq))) m.ndt_slot[s] = -1;
  }
  if (t0 == 0) {
    *m.region_count = m.calls->region_start;
    *m.ndt_count = m.calls->ndt_start;
    m.free_info[1] = m.calls->free_used_start;
    m.free_info[3] = m.calls->ndt_free_used_start;
  }
}

}  // namespace ohm
