// Ray integration kernels (Sec. III-B, III-C of arxiv 2206.06079, re-designed
// for sm_103a).
//
// One integrate call is one "ray set".  Kernels, in stream order:
//   k_prepare_occ    per ray: fixed-point quantisation, max-range truncation,
//                    region walk with hash insertion (the paper does this on
//                    the CPU, Sec. III-B; here it is a device pass), the
//                    segment table (Sec. III-B ray segments), and the NDT
//                    block of the sample's region
//   k_ndt_alloc      sample rays prepare left: give their regions an NDT layer
//   k_prepare_tsdf   per ray: TSDF band end points and their regions
//   k_walk_fast      per segment: exact voxel walk, miss update per voxel,
//                    counts and decay path lengths
//   k_hits           per sample: hit update, hit count, NDT moments
//   k_tsdf_walk      per ray: band walk, fixed-point s sums and counts
//   k_tsdf_apply     per touched voxel: weighted average, scratch cleared
//   k_end            if any kernel latched a failure: undo the allocations;
//                    counters and rollback point made ready for the next call
// Every kernel returns at once when the status word is set, so
// a failed call changes no voxel.
#include "ohm_kernels.cuh"

namespace ohm {

#define OHM_GRID_STRIDE(i, n) \
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < (n); i += (long long)gridDim.x * blockDim.x)

// Bound by latency and divergence: a ray is one thread's chain of region
// lookups, so in a call that fits one wave the SM with the most rays ends it.
// Blocks of 128 rays share such a call out more evenly than blocks of 256 (131,072
// rays on 152 SMs: at most 7 x 128 a SM instead of 4 x 256): a tunnel scan
// 51.0 -> 47.2 us, outdoors 35.5 -> 34.9.  A call of several waves is faster in
// blocks of 256 (262,144 rays: 67.3 against 72.7 us).
constexpr int kPrepareWaveBlock = 128;
template <int kThreads>
__global__ void __launch_bounds__(kThreads, OHM_PREPARE_MIN_BLOCKS * kBlock / kThreads)
    k_prepare_occ(DeviceMap m, CallArgs args) {
  chain_enter();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  prepare_occ_ray(m, args, i, i < args.n);
}

// Blocks of the NDT pass: it has only the rays prepare could not settle (a
// few per scan), read from the device-side count.
constexpr int kNdtPendingGrid = 64;

// The sample rays whose region slot prepare did not learn (another thread
// was inserting the region at the time): their regions get NDT blocks here.
__global__ void __launch_bounds__(kBlock) k_ndt_alloc(DeviceMap m) {
  chain_enter();
  if (latched(m)) return;
  const long long n = (long long)m.calls->ndt_pending;
  OHM_GRID_STRIDE(k, n) ndt_alloc_ray(m, m.ndt_pending[k]);
}

// The miss walk (walk_segments); kVariant: walk_variant.
template <int kVariant>
__global__ void __launch_bounds__(kBlock, OHM_FAST_MIN_BLOCKS) k_walk_fast(DeviceMap m) {
  constexpr bool kOcc = (kVariant & 4) != 0, kCounts = (kVariant & 2) != 0, kCas = (kVariant & 1) != 0;
  constexpr bool kDecay = (kVariant & kWalkDecay) != 0;
  chain_enter();
  if (latched(m)) return;
  __shared__ WalkShared sh;
  const long long nseg = (long long)m.calls->segments;
  const long long stride = (long long)gridDim.x * kBlock;
  unsigned int ops = 0;
  walk_shared_init(sh);
  long long si = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  int2 sg = si < nseg ? m.segs[si] : make_int2(0, 0);
  // whole warps iterate together
  for (; si - (threadIdx.x & 31) < nseg; si += stride) {
    // the next segment's table entry is loaded while this one walks
    const int2 next = si + stride < nseg ? m.segs[si + stride] : make_int2(-1, 0);
    walk_segments<kOcc, kCounts, kCas, kDecay>(m, si < nseg, sg, sh, ops, next.x >= 0 ? m.rays + next.x : nullptr);
    sg = next;
  }
  if (kOcc && !kCas) ops += drain_open(m, sh, 1u);
  // every thread gets here: one atomic per warp for the call's atomic count
  ops = __reduce_add_sync(0xffffffffu, ops);
  if ((threadIdx.x & 31) == 0 && ops) atomicAdd(&m.calls->atomics, (unsigned long long)ops);
}

template <bool kOcc, bool kCounts, bool kNdt>
__global__ void __launch_bounds__(kBlock) k_hits(DeviceMap m, long long n) {
  chain_enter();
  if (latched(m)) return;
  __shared__ HitShared sh;
  // whole warps iterate together (the update is warp-collective)
  const long long np = (n + 31) & ~31LL;
  OHM_GRID_STRIDE(i, np) hit_ray<kOcc, kCounts, kNdt>(m, i, i < n, &sh);
}

// Runs for failed calls too: it then only clears the per-call sums.
__global__ void __launch_bounds__(kBlock) k_mean_apply(DeviceMap m) {
  chain_enter();
  const bool apply = !latched(m);
  const long long nt = mean_touched_count(m);
  OHM_GRID_STRIDE(t, nt) mean_apply_one(m, t, apply);
}

// Compiled for 4 blocks per SM (64 registers; 78 unbounded, which fits 3).
__global__ void __launch_bounds__(kBlock, 4) k_prepare_tsdf(DeviceMap m, CallArgs args) {
  chain_enter();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  prepare_tsdf_ray(m, args, i, i < args.n);
}

// Compiled for 4 blocks per SM, which the launch counts on.
__global__ void __launch_bounds__(kBlock, 4) k_tsdf_walk(DeviceMap m, long long n) {
  chain_enter();
  if (latched(m)) return;
  __shared__ uint32_t tab[8 * kBlock];
  __shared__ uint32_t acc[2 * kBlock];
  acc[threadIdx.x] = acc[kBlock + threadIdx.x] = 0;
  __syncthreads();
  // whole warps iterate together (the walk is warp-collective)
  const long long np = (n + 31) & ~31LL;
  OHM_GRID_STRIDE(i, np) tsdf_walk_ray(m, i, i < n, tab + threadIdx.x, acc + 2 * (threadIdx.x & ~31u));
}

__global__ void __launch_bounds__(kBlock) k_tsdf_apply(DeviceMap m) {
  chain_enter();
  if (latched(m)) return;
  const long long nt = touched_count(m);
  OHM_GRID_STRIDE(t, nt) tsdf_apply_one(m, t);
}

__global__ void k_end(DeviceMap m, long long n) {
  chain_enter();
  if (blockIdx.x == 0 && threadIdx.x == 0) finish_call(m, n);
  if (!latched(m)) return;
  rollback_call(m, (long long)blockIdx.x * blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x);
}

// The pool counters changed between calls (region cache).
__global__ void k_snapshot(DeviceMap m) { snapshot_pool(m); }

// ---------------------------------------------------------------------------
// Query and export.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kBlock) k_query(DeviceMap m, const float* pts, long long n, float* occupancy,
                                                   uint8_t* known, float* ndt, float* tsdf, uint32_t* counts,
                                                   unsigned long long* path_sum, float* mean) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int F = m.frac_bits;
  long long q[3];
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 3; ++k) ok = quantise_coord(m, pts[3 * i + k], k, &q[k]) && ok;
  ok = ok && in_extent(q, F);
  int32_t slot = -1;
  uint32_t mo = 0;
  int32_t v[3] = {0, 0, 0};
  if (ok) {
    v[0] = (int32_t)(q[0] >> F);
    v[1] = (int32_t)(q[1] >> F);
    v[2] = (int32_t)(q[2] >> F);
    slot = region_slot_of(m, v[0], v[1], v[2]);
    mo = local_morton(v[0], v[1], v[2]);
  }
  const long long off = voxel_offset(slot, mo);
  if (occupancy || known) {
    float l = __int_as_float(0x7fc00000);
    if (slot >= 0 && (m.layers & kLayerOcc)) l = logodds_read(m.occ[off], m.l_min);
    if (occupancy) occupancy[i] = l;
    if (known) known[i] = (l == l) ? 1 : 0;
  }
  if (path_sum) path_sum[i] = (slot >= 0 && (m.layers & kLayerDecay)) ? m.decay[off] : 0ULL;
  if (mean) {
    const unsigned long long w = (slot >= 0 && (m.layers & kLayerMean)) ? m.vmean[off] : 0ULL;
    const unsigned long long cnt = w >> 32;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double frac = ((double)((w >> (10 * k)) & 1023ULL) + 0.5) / 1024.0;
      mean[4 * i + k] = cnt ? (float)(m.origin[k] + ((double)v[k] + frac) * m.voxel_size) : __int_as_float(0x7fc00000);
    }
    mean[4 * i + 3] = (float)cnt;
  }
  if (counts) {
    unsigned long long c = 0;
    if (slot >= 0 && (m.layers & kLayerCounts)) c = m.counts[off];
    counts[2 * i + 0] = (uint32_t)(c >> 32);
    counts[2 * i + 1] = (uint32_t)(c & 0xffffffffu);
  }
  if (tsdf) {
    float2 dw = make_float2(0.f, 0.f);
    if (slot >= 0 && (m.layers & kLayerTsdf)) dw = m.tsdf[off];
    tsdf[2 * i + 0] = dw.x;
    tsdf[2 * i + 1] = dw.y;
  }
  if (ndt) {
    float out[10];
#pragma unroll
    for (int k = 0; k < 10; ++k) out[k] = 0.f;
    const int32_t ns = (slot >= 0 && (m.layers & kLayerNdt)) ? m.ndt_slot[slot] : -1;
    if (ns >= 0) {
      const longlong2* base = reinterpret_cast<const longlong2*>(ndt_moments(m, ns, mo));
      long long s[10];
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        const longlong2 p = base[k];
        s[2 * k] = p.x;
        s[2 * k + 1] = p.y;
      }
      if (s[0] > 0) {
        // In double, with one reciprocal for the nine quotients (a rounding
        // or two of 2^-53 more each, far below the float outputs') and the
        // exact numerators of the covariance in 64 bits where they fit:
        // n Sxx <= n^2 2^(2F) < 2^62.  A double instruction takes a warp 64
        // cycles of a scheduler; nine divisions and six 128-bit conversions
        // made this 18.5 us for 20,000 points; 10.3 us this way.
        const double cnt = (double)s[0], inv = 1.0 / cnt;
        const double cell = m.voxel_size / (double)(1LL << F);
        out[0] = (float)cnt;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const double corner = (double)((long long)v[k] * (1LL << F));
          out[1 + k] = (float)(m.origin[k] + (corner + (double)s[1 + k] * inv) * cell);
        }
        const int pa[6] = {0, 0, 0, 1, 1, 2}, pb[6] = {0, 1, 2, 1, 2, 2};
        const double scale = inv * cell, scale2 = scale * scale;
        if (s[0] < (1LL << (31 - F))) {
#pragma unroll
          for (int k = 0; k < 6; ++k)
            out[4 + k] = (float)((double)(s[0] * s[4 + k] - s[1 + pa[k]] * s[1 + pb[k]]) * scale2);
        } else {
#pragma unroll 1
          for (int k = 0; k < 6; ++k) {
            const __int128 num = (__int128)s[0] * s[4 + k] - (__int128)s[1 + pa[k]] * s[1 + pb[k]];
            out[4 + k] = (float)((double)num * scale2);
          }
        }
      }
    }
#pragma unroll
    for (int k = 0; k < 10; ++k) ndt[10 * i + k] = out[k];
  }
}

// Two neighbouring elements of an exported row; in one store where the output
// is aligned for it (kWide).
template <bool kWide, typename T, typename T2>
__device__ __forceinline__ void store_pair(T* out, T2 v) {
  if (kWide) {
    *reinterpret_cast<T2*>(out) = v;
  } else {
    out[0] = v.x;
    out[1] = v.y;
  }
}

// Export of regions in allocation order, voxels x fastest.  One block per slab
// of two z layers of a region, one 2 x 2 x 2 brick of voxels per thread: in
// Morton order a brick is contiguous (a sector of floats), so every layer is
// read with whole 16-byte loads and written as four x pairs, 16 lanes side by
// side filling a row.  NDT moments are copied row by row in 16-byte pieces,
// five per voxel.  Bound by memory: a map of 192 regions with occupancy,
// counts and NDT (1.16 GB moved) and a lookup took 429 us as one voxel per
// thread, which read scattered floats and wrote 80-byte-strided words; this
// form takes 205 us, 84 % of copy bandwidth.
// kWide: every output pointer is 16-byte aligned.
constexpr int kExportSlabs = 16;
template <bool kWide>
__global__ void __launch_bounds__(kBlock) k_export(DeviceMap m, long long first, int32_t* keys, float* occupancy,
                                                    uint32_t* counts, long long* ndt, float* tsdf,
                                                    unsigned long long* path_sum, unsigned long long* mean) {
  const long long r = blockIdx.x / kExportSlabs;
  const int slab = blockIdx.x % kExportSlabs, t = threadIdx.x;
  const int32_t slot = (int32_t)(first + r);
  if (keys && slab == 0 && t < 3) keys[3 * r + t] = m.region_coords[3 * slot + t];
  const int x = 2 * (t & 15), y = 2 * (t >> 4), z = 2 * slab;
  const long long off = voxel_offset(slot, morton(x, y, z));       // the brick's first voxel
  const long long lin = r * kRegionVoxels + x + 32 * (y + 32 * z);  // and its place in the outputs
  // rows of the brick: (y, z), (y + 1, z), (y, z + 1), (y + 1, z + 1)
  const int row[4] = {0, 32, 1024, 1056};
  if (occupancy) {
    const float4* src = reinterpret_cast<const float4*>(m.occ + off);
    const float4 a = src[0], b = src[1];
    const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
    for (int k = 0; k < 4; ++k)
      store_pair<kWide>(occupancy + lin + row[k],
                        make_float2(logodds_read(v[2 * k], m.l_min), logodds_read(v[2 * k + 1], m.l_min)));
  }
  if (counts) {
    const ulonglong2* src = reinterpret_cast<const ulonglong2*>(m.counts + off);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const ulonglong2 c = src[k];
      uint32_t* o = counts + 2 * (lin + row[k]);
      const uint4 v = make_uint4((uint32_t)(c.x >> 32), (uint32_t)c.x, (uint32_t)(c.y >> 32), (uint32_t)c.y);
      if (kWide) {
        *reinterpret_cast<uint4*>(o) = v;
      } else {
        o[0] = v.x;
        o[1] = v.y;
        o[2] = v.z;
        o[3] = v.w;
      }
    }
  }
  auto words = [&](const unsigned long long* layer, unsigned long long* out) {
    const ulonglong2* src = reinterpret_cast<const ulonglong2*>(layer + off);
#pragma unroll
    for (int k = 0; k < 4; ++k) store_pair<kWide>(out + lin + row[k], src[k]);
  };
  if (path_sum) words(m.decay, path_sum);
  if (mean) words(m.vmean, mean);
  if (tsdf) {
    const float4* src = reinterpret_cast<const float4*>(m.tsdf + off);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float4 v = src[k];
      float* o = tsdf + 2 * (lin + row[k]);
      if (kWide) {
        *reinterpret_cast<float4*>(o) = v;
      } else {
        o[0] = v.x;
        o[1] = v.y;
        o[2] = v.z;
        o[3] = v.w;
      }
    }
  }
  if (ndt) {
    const int32_t ns = m.ndt_slot[slot];
    longlong2* const out = reinterpret_cast<longlong2*>(ndt + (r * kRegionVoxels + 2048LL * slab) * 10);
    // 64 rows of 32 voxels of 5 pieces
#pragma unroll 8
    for (int i = t; i < 64 * 160; i += kBlock) {
      const int vox = i / 5, part = i - 5 * vox;
      longlong2 v = make_longlong2(0, 0);
      if (ns >= 0)
        v = reinterpret_cast<const longlong2*>(ndt_moments(m, ns, morton(vox & 31, (vox >> 5) & 31, z + (vox >> 10))))[part];
      store_pair<kWide>(reinterpret_cast<long long*>(out + i), v);
    }
  }
}

// ---------------------------------------------------------------------------
// Host launchers.
// ---------------------------------------------------------------------------
int walk_blocks_per_sm() {
  int b = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_walk_fast<4>, kBlock, 0);
  return b > 0 ? b : 1;
}

static long long blocks_for(long long n) { return (n + kBlock - 1) / kBlock; }


// Launch one kernel as stage `stage`, with event timing when it is profiled.
#define OHM_LAUNCH(stage, ...)                  \
  do {                                          \
    cudaEvent_t ev_ = nullptr;                  \
    stage_begin(map, (stage), stream, &ev_);    \
    __VA_ARGS__;                                \
    stage_end(map, (stage), stream, ev_);       \
    map->launches += 1;                         \
  } while (0)

cudaError_t launch_integrate(ohm_map* map, const CallArgs& args, cudaStream_t stream) {
  DeviceMap& m = map->d;
  map->profile_call += 1;  // the call's index for sampled stage timing
  const bool occ = (m.layers & kLayerOcc) != 0, cnt = (m.layers & kLayerCounts) != 0, ndt = (m.layers & kLayerNdt) != 0;
  const bool tsdf = (m.layers & kLayerTsdf) != 0;
  const bool mean = (m.layers & kLayerMean) != 0;
  const bool occ_like = occ || cnt || ndt || mean || (m.layers & kLayerDecay);
  const long long n = args.n;
  const int grid = map->walk_blocks;
  // the walk's grid-stride loop runs on OHM_WALK_OVERSUBSCRIBE times the
  // resident blocks: a block whose segments took longer holds its SM while
  // blocks that finished early are replaced by new ones (no long tail)
  const int wgrid = grid * OHM_WALK_OVERSUBSCRIBE;
  const long long per_ray_blocks = blocks_for(n) > 0 ? blocks_for(n) : 1;
  const int ray_grid = (int)(per_ray_blocks < grid ? per_ray_blocks : grid);
  const unsigned prb = (unsigned)per_ray_blocks;
  if (occ_like) {
    if (n <= (long long)map->num_sms * OHM_PREPARE_MIN_BLOCKS * kBlock) {
      const unsigned wave_blocks = (unsigned)((n + kPrepareWaveBlock - 1) / kPrepareWaveBlock);
      OHM_LAUNCH(OHM_STAGE_PREPARE, launch_chained_of(kPrepareWaveBlock, k_prepare_occ<kPrepareWaveBlock>,
                                                      wave_blocks > 0 ? wave_blocks : 1u, stream, m, args));
    } else {
      OHM_LAUNCH(OHM_STAGE_PREPARE, launch_chained(k_prepare_occ<kBlock>, prb, stream, m, args));
    }
    if (ndt) OHM_LAUNCH(OHM_STAGE_NDT_ALLOC, launch_chained(k_ndt_alloc, kNdtPendingGrid, stream, m));
  }
  if (tsdf) OHM_LAUNCH(OHM_STAGE_PREPARE_TSDF, launch_chained(k_prepare_tsdf, prb, stream, m, args));
  switch (walk_variant(m.layers, m.miss, m.ndt_clear)) {
#define OHM_WALK_CASE(v) \
  case v: OHM_LAUNCH(OHM_STAGE_WALK, launch_chained(k_walk_fast<v>, wgrid, stream, m)); break;
    OHM_WALK_VARIANTS(OHM_WALK_CASE)
#undef OHM_WALK_CASE
    default: break;  // kWalkNone
  }
  if (occ || cnt || ndt || mean) {
    const int sel = (occ ? 4 : 0) | (cnt ? 2 : 0) | (ndt ? 1 : 0);
    switch (sel) {
      case 7: OHM_LAUNCH(OHM_STAGE_HITS, launch_chained(k_hits<true, true, true>, ray_grid, stream, m, n)); break;
      case 6: OHM_LAUNCH(OHM_STAGE_HITS, launch_chained(k_hits<true, true, false>, ray_grid, stream, m, n)); break;
      case 5: OHM_LAUNCH(OHM_STAGE_HITS, launch_chained(k_hits<true, false, true>, ray_grid, stream, m, n)); break;
      case 4: OHM_LAUNCH(OHM_STAGE_HITS, launch_chained(k_hits<true, false, false>, ray_grid, stream, m, n)); break;
      case 3: OHM_LAUNCH(OHM_STAGE_HITS, launch_chained(k_hits<false, true, true>, ray_grid, stream, m, n)); break;
      case 2: OHM_LAUNCH(OHM_STAGE_HITS, launch_chained(k_hits<false, true, false>, ray_grid, stream, m, n)); break;
      case 1: OHM_LAUNCH(OHM_STAGE_HITS, launch_chained(k_hits<false, false, true>, ray_grid, stream, m, n)); break;
      default: OHM_LAUNCH(OHM_STAGE_HITS, launch_chained(k_hits<false, false, false>, ray_grid, stream, m, n)); break;
    }
    if (mean) OHM_LAUNCH(OHM_STAGE_MEAN_APPLY, launch_chained(k_mean_apply, ray_grid, stream, m));
  }
  if (tsdf) {
    OHM_LAUNCH(OHM_STAGE_TSDF_WALK, launch_chained(k_tsdf_walk, ray_grid, stream, m, n));
    OHM_LAUNCH(OHM_STAGE_TSDF_APPLY, launch_chained(k_tsdf_apply, grid, stream, m));
  }
  // one block per SM: the body only runs (a grid-stride rollback) after a failure
  OHM_LAUNCH(OHM_STAGE_END, launch_chained(k_end, (unsigned)map->num_sms, stream, m, n));
  return cudaGetLastError();
}

// 64-bit finaliser of SplitMix64 (Steele, Lea, Flood 2014), a published mixer.
__device__ __forceinline__ unsigned long long splitmix64_mix(unsigned long long z) {
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
  return z ^ (z >> 31);
}

// Throughput probe: per round, four random words are loaded, then each is
// compare-and-swapped to its value + 1.
__global__ void __launch_bounds__(kBlock, 4) k_probe_cas(unsigned int* buf, unsigned long long mask, int rounds) {
  const unsigned long long threads = (unsigned long long)gridDim.x * blockDim.x;
  const unsigned long long t = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (int r = 0; r < rounds; ++r) {
    unsigned long long a[4];
    unsigned int old[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) a[j] = splitmix64_mix((unsigned long long)r * threads * 4 + t * 4 + j) & mask;
#pragma unroll
    for (int j = 0; j < 4; ++j) old[j] = buf[a[j]];
#pragma unroll
    for (int j = 0; j < 4; ++j) atomicCAS(buf + a[j], old[j], old[j] + 1u);
  }
}

cudaError_t probe_cas_rate(int device, long long words, long long ops, double* rate) {
  int sms = 0;
  cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  if (e != cudaSuccess) return e;
  const unsigned long long threads = (unsigned long long)sms * 4 * kBlock;
  int rounds = (int)(ops / (long long)(threads * 4));
  if (rounds < 1) rounds = 1;
  unsigned int* buf = nullptr;
  e = cudaMalloc(reinterpret_cast<void**>(&buf), sizeof(unsigned int) * (size_t)words);
  if (e != cudaSuccess) return e;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  e = cudaMemset(buf, 0, sizeof(unsigned int) * (size_t)words);
  if (e == cudaSuccess) e = cudaEventCreate(&e0);
  if (e == cudaSuccess) e = cudaEventCreate(&e1);
  if (e == cudaSuccess) {
    k_probe_cas<<<sms * 4, kBlock>>>(buf, (unsigned long long)words - 1, rounds);  // warm-up
    cudaEventRecord(e0);
    k_probe_cas<<<sms * 4, kBlock>>>(buf, (unsigned long long)words - 1, rounds);
    cudaEventRecord(e1);
    e = cudaEventSynchronize(e1);
  }
  float ms = 0.f;
  if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
  if (e == cudaSuccess) *rate = (double)threads * 4.0 * rounds / (ms * 1e-3);
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  cudaFree(buf);
  return e;
}

// Probe kernels for ohm_probe_rate; per round each thread touches kProbeInFlight
// random locations: a float atomic add of 1 to a word (fire and forget), a
// load then compare-and-swap of a word, or a load of a word of a random
// 32-byte sector then a store of it plus one (the sector is read from and
// written back to memory when the buffer is larger than L2).
constexpr int kProbeInFlight = 8;
template <int kKind>
__global__ void __launch_bounds__(kBlock) k_probe(unsigned int* buf, unsigned long long mask, int rounds) {
  const unsigned long long threads = (unsigned long long)gridDim.x * blockDim.x;
  const unsigned long long t = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (int r = 0; r < rounds; ++r) {
    unsigned long long a[kProbeInFlight];
#pragma unroll
    for (int j = 0; j < kProbeInFlight; ++j)
      a[j] = splitmix64_mix(((unsigned long long)r * threads + t) * kProbeInFlight + j) & mask;
    if (kKind == OHM_PROBE_L2_ADD) {
#pragma unroll
      for (int j = 0; j < kProbeInFlight; ++j) atomicAdd(reinterpret_cast<float*>(buf) + a[j], 1.0f);
    } else {
      unsigned int old[kProbeInFlight];
      if (kKind == OHM_PROBE_SECTOR_RMW) {
#pragma unroll
        for (int j = 0; j < kProbeInFlight; ++j) a[j] = (a[j] << 3) | (t & 7);  // word t % 8 of sector a
      }
#pragma unroll
      for (int j = 0; j < kProbeInFlight; ++j) old[j] = buf[a[j]];
#pragma unroll
      for (int j = 0; j < kProbeInFlight; ++j) {
        if (kKind == OHM_PROBE_L2_CAS)
          atomicCAS(buf + a[j], old[j], old[j] + 1u);
        else
          buf[a[j]] = old[j] + 1u;
      }
    }
  }
}

cudaError_t probe_rate(int device, int kind, long long units, long long ops, double* rate) {
  int sms = 0;
  cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  if (e != cudaSuccess) return e;
  const int blocks = sms * 8;
  const unsigned long long threads = (unsigned long long)blocks * kBlock;
  int rounds = (int)(ops / (long long)(threads * kProbeInFlight));
  if (rounds < 1) rounds = 1;
  const long long words = kind == OHM_PROBE_SECTOR_RMW ? units * 8 : units;
  unsigned int* buf = nullptr;
  e = cudaMalloc(reinterpret_cast<void**>(&buf), sizeof(unsigned int) * (size_t)words);
  if (e != cudaSuccess) return e;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  e = cudaMemset(buf, 0, sizeof(unsigned int) * (size_t)words);
  if (e == cudaSuccess) e = cudaEventCreate(&e0);
  if (e == cudaSuccess) e = cudaEventCreate(&e1);
  const unsigned long long mask = (unsigned long long)units - 1;
  auto launch = [&]() {
    if (kind == OHM_PROBE_L2_ADD)
      k_probe<OHM_PROBE_L2_ADD><<<blocks, kBlock>>>(buf, mask, rounds);
    else if (kind == OHM_PROBE_L2_CAS)
      k_probe<OHM_PROBE_L2_CAS><<<blocks, kBlock>>>(buf, mask, rounds);
    else
      k_probe<OHM_PROBE_SECTOR_RMW><<<blocks, kBlock>>>(buf, mask, rounds);
  };
  float best = 0.f;
  if (e == cudaSuccess) {
    launch();  // warm-up (and L2 fill for the L2-resident kinds)
    for (int rep = 0; rep < 3 && e == cudaSuccess; ++rep) {
      cudaEventRecord(e0);
      launch();
      cudaEventRecord(e1);
      e = cudaEventSynchronize(e1);
      float ms = 0.f;
      if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
      if (e == cudaSuccess && (best == 0.f || ms < best)) best = ms;
    }
  }
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e == cudaSuccess) *rate = (double)threads * kProbeInFlight * rounds / (best * 1e-3);
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  cudaFree(buf);
  return e;
}

cudaError_t launch_snapshot(ohm_map* map, cudaStream_t stream) {
  k_snapshot<<<1, 1, 0, stream>>>(map->d);
  return cudaGetLastError();
}

cudaError_t launch_query(ohm_map* map, const float* points, long long n, float* occupancy, uint8_t* known, float* ndt,
                         float* tsdf, uint32_t* counts, unsigned long long* path_sum, float* mean,
                         cudaStream_t stream) {
  if (n > 0)
    k_query<<<(unsigned)blocks_for(n), kBlock, 0, stream>>>(map->d, points, n, occupancy, known, ndt, tsdf, counts,
                                                            path_sum, mean);
  return cudaGetLastError();
}

cudaError_t launch_export(ohm_map* map, long long first, long long count, int32_t* keys, float* occupancy,
                          uint32_t* counts, long long* ndt, float* tsdf, unsigned long long* path_sum,
                          unsigned long long* mean, cudaStream_t stream) {
  if (count > 0) {
    const unsigned blocks = (unsigned)(count * kExportSlabs);  // at most 2^20
    uintptr_t low = 0;
    for (const void* p : {(const void*)occupancy, (const void*)counts, (const void*)ndt, (const void*)tsdf,
                          (const void*)path_sum, (const void*)mean})
      low |= reinterpret_cast<uintptr_t>(p);
    if (low & 15)
      k_export<false><<<blocks, kBlock, 0, stream>>>(map->d, first, keys, occupancy, counts, ndt, tsdf, path_sum, mean);
    else
      k_export<true><<<blocks, kBlock, 0, stream>>>(map->d, first, keys, occupancy, counts, ndt, tsdf, path_sum, mean);
  }
  return cudaGetLastError();
}

}  // namespace ohm
