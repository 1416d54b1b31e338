// Host-side check of the local walk (LWalker, piece_start of ohm_device.cuh)
// that the integrate kernels' miss walk runs: compiles it for the CPU and
// prints, for every ray, the voxels visited by the pieces of all its segments
// in order, with the kernels' six-bit sign-normalised Morton stepping.
//
// stdin:  F S n, then n lines "ax ay az bx by bz" (fixed point)
// stdout: per ray "count" then count lines "x y z"
// stderr: "exact <n> steps <n>" -- near-ties decided exactly, steps taken
// exit codes: 2 Morton or region bit mismatch, 5 piece end or start mismatch
#include <cstdio>

#include "../../paper_2206_06079_gb300/csrc/ohm_device.cuh"

static int vox[1 << 20][3];

int main() {
  int F, S;
  long long n;
  if (scanf("%d %d %lld", &F, &S, &n) != 3) return 1;
  long long exact_steps = 0, all_steps = 0;
  for (long long i = 0; i < n; ++i) {
    long long a[3], b[3];
    if (scanf("%lld %lld %lld %lld %lld %lld", &a[0], &a[1], &a[2], &b[0], &b[1], &b[2]) != 6) return 1;
    const int M = ohm::longest_axis(a, b);
    ohm::RayRec rec;
    long long nsteps = 0;
    rec.flags = 0;
    ohm::ray_constants(a, b, F, &rec);
    for (int k = 0; k < 3; ++k) nsteps += rec.n[k];
    const int32_t nmaj = rec.n[M];
    rec.inv = ohm::reciprocal64((unsigned long long)rec.A[M]);
    const ohm::SegSplit sp = ohm::ray_segment_split(nmaj, nsteps, S);
    rec.flags |= (M << ohm::kRayAxisShift) | (int32_t)((uint32_t)sp.q << ohm::kRaySegShift);
    rec.nseg = sp.nseg;
    long long c = 0;
    int32_t expect[3] = {rec.v0[0], rec.v0[1], rec.v0[2]};  // where the next piece must start
    for (int j = 0; j < rec.nseg; ++j) {
      long long K0, K1;
      ohm::segment_bounds(nmaj, rec.nseg, sp.q, j, &K0, &K1);
      for (long long k = K0; k < K1; k += ohm::kPieceSlots) {
        const long long ke = k + ohm::kPieceSlots < K1 ? k + ohm::kPieceSlots : K1;
        ohm::PieceStart p;
        ohm::LWalker w;
        ohm::piece_start(rec, F, (int32_t)k, (int32_t)ke, ke == (long long)nmaj + 1, &p, &w);
        const uint32_t neg = ohm::morton_neg(rec.flags);
        uint32_t mo = ohm::region_morton(p.v[0], p.v[1], p.v[2]) ^ neg;
        int32_t v[3] = {p.v[0], p.v[1], p.v[2]};
        for (int d = 0; d < 3; ++d)
          if (v[d] != expect[d]) return 5;
        for (int left = p.visits; left > 0; --left) {
          if (((mo ^ neg) & 0x7fffu) != ohm::region_morton(v[0], v[1], v[2])) return 2;
          for (int d = 0; d < 3; ++d) {
            const int sg = ((rec.flags >> (ohm::kRaySignShift + d)) & 1) ? -1 : 1;
            if ((v[d] >> 5) != (p.v[d] >> 5) + sg * (int)((mo >> (15 + d)) & 1u)) return 2;
          }
          if (c < (1 << 20)) {
            vox[c][0] = v[0];
            vox[c][1] = v[1];
            vox[c][2] = v[2];
          }
          ++c;
          if (left == 1 && (v[0] != p.ve[0] || v[1] != p.ve[1] || v[2] != p.ve[2])) return 5;
          if (left == 1 && ke == (long long)nmaj + 1) break;
          // the step may open the next piece: its region bit is not kept here
          uint32_t to = mo, exact = 0;
          ++all_steps;
          if (!ohm::lwalker_step(w, to)) {
            to = mo;
            ohm::piece_exact_steps(rec, F, (int32_t)k, w, to, 1, &exact);
            if (exact != to) return 2;
            ++exact_steps;
          }
          int axis = -1;
          for (int d = 0; d < 3; ++d)
            if (ohm::morton_coord6(to, d) != ohm::morton_coord6(mo, d)) axis = d;
          v[axis] += ((rec.flags >> (ohm::kRaySignShift + axis)) & 1) ? -1 : 1;
          mo = to;
        }
        for (int d = 0; d < 3; ++d) expect[d] = v[d];
      }
    }
    printf("%lld\n", c);
    for (long long k = 0; k < c && k < (1 << 20); ++k) printf("%d %d %d\n", vox[k][0], vox[k][1], vox[k][2]);
  }
  fprintf(stderr, "exact %lld steps %lld\n", exact_steps, all_steps);
  return 0;
}
