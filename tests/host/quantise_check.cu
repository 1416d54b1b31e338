// Host check of quantise_ff and truncate_ff (ohm_device.cuh) against the double
// evaluations they settle: random points and origins, points built onto
// half-integers of the fixed-point grid, rays around and beyond a range limit.
// Prints "points <n> settled <n> random <n> settled <n> rays <n> settled <n>"
// (random: the random points that the stated bounds say must be settled);
// exit code 2 / 3 on a point / ray settled differently.
#include <cstdio>
#include <random>

#include "../../paper_2206_06079_gb300/csrc/ohm_device.cuh"

int main() {
  std::mt19937_64 g(11);
  std::uniform_real_distribution<double> U(-1.0, 1.0);
  long long n = 0, ok = 0, nr = 0, okr = 0;
  const double voxels[] = {0.1, 0.05, 0.08, 1.0, 0.037};
  for (int i = 0; i < 2000000; ++i) {
    const double voxel = voxels[i % 5], scale = std::ldexp(1.0, i % 7 == 0 ? 20 : 16) / voxel;
    const double range = std::pow(10.0, 2.0 * U(g)) * voxel * 100.0;
    const double origin = i % 3 == 0 ? 0.0 : U(g) * range * (i % 3 == 1 ? 1.0 : 50.0);
    double xd = origin + U(g) * range;
    const bool random = i % 4 != 0;
    if (!random) {  // close to a half-integer of the grid
      const double k = std::rint((xd - origin) * scale) + 0.5;
      xd = origin + k / scale;
    }
    float x = (float)xd;
    if (i % 1000003 == 5) x = INFINITY;
    if (i % 1000003 == 6) x = NAN;
    const double s = ((double)x - origin) * scale;
    long long q;
    const bool settled = ohm::quantise_ff(x, ohm::ff_of_double(origin), ohm::ff_of_double(scale), &q);
    if (settled && !(std::fabs(s) < 4503599627370496.0)) return 2;
    if (settled && q != std::llrint(s)) return 2;
    ++n;
    ok += settled;
    // a point farther than the stated E (and the 1e-6 of the last roundings,
    // both doubled) from a half-integer has to be settled
    const double E = std::ldexp(std::fabs((double)x) + std::fabs(origin), -44) * scale;
    if (random && std::fabs(s) < 1.2e8 && std::fabs(s - std::floor(s) - 0.5) > 2.0 * E + 2e-6) {
      ++nr;
      okr += settled;
    }
  }
  long long rays = 0, rays_ok = 0;
  for (int i = 0; i < 1000000; ++i) {
    const double rmax = 1000.0 + 4.0e7 * std::fabs(U(g)) * (i % 2 ? 1.0 : 0.01);
    const double over = i % 3 == 0 ? 1.0 + 1e-7 * std::fabs(U(g)) : 1.0 + 2.0 * std::fabs(U(g));
    double v[3] = {U(g), U(g), i % 5 == 0 ? 0.0 : U(g)};
    const double norm = std::sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
    int32_t d[3], out[3];
    unsigned long long l2 = 0;
    bool fits = true;
    for (int k = 0; k < 3; ++k) {
      const double c = v[k] / norm * rmax * over;
      fits = fits && std::fabs(c) < 9.0e7;
      d[k] = (int32_t)std::rint(fits ? c : 0.0);
      l2 += (unsigned long long)((long long)d[k] * d[k]);
    }
    if (!fits || l2 >= (1ULL << 53)) continue;
    const double len = std::sqrt((double)l2);
    if (!(len > rmax)) continue;
    ++rays;
    if (!ohm::truncate_ff(d, l2, ohm::ff_of_double(rmax), out)) continue;
    ++rays_ok;
    const double ratio = rmax / len;
    for (int k = 0; k < 3; ++k)
      if (out[k] != (int32_t)std::llrint((double)d[k] * ratio)) return 3;
  }
  printf("points %lld settled %lld random %lld settled %lld rays %lld settled %lld\n", n, ok, nr, okr, rays, rays_ok);
  return 0;
}
