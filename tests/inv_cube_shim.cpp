// Test-only C entry point over the integer evaluation of mu |d|^-3
// (paper_2112_15079_gb300/csrc/inv_cube.h).  tests/test_inv_cube.py builds
// it with g++; the seed's relative error is the caller's, so that the GPU
// instruction's whole error range is covered on the CPU.
#include <cstdint>

#include "inv_cube.h"

namespace {
struct Seed {
  double off;
  float operator()(float x) const { return static_cast<float>((1.0 + off) / std::sqrt(static_cast<double>(x))); }
};
}  // namespace

// out[i] = mu[i] |d_i|^-power (power 1, 2 or 3); taken[i] = whether the integer path takes the pair.
extern "C" void ic_factors(int64_t n, int32_t power, const double *dx, const double *dy, const double *dz, const double *mu,
                           const double *off, double *out, int32_t *taken) {
  using namespace nb::ic;
  for (int64_t i = 0; i < n; ++i) {
    const uint32_t em = max_exp(dx[i], dy[i], dz[i]);
    const Mass m = pack_mass(mu[i]);
    taken[i] = exp_in_range(em) && mass_in_range(m);
    if (!taken[i]) continue;
    const uint64_t R = square_sum(dx[i], dy[i], dz[i], em);
    const Seed seed{off[i]};
    const CubeSquare c = inv_cube_square(R, em, seed);
    out[i] = mass_times(m, power == 3 ? c.cube : power == 2 ? c.square : inv_dist(R, em, seed));
    const Cube q = inv_cube(R, em, seed);
    if (q.lo != c.cube.lo || q.hi != c.cube.hi || q.e != c.cube.e) taken[i] = -2;
    if (unpack_mass(m) != mu[i]) taken[i] = -1;
  }
}
