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

// Fixed-point differences xj - xi (three components each, [3][n]) at the
// exponent field E[i]: out[c][i], the factor |d|^-3 in cube[i], and whether the
// pair is taken.
extern "C" void ic_differences(int64_t n, const double *xi, const double *xj, const int32_t *E, double *out,
                               double *cube, int32_t *taken) {
  using namespace nb::ic;
  for (int64_t i = 0; i < n; ++i) {
    Fix a[3], b[3];
    for (int c = 0; c < 3; ++c) {
      a[c] = to_fix(xi[c * n + i], static_cast<uint32_t>(E[i]));
      b[c] = to_fix(xj[c * n + i], static_cast<uint32_t>(E[i]));
    }
    const FixDiff f = fix_diff(b, a, static_cast<uint32_t>(E[i]));
    taken[i] = fix_in_range(static_cast<uint32_t>(E[i])) && f.ok;
    if (!taken[i]) continue;
    for (int c = 0; c < 3; ++c) out[c * n + i] = fix_value(f, c);
    cube[i] = mass_times(pack_mass(1.0), cube_of(inv_root(square_sum(f), Rsqrt{}), f.em));
  }
}
