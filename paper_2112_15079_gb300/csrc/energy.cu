// Energy (Sections 2 and 4), FP64:
//   E = sum_p (1/2) m_p |v_p|^2 - sum_{p<j} G m_p m_j / |r_j - r_p|.
//
// Each system's bodies are cut into blocks of 32 T; the work items are the
// block pairs (I, J), I <= J, one CTA each.  A warp holds a 32-body tile of
// block I, one body a lane, and rotates the tiles of block J past it with
// shuffles, so every unordered pair is evaluated once.  mu_j / |d| comes from
// the integer pipes (inv_cube.h), which leaves 4 FP64 operations to a pair: 3
// differences and the sum.  A lane adds the 32 terms of a tile plainly, and
// m_p times that sum enters its double-double through TwoSum; the lanes'
// double-doubles are added in a fixed order, the items' by one CTA per
// system, so the result does not depend on scheduling.  Diagonal items also
// take their block's kinetic energy.
//
// The FP64 pipe bounds it: 4 x 76 cycles a pair and warp step is 0.41 ms at
// 10,425 bodies.  Measured there, the call with its copy back: 0.58 ms,
// against 9.76 ms for one CTA per 256 bodies evaluating every ordered pair (41
// CTAs for 152 SMs, 13 FP64 operations an interaction).
#include "nbody_dev.cuh"

namespace nb {

namespace {

constexpr int kWarps = 4;

struct DD {
  double hi, lo;
};
// Double-double sum: Knuth's TwoSum, then Dekker's Fast2Sum.
__device__ __forceinline__ DD dd_add(DD a, DD b) {
  const double s = a.hi + b.hi;
  const double bb = s - a.hi;
  const double e = (a.hi - (s - bb)) + (b.hi - bb) + (a.lo + b.lo);
  const double hi = s + e;
  return {hi, e - (hi - s)};
}

// The CTA's (kWarps x 32 lanes') double-doubles, in lane 0 of warp 0: a fixed
// tree, by one warp (FP64 work costs the same for one lane as for 32).
__device__ __forceinline__ DD cta_sum(DD v, DD (*buf)[32]) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  buf[w][lane] = v;
  __syncthreads();
  if (w != 0) return v;
  for (int k = 1; k < kWarps; ++k) v = dd_add(v, buf[k][lane]);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const DD o = {__shfl_down_sync(0xffffffffu, v.hi, off), __shfl_down_sync(0xffffffffu, v.lo, off)};
    v = dd_add(v, o);
  }
  return v;
}

// Body il of a system (first body b, ns bodies) with mu = G m; past the end an
// inert one: massless, far away, at a position of its own.
__device__ __forceinline__ double4_32a energy_load(const EnergyArgs &a, int b, int il, int ns, double pad) {
  if (il >= ns) return make_double4_32a(pad, 0.0, 0.0, 0.0);
  return make_double4_32a(a.x[b + il], a.y[b + il], a.z[b + il], a.G * a.m[b + il]);
}

// sum over the tile's sources j of mu_j / |r_j - r_p| for this lane's target.
// SELF: the tile with itself, each unordered pair once: offsets 1..15 in every
// lane, 16 in the lower half.
template <bool SELF>
__device__ __forceinline__ double tile_potential(const double4_32a &p, const double4_32a &j, int lane) {
  double xj = j.x, yj = j.y, zj = j.z;
  ic::Mass mu = ic::pack_mass(j.w);
  const bool fits = __all_sync(0xffffffffu, ic::mass_in_range(mu));
  const int src = (lane + 1) & 31;
  double t = 0.0;
#pragma unroll 2
  for (int k = 0; k < (SELF ? 17 : 32); ++k) {
    if (!SELF || k > 0) {
      const double dx = xj - p.x, dy = yj - p.y, dz = zj - p.z;
      const uint32_t em = ic::max_exp(dx, dy, dz);
      double v = ic::mass_times(mu, ic::inv_dist(ic::square_sum(dx, dy, dz, em), em, ic::Rsqrt{}));
      if (!(fits && ic::exp_in_range(em)))
        v = ic::unpack_mass(mu) * inv_r1(fma(dz, dz, fma(dy, dy, dx * dx)));
      if (!SELF || k < 16 || lane < 16) t += v;
    }
    xj = __shfl_sync(0xffffffffu, xj, src);
    yj = __shfl_sync(0xffffffffu, yj, src);
    zj = __shfl_sync(0xffffffffu, zj, src);
    mu.u = __shfl_sync(0xffffffffu, mu.u, src);
    mu.w = __shfl_sync(0xffffffffu, mu.w, src);
  }
  return t;
}

__global__ void __launch_bounds__(32 * kWarps) energy_kernel(const EnergyArgs a) {
  __shared__ DD buf[kWarps][32];
  const int4 it = a.items[blockIdx.x];  // (first body of the system, its bodies, block I, block J)
  const int b = it.x, ns = it.y, T = a.tiles, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i0 = it.z * 32 * T, j0 = it.w * 32 * T;
  const bool diag = it.z == it.w;
  DD pot = {0.0, 0.0}, kin = {0.0, 0.0};
  for (int r = w; r < T && i0 + 32 * r < ns; r += kWarps) {
    const int il = i0 + 32 * r + lane;
    const double4_32a p = energy_load(a, b, il, ns, kInertPlace * (lane + 1));
    const double mp = il < ns ? a.m[b + il] : 0.0;
    for (int q = diag ? r : 0; q < T && j0 + 32 * q < ns; ++q) {
      const double4_32a j = energy_load(a, b, j0 + 32 * q + lane, ns, kInertPlace * (lane + 1) + 0.5 * kInertPlace);
      const double t = diag && q == r ? tile_potential<true>(p, j, lane) : tile_potential<false>(p, j, lane);
      two_sum_acc(pot.hi, pot.lo, -mp * t);
    }
    if (diag && il < ns) {
      const double vx = a.vx[b + il], vy = a.vy[b + il], vz = a.vz[b + il];
      two_sum_acc(kin.hi, kin.lo, 0.5 * mp * fma(vz, vz, fma(vy, vy, vx * vx)));
    }
  }
  pot = cta_sum(pot, buf);
  if (diag) kin = cta_sum(kin, buf);
  if (threadIdx.x == 0) {
    double *o = a.part + 4 * static_cast<size_t>(blockIdx.x);
    o[0] = kin.hi;
    o[1] = kin.lo;
    o[2] = pot.hi;
    o[3] = pot.lo;
  }
}

// One CTA per system: its items' double-doubles in a fixed order.
__global__ void __launch_bounds__(32 * kWarps) energy_reduce_kernel(const EnergyArgs a) {
  __shared__ DD buf[kWarps][32];
  DD k = {0.0, 0.0}, q = {0.0, 0.0};
  for (int i = a.item_off[blockIdx.x] + threadIdx.x; i < a.item_off[blockIdx.x + 1]; i += 32 * kWarps) {
    const double *o = a.part + 4 * static_cast<size_t>(i);
    if (a.items[i].z == a.items[i].w) k = dd_add(k, DD{o[0], o[1]});
    q = dd_add(q, DD{o[2], o[3]});
  }
  k = cta_sum(k, buf);
  q = cta_sum(q, buf);
  if (threadIdx.x == 0) {
    a.out[blockIdx.x] = k.hi + k.lo;
    a.out[a.n_systems + blockIdx.x] = q.hi + q.lo;
  }
}

}  // namespace

cudaError_t launch_energy(const EnergyArgs &a, cudaStream_t s) {
  energy_kernel<<<a.n_items, 32 * kWarps, 0, s>>>(a);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  energy_reduce_kernel<<<a.n_systems, 32 * kWarps, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace nb
