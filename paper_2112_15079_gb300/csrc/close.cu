// Close-encounter handling: impulse multiple time stepping of close pairs
// (Tuckerman, Berne and Martyna 1992), FP64, for the members of clusters of
// close pairs (close_pairs.h).
//
// Per Verlet step the force launch evaluates Eq. 1 at the staged positions
// and the per-body Verlet kernel closes the step for every body (bodies in
// no cluster are then done: with no near force the scheme is Verlet).  Two
// kernels then correct the cluster members and start their next step:
//   close_far_kernel: A_far of each member at its position -- Eq. 1 over
//     every source of its system except itself and its close partners,
//     summed directly (not as A - A_near, which would carry the rounding of
//     the dominant near term into a far force many orders smaller);
//   close_kernel, per cluster:
//     complete: v <- vh + dt/2 A_far       (vh saved by the previous sub-cycle)
//     start:    vh <- v + dt/2 A_far
//               k times, h = dt/k:  vh += h/2 a_near; r += h vh;
//                                   a_near <- A_near(r); vh += h/2 a_near
//               stage r for the next force launch; save vh, a_near.
// A_near(r)_p = sum over p's close pairs (p, j), j ascending, of
// mu_j (r_j - r_p) |r_j - r_p|^-3 (mu_j = G m_j), in the force kernel's FP64
// pair arithmetic.  At the start of an nbody_step call (start only) a_near
// is computed from the state.
#include "nbody_dev.cuh"

namespace nb {

constexpr int kFarThreads = 256;

// One CTA per chunk: the chunk's share of its member's far force, reduced in
// a fixed order (a tree over the threads' sums) into far_part.
__global__ void __launch_bounds__(kFarThreads) close_far_kernel(const CloseArgs a) {
  __shared__ double s_red[3][kFarThreads];
  __shared__ int32_t s_part[kFarPartners];
  grid_dependency_wait();    // positions written by the Verlet kernel
  grid_dependency_launch();  // the cluster kernel may start launching (it waits for us)
  const int g = blockIdx.x, t = threadIdx.x;
  const int mi = a.fc_mem[g], j0 = a.fc_j0[g], j1 = a.fc_j1[g];
  const int p = a.mem_body[mi];
  const double px = a.x[p], py = a.y[p], pz = a.z[p];
  // this member's close partners (at most kFarPartners, checked at init)
  const int e0 = a.mp_off[mi], ne = a.mp_off[mi + 1] - e0;
  if (t < ne) {
    const int q = a.mp_pair[e0 + t];
    const int ba = a.mem_body[a.pr_a[q]], bb = a.mem_body[a.pr_b[q]];
    s_part[t] = ba == p ? bb : ba;
  }
  __syncthreads();
  double sx = 0.0, sy = 0.0, sz = 0.0;
  for (int j = j0 + t; j < j1; j += kFarThreads) {
    if (j == p) continue;
    bool partner = false;
    for (int u = 0; u < ne; ++u) partner |= s_part[u] == j;
    if (partner) continue;
    const double dx = a.x[j] - px, dy = a.y[j] - py, dz = a.z[j] - pz;
    const double f = source_factor(dx, dy, dz, ic::pack_mass(a.G * a.m[j]));
    sx = fma(f, dx, sx);
    sy = fma(f, dy, sy);
    sz = fma(f, dz, sz);
  }
  s_red[0][t] = sx;
  s_red[1][t] = sy;
  s_red[2][t] = sz;
  for (int w = kFarThreads / 2; w > 0; w >>= 1) {
    __syncthreads();
    if (t < w)
      for (int d = 0; d < 3; ++d) s_red[d][t] += s_red[d][t + w];
  }
  if (t == 0)
    for (int d = 0; d < 3; ++d) a.far_part[static_cast<size_t>(d) * a.n_chunks + g] = s_red[d][0];
}

// Component c of body b's position for the next force launch.
__device__ __forceinline__ void close_stage(const CloseArgs &a, int b, int c, double r, double *Rc) {
  if (a.precision == 0) {
    double *q = reinterpret_cast<double *>(static_cast<double4_32a *>(a.stage) + b);
    q[c] = r;
    if (c == 0) q[3] = a.G * a.m[b];
  } else {
    Rc[b] = r;
    float *w = static_cast<float *>(a.stage) + pair_off(a.qidx[b]);
    r = times_pow2(r, a.unit);
    const float h = hi_part(r);
    w[kXh + 2 * c] = h;
    w[kXl + 2 * c] = lo_part(r, h);
  }
}

// One cluster.  A sub-step is a chain of dependent operations on a handful of
// bodies, so the work is spread by component: groups of three lanes, lane c of
// a group working on component c, ten groups to a warp.  Group t evaluates
// the force term on one side of one pair (t = 2 pair + side), another group
// holds one member; positions and terms pass through shared memory, with a
// barrier over the warps in use only (one warp up to 5 pairs).  Measured on
// GB300, 131 bodies with 23 close pairs in 13 clusters, k <= 292: 2.07 ->
// 0.92 us per sub-step (one thread per pair and per member and two barriers
// of 256 threads a sub-step before).
//
// The near forces keep the FP64 series and the two half kicks of the scheme as
// written, although the integer factors (inv_cube.h) and one kick for two
// would take 0.74 us: a member's position is rounded at its heliocentric
// magnitude, some 1e-11 of a fast moon's orbit, and each such rounding that
// falls the other way moves the orbit's phase by as much per radian, so other
// low bits in the near force part two runs by 1e-9 within a few steps.
constexpr int kGroups = 10;  // groups of three lanes per warp
constexpr int kCloseWarps = kCloseThreads / 32;
// Members a group holds at most: one unless every warp is in use.
constexpr int kHeldMax = (kCloseThreads + kGroups * kCloseWarps - 1) / (kGroups * kCloseWarps);

struct CloseShared {
  double (*r)[3];       // positions of the members
  double (*u)[3];       // term of side t & 1 of pair t >> 1
  const double *mu;
  const int16_t *ia, *ib;  // the pairs' members
  const int16_t *task;     // the members' terms, each in ascending partner order
};

// The cluster with `W` warps; each group holds up to HELD members: group,
// group + 10 W, ...
template <int HELD>
__device__ __forceinline__ void close_run(const CloseArgs &a, const CloseShared &sh, int cl, int W, int warp,
                                          int lane) {
  const int m0 = a.cl_off[cl], nm = a.cl_off[cl + 1] - m0, np = a.pr_off[cl + 1] - a.pr_off[cl];
  const int e0 = a.mp_off[m0], k = a.cl_k[cl];
  const int g = lane / 3, c = lane % 3;  // (lanes 30 and 31: no group)
  const bool live = g < kGroups;
  const int stride = kGroups * W, group = warp * kGroups + g;
  auto sync = [&]() {
    if (W == 1)
      __syncwarp();
    else
      asm volatile("bar.sync 1, %0;" ::"r"(32 * W) : "memory");
  };
  const size_t M = static_cast<size_t>(a.n_mem);
  const double h = a.dt / k, hh = 0.5 * h;
  auto pick = [&](double *x, double *y, double *z) { return c == 0 ? x : c == 1 ? y : z; };
  double *const Xc = pick(a.x, a.y, a.z), *const Vc = pick(a.vx, a.vy, a.vz), *const Rc = pick(a.Rx, a.Ry, a.Rz);
  double r[HELD], vh[HELD], an[HELD];
  int eb[HELD], ee[HELD], first[HELD];  // the member's terms: task[eb .. ee), the first of them
  bool own[HELD];
#pragma unroll
  for (int s = 0; s < HELD; ++s) {
    const int t = group + s * stride;
    own[s] = live && t < nm;
    r[s] = vh[s] = an[s] = 0.0;
    eb[s] = ee[s] = first[s] = 0;
    if (!own[s]) continue;
    const int mi = m0 + t, b = a.mem_body[mi];
    eb[s] = a.mp_off[mi] - e0;
    ee[s] = a.mp_off[mi + 1] - e0;
    first[s] = sh.task[eb[s]];  // (a member has a partner)
    double af = 0.0, v;
    for (int f = a.mch_off[mi]; f < a.mch_off[mi + 1]; ++f) af += a.far_part[static_cast<size_t>(c) * a.n_chunks + f];
    if (a.complete) {
      an[s] = a.an[c * M + mi];
      v = fma(a.half_dt, af, a.vh[c * M + mi]);
      Vc[b] = v;
    } else {
      v = Vc[b];
    }
    r[s] = Xc[b];
    vh[s] = fma(a.half_dt, af, v);
  }
  // This lane's first pair side (with few pairs the only one).
  const int t1 = live && group < 2 * np ? group : 0;
  const int ia1 = sh.ia[t1 >> 1], ib1 = sh.ib[t1 >> 1];
  const double mu1 = sh.mu[t1 & 1 ? ia1 : ib1];
  auto term = [&](int t, int ia, int ib, double mu, bool real) {
    const double d = sh.r[ib][c] - sh.r[ia][c];
    const int l0 = lane - c;
    const double dx = __shfl_sync(0xffffffffu, d, l0), dy = __shfl_sync(0xffffffffu, d, min(l0 + 1, 31)),
                 dz = __shfl_sync(0xffffffffu, d, min(l0 + 2, 31));
    if (real) sh.u[t][c] = mu * inv_r3(fma(dz, dz, fma(dy, dy, dx * dx))) * (t & 1 ? -d : d);
  };
  // A_near at the positions in sh.r, into an.
  auto near = [&]() {
    sync();  // positions written
    term(t1, ia1, ib1, mu1, live && group < 2 * np);
    for (int t0 = warp * kGroups + stride; t0 < 2 * np; t0 += stride) {  // warp-uniform
      const bool real = live && t0 + g < 2 * np;
      const int t = real ? t0 + g : 0, ia = sh.ia[t >> 1], ib = sh.ib[t >> 1];
      term(t, ia, ib, sh.mu[t & 1 ? ia : ib], real);
    }
    sync();  // terms written (and every read of the positions done)
#pragma unroll
    for (int s = 0; s < HELD; ++s) {
      if (!own[s]) continue;
      double sum = sh.u[first[s]][c];
      for (int e = eb[s] + 1; e < ee[s]; ++e) sum += sh.u[sh.task[e]][c];
      an[s] = sum;
    }
  };
  if (!a.complete) near();
#pragma unroll 1
  for (int sub = 0; sub < k; ++sub) {
    // (the previous near() ended with a barrier after its last read of the
    // positions, so they may be overwritten now)
#pragma unroll
    for (int s = 0; s < HELD; ++s) {
      if (!own[s]) continue;
      vh[s] = fma(hh, an[s], vh[s]);
      r[s] = fma(h, vh[s], r[s]);
      sh.r[group + s * stride][c] = r[s];
    }
    near();
#pragma unroll
    for (int s = 0; s < HELD; ++s) vh[s] = fma(hh, an[s], vh[s]);
  }
#pragma unroll
  for (int s = 0; s < HELD; ++s) {
    if (!own[s]) continue;
    const int mi = m0 + group + s * stride, b = a.mem_body[mi];
    if (!(isfinite(an[s]) && isfinite(vh[s]))) atomicOr(a.flags, kFlagNonFinite);
    a.vh[c * M + mi] = vh[s];
    a.an[c * M + mi] = an[s];
    close_stage(a, b, c, r[s], Rc);
  }
}

__global__ void __launch_bounds__(kCloseThreads) close_kernel(const CloseArgs a) {
  __shared__ double s_r[kCloseThreads][3];
  __shared__ double s_u[2 * kCloseMaxPairs][3];  // term of side t & 1 of pair t >> 1
  __shared__ double s_mu[kCloseThreads];
  __shared__ int16_t s_ia[kCloseMaxPairs], s_ib[kCloseMaxPairs];
  __shared__ int16_t s_task[2 * kCloseMaxPairs];  // the members' terms, each in ascending partner order
  grid_dependency_wait();    // the far forces, and the state and stage the Verlet kernel wrote
  grid_dependency_launch();  // the next kernel may start launching (it waits for us)
  const int cl = blockIdx.x;
  const int m0 = a.cl_off[cl], nm = a.cl_off[cl + 1] - m0;
  const int p0 = a.pr_off[cl], np = a.pr_off[cl + 1] - p0;
  const int e0 = a.mp_off[m0];
  for (int t = threadIdx.x; t < np; t += kCloseThreads) {
    s_ia[t] = static_cast<int16_t>(a.pr_a[p0 + t] - m0);
    s_ib[t] = static_cast<int16_t>(a.pr_b[p0 + t] - m0);
  }
  for (int t = threadIdx.x; t < nm; t += kCloseThreads) {
    const int b = a.mem_body[m0 + t];
    s_mu[t] = a.G * a.m[b];
    s_r[t][0] = a.x[b];
    s_r[t][1] = a.y[b];
    s_r[t][2] = a.z[b];
    for (int e = a.mp_off[m0 + t]; e < a.mp_off[m0 + t + 1]; ++e) {
      const int q = a.mp_pair[e] - p0;
      s_task[e - e0] = static_cast<int16_t>(2 * q + (a.pr_a[p0 + q] - m0 == t ? 0 : 1));
    }
  }
  __syncthreads();
  const int W = min(kCloseWarps, (max(2 * np, nm) + kGroups - 1) / kGroups);  // warps in use
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp >= W) return;
  const CloseShared sh{s_r, s_u, s_mu, s_ia, s_ib, s_task};
  if (W < kCloseWarps)
    close_run<1>(a, sh, cl, W, warp, lane);
  else
    close_run<kHeldMax>(a, sh, cl, W, warp, lane);
}

namespace {
template <typename Kernel>
cudaError_t launch_pdl(Kernel k, int grid, int block, const CloseArgs &a, cudaStream_t s, bool chained) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = chained ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, a);
}
}  // namespace

cudaError_t launch_close_far(const CloseArgs &a, cudaStream_t s, bool chained) {
  if (a.n_chunks <= 0) return cudaSuccess;
  return launch_pdl(close_far_kernel, a.n_chunks, kFarThreads, a, s, chained);
}

cudaError_t launch_close(const CloseArgs &a, int n_clusters, cudaStream_t s, bool chained) {
  if (n_clusters <= 0) return cudaSuccess;
  return launch_pdl(close_kernel, n_clusters, kCloseThreads, a, s, chained);
}

}  // namespace nb
