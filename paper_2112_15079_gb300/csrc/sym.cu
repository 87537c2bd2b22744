// Eq. 1 force kernel of the FP64 path, each pair once (Newton's third law).
//
// The FP64 pipe bounds this path (an operation of a warp every 76 cycles per
// SM sub-partition).  The pair (p, j) and its reaction share the difference
// and |d|^-3, so evaluating each unordered pair once takes 20 FP64 operations
// for two interactions.  |d|^2, |d|^-3 and the mass products, 11 of them, and
// the differences run on the integer pipes (inv_cube.h), about 185
// instructions beside the 6 FP64 accumulations that are left.  Measured on
// GB300, 10,425 bodies: 2.03 ms per step with 20 FP64 operations, 0.94 ms with
// 9 (FP64 differences), 0.65 ms with 6 (the launch 0.62 ms; 6 x 76 cycles a pair
// and warp step are 0.61: the FP64 pipe stays the bound).
//
// Decomposition: each system's bodies are cut into blocks of 64 (two warp
// tiles of 32); the work items are the block pairs (I, J), I <= J, handed
// out by a counter (off-diagonal pairs first, the cheaper diagonal ones
// last).  A CTA of two warps takes an item: warp w keeps the 32 bodies of
// tile w of block I in registers and, for each tile t of block J, loads its
// 32 bodies as the "sources" and rotates them (positions, masses and their
// reaction sums) once around the warp with shuffles: after 32 steps every
// source has met every target once and its reaction sum is back in its own
// lane, with no FP64 reduction.  A tile paired with itself (diagonal items)
// rotates 16 steps (the 16th for the target side only: lanes L and L + 16
// meet twice).  The two warps' reaction sums for a J tile are added in a
// fixed order in shared memory.
//
// Output: block I's sums go to partial row J of its bodies, block J's to row
// I (a diagonal item adds both into row I); the Verlet kernel adds a body's
// rows 0 .. blocks-1 in order, so the result does not depend on which CTA
// took which item.
#include "nbody_dev.cuh"

namespace nb {

namespace {

__device__ __forceinline__ double4_32a sym_load(const double4_32a *cur, int64_t sb, int il, int ns, double pad) {
  if (il < ns) return cur[sb + il];
  // outside the system: inert (massless, far away, distinct per lane: kInertPlace)
  return make_double4_32a(pad, 0.0, 0.0, 0.0);
}

__device__ __forceinline__ void sym_pair(double xi, double yi, double zi, double mi, double xj, double yj, double zj,
                                         double mj, double &ax, double &ay, double &az, double &bx, double &by,
                                         double &bz, bool react) {
  const double dx = xj - xi, dy = yj - yi, dz = zj - zi;
  const double s3 = inv_r3(fma(dz, dz, fma(dy, dy, dx * dx)));
  const double fi = mj * s3;
  ax = fma(fi, dx, ax);
  ay = fma(fi, dy, ay);
  az = fma(fi, dz, az);
  if (react) {
    const double fj = mi * s3;
    bx = fma(-fj, dx, bx);
    by = fma(-fj, dy, by);
    bz = fma(-fj, dz, bz);
  }
}

// Both terms of one pair with the factors mu_j |d|^-3, mu_i |d|^-3 from the
// integer pipes (inv_cube.h): 9 FP64 operations instead of 20.
__device__ __forceinline__ void sym_pair_int(double xi, double yi, double zi, const ic::Mass &mi, double xj, double yj,
                                             double zj, const ic::Mass &mj, double &ax, double &ay, double &az,
                                             double &bx, double &by, double &bz, bool react) {
  const double dx = xj - xi, dy = yj - yi, dz = zj - zi;
  double f, fr;
  pair_factors(dx, dy, dz, mj, mi, f, fr);
  ax = fma(f, dx, ax);
  ay = fma(f, dy, ay);
  az = fma(f, dz, az);
  if (react) {
    bx = fma(-fr, dx, bx);
    by = fma(-fr, dy, by);
    bz = fma(-fr, dz, bz);
  }
}

// One tile pair: the 32 targets pi (one per lane) against the 32 sources pj,
// rotated once around the warp; (ax, ay, az) take the targets' sums, (bx, by,
// bz) return the sources' reaction sums, each in its source's own lane.
// SELF: the tile with itself, offsets 1..15 both ways and 16 one way (lanes L
// and L + 16 meet twice).  ri, rj: whether this lane's target and source are
// real bodies of the system.
//
// The differences are taken in fixed point (inv_cube.h), which leaves 6 FP64
// operations to a pair, the accumulations; pairs too close for it take 3
// FP64 differences (their sources' coordinates come from their own lanes, so
// the whole warp takes part).  A tile pair with many of them (planets among
// their moons: after kCloseSteps steps that had one), or with magnitudes
// beyond the fixed-point range, goes on with FP64 differences throughout,
// and masses beyond the integer range (never in a physical model) take the
// FP64 series.
constexpr int kCloseSteps = 3;

template <bool SELF>
__device__ __forceinline__ void sym_tile(const double4_32a &pi, const double4_32a &pj, bool ri, bool rj, int lane,
                                         double &ax, double &ay, double &az, double &bx, double &by, double &bz) {
  constexpr int kFirst = SELF ? 1 : 0, kEnd = SELF ? 17 : 32;
  bx = by = bz = 0.0;
  const int src = (lane + 1) & 31;
  auto rotate = [&]() {
    bx = __shfl_sync(0xffffffffu, bx, src);
    by = __shfl_sync(0xffffffffu, by, src);
    bz = __shfl_sync(0xffffffffu, bz, src);
  };
  const uint32_t ei = ri ? ic::max_exp(pi.x, pi.y, pi.z) : 0u, ej = rj ? ic::max_exp(pj.x, pj.y, pj.z) : 0u;
  const uint32_t E = __reduce_max_sync(0xffffffffu, max(ei, ej)) >> 20;
  const bool masses = __all_sync(0xffffffffu, mass_fits(pi.w) && mass_fits(pj.w));
  int k = kFirst;
  if (masses && ic::fix_in_range(E)) {
    const ic::Mass mi = ic::pack_mass(pi.w);
    ic::Mass mj = ic::pack_mass(pj.w);
    ic::Fix xi[3] = {ic::to_fix(pi.x, E), ic::to_fix(pi.y, E), ic::to_fix(pi.z, E)};
    ic::Fix xj[3] = {ic::to_fix(pj.x, E), ic::to_fix(pj.y, E), ic::to_fix(pj.z, E)};
    // (a lane outside the system: beyond every body of the tiles, massless)
    if (!ri) xi[0] = xi[1] = xi[2] = ic::fix_pad();
    if (!rj) xj[0] = xj[1] = xj[2] = ic::fix_pad();
    auto rotate_source = [&]() {
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int u = 0; u < 3; ++u) xj[c].w[u] = __shfl_sync(0xffffffffu, xj[c].w[u], src);
      mj.u = __shfl_sync(0xffffffffu, mj.u, src);
      mj.w = __shfl_sync(0xffffffffu, mj.w, src);
    };
    int close = 0;  // steps that had a close pair
#pragma unroll 1
    for (; k < kEnd && close < kCloseSteps; ++k) {
      if (SELF) {
        rotate();
        rotate_source();
      }
      const ic::FixDiff f = ic::fix_diff(xj, xi, E);
      double dx = ic::fix_value(f, 0), dy = ic::fix_value(f, 1), dz = ic::fix_value(f, 2);
      const ic::Cube c = ic::cube_of(ic::inv_root(ic::square_sum(f), ic::Rsqrt{}), f.em);
      double fj = ic::mass_times(mj, c), fi = ic::mass_times(mi, c);
      if (__any_sync(0xffffffffu, !f.ok)) {
        ++close;
        const int from = (lane + k) & 31;
        const double sx = __shfl_sync(0xffffffffu, pj.x, from), sy = __shfl_sync(0xffffffffu, pj.y, from),
                     sz = __shfl_sync(0xffffffffu, pj.z, from);
        if (!f.ok) {
          dx = sx - pi.x;
          dy = sy - pi.y;
          dz = sz - pi.z;
          pair_factors(dx, dy, dz, mj, mi, fj, fi);
        }
      }
      ax = fma(fj, dx, ax);
      ay = fma(fj, dy, ay);
      az = fma(fj, dz, az);
      if (!SELF || k < 16) {
        bx = fma(-fi, dx, bx);
        by = fma(-fi, dy, by);
        bz = fma(-fi, dz, bz);
      }
      if (!SELF) {
        rotate();
        rotate_source();
      }
    }
  }
  if (k < kEnd) {
    const int at = (lane + k - kFirst) & 31;  // the source here before step k
    double xj = __shfl_sync(0xffffffffu, pj.x, at), yj = __shfl_sync(0xffffffffu, pj.y, at),
           zj = __shfl_sync(0xffffffffu, pj.z, at), wj = __shfl_sync(0xffffffffu, pj.w, at);
    auto rotate_source = [&]() {
      xj = __shfl_sync(0xffffffffu, xj, src);
      yj = __shfl_sync(0xffffffffu, yj, src);
      zj = __shfl_sync(0xffffffffu, zj, src);
      wj = __shfl_sync(0xffffffffu, wj, src);
    };
    const ic::Mass mi = ic::pack_mass(pi.w);
#pragma unroll 1
    for (; k < kEnd; ++k) {
      if (SELF) {
        rotate();
        rotate_source();
      }
      const bool react = !SELF || k < 16;
      if (masses)
        sym_pair_int(pi.x, pi.y, pi.z, mi, xj, yj, zj, ic::pack_mass(wj), ax, ay, az, bx, by, bz, react);
      else
        sym_pair(pi.x, pi.y, pi.z, pi.w, xj, yj, zj, wj, ax, ay, az, bx, by, bz, react);
      if (!SELF) {
        rotate();
        rotate_source();
      }
    }
  }
  if (SELF) {  // lane L holds the sums of lane L + 16: hand them back
    const int back = (lane + 16) & 31;
    bx = __shfl_sync(0xffffffffu, bx, back);
    by = __shfl_sync(0xffffffffu, by, back);
    bz = __shfl_sync(0xffffffffu, bz, back);
  }
}

}  // namespace

__global__ void __launch_bounds__(kSymThreads) force_sym_kernel(const SymArgs a) {
  __shared__ double s_b[2][2][3][32];  // reaction sums [warp][J tile][component][lane]
  __shared__ int s_item;
  grid_dependency_wait();    // staged sources of this step are complete
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const size_t N = static_cast<size_t>(a.N);
  for (;;) {
    __syncthreads();  // the previous item's shared sums are consumed
    if (tid == 0) s_item = atomicAdd(a.ctr, 1);
    __syncthreads();
    const int item = s_item;
    if (item >= a.n_pairs) {
      // The Verlet kernel may launch as the CTAs run out of items.  (Let in at
      // the start, its CTAs that found no room beside ours piled onto the SMs
      // that finished first: 10,425 bodies 691 us per step, 650 so; 3,001 87 and 73.)
      grid_dependency_launch();
      break;
    }
    const int4 pr = a.pairs[item];  // (first body of the system, its bodies, block I, block J)
    const int64_t sb = pr.x;
    const int ns = pr.y, I = pr.z, J = pr.w;
    const double4_32a pi = sym_load(a.cur, sb, I * kSymBlock + w * 32 + lane, ns, kInertPlace * (lane + 1));
    double ax = 0.0, ay = 0.0, az = 0.0;
    for (int t = 0; t < 2; ++t) {
      double bx = 0.0, by = 0.0, bz = 0.0;
      if (!(I == J && t < w)) {  // tile pair (w, t) with t < w of a diagonal item is (t, w), warp t's
        const double4_32a pj0 = sym_load(a.cur, sb, J * kSymBlock + t * 32 + lane, ns,
                                         kInertPlace * (lane + 1) + 0.5 * kInertPlace);
        const bool ri = I * kSymBlock + w * 32 + lane < ns, rj = J * kSymBlock + t * 32 + lane < ns;
        if (I == J && t == w)
          sym_tile<true>(pi, pj0, ri, rj, lane, ax, ay, az, bx, by, bz);
        else
          sym_tile<false>(pi, pj0, ri, rj, lane, ax, ay, az, bx, by, bz);
      }
      s_b[w][t][0][lane] = bx;
      s_b[w][t][1][lane] = by;
      s_b[w][t][2][lane] = bz;
    }
    __syncthreads();
    // thread (w, lane): body J*64 + tid of block J (reaction sums of both
    // warps, warp 0 first) and body I*64 + tid of block I (its own sums)
    const int jl = J * kSymBlock + tid, il = I * kSymBlock + tid;
    double rj[3];
    for (int d = 0; d < 3; ++d) rj[d] = s_b[0][w][d][lane] + s_b[1][w][d][lane];
    if (I == J) {
      if (il < ns) {
        double *row = a.partial + static_cast<size_t>(I) * 3 * N;
        row[sb + il] = ax + rj[0];
        row[N + sb + il] = ay + rj[1];
        row[2 * N + sb + il] = az + rj[2];
      }
    } else {
      if (il < ns) {
        double *row = a.partial + static_cast<size_t>(J) * 3 * N;
        row[sb + il] = ax;
        row[N + sb + il] = ay;
        row[2 * N + sb + il] = az;
      }
      if (jl < ns) {
        double *row = a.partial + static_cast<size_t>(I) * 3 * N;
        row[sb + jl] = rj[0];
        row[N + sb + jl] = rj[1];
        row[2 * N + sb + jl] = rj[2];
      }
    }
  }
  // The last CTA out resets the item counter for the next launch.
  if (tid == 0) {
    __threadfence();
    if (atomicAdd(a.ctr + 1, 1) == static_cast<int>(gridDim.x) - 1) {
      atomicExch(a.ctr, 0);
      atomicExch(a.ctr + 1, 0);
    }
  }
}

// Wide blocks, for systems whose 64-body blocks would need too many partial
// rows (one per block): blocks of B = 32 T bodies (T tiles, a power of two,
// kSymWideMinTiles .. kSymWideMaxTiles), so a body has one row per B bodies
// of its system.  A CTA of W warps takes an item (I, J).  In
// round r warp w holds tile p = r W + w of block I in registers; in phase
// t = 0 .. T-1 it rotates tile q = (p + t) mod T of block J past it, as
// force_sym_kernel does, and adds the tile's reaction sums into block J's
// sums in shared memory.  A CTA barrier closes each phase, and within a
// phase the warps' q differ, so each tile's shared sums take their terms in
// phase order, whichever warp runs first.  Block I's sums of a tile are
// added per tile pair, in phase order.  Off-diagonal items: block I's sums
// go to row J, block J's shared sums to row I.  A diagonal item takes the
// tile pairs q >= p only (q == p as the 16-step half rotation); each warp
// adds its tile's own sums into the shared sums after its round, and the
// total goes to row I.  Tiles past the end of the system are skipped.
// W is kSymWideWarps, four CTAs to an SM, and twice that for the widest
// blocks, whose 96 KB of shared sums leave two CTAs: 16 warps an SM either way.
// With 8, 1,048,576 bodies took 8.48 s per step, 6.24 so.
__global__ void __launch_bounds__(2 * kSymWideThreads, 2) force_sym_wide_kernel(const SymArgs a) {
  extern __shared__ double s_acc[];  // [3][32 T]: block J's reaction sums of the item
  __shared__ int s_item;
  grid_dependency_wait();    // staged sources of this step are complete
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const int T = a.tiles, BT = 32 * T, W = blockDim.x >> 5;
  const size_t N = static_cast<size_t>(a.N);
  for (;;) {
    __syncthreads();  // the previous item's shared sums are consumed
    if (tid == 0) s_item = atomicAdd(a.ctr, 1);
    for (int k = tid; k < 3 * BT; k += 32 * W) s_acc[k] = 0.0;
    __syncthreads();
    const int item = s_item;
    if (item >= a.n_pairs) break;
    const int4 pr = a.pairs[item];  // (first body of the system, its bodies, block I, block J)
    const int64_t sb = pr.x;
    const int ns = pr.y, I = pr.z, J = pr.w;
    const bool diag = I == J;
    const int i0 = I * BT, j0 = J * BT;  // first body of each block within the system
    for (int r = 0; r < T; r += W) {
      const int p = r + w;
      const bool p_live = i0 + p * 32 < ns;  // warp-uniform
      const double4_32a pi = sym_load(a.cur, sb, i0 + p * 32 + lane, ns, kInertPlace * (lane + 1));
      double ax = 0.0, ay = 0.0, az = 0.0;
      // the next phase's J tile, loaded a phase ahead
      int q = p;
      double4_32a pn = sym_load(a.cur, sb, j0 + q * 32 + lane, ns, kInertPlace * (lane + 1) + 0.5 * kInertPlace);
      for (int t = 0; t < T; ++t) {
        const double4_32a pj0 = pn;
        const int qn = (p + t + 1) & (T - 1);
        if (t + 1 < T) pn = sym_load(a.cur, sb, j0 + qn * 32 + lane, ns,
                                     kInertPlace * (lane + 1) + 0.5 * kInertPlace);
        if (p_live && j0 + q * 32 < ns && !(diag && q < p)) {  // (q < p on a diagonal item: tile q's warp's pair)
          double tx = 0.0, ty = 0.0, tz = 0.0, bx, by, bz;
          const bool ri = i0 + p * 32 + lane < ns, rj = j0 + q * 32 + lane < ns;
          if (diag && q == p)
            sym_tile<true>(pi, pj0, ri, rj, lane, tx, ty, tz, bx, by, bz);
          else
            sym_tile<false>(pi, pj0, ri, rj, lane, tx, ty, tz, bx, by, bz);
          ax += tx;
          ay += ty;
          az += tz;
          double *acc = s_acc + q * 32 + lane;
          acc[0] += bx;
          acc[BT] += by;
          acc[2 * BT] += bz;
        }
        q = qn;
        __syncthreads();  // phase done: the J tiles change hands
      }
      if (p_live) {
        const int il = i0 + p * 32 + lane;
        if (diag) {  // tile p's own sums join its shared sums (no warp takes tile p until the next barrier)
          double *acc = s_acc + p * 32 + lane;
          acc[0] += ax;
          acc[BT] += ay;
          acc[2 * BT] += az;
        } else if (il < ns) {
          double *row = a.partial + static_cast<size_t>(J) * 3 * N;
          row[sb + il] = ax;
          row[N + sb + il] = ay;
          row[2 * N + sb + il] = az;
        }
      }
    }
    __syncthreads();
    // block J's sums (on a diagonal item, the block's whole sums) to row I
    double *row = a.partial + static_cast<size_t>(I) * 3 * N;
    for (int k = tid; k < BT && j0 + k < ns; k += 32 * W) {
      row[sb + j0 + k] = s_acc[k];
      row[N + sb + j0 + k] = s_acc[BT + k];
      row[2 * N + sb + j0 + k] = s_acc[2 * BT + k];
    }
  }
  // The last CTA out resets the item counter for the next launch.
  if (tid == 0) {
    __threadfence();
    if (atomicAdd(a.ctr + 1, 1) == static_cast<int>(gridDim.x) - 1) {
      atomicExch(a.ctr, 0);
      atomicExch(a.ctr + 1, 0);
    }
  }
}

// The adjoint's vector-Jacobian product of Eq. 1 (see vjp.cu), each pair
// once.  For the pair (q, j), d = r_j - r_q, s3 = |d|^-3, s5 = |d|^-5 and
// u = mu_q w_j - mu_j w_q, the q term s3 u - 3 s5 (d.u) d changes sign
// under q <-> j (K(d) is even in d, u is odd), and the mass terms are
// s3 (w_j . d) for q and -s3 (w_q . d) for j.  With f_q = mu_q s3,
// f_j = mu_j s3, a = w_j . d, b = w_q . d and z = 3 |d|^-2 the q term is
//   f_q w_j - f_j w_q - z (f_q a - f_j b) d:
// f_q, f_j, s3 and z come from the integer pipes (inv_cube.h), which leaves 29
// FP64 operations to a pair (3 differences, 6 for a and b, 3 for the last
// factor, 9 for the term, 6 + 2 accumulations) of the 48 that |d|^-1, its
// powers and u took: 2,131 bodies 240 -> 156 us per product and reverse
// step.  Rows hold 4 values per body (the three components and the mass
// sum), block I's sums in row J, block J's in row I, as in force_sym_kernel.
__global__ void __launch_bounds__(kSymThreads) vjp_sym_kernel(const VjpSymArgs a) {
  __shared__ double s_b[2][2][4][32];  // reaction sums [warp][J tile][component][lane]
  __shared__ int s_item;
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const size_t N = static_cast<size_t>(a.N);
  const ic::Mass one = ic::pack_mass(1.0), three = ic::pack_mass(3.0);
  for (;;) {
    __syncthreads();
    if (tid == 0) s_item = atomicAdd(a.ctr, 1);
    __syncthreads();
    const int item = s_item;
    if (item >= a.n_pairs) break;
    const int4 pr = a.pairs[item];
    const int64_t sb = pr.x;
    const int ns = pr.y, I = pr.z, J = pr.w;
    const int iq = I * kSymBlock + w * 32 + lane;
    const double4_32a pq = sym_load(a.pos, sb, iq, ns, kInertPlace * (lane + 1));
    const double4_32a wq = iq < ns ? a.w[sb + iq] : make_double4_32a(0.0, 0.0, 0.0, 0.0);
    const ic::Mass mq = ic::pack_mass(pq.w);
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int t = 0; t < 2; ++t) {
      double b[4] = {0.0, 0.0, 0.0, 0.0};
      if (!(I == J && t < w)) {  // tile pair (w, t) with t < w of a diagonal item is (t, w), warp t's
        const int ij = J * kSymBlock + t * 32 + lane;
        const double4_32a pj0 = sym_load(a.pos, sb, ij, ns, kInertPlace * (lane + 1) + 0.5 * kInertPlace);
        const double4_32a wj0 = ij < ns ? a.w[sb + ij] : make_double4_32a(0.0, 0.0, 0.0, 0.0);
        double xj = pj0.x, yj = pj0.y, zj = pj0.z, wjx = wj0.x, wjy = wj0.y, wjz = wj0.z;
        ic::Mass mj = ic::pack_mass(pj0.w);
        auto rotate = [&]() {
          const int src = (lane + 1) & 31;
          xj = __shfl_sync(0xffffffffu, xj, src);
          yj = __shfl_sync(0xffffffffu, yj, src);
          zj = __shfl_sync(0xffffffffu, zj, src);
          mj.u = __shfl_sync(0xffffffffu, mj.u, src);
          mj.w = __shfl_sync(0xffffffffu, mj.w, src);
          wjx = __shfl_sync(0xffffffffu, wjx, src);
          wjy = __shfl_sync(0xffffffffu, wjy, src);
          wjz = __shfl_sync(0xffffffffu, wjz, src);
#pragma unroll
          for (int c = 0; c < 4; ++c) b[c] = __shfl_sync(0xffffffffu, b[c], src);
        };
        auto pair = [&](bool react) {
          const double dx = xj - pq.x, dy = yj - pq.y, dz = zj - pq.z;
          const VjpFactors f = vjp_factors(dx, dy, dz, mq, mj, one, three, false);
          const double al = fma(wjz, dz, fma(wjy, dy, wjx * dx));
          const double be = fma(wq.z, dz, fma(wq.y, dy, wq.x * dx));
          const double c = f.z * fma(-f.fj, be, f.fq * al);
          const double tx = fma(-c, dx, fma(-f.fj, wq.x, f.fq * wjx));
          const double ty = fma(-c, dy, fma(-f.fj, wq.y, f.fq * wjy));
          const double tz = fma(-c, dz, fma(-f.fj, wq.z, f.fq * wjz));
          acc[0] += tx;
          acc[1] += ty;
          acc[2] += tz;
          acc[3] = fma(f.s3, al, acc[3]);
          if (react) {
            b[0] -= tx;
            b[1] -= ty;
            b[2] -= tz;
            b[3] = fma(-f.s3, be, b[3]);
          }
        };
        if (I == J && t == w) {
#pragma unroll 1
          for (int k = 1; k <= 16; ++k) {
            rotate();
            pair(k < 16);
          }
          const int back = (lane + 16) & 31;
#pragma unroll
          for (int c = 0; c < 4; ++c) b[c] = __shfl_sync(0xffffffffu, b[c], back);
        } else {
#pragma unroll 2
          for (int k = 0; k < 32; ++k) {
            pair(true);
            rotate();
          }
        }
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) s_b[w][t][c][lane] = b[c];
    }
    __syncthreads();
    const int jl = J * kSymBlock + tid, il = I * kSymBlock + tid;
    double rj[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) rj[c] = s_b[0][w][c][lane] + s_b[1][w][c][lane];
    if (I == J) {
      if (il < ns) {
        double *row = a.partial + static_cast<size_t>(I) * 4 * N;
#pragma unroll
        for (int c = 0; c < 4; ++c) row[c * N + sb + il] = acc[c] + rj[c];
      }
    } else {
      if (il < ns) {
        double *row = a.partial + static_cast<size_t>(J) * 4 * N;
#pragma unroll
        for (int c = 0; c < 4; ++c) row[c * N + sb + il] = acc[c];
      }
      if (jl < ns) {
        double *row = a.partial + static_cast<size_t>(I) * 4 * N;
#pragma unroll
        for (int c = 0; c < 4; ++c) row[c * N + sb + jl] = rj[c];
      }
    }
  }
  if (tid == 0) {
    __threadfence();
    if (atomicAdd(a.ctr + 1, 1) == static_cast<int>(gridDim.x) - 1) {
      atomicExch(a.ctr, 0);
      atomicExch(a.ctr + 1, 0);
    }
  }
}

cudaError_t launch_vjp_sym(const VjpSymArgs &a, int grid, cudaStream_t s) {
  vjp_sym_kernel<<<grid, kSymThreads, 0, s>>>(a);
  return cudaGetLastError();
}

size_t force_sym_smem_bytes(int tiles) {
  return tiles == 2 ? 0 : sizeof(double) * 3 * 32 * static_cast<size_t>(tiles);
}

namespace {
int sym_wide_threads(int tiles) { return tiles == kSymWideMaxTiles ? 2 * kSymWideThreads : kSymWideThreads; }
}  // namespace

cudaError_t launch_force_sym(const SymArgs &a, int grid, cudaStream_t s, bool chained) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(a.tiles == 2 ? kSymThreads : sym_wide_threads(a.tiles));
  cfg.dynamicSmemBytes = force_sym_smem_bytes(a.tiles);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = chained ? 1 : 0;
  if (a.tiles == 2) return cudaLaunchKernelEx(&cfg, force_sym_kernel, a);
  return cudaLaunchKernelEx(&cfg, force_sym_wide_kernel, a);
}

int force_sym_ctas_per_sm(int tiles) {
  int occ = 0;
  cudaError_t e;
  if (tiles == 2) {
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, force_sym_kernel, kSymThreads, 0);
  } else {
    const size_t smem = force_sym_smem_bytes(tiles);
    e = cudaFuncSetAttribute(force_sym_wide_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(force_sym_smem_bytes(kSymWideMaxTiles)));
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, force_sym_wide_kernel, sym_wide_threads(tiles), smem);
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return occ;
}

}  // namespace nb
