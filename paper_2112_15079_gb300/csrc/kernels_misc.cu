// Per-body kernels around the Eq. 1 force launches: the Verlet step
// completion (Eqs. 4 and 3), the RK4 stage completion and stage-1 prep, the
// staging / pre-drift kernel, and the force-launch dispatcher.
#include <mutex>
#include <type_traits>

#include "nbody_dev.cuh"

namespace nb {

bool force_fp64_supported(int threads, int ipt);
bool force_mixed_supported(int threads, int ipt);
cudaError_t run_force_fp64(int op, int threads, int ipt, int grid, size_t smem, const ForceArgs &a, cudaStream_t s,
                           bool chained, int *occ);
cudaError_t run_force_mixed(int op, int threads, int ipt, int grid, size_t smem, const ForceArgs &a, cudaStream_t s,
                            bool chained, int *occ);

static cudaError_t run_force(int precision, int op, int threads, int ipt, int grid, size_t smem, const ForceArgs &a,
                             cudaStream_t s, bool chained, int *occ) {
  return precision == 0 ? run_force_fp64(op, threads, ipt, grid, smem, a, s, chained, occ)
                        : run_force_mixed(op, threads, ipt, grid, smem, a, s, chained, occ);
}

cudaError_t launch_force(int precision, int threads, int ipt, int grid, size_t smem, const ForceArgs &a,
                         cudaStream_t s, bool chained) {
  return run_force(precision, 0, threads, ipt, grid, smem, a, s, chained, nullptr);
}

cudaError_t force_set_smem(int precision, int threads, int ipt, size_t smem) {
  // Read-and-raise of a limit shared by every context (and host thread).
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  return run_force(precision, 1, threads, ipt, 0, smem, ForceArgs{}, nullptr, false, nullptr);
}

int force_max_ctas_per_sm(int precision, int threads, int ipt, size_t smem) {
  int occ = 0;
  if (run_force(precision, 2, threads, ipt, 0, smem, ForceArgs{}, nullptr, false, &occ) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return occ;
}

bool force_config_supported(int precision, int threads, int ipt) {
  return precision == 0 ? force_fp64_supported(threads, ipt) : force_mixed_supported(threads, ipt);
}

size_t force_smem_bytes(int precision, int tj, int stages) {
  // 32 bytes per staged source in both layouts; the mixed stage also holds
  // the boxes of the source groups its tile touches
  return static_cast<size_t>(stages) * (static_cast<size_t>(tj) * 32 + (precision == 1 ? (tj / 64 + 2) * 32 : 0));
}

// ---------------------------------------------------------------------------
// Widened boxes of the mixed stage's source groups for the next force launch:
// group g = stage pairs [kBoxPairs g, kBoxPairs (g + 1)), one warp per group,
// lane l reading pairs kBoxPairs g + l + 32 i.  The box of the hi parts is widened on
// every side by kFarKappa times the largest lo part (see step_kernel.cuh).
// Padding sources (coordinate kPadCoord, mu = 0) stay out of the box; a group
// of padding only gets an empty box (low corner +inf, high corner -inf),
// which the far test finds far from every warp.
// ---------------------------------------------------------------------------
constexpr int kBoxWarps = 8;  // groups per CTA

__global__ void __launch_bounds__(32 * kBoxWarps) box_kernel(const float4 *stage, int64_t n_pairs, float4 *boxes) {
  grid_dependency_wait();  // the stage was written by the previous kernel
  grid_dependency_launch();
  const int64_t g = static_cast<int64_t>(blockIdx.x) * kBoxWarps + threadIdx.x / 32;
  const int64_t n_groups = (n_pairs + kBoxPairs - 1) / kBoxPairs;
  if (g >= n_groups) return;  // warp-uniform
  float mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY}, lo[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int i = 0; i < kBoxPairs / 32; ++i) {
    const int64_t b = g * kBoxPairs + (threadIdx.x & 31) + 32 * i;
    if (b >= n_pairs) break;
    // (xh0 xh1 yh0 yh1) (zh0 zh1 mu0 mu1) (xl0 xl1 yl0 yl1) (zl0 zl1 - -)
    const float4 A = stage[4 * b], B = stage[4 * b + 1], C = stage[4 * b + 2], D = stage[4 * b + 3];
    const float hx[2] = {A.x, A.y}, hy[2] = {A.z, A.w}, hz[2] = {B.x, B.y}, mu[2] = {B.z, B.w};
    const float lx[2] = {C.x, C.y}, ly[2] = {C.z, C.w}, lz[2] = {D.x, D.y};
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      if (hx[e] == kPadCoord && mu[e] == 0.f) continue;
      mn[0] = fminf(mn[0], hx[e]);
      mn[1] = fminf(mn[1], hy[e]);
      mn[2] = fminf(mn[2], hz[e]);
      mx[0] = fmaxf(mx[0], hx[e]);
      mx[1] = fmaxf(mx[1], hy[e]);
      mx[2] = fmaxf(mx[2], hz[e]);
      lo[0] = fmaxf(lo[0], fabsf(lx[e]));
      lo[1] = fmaxf(lo[1], fabsf(ly[e]));
      lo[2] = fmaxf(lo[2], fabsf(lz[e]));
    }
  }
  warp_box(mn[0], mn[1], mn[2], mx[0], mx[1], mx[2], lo[0], lo[1], lo[2], boxes + 2 * g);
}

cudaError_t launch_boxes(const void *stage, int64_t n_pairs, float4 *boxes, cudaStream_t s, bool chained) {
  const int64_t n_groups = (n_pairs + kBoxPairs - 1) / kBoxPairs;
  if (n_groups <= 0) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>((n_groups + kBoxWarps - 1) / kBoxWarps));
  cfg.blockDim = dim3(32 * kBoxWarps);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = chained ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, box_kernel, static_cast<const float4 *>(stage), n_pairs, boxes);
}

// ---------------------------------------------------------------------------
// Completes a step for VerletShape<PREC>::kBodies consecutive bodies per CTA.
//   Phase A (kLanes threads per body): a_new = the sum of the body's force
//   partials in a fixed order.  Lane l takes rows l, l + kLanes, ... (TwoSum:
//   FP64 pairs for the FP64 path, float pairs for the mixed path), its loads
//   issued kUnroll rows at a time; for kLanes > 1 a fixed-shape shuffle tree
//   then combines the lanes, so the summation order never changes.
//   Phase B (one component of a body per thread): for kModeStep,
//     Eq. 4  v_{i+1} = v_i + dt/2 (a_i + a_{i+1}),
//     the caller's position receives r_{i+1} (the staged positions),
//     Eq. 3  r_{i+2} = r_{i+1} + v_{i+1} dt + dt^2/2 a_{i+1} -> next stage.
// GB300 runs FP64 at 1/64 of the FP32 rate and charges a warp instruction
// for all 32 lanes whatever the active mask, so FP64 work runs one body per
// lane, and warp c < 3 of a CTA of 32 bodies takes component c: the mixed path
// sums its float-pair rows 8 lanes per body (short latency) and hands the sums
// to those warps for phase B; the FP64 path, whose row sums are FP64
// themselves, sums them there too.  (One thread for all three components
// left most sub-partitions idle at 10,425 bodies: 55 -> 37 us per launch with
// its 163 rows.)
// ---------------------------------------------------------------------------
template <int PREC>
struct VerletShape {
  static constexpr int kBodies = 32;
  static constexpr int kLanes = PREC == 0 ? 1 : 8;   // threads per body (FP64: and component) in phase A
  static constexpr int kBlock = PREC == 0 ? 96 : 256;
  static constexpr int kUnroll = PREC == 0 ? 8 : 4;  // rows per lane whose loads go out together
};

// (hi, lo) pair sums: FP64 pairs for the FP64 path, float pairs for mixed.
template <typename T>
__device__ __forceinline__ void pair_add(T &hi, T &lo, T vhi, T vlo) {
  two_sum_acc(hi, lo, vhi);
  lo += vlo;
}

// Phase A of the per-body kernels, FP64: component c of body p's force partials
// (rows 0..rows-1).  The (up to) U loaded rows are added plainly in row order,
// then the group sum goes into the (hi, lo) pair: one TwoSum per U rows (the
// pair-once kernel leaves a row per 64-body block, ~160 per body at
// N = 10,425; each row is a sum of at most 128 terms).
__device__ __forceinline__ double sum_rows_fp64(const double *partial, int rows, size_t N, int p, int c) {
  constexpr int U = VerletShape<0>::kUnroll;
  double s = 0.0, e = 0.0;
  for (int r0 = 0; r0 < rows; r0 += U) {
    double v[U], g = 0.0;
#pragma unroll
    for (int u = 0; u < U; ++u)  // all loads first, then the sums in row order
      v[u] = r0 + u < rows ? __ldg(partial + (static_cast<size_t>(r0 + u) * 3 + c) * N + p) : 0.0;
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (r0 + u < rows) g += v[u];
    two_sum_acc(s, e, g);
  }
  return s + e;
}

// Mixed: the same by 8 lanes per body, every row through the float pair; the
// sums of the three components, unevaluated (hi, lo) pairs, end in lane 0.
__device__ __forceinline__ void sum_rows_mixed(const double *partial, int rows, size_t N, int p, int lane, float &sx,
                                               float &ex, float &sy, float &ey, float &sz, float &ez) {
  constexpr int L = VerletShape<1>::kLanes, U = VerletShape<1>::kUnroll;
  sx = sy = sz = ex = ey = ez = 0.f;
  const float2 *part = reinterpret_cast<const float2 *>(partial);  // row c of body p: part[c*3N + k*N + p]
  for (int c0 = lane; c0 < rows; c0 += U * L) {
    float2 vx_[U], vy_[U], vz_[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {  // all loads first, then the sums in row order
      const int c = c0 + u * L;
      if (c < rows) {
        const float2 *row = part + static_cast<size_t>(c) * 3 * N;
        vx_[u] = __ldg(row + p);
        vy_[u] = __ldg(row + N + p);
        vz_[u] = __ldg(row + 2 * N + p);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (c0 + u * L < rows) {
        pair_add(sx, ex, vx_[u].x, vx_[u].y);
        pair_add(sy, ey, vy_[u].x, vy_[u].y);
        pair_add(sz, ez, vz_[u].x, vz_[u].y);
      }
    }
  }
#pragma unroll
  for (int off = 1; off < L; off <<= 1) {
    const float hx = __shfl_down_sync(0xffffffffu, sx, off), lx = __shfl_down_sync(0xffffffffu, ex, off);
    const float hy = __shfl_down_sync(0xffffffffu, sy, off), ly = __shfl_down_sync(0xffffffffu, ey, off);
    const float hz = __shfl_down_sync(0xffffffffu, sz, off), lz = __shfl_down_sync(0xffffffffu, ez, off);
    if ((lane & (2 * off - 1)) == 0) {
      pair_add(sx, ex, hx, lx);
      pair_add(sy, ey, hy, ly);
      pair_add(sz, ez, hz, lz);
    }
  }
}

// Phase A of a CTA: the acceleration component `comp` of body p0 + k for the
// thread's phase B (0 beyond component 2).  rows_a: the rows of the thread's
// phase A body; unit: VerletArgs::unit.  Mixed: every thread of the CTA takes part.
template <int PREC>
__device__ __forceinline__ double sum_rows(const double *partial, size_t N, int p0, int rows_a, int comp, int k,
                                           int32_t unit) {
  if constexpr (PREC == 0) {
    return sum_rows_fp64(partial, rows_a, N, p0 + k, comp);
  } else {
    constexpr int L = VerletShape<1>::kLanes, NB = VerletShape<1>::kBodies;
    __shared__ float s_hi[3][NB], s_lo[3][NB];
    const int b = threadIdx.x / L, lane = threadIdx.x % L;
    float sx, sy, sz, ex, ey, ez;
    sum_rows_mixed(partial, rows_a, N, p0 + b, lane, sx, ex, sy, ey, sz, ez);
    if (lane == 0) {
      s_hi[0][b] = sx;
      s_lo[0][b] = ex;
      s_hi[1][b] = sy;
      s_lo[1][b] = ey;
      s_hi[2][b] = sz;
      s_lo[2][b] = ez;
    }
    __syncthreads();
    if (comp >= 3) return 0.0;
    return times_pow2(static_cast<double>(s_hi[comp][k]) + static_cast<double>(s_lo[comp][k]), -unit);
  }
}

// One component of the per-body update after a force evaluation `an` at the
// staged position r (from velocity v, previous acceleration ao):
//   Verlet (Eqs. 4, 3): v' = v + dt/2 (ao + an); the state position is r;
//     the next staged position is r + v' dt + dt^2/2 an.
//   Leapfrog, drift-kick-drift (r is the half-step position r_{n+1/2}):
//     v' = v + dt an; the state position is r + dt/2 v'; the next staged
//     position is that plus dt/2 v' (the next half step).
// Returns the state position; v becomes v', *next the next staged position.
__device__ __forceinline__ double step_component(bool leap, double r, double &v, double ao, double an, double dt,
                                                 double half_dt, double half_dt2, double *next) {
  if (leap) {
    v = fma(dt, an, v);
    const double x = fma(half_dt, v, r);
    *next = fma(half_dt, v, x);
    return x;
  }
  v = kick(v, ao, an, half_dt);
  *next = drift(r, v, an, dt, half_dt2);
  return r;
}

// Stage position (rx, ry, rz) of body q for the next force launch, with mu
// copied from the current stage: FP64 double4 at q, or the mixed hi/lo pair
// block at qidx[q] (mixed: *o is the pair offset, *muf the staged mu; the
// position in units of 2^-unit).
template <int PREC>
__device__ __forceinline__ void stage_position(void *nxt, int q, size_t o, double rx, double ry, double rz, double mu,
                                               float muf, int32_t unit) {
  if (PREC == 0) {
    static_cast<double4_32a *>(nxt)[q] = make_double4_32a(rx, ry, rz, mu);
  } else {
    float *w = static_cast<float *>(nxt) + o;
    rx = times_pow2(rx, unit);
    ry = times_pow2(ry, unit);
    rz = times_pow2(rz, unit);
    const float hx = hi_part(rx), hy = hi_part(ry), hz = hi_part(rz);
    w[kXh] = hx;
    w[kYh] = hy;
    w[kZh] = hz;
    w[kMu] = muf;
    w[kXl] = lo_part(rx, hx);
    w[kYl] = lo_part(ry, hy);
    w[kZl] = lo_part(rz, hz);
  }
}

// The same, component c by itself (c = 0 also writes mu).
template <int PREC>
__device__ __forceinline__ void stage_component(void *nxt, int q, size_t o, int c, double r, double mu, float muf,
                                                int32_t unit) {
  if (PREC == 0) {
    double *w = reinterpret_cast<double *>(static_cast<double4_32a *>(nxt) + q);
    w[c] = r;
    if (c == 0) w[3] = mu;
  } else {
    float *w = static_cast<float *>(nxt) + o;
    r = times_pow2(r, unit);
    const float h = hi_part(r);
    w[kXh + 2 * c] = h;
    w[kXl + 2 * c] = lo_part(r, h);
    if (c == 0) w[kMu] = muf;
  }
}

template <int PREC, int MODE>  // MODE: kModeForce, kModeStep or kModeLeapfrog (a.mode)
__global__ void __launch_bounds__(VerletShape<PREC>::kBlock) verlet_kernel(const VerletArgs a) {
  // Where the host says so the next kernel may launch now, so that its launch
  // overlaps this kernel (its own griddepcontrol.wait still waits for our
  // completion).  Otherwise release only at the end (below).
  if (a.release_early) grid_dependency_launch();
  constexpr int L = VerletShape<PREC>::kLanes, NB = VerletShape<PREC>::kBodies;
  // Phase B: warp c < 3 takes component c of the CTA's 32 bodies, lane = body,
  // so each warp issues a third of the FP64 instructions (GB300's FP64 pipe
  // spends 76 cycles on every warp instruction, so this is the latency).
  const int p0 = a.p_begin + blockIdx.x * NB;  // bodies [p_begin, p_end) (a row shard, or all)
  const int comp = threadIdx.x >> 5, k = threadIdx.x & 31, q = p0 + k;
  const bool own = comp < 3 && q < a.p_end;
  const size_t N = static_cast<size_t>(a.N);
  constexpr bool step = MODE != kModeForce;
  constexpr bool leap = MODE == kModeLeapfrog;
  // This thread's component arrays.
  auto pick = [&](double *x, double *y, double *z) { return comp == 0 ? x : comp == 1 ? y : z; };
  double *const Xc = pick(a.x, a.y, a.z), *const Vc = pick(a.vx, a.vy, a.vz), *const Ac = pick(a.ax, a.ay, a.az);
  double *const Rc = pick(a.Rx, a.Ry, a.Rz);

  // Before the wait: everything this step's force kernel does not write (it
  // writes only the partial rows), so these loads overlap its tail.
  const int pa = PREC == 0 ? q : p0 + static_cast<int>(threadIdx.x) / L;  // phase A body
  const int rows = pa < a.p_end ? a.nsl[pa] : 0;
  double v = 0.0, ao = 0.0, r = 0.0, mu = 0.0;
  float muf = 0.f;
  size_t o = 0;
  if (own && step) {
    v = Vc[q];
    ao = Ac[q];
    if (PREC == 0) {
      const double *rr = reinterpret_cast<const double *>(static_cast<const double4_32a *>(a.cur) + q);
      r = rr[comp];
      if (comp == 0) mu = rr[3];
    } else {
      r = Rc[q];
      o = pair_off(a.qidx[q]);
      if (comp == 0) muf = static_cast<const float *>(a.cur)[o + kMu];
    }
  }
  grid_dependency_wait();  // the force partials of this step are complete

  const double an = sum_rows<PREC>(a.partial, N, p0, rows, comp, k, a.unit);  // phase A
  if (!own) {
    if (!a.release_early) grid_dependency_launch();
    return;
  }
  // ---- phase B: Eqs. 4 and 3, component `comp` of body q ----------------------
  if (!isfinite(an)) atomicOr(a.flags, kFlagNonFinite);
  if (step) {
    double vn = v, nr;
    const double x = step_component(leap, r, vn, ao, an, a.dt, a.half_dt, a.half_dt2, &nr);
    stage_component<PREC>(a.nxt, q, o, comp, nr, mu, muf, a.unit);
    if (PREC == 1) Rc[q] = nr;
    Xc[q] = x;
    Vc[q] = vn;
  }
  Ac[q] = an;
  // Otherwise only now may the next force launch be placed: its CTAs then
  // land on an idle GPU, one share per slot, as the equal-share decomposition
  // assumes (an early launch let several CTAs pile onto the SMs that freed
  // first).
  if (!a.release_early) grid_dependency_launch();
}

cudaError_t launch_verlet(int precision, const VerletArgs &a, cudaStream_t s, bool chained) {
  if (a.p_end <= a.p_begin) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  const int64_t nb = precision == 0 ? VerletShape<0>::kBodies : VerletShape<1>::kBodies;
  cfg.gridDim = dim3(static_cast<unsigned>((static_cast<int64_t>(a.p_end - a.p_begin) + nb - 1) / nb));
  cfg.blockDim = dim3(precision == 0 ? VerletShape<0>::kBlock : VerletShape<1>::kBlock);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = chained ? 1 : 0;
#define NB_VERLET(P, M) \
  if (precision == P && a.mode == M) return cudaLaunchKernelEx(&cfg, verlet_kernel<P, M>, a);
  NB_VERLET(0, kModeForce)
  NB_VERLET(0, kModeStep)
  NB_VERLET(0, kModeLeapfrog)
  NB_VERLET(1, kModeForce)
  NB_VERLET(1, kModeStep)
  NB_VERLET(1, kModeLeapfrog)
#undef NB_VERLET
  return cudaErrorInvalidValue;
}

// ---------------------------------------------------------------------------
// Classical RK4 (the higher-order method Section 2 names) on y = (r, v),
// y' = (v, A(r)): stage completion, s = 2..5 (stage 1 is rk_prep or the end
// of s = 5).  Phase A as in the Verlet kernel; phase B, one body per thread:
//   s = 2, 3: AR += 2 v_s, AV += 2 a_s; r_{s+1} = r + c v_s, v_{s+1} = v + c a_s
//             (c = dt/2 at s = 2, dt at s = 3);
//   s = 4:    r <- r + dt/6 (AR + v_4), v <- v + dt/6 (AV + a_4), stage r;
//   s = 5:    a <- a_5 = A(r); then stage 1 of the next step:
//             AR = v, AV = a, v_2 = v + dt/2 a, stage r_2 = r + dt/2 v.
// ---------------------------------------------------------------------------
template <int PREC>
__global__ void __launch_bounds__(VerletShape<PREC>::kBlock) rk_stage_kernel(const RkArgs a) {
  if (a.release_early) grid_dependency_launch();
  constexpr int L = VerletShape<PREC>::kLanes, NB = VerletShape<PREC>::kBodies;
  const int p0 = blockIdx.x * NB;
  const int c = threadIdx.x >> 5, k = threadIdx.x & 31, q = p0 + k;  // (as the Verlet kernel: warp c, component c)
  const bool own = c < 3 && q < a.N;
  const size_t N = static_cast<size_t>(a.N);
  const int pa = PREC == 0 ? q : p0 + static_cast<int>(threadIdx.x) / L;  // phase A body
  const int rows = pa < a.N ? a.nsl[pa] : 0;
  auto sel = [&](double *x, double *y, double *z) { return c == 0 ? x : c == 1 ? y : z; };
  const size_t i = c * N + q;
  // Prefetch what the force launch does not write (the state, the RK sums).
  double rn = 0.0, vn = 0.0, vs = 0.0, ar = 0.0, av = 0.0, mu = 0.0;
  float muf = 0.f;
  size_t o = 0;
  if (own) {
    rn = sel(a.x, a.y, a.z)[q];
    vn = sel(a.vx, a.vy, a.vz)[q];
    if (a.stage <= 4) {
      vs = a.V[i];
      ar = a.AR[i];
      av = a.AV[i];
    }
    if (PREC == 0) {
      if (c == 0) mu = static_cast<const double4_32a *>(a.cur)[q].w;
    } else {
      o = pair_off(a.qidx[q]);
      if (c == 0) muf = static_cast<const float *>(a.cur)[o + kMu];
    }
  }
  grid_dependency_wait();  // the force partials of this stage are complete
  const double as = sum_rows<PREC>(a.partial, N, p0, rows, c, k, a.unit);
  if (!own) {
    if (!a.release_early) grid_dependency_launch();
    return;
  }
  double rnext;
  if (a.stage == 2 || a.stage == 3) {
    const double cc = a.stage == 2 ? 0.5 * a.dt : a.dt;
    a.AR[i] = ar + 2.0 * vs;
    a.AV[i] = av + 2.0 * as;
    rnext = rn + cc * vs;
    a.V[i] = vn + cc * as;
  } else if (a.stage == 4) {
    const double h = a.dt / 6.0;
    rnext = rn + h * (ar + vs);
    sel(a.x, a.y, a.z)[q] = rnext;
    sel(a.vx, a.vy, a.vz)[q] = vn + h * (av + as);
  } else {  // s = 5: A at the new state, then stage 1 of the next step
    sel(a.ax, a.ay, a.az)[q] = as;
    const double cc = 0.5 * a.dt;
    a.AR[i] = vn;
    a.AV[i] = as;
    rnext = rn + cc * vn;
    a.V[i] = vn + cc * as;
  }
  if (!isfinite(as)) atomicOr(a.flags, kFlagNonFinite);
  stage_component<PREC>(a.nxt, q, o, c, rnext, mu, muf, a.unit);
  if (!a.release_early) grid_dependency_launch();
}

cudaError_t launch_rk_stage(int precision, const RkArgs &a, cudaStream_t s, bool chained) {
  if (a.N <= 0) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  const int64_t nb = precision == 0 ? VerletShape<0>::kBodies : VerletShape<1>::kBodies;
  cfg.gridDim = dim3(static_cast<unsigned>((static_cast<int64_t>(a.N) + nb - 1) / nb));
  cfg.blockDim = dim3(precision == 0 ? VerletShape<0>::kBlock : VerletShape<1>::kBlock);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = chained ? 1 : 0;
  return precision == 0 ? cudaLaunchKernelEx(&cfg, rk_stage_kernel<0>, a)
                        : cudaLaunchKernelEx(&cfg, rk_stage_kernel<1>, a);
}

// RK4 stage 1 from the state (r, v, a = A(r)): AR = v, AV = a,
// V = v + dt/2 a, and the staged sources r_2 = r + dt/2 v with mu = G m.
template <int PREC>
__global__ void rk_prep_kernel(const RkArgs a) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= a.N) return;
  const size_t N = static_cast<size_t>(a.N);
  const double rn[3] = {a.x[q], a.y[q], a.z[q]}, vn[3] = {a.vx[q], a.vy[q], a.vz[q]};
  const double an[3] = {a.ax[q], a.ay[q], a.az[q]};
  const double c = 0.5 * a.dt;
  double r2[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    a.AR[k * N + q] = vn[k];
    a.AV[k * N + q] = an[k];
    r2[k] = rn[k] + c * vn[k];
    a.V[k * N + q] = vn[k] + c * an[k];
  }
  const double mu = a.G * a.m[q];
  const size_t o = PREC == 0 ? 0 : pair_off(a.qidx[q]);
  stage_position<PREC>(a.nxt, q, o, r2[0], r2[1], r2[2], mu, static_cast<float>(mu), a.unit);
}

cudaError_t launch_rk_prep(int precision, const RkArgs &a, cudaStream_t s) {
  if (a.N <= 0) return cudaSuccess;
  const unsigned grid = static_cast<unsigned>((static_cast<int64_t>(a.N) + 255) / 256);
  if (precision == 0)
    rk_prep_kernel<0><<<grid, 256, 0, s>>>(a);
  else
    rk_prep_kernel<1><<<grid, 256, 0, s>>>(a);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Stage the sources of the next force launch: r (drift == 0) or the Eq. 3
// drift of (r, v, a) (drift == 1), with mu = G m.
//   FP64: double4 (x, y, z, mu) at index p.
//   Mixed: FP64 positions R[p], and hi = fl32(r'), lo = fl32(r' - hi) with
//   r' = 2^a.unit r, mu into the pair block of stage entry q = qidx[p] (layout
//   in step_kernel.cuh).
// ---------------------------------------------------------------------------
template <int PREC>
__global__ void prep_kernel(const PrepArgs a) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= a.N) return;
  double rx = a.x[p], ry = a.y[p], rz = a.z[p];
  const double m = a.m[p];
  if (a.check) {
    const bool ok = finite3(rx, ry, rz) && finite3(a.vx[p], a.vy[p], a.vz[p]) && isfinite(m) && m >= 0.0;
    if (!ok) atomicOr(a.flags, kFlagBadInput);
  }
  if (a.drift == 1) {  // Eq. 3
    rx = drift(rx, a.vx[p], a.ax[p], a.dt, a.half_dt2);
    ry = drift(ry, a.vy[p], a.ay[p], a.dt, a.half_dt2);
    rz = drift(rz, a.vz[p], a.az[p], a.dt, a.half_dt2);
  } else if (a.drift == 2) {  // leapfrog: the first half-step drift
    const double h = 0.5 * a.dt;
    rx = fma(h, a.vx[p], rx);
    ry = fma(h, a.vy[p], ry);
    rz = fma(h, a.vz[p], rz);
  }
  const double mu = a.G * m;
  if (PREC == 0) {
    static_cast<double4_32a *>(a.stage)[p] = make_double4_32a(rx, ry, rz, mu);
  } else {
    a.Rx[p] = rx;
    a.Ry[p] = ry;
    a.Rz[p] = rz;
    const int q = a.qidx[p];
    float *w = static_cast<float *>(a.stage) + pair_off(q);
    rx = times_pow2(rx, a.unit);
    ry = times_pow2(ry, a.unit);
    rz = times_pow2(rz, a.unit);
    const float hx = hi_part(rx), hy = hi_part(ry), hz = hi_part(rz);
    w[kXh] = hx;
    w[kYh] = hy;
    w[kZh] = hz;
    w[kMu] = static_cast<float>(mu);
    w[kXl] = lo_part(rx, hx);
    w[kYl] = lo_part(ry, hy);
    w[kZl] = lo_part(rz, hz);
    w[14] = 0.f;
  }
}

cudaError_t launch_prep(int precision, const PrepArgs &a, cudaStream_t s) {
  if (a.N <= 0) return cudaSuccess;
  const int grid = (a.N + 255) / 256;
  if (precision == 0)
    prep_kernel<0><<<grid, 256, 0, s>>>(a);
  else
    prep_kernel<1><<<grid, 256, 0, s>>>(a);
  return cudaGetLastError();
}

// Padding sources of the mixed layout: hi = (kPadCoord, kPadCoord,
// kPadCoord), mu = 0, lo = 0.  Against any real target r2 ~ 3e30 stays
// finite in FP32, q = r2^{-1/2} is tiny and mu = 0 makes the term exactly 0.
__global__ void pad_fill_kernel(float *stage, int64_t n_pairs) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n_pairs * 16) return;
  const int f = static_cast<int>(i & 15);
  stage[i] = f < 6 ? kPadCoord : 0.f;
}

// Padding sources of the FP64 layout (row shards pad the stage to equal
// chunks): (kPadCoord, kPadCoord, kPadCoord, mu = 0); the term of each is
// exactly 0 against any real target.
__global__ void pad_fill_fp64_kernel(double4_32a *stage, int64_t n) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i < n) stage[i] = make_double4_32a(kPadCoord, kPadCoord, kPadCoord, 0.0);
}

cudaError_t launch_pad_fill_fp64(void *stage, int64_t n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  pad_fill_fp64_kernel<<<static_cast<unsigned>((n + 255) / 256), 256, 0, s>>>(static_cast<double4_32a *>(stage), n);
  return cudaGetLastError();
}

cudaError_t launch_pad_fill(void *stage, int64_t n_pairs, cudaStream_t s) {
  if (n_pairs <= 0) return cudaSuccess;
  const int64_t n = n_pairs * 16;
  pad_fill_kernel<<<static_cast<unsigned>((n + 255) / 256), 256, 0, s>>>(static_cast<float *>(stage), n_pairs);
  return cudaGetLastError();
}

}  // namespace nb
