// Eq. 1 force kernel of the mixed path, each pair once (Newton's third law).
//
// One pair (p, j) gives the term on p, mu_j |d|^-3 d, and the reaction on
// j, -mu_p |d|^-3 d, from one difference d = r_j - r_p, one |d|^2 and one
// |d|^-3: 16 FP32 lane operations for the two interactions of a far pair
// (hi-only difference) instead of 24, 22 instead of 36 for a near pair
// (hi/lo difference).  The arithmetic of each term is that of the
// every-ordered-pair kernel (step_kernel.cuh): the same hi/lo split, the
// same far test, MUFU rsqrt.
//
// Decomposition: each system's stage (spatial order) is cut into blocks of
// B = 32 T entries; the work items are the block pairs (I, J), I <= J,
// handed out by a counter.  A CTA of W = T / 4 warps takes an item: warp p
// holds block I's entries [128 p, 128 p + 128) in registers, four per lane
// (slot a: entry 128 p + 32 a + lane).  Block J is cut into chunks of 64
// entries; in phase t the warp takes chunk c = (2 p + t) mod (T / 2).  The
// chunk's 32 stage pair blocks (two entries each, 64 B) are copied
// (cp.async) into the warp's shared memory a phase ahead, the four 16-byte
// pieces of each block into four arrays, so that at step k lane l reads
// pair block (l + k) mod 32 without bank conflicts, its two entries already
// packed as f32x2 operands: in 32 steps every source meets every target
// once, eight pairs per lane and step, the two sources of a lane in one
// packed instruction.  The sources' reaction sums rotate around the warp
// with shuffles, one lane per step.  A chunk passes from warp p + 1 (phase
// t - 2) to warp p (phase t), so its sums in shared memory take their terms
// in phase order; a warp waits for that one neighbour only, two phases back,
// so warps with near chunks and warps with far ones drift instead of meeting
// at a barrier per phase (262,144 bodies: 25.4 -> 23.3 ms per step, 21.7 with the unrolled steps).
//
// Sums, all float pairs (hi, lo) fed through TwoSum: a target's packed
// per-slot sums every two phases (64 terms per half), a source's reaction
// sums twice per phase (after 16 steps, when the sums of the sources of pair
// block l sit in lane l - 16, and at the end; 64 terms per half).
// Off-diagonal items: block I's sums go to row J of its bodies, block J's to
// row I.  Diagonal items (I == J) take each pair (target entry e, source
// entry f) with e < f, by weights on the two chunks that meet the warp's
// own entries (the others are wholly above or below them); each warp adds
// its targets' sums into the block's shared sums after the last phase, and
// the total goes to row I.  Entries past the end of a system's stage are
// inert (massless, far away, distinct).
//
// Far test: a chunk takes the hi-only difference when the union of the
// widened boxes (box_kernel) of the 64-entry stage groups holding the
// warp's targets and the one of the groups holding the chunk are disjoint
// (the bound of step_kernel.cuh holds for either term of the pair).
#include "nbody_dev.cuh"

namespace nb {

namespace {

// Polls of a neighbour's progress in shared memory before it is given up
// (tens of milliseconds; a phase takes tens of microseconds).  The warp then
// says so to the CTA, sets kFlagTimeout and takes no further phase, nor does a
// warp that would wait for it, and the CTA takes no further item (the host
// reports the timeout: the rows it wrote and left out are not used).
constexpr int kMsymPolls = 1 << 21;

// Per-warp shared scratch: two chunk buffers, the targets' negated lo parts
// (duplicated in both halves, read by the near path) and their running
// float-pair sums.
struct MsymWarp {
  // [buffer][piece][pair block]: the 16-byte pieces (xh0 xh1 yh0 yh1),
  // (zh0 zh1 mu0 mu1), (xl0 xl1 yl0 yl1), (zl0 zl1 - -) of a chunk's pair blocks
  float4 src[2][4][32];
  f2 tlo[4][3][32];     // [slot a][component][lane]
  float sum[4][6][32];  // [slot a][x hi, x lo, y hi, y lo, z hi, z lo][lane]
  float4 box[2];        // the union of the widened boxes of the targets' groups
};

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// One arrival on `bar` when this thread's copies so far have landed.
__device__ __forceinline__ void cp_async_arrive(uint64_t *bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Union of the widened boxes of the stage groups that hold entries [e0, e1).
__device__ __forceinline__ void box_union(const float4 *boxes, int e0, int e1, float4 &lo, float4 &hi) {
  lo = make_float4(INFINITY, INFINITY, INFINITY, 0.f);
  hi = make_float4(-INFINITY, -INFINITY, -INFINITY, 0.f);
  for (int g = (e0 >> 1) / kBoxPairs; g <= ((e1 - 1) >> 1) / kBoxPairs; ++g) {
    const float4 l = boxes[2 * g], h = boxes[2 * g + 1];
    lo.x = fminf(lo.x, l.x);
    lo.y = fminf(lo.y, l.y);
    lo.z = fminf(lo.z, l.z);
    hi.x = fmaxf(hi.x, h.x);
    hi.y = fmaxf(hi.y, h.y);
    hi.z = fmaxf(hi.z, h.z);
  }
}

__device__ __forceinline__ bool boxes_apart(const float4 &alo, const float4 &ahi, const float4 &blo,
                                            const float4 &bhi) {
  return alo.x > bhi.x || alo.y > bhi.y || alo.z > bhi.z || blo.x > ahi.x || blo.y > ahi.y || blo.z > ahi.z;
}

// Position (hi) and mu of local entry e of a system's stage (first stage
// entry s0, nst entries); past the end an inert entry: massless, far away,
// at a position of its own.
__device__ __forceinline__ float4 msym_hi(const float *cur, int s0, int e, int nst) {
  if (e < nst) {
    const float *q = cur + pair_off(s0 + e);
    return make_float4(q[kXh], q[kYh], q[kZh], q[kMu]);
  }
  const float x = 2.f * kPadCoord + 1e12f * static_cast<float>(e - nst);
  return make_float4(x, x, x, 0.f);
}

__device__ __forceinline__ float4 msym_lo(const float *cur, int s0, int e, int nst) {
  if (e < nst) {
    const float *q = cur + pair_off(s0 + e);
    return make_float4(q[kXl], q[kYl], q[kZl], 0.f);
  }
  return make_float4(0.f, 0.f, 0.f, 0.f);
}

// Steps [K0, K0 + 16) of a chunk's rotation past the lane's four targets: at
// step k lane l takes the two entries of pair block m = (l + k) mod 32 of the
// chunk (cb: its first piece; piece q of block m at cb[q PS + m]), and the
// block's reaction sums, (bx, by, bz), move one lane down.  The sums start at
// zero, and end as those of pair block (l + K0 + 16) mod 32.  MASKED (a
// diagonal item): a pair counts only if the target's entry, et0 + 32 a,
// precedes the source's, jc + 2 m + h.  MU_SMEM: the targets' mu come from wmu
// ([slot a][lane], shared memory) instead of registers; tlo: the targets'
// negated lo parts, [slot][component][lane], both halves alike.
template <bool NEAR, bool MASKED, bool MU_SMEM, int PS>
__device__ __forceinline__ void msym_half(const float4 *cb, const f2 (&nxh)[4], const f2 (&nyh)[4],
                                          const f2 (&nzh)[4], const f2 (&tmu)[4], const f2 (*wmu)[32],
                                          const f2 (*tlo)[3][32], int lane, int et0, f2 (&ax)[4], f2 (&ay)[4],
                                          f2 (&az)[4], f2 &bx, f2 &by, f2 &bz, int jc, int K0) {
  bx = by = bz = 0ull;
  auto step = [&](int k) {
    const int m = (lane + k) & 31;
    const float4 A = cb[m], B = cb[PS + m];
    const f2 sx = pk(A.x, A.y), sy = pk(A.z, A.w), sz = pk(B.x, B.y), sm = pk(B.z, B.w);
    f2 sxl = 0ull, syl = 0ull, szl = 0ull;
    if (NEAR) {
      const float4 C = cb[2 * PS + m];
      const float2 D = *reinterpret_cast<const float2 *>(cb + 3 * PS + m);  // (zl0, zl1)
      sxl = pk(C.x, C.y);
      syl = pk(C.z, C.w);
      szl = pk(D.x, D.y);
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      f2 dx = add2(sx, nxh[a]), dy = add2(sy, nyh[a]), dz = add2(sz, nzh[a]);
      if (NEAR) {
        dx = add2(dx, add2(sxl, tlo[a][0][lane]));
        dy = add2(dy, add2(syl, tlo[a][1][lane]));
        dz = add2(dz, add2(szl, tlo[a][2][lane]));
      }
      f2 r2 = mul2(dx, dx);
      r2 = fma2(dy, dy, r2);
      r2 = fma2(dz, dz, r2);
      float ra, rb;
      upk(r2, ra, rb);
      float w0 = 1.f, w1 = 1.f;
      if (MASKED) {
        const int et = et0 + 32 * a, es = jc + 2 * m;
        w0 = et < es ? 1.f : 0.f;
        w1 = et < es + 1 ? 1.f : 0.f;
        ra = w0 != 0.f ? ra : 1.f;  // (a target with itself: r2 = 0)
        rb = w1 != 0.f ? rb : 1.f;
      }
      const f2 q = pk(rsqrt_approx(ra), rsqrt_approx(rb));
      const f2 q3 = mul2(mul2(q, q), q);
      f2 fi = mul2(sm, q3), fj = mul2(MU_SMEM ? wmu[a][lane] : tmu[a], q3);
      if (MASKED) {
        const f2 wgt = pk(w0, w1);
        fi = mul2(fi, wgt);
        fj = mul2(fj, wgt);
      }
      ax[a] = fma2(fi, dx, ax[a]);
      ay[a] = fma2(fi, dy, ay[a]);
      az[a] = fma2(fi, dz, az[a]);
      bx = fma2(fj, dx, bx);
      by = fma2(fj, dy, by);
      bz = fma2(fj, dz, bz);
    }
    const int src = (lane + 1) & 31;  // the sums follow their sources to the next lane's step
    bx = __shfl_sync(0xffffffffu, bx, src);
    by = __shfl_sync(0xffffffffu, by, src);
    bz = __shfl_sync(0xffffffffu, bz, src);
  };
  // (Unrolled 4 deep against 1: 65,536 bodies 1.62 -> 1.50 ms per step with the
  // waits above; 8 is 2 % better with mu in shared memory, 1 % worse without.)
#pragma unroll(MU_SMEM ? 8 : 4)
  for (int k = 0; k < 16; ++k) step(K0 + k);
}

// One chunk, all 32 steps: every source meets every target once.  The
// reaction sums fold into the chunk's float pairs s_j (local chunk entries
// jc + 2 m + h for pair block m) half way and at the end.
template <bool NEAR, bool MASKED, bool MU_SMEM>
__device__ __forceinline__ void msym_chunk(const float4 (*cb)[32], const f2 (&nxh)[4], const f2 (&nyh)[4],
                                           const f2 (&nzh)[4], const f2 (&tmu)[4], const f2 (*wmu)[32],
                                           const MsymWarp &ws, int lane, int et0, f2 (&ax)[4], f2 (&ay)[4],
                                           f2 (&az)[4], float *s_j, int BT, int jc) {
#pragma unroll 1
  for (int K0 = 0; K0 < 32; K0 += 16) {
    f2 bx, by, bz;
    msym_half<NEAR, MASKED, MU_SMEM, 32>(cb[0], nxh, nyh, nzh, tmu, wmu, ws.tlo, lane, et0, ax, ay, az, bx, by, bz, jc,
                                         K0);
    const f2 b[3] = {bx, by, bz};
    const int e0 = jc + 2 * ((lane + K0 + 16) & 31);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      float b0, b1;
      upk(b[d], b0, b1);
      two_sum_acc(s_j[(2 * d) * BT + e0], s_j[(2 * d + 1) * BT + e0], -b0);
      two_sum_acc(s_j[(2 * d) * BT + e0 + 1], s_j[(2 * d + 1) * BT + e0 + 1], -b1);
    }
  }
}

}  // namespace

// MU_SMEM: the targets' mu in shared memory, which frees 8 registers in the
// rotation loop.  Used with 2,048-entry blocks (16-warp CTAs, one per SM),
// where it measured faster on GB300 (1,048,576 bodies: 395 against 403 ms
// per step, then with a barrier per phase); with 512-entry blocks its 4 KB per
// CTA cost an SM its fourth CTA (65,536 bodies: 1.71 against 1.64 ms), so
// they keep mu in registers.
template <bool MU_SMEM>
__global__ void __launch_bounds__(32 * kMsymMaxWarps, 1) force_msym_kernel(const MsymArgs a) {
  extern __shared__ __align__(16) unsigned char msym_smem[];
  __shared__ int s_item;
  __shared__ volatile int s_done[kMsymMaxWarps];  // phases each warp has finished
  __shared__ volatile int s_lost;                 // a wait ran out
  grid_dependency_wait();    // staged sources and boxes of this step are complete
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const int W = a.warps, T = a.tiles, BT = 32 * T, NC = T / 2;
  MsymWarp &ws = reinterpret_cast<MsymWarp *>(msym_smem)[w];
  // block J's sums of the item: [x hi, x lo, y hi, y lo, z hi, z lo][BT]
  float *s_j = reinterpret_cast<float *>(msym_smem + static_cast<size_t>(W) * sizeof(MsymWarp));
  // MU_SMEM: this warp's targets' mu, after the sums
  f2 (*wmu)[32] = reinterpret_cast<f2 (*)[32]>(s_j + 6 * BT) + 4 * w;
  const size_t N = static_cast<size_t>(a.N);
  const float *cur = a.cur;
  if (tid == 0) s_lost = 0;
  for (;;) {
    __syncthreads();  // the previous item's shared sums are consumed
    if (tid == 0) s_item = atomicAdd(a.ctr, 1);
    if (lane == 0) s_done[w] = 0;
    for (int k = tid; k < 6 * BT; k += 32 * W) s_j[k] = 0.f;
    __syncthreads();
    const int item = s_lost ? a.n_pairs : s_item;
    if (item >= a.n_pairs) {
      grid_dependency_launch();  // the Verlet kernel may launch as the CTAs run out of items
      break;
    }
    const int4 pr = a.pairs[item];  // (first stage entry of the system, its bodies, block I, block J)
    const int s0 = pr.x, ns = pr.y, I = pr.z, J = pr.w;
    const int nst = (ns + 1) & ~1;  // the system's stage entries (padded to even)
    const bool diag = I == J;
    const int i0 = I * BT, j0 = J * BT;
    {
      const int p = w;               // one round: W = T / 4 warps cover block I
      const int ib = i0 + 128 * p;   // this warp's targets: local entries [ib, ib + 128)
      const bool p_live = ib < nst;  // warp-uniform
      // chunk cc into buffer bb: lane l copies pair block l (its four
      // pieces) if it lies inside the system, else writes two inert entries
      auto stage_chunk = [&](int cc, int bb) {
        const int jb = j0 + 64 * cc;
        const int e0 = jb + 2 * lane;  // the block's first local entry
        if (e0 < nst) {
          const float4 *src = reinterpret_cast<const float4 *>(cur) + static_cast<size_t>((s0 + e0) >> 1) * 4;
#pragma unroll
          for (int q = 0; q < 4; ++q) cp_async16(&ws.src[bb][q][lane], src + q);
        } else {
          const float x0 = 2.f * kPadCoord + 1e12f * static_cast<float>(e0 - nst), x1 = x0 + 1e12f;
          ws.src[bb][0][lane] = make_float4(x0, x1, x0, x1);
          ws.src[bb][1][lane] = make_float4(x0, x1, 0.f, 0.f);
          ws.src[bb][2][lane] = make_float4(0.f, 0.f, 0.f, 0.f);
          ws.src[bb][3][lane] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        cp_async_commit();
      };
      int c = (2 * p) % NC;
      if (p_live) stage_chunk(c, 0);
      f2 nxh[4], nyh[4], nzh[4], tmu[4], ax[4], ay[4], az[4];
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const int e = ib + 32 * s + lane;
        const float4 h = msym_hi(cur, s0, e, nst), l = msym_lo(cur, s0, e, nst);
        nxh[s] = pk(-h.x, -h.x);
        nyh[s] = pk(-h.y, -h.y);
        nzh[s] = pk(-h.z, -h.z);
        tmu[s] = pk(h.w, h.w);
        if (MU_SMEM) wmu[s][lane] = tmu[s];
        ws.tlo[s][0][lane] = pk(-l.x, -l.x);
        ws.tlo[s][1][lane] = pk(-l.y, -l.y);
        ws.tlo[s][2][lane] = pk(-l.z, -l.z);
#pragma unroll
        for (int f = 0; f < 6; ++f) ws.sum[s][f][lane] = 0.f;
        ax[s] = ay[s] = az[s] = 0ull;
      }
      if (p_live && lane == 0) box_union(a.boxes, s0 + ib, s0 + min(ib + 128, nst), ws.box[0], ws.box[1]);
      __syncwarp();
      // the targets' packed sums into their float pairs
      auto fold_targets = [&]() {
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const f2 v[3] = {ax[s], ay[s], az[s]};
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            float v0, v1;
            upk(v[d], v0, v1);
            two_sum_acc(ws.sum[s][2 * d][lane], ws.sum[s][2 * d + 1][lane], v0);
            two_sum_acc(ws.sum[s][2 * d][lane], ws.sum[s][2 * d + 1][lane], v1);
          }
          ax[s] = ay[s] = az[s] = 0ull;
        }
      };
      for (int t = 0; t < NC; ++t) {
        const int cc = c;
        c = (2 * p + t + 1) % NC;
        const int jb = j0 + 64 * cc;  // the chunk: local entries [jb, jb + 64)
        // diagonal item: chunk tiles 2 cc, 2 cc + 1 against the warp's 4 p .. 4 p + 3
        const bool skip = diag && 2 * cc + 1 < 4 * p;
        const bool masked = diag && 2 * cc <= 4 * p + 3;
        if (p_live) {
          cp_async_wait_all();
          __syncwarp();  // every lane's copies (and inert entries) are in buffer t & 1
          // the next chunk into the other buffer, read last in the previous phase
          if (t + 1 < NC) stage_chunk(c, (t + 1) & 1);
          if (jb < nst && !skip) {
            float4 jlo, jhi;
            box_union(a.boxes, s0 + jb, s0 + min(jb + 64, nst), jlo, jhi);
            const bool far = boxes_apart(ws.box[0], ws.box[1], jlo, jhi);
            const float4(*cb)[32] = ws.src[t & 1];
            const int jc = 64 * cc, et0 = 128 * p + lane;
            if (far && !masked)
              msym_chunk<false, false, MU_SMEM>(cb, nxh, nyh, nzh, tmu, wmu, ws, lane, et0, ax, ay, az, s_j, BT, jc);
            else if (masked)
              msym_chunk<true, true, MU_SMEM>(cb, nxh, nyh, nzh, tmu, wmu, ws, lane, et0, ax, ay, az, s_j, BT, jc);
            else
              msym_chunk<true, false, MU_SMEM>(cb, nxh, nyh, nzh, tmu, wmu, ws, lane, et0, ax, ay, az, s_j, BT, jc);
          }
        }
        if ((t & 1) || t + 1 == NC) fold_targets();
        // Phase done.  The chunk of the next phase was the neighbour's two
        // phases before it: wait for that one only.
        if (W > 1) {
          __syncwarp();
          __threadfence_block();
          if (lane == 0) s_done[w] = t + 1;
          const int next = w + 1 < W ? w + 1 : 0;
          int polls = kMsymPolls;
          while (s_done[next] < t + a.stall && polls > 0) polls = s_lost ? 0 : polls - 1;
          if (__any_sync(0xffffffffu, polls == 0)) {
            if (lane == 0) {
              s_lost = 1;
              atomicOr(a.flags, kFlagTimeout);
            }
            break;
          }
          __threadfence_block();
        }
      }
      __syncthreads();  // all phases done
      if (p_live) {
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const int e = ib + 32 * s + lane;
          if (diag) {  // into the block's shared sums (no warp takes these entries until the next barrier)
#pragma unroll
            for (int d = 0; d < 3; ++d) {
              const int k = 128 * p + 32 * s + lane;
              two_sum_acc(s_j[(2 * d) * BT + k], s_j[(2 * d + 1) * BT + k], ws.sum[s][2 * d][lane]);
              s_j[(2 * d + 1) * BT + k] += ws.sum[s][2 * d + 1][lane];
            }
          } else if (e < ns) {
            float2 *row = reinterpret_cast<float2 *>(a.partial) + static_cast<size_t>(J) * 3 * N;
            const int b = a.perm[s0 + e];
            row[b] = make_float2(ws.sum[s][0][lane], ws.sum[s][1][lane]);
            row[N + b] = make_float2(ws.sum[s][2][lane], ws.sum[s][3][lane]);
            row[2 * N + b] = make_float2(ws.sum[s][4][lane], ws.sum[s][5][lane]);
          }
        }
      }
    }
    __syncthreads();
    // block J's sums (on a diagonal item, the block's whole sums) to row I
    float2 *row = reinterpret_cast<float2 *>(a.partial) + static_cast<size_t>(I) * 3 * N;
    for (int k = tid; k < BT && j0 + k < ns; k += 32 * W) {
      const int b = a.perm[s0 + j0 + k];
      row[b] = make_float2(s_j[k], s_j[BT + k]);
      row[N + b] = make_float2(s_j[2 * BT + k], s_j[3 * BT + k]);
      row[2 * N + b] = make_float2(s_j[4 * BT + k], s_j[5 * BT + k]);
    }
  }
  cp_async_wait_all();  // (a chunk is on its way if a wait ran out)
  // The last CTA out resets the item counter for the next launch.
  if (tid == 0) {
    __threadfence();
    if (atomicAdd(a.ctr + 1, 1) == static_cast<int>(gridDim.x) - 1) {
      atomicExch(a.ctr, 0);
      atomicExch(a.ctr + 1, 0);
    }
  }
}

// 128-entry blocks (force_msym_block_kernel): an item is small, so a CTA of
// four warps takes it together.  All four hold block I's 128 targets; warp w
// takes the 16 rotation steps from 16 (w & 1) of chunk w >> 1 of block J.
// Block I and block J (4 KB each) and their boxes are copied to shared memory
// an item ahead, descriptors fetched two and item numbers three ahead, so
// only the barriers at an item's ends and its sums' combination are left
// outside the rotation (loading them at the item's start kept the warps
// waiting for memory 2.4 issue slots in 7: 65.4 us per step at 10,425 bodies,
// 61.3 so).  One warp per item, two 32-step chunks one after the other, left
// an SM with 1.4 rounds of long items: 70 us.  ncu at 10,425 bodies: FMA pipe
// 52 % busy while SMs are active, of the ~76 % its register reads allow.
//
// Sums: a target has 16 terms per warp and half; the two halves and the two
// warps of a chunk are added plainly (64 terms, as everywhere in the mixed
// path), the two chunks' sums through TwoSum.  A source has 64 terms from each
// of its two warps, added through TwoSum.  Every order is fixed.
constexpr int kBlkWarps = 4;

struct MsymBlockShared {
  float4 src[2][2][4][64];        // [buffer][block I, J][piece][pair block]
  float4 box[2][2][3][2];         // [buffer][block I, J][stage group of its entries][low, high corner]
  f2 ti[kBlkWarps][4][3][32];     // per warp: the targets' negated lo parts, then their packed sums
  f2 tj[kBlkWarps][3][32];        // per warp: reaction sums of its chunk's pair blocks
};

__global__ void __launch_bounds__(32 * kBlkWarps, 4) force_msym_block_kernel(const MsymArgs a) {
  extern __shared__ __align__(16) unsigned char msym_smem[];
  MsymBlockShared &sh = *reinterpret_cast<MsymBlockShared *>(msym_smem);
  __shared__ int s_item;
  grid_dependency_wait();    // staged sources and boxes of this step are complete
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const int chunk = w >> 1, K0 = 16 * (w & 1);
  const size_t N = static_cast<size_t>(a.N);
  // An item's descriptor: (first stage entry of the system, its bodies, block
  // I, block J); no bodies past the last item.
  auto describe = [&](int item) { return item < a.n_pairs ? a.pairs[item] : make_int4(0, 0, 0, 0); };
  // Blocks I and J of an item, and the boxes of the stage groups they touch,
  // into buffer bb.
  auto stage_item = [&](const int4 &pr, int bb) {
    if (pr.y > 0) {
      const int nst = (pr.y + 1) & ~1;
#pragma unroll
      for (int u = 0; u < 4; ++u) {  // (4 x 128 threads: 2 blocks x 64 pair blocks x 4 pieces)
        const int blk = u >> 1, pb = tid >> 1, q = 2 * (u & 1) + (tid & 1);
        const int e0 = 128 * (blk ? pr.w : pr.z) + 2 * pb;
        float4 *dst = &sh.src[bb][blk][q][pb];
        if (e0 < nst) {
          cp_async16(dst, reinterpret_cast<const float4 *>(a.cur) + static_cast<size_t>((pr.x + e0) >> 1) * 4 + q);
        } else {  // past the end of the system: inert, each entry at a position of its own
          const float x0 = 2.f * kPadCoord + 1e12f * static_cast<float>(e0 - nst), x1 = x0 + 1e12f;
          *dst = q == 0 ? make_float4(x0, x1, x0, x1) : q == 1 ? make_float4(x0, x1, 0.f, 0.f)
                                                               : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
      if (tid < 12) {
        const int blk = tid / 6, u = (tid % 6) >> 1, e0 = 128 * (blk ? pr.w : pr.z);
        const int g = ((pr.x + e0) >> 1) / kBoxPairs + u, last = ((pr.x + min(e0 + 128, nst) - 1) >> 1) / kBoxPairs;
        float4 *dst = &sh.box[bb][blk][u][tid & 1];
        if (g <= last)
          cp_async16(dst, a.boxes + 2 * g + (tid & 1));
        else  // empty
          *dst = tid & 1 ? make_float4(-INFINITY, -INFINITY, -INFINITY, 0.f)
                         : make_float4(INFINITY, INFINITY, INFINITY, 0.f);
      }
    }
    cp_async_commit();
  };
  // The item numbers run three ahead (the first is the CTA's own, the others
  // from the counter), descriptors two, data one.
  int fetched = 0;  // thread 0
  if (tid == 0) {
    s_item = static_cast<int>(gridDim.x) + atomicAdd(a.ctr, 1);
    fetched = static_cast<int>(gridDim.x) + atomicAdd(a.ctr, 1);
  }
  int4 pr = describe(blockIdx.x);
  stage_item(pr, 0);
  __syncthreads();
  int4 pn = describe(s_item);
  int bb = 0;
  while (pr.y > 0) {
    cp_async_wait_all();
    __syncthreads();  // this item's blocks are in; the previous item's sums (and s_item) are consumed
    if (tid == 0) {
      s_item = fetched;
      fetched = static_cast<int>(gridDim.x) + atomicAdd(a.ctr, 1);  // used an item later
    }
    stage_item(pn, bb ^ 1);
    const int s0 = pr.x, ns = pr.y, I = pr.z, J = pr.w;
    const int nst = (ns + 1) & ~1;
    const bool diag = I == J;
    const int i0 = 128 * I, j0 = 128 * J, jc = 64 * chunk;
    const int bi = i0 + tid < ns ? a.perm[s0 + i0 + tid] : -1, bj = j0 + tid < ns ? a.perm[s0 + j0 + tid] : -1;
    bool far = false;
    {
      float4 ilo = sh.box[bb][0][0][0], ihi = sh.box[bb][0][0][1];
#pragma unroll
      for (int u = 1; u < 3; ++u) {
        const float4 l = sh.box[bb][0][u][0], h = sh.box[bb][0][u][1];
        ilo = make_float4(fminf(ilo.x, l.x), fminf(ilo.y, l.y), fminf(ilo.z, l.z), 0.f);
        ihi = make_float4(fmaxf(ihi.x, h.x), fmaxf(ihi.y, h.y), fmaxf(ihi.z, h.z), 0.f);
      }
      // the chunk's entries lie in one or two of block J's groups
      const int gj = ((s0 + j0) >> 1) / kBoxPairs, g0 = ((s0 + j0 + jc) >> 1) / kBoxPairs - gj,
                g1 = ((s0 + min(j0 + jc + 64, nst) - 1) >> 1) / kBoxPairs - gj;
      if (j0 + jc < nst)
        far = boxes_apart(ilo, ihi, sh.box[bb][1][g0][0], sh.box[bb][1][g0][1]) &&
              boxes_apart(ilo, ihi, sh.box[bb][1][g1][0], sh.box[bb][1][g1][1]);
    }
    f2 ax[4], ay[4], az[4], bx = 0ull, by = 0ull, bz = 0ull;
#pragma unroll
    for (int s = 0; s < 4; ++s) ax[s] = ay[s] = az[s] = 0ull;
    if (j0 + jc < nst) {  // (warp-uniform; a diagonal item's chunk 1 meets targets of both halves, chunk 0 too)
      f2 nxh[4], nyh[4], nzh[4], tmu[4];
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        // target entry 32 s + lane: pair block 16 s + lane / 2, half lane & 1
        const float *p0 = reinterpret_cast<const float *>(&sh.src[bb][0][0][16 * s + (lane >> 1)]) + (lane & 1);
        const float *p1 = reinterpret_cast<const float *>(&sh.src[bb][0][1][16 * s + (lane >> 1)]) + (lane & 1);
        const float *p2 = reinterpret_cast<const float *>(&sh.src[bb][0][2][16 * s + (lane >> 1)]) + (lane & 1);
        const float *p3 = reinterpret_cast<const float *>(&sh.src[bb][0][3][16 * s + (lane >> 1)]) + (lane & 1);
        nxh[s] = pk(-p0[0], -p0[0]);
        nyh[s] = pk(-p0[2], -p0[2]);
        nzh[s] = pk(-p1[0], -p1[0]);
        tmu[s] = pk(p1[2], p1[2]);
        sh.ti[w][s][0][lane] = pk(-p2[0], -p2[0]);
        sh.ti[w][s][1][lane] = pk(-p2[2], -p2[2]);
        sh.ti[w][s][2][lane] = pk(-p3[0], -p3[0]);
      }
      __syncwarp();
      const float4 *cb = &sh.src[bb][1][0][32 * chunk];
      if (diag)
        msym_half<true, true, false, 64>(cb, nxh, nyh, nzh, tmu, nullptr, sh.ti[w], lane, lane, ax, ay, az, bx, by, bz,
                                         jc, K0);
      else if (far)
        msym_half<false, false, false, 64>(cb, nxh, nyh, nzh, tmu, nullptr, sh.ti[w], lane, lane, ax, ay, az, bx, by,
                                           bz, jc, K0);
      else
        msym_half<true, false, false, 64>(cb, nxh, nyh, nzh, tmu, nullptr, sh.ti[w], lane, lane, ax, ay, az, bx, by,
                                          bz, jc, K0);
      __syncwarp();  // the lo parts are read
    }
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      sh.ti[w][s][0][lane] = ax[s];
      sh.ti[w][s][1][lane] = ay[s];
      sh.ti[w][s][2][lane] = az[s];
    }
    const int m = (lane + K0 + 16) & 31;  // the pair block whose sums this lane holds
    sh.tj[w][0][m] = bx;
    sh.tj[w][1][m] = by;
    sh.tj[w][2][m] = bz;
    __syncthreads();
    // thread t: target entry t and source entry t
    float hi[3], lo[3], rh[3], rl[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      float e[kBlkWarps], o[kBlkWarps];
#pragma unroll
      for (int k = 0; k < kBlkWarps; ++k) upk(sh.ti[k][tid >> 5][d][lane], e[k], o[k]);
      hi[d] = (e[0] + o[0]) + (e[1] + o[1]);
      lo[d] = 0.f;
      two_sum_acc(hi[d], lo[d], (e[2] + o[2]) + (e[3] + o[3]));
      // source entry t: chunk t / 64, pair block (t / 2) % 32, half t % 2
      const int c2 = 2 * (tid >> 6), mb = (tid >> 1) & 31;
      const float *r0 = reinterpret_cast<const float *>(&sh.tj[c2][d][mb]) + (tid & 1);
      const float *r1 = reinterpret_cast<const float *>(&sh.tj[c2 + 1][d][mb]) + (tid & 1);
      rh[d] = -*r0;
      rl[d] = 0.f;
      two_sum_acc(rh[d], rl[d], -*r1);
    }
    float2 *part = reinterpret_cast<float2 *>(a.partial);
    if (diag) {
      if (bi >= 0) {
        float2 *row = part + static_cast<size_t>(I) * 3 * N + bi;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          two_sum_acc(hi[d], lo[d], rh[d]);
          row[d * N] = make_float2(hi[d], lo[d] + rl[d]);
        }
      }
    } else {
      if (bi >= 0) {
        float2 *row = part + static_cast<size_t>(J) * 3 * N + bi;
#pragma unroll
        for (int d = 0; d < 3; ++d) row[d * N] = make_float2(hi[d], lo[d]);
      }
      if (bj >= 0) {
        float2 *row = part + static_cast<size_t>(I) * 3 * N + bj;
#pragma unroll
        for (int d = 0; d < 3; ++d) row[d * N] = make_float2(rh[d], rl[d]);
      }
    }
    pr = pn;
    pn = describe(s_item);  // (written before the barrier above; used an item later)
    bb ^= 1;
  }
  // The Verlet kernel may launch as the CTAs run out of items (let in at the
  // start, its CTAs that found no room piled onto the SMs that finished first:
  // 4,096 bodies 19.3 us per step, 17.4 so; 65,536 1.498 and 1.487 ms).
  grid_dependency_launch();
  cp_async_wait_all();
  __syncthreads();
  // The last CTA out resets the item counter for the next launch.
  if (tid == 0) {
    __threadfence();
    if (atomicAdd(a.ctr + 1, 1) == static_cast<int>(gridDim.x) - 1) {
      atomicExch(a.ctr, 0);
      atomicExch(a.ctr + 1, 0);
    }
  }
}

// The adjoint's vector-Jacobian product of Eq. 1 (see vjp.cu), each pair once,
// mixed: 128-entry blocks and items as above, hi/lo differences throughout.
// Warp w takes the 64 targets of half w >> 1 of block I, two per lane, and the
// 64 entries of chunk w & 1 of block J, all 32 rotation steps.  With
// f_q = mu_q |d|^-3, f_j = mu_j |d|^-3, al = w_j . d and be = -w_q . d the term
//   t = f_q w_j - f_j w_q - 3 |d|^-2 (f_q al + f_j be) d
// goes to q and -t to j, |d|^-3 al to q's mass sum and |d|^-3 be to j's: 43
// packed operations for the two interactions of two source pairs against 72
// in the ordered-pair kernel.  A product, reverse step and recomputed forward
// step together: 2,131 bodies 64.6 -> 34.7 us, 10,425 bodies 209 -> 179.
//
// Sums: a target has 32 terms per half and warp; its halves are added plainly
// (64 terms), its two warps' sums through TwoSum; a source has 64 terms from
// each of its two warps, added through TwoSum.
//
// An item's copies arrive on the mbarrier of its buffer, and the CTA waits for
// them with a limit: a wait that runs out sets kFlagTimeout and the CTA leaves.
// Test hook: with a.stall set, thread 0 of CTA 0 leaves out its first arrival.
struct VjpBlockShared {
  float4 src[2][2][4][64];     // [buffer][block I, J][piece][pair block]
  float4 wsrc[2][2][2][64];    // the same of w: (wx0 wx1 wy0 wy1), (wz0 wz1 - -)
  f2 ti[kBlkWarps][2][4][32];  // per warp and target slot: negated lo parts (0..2), then the packed sums
  f2 tj[kBlkWarps][4][32];     // per warp: reaction sums of its chunk's pair blocks
};

template <bool MASKED>
__device__ __forceinline__ void vjp_rotate(const float4 *cb, const float4 *wb, const f2 (&nx)[2][3],
                                           const f2 (&mq)[2], const f2 (&nw)[2][3], const f2 (*tlo)[4][32], int lane,
                                           int et0, int jc, f2 (&acc)[2][4], f2 (&b)[4]) {
  const f2 m3 = pk(-3.f, -3.f);
#pragma unroll 2
  for (int k = 0; k < 32; ++k) {
    const int m = (lane + k) & 31;
    const float4 A = cb[m], B = cb[64 + m], C = cb[128 + m], W = wb[m];
    const float2 D = *reinterpret_cast<const float2 *>(cb + 192 + m), V = *reinterpret_cast<const float2 *>(wb + 64 + m);
    const f2 sh[3] = {pk(A.x, A.y), pk(A.z, A.w), pk(B.x, B.y)}, sl[3] = {pk(C.x, C.y), pk(C.z, C.w), pk(D.x, D.y)};
    const f2 wj[3] = {pk(W.x, W.y), pk(W.z, W.w), pk(V.x, V.y)}, sm = pk(B.z, B.w);
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      f2 d[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) d[c] = add2(add2(sh[c], nx[a][c]), add2(sl[c], tlo[a][c][lane]));
      f2 r2 = mul2(d[0], d[0]);
      r2 = fma2(d[1], d[1], r2);
      r2 = fma2(d[2], d[2], r2);
      float ra, rb;
      upk(r2, ra, rb);
      float w0 = 1.f, w1 = 1.f;
      if (MASKED) {  // a pair counts only if the target's entry precedes the source's
        const int et = et0 + 32 * a, es = jc + 2 * m;
        w0 = et < es ? 1.f : 0.f;
        w1 = et < es + 1 ? 1.f : 0.f;
        ra = w0 != 0.f ? ra : 1.f;
        rb = w1 != 0.f ? rb : 1.f;
      }
      const f2 q = pk(rsqrt_approx(ra), rsqrt_approx(rb));
      const f2 q2 = mul2(q, q);
      f2 s3 = mul2(q, q2);
      if (MASKED) s3 = mul2(s3, pk(w0, w1));
      const f2 fq = mul2(mq[a], s3), fj = mul2(sm, s3);
      f2 al = mul2(wj[0], d[0]);
      al = fma2(wj[1], d[1], al);
      al = fma2(wj[2], d[2], al);
      f2 be = mul2(nw[a][0], d[0]);
      be = fma2(nw[a][1], d[1], be);
      be = fma2(nw[a][2], d[2], be);
      const f2 g = mul2(mul2(fma2(fj, be, mul2(fq, al)), q2), m3);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const f2 t = fma2(g, d[c], fma2(fj, nw[a][c], mul2(fq, wj[c])));
        acc[a][c] = add2(acc[a][c], t);
        b[c] = add2(b[c], t);
      }
      acc[a][3] = fma2(s3, al, acc[a][3]);
      b[3] = fma2(s3, be, b[3]);
    }
    const int src = (lane + 1) & 31;
#pragma unroll
    for (int c = 0; c < 4; ++c) b[c] = __shfl_sync(0xffffffffu, b[c], src);
  }
}

__global__ void __launch_bounds__(32 * kBlkWarps, 4) vjp_msym_block_kernel(const VjpMsymArgs a) {
  extern __shared__ __align__(16) unsigned char msym_smem[];
  VjpBlockShared &sh = *reinterpret_cast<VjpBlockShared *>(msym_smem);
  __shared__ int s_item;
  __shared__ __align__(8) uint64_t bar[2];
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const int half = w >> 1, chunk = w & 1;
  const size_t N = static_cast<size_t>(a.N);
  auto describe = [&](int item) { return item < a.n_pairs ? a.pairs[item] : make_int4(0, 0, 0, 0); };
  auto stage_item = [&](const int4 &pr, int bb, bool stall) {
    if (pr.y > 0) {
      const int nst = (pr.y + 1) & ~1;
#pragma unroll
      for (int u = 0; u < 6; ++u) {  // per block: 64 pair blocks x (4 + 2) pieces, 128 threads
        const int blk = u / 3, pb = tid >> 1, v = u % 3, q = 2 * (v & 1) + (tid & 1);
        const int e0 = 128 * (blk ? pr.w : pr.z) + 2 * pb;
        const size_t block = static_cast<size_t>((pr.x + e0) >> 1);
        float4 *dst = v < 2 ? &sh.src[bb][blk][q][pb] : &sh.wsrc[bb][blk][tid & 1][pb];
        if (e0 < nst) {
          cp_async16(dst, v < 2 ? reinterpret_cast<const float4 *>(a.pos) + block * 4 + q
                                : reinterpret_cast<const float4 *>(a.w) + block * 2 + (tid & 1));
        } else {  // past the end of the system: inert, each entry at a position of its own
          const float x0 = 2.f * kPadCoord + 1e12f * static_cast<float>(e0 - nst), x1 = x0 + 1e12f;
          *dst = v == 2 || q >= 2 ? make_float4(0.f, 0.f, 0.f, 0.f)
                 : q == 0         ? make_float4(x0, x1, x0, x1)
                                  : make_float4(x0, x1, 0.f, 0.f);
        }
      }
      if (!stall) cp_async_arrive(&bar[bb]);
    }
  };
  // (item numbers, descriptors and data run ahead as in force_msym_block_kernel)
  int fetched = 0;  // thread 0
  if (tid == 0) {
    s_item = static_cast<int>(gridDim.x) + atomicAdd(a.ctr, 1);
    fetched = static_cast<int>(gridDim.x) + atomicAdd(a.ctr, 1);
    mbar_init(&bar[0], 32 * kBlkWarps);
    mbar_init(&bar[1], 32 * kBlkWarps);
    mbar_init_fence();
  }
  int4 pr = describe(blockIdx.x);
  __syncthreads();
  stage_item(pr, 0, a.stall != 0 && blockIdx.x == 0 && tid == 0);
  int4 pn = describe(s_item);
  int bb = 0;
  uint32_t parity = 0;
  while (pr.y > 0) {
    if (__syncthreads_or(!mbar_wait(&bar[bb], parity))) {
      if (tid == 0) atomicOr(a.flags, kFlagTimeout);
      break;
    }  // this item's blocks are in; the previous item's sums (and s_item) are consumed
    if (tid == 0) {
      s_item = fetched;
      fetched = static_cast<int>(gridDim.x) + atomicAdd(a.ctr, 1);
    }
    stage_item(pn, bb ^ 1, false);
    const int s0 = pr.x, ns = pr.y, I = pr.z, J = pr.w;
    const int nst = (ns + 1) & ~1;
    const bool diag = I == J;
    const int i0 = 128 * I, j0 = 128 * J, jc = 64 * chunk;
    const int bi = i0 + tid < ns ? a.perm[s0 + i0 + tid] : -1, bj = j0 + tid < ns ? a.perm[s0 + j0 + tid] : -1;
    f2 acc[2][4], b[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[0][c] = acc[1][c] = b[c] = 0ull;
    // (a diagonal item's second half precedes none of the first chunk)
    if (j0 + jc < nst && i0 + 64 * half < nst && !(diag && half > chunk)) {
      f2 nx[2][3], mq[2], nw[2][3];
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        // target entry 64 half + 32 s + lane: pair block 32 half + 16 s + lane / 2, half lane & 1
        const int pb = 32 * half + 16 * s + (lane >> 1), h = lane & 1;
        const float *p[4], *v[2];
#pragma unroll
        for (int q = 0; q < 4; ++q) p[q] = reinterpret_cast<const float *>(&sh.src[bb][0][q][pb]) + h;
#pragma unroll
        for (int q = 0; q < 2; ++q) v[q] = reinterpret_cast<const float *>(&sh.wsrc[bb][0][q][pb]) + h;
        nx[s][0] = pk(-p[0][0], -p[0][0]);
        nx[s][1] = pk(-p[0][2], -p[0][2]);
        nx[s][2] = pk(-p[1][0], -p[1][0]);
        mq[s] = pk(p[1][2], p[1][2]);
        nw[s][0] = pk(-v[0][0], -v[0][0]);
        nw[s][1] = pk(-v[0][2], -v[0][2]);
        nw[s][2] = pk(-v[1][0], -v[1][0]);
        sh.ti[w][s][0][lane] = pk(-p[2][0], -p[2][0]);
        sh.ti[w][s][1][lane] = pk(-p[2][2], -p[2][2]);
        sh.ti[w][s][2][lane] = pk(-p[3][0], -p[3][0]);
      }
      __syncwarp();
      const float4 *cb = &sh.src[bb][1][0][32 * chunk], *wb = &sh.wsrc[bb][1][0][32 * chunk];
      if (diag && half == chunk)
        vjp_rotate<true>(cb, wb, nx, mq, nw, sh.ti[w], lane, 64 * half + lane, jc, acc, b);
      else
        vjp_rotate<false>(cb, wb, nx, mq, nw, sh.ti[w], lane, 64 * half + lane, jc, acc, b);
      __syncwarp();  // the lo parts are read
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      sh.ti[w][0][c][lane] = acc[0][c];
      sh.ti[w][1][c][lane] = acc[1][c];
      sh.tj[w][c][lane] = b[c];  // (a whole rotation: pair block `lane`)
    }
    __syncthreads();
    // thread t: target entry t and source entry t
    float2 *part = reinterpret_cast<float2 *>(a.partial);
    float2 *row_i = part + static_cast<size_t>(J) * 4 * N + max(bi, 0), *row_j = part + static_cast<size_t>(I) * 4 * N + max(bj, 0);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int tw = 2 * (tid >> 6), sw = tid >> 6, mb = (tid >> 1) & 31;
      float e0, o0, e1, o1;
      upk(sh.ti[tw][(tid >> 5) & 1][c][lane], e0, o0);
      upk(sh.ti[tw + 1][(tid >> 5) & 1][c][lane], e1, o1);
      float hi = e0 + o0, lo = 0.f;
      two_sum_acc(hi, lo, e1 + o1);
      const float sg = c < 3 ? -1.f : 1.f;
      float rh = sg * *(reinterpret_cast<const float *>(&sh.tj[sw][c][mb]) + (tid & 1)), rl = 0.f;
      two_sum_acc(rh, rl, sg * *(reinterpret_cast<const float *>(&sh.tj[2 + sw][c][mb]) + (tid & 1)));
      if (diag) {
        two_sum_acc(hi, lo, rh);
        if (bi >= 0) row_i[c * N] = make_float2(hi, lo + rl);
      } else {
        if (bi >= 0) row_i[c * N] = make_float2(hi, lo);
        if (bj >= 0) row_j[c * N] = make_float2(rh, rl);
      }
    }
    pr = pn;
    pn = describe(s_item);  // (written before the barrier above; used an item later)
    bb ^= 1;
    parity ^= bb ^ 1;  // each buffer's every second use
  }
  cp_async_wait_all();
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    if (atomicAdd(a.ctr + 1, 1) == static_cast<int>(gridDim.x) - 1) {
      atomicExch(a.ctr, 0);
      atomicExch(a.ctr + 1, 0);
    }
  }
}

namespace {
bool msym_mu_smem(int tiles) { return tiles == kMsymMaxTiles; }
}  // namespace

size_t force_msym_smem_bytes(int tiles, int warps) {
  if (tiles == kMsymMinTiles) return sizeof(MsymBlockShared);
  return static_cast<size_t>(warps) * sizeof(MsymWarp) + sizeof(float) * 6 * 32 * static_cast<size_t>(tiles) +
         (msym_mu_smem(tiles) ? sizeof(f2) * 4 * 32 * static_cast<size_t>(warps) : 0);
}

cudaError_t launch_force_msym(const MsymArgs &a, int grid, cudaStream_t s, bool chained) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(a.tiles == kMsymMinTiles ? 32 * kBlkWarps : 32 * a.warps);
  cfg.dynamicSmemBytes = force_msym_smem_bytes(a.tiles, a.warps);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = chained ? 1 : 0;
  if (a.tiles == kMsymMinTiles) return cudaLaunchKernelEx(&cfg, force_msym_block_kernel, a);
  if (msym_mu_smem(a.tiles)) return cudaLaunchKernelEx(&cfg, force_msym_kernel<true>, a);
  return cudaLaunchKernelEx(&cfg, force_msym_kernel<false>, a);
}

int force_msym_ctas_per_sm(int tiles, int warps) {
  int occ = 0;
  const int max_smem = static_cast<int>(force_msym_smem_bytes(kMsymMaxTiles, kMsymMaxWarps));
  const auto kernel = tiles == kMsymMinTiles ? force_msym_block_kernel
                      : msym_mu_smem(tiles)  ? force_msym_kernel<true>
                                             : force_msym_kernel<false>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, tiles == kMsymMinTiles ? 32 * kBlkWarps : 32 * warps,
                                                      force_msym_smem_bytes(tiles, warps));
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return occ;
}

int vjp_msym_ctas_per_sm() {
  int occ = 0;
  cudaError_t e = cudaFuncSetAttribute(vjp_msym_block_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(sizeof(VjpBlockShared)));
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, vjp_msym_block_kernel, 32 * kBlkWarps, sizeof(VjpBlockShared));
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return occ;
}

cudaError_t launch_vjp_msym(const VjpMsymArgs &a, int grid, cudaStream_t s) {
  vjp_msym_block_kernel<<<grid, 32 * kBlkWarps, sizeof(VjpBlockShared), s>>>(a);
  return cudaGetLastError();
}

}  // namespace nb
