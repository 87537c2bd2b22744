// nbody_accel_static: all-pairs gravitational accelerations of one system,
// FP64, without allocating device memory.  Some callers cannot allocate: hosts that reserve all device
// memory up front and forbid allocation afterwards (real-time or embedded
// loops, services with a fixed memory budget), and components that run while
// another allocator owns the device memory, where an extra cudaMalloc may fail
// or stall.  This entry point therefore keeps its scratch (the staged
// sources, the partial sums, the work tables and the fault flags) in one
// file-scope __device__ array of fixed size instead of asking for memory.
//
// The array is shared by every call on a device and keeps the previous
// call's contents; each call rewrites the staged sources and work tables it
// reads and clears the fault flags and the work counter, which must start
// at zero.  Calls whose work overlaps on the GPU
// (concurrent streams, or several host threads) race on the array and give
// wrong results: serialise them.  Every GPU that loads this library holds the
// array (kStaticScratchBytes) until the process exits.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>

#include <cuda_runtime.h>

#include "nbody.h"
#include "nbody_internal.h"

namespace {

constexpr int64_t kMaxBodies = NBODY_STATIC_MAX_BODIES;
constexpr int kThreads = 128;  // targets per block (IPT 1)
constexpr int kTj = 256;       // sources per shared-memory stage
constexpr int kMaxBlocks = static_cast<int>((kMaxBodies + kThreads - 1) / kThreads);
// The work -- the blocks' sources, block after block -- is cut into equal
// pieces, one CTA each: kPiecesPerSm per SM (all resident; 16 warps hide the
// integer chains), at least as many as blocks (so a piece meets two blocks at
// most), and fewer where a piece would get less than 2 sqrt(n) sources (each
// piece of a block is a partial row of its bodies).  10,425 bodies measured
// on GB300: 6.18 ms with one CTA per block (82 for 152 SMs; 4.48 with the
// reciprocal cube on the integer pipes), 1.30 ms so.
constexpr int kPiecesPerSm = 4;
constexpr int kMaxPieces = 1024;
static_assert(kMaxBlocks <= kMaxPieces, "a piece per block at least");
// Rows x bodies: G pieces over nb blocks leave a body at most G / nb + 2 rows,
// and n <= kThreads nb.
constexpr int64_t kPartialEntries = int64_t(kThreads) * (kMaxPieces + 2 * kMaxBlocks);

constexpr size_t align256(size_t b) { return (b + 255) / 256 * 256; }

// Layout of the static scratch (byte offsets, each 256-byte aligned).
constexpr size_t kOffStage = 0;                                                  // double4 (x, y, z, G m) [max]
constexpr size_t kOffPartial = kOffStage + 32 * kMaxBodies;                      // double [rows][3][n]
constexpr size_t kOffNsl = kOffPartial + 24 * kPartialEntries;                   // uint16 [max]
constexpr size_t kOffBlks = kOffNsl + align256(2 * kMaxBodies);                  // Blk [kMaxBlocks]
constexpr size_t kOffSegs = kOffBlks + align256(sizeof(nb::Blk) * kMaxBlocks);   // Seg [kMaxPieces + kMaxBlocks]
constexpr size_t kOffSegOff = kOffSegs + align256(sizeof(nb::Seg) * (kMaxPieces + kMaxBlocks));  // int32 [kMaxPieces + 1]
constexpr size_t kOffFlags = kOffSegOff + align256(sizeof(int32_t) * (kMaxPieces + 1));  // unsigned
constexpr size_t kOffDyn = kOffFlags + 16;                                       // int32 [2] chunk counter
constexpr size_t kStaticScratchBytes = kOffFlags + 256;

__device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

// Device addresses of g_static_scratch, looked up once per device.
constexpr int kMaxDevices = 64;
std::mutex g_mu;
void *g_addr[kMaxDevices] = {};

// Failure messages go where nbody_last_error(NULL) reads them.
nbody_status fail(nbody_status st, const char *msg) {
  nb::set_last_error(msg);
  return st;
}

// The work tables for n bodies in nb blocks and G pieces.  Position x of the
// line is source x % n of block x / n; piece g covers [cut(g), cut(g + 1)).
// CTA 0 (kMaxPieces threads, one per piece) writes blocks and segments, the
// others the rows of each body.
__global__ void __launch_bounds__(kMaxPieces) static_tables_kernel(int32_t n, int32_t nb, int32_t G, nb::Blk *blks,
                                                                   nb::Seg *segs, int32_t *seg_off, uint16_t *nsl) {
  __shared__ int s_scan[kMaxPieces];
  const int64_t W = static_cast<int64_t>(nb) * n;
  auto cut = [&](int64_t g) { return g * W / G; };
  auto piece_of = [&](int64_t x) {  // the piece that holds position x
    int64_t g = x * G / W;
    while (cut(g) > x) --g;
    while (cut(g + 1) <= x) ++g;
    return static_cast<int>(g);
  };
  auto first_body = [&](int64_t k) { return static_cast<int32_t>(n * k / nb); };
  const int t = threadIdx.x;
  if (blockIdx.x > 0) {
    const int p = (blockIdx.x - 1) * blockDim.x + t;
    if (p >= n) return;
    int64_t k = static_cast<int64_t>(p) * nb / n;  // the block that holds body p
    while (first_body(k) > p) --k;
    while (first_body(k + 1) <= p) ++k;
    nsl[p] = static_cast<uint16_t>(piece_of((k + 1) * n - 1) - piece_of(k * n) + 1);
    return;
  }
  if (t < nb) {
    nb::Blk k;
    k.i0 = first_body(t);
    k.i1 = first_body(t + 1);
    k.q0 = k.i0;
    k.nsplit = piece_of(static_cast<int64_t>(t + 1) * n - 1) - piece_of(static_cast<int64_t>(t) * n) + 1;
    blks[t] = k;
  }
  const int64_t lo = t < G ? cut(t) : 0, hi = t < G ? cut(t + 1) : 0;
  const int b0 = static_cast<int>(lo / n), mine = t < G ? static_cast<int>((hi - 1) / n) - b0 + 1 : 0;
  s_scan[t] = mine;
  __syncthreads();
  for (int off = 1; off < kMaxPieces; off <<= 1) {  // inclusive sums
    const int v = t >= off ? s_scan[t - off] : 0;
    __syncthreads();
    s_scan[t] += v;
    __syncthreads();
  }
  if (t >= G) return;
  const int at = s_scan[t] - mine;
  seg_off[t] = at;
  if (t == G - 1) seg_off[G] = s_scan[t];
  for (int k = 0; k < mine; ++k) {
    const int64_t base = static_cast<int64_t>(b0 + k) * n;
    nb::Seg sg;
    sg.blk = b0 + k;
    sg.s0 = static_cast<int32_t>((lo > base ? lo : base) - base);
    sg.s1 = static_cast<int32_t>((hi < base + n ? hi : base + n) - base);
    sg.slot = t - piece_of(base);
    segs[at + k] = sg;
  }
}

}  // namespace

extern "C" nbody_status nbody_accel_static(int64_t n, double G, const double *x, const double *y, const double *z,
                                           const double *m, double *ax, double *ay, double *az, void *cuda_stream) {
  nb::set_last_error("");
  if (n < 1 || n > kMaxBodies) return fail(NBODY_EINVAL, "n must be in [1, NBODY_STATIC_MAX_BODIES]");
  if (!x || !y || !z || !m || !ax || !ay || !az) return fail(NBODY_EINVAL, "a pointer is NULL");
  if (!(G > 0.0)) return fail(NBODY_EINVAL, "G must be > 0");
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices)
    return fail(NBODY_ECUDA, "no usable CUDA device");
  // The call ends with a copy to pageable host memory and a synchronize,
  // which a stream capture cannot hold: refuse before touching the stream.
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(static_cast<cudaStream_t>(cuda_stream), &cap) != cudaSuccess)
    return fail(NBODY_ECUDA, "cudaStreamIsCapturing failed");
  if (cap != cudaStreamCaptureStatusNone) return fail(NBODY_EINVAL, "the stream is being captured into a graph");
  void *base = nullptr;
  {
    // First call on this device: find the device address of the array (the
    // host-side symbol is only a stand-in and must never reach a kernel).
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_addr[dev]) {
      void *p = nullptr;
      cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
      if (e != cudaSuccess || !p) return fail(NBODY_ECUDA, "cudaGetSymbolAddress failed for the static scratch");
      g_addr[dev] = p;
    }
    base = g_addr[dev];
  }
  unsigned char *s = static_cast<unsigned char *>(base);
  void *stage = s + kOffStage;
  double *partial = reinterpret_cast<double *>(s + kOffPartial);
  uint16_t *nsl = reinterpret_cast<uint16_t *>(s + kOffNsl);
  nb::Blk *blks = reinterpret_cast<nb::Blk *>(s + kOffBlks);
  nb::Seg *segs = reinterpret_cast<nb::Seg *>(s + kOffSegs);
  int32_t *seg_off = reinterpret_cast<int32_t *>(s + kOffSegOff);
  unsigned *flags = reinterpret_cast<unsigned *>(s + kOffFlags);
  int32_t *dyn = reinterpret_cast<int32_t *>(s + kOffDyn);
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const int N = static_cast<int>(n);
  const int n_blocks = (N + kThreads - 1) / kThreads;
  int nsm = 0;
  if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return fail(NBODY_ECUDA, "cudaDeviceGetAttribute failed");
  const int64_t least = static_cast<int64_t>(2.0 * std::sqrt(static_cast<double>(N)));
  const int64_t fit = static_cast<int64_t>(n_blocks) * N / std::max<int64_t>(least, 1);
  const int pieces = static_cast<int>(
      std::max<int64_t>(n_blocks, std::min<int64_t>({fit, int64_t(kPiecesPerSm) * nsm, int64_t(kMaxPieces)})));

  // The fault flags and the chunk counter start at zero on every call; the
  // tables are rewritten.
  if (cudaMemsetAsync(flags, 0, 256, st) != cudaSuccess) return fail(NBODY_ECUDA, "cudaMemsetAsync failed");
  static_tables_kernel<<<1 + (N + kMaxPieces - 1) / kMaxPieces, kMaxPieces, 0, st>>>(N, n_blocks, pieces, blks, segs,
                                                                                    seg_off, nsl);
  if (cudaGetLastError() != cudaSuccess) return fail(NBODY_ECUDA, "table launch failed");

  nb::PrepArgs p{};
  // The staging kernel validates positions and masses; it also reads
  // velocities for that check, which this entry point does not take, so the
  // positions stand in for them.
  p.x = x; p.y = y; p.z = z; p.vx = x; p.vy = y; p.vz = z;
  p.m = m;
  p.stage = stage;
  p.flags = flags;
  p.N = N;
  p.drift = 0;
  p.check = 1;
  p.G = G;
  if (nb::launch_prep(0, p, st) != cudaSuccess) return fail(NBODY_ECUDA, "staging launch failed");

  nb::ForceArgs fa{};
  fa.cur = stage;
  fa.partial = partial;
  fa.flags = flags;
  fa.blks = blks;
  fa.segs = segs;
  fa.seg_off = seg_off;
  fa.dyn_ctr = dyn;
  fa.n_dyn = 0;
  fa.N = N;
  fa.tj = kTj;
  fa.stages = nb::kStages;
  if (nb::launch_force(0, kThreads, 1, pieces, nb::force_smem_bytes(0, kTj, nb::kStages), fa, st, false) != cudaSuccess)
    return fail(NBODY_ECUDA, "force launch failed");
  nb::VerletArgs va{};
  va.ax = ax; va.ay = ay; va.az = az;
  va.partial = partial;
  va.nsl = nsl;
  va.flags = flags;
  va.N = N;
  va.p_begin = 0;
  va.p_end = N;
  va.mode = nb::kModeForce;
  if (nb::launch_verlet(0, va, st, false) != cudaSuccess) return fail(NBODY_ECUDA, "sum launch failed");

  unsigned f = 0;
  if (cudaMemcpyAsync(&f, flags, sizeof f, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return fail(NBODY_ECUDA, "synchronisation failed");
  if (f & nb::kFlagBadInput) return fail(NBODY_EINVAL, "non-finite position or negative/non-finite mass");
  if (f & nb::kFlagTimeout) return fail(NBODY_ETIMEOUT, "a bounded device wait ran out");
  if (f & nb::kFlagNonFinite) return fail(NBODY_EINVAL, "non-finite acceleration: two bodies coincide");
  return NBODY_OK;
}
