// Block size of the pair-once force kernels (sym.cu, sym_mixed.cu) for a
// context, host side.  Plain C++ without CUDA, so the library and a CPU test
// build the same code.
//
// A body keeps one partial row (24 B) per block of its system, and the
// per-body kernel reads them every step; the block pairs (I, J), I <= J, are
// the work items.  The choice:
//   FP64 (bodies per block): 64 when every system has at most kSymMaxBodies
//   (rows <= 1.6 GB at 65,536); else the narrowest wide block (256 .. 4,096
//   bodies) whose rows fit in kSymRowBudget, else 4,096 if they fit in
//   kSymRowLimit (else none); used when the systems hold at least 1.5 block
//   pairs per SM (with fewer, one CTA carries a system's whole sum; measured
//   on GB300, us per step, pair-once against every ordered pair: 600 bodies
//   44.6 / 22.2, 1,031 bodies / 153 pairs 46.0 / 40.9, 1,283 bodies / 231 pairs
//   47.0 / 51.2, 10,425 bodies 649 / 1,224).
//   Mixed (stage entries per block): for a largest system of at least
//   kMsymMinBodies (measured on GB300: 65,536 bodies 1.50 against 1.82 ms
//   per step, 1,048,576 bodies 340 against 430 ms), the narrowest block (128 ..
//   2,048 entries) that leaves the largest system at most kMsymMaxRows rows
//   per body, if the rows fit in kSymRowLimit and the block pairs give at
//   least 8 warps per SM (each warp holds 128 targets); smaller systems:
//   msym_small_block.
// A requested block size is used as asked (nbody_init checks its rows
// against kSymRowLimit and 65,535 blocks per system).
#pragma once

#include <algorithm>
#include <cstdint>
#include <vector>

namespace nb {

// FP64, 64-body blocks (force_sym_kernel): pairs (I, J), I <= J.
constexpr int kSymBlock = 64;
constexpr int kSymThreads = 64;       // two warps: one 32-body tile of block I each
constexpr int kSymMaxBodies = 65536;  // per system, by default (the partial rows are [blocks][3][N])
// FP64 wide blocks of 32 T bodies (force_sym_wide_kernel) above that: T tiles.
constexpr int kSymWideWarps = 4;       // per CTA (the widest blocks: 8)
constexpr int kSymWideThreads = 32 * kSymWideWarps;
constexpr int kSymWideMinTiles = 8;    // 256 bodies
constexpr int kSymWideMaxTiles = 128;  // 4,096 bodies (96 KB of shared sums)
// Mixed blocks of 32 T stage entries (force_msym_kernel), W = T / 4 warps.
constexpr int kMsymMinTiles = 4;   // 128 entries: one warp's four target tiles
constexpr int kMsymMaxTiles = 64;  // 2,048 entries
constexpr int kMsymMaxWarps = kMsymMaxTiles / 4;

constexpr int64_t kSymRowBudget = int64_t(2) << 30;
constexpr int64_t kSymRowLimit = int64_t(16) << 30;
constexpr int64_t kMsymMaxRows = 128;
constexpr int64_t kMsymMinBodies = 65536;

// Rows per body of the largest system with blocks of B, and their bytes
// ([rows][3][N], 8 B per entry) for N bodies in all.
inline int64_t pair_once_rows(const std::vector<int64_t> &sizes, int64_t B) {
  int64_t rows = 1;
  for (int64_t n : sizes) rows = std::max(rows, (n + B - 1) / B);
  return rows;
}

inline int64_t pair_once_row_bytes(const std::vector<int64_t> &sizes, int64_t B) {
  int64_t N = 0;
  for (int64_t n : sizes) N += n;
  return pair_once_rows(sizes, B) * 3 * 8 * N;
}

// The block pairs (I, J), I <= J, of all systems.
inline int64_t pair_once_items(const std::vector<int64_t> &sizes, int64_t B) {
  int64_t pairs = 0;
  for (int64_t n : sizes) {
    const int64_t nb = (n + B - 1) / B;
    pairs += nb * (nb + 1) / 2;
  }
  return pairs;
}

// Unit of the mixed pair-once stage.  These kernels share |d|^-3 between a
// pair's two terms and multiply by mu afterwards; in FP32 |d|^-3 alone loses
// bits from |d| = 2^42 on and overflows below 2^-43, where the every-ordered-pair
// kernel's (mu |d|^-1)(|d|^-2) does neither.  (That form here would cost an
// operation of 16 and 3 % of the time: 65,536 bodies 1.504 -> 1.556 ms per
// step, 10,425 bodies 62.0 -> 63.6 us.)  So the stage has a unit of length of its
// own: positions 2^k r, mu 2^3k G m, accelerations 2^k a, the same bits as
// without where FP32's range holds both.  lo, hi: the smallest and the largest,
// over the systems, of the exponent of a system's largest |coordinate|.  k = 0
// while these leave room on both sides (astronomical units: 5); else the
// largest becomes 2^24, 2^66 above the closest pair that FP32 then takes and 2^17
// below the farthest.  Systems whose sizes lie further apart than 2^30 (the
// smallest then has 2^36 left for its closest pairs) cannot share a unit and
// keep the ordered-pair kernel (unless a block size was asked for).
constexpr int kUnitLow = -4, kUnitHigh = 24, kUnitTo = 24, kUnitSpread = 30;

inline bool stage_unit_fits(int lo, int hi) { return hi - lo <= kUnitSpread; }
inline int stage_unit_exp(int lo, int hi) {
  if (lo >= kUnitLow && hi <= kUnitHigh) return 0;
  return std::min(100, std::max(-100, kUnitTo - hi));
}

// sizes: bodies per system; nsm: the GPU's SMs; requested: the caller's
// block size (0 = automatic).  Returns the block size, or 0 for the
// every-ordered-pair kernel.
inline int pair_once_block(const std::vector<int64_t> &sizes, bool mixed, int64_t nsm, int requested) {
  if (requested > 0) return requested;
  int64_t nmax = 0;
  for (int64_t n : sizes) nmax = std::max(nmax, n);
  if (mixed) {
    if (nmax < kMsymMinBodies) return 0;
    int64_t B = 32 * kMsymMinTiles;
    while (B < 32 * kMsymMaxTiles && pair_once_rows(sizes, B) > kMsymMaxRows) B *= 2;
    if (pair_once_row_bytes(sizes, B) > kSymRowLimit) return 0;
    return pair_once_items(sizes, B) * (B / 128) >= 8 * nsm ? static_cast<int>(B) : 0;
  }
  int64_t B = kSymBlock;
  if (nmax > kSymMaxBodies) {
    B = 32 * kSymWideMinTiles;
    while (B < 32 * kSymWideMaxTiles && pair_once_row_bytes(sizes, B) > kSymRowBudget) B *= 2;
    if (pair_once_row_bytes(sizes, B) > kSymRowLimit) return 0;
  }
  return 2 * pair_once_items(sizes, B) >= 3 * nsm ? static_cast<int>(B) : 0;
}

// Mixed systems below kMsymMinBodies: 128-entry blocks (force_msym_block_kernel,
// four warps to a block pair), or 512, or 0 for the every-ordered-pair
// kernel.  Measured on GB300, us per step, every ordered pair / 128 / 512:
//   bodies     31   300  1,031  2,131  4,096  5,003  8,192  9,000  10,425  20,011  32,768  50,001
//   ordered   8.9  10.7   14.8   18.0   24.0   27.1   46.3   53.9    68.6     207     516    1075
//   128      10.0  10.2   11.0   12.5   18.0   36.2   47.4   49.9    62.4     184     702    2057
//   512      18.5  41.1   58.7   58.8   59.4   60.1   60.9   84.8    86.3     197     429     893
//   systems x bodies  64 x 40..400  2,000 x 500  10 x 5,000  100 x 5,000  64 x 1,000..20,000
//   ordered                   22.4          610         171         1338                4529
//   128                       14.1          484         140         1871                9027
//   512                       54.9          534         154         1135                3745
//   (calls of 10 steps, ordered / 128)  2 x 2,048 20.5 / 13.8, 3 x 2,048 22.1 / 16.4, 2 x 3,000
//   25.5 / 19.4, 2,048 + 100 22.1 / 11.3, 3,100 x 10 44.0 / 42.4, 10,000 x 31 419 / 146
// 128: while the rows written per step (24 B per body and block) stay in the
// L2 cache (kMsymRowBytes) or are few (kMsymFewRows per body), and the block
// pairs fill the GPU's 4 x SMs CTAs once at most or at least five times
// (between, the second round runs half empty: 128 loses up to 8,192 bodies; it
// wins from about 8,500, so the line at five rounds, 9,857 bodies, leaves up to
// 9 % there), for a largest system of at least kMsymSmallBodies or block pairs
// enough for five rounds; else 512 where that gives 8 warps per SM and the rows
// would have left the cache.  Below kMsymSmallBodies 128 would win too (1,031
// bodies by a quarter); contexts there keep the kernel whose tiles the caller
// can set and tune.  (4 CTAs per SM and the 80 MB, 62 % of GB300's L2, are this
// GPU's.)
constexpr int64_t kMsymRowBytes = 80000000;
constexpr int64_t kMsymFewRows = 8;
constexpr int64_t kMsymSmallBodies = 2048;

inline int msym_small_block(const std::vector<int64_t> &sizes, int64_t nsm) {
  constexpr int64_t B = 32 * kMsymMinTiles, Bw = 4 * B;
  int64_t nmax = 0, N = 0, rows = 0;
  for (int64_t n : sizes) {
    nmax = std::max(nmax, n);
    N += n;
    rows += (n + B - 1) / B * n;
  }
  if (nmax >= kMsymMinBodies) return 0;  // pair_once_block decides
  if (24 * rows > kMsymRowBytes && rows > kMsymFewRows * N)
    return pair_once_row_bytes(sizes, Bw) <= kSymRowLimit / 4 && pair_once_items(sizes, Bw) * (Bw / B) >= 8 * nsm
               ? static_cast<int>(Bw)
               : 0;
  if (pair_once_row_bytes(sizes, B) > kSymRowLimit / 4) return 0;
  const int64_t items = pair_once_items(sizes, B);
  const bool fills = items >= 20 * nsm;
  return fills || (nmax >= kMsymSmallBodies && items <= 4 * nsm) ? static_cast<int>(B) : 0;
}

}  // namespace nb
