// mu |d|^-3 of a pair in full FP64 accuracy on the integer pipes.
//
// GB300 issues an FP64 operation of a warp every 76 cycles per SM
// sub-partition (measured; 1/64 of the FP32 rate), a 32x32+64-bit integer
// multiply-add every 2.  The part of Eq. 1 between the difference d and the
// factors mu_j |d|^-3, mu_i |d|^-3 -- |d|^2, the reciprocal cube and the two
// mass products, 11 of a pair's 20 FP64 operations -- is therefore done in
// 64-bit fixed point, about 120 integer instructions, which run beside the
// 9 FP64 operations that are left (3 differences, 6 accumulations).  The
// differences too can be had in fixed point (further below).
//
// Method (own derivation; the numbers are integers, errors in brackets are
// relative):
//   1. The components of |d| are aligned to the largest one's exponent em:
//      A_c = (h_c, l_c) with the largest in [2^61, 2^62); smaller ones lose
//      bits below 2^-61 of it.
//   2. R = sum h_c^2 + 2 sum h_c l_c / 2^32 ~ |A|^2 / 2^64 (the l_c^2 / 2^64 are
//      dropped: < 3 units of R >= 2^58), then scaled by 4 if below 2^60:
//      R in [2^60, 2^62)  [< 2^-57].
//   3. Y ~ 2^51 R^-1/2, an integer of at most 21 bits, from the FP32
//      reciprocal square root of R's upper word; T = Y^3 exactly.
//   4. e = 1 - R Y^2 / 2^102 from the low 64 bits of R Y^2 / 2^32 (the upper
//      ones cancel), |e| < 2^-19, in units of 2^-70 [2^-69].
//   5. R^-3/2 = 2^-153 T (1 - e)^-3/2 = 2^-153 T (1 + 3e/2 + 15e^2/8 + ...)
//      (binomial series; the dropped 35/16 e^3 is below 2^-56).
//   6. The products with the masses' 53-bit mantissas keep 63 bits and round
//      once to FP64.
// The exponents are kept apart throughout.  Against exact arithmetic the
// factor is within 0.77 units in the last place by the bounds above and the
// final rounding (largest of 60 million draws: 0.57; of the FP64 series it
// replaces: 4.8), see the CPU test.  Differences or masses whose
// exponents leave the range below (d zero, subnormal, infinite, NaN, beyond
// 2^+-200; masses beyond 2^+-400) take the FP64 series instead.
//
// Plain C++ (a CPU test builds the same code); __CUDACC__ adds the
// instructions.
#pragma once

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define NB_HD __host__ __device__ __forceinline__
#else
#include <cmath>
#define NB_HD inline
#endif

namespace nb {
namespace ic {

// Exponent fields (of an FP64 number) of differences and masses that the
// integer path takes: |d| in [2^-200, 2^200], mu in [2^-400, 2^400] or 0.
constexpr uint32_t kDExpMin = 1023 - 200, kDExpSpan = 400;
constexpr uint32_t kMExpMin = 1023 - 400, kMExpSpan = 800;

NB_HD uint64_t wide(uint32_t a, uint32_t b) { return static_cast<uint64_t>(a) * b; }
NB_HD uint32_t mulhi(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
  return __umulhi(a, b);
#else
  return static_cast<uint32_t>(wide(a, b) >> 32);
#endif
}
NB_HD int32_t mulhi_s(int32_t a, int32_t b) {
#ifdef __CUDA_ARCH__
  return __mulhi(a, b);
#else
  return static_cast<int32_t>((static_cast<int64_t>(a) * b) >> 32);
#endif
}
// (hi:lo) << s, upper word (s < 32) / >> s, lower word (s <= 32: clamped)
NB_HD uint32_t fshl(uint32_t lo, uint32_t hi, uint32_t s) {
#ifdef __CUDA_ARCH__
  return __funnelshift_l(lo, hi, s);
#else
  return static_cast<uint32_t>((((static_cast<uint64_t>(hi) << 32) | lo) << (s & 31)) >> 32);
#endif
}
NB_HD uint32_t fshr(uint32_t lo, uint32_t hi, uint32_t s) {
#ifdef __CUDA_ARCH__
  return __funnelshift_rc(lo, hi, s);
#else
  return static_cast<uint32_t>(((static_cast<uint64_t>(hi) << 32) | lo) >> (s > 32 ? 32 : s));
#endif
}
NB_HD uint32_t shr(uint32_t v, uint32_t s) {  // 0 for s >= 32
#ifdef __CUDA_ARCH__
  uint32_t r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(s));
  return r;
#else
  return s >= 32 ? 0u : v >> s;
#endif
}
NB_HD uint32_t clz32(uint32_t v) {
#ifdef __CUDA_ARCH__
  return static_cast<uint32_t>(__clz(static_cast<int>(v)));
#else
  return v ? static_cast<uint32_t>(__builtin_clz(v)) : 32u;
#endif
}
NB_HD uint32_t lo32(uint64_t v) { return static_cast<uint32_t>(v); }
NB_HD uint32_t hi32(uint64_t v) { return static_cast<uint32_t>(v >> 32); }
NB_HD uint64_t make64(uint32_t lo, uint32_t hi) { return (static_cast<uint64_t>(hi) << 32) | lo; }
NB_HD uint64_t bits(double x) {
#ifdef __CUDA_ARCH__
  return static_cast<uint64_t>(__double_as_longlong(x));
#else
  uint64_t u;
  std::memcpy(&u, &x, 8);
  return u;
#endif
}
NB_HD double from_bits(uint32_t lo, uint32_t hi) {
#ifdef __CUDA_ARCH__
  return __hiloint2double(static_cast<int>(hi), static_cast<int>(lo));
#else
  const uint64_t u = make64(lo, hi);
  double x;
  std::memcpy(&x, &u, 8);
  return x;
#endif
}

// A mass as the product takes it: u = the mantissa's upper 32 bits (leading
// one at bit 31; 0 for a massless body), w = its lower 21 bits, then the
// 11-bit exponent field.
struct Mass {
  uint32_t u, w;
};
NB_HD Mass pack_mass(double mu) {
  const uint64_t b = bits(mu);
  const uint32_t lo = lo32(b), hi = hi32(b);
  Mass m;
  m.u = ((hi << 1) | lo) == 0u ? 0u : fshl(lo, hi, 11) | 0x80000000u;  // (an FP64 compare would cost a pipe slot)
  m.w = (lo << 11) | ((hi >> 20) & 0x7ffu);
  return m;
}
NB_HD bool mass_in_range(const Mass &m) { return m.u == 0u || (m.w & 0x7ffu) - kMExpMin <= kMExpSpan; }
NB_HD double unpack_mass(const Mass &m) {  // exact for every mu >= 0
  return from_bits((m.w >> 11) | (m.u << 21), m.u ? ((m.w & 0x7ffu) << 20) | ((m.u & 0x7fffffffu) >> 11) : 0u);
}

// |d|^-3 (or |d|^-1) as a 64-bit mantissa, its leading one at bit 63, and the
// exponent that mass_times adds to the mass's own exponent field.
struct Cube {
  uint32_t lo, hi;
  int32_t e;
};

// FP32 reciprocal square root of the seed (`rsq` lets a test perturb it).
struct Rsqrt {
  NB_HD float operator()(float x) const {
#ifdef __CUDA_ARCH__
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
#else
    return static_cast<float>(1.0 / std::sqrt(static_cast<double>(x)));
#endif
  }
};

// Largest exponent field of the components (in place, bits 20..30).
NB_HD uint32_t max_exp(double dx, double dy, double dz) {
  const uint32_t ex = hi32(bits(dx)) & 0x7ff00000u, ey = hi32(bits(dy)) & 0x7ff00000u,
                 ez = hi32(bits(dz)) & 0x7ff00000u;
  const uint32_t m = ex > ey ? ex : ey;
  return m > ez ? m : ez;
}
// Whether the integer path takes a difference with this largest exponent.
NB_HD bool exp_in_range(uint32_t em20) { return (em20 >> 20) - kDExpMin <= kDExpSpan; }

// R in [2^58, 2^62) of the aligned components, see (1) and (2); em20 =
// max_exp(d), in range.
NB_HD uint64_t square_sum(double dx, double dy, double dz, uint32_t em20) {
  const double d[3] = {dx, dy, dz};
  uint64_t R = 0, C = uint64_t(3) << 30;  // (C starts at the mean of what (2) and the shift drop: 1.5 units of R)
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int c = 0; c < 3; ++c) {
    const uint64_t b = bits(d[c]);
    const uint32_t lo = lo32(b), hi = hi32(b);
    const uint32_t s = (em20 - (hi & 0x7ff00000u)) >> 20;
    const uint32_t mh = (hi & 0x000fffffu) | 0x00100000u;  // (a zero component: exponent 0, shifted out)
    const uint32_t ah = fshl(lo, mh, 9), al = lo << 9;
    const uint32_t h = shr(ah, s), l = fshr(al, ah, s);
    R += wide(h, h);
    C += wide(h, l);
  }
  return R + (C >> 31);
}

// Steps (2) .. (4): R scaled by 2^k (k = 0 or 2), Y and T2 = Y^2 = (th, tl), and
// e = 1 - R Y^2 / 2^102: ne = -e in units of 2^-70, q = e^2 in units of 2^-66.
struct Root {
  uint32_t k, Y, th, tl;
  int64_t ne;
  int32_t q;
};
template <class Rsq>
NB_HD Root inv_root(uint64_t R, const Rsq &rsq) {
  Root o;
  o.k = hi32(R) < (1u << 28) ? 2u : 0u;  // scale by 4 below 2^60
  const uint32_t Rh = fshl(lo32(R), hi32(R), o.k), Rl = lo32(R) << o.k;
  const float y = rsq(static_cast<float>(Rh));  // Rh in [2^28, 2^30)
#ifdef __CUDA_ARCH__
  const uint32_t Yr = static_cast<uint32_t>(__float_as_int(__fmaf_rn(y, 34359738368.0f, 8388608.0f))) - 0x4b000000u;
#else
  const float z = std::fmaf(y, 34359738368.0f, 8388608.0f);  // 2^35 y + 2^23: Y in the low mantissa bits
  uint32_t zb;
  std::memcpy(&zb, &z, 4);
  const uint32_t Yr = zb - 0x4b000000u;
#endif
  o.Y = Yr < 0x1fffffu ? Yr : 0x1fffffu;  // Y^3 < 2^63
  const uint64_t t = wide(o.Y, o.Y);
  o.th = hi32(t);
  o.tl = lo32(t);
  // R t / 2^32 mod 2^64 = -e in units of 2^-70
  uint64_t Q = wide(Rh, o.tl) + wide(Rl, o.th) + mulhi(Rl, o.tl);
  Q += static_cast<uint64_t>(Rh * o.th) << 32;
  o.ne = static_cast<int64_t>(Q);
  const int32_t e1 = static_cast<int32_t>(o.ne >> 21);  // -e in units of 2^-49
  o.q = mulhi_s(e1, e1);
  return o;
}

// The mantissa S, its leading one shifted to bit 63, and the exponent.
NB_HD Cube normalised(uint64_t S, int32_t e) {
  const uint32_t n = clz32(hi32(S));
  Cube c;
  c.hi = fshl(lo32(S), hi32(S), n);
  c.lo = lo32(S) << n;
  c.e = e - static_cast<int32_t>(n);
  return c;
}

// |d|^-3, step (5); em: the exponent field of |d|'s largest component.
NB_HD Cube cube_of(const Root &o, uint32_t em) {
  const int64_t g = static_cast<int64_t>(o.q) * 30 - (o.ne + (o.ne >> 1));  // 3e/2 + 15e^2/8 in units of 2^-70
  uint64_t T = wide(o.Y, o.tl);  // Y^3
  T += static_cast<uint64_t>(o.Y * o.th) << 32;
  // T g / 2^70 = (Th 2^32 + Tl) (gh 2^32 + gl) / 2^70
  const uint32_t Th = hi32(T), Tl = lo32(T);
  const int32_t gh = static_cast<int32_t>(g >> 32);
  const uint32_t gl = lo32(static_cast<uint64_t>(g));
  int64_t V = static_cast<int64_t>(static_cast<int32_t>(Th)) * gh;
  V += mulhi(Th, gl);
  V += 2 * static_cast<int64_t>(mulhi_s(static_cast<int32_t>(Tl >> 1), gh));
  return normalised(T + static_cast<uint64_t>(V >> 6),
                    3065 + static_cast<int32_t>(o.k + (o.k >> 1)) - 3 * static_cast<int32_t>(em));
}
template <class Rsq>
NB_HD Cube inv_cube(uint64_t R, uint32_t em20, const Rsq &rsq) {
  return cube_of(inv_root(R, rsq), em20 >> 20);
}

// |d|^-3 and |d|^-2 of one difference: R^-1 = 2^-102 Y^2 (1 - e)^-1 = 2^-102 Y^2 (1 + e +
// e^2 + ...) (the dropped e^3 is below 2^-57).
NB_HD int64_t mulhi64(int64_t a, int64_t b) {
#ifdef __CUDA_ARCH__
  return __mul64hi(a, b);
#else
  return static_cast<int64_t>((static_cast<__int128>(a) * b) >> 64);
#endif
}
struct CubeSquare {
  Cube cube, square;
};
template <class Rsq>
NB_HD CubeSquare inv_cube_square(uint64_t R, uint32_t em20, const Rsq &rsq) {
  const Root o = inv_root(R, rsq);
  CubeSquare r;
  r.cube = cube_of(o, em20 >> 20);
  const uint64_t t = make64(o.tl, o.th);  // <= 2^42
  const int64_t g = static_cast<int64_t>(o.q) * 16 - o.ne;  // e + e^2 in units of 2^-70
  const uint64_t S = (t << 20) + static_cast<uint64_t>(mulhi64(static_cast<int64_t>(t << 14), g));  // 2^20 t (1 + g)
  r.square = normalised(S, 2044 + static_cast<int32_t>(o.k) - 2 * static_cast<int32_t>(em20 >> 20));
  return r;
}

// |d|^-1 likewise: 2^-51 Y (1 - e)^-1/2 = 2^-51 Y (1 + e/2 + 3e^2/8 + ...)
// (the dropped 5/16 e^3 is below 2^-59).
template <class Rsq>
NB_HD Cube inv_dist(uint64_t R, uint32_t em20, const Rsq &rsq) {
  const Root o = inv_root(R, rsq);
  const int64_t g = static_cast<int64_t>(o.q) * 6 - (o.ne >> 1);  // e/2 + 3e^2/8 in units of 2^-70
  const int32_t gh = static_cast<int32_t>(g >> 32);
  const uint32_t gl = lo32(static_cast<uint64_t>(g));
  // S = 2^42 Y (1 + g): Y g / 2^28 from the two words of g
  const int64_t V = ((static_cast<int64_t>(static_cast<int32_t>(o.Y)) * gh) << 4) +
                    static_cast<int64_t>(wide(o.Y, gl) >> 28);
  const uint64_t S = make64(0u, o.Y << 10) + static_cast<uint64_t>(V);
  return normalised(S, 1021 + static_cast<int32_t>(o.k >> 1) - static_cast<int32_t>(em20 >> 20));
}

// mu |d|^-3 (mu |d|^-1), rounded to FP64 (half up in the 63-bit product).
NB_HD double mass_times(const Mass &m, const Cube &c) {
  const uint32_t ul = m.w & 0xfffff800u;
  const uint64_t F = wide(m.u, c.hi) + mulhi(m.u, c.lo) + mulhi(ul, c.hi);  // [2^62, 2^64)
  const uint32_t b = hi32(F) >> 31;
  const uint32_t l = fshr(lo32(F), hi32(F), b), h = hi32(F) >> b;
  const uint64_t M = make64(l, h) + 0x200u;
  const uint32_t lo = fshr(lo32(M), hi32(M), 10);
  const uint32_t hi = (hi32(M) >> 10) + ((static_cast<uint32_t>(c.e) + (m.w & 0x7ffu) + b) << 20);
  return from_bits(lo, m.u ? hi : 0u);
}

// ---------------------------------------------------------------------------
// Differences in fixed point.  Within a pair of 32-body tiles the coordinates
// become 96-bit integers X = x 2^(1115 - E), E the largest exponent field among
// them, so |X| < 2^93: exact for a coordinate of at least 2^-40 of the largest,
// to one unit otherwise.  D = Xj - Xi is the difference, exact or within 2^-92
// of the tiles' largest coordinate; its upper 64 bits, shifted, are the
// aligned components that the square sum takes, and each component rounds
// once to FP64 for the accumulations -- without the FP64 pipe and as exact as
// its subtraction (64-bit integers are not: a component much smaller than
// the others then loses bits that FP64 keeps).  Pairs closer than 2^-7 of the
// scale, and those with a component below 2^-30 of the largest, are left to
// FP64.
// ---------------------------------------------------------------------------

// Exponent fields E for which every difference taken is in the range above.
NB_HD bool fix_in_range(uint32_t E) { return E - (kDExpMin + 8) <= kDExpSpan - 16; }

struct Fix {
  uint32_t w[3];  // two's complement, w[2] the uppermost
};
NB_HD Fix fix_of(unsigned __int128 v) {
  Fix f;
  f.w[0] = static_cast<uint32_t>(v);
  f.w[1] = static_cast<uint32_t>(v >> 32);
  f.w[2] = static_cast<uint32_t>(v >> 64);
  return f;
}
// Beyond every coordinate: the place of a lane outside the system.
NB_HD Fix fix_pad() { return fix_of(static_cast<unsigned __int128>(1) << 93); }

NB_HD Fix to_fix(double x, uint32_t E) {
  const uint64_t b = bits(x);
  const uint32_t hi = hi32(b), s = E - ((hi >> 20) & 0x7ffu);
  const uint64_t m = make64(lo32(b), (hi & 0x000fffffu) | 0x00100000u);  // (a subnormal x: shifted out)
  const unsigned __int128 v = s <= 40u ? static_cast<unsigned __int128>(m) << (40u - s) : s < 104u ? m >> (s - 40u) : 0u;
  return fix_of(static_cast<int32_t>(hi) < 0 ? -v : v);
}

// a - b, and |a - b| with the sign in *neg (all ones if negative).
NB_HD void fix_abs_diff(const Fix &a, const Fix &b, uint32_t (&m)[3], uint32_t *neg) {
#ifdef __CUDA_ARCH__
  uint32_t d0, d1, d2;
  asm("sub.cc.u32 %0, %3, %6;\n\tsubc.cc.u32 %1, %4, %7;\n\tsubc.u32 %2, %5, %8;"
      : "=r"(d0), "=r"(d1), "=r"(d2)
      : "r"(a.w[0]), "r"(a.w[1]), "r"(a.w[2]), "r"(b.w[0]), "r"(b.w[1]), "r"(b.w[2]));
  const uint32_t s = static_cast<uint32_t>(static_cast<int32_t>(d2) >> 31);
  asm("sub.cc.u32 %0, %3, %6;\n\tsubc.cc.u32 %1, %4, %6;\n\tsubc.u32 %2, %5, %6;"
      : "=r"(m[0]), "=r"(m[1]), "=r"(m[2])
      : "r"(d0 ^ s), "r"(d1 ^ s), "r"(d2 ^ s), "r"(s));
  *neg = s;
#else
  auto whole = [](const Fix &f) {
    return static_cast<__int128>((static_cast<unsigned __int128>(static_cast<int64_t>(static_cast<int32_t>(f.w[2]))) << 64) |
                                 make64(f.w[0], f.w[1]));
  };
  const __int128 d = whole(a) - whole(b);
  const Fix f = fix_of(static_cast<unsigned __int128>(d < 0 ? -d : d));
  m[0] = f.w[0];
  m[1] = f.w[1];
  m[2] = f.w[2];
  *neg = d < 0 ? ~0u : 0u;
#endif
}

// A difference from fixed point: magnitudes (h, l, t) with the largest h in
// [2^29, 2^30), signs, em as above; ok false where FP64 has to take it.
struct FixDiff {
  uint32_t h[3], l[3], t[3], sign[3];
  uint32_t em;
  bool ok;
};
NB_HD FixDiff fix_diff(const Fix (&xj)[3], const Fix (&xi)[3], uint32_t E) {
  FixDiff f;
  uint32_t mx = 0u, mn = ~0u;
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int c = 0; c < 3; ++c) {
    uint32_t m[3], neg;
    fix_abs_diff(xj[c], xi[c], m, &neg);
    f.sign[c] = neg & 0x80000000u;
    f.h[c] = m[2];
    f.l[c] = m[1];
    f.t[c] = m[0];
    mx = m[2] > mx ? m[2] : mx;
  }
  f.ok = mx >= (1u << 22);
  const uint32_t n = clz32(mx), s = n - 2u;  // (|D| < 2^94: n >= 2)
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int c = 0; c < 3; ++c) {
    f.h[c] = fshl(f.l[c], f.h[c], s);
    f.l[c] = fshl(f.t[c], f.l[c], s);
    f.t[c] <<= s & 31u;
    mn = f.h[c] < mn ? f.h[c] : mn;
  }
  f.ok = f.ok && mn != 0u;
  f.em = E + 3u - n;
  return f;
}
NB_HD uint64_t square_sum(const FixDiff &f) {
  uint64_t R = 0, C = uint64_t(3) << 30;
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int c = 0; c < 3; ++c) {
    R += wide(f.h[c], f.h[c]);
    C += wide(f.h[c], f.l[c]);
  }
  return R + (C >> 31);
}
// Component c, rounded to FP64.
NB_HD double fix_value(const FixDiff &f, int c) {
  const uint32_t m = clz32(f.h[c]), s = m - 1u;  // (2 <= m < 32)
  const uint64_t v = make64(fshl(f.t[c], f.l[c], s), fshl(f.l[c], f.h[c], s)) + 0x200u;  // leading one at bit 62
  const uint32_t hi = (hi32(v) >> 10) + ((f.em + 1u - m) << 20);
  return from_bits(fshr(lo32(v), hi32(v), 10), hi | f.sign[c]);
}

}  // namespace ic
}  // namespace nb
