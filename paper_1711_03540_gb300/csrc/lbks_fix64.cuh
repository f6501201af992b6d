// The collision of one site of FP64 storage in 64-bit block fixed point, on the integer
// pipes.  (Plain C++ apart from a few one-instruction helpers, so that host tests run the
// same arithmetic.)
//
// Why: an SM of this part issues 1.7 FP64 operations per clock against 55 32 x 32 -> 64-bit
// multiply-adds, 60 shifts and 110 32-bit adds (measured), so the collision's 29 FP64
// operations (D1Q7) take 17 clocks of an SM however they are arranged: 1.9e10
// site-updates/s on 152 SMs, which the plain kernel ran at.  Here:
//  1. Every pair of planes +-p has a grid of its own, kp[p] binades finer than g_0's: f^eq_p is
//     that much smaller than rho (fix_coef).  The site's exponent e is the largest of g_0's and
//     of the planes' plus kp[p], so that each plane has 56 bits for its share of the largest
//     density about the site.  (One grid for all planes rounds the small ones coarsely, and the
//     same way for many steps where a step changes little: errors of 5 to 10 times FP64
//     arithmetic's after 200000 steps.)  Bits below the grid are jammed into the last one (it is
//     set when any is lost): unlike truncation, and unlike rounding halves away, that has no
//     bias, which would drift the conserved mass linearly in time.
//  2. s = sum g_i is rounded once to g_0's grid.  With u, w the sum and the difference of a
//     pair, its new values are even + odd and even - odd, even = r u / 2 + a_p s and
//     odd = r w / 2 + b_p s^2, sums of limb products (32 x 32 -> 64-bit multiply-adds) on half
//     the plane's grid, rounded.  The products of two low limbs are left out; their mean, where
//     it is not zero, is added (the sign of g_i with r).
//  3. g_0 takes s minus the others, exactly, to 32 bits below its grid.  What its 53 bits cannot
//     hold is not dropped but handed to the planes +-1 (a sixteenth or half of it to +-2), so that the
//     collision keeps the mass to the other planes' conversions.  FP64 arithmetic keeps it
//     too, by adding and subtracting the same rounded values; rounding g_0 alone lets the
//     long waves and the mass walk randomly, up to twice its error.
//  4. The hardware's conversion (64-bit integer to FP64, round to nearest even, on the idle
//     FP64 pipe) rounds each result once.
// Lattices advanced 16000 to 400000 steps end 0.03 to 0.6 times as far from a long double run as
// with FP64 arithmetic (spacings 0.0245-0.6, tau 1-3, means 0 to 3.7, time steps down to where
// the planes +-1 are 16 to 18 binades below g_0; there FP64 arithmetic takes over).  Where a
// lattice decays until a step no longer changes it, both stop short, this one at 0.1 of the
// distance.
// About 500 instructions per site instead of 29 FP64 ones.  What bounds the many-step kernel
// (3.9e10 site-updates/s on the 4096-lattice ensemble) is the pipe of shifts, logic and adds, 73 % busy,
// then multiply-adds (0.49) and the conversions (7 of 2 a clock).  Written for that pipe: signs by
// multiplication, pairs as sum and difference (12 products instead of 17), shifts by a run's
// constants as products.  One grid per site took 440 instructions, 4.5e10.
#pragma once

#include <cstdint>

#if defined(__CUDACC__)
#define LBKS_HD __host__ __device__ __forceinline__
#define LBKS_UNROLL _Pragma("unroll")
#else
#define LBKS_HD inline
#define LBKS_UNROLL
#endif

namespace lbks {

// A run's coefficients as fixed-point numbers in two signed limbs, value = h 2^28 + l
// with -2^27 <= l < 2^27 (fix_coef): r at 2^56, a_p = a_{+p} = a_{-p} at 2^(57 + kp[p]),
// b_p = b_{+p} = -b_{-p} at 2^(kb + kp[p]), kb the largest with |b_p| 2^(kb + kp[p]) < 2^55 for
// every p.  kp[p]: the planes +-p lie that many binades below the site's scale.
struct FixCoef {
  int32_t rh, rl, ah[3], al[3], bh[3], bl[3];
  int16_t kp[3];
  int16_t z0;  // kb - 55 + 1022; 0: out of range, every site of the run takes FP64 arithmetic
};

namespace fix64 {

constexpr int kLimb = 28;             // bits of a low limb
constexpr int32_t kMask = (1 << kLimb) - 1;

// Shifts whose result is 0 once the count reaches the width (as the hardware's are).
LBKS_HD uint32_t shr32(uint32_t x, uint32_t n) {
#if defined(__CUDA_ARCH__)
  uint32_t r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(n));
  return r;
#else
  return n > 31 ? 0u : x >> n;
#endif
}
LBKS_HD uint32_t shl32(uint32_t x, uint32_t n) {
#if defined(__CUDA_ARCH__)
  uint32_t r;
  asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(n));
  return r;
#else
  return n > 31 ? 0u : x << n;
#endif
}
LBKS_HD uint64_t shr64(uint64_t x, uint32_t n) {
#if defined(__CUDA_ARCH__)
  uint64_t r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
  return r;
#else
  return n > 63 ? 0u : x >> n;
#endif
}
// x >> n and x << n of 64 bits for n < 32, and x's bits that x >> n loses, at the top of a word
LBKS_HD int64_t sra64(int64_t x, uint32_t n) {
#if defined(__CUDA_ARCH__)
  const uint32_t lo = __funnelshift_r((uint32_t)x, (uint32_t)((uint64_t)x >> 32), n);
  return (int64_t)((uint64_t)(uint32_t)((int32_t)(x >> 32) >> n) << 32 | lo);
#else
  return x >> n;
#endif
}
LBKS_HD uint32_t below64(int64_t x, uint32_t n) { return shl32((uint32_t)x, 32u - n); }
// the high word of (hi : lo) << n for n < 32
LBKS_HD int32_t shl_pair(int32_t hi, uint32_t lo, uint32_t n) {
#if defined(__CUDA_ARCH__)
  return (int32_t)__funnelshift_l(lo, (uint32_t)hi, n);
#else
  return (int32_t)(uint32_t)((((uint64_t)(uint32_t)hi << 32 | lo) << n) >> 32);
#endif
}
LBKS_HD int64_t mul(int32_t a, int32_t b) { return (int64_t)a * b; }
LBKS_HD int64_t mad(int32_t a, int32_t b, int64_t c) { return (int64_t)a * b + c; }

LBKS_HD int32_t hi_limb(int64_t x) { return (int32_t)(x >> kLimb); }
LBKS_HD int32_t lo_limb(int64_t x) { return (int32_t)((uint32_t)x & (uint32_t)kMask); }
LBKS_HD uint32_t hi32(uint64_t x) { return (uint32_t)(x >> 32); }

// A value as h 2^28 + l in units of 2^(e - 1078), |g| <= 2^(e - 1022) (both limbs carry the sign
// sg), a lost bit jammed into l.  FAR: the value may lie more than 35 binades below 2^(e - 1022).
template <bool FAR>
LBKS_HD void to_limbs(uint64_t bits, uint32_t e, int32_t& h, int32_t& l, int32_t& sg) {
  const uint32_t hi = hi32(bits), lo = (uint32_t)bits, mag = hi & 0x7fffffffu;
  const uint32_t ei = mag >> 20;
  const uint64_t p = (bits << 11) | ((uint64_t)0x80000000u << 32);   // mantissa, leading bit at 63
  // the bits below the grid: of the low word alone down to 35 binades, then of all of the
  // mantissa, and from 56 on the leading one too, which every value but zero has
  uint32_t rest = shl32(lo, ei + (35u - e));
  if (FAR && e - ei > 35u) rest = e - ei > 55u ? mag : lo | shl32(hi, ei + (67u - e));
  sg = ((int32_t)hi >> 31) | 1;
  h = (int32_t)shr32(hi32(p), (e + 4u) - ei) * sg;
  l = (int32_t)(((uint32_t)shr64(p, (e + 8u) - ei) & (uint32_t)kMask) | (rest < 1u ? rest : 1u)) * sg;
}
LBKS_HD void to_limbs(uint64_t bits, uint32_t e, int32_t& h, int32_t& l, int32_t& sg) {
  to_limbs<true>(bits, e, h, l, sg);
}

// y != 0 in units of 2^(e - 1079) rounded to the nearest FP64 (ties to even) by the
// conversion unit; adj = (e - 1079) 2^20 moves the exponent.  low: the smallest high word
// of the converted values (0 for y = 0).
LBKS_HD uint64_t to_fp64(int64_t y, uint32_t adj, uint32_t& low) {
  const double v = (double)y;
#if defined(__CUDA_ARCH__)
  const uint64_t b = (uint64_t)__double_as_longlong(v);
#else
  uint64_t b;
  __builtin_memcpy(&b, &v, 8);
#endif
  low = hi32(b) < low ? hi32(b) : low;
  return b + ((uint64_t)adj << 32);
}

}  // namespace fix64

// Collision of one site, bits of g_i in and out.  False when it is out of range (`out` is
// then meaningless): all values zero, tiny, infinite or NaN, b_p s^2 beyond four times the
// scale of plane p, or a run whose coefficients are (FixCoef::z0).
template <int Q>
LBKS_HD bool fix_collide(const uint64_t (&g)[Q], uint64_t (&out)[Q], const FixCoef& k) {
  using namespace fix64;
  constexpr int P = (Q - 1) / 2;
  // the site's scale 2^(e - 1022): g_0 below it and the planes +-p kp[p] binades further down
  const uint32_t m0 = hi32(g[0]) & 0x7fffffffu;
  uint32_t top = m0, least = 0xffffffffu;
  LBKS_UNROLL
  for (int p = 0; p < P; ++p) {
    const uint32_t u = hi32(g[2 * p + 1]) & 0x7fffffffu, v = hi32(g[2 * p + 2]) & 0x7fffffffu;
    const uint32_t scale = (uint32_t)k.kp[p] << 20, w = (u > v ? u : v) + scale, x = (u > v ? v : u) + scale;
    top = w > top ? w : top;
    least = x < least ? x : least;
  }
  const uint32_t e = top >> 20;
  const uint32_t zn = (uint32_t)k.z0 - e;  // shift of s^2; negative for z0 = 0 (and NaN, infinities)
  int32_t h[Q], l[Q], sg[Q];
  // (g_0 may be far below the scale, about a zero of the density, where the planes are not: a
  // lattice odd in x has such sites at all times)
  to_limbs<true>(g[0], e, h[0], l[0], sg[0]);
  LBKS_UNROLL
  for (int i = 1; i < Q; ++i) to_limbs<false>(g[i], e - (uint32_t)k.kp[(i - 1) / 2], h[i], l[i], sg[i]);
  if (e - (least >> 20) > 35u) {
  LBKS_UNROLL
    for (int i = 1; i < Q; ++i) to_limbs<true>(g[i], e - (uint32_t)k.kp[(i - 1) / 2], h[i], l[i], sg[i]);
  }
  // of each pair its sum (in h, l, sg of the first) and difference (of the second); s = sum g_i,
  // rounded to g_0's grid
  int64_t y0 = mad(h[0], 1 << kLimb, (int64_t)l[0]), s = y0;
  int32_t part = 1 << (kLimb - 1);
  LBKS_UNROLL
  for (int p = 0; p < P; ++p) {
    const int i = 2 * p + 1, j = i + 1, kp = k.kp[p];
    const int32_t dh = h[i] - h[j], dl = l[i] - l[j], ds = sg[i] - sg[j];
    h[i] += h[j];
    l[i] += l[j];
    sg[i] += sg[j];
    h[j] = dh;
    l[j] = dl;
    sg[j] = ds;
    s = mad(h[i], (1 << kLimb) >> kp, s);
    part += (l[i] + ((1 << kp) >> 1)) >> kp;
  }
  s += part;
  // its low limb balanced: s^2 without that limb's square is then never negative (it was for a
  // small negative s, the sum of populations that cancel)
  const int32_t sh = hi_limb(s), sl = lo_limb(s) - (1 << (kLimb - 1));
  // s^2 on the grid that makes b_p s^2 come out on the results', its low limb balanced too
  const uint64_t zz = 4 * (uint64_t)mul(sh, sh) + (uint64_t)(mad(sh, sl, 1 << (kLimb - 4)) >> (kLimb - 3));
  const uint64_t zr = shr64(zz, zn) + ((1u << (kLimb - 1)) + ((uint32_t)shr64(zz, zn - 1u) & 1u));
  const int32_t zh = hi_limb((int64_t)zr), zl = lo_limb((int64_t)zr) - (1 << (kLimb - 1));
  if (e < 128u || (int32_t)zn < 0 || (uint32_t)(zr >> 59) != 0u) return false;
  // results in units of half the planes' grids: even + odd and even - odd
  const int32_t rhalf = k.rl >> 1;
  int64_t y[Q];
  uint32_t low = 0xffffffffu;
  uint64_t f = 0;  // what y0 holds below its unit, in 2^-32 of it
  LBKS_UNROLL
  for (int p = P - 1; p >= 0; --p) {
    const int i = 2 * p + 1, j = i + 1;
    const int64_t el = mad(l[i], k.rh, mad(h[i], k.rl, mad(sg[i], rhalf, 1 << (kLimb - 1))));
    const int64_t ol = mad(l[j], k.rh, mad(h[j], k.rl, mad(sg[j], rhalf, 1 << (kLimb - 1))));
    const int64_t even = mad(sh, k.ah[p], mul(h[i], k.rh)) + (mad(sl, k.ah[p], mad(sh, k.al[p], el)) >> kLimb);
    const int64_t odd = mad(zh, k.bh[p], mul(h[j], k.rh)) + (mad(zl, k.bh[p], mad(zh, k.bl[p], ol)) >> kLimb);
    y[i] = even + odd;
    y[j] = even - odd;
    const int64_t d = mad(h[i], 1 << kLimb, (int64_t)l[i]) - even;
    if (p == 2) {
      out[i] = to_fp64(y[i], (e - (uint32_t)k.kp[p] - 1079u) << 20, low);
      out[j] = to_fp64(y[j], (e - (uint32_t)k.kp[p] - 1079u) << 20, low);
    }
    y0 += sra64(d, (uint32_t)k.kp[p]);
    f += below64(d, (uint32_t)k.kp[p]);
  }
  y0 += (int64_t)(f >> 32);
  // g_0 keeps the bits it had room for; what is left goes to the planes +-1, half each (the odd
  // unit to either in turn), but for a sixteenth that the planes +-2 take (so that none takes as
  // much as a quarter of g_0's last bit; where their grid is fine enough).  They take half where
  // the planes are so small that short waves stay long: four directions make less noise than two.
  const uint32_t gap = e - (m0 >> 20), bit = gap < 3u ? 8u >> gap : 1u;
  const int64_t v0 = (y0 + (int64_t)(gap < 3u ? bit >> 1 : (uint32_t)f >> 31)) & -(int64_t)bit;
  const int32_t left = (int32_t)((uint32_t)y0 - (uint32_t)v0);
  const int32_t share = k.kp[1] < 2 ? 0 : k.kp[0] > 14 ? 8 : 1;
  const int32_t far = (left * share + (share < 2 ? 2 * share : 4)) >> 2;
  const uint32_t lo = (uint32_t)f - ((uint32_t)far << 30);
  const int32_t hi = left - (far >> 2) - (lo > (uint32_t)f ? 1 : 0);
  const int32_t near = shl_pair(hi, lo, (uint32_t)k.kp[0] + 1u) | (shl32(lo, (uint32_t)k.kp[0] + 1u) ? 1 : 0);
  const int32_t half = (near >> 1) + (near & (int32_t)((uint32_t)y[1] >> 4) & 1), half2 = far * ((1 << k.kp[1]) >> 2);
  y[1] += half;
  y[2] += near - half;
  y[3] += half2;
  y[4] += half2;
  out[0] = to_fp64(v0, (e - 1078u) << 20, low);
  LBKS_UNROLL
  for (int i = 1; i < 5; ++i) out[i] = to_fp64(y[i], (e - (uint32_t)k.kp[(i - 1) / 2] - 1079u) << 20, low);
  if (low == 0u) {  // a result of zero
  LBKS_UNROLL
    for (int i = 0; i < Q; ++i)
      if (out[i] == (uint64_t)((e - (i ? (uint32_t)k.kp[(i - 1) / 2] + 1079u : 1078u)) << 20) << 32) out[i] = 0;
  }
  return true;
}

// The limbs of a run's coefficients (r, a_i, b_i as in RunDesc, i in speed order).
LBKS_HD void fix_limbs(double v, double scale, int32_t& h, int32_t& l) {
#if defined(__CUDA_ARCH__)
  const int64_t q = __double2ll_rn(v * scale);
#else
  const int64_t q = (int64_t)__builtin_nearbyint(v * scale);
#endif
  h = (int32_t)((q + (1 << (fix64::kLimb - 1))) >> fix64::kLimb);
  l = (int32_t)(q - (int64_t)h * (1 << fix64::kLimb));
}

LBKS_HD FixCoef fix_coef(int Q, double r, double rhobar, const double* a, const double* b) {
  FixCoef k{};
  const int P = (Q - 1) / 2;
  double asum = 0.0, bmax = 0.0, scale[3] = {};
  bool pairs = true;
  for (int p = 0; p < P; ++p) {
    const double x = a[2 * p + 1], y = b[2 * p + 1];
    pairs = pairs && x == a[2 * p + 2] && y == -b[2 * p + 2];
    const double ax = x < 0.0 ? -x : x, ay = y < 0.0 ? -y : y;
    asum += 2.0 * ax;
    // f^eq_p / rho = A_p + B_p rho: the larger of |A_p| and 4 |B_p| (A_p = a_p / (1 - r)) as a
    // power of two, so that a plane's share of b_p s^2 has room up to |rho| = 8 tau at least
    const double size = ax > 4.0 * ay ? ax : 4.0 * ay;
    scale[p] = 1.0;
    while (k.kp[p] < 27 && 4.0 * scale[p] * size <= 1.0 - r) { scale[p] *= 2.0; ++k.kp[p]; }
    pairs = pairs && (size == 0.0 || 32.0 * scale[p] * size >= 1.0 - r);  // (a_p exact in its limbs)
    bmax = ay * scale[p] > bmax ? ay * scale[p] : bmax;
  }
  // Planes so small that a step hardly changes a lattice: what g_0 hands them stops being random
  // there, and errors reach 1.4 times FP64 arithmetic's (18 binades at tau 1.05, 20 at 1.5; 0.7 up
  // to these limits)
  if (k.kp[0] > (r < 0.3 ? 16 : 18)) return FixCoef{};
  // Limits that keep every sum below 64 bits: |s| < 2^58.8, 1 + sum |a_i| <= 8 (NaNs fail)
  if (!(pairs && rhobar == 0.0 && r >= 0.0 && r <= 1.0 && asum <= 7.0 && bmax >= 0x1p-60 && bmax <= 0x1p3))
    return FixCoef{};
  int kb = 48;
  double sb = 0x1p48;
  while (2.0 * sb * bmax < 0x1p55) { sb *= 2.0; ++kb; }
  fix_limbs(r, 0x1p56, k.rh, k.rl);
  for (int p = 0; p < P; ++p) {
    fix_limbs(a[2 * p + 1], scale[p] * 0x1p57, k.ah[p], k.al[p]);
    fix_limbs(b[2 * p + 1], scale[p] * sb, k.bh[p], k.bl[p]);
  }
  k.z0 = (int16_t)(kb - 55 + 1022);
  return k;
}

}  // namespace lbks
