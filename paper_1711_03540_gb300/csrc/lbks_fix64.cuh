// The collision of one site of FP64 storage in 64-bit block fixed point, on the integer
// pipes.  (Plain C++ apart from a few one-instruction helpers, so that host tests run the
// same arithmetic.)
//
// Why: an SM of this part issues 1.7 FP64 operations per clock against 55 32 x 32 -> 64-bit
// multiply-adds, 60 shifts and 110 32-bit adds (measured), so the collision's 29 FP64
// operations (D1Q7) take 17 clocks of an SM however they are arranged: 1.9e10
// site-updates/s on 152 SMs, which the plain kernel ran at.  Here:
//  1. The site's largest exponent e sets a grid of 2^(e - 1078): 56 bits for its largest
//     population.  Each population becomes two signed limbs of 28 bits on it (to_limbs).
//     Bits below the grid are jammed into the last one (it is set when any is lost): unlike
//     truncation, and unlike rounding halves away, that has no bias, which would drift the
//     conserved mass linearly in time instead of as a random walk.
//  2. s = sum g_i is exact on the grid; r g_i + a_i s + b_i s^2 are sums of limb products
//     (32 x 32 -> 64-bit multiply-adds), on a grid of 2^(e - 1079).  The products of two low
//     limbs are left out; their mean, where it is not zero, is added (the sign of g_i with r).
//  3. g_0 takes s minus the others, in integers: the collision keeps mass to the conversions.
//  4. The hardware's conversion (64-bit integer to FP64, round to nearest even, on the idle
//     FP64 pipe) rounds each result once.
// Each result is within a few units of 2^(e - 1079) and half an ulp of the exact value,
// where the FP64 form rounds three (g_0: twelve) times; lattices advanced 1500 to 20000
// steps end 0.2 to 0.65 times as far from a long double run as with FP64 arithmetic (over
// spacings 0.0245-0.6, time steps 1e-7 to 1e-3, tau 1-3, means 0 and 2).
// About 370 instructions per site instead of 29 FP64 ones: the plain kernel on the
// 4096-lattice ensemble went from 1.90e10 to 3.5e10 site-updates/s.  What bounds the many-step
// kernel (4.5e10) now is the integer pipe (ALU 55 % busy) and the conversions (FP64 pipe 56 %).
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
// with -2^27 <= l < 2^27 (fix_coef): r and a_p = a_{+p} = a_{-p} at 2^57 (a_p with 14 more
// bits in ae), b_p = b_{+p} = -b_{-p} at 2^kb, kb the largest with |b_p| 2^kb < 2^52.
struct FixCoef {
  int32_t rh, rl, ah[3], al[3], bh[3], bl[3];
  int16_t ae[3];
  int16_t z0;  // kb - 57 + 1022; 0: out of range, every site of the run takes FP64 arithmetic
};

namespace fix64 {

constexpr int kLimb = 28;             // bits of a low limb
constexpr int kHalf = kLimb / 2;
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
LBKS_HD int64_t mul(int32_t a, int32_t b) { return (int64_t)a * b; }
LBKS_HD int64_t mad(int32_t a, int32_t b, int64_t c) { return (int64_t)a * b + c; }

LBKS_HD uint32_t hi32(uint64_t x) { return (uint32_t)(x >> 32); }

// A value on the site's grid: |g| <= 2^(e - 1022), as h 2^28 + l in units of 2^(e - 1078)
// (both limbs carry the sign sg), a lost bit jammed into l.
LBKS_HD void to_limbs(uint64_t bits, uint32_t e, int32_t& h, int32_t& l, int32_t& sg) {
  const uint32_t hi = hi32(bits), lo = (uint32_t)bits, mag = hi & 0x7fffffffu;
  const uint32_t ei = mag >> 20;
  const uint64_t p = (bits << 11) | ((uint64_t)0x80000000u << 32);   // mantissa, leading bit at 63
  // the bits below the grid: of the low word alone down to 35 binades, then of all of the
  // mantissa, and from 56 on the leading one too, which every value but zero has
  const uint32_t n = e - ei;
  uint32_t rest = shl32(lo, 35u - n);
  if (n > 35u) rest = n > 55u ? mag : lo | shl32(hi, 67u - n);
  sg = ((int32_t)hi >> 31) | 1;
  h = (int32_t)shr32(hi32(p), (e + 4u) - ei) * sg;
  l = (int32_t)(((uint32_t)shr64(p, (e + 8u) - ei) & (uint32_t)kMask) | (rest < 1u ? rest : 1u)) * sg;
}

// Y != 0 in units of 2^(e - 1079) rounded to the nearest FP64 (ties to even) by the
// conversion unit; adj = (e - 1079) 2^20 moves the exponent.  low: the smallest high word
// of the converted values (0 for Y = 0).
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
// then meaningless): all values zero, tiny, infinite or NaN, |s| beyond about 2^-5 / b, a
// result of exactly zero, or a run whose coefficients are (FixCoef::z0).
template <int Q>
LBKS_HD bool fix_collide(const uint64_t (&g)[Q], uint64_t (&out)[Q], const FixCoef& k) {
  using namespace fix64;
  constexpr int P = (Q - 1) / 2;
  uint32_t top = hi32(g[0]) & 0x7fffffffu;
  LBKS_UNROLL
  for (int i = 1; i < Q; ++i) {
    const uint32_t v = hi32(g[i]) & 0x7fffffffu;
    top = v > top ? v : top;
  }
  const uint32_t e = top >> 20;
  const uint32_t zn = (uint32_t)k.z0 - e;  // shift of s^2; negative for z0 = 0 (and NaN, infinities)
  bool bad = e < 64u || (int32_t)zn < 0;
  int32_t h[Q], l[Q], sg[Q];
  const int32_t rhalf = k.rl >> 1;
  LBKS_UNROLL
  for (int i = 0; i < Q; ++i) to_limbs(g[i], e, h[i], l[i], sg[i]);
  int32_t sh = h[0], sl = l[0];
  LBKS_UNROLL
  for (int i = 1; i < Q; ++i) { sh += h[i]; sl += l[i]; }
  // (the low limb balanced: s^2 without its low limb's square is then never negative, as it was
  // for a small negative s, the sum of populations that cancel)
  sl += 1 << (kLimb - 1);
  sh += sl >> kLimb;
  sl = (sl & kMask) - (1 << (kLimb - 1));
  // s^2 on the grid that makes b_p s^2 come out on the results', its low limb balanced
  const uint64_t z = shr64((uint64_t)(mul(sh, sh) + (mul(sh, sl) >> (kLimb - 1))), zn);
  const uint64_t zr = z + (1u << (kLimb - 1));
  const int32_t zh = (int32_t)(zr >> kLimb), zl = (int32_t)((uint32_t)zr & (uint32_t)kMask) - (1 << (kLimb - 1));
  bad = bad || (uint32_t)(z >> 58) != 0u;
  const int32_t nh = -zh, nl = -zl;
  int64_t y0 = mad(sh, 1 << (kLimb + 1), (int64_t)(2 * (int64_t)sl));
  const uint32_t adj = (e - 1079u) << 20;
  uint32_t low = 0xffffffffu;
  LBKS_UNROLL
  for (int p = 0; p < P; ++p) {
    const int64_t th = mul(sh, k.ah[p]);
    const int64_t tl = mad(sl, k.ah[p], mad(sh, k.al[p], mad(sh >> kHalf, k.ae[p], 1 << (kLimb - 1))));
  LBKS_UNROLL
    for (int m = 0; m < 2; ++m) {
      const int i = 2 * p + 1 + m;
      const int32_t wh = m ? nh : zh, wl = m ? nl : zl;
      const int64_t ch = mad(h[i], k.rh, mad(wh, k.bh[p], th));
      const int64_t cl = mad(sg[i], rhalf, mad(h[i], k.rl, mad(l[i], k.rh, mad(wl, k.bh[p], mad(wh, k.bl[p], tl)))));
      const int64_t y = ch + (cl >> kLimb);
      out[i] = to_fp64(y, adj, low);
      y0 -= y;
    }
  }
  out[0] = to_fp64(y0, adj, low);
  return !(bad || low == 0u);
}

// The limbs of a run's coefficients (r, a_i, b_i as in RunDesc, i in speed order).
LBKS_HD void fix_limbs(double v, double scale, int32_t& h, int32_t& l) {
#if defined(__CUDA_ARCH__)
  const int64_t q = __double2ll_rn(v * scale);
#else
  const int64_t q = (int64_t)__builtin_nearbyint(v * scale);
#endif
  h = (int32_t)((q + (1 << (fix64::kLimb - 1))) >> fix64::kLimb);
  l = (int32_t)(q - ((int64_t)h << fix64::kLimb));
}

LBKS_HD FixCoef fix_coef(int Q, double r, double rhobar, const double* a, const double* b) {
  FixCoef k{};
  const int P = (Q - 1) / 2;
  double asum = 0.0, bmax = 0.0;
  bool pairs = true;
  for (int p = 0; p < P; ++p) {
    const double x = a[2 * p + 1], y = b[2 * p + 1];
    pairs = pairs && x == a[2 * p + 2] && y == -b[2 * p + 2];
    asum += 2.0 * (x < 0.0 ? -x : x);
    const double ay = y < 0.0 ? -y : y;
    bmax = ay > bmax ? ay : bmax;
  }
  // Limits that keep every sum below 64 bits: |s| < 2^58.8, 1 + sum |a_i| <= 8 (NaNs fail)
  if (!(pairs && rhobar == 0.0 && r >= 0.0 && r <= 1.0 && asum <= 7.0 && bmax >= 0x1p-60 && bmax <= 0x1p3)) return k;
  int kb = 48;
  double sb = 0x1p48;
  while (2.0 * sb * bmax < 0x1p52) { sb *= 2.0; ++kb; }
  fix_limbs(r, 0x1p57, k.rh, k.rl);
  for (int p = 0; p < P; ++p) {
    fix_limbs(a[2 * p + 1], 0x1p57, k.ah[p], k.al[p]);
    int32_t x, y;  // (the difference is exact)
    fix_limbs(a[2 * p + 1] - ((double)k.ah[p] * 0x1p28 + (double)k.al[p]) * 0x1p-57, 0x1p71, x, y);
    k.ae[p] = (int16_t)y;
    fix_limbs(b[2 * p + 1], sb, k.bh[p], k.bl[p]);
  }
  k.z0 = (int16_t)(kb - 57 + 1022);
  return k;
}

}  // namespace lbks
