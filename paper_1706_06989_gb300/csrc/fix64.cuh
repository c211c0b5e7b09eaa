// fix64.cuh -- the FP64 near field's arithmetic in integers.
//
// GB300 retires 1.7 to 2 FP64 operations per clock and SM, but 32 32 x 32 ->
// 64-bit integer products and 64 shifts or additions (measured), so a sum that
// is bound by the FP64 pipe runs faster in fixed point, and no less exactly: on
// systems of every kind tested the rms error is 0.15 to 0.5 of that of FP64
// arithmetic.  One ordered body pair (target i, source j) takes about 145 integer
// instructions, 36 of them products, and no FP64 one.
//
// Formats
//   positions  96-bit two's complement, in units of 2^(Eext - 95) where
//              2^Eext bounds the extent of the system's cube, kept modulo
//              2^96: only differences are used, and they fit.  A coordinate
//              keeps all of its 53 bits unless it lies within 2^-43 of the
//              extent from zero.
//   window     for a batch of source bodies, differences are bounded by
//              2^57 units of 2^gd; positions relative to a common origin are
//              rounded to that grid and split as v = H 2^29 + L, 0 <= L < 2^29.
//   r^2        the integer S2 2^58 + S1 2^30 + S0 of the digits' products.
//   r^-3       a 64-bit mantissa from a hardware seed of r^-1 (about 2^-22),
//              one step in 32-bit integers (2^-29), one in 64-bit ones: the
//              relative error is below 2^-55.
//   sums       three accumulators per component in a unit chosen before the
//              first term: a sum rounds nothing but its terms, to 2^-79 of
//              the largest factor the unit allows.
// A close pair takes a window of its own from the 96-bit positions
// (close_digits): closer than 2^-5 of the window when the window rounds a
// position (coordinates within 2^-4 of the window from zero; a difference there is
// good to 2^-52 of itself), else closer than 2^-10, the least the digits'
// normalisation takes.  Softened pairs closer than 2^-5, by r^2 without eps^2, are
// left to FP64: their terms m d / (r^2 + eps^2)^(3/2) shrink with d, and with it the
// bits that d's digits and the sums' unit leave them.
#pragma once
#include <math.h>
#include <stdint.h>

#ifdef __CUDACC__
#define AMFMM_HD __host__ __device__ __forceinline__
#else
#define AMFMM_HD static inline
#endif

namespace amfmm {
namespace fix {

constexpr int kDig = 29;  // bits of a digit
constexpr uint32_t kDigMask = (1u << kDig) - 1;
constexpr int kWin = 57;  // |difference| <= 2^kWin
// r^2 / 2^58, high word, below which a pair is close: 2^46 and 2^36 (signed:
// hi is -1 for the closest pairs, whose rem makes up for it)
constexpr int32_t kCloseRounded = 1 << (46 - 32), kCloseExact = 1 << (36 - 32);
AMFMM_HD bool is_close(int64_t hi, int32_t bound) { return static_cast<int32_t>(hi >> 32) < bound; }
constexpr int kFieldUp = 26;   // fraction bits a factor keeps below its mantissa
constexpr int kMaxTerms = 32;  // terms before the carries are propagated (a term adds below 2^58 to a1, 2^26 to a0)

AMFMM_HD int clz32(uint32_t v) {
#ifdef __CUDA_ARCH__
  return __clz(static_cast<int>(v));
#else
  return v ? __builtin_clz(v) : 32;
#endif
}
// low word of (hi:lo) >> s, 0 <= s < 32
AMFMM_HD uint32_t funnel_r(uint32_t lo, uint32_t hi, int s) {
#ifdef __CUDA_ARCH__
  return __funnelshift_r(lo, hi, s);
#else
  return static_cast<uint32_t>(((static_cast<uint64_t>(hi) << 32) | lo) >> (s & 31));
#endif
}
// A reciprocal square root good to about 22 bits.  The host form (tests)
// takes a relative perturbation so that a test covers any such seed.
#ifndef __CUDA_ARCH__
extern float seed_error;
#endif
AMFMM_HD float rsqrt_seed(float v) {
#ifdef __CUDA_ARCH__
  return rsqrtf(v);
#else
  return static_cast<float>(1.0 / __builtin_sqrt(static_cast<double>(v)) * (1.0 + seed_error));
#endif
}
AMFMM_HD uint32_t to_u32(float v) {
#ifdef __CUDA_ARCH__
  return __float2uint_rn(v);
#else
  return static_cast<uint32_t>(v);
#endif
}
// 32 x 32 -> 64 bits, and the high word.  With the wide products as C expressions,
// int64_t(a) * b, the near field took 9.40 ms instead of 7.39 at N = 1,048,576, with
// the high words from wide products instead of __mulhi 7.39 instead of 7.31 (softened,
// N = 262,144: 2.19 instead of 2.20).
AMFMM_HD int64_t mul_wide(int32_t a, int32_t b) {
#ifdef __CUDA_ARCH__
  int64_t d;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
  return d;
#else
  return static_cast<int64_t>(a) * b;
#endif
}
AMFMM_HD uint64_t mul_wide_u(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
  uint64_t d;
  asm("mul.wide.u32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
  return d;
#else
  return static_cast<uint64_t>(a) * b;
#endif
}
AMFMM_HD int32_t mul_hi(int32_t a, int32_t b) {
#ifdef __CUDA_ARCH__
  return __mulhi(a, b);
#else
  return static_cast<int32_t>(mul_wide(a, b) >> 32);
#endif
}
AMFMM_HD uint32_t mul_hi_u(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
  return __umulhi(a, b);
#else
  return static_cast<uint32_t>(mul_wide_u(a, b) >> 32);
#endif
}

// 64-bit shifts by 0 .. 64 and beyond: what is shifted out is zero.
AMFMM_HD uint64_t shr64(uint64_t v, unsigned s) {
#ifdef __CUDA_ARCH__
  uint64_t d;
  asm("shr.u64 %0, %1, %2;" : "=l"(d) : "l"(v), "r"(s));
  return d;
#else
  return s < 64 ? v >> s : 0;
#endif
}
AMFMM_HD uint64_t shl64(uint64_t v, unsigned s) {
#ifdef __CUDA_ARCH__
  uint64_t d;
  asm("shl.b64 %0, %1, %2;" : "=l"(d) : "l"(v), "r"(s));
  return d;
#else
  return s < 64 ? v << s : 0;
#endif
}

// ---- conversion of the inputs ------------------------------------------
struct W96 {
  uint32_t w[3];
};

// x in units of 2^g, modulo 2^96 (rounded to the nearest unit, halves up in
// magnitude, when its own last place is finer).
AMFMM_HD W96 fixed96(double x, int g) {
  union {
    double d;
    uint64_t u;
  } b;
  b.d = x;
  int e = static_cast<int>((b.u >> 52) & 0x7ff);
  uint64_t m = b.u & 0xfffffffffffffull;
  if (e) m |= 1ull << 52;
  else e = 1;
  const int sh = e - 1075 - g;
  unsigned __int128 v = 0;
  if (sh >= 0) {
    if (sh < 96) v = static_cast<unsigned __int128>(m) << sh;
  } else if (sh > -64) {
    v = (m + (1ull << (-sh - 1))) >> -sh;
  }
  if (b.u >> 63) v = ~v + 1;
  W96 r;
  r.w[0] = static_cast<uint32_t>(v);
  r.w[1] = static_cast<uint32_t>(v >> 32);
  r.w[2] = static_cast<uint32_t>(v >> 64);
  return r;
}

// m > 0 as M 2^-64 2^e with M in [2^63, 2^64)
AMFMM_HD void mantissa64(double m, uint64_t *M, int *e) {
  union {
    double d;
    uint64_t u;
  } b;
  b.d = m;
  int ex = static_cast<int>((b.u >> 52) & 0x7ff);
  uint64_t f = b.u & 0xfffffffffffffull;
  if (ex) f |= 1ull << 52;
  else ex = 1;
  int up = 11;
  while (f && !(f >> 52)) {  // subnormal
    f <<= 1;
    ++up;
  }
  *M = f << 11;
  *e = ex - 1075 - up + 64;
}

// Exponent of a cube's extent from its key scale 2^21 / extent (a factor two
// of room; 0 for a cube without extent, whose differences are all zero or
// left to FP64).
AMFMM_HD int extent_exponent(double scale) {
  union {
    double d;
    uint64_t u;
  } b;
  b.d = scale;
  const int e = static_cast<int>((b.u >> 52) & 0x7ff);
  if (e == 0 || e == 0x7ff) return 0;
  return 22 - (e - 1023);
}

AMFMM_HD W96 sub96(const W96 &a, const W96 &b) {
  const uint64_t lo = (static_cast<uint64_t>(a.w[1]) << 32 | a.w[0]) - (static_cast<uint64_t>(b.w[1]) << 32 | b.w[0]);
  const uint64_t al = static_cast<uint64_t>(a.w[1]) << 32 | a.w[0];
  W96 r;
  r.w[0] = static_cast<uint32_t>(lo);
  r.w[1] = static_cast<uint32_t>(lo >> 32);
  r.w[2] = a.w[2] - b.w[2] - (lo > al ? 1u : 0u);
  return r;
}

// |top word| of an offset, rounded so that |offset| < (mag + 1) 2^64 units
AMFMM_HD uint32_t top_mag(const W96 &o) {
  const int32_t t = static_cast<int32_t>(o.w[2]);
  return static_cast<uint32_t>(t ^ (t >> 31));
}

// Shift that brings differences of offsets, |a| < (ma + 1) 2^64 and
// |b| < (mb + 1) 2^64, to at most 2^kWin: between 9 and 39 (offsets stay below 2^94).
AMFMM_HD int window_shift(uint32_t ma, uint32_t mb) {
  const uint32_t s = ma + mb + 2;  // < 2^32: magnitudes are below 2^31
  return 64 + (32 - clz32(s)) - kWin;
}

// Offset rounded to the window's grid, as digits; true if that rounded it.
AMFMM_HD bool digits(const W96 &o, int sh, int32_t *H, int32_t *L) {
  // + half a unit
  const uint64_t half = 1ull << (sh - 1);
  const uint64_t lo = (static_cast<uint64_t>(o.w[1]) << 32 | o.w[0]) + half;
  const uint32_t w0 = static_cast<uint32_t>(lo), w1 = static_cast<uint32_t>(lo >> 32);
  const uint32_t w2 = o.w[2] + (lo < half ? 1u : 0u);
  uint32_t vl, vh;
  if (sh < 32) {
    vl = funnel_r(w0, w1, sh);
    vh = funnel_r(w1, w2, sh);
  } else {
    vl = funnel_r(w1, w2, sh - 32);
    vh = static_cast<uint32_t>(static_cast<int32_t>(w2) >> (sh - 32));
  }
  *H = static_cast<int32_t>(funnel_r(vl, vh, kDig));
  *L = static_cast<int32_t>(vl & kDigMask);
  return (((static_cast<uint64_t>(o.w[1]) << 32 | o.w[0]) << (64 - sh)) != 0);
}

// ---- the pair ----------------------------------------------------------
// Digits of a close pair's difference d = a - b at the finest window that
// holds it: the largest component lies in [2^(kWin - 1), 2^kWin).  Returns
// the window's shift, or kNoDigits when the positions agree to 2^53 units
// (2^-42 of the system's extent), where their rounding shows.
constexpr int kNoDigits = -1000;
AMFMM_HD int close_digits(const W96 a[3], const W96 b[3], int32_t H[3], int32_t L[3]) {
  __int128 d[3];
  unsigned __int128 m = 0;
  for (int c = 0; c < 3; ++c) {
    const W96 e = sub96(a[c], b[c]);
    d[c] = (static_cast<__int128>(static_cast<int32_t>(e.w[2])) << 64) |
           (static_cast<unsigned __int128>(e.w[1]) << 32 | e.w[0]);
    m |= static_cast<unsigned __int128>(d[c] < 0 ? -d[c] : d[c]);
  }
  const uint32_t m2 = static_cast<uint32_t>(m >> 64), m1 = static_cast<uint32_t>(m >> 32), m0 = static_cast<uint32_t>(m);
  const int bits = m2 ? 95 - clz32(m2) : m1 ? 63 - clz32(m1) : 31 - clz32(m0);
  if (bits < 53) return kNoDigits;
  const int sh = bits - (kWin - 1);
  for (int c = 0; c < 3; ++c) {
    const __int128 v = sh > 0 ? (d[c] + (static_cast<__int128>(1) << (sh - 1))) >> sh : d[c] << -sh;
    H[c] = static_cast<int32_t>(v >> kDig);
    L[c] = static_cast<int32_t>(static_cast<uint32_t>(v) & kDigMask);
  }
  return sh;
}

// r^2 of the digits' difference, in units of 2^58 (hi) and 2^32 (rem, the
// rest, below 2^28): S2 2^58 + S1 2^30 + S0, S0 less its low words.
AMFMM_HD void square(const int32_t dH[3], const int32_t dL[3], int64_t *hi, uint32_t *rem) {
  const int64_t S2 = (mul_wide(dH[0], dH[0]) + mul_wide(dH[1], dH[1])) + mul_wide(dH[2], dH[2]);
  const int64_t S1 = (mul_wide(dH[0], dL[0]) + mul_wide(dH[1], dL[1])) + mul_wide(dH[2], dL[2]);
  const int32_t S0 = mul_hi(dL[0], dL[0]) + mul_hi(dL[1], dL[1]) + mul_hi(dL[2], dL[2]);
  *hi = S2 + (S1 >> 28);
  *rem = ((static_cast<uint32_t>(S1) & 0xfffffffu) >> 2) + static_cast<uint32_t>(S0);
}

// Softening, for digits in units of 2^gd.  The window is that of the positions
// alone, so that a length far above the separations takes no bits from the
// differences: eps^2 = eh 2^58 + el 2^32, like r^2, in units of 2^(2 (gd + t)), t = 0
// while eps^2 fits.
struct Soft {
  int t, s2, room;  // s2 (of inv_cube) at the window's bound; 3 x what it grows by down to the closest pairs
  int64_t eh;
  uint32_t el;
};
AMFMM_HD int soft_s2(const Soft &s, int bits) {  // at r^2 = 2^bits in units of 2^(2 gd + 58)
  const int64_t v = s.eh + (bits >= 2 * s.t ? 1ll << (bits - 2 * s.t) : 0);
  return (clz32(static_cast<uint32_t>(v >> 32)) - 1) >> 1;
}
AMFMM_HD Soft soft_window(double eps2, int gd) {
  Soft s;
  const int up = ilogb(eps2) - 2 * gd - 2 * kDig - 59;  // eh stays below 2^60
  s.t = up > 0 ? (up + 1) / 2 : 0;
  const double e = scalbn(eps2, -2 * (gd + s.t) - 2 * kDig);
  s.eh = static_cast<int64_t>(e);
  s.el = static_cast<uint32_t>(scalbn(e - static_cast<double>(s.eh), 2 * kDig - 32));
  s.s2 = soft_s2(s, 56);
  s.room = 3 * (soft_s2(s, 46) - s.s2);
  return s;
}
// r^2 + eps^2 from r^2 of the digits' difference
AMFMM_HD void soften(const Soft &s, int64_t *hi, uint32_t *rem) {
  if (s.t) {  // the same for a whole batch
    const unsigned d = 2 * static_cast<unsigned>(s.t);
    const uint64_t h = static_cast<uint64_t>(*hi);
    *rem = (d < 26 ? static_cast<uint32_t>(h << (26 - d)) : static_cast<uint32_t>(shr64(h, d - 26))) & 0x3ffffffu;
    *hi = static_cast<int64_t>(shr64(h, d));
  }
  *hi += s.eh;
  *rem += s.el;
}

// r^-3 = w 2^-58 2^(-3 (60 - s2 + gd)) for r^2 = (hi 2^58 + rem 2^32) 2^(2 gd),
// hi >= 2^36; w in [2^56, 2^60).
AMFMM_HD uint64_t inv_cube(int64_t hi, uint32_t rem, int *s2out) {
  const uint32_t hh = static_cast<uint32_t>(static_cast<uint64_t>(hi) >> 32);
  const int s2 = (clz32(hh) - 1) >> 1, s = 2 * s2;
  // r^2 = Rm 2^(58 - s + 2 gd), Rm in [2^61, 2^63]; rho = Rm 2^-62, y = rho^-1/2
  const uint64_t Rm = (static_cast<uint64_t>(hi) << s) + (rem >> (26 - s));
  const uint32_t A1 = static_cast<uint32_t>(Rm >> 32), A0 = static_cast<uint32_t>(Rm);
  const uint32_t Y = to_u32(rsqrt_seed(static_cast<float>(A1)) * 35184372088832.0f);  // y 2^30
  // y1 = Y (1 + e/2), e = 1 - rho Y^2 to 2^-29.  The 9 centres the errors of
  // the truncations (A1, Y^2, the product's high word and its half), so that
  // 3/2 e1 stays below 2^31 units with a factor of two to spare.
  const uint64_t P = mul_wide_u(A1, static_cast<uint32_t>(mul_wide_u(Y, Y) >> 30));  // 2^60 (1 - e)
  const int32_t en = static_cast<int32_t>(static_cast<uint32_t>(P >> 28)) + 9;       // -e 2^32
  const uint32_t y1 = Y - static_cast<uint32_t>(mul_hi(en, static_cast<int32_t>(Y)) >> 1);
  // e1 = 1 - rho y1^2 in units of 2^-58: the product modulo 2^32
  const uint64_t Y2 = mul_wide_u(y1, y1);  // y^2 2^60
  const uint32_t B1 = static_cast<uint32_t>(Y2 >> 32), B0 = static_cast<uint32_t>(Y2);
  const int32_t Ln = static_cast<int32_t>(A1 * B1 + mul_hi_u(A1, B0) + mul_hi_u(A0, B1));  // -e1
  const uint64_t V = mul_wide_u(B1, y1) + mul_hi_u(B0, y1);                              // y^3 2^58
  const int32_t e15 = -(Ln + (Ln >> 1));                                                   // 3/2 e1
  *s2out = s2;
  return V + static_cast<uint64_t>(mul_wide(static_cast<int32_t>(static_cast<uint32_t>(V >> 29)), e15) >> 29);
}

// w M 2^-64, M = (m1:m0) in [2^63, 2^64): 2^55 .. 2^60
AMFMM_HD uint64_t times_mass(uint64_t w, uint32_t m1, uint32_t m0) {
  const uint32_t w1 = static_cast<uint32_t>(w >> 32), w0 = static_cast<uint32_t>(w);
  return mul_wide_u(w1, m1) + mul_hi_u(w1, m0) + mul_hi_u(w0, m1);
}

// ---- sums --------------------------------------------------------------
struct Acc {
  int64_t a2[3], a1[3];  // weights 2^58 and 2^29, in units of 2^(Ua + 29)
  int32_t a0[3], b0[3];  // weight 2^32: the low digits' products, their low words dropped
  int Ua;
};

AMFMM_HD void acc_clear(Acc &a) {
  for (int c = 0; c < 3; ++c) a.a2[c] = a.a1[c] = a.a0[c] = a.b0[c] = 0;
  a.Ua = 0;
}

// Propagates the carries after terms <= kMaxTerms terms, and makes room (the
// sums shifted right by 12 bits, rare) when one has grown to 2^59 in its top
// accumulator: kMaxTerms terms add below 2^61 there.  The low words that a0 and
// b0 drop are half a unit each on average; that much per term is added back.
AMFMM_HD void acc_carry(Acc &a, int terms) {
  uint32_t m = 0;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int64_t v = a.a1[c] + (static_cast<int64_t>(a.a0[c]) + a.b0[c] + terms) * 8;
    a.a0[c] = a.b0[c] = 0;
    a.a1[c] = static_cast<int64_t>(static_cast<uint32_t>(v) & kDigMask);
    a.a2[c] += v >> kDig;
    const uint32_t h = static_cast<uint32_t>(static_cast<uint64_t>(a.a2[c]) >> 32);
    m |= h ^ static_cast<uint32_t>(static_cast<int32_t>(h) >> 31);
  }
  if (m >> 27) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      a.a1[c] = static_cast<int64_t>((static_cast<uint64_t>(a.a2[c]) & 0xfffu) << (kDig - 12)) | (a.a1[c] >> 12);
      a.a2[c] >>= 12;
    }
    a.Ua += 12;
  }
}

// Digits (weights 2^58, 2^29, 1) of a factor q 2^eq in the sums' unit, where
// k = Ua + 26 - eq - gd in [0, kShiftEnd) places it; kNoTerm gives zeros.
constexpr unsigned kShiftEnd = 52;  // (the middle digit of a term is then never zero)
constexpr int kNoTerm = 128;
AMFMM_HD void factor_digits(uint64_t q, int k, int32_t d[3]) {
  const uint64_t a = shr64(q, static_cast<unsigned>(k));
  const uint32_t b = static_cast<uint32_t>(shl64(q, 64u - static_cast<unsigned>(k)) >> 32);
  const uint32_t ah = static_cast<uint32_t>(a >> 32), al = static_cast<uint32_t>(a);
  // q 2^32 >> k in 96 bits (ah:al:b); its digits from bit 6 up
  d[2] = static_cast<int32_t>(ah);
  d[1] = static_cast<int32_t>(al >> 3);
  d[0] = static_cast<int32_t>(funnel_r(b, al, 6) & kDigMask);
}

// Adds a factor's digits times the difference.
AMFMM_HD void acc_add(Acc &a, const int32_t q[3], const int32_t dH[3], const int32_t dL[3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    a.a2[c] += mul_wide(q[2], dH[c]);
    a.a1[c] += mul_wide(q[1], dH[c]) + mul_wide(q[2], dL[c]);
    a.a0[c] += mul_hi(q[0], dH[c]);
    a.b0[c] += mul_hi(q[1], dL[c]);
  }
}

// A unit for sums over sources in a window of exponent gd, em the heaviest one's
// mass exponent: at the window's bound that source gets k = 24 and fits down to
// 2^-8 of the window (closer ones: the caller's FP64 path).  A unit is kept while
// it stays within 2^kUnitSpan of the one that the sources at hand ask for (a window
// wider or narrower by 2^kWinSpan, or other masses): k is 18 to 30 then, and a
// source lighter by 2^kClassSpan still gets k < kShiftEnd.  A term rounds to
// 2^(k - 79) of itself at the window's bound (less when it is closer), so all of
// them to 2^-49 of the heaviest one's term at worst.
constexpr int kWinSpan = 3, kUnitSpan = 2 * kWinSpan, kClassSpan = 21;
AMFMM_HD int unit_guess(int gd, int em) { return 24 + em + 9 - (kFieldUp + 238 + 2 * gd); }

// Softened, a heavy source next to the row adds little, so every term keeps its own
// bits: classes span 2^kSoftClassSpan, and the unit gives the heaviest source k = 2
// at the closest.  The lightest has at most 2^(28 - 79) of its term rounded away.
constexpr int kSoftUnitSpan = 2, kSoftClassSpan = 9;
AMFMM_HD int unit_soft(int gd, int em, const Soft &s) {
  return s.room + 2 + em + 3 * (s.s2 - s.t) - (kFieldUp + 238 + 2 * gd);
}

// Constant part of k for a batch of window exponent gd: k = base - em - 3 s2
// with em the source mass's exponent (eq = em - 238 + 3 s2 - 3 gd; softened, gd + t).
AMFMM_HD int k_base(int Ua, int gd) { return Ua + kFieldUp + 238 + 2 * gd; }

}  // namespace fix
}  // namespace amfmm
