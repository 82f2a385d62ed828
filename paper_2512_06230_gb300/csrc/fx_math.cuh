// Exponential, logarithm, sine and cosine in 64-bit integer arithmetic, for
// FP64 callers.  An SM issues an FP64 instruction every 16 cycles for a warp
// and an integer one on each of its four schedulers every cycle or two, so
// these cost a fraction of the FP64 library functions; each result is off by
// no more than theirs (about half a unit in the last place of the result, the
// library's being one; tests/test_fx_*.py check them against extended and
// 70-digit arithmetic).  The series are Taylor's, the tables come from the
// series at compile time.
#pragma once
#include <stdint.h>

#include <cmath>
#include <cstring>

#if defined(__CUDACC__)
#define FX_FN __host__ __device__ __forceinline__
#else
#define FX_FN inline
#endif

namespace glmb {
namespace fx {

using u64 = unsigned long long;
using u128 = unsigned __int128;

FX_FN u64 mulhi(u64 a, u64 b) {
#if defined(__CUDA_ARCH__)
  return __umul64hi(a, b);
#else
  return (u64)(((u128)a * b) >> 64);
#endif
}
FX_FN long long mulhi_s(long long a, long long b) {
#if defined(__CUDA_ARCH__)
  return __mul64hi(a, b);
#else
  return (long long)(((__int128)a * b) >> 64);
#endif
}
FX_FN int clz(u64 v) {
#if defined(__CUDA_ARCH__)
  return __clzll((long long)v);
#else
  return v ? __builtin_clzll(v) : 64;
#endif
}
FX_FN double from_bits(u64 b) {
#if defined(__CUDA_ARCH__)
  return __longlong_as_double((long long)b);
#else
  double d;
  std::memcpy(&d, &b, 8);
  return d;
#endif
}
FX_FN u64 to_bits(double d) {
#if defined(__CUDA_ARCH__)
  return (u64)__double_as_longlong(d);
#else
  u64 b;
  std::memcpy(&b, &d, 8);
  return b;
#endif
}

// v 2^e as a double, rounded to nearest (v > 0 with a normal result, or 0)
FX_FN double to_double(u64 v, int e) {
  if (v == 0ull) return 0.0;
  const int lz = clz(v);
  const u64 m = v << lz;
  return from_bits(((u64)(1085 - lz + e) << 52) + (m >> 11) + ((m >> 10) & 1ull));
}

// a value v 2^e still in fixed point
struct Val {
  u64 v;
  int e;
};
FX_FN double to_double(Val x) { return to_double(x.v, x.e); }

// ---- tables ----
// 2^(-j/64) 2^63 and -ln(k_j / 1024) 2^59, k_j = round(1024 / (1 + (j + 1/2) / 128)),
// from exp's and atanh's series with 100-bit fractions
struct Tables {
  u64 exp2[64];
  u64 nlog[128];
  uint16_t inv[128];
  constexpr Tables() : exp2{}, nlog{}, inv{} {
    constexpr u128 one = (u128)1 << 100;
    constexpr u128 ln2 = ((u128)0xB17217F7Dull << 64) | 0x1CF79ABC9E3B3980ull;   // ln(2) 2^100
    for (int j = 0; j < 64; ++j) {
      const u128 x = (ln2 * (u128)j) >> 6;   // j ln(2) / 64
      // exp(-x) by Horner's rule, 1 - x (1 - x/2 (1 - x/3 (...)))
      u128 s = one;
      for (int k = 34; k >= 1; --k) {
        // x s / k with 100-bit fractions: the halves of s separately
        const u128 sh = s >> 50, sl = s & (((u128)1 << 50) - 1);
        const u128 xs = x >> 26;   // 74 fraction bits are left of x
        s = one - (((xs * sh) >> 24) + ((xs * sl) >> 74)) / (u128)k;
      }
      exp2[j] = (u64)((s + ((u128)1 << 36)) >> 37);
    }
    for (int j = 0; j < 128; ++j) {
      const int k = (1024 * 256 + (257 + 2 * j) / 2) / (257 + 2 * j);
      inv[j] = (uint16_t)k;
      // -ln(k / 1024) = 2 atanh(y), y = (1024 - k) / (1024 + k)
      const u128 n = (u128)(1024 - k), d = (u128)(1024 + k);
      u128 term = one * n / d, sum = 0;
      for (int i = 1; term != 0 && i < 200; i += 2) {
        sum += term / (u128)i;
        term = term * n / d * n / d;
      }
      nlog[j] = (u64)((2 * sum + ((u128)1 << 40)) >> 41);
    }
  }
};

// exp(-r 2^-64) 2^63 for r 2^-64 < 0.022, by Taylor's series
FX_FN u64 exp_poly(u64 r) {
  // 1 - r (1 - r/2 (1 - r/3 (...))), the inner terms in 32 bits
  const uint32_t rh = (uint32_t)(r >> 32);
  uint32_t q = 35791394u - (uint32_t)(((u64)rh * 5965232u) >> 32);     // (1/120 - r/720) 2^32
  q = 178956971u - (uint32_t)(((u64)rh * q) >> 32);
  u64 p = 0x1555555555555555ull - mulhi(r, (u64)q << 31);              // (1/6 - ...) 2^63
  p = 0x4000000000000000ull - mulhi(r, p);
  p = 0x8000000000000000ull - mulhi(r, p);
  return 0x8000000000000000ull - mulhi(r, p);
}

// ---- exp(-x), x >= 0 and not -0 (0 from 708 on; NaN for NaN) ----
// (exp_weight below goes on to the last subnormal)
// x = n ln(2) / 64 + r: a table entry times the polynomial of exp(-r).
FX_FN double exp_neg(double x, const u64* exp2) {
  const u64 b = to_bits(x);
  if (b >= 0x4086200000000000ull) return b > 0x7FF0000000000000ull ? x : 0.0;   // 708 and beyond; NaN
  const int e = (int)(b >> 52) - 1075;                        // x = m 2^e (x >= 0)
  const u64 m = (b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
  // X = x 2^53, rounded
  const int sh = e + 53;
  const u64 X = sh >= 0 ? m << sh : sh < -54 ? 0ull : (m + (1ull << (-sh - 1))) >> -sh;
  // n <= x 64 / ln 2, short of it by less than 2
  const uint32_t n = (uint32_t)(((u64)(uint32_t)(X >> 32) * 0xB8AA3B29u) >> 46);
  // r 2^64 (the integer part of x cancels modulo 2^64)
  const u64 r = (X << 11) - (u64)n * 0x2C5C85FDF473DE6ull - (((u64)n * 0xAF278ECEull) >> 32);
  const u64 t = mulhi(exp_poly(r), exp2[n & 63u]);                     // 2^62
  return to_double(t, -62 - (int)(n >> 6));
}

// exp(l) of a log-weight difference, l <= 0 but for rounding; the library's
// function above 0 and where the result is below the normal range or near it
// (-708 down to -746, from where it is 0)
FX_FN double exp_weight(double l, const u64* exp2) {
  const u64 b = to_bits(l);
  if ((b << 1) == 0ull) return 1.0;
  if (b >> 63) {
    if (b < 0xC086200000000000ull) return exp_neg(-l, exp2);
    if (b >= 0xC087500000000000ull && b <= 0xFFF0000000000000ull) return 0.0;
  }
  return exp(l);
}

// ---- exp(-d 2^-32), d >= 0: sums of many such values beside a large one ----
// d log2(e) = i + j/64 + r / ln 2: the table's 2^(-j/64) times the polynomial
// of exp(-r).  t 2^(-62 - i), t in [2^61, 2^62], is the value to 2^-54 of it.
struct ExpParts {
  u64 t;
  int i;
};
FX_FN ExpParts exp_parts(u64 d, const u64* exp2) {                     // d < 2^39
  const u64 y = mulhi(d << 25, 0x5C551D94AE0BF85Eull);                 // d log2(e) 2^(55 - 32)
  const u64 r = mulhi((y & 0x1FFFFFFFFFFFFull) << 9, 0xB17217F7D1CF79ACull);
  return ExpParts{mulhi(exp_poly(r), exp2[(y >> 49) & 63u]), (int)(y >> 55)};
}
// Up to 31 values summed in units of 2^-90: of 2^30 values beside one of 1 the
// sum is off by 2^-60 (0 from d = 63 2^32 on, where the value is below 2^-90).
struct ExpSum {
  u64 hi = 0ull, lo = 0ull;                                            // 2^-58 and 2^-90 units (lo: carries above bit 32)
  FX_FN void add(u64 d, const u64* exp2) {
    if (d >= (63ull << 32)) return;
    const ExpParts e = exp_parts(d, exp2);                             // 0 <= i <= 90
    if (e.i < 60) {
      hi += e.t >> (4 + e.i);
      lo += (e.t << (60 - e.i)) >> 32;
    } else {
      lo += (e.t >> (e.i - 60)) >> 32;
    }
  }
  FX_FN bool any() const { return (hi | lo) != 0ull; }
  FX_FN double value() const {
    const u64 h = hi + (lo >> 32), l = lo << 32;
    if (h == 0ull) return to_double(l >> 32, -90);
    const int lz = clz(h);
    return to_double((h << lz) | ((l >> 1) >> (63 - lz)), -58 - lz);
  }
};
// one value, rounded (d < 2^39, beyond it 0: the value is below 2^-184)
FX_FN double exp_fixed(u64 d, const u64* exp2) {
  if (d >> 39) return 0.0;
  const ExpParts e = exp_parts(d, exp2);
  return to_double(e.t, -62 - e.i);
}

// ---- -2 ln((2 w + 1) / 2^33) ----
FX_FN Val neg2_log_unit(uint32_t w, const u64* nlog, const uint16_t* inv) {
  const u64 a = 2ull * w + 1ull;
  const u64 dl = (1ull << 33) - a;
  if (dl < (1ull << 26)) {
    // near 1: d (1 + d/2 + d^2/3 + ...), d = dl 2^-33 < 2^-7
    const u64 d = dl << 31;
    u64 q = 0x071C71C71C71C71Cull;                                     // 1/9 2^62
    q = 0x0800000000000000ull + mulhi(d, q);
    q = 0x0924924924924925ull + mulhi(d, q);
    q = 0x0AAAAAAAAAAAAAABull + mulhi(d, q);
    q = 0x0CCCCCCCCCCCCCCDull + mulhi(d, q);
    q = 0x1000000000000000ull + mulhi(d, q);
    q = 0x1555555555555555ull + mulhi(d, q);
    q = 0x2000000000000000ull + mulhi(d, q);
    q = 0x4000000000000000ull + mulhi(d, q);
    const int ln = clz(dl);
    return Val{mulhi(dl << ln, q), 3 - ln - 33};
  }
  const int lz = clz(a);
  const u64 mm = (a << lz) >> 31;                                      // [1, 2) 2^32, exact
  const int j = (int)(mm >> 25) & 127;
  // r = m' k / 1024 - 1, |r| < 2^-7.6, exact; r 2^64
  const long long r = (long long)((mm * inv[j] - (1ull << 42)) << 22);
  long long p = 0x0924924924924925ll;                                  // 1/7 2^62
  p = 0x0AAAAAAAAAAAAAABll - mulhi_s(r, p);
  p = 0x0CCCCCCCCCCCCCCDll - mulhi_s(r, p);
  p = 0x1000000000000000ll - mulhi_s(r, p);
  p = 0x1555555555555555ll - mulhi_s(r, p);
  p = 0x2000000000000000ll - mulhi_s(r, p);
  p = 0x4000000000000000ll - mulhi_s(r, p);
  const long long l1 = mulhi_s(r, p);                                  // ln(1 + r) 2^62
  // E ln 2 + ln(k / 1024) - ln(1 + r), 2^59
  const u64 E = (u64)(lz - 30);
  const u64 L = E * 0x058B90BFBE8E7BCDull + ((E * 0x5E4F1D9Cull) >> 32) - nlog[j] - (u64)((l1 + 4) >> 3);
  return Val{L, -58};
}

// ---- sine and cosine of (octant + t / 2^64) / 8 of a turn, 0 <= t < 2^64 ----
// both polynomials in q = (t / 2^64)^2, x = (pi / 4) t / 2^64
FX_FN u64 cos_oct(u64 q) {                                             // cos x 2^63
  u64 p = 0x13ull;
  p = 0x2419ull - mulhi(q, p);
  p = 0x36DC4Aull - mulhi(q, p);
  p = 0x3F3A7147ull - mulhi(q, p);
  p = 0x34DA3E5441ull - mulhi(q, p);
  p = 0x1E1F506891BBull - mulhi(q, p);
  p = 0xAAE9E3F1E5FFDull - mulhi(q, p);
  p = 0x20783E1036B5876ull - mulhi(q, p);
  p = 0x277A79937C8BBCB5ull - mulhi(q, p);
  return 0x8000000000000000ull - mulhi(q, p);
}
FX_FN u64 sin_oct(u64 t, u64 q) {                                      // sin x 2^63
  u64 p = 0x1ABull;
  p = 0x2DF5Bull - mulhi(q, p);
  p = 0x3D1E86Aull - mulhi(q, p);
  p = 0x3C60E9FBDull - mulhi(q, p);
  p = 0x2A0F0690FDDull - mulhi(q, p);
  p = 0x132D2CCE62BD8ull - mulhi(q, p);
  p = 0x519AF19DD6AB87ull - mulhi(q, p);
  p = 0x0A55DE7312DF295Full - mulhi(q, p);
  p = 0x6487ED5110B4611Aull - mulhi(q, p);
  return mulhi(t, p);
}

// square root of x > 0, to about 2^-58 of its value: a 22-bit reciprocal root,
// one correction of second order
FX_FN Val root(Val x) {
  const int lz = clz(x.v);
  u64 M = x.v << lz;                                                   // x = M 2^E
  int E = x.e - lz;
  if (E & 1) {
    M >>= 1;
    ++E;
  }
  const float xf = (float)(uint32_t)(M >> 32) * 9.313225746154785e-10f;   // M 2^-62, in [1, 4)
#if defined(__CUDA_ARCH__)
  const float y = rsqrtf(xf);
#else
  const float y = 1.0f / std::sqrt(xf);
#endif
  const uint32_t Y = (uint32_t)(y * 2147483648.0f);                    // 1 / sqrt(x) 2^31
  // r = 1 - x y^2 (2^-60 units); sqrt(x) = x y (1 + r/2 + 3 r^2 / 8 + ...)
  const long long r = (long long)((1ull << 60) - mulhi(M, (u64)Y * Y));
  const long long rh = r >> 20;
  const long long c = (r >> 1) + ((3 * rh * rh) >> 23);
  const u64 s0 = mulhi(M, (u64)Y << 32);                               // x y 2^61
  return Val{s0 + (u64)mulhi_s((long long)s0, c << 4), E / 2 - 30};
}

// cos(2 pi (2 w + 1) / 2^33), its magnitude
FX_FN Val cos_turn(uint32_t w, bool& neg) {
  const u64 a = 2ull * w + 1ull;
  const uint32_t oct = (uint32_t)(a >> 30);
  uint32_t t30 = (uint32_t)a & 0x3FFFFFFFu;                            // odd
  if (oct & 1u) t30 = 0x40000000u - t30;
  const u64 q = ((u64)t30 * t30) << 4;
  neg = oct >= 2u && oct < 6u;
  if (((oct + 1u) & 2u) == 0u) return Val{cos_oct(q), -63};
  // octants 1, 2, 5, 6: t30 times the sine's polynomial, normalised, for
  // relative accuracy near 0 too
  const int ln = clz(t30);
  return Val{sin_oct((u64)t30 << ln, q), 1 - ln - 30};
}

// A standard normal of two words (Box and Muller's cosine branch):
// sqrt(-2 ln u0) cos(2 pi u1), u = (word + 1/2) / 2^32, rounded once.
FX_FN double normal(uint32_t w0, uint32_t w1, const u64* nlog, const uint16_t* inv) {
  bool neg;
  const Val s = root(neg2_log_unit(w0, nlog, inv)), c = cos_turn(w1, neg);
  const double n = to_double(mulhi(s.v, c.v), s.e + c.e + 64);
  return neg ? -n : n;
}

// A fraction of a turn, (hi 2^64 + lo) 2^-128.
struct Turn {
  u64 hi, lo;
};
FX_FN Turn operator+(Turn a, Turn b) {
  const u64 lo = a.lo + b.lo;
  return Turn{a.hi + b.hi + (lo < a.lo ? 1ull : 0ull), lo};
}

// 0, or a magnitude from 2^-60 up to below `limit`: what the functions below
// take without losing more than 2^-57 of the result (a smaller angle would
// have its own bits below 2^-128 of a turn)
FX_FN bool in_turn_range(double x, double limit) {
  const u64 b = to_bits(x) & 0x7FFFFFFFFFFFFFFFull;
  return b == 0ull || b - 0x3C30000000000000ull < to_bits(limit) - 0x3C30000000000000ull;
}

// x / (2 pi) modulo 1, x in range (below 2^30): the significand times 192 bits
// of 1 / (2 pi), so that the distance from a zero of the sine or the cosine,
// however small, has its full precision too
FX_FN Turn turn(double x) {
  const u64 b = to_bits(x);
  const int E = (int)((b >> 52) & 0x7FFull) - 1023;
  const u64 M = ((b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull) << 11;   // |x| = M 2^(E - 63)
  constexpr u64 I2 = 0x28BE60DB9391054Aull, I1 = 0x7F09D5F47D4D3770ull, I0 = 0x36D8A5664F10E410ull;
  // M I, from the units down: w2 (the integer part), w1, w0 (2^-128)
  u64 w0 = M * I1, w1 = M * I2, w2 = mulhi(M, I2);
  const u64 c0 = mulhi(M, I0), c1 = mulhi(M, I1);
  w0 += c0;
  const u64 k0 = w0 < c0 ? 1ull : 0ull;
  w1 += c1;
  w2 += w1 < c1 ? 1ull : 0ull;
  w1 += k0;
  w2 += w1 < k0 ? 1ull : 0ull;
  // times 2^(E + 1) (b == 0: nothing, E = -1023)
  const int sh = E + 1;
  Turn f;
  if (sh >= 0) {
    f.hi = (w2 << sh) | ((w1 >> 1) >> (63 - sh));
    f.lo = (w1 << sh) | ((w0 >> 1) >> (63 - sh));
  } else if (sh > -64) {
    f.hi = w2 >> -sh;
    f.lo = (w2 << (64 + sh)) | (w1 >> -sh);
  } else {
    f.hi = f.lo = 0ull;
  }
  if (b >> 63) {
    f.lo = 0ull - f.lo;
    f.hi = 0ull - f.hi - (f.lo != 0ull ? 1ull : 0ull);
  }
  return f;
}
// sine and cosine of a fraction of a turn, each to 2^-57 of itself beside its
// rounding
FX_FN void sincos_turn(Turn f, double& s, double& c) {
  const uint32_t oct = (uint32_t)(f.hi >> 61);
  u64 t1 = (f.hi << 3) | (f.lo >> 61), t0 = f.lo << 3;                    // (t1 2^64 + t0) 2^-128 of an octant
  if (oct & 1u) {
    t1 = ~t1;                                                             // 1 - t to 2^-128
    t0 = ~t0;
  }
  const u64 q = mulhi(t1, t1);
  // the sine's polynomial times t, normalised: the zero it has at t = 0 is the
  // sine's own or, in the swapped octants, the cosine's
  int e = -63;
  if (t1 == 0ull) {
    t1 = t0;
    t0 = 0ull;
    e = -127;
  }
  const int lz = clz(t1) & 63;                                            // (t = 0 stays 0)
  const u64 tn = (t1 << lz) | ((t0 >> 1) >> (63 - lz));
  const double vs = to_double(sin_oct(tn, q), e - lz), vc = to_double(cos_oct(q), -63);
  const bool swap = ((oct + 1u) & 2u) != 0u;
  const double as = swap ? vc : vs, ac = swap ? vs : vc;
  s = oct >= 4u ? -as : as;
  c = (oct >= 2u && oct < 6u) ? -ac : ac;
}

// sin(h) / h, |h| < 1/2 (checked by the caller)
FX_FN double sinc(double h) {
  const u64 b = to_bits(h) & 0x7FFFFFFFFFFFFFFFull;
  const int sh = 1022 - (int)(b >> 52);                                   // |h| = M 2^-(sh + 64)
  const u64 M = ((b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull) << 11;
  const u64 x = sh < 64 ? M >> sh : 0ull;
  const u64 q = mulhi(x, x);
  u64 p = 0x654Bull;                                                      // 1/17! 2^63
  p = 0x6B9FD0ull - mulhi(q, p);
  p = 0x5849184Full - mulhi(q, p);
  p = 0x35CC8ACFEBull - mulhi(q, p);
  p = 0x171DE3A556C7ull - mulhi(q, p);
  p = 0x6806806806807ull - mulhi(q, p);
  p = 0x111111111111111ull - mulhi(q, p);
  p = 0x1555555555555555ull - mulhi(q, p);
  return to_double(0x8000000000000000ull - mulhi(q, p), -63);
}

}  // namespace fx
}  // namespace glmb
