// FP64 elementary functions of the FP64 form's particle update, written for a GPU whose FP64
// pipe is its narrowest: an FP64 warp instruction holds a scheduler's pipe for 64 cycles
// whatever it does, so what counts is the number of FP64 operations.  Arguments are taken
// apart with integer operations, seeds come from the FP32 special-function unit, and tables
// shorten the series.  FP64 operations (library function on this GPU, from latencies):
// reciprocal 4 (9), square root 6 (10), quotient 5 (10), inverse cube root 8 (about 25), -2 ln u
// 10 (about 25), cos and sin of 2 pi u 14 (about 30).  None is less accurate than the library's:
// largest errors found on the device in units in the last place, over half a million arguments and
// more of the ranges met (library): reciprocal, square root and quotient 0.500 (0.500), inverse
// cube root 0.500 (0.753), -2 ln u 0.501 (0.531), cosine 1.02 (1.44), sine 1.11 (1.42).
//
// Plain C++ as well as CUDA, so that a test runs the same code on the host.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#if defined(__CUDACC__)
#define PDFX_M64 __device__ __forceinline__
#else
#define PDFX_M64 inline
#endif

namespace pdfx {
namespace m64 {

#if defined(__CUDA_ARCH__)
PDFX_M64 int64_t bits(double x) { return __double_as_longlong(x); }
PDFX_M64 double from_bits(int64_t b) { return __longlong_as_double(b); }
PDFX_M64 int32_t hi_word(double x) { return __double2hiint(x); }
PDFX_M64 uint32_t fbits(float x) { return __float_as_uint(x); }
PDFX_M64 float from_fbits(uint32_t b) { return __uint_as_float(b); }
PDFX_M64 int top_bit(uint64_t m) { return 63 - __clzll(static_cast<long long>(m)); }
PDFX_M64 float seed_rsqrt(float x) { return rsqrtf(x); }
PDFX_M64 float seed_rcp(float x) { return __fdividef(1.0f, x); }
PDFX_M64 float seed_rcbrt(float x) { return exp2f(__log2f(x) * (-1.0f / 3.0f)); }
#else
inline int64_t bits(double x) { int64_t b; std::memcpy(&b, &x, 8); return b; }
inline double from_bits(int64_t b) { double x; std::memcpy(&x, &b, 8); return x; }
inline int32_t hi_word(double x) { return static_cast<int32_t>(bits(x) >> 32); }
inline uint32_t fbits(float x) { uint32_t b; std::memcpy(&b, &x, 4); return b; }
inline float from_fbits(uint32_t b) { float x; std::memcpy(&x, &b, 4); return x; }
inline int top_bit(uint64_t m) { return 63 - __builtin_clzll(m); }
inline float seed_rsqrt(float x) { return 1.0f / std::sqrt(x); }
inline float seed_rcp(float x) { return 1.0f / x; }
inline float seed_rcbrt(float x) { return 1.0f / std::cbrt(x); }
#endif

// ---------------------------------------------------------------------------------------
// Tables, formed at compile time in pairs of doubles (about 100 bits) by recurrences.
// ---------------------------------------------------------------------------------------
struct DD {   // hi + lo
  double h, l;
};
constexpr DD dd_sum(double a, double b) {
  const double s = a + b, bb = s - a;
  return {s, (a - (s - bb)) + (b - bb)};
}
constexpr DD dd_prod(double a, double b) {   // Dekker's exact product
  const double ca = 134217729.0 * a, cb = 134217729.0 * b;
  const double ah = ca - (ca - a), al = a - ah, bh = cb - (cb - b), bl = b - bh;
  const double p = a * b;
  return {p, ((ah * bh - p) + ah * bl + al * bh) + al * bl};
}
constexpr DD dd_add(DD a, DD b) {
  const DD s = dd_sum(a.h, b.h);
  const DD t = dd_sum(a.l, b.l);
  const DD u = dd_sum(s.h, s.l + t.h);
  return dd_sum(u.h, u.l + t.l);
}
constexpr DD dd_mul(DD a, DD b) {
  const DD p = dd_prod(a.h, b.h);
  return dd_sum(p.h, p.l + (a.h * b.l + a.l * b.h));
}
constexpr DD dd_over(DD a, double n) {   // n a small integer
  const double q = a.h / n;
  const DD p = dd_prod(q, n);
  const double r = ((a.h - p.h) - p.l + a.l) / n;
  return dd_sum(q, r);
}

// A multiple of 2^-47 within 2^-47 of x, -16 < x < 80.
constexpr double head(double x) { return (x + 48.0) - 48.0; }

constexpr int kLogCells = 1024;   // cells of [1, 2) in the logarithm's table
constexpr int kTrigCells = 512;   // cells of a quarter turn

// 2^12 / f rounded to an integer, f = 1 + i / kLogCells
constexpr int log_recip(int i) { return (2 * 4096 * kLogCells / (kLogCells + i) + 1) / 2; }

struct alignas(32) Tables {
  double cs[kTrigCells + 1][4];   // cos and its rest, sin and its rest of (pi / 2) i / kTrigCells
  // 2 ln(C_i / 2^12), from i = kLogCells / 2 on 2 ln(C_i / 2^11), and 2 j ln 2, the exponent's
  // part of -2 ln u: multiples of 2^-47, whose sums are exact, and the rest
  double t[kLogCells + 1], tl[kLogCells + 1], e[34], el[34];
  uint16_t r[kLogCells + 1];   // C_i
  constexpr Tables() : cs(), t(), tl(), e(), el(), r() {
    // ln n for n = 2048 .. 4096 from ln 2048 by ln(n + 1) = ln n + 2 atanh(1 / (2 n + 1))
    DD ln2 = {0.69314718055994530942, 2.3190468138462996e-17};
    for (int j = 0; j < 34; ++j) {
      const DD v = dd_mul(ln2, DD{2.0 * j, 0.0});
      e[j] = head(v.h);
      el[j] = (v.h - e[j]) + v.l;
    }
    DD rel = {0.0, 0.0};   // ln(n / 2048)
    int i = kLogCells;     // log_recip falls as i rises
    for (int n = 2048; n <= 4096; ++n) {
      while (i >= 0 && log_recip(i) == n) {
        r[i] = static_cast<uint16_t>(n);
        const DD below = dd_add(rel, DD{-ln2.h, -ln2.l});   // ln(n / 4096)
        const DD v = i >= kLogCells / 2 ? rel : (n == 4096 ? DD{0.0, 0.0} : below);
        t[i] = head(2.0 * v.h);
        tl[i] = (2.0 * v.h - t[i]) + 2.0 * v.l;
        --i;
      }
      const double m = 2.0 * n + 1.0;
      DD z = dd_over(DD{1.0, 0.0}, m);
      const DD z2 = dd_mul(z, z);
      DD sum = {0.0, 0.0};
      for (int k = 1; k <= 9; k += 2) {
        sum = dd_add(sum, dd_over(z, k));
        z = dd_mul(z, z2);
      }
      rel = dd_add(rel, DD{2.0 * sum.h, 2.0 * sum.l});
    }
    // one cell's turn by its series, then rotations
    const DD a = dd_over(DD{1.5707963267948966192, 6.123233995736766e-17}, kTrigCells);
    DD c1 = {1.0, 0.0}, s1 = {0.0, 0.0}, term = {1.0, 0.0};
    for (int k = 1; k <= 16; ++k) {
      term = k == 1 ? a : dd_over(dd_mul(term, a), k);
      const double sg = (k / 2) % 2 ? -1.0 : 1.0;
      const DD v = {sg * term.h, sg * term.l};
      if (k % 2) s1 = dd_add(s1, v);
      else c1 = dd_add(c1, v);
    }
    DD cc = {1.0, 0.0}, ss = {0.0, 0.0};
    for (int k = 0; k <= kTrigCells / 2; ++k) {   // up to an eighth of a turn, the rest by symmetry
      cs[k][0] = cs[kTrigCells - k][2] = cc.h;
      cs[k][1] = cs[kTrigCells - k][3] = cc.l;
      cs[k][2] = cs[kTrigCells - k][0] = ss.h;
      cs[k][3] = cs[kTrigCells - k][1] = ss.l;
      const DD nc = dd_add(dd_mul(cc, c1), [](DD x) { return DD{-x.h, -x.l}; }(dd_mul(ss, s1)));
      ss = dd_add(dd_mul(ss, c1), dd_mul(cc, s1));
      cc = nc;
    }
  }
};
#if defined(__CUDACC__)
__device__ const Tables g_tables = Tables();
PDFX_M64 const Tables& tables() { return g_tables; }
#else
constexpr Tables h_tables = Tables();
inline const Tables& tables() { return h_tables; }
#endif

// A signed integer below 2^51 in magnitude as a double: one FP64 addition.
PDFX_M64 double of_int(int64_t v) { return from_bits(0x4338000000000000ll + v) - 6755399441055744.0; }

// Positive and between 2^-100 and 2^100: the FP32 seeds below hold there.
PDFX_M64 bool seedable(double x) {
  return static_cast<uint32_t>(hi_word(x) - 0x39b00000) < 0x46300000u - 0x39b00000u;
}
// The FP32 number nearest below a seedable double, and a positive normal FP32 number as a
// double, by moving bits.
PDFX_M64 float narrow(double x) {
  return from_fbits(static_cast<uint32_t>((bits(x) - (int64_t(896) << 52)) >> 29));
}
PDFX_M64 double widen(float x) { return from_bits((static_cast<int64_t>(fbits(x)) << 29) + (int64_t(896) << 52)); }

// 1 / x: Newton's step doubles the seed's bits, a second one from the exact remainder rounds.
PDFX_M64 double rcp(double x) {
  if (!seedable(x)) return 1.0 / x;
  double y = widen(seed_rcp(narrow(x)));
  y = fma(fma(-x, y, 1.0), y, y);
  return fma(fma(-x, y, 1.0), y, y);
}
// a / b: Markstein's correction (1990) of the product with 1 / b.
PDFX_M64 double quotient(double a, double b) {
  if (!seedable(a) || !seedable(b)) return a / b;
  double y = widen(seed_rcp(narrow(b)));
  y = fma(fma(-b, y, 1.0), y, y);
  const double q = a * y;
  return fma(fma(-q, b, a), y, q);
}
// sqrt(x): g near sqrt(x) and h near 1 / (2 sqrt(x)) from the seed, both with twice its bits
// after one step (r = 1/2 - g h), then g from the exact remainder x - g^2.
PDFX_M64 double root(double x) {
  if (!seedable(x)) return sqrt(x);
  const double y = widen(seed_rsqrt(narrow(x)));
  const double h0 = from_bits(bits(y) - (int64_t(1) << 52));
  const double g0 = x * y;
  const double r = fma(-g0, h0, 0.5);
  const double g = fma(g0, r, g0), h = fma(h0, r, h0);
  return fma(fma(-g, g, x), h, g);
}
// x^(-1/3) of a normal number x = m 8^k, 1 <= m < 8: the seed z of m^(-1/3), where the FP32
// logarithm's error is small, e = 1 - m z^3 with the product's rounding taken along (z^2 is
// exact), then z (1 + e / 3 + 2 e^2 / 9), and the exponent back.
PDFX_M64 double rcbrt(double x) {
  const int b = hi_word(x) >> 20;   // sign and exponent
  if (b <= 0 || b >= 0x7ff) return 1.0 / cbrt(x);
  const int k = b / 3 - 341;        // 3 k <= b - 1023 < 3 k + 3
  const double m = from_bits(bits(x) - (static_cast<int64_t>(3 * k) << 52));
  const double z = widen(seed_rcbrt(narrow(m)));
  const double z2 = z * z, p = m * z;
  const double e = fma(-fma(m, z, -p), z2, fma(-p, z2, 1.0));
  const double w = fma(fma(e, 2.0 / 9.0, 1.0 / 3.0) * e, z, z);
  return from_bits(bits(w) - (static_cast<int64_t>(k) << 52));
}

// Any FP32 number as FP64 by its bits (the conversion takes the FP64 pipe like any other FP64
// operation): the exponent is re-biased; zero keeps its sign; subnormal, infinite and NaN go
// through the conversion.
PDFX_M64 double widened(float x) {
  const uint32_t b = fbits(x), m = b & 0x7fffffffu;
  const bool normal = m - 0x00800000u < 0x7f000000u;
  if (!normal && m != 0u) return static_cast<double>(x);
  const uint32_t hi = (b & 0x80000000u) | (normal ? (m >> 3) + 0x38000000u : 0u);
  return from_bits(static_cast<int64_t>(static_cast<uint64_t>(hi) << 32 | static_cast<uint64_t>(b << 29)));
}
PDFX_M64 double widened(double x) { return x; }

// x >= 0 (a zero of either sign; false for NaN) and x < c for a positive c, on the bits.
PDFX_M64 bool nonneg(double x) {
  const uint64_t b = static_cast<uint64_t>(bits(x));
  return b <= 0x7ff0000000000000ull || b == 0x8000000000000000ull;
}
PDFX_M64 bool below_pos(double x, double c) {
  const int64_t b = bits(x);
  return b < bits(c) && static_cast<uint64_t>(b) <= 0xfff0000000000000ull;
}

// -2 ln u of u = (w + 1/2) 2^-32 = m 2^-33, m = 2 w + 1: m = f 2^p, 1 <= f < 2; f C_i / 2^12
// = 1 + r exactly (integers of 46 bits), |r| < 2^-10; the tables give the rest.  From f = 1.5
// on the logarithm is that of f / 2, so that nothing cancels as u nears 1.
PDFX_M64 double minus_two_log(uint32_t w) {
  const uint64_t m = 2 * static_cast<uint64_t>(w) + 1;
  const int p = top_bit(m);                                  // 0 .. 32
  const uint64_t F = m << (32 - p);                          // f 2^32
  const uint32_t i = (static_cast<uint32_t>(F >> 21) - (1u << 11) + 1u) >> 1;   // nearest cell, 0 .. kLogCells
  const Tables& T = tables();
  const int64_t R = static_cast<int64_t>(F * T.r[i]) - (int64_t(1) << 44);
  const double x = of_int(R);                                // r 2^44
  // -2 ln(1 + r) = -2 r + r^2 - 2/3 r^3 + 1/2 r^4 - 2/5 r^5; the first term joins the tables'
  // heads exactly (multiples of 2^-47 below 64), so that one rounding is left
  constexpr double k1 = 5.684341886080802e-14, k2 = k1 * k1;   // 2^-44, 2^-88
  double q = fma(x, -0.4 * k2 * k2 * k1, 0.5 * k2 * k2);
  q = fma(x, q, -2.0 / 3.0 * k2 * k1);
  q = fma(x, q, k2);
  const int j = 33 - p - (i >= kLogCells / 2 ? 1 : 0);
  return fma(x, -2.0 * k1, T.e[j] + T.t[i]) + fma(x * x, q, T.el[j] + T.tl[i]);
}

// (cos, sin) of 2 pi u, u = (w + 1/2) 2^-32: the quarter turn and the nearest of its cells
// from the bits, the rest delta = (pi / 2) R 2^-31, |R| <= 2^21, by its series.
PDFX_M64 void turn(uint32_t w, double& cs, double& sn) {
  const uint64_t m = 2 * static_cast<uint64_t>(w) + 1;       // u 2^33
  const uint32_t quarter = w >> 30;
  const uint32_t t = static_cast<uint32_t>(m) & 0x7fffffffu;
  const uint32_t i = (t + (1u << 21)) >> 22;                 // 0 .. kTrigCells
  const double x = of_int(static_cast<int32_t>(t - (i << 22)));
  constexpr double a = 1.5707963267948966 * 4.656612873077393e-10;   // (pi / 2) 2^-31
  const double x2 = x * x;
  // sin(delta) rounded once: x a and the rest (a's own, the series')
  constexpr double al = 6.123233995736766e-17 * 4.656612873077393e-10;
  const double sd = fma(x, a, x * fma(x2, fma(x2, a * a * a * a * a / 120.0, -a * a * a / 6.0), al));
  const double cm = x2 * fma(x2, a * a * a * a / 24.0, -a * a / 2.0);
  const double* T = tables().cs[i];
#if defined(__CUDA_ARCH__)
  const double2 tc = *reinterpret_cast<const double2*>(T), ts = *reinterpret_cast<const double2*>(T + 2);
  const double C = tc.x, Cl = tc.y, S = ts.x, Sl = ts.y;
#else
  const double C = T[0], Cl = T[1], S = T[2], Sl = T[3];
#endif
  const double c = C + fma(-S, sd, fma(C, cm, Cl));   // the smallest terms first
  const double s = S + fma(C, sd, fma(S, cm, Sl));
  const double u = quarter & 1 ? s : c, v = quarter & 1 ? c : s;
  const int64_t top = int64_t(1) << 63;
  cs = from_bits(bits(u) ^ ((quarter == 1 || quarter == 2) ? top : 0));
  sn = from_bits(bits(v) ^ (quarter & 2 ? top : 0));
}

}  // namespace m64
}  // namespace pdfx
