// Largest errors of csrc/math64.h in units in the last place, against long double, one line
// per function: the uniforms' words at their ends, at powers of two and at random, and
// positive numbers over the range the FP32 seeds take, its ends and beyond.
#include <cstdio>
#include <random>

#include "math64.h"

using namespace pdfx::m64;
typedef long double LD;

static double ulp(double x) { x = std::fabs(x); return std::nextafter(x, INFINITY) - x; }
static void worst(double& w, double got, LD want) {
  const double e = static_cast<double>(fabsl(got - want)) / ulp(static_cast<double>(want));
  if (!(e <= w)) w = e;
}

int main() {
  std::mt19937_64 g(1);
  double wl = 0, wc = 0, ws = 0, wr = 0, wq = 0, w3 = 0;
  const LD quarter_pi = 0.785398163397448309615660845819875721L;
  auto word = [&](uint32_t w) {
    worst(wl, minus_two_log(w), -2 * logl((static_cast<LD>(w) + 0.5L) / 4294967296.0L));
    // the angle from the nearest multiple of a quarter turn, so that its sine stays exact
    const uint64_t m = 2 * static_cast<uint64_t>(w) + 1;
    const int q = static_cast<int>(w >> 30);
    const LD t = static_cast<LD>(m - (static_cast<uint64_t>(q) << 31)) / 2147483648.0L;
    const LD c0 = t <= 0.5L ? cosl(2 * quarter_pi * t) : sinl(2 * quarter_pi * (1 - t));
    const LD s0 = t <= 0.5L ? sinl(2 * quarter_pi * t) : cosl(2 * quarter_pi * (1 - t));
    const LD C = q == 0 ? c0 : q == 1 ? -s0 : q == 2 ? -c0 : s0;
    const LD S = q == 0 ? s0 : q == 1 ? c0 : q == 2 ? -s0 : -c0;
    double c, s;
    turn(w, c, s);
    worst(wc, c, C);
    worst(ws, s, S);
  };
  for (int k = 0; k < 32; ++k)
    for (int d = -3; d <= 3; ++d) word((1u << k) + static_cast<uint32_t>(d));
  for (uint32_t i = 0; i < 1025; ++i)   // around the tables' cell boundaries
    for (int d = -2; d <= 2; ++d) word((i << 22) + (1u << 21) + static_cast<uint32_t>(d));
  for (uint32_t k = 0; k < 20000; ++k) { word(k); word(0xffffffffu - k); }
  for (int k = 0; k < 300000; ++k) word(static_cast<uint32_t>(g()));
  auto number = [&](double x) {
    const LD X = x;
    worst(wr, rcp(x), 1 / X);
    worst(wq, root(x), sqrtl(X));
    worst(w3, rcbrt(x), 1 / cbrtl(X));
  };
  std::uniform_real_distribution<double> e(-120, 120);
  for (int k = 0; k < 300000; ++k) number(std::exp2(e(g)));
  for (int k = -130; k <= 130; ++k)
    for (double x : {std::ldexp(1.0, k), std::nextafter(std::ldexp(1.0, k), 0.0), std::nextafter(std::ldexp(1.0, k), INFINITY)}) number(x);
  std::printf("log %.3f\ncos %.3f\nsin %.3f\nrcp %.3f\nroot %.3f\nrcbrt %.3f\n", wl, wc, ws, wr, wq, w3);
  bool ok = root(0.0) == 0.0 && std::isinf(rcp(0.0)) && std::isnan(root(-1.0)) && std::isnan(rcp(NAN));
  ok = ok && nonneg(0.0) && nonneg(-0.0) && nonneg(INFINITY) && !nonneg(NAN) && !nonneg(-NAN) && !nonneg(-1e-320);
  ok = ok && below_pos(-1.0, 1e-30) && below_pos(0.0, 1e-30) && !below_pos(1e-30, 1e-30) && !below_pos(NAN, 1e-30) &&
       !below_pos(-NAN, 1e-30) && below_pos(-INFINITY, 1e-30);
  std::printf("special %d\n", ok ? 1 : 0);
}
