// csrc/math64.h's widened against the conversion, bit for bit, over every sign and exponent of
// an FP32 number with mantissas at their ends and at random.
#include <cstdio>
#include <random>

#include "math64.h"

int main() {
  std::mt19937 g(1);
  long bad = 0, n = 0;
  auto check = [&](uint32_t b) {
    const float x = pdfx::m64::from_fbits(b);
    bad += pdfx::m64::bits(pdfx::m64::widened(x)) != pdfx::m64::bits(static_cast<double>(x));
    ++n;
  };
  for (uint32_t se = 0; se < 512; ++se) {
    for (uint32_t m : {0u, 1u, 2u, 0x3fffffu, 0x400000u, 0x400001u, 0x7ffffeu, 0x7fffffu}) check(se << 23 | m);
    for (int k = 0; k < 2000; ++k) check(se << 23 | (g() & 0x7fffffu));
  }
  std::printf("%ld %ld\n", bad, n);
}
