// The largest errors on the device of csrc/math64.h's functions and of the library's that they stand
// for, in units in the last place against long double: the uniforms' words at their ends, at powers
// of two, around the tables' cells and at random, and positive numbers of every exponent that the
// functions meet.  One line per function: its error and the library's.
#include <cstdio>
#include <random>
#include <vector>

#include <cuda_runtime.h>

#include "math64.h"

namespace m64 = pdfx::m64;
typedef long double LD;
constexpr int kOut = 8;   // of a word: log, cos, sin; of a number: rcp, root, rcbrt, quotient; then the library's

// The number that number i is divided by.
__host__ __device__ inline int partner(int i, int n) { return static_cast<int>((i * 7919ll + 1) % n); }

__global__ void words_kernel(const uint32_t* w, int n, double* out) {
  const int i = static_cast<int>(blockIdx.x * blockDim.x + threadIdx.x);
  if (i >= n) return;
  double* o = out + static_cast<size_t>(kOut) * i;
  o[0] = m64::minus_two_log(w[i]);
  m64::turn(w[i], o[1], o[2]);
  const double u = (static_cast<double>(w[i]) + 0.5) * 2.3283064365386963e-10;
  o[4] = -2.0 * log(u);
  sincospi(2.0 * u, o + 6, o + 5);
}
__global__ void numbers_kernel(const double* x, int n, double* out) {
  const int i = static_cast<int>(blockIdx.x * blockDim.x + threadIdx.x);
  if (i >= n) return;
  double* o = out + static_cast<size_t>(kOut) * i;
  o[0] = m64::rcp(x[i]);
  o[1] = m64::root(x[i]);
  o[2] = m64::rcbrt(x[i]);
  o[3] = m64::quotient(x[i], x[partner(i, n)]);
  o[4] = 1.0 / x[i];
  o[5] = sqrt(x[i]);
  o[6] = cbrt(1.0 / x[i]);
  o[7] = x[i] / x[partner(i, n)];
}

static double worst[2][7] = {};
static void add(int h, int k, double got, LD want) {
  const double w = std::fabs(static_cast<double>(want));
  const double e = static_cast<double>(fabsl(static_cast<LD>(got) - want)) / (std::nextafter(w, INFINITY) - w);
  if (!(e <= worst[h][k])) worst[h][k] = e;
}

template <typename T, typename Kernel>
static std::vector<double> run(const std::vector<T>& in, Kernel kernel) {
  const int n = static_cast<int>(in.size());
  std::vector<double> out(static_cast<size_t>(kOut) * n);
  T* d = nullptr;
  double* o = nullptr;
  if (cudaMalloc(&d, sizeof(T) * n) != cudaSuccess || cudaMalloc(&o, sizeof(double) * out.size()) != cudaSuccess) return {};
  cudaMemcpy(d, in.data(), sizeof(T) * n, cudaMemcpyHostToDevice);
  kernel<<<(n + 255) / 256, 256>>>(d, n, o);
  const cudaError_t e = cudaMemcpy(out.data(), o, sizeof(double) * out.size(), cudaMemcpyDeviceToHost);
  cudaFree(d);
  cudaFree(o);
  return e == cudaSuccess ? out : std::vector<double>();
}

int main() {
  std::mt19937_64 g(1);
  std::vector<uint32_t> w;
  for (int k = 0; k < 32; ++k)
    for (int d = -3; d <= 3; ++d) w.push_back((1u << k) + static_cast<uint32_t>(d));
  for (uint32_t i = 0; i < 2049; ++i)
    for (int d = -2; d <= 2; ++d) w.push_back((i << 21) + static_cast<uint32_t>(d));
  for (uint32_t k = 0; k < 20000; ++k) { w.push_back(k); w.push_back(0xffffffffu - k); }
  for (int k = 0; k < 400000; ++k) w.push_back(static_cast<uint32_t>(g()));
  for (int k = 0; k < 200000; ++k) w.push_back(~static_cast<uint32_t>(g() >> (32 + k % 24)));   // u near 1
  std::vector<double> x;
  std::uniform_real_distribution<double> e(-120, 120), m(1.0, 2.0);
  for (int k = 0; k < 400000; ++k) x.push_back(std::exp2(e(g)));
  for (int k = -110; k <= 110; ++k) {
    for (double v : {1.0, std::nextafter(1.0, 2.0), std::nextafter(2.0, 0.0)}) x.push_back(std::ldexp(v, k));
    for (int j = 0; j < 500; ++j) x.push_back(std::ldexp(m(g), k));
  }
  const std::vector<double> ow = run(w, words_kernel), ox = run(x, numbers_kernel);
  if (ow.empty() || ox.empty()) return 1;
  const LD quarter_pi = 0.785398163397448309615660845819875721049L;
  for (size_t i = 0; i < w.size(); ++i) {
    const double* o = ow.data() + kOut * i;
    const LD u = (static_cast<LD>(w[i]) + 0.5L) / 4294967296.0L;
    const LD lg = w[i] > 0x80000000u ? log1pl(u - 1) : logl(u);
    // the angle from the nearest multiple of a quarter turn, so that its sine stays exact
    const uint64_t mm = 2 * static_cast<uint64_t>(w[i]) + 1;
    const int q = static_cast<int>(w[i] >> 30);
    const LD t = static_cast<LD>(mm - (static_cast<uint64_t>(q) << 31)) / 2147483648.0L;
    const LD c0 = t <= 0.5L ? cosl(2 * quarter_pi * t) : sinl(2 * quarter_pi * (1 - t));
    const LD s0 = t <= 0.5L ? sinl(2 * quarter_pi * t) : cosl(2 * quarter_pi * (1 - t));
    const LD C = q == 0 ? c0 : q == 1 ? -s0 : q == 2 ? -c0 : s0;
    const LD S = q == 0 ? s0 : q == 1 ? c0 : q == 2 ? -s0 : -c0;
    for (int h = 0; h < 2; ++h) {
      add(h, 0, o[4 * h], -2 * lg);
      add(h, 1, o[4 * h + 1], C);
      add(h, 2, o[4 * h + 2], S);
    }
  }
  for (size_t i = 0; i < x.size(); ++i) {
    const double* o = ox.data() + kOut * i;
    const LD X = x[i];
    for (int h = 0; h < 2; ++h) {
      add(h, 3, o[4 * h], 1 / X);
      add(h, 4, o[4 * h + 1], sqrtl(X));
      add(h, 5, o[4 * h + 2], 1 / cbrtl(X));
      add(h, 6, o[4 * h + 3], X / x[partner(static_cast<int>(i), static_cast<int>(x.size()))]);
    }
  }
  const char* names[] = {"log", "cos", "sin", "rcp", "root", "rcbrt", "quotient"};
  for (int k = 0; k < 7; ++k) std::printf("%s %.4f %.4f\n", names[k], worst[0][k], worst[1][k]);
  return 0;
}
