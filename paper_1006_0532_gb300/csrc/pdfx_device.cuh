// Device building blocks shared by the pdfx kernels: counter-based random numbers,
// Gaussian and gamma sampling, and the per-element data layout.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "math64.h"

namespace pdfx {

constexpr int kNF = 32;            // nodal field slots
constexpr int kNS = 13;            // statistics per element / node
constexpr int kHopLimit = 64;      // neighbour-walk hops before the fall-back search
constexpr int kGammaAttempts = 32; // Marsaglia-Tsang attempts before falling back to the mean

// Philox counter word 2 ("purpose"): independent streams per use.
enum Purpose : uint32_t { kPurStep = 0, kPurInit = 1, kPurWallGamma = 2, kPurRedist = 3,
                          kPurInitGamma = 4 };

// Diagnostic counter slots (int64 each).
enum Diag : int {
  kDiagHops = 0, kDiagFallback, kDiagBrute, kDiagLost, kDiagWall, kDiagFreeSlip,
  kDiagOmegaReflect, kDiagC0Clamp, kDiagGammaExhausted, kDiagMoves, kDiagSource,
  kDiagCapacity, kDiagNonFinite, kDiagHopHist0, kDiagLostRecord = kDiagHopHist0 + 8,
  kDiagBadElement, kDiagCount
};
constexpr int kLostRecords = 4;    // (x, y, old element, particle id) of the first lost particles
constexpr int kBruteCap = 4096;    // particles per step that may need the brute-force search

// Per-element geometry: the coordinates of the three nodes (x in [0, period), the canonical
// image) and 1 / (2 A_e).  FP64 form: plain FP64.  FP32 form: each coordinate as an
// unevaluated sum hi + lo of two FP32 numbers (about 48 significant bits), so that a
// particle's offset from a node, and with it the area coordinates, keep FP32 precision
// relative to the cell rather than to the domain (a first cell 4.6e-5 high at y = 1 is 770
// FP32 spacings of y).
//
// Both keep each edge's vector, from the edge's lower-numbered node (its pivot) to the other,
// computed once in FP64 from the nodes' coordinates (and in the FP32 form rounded): the same
// numbers for both elements of the edge.
template <typename T>
struct ElemGeo;
// FP64 form: code holds, for the edge opposite local vertex k, the pivot's local index (bits
// 3k, 3k + 1) and whether the pivot is the edge's second node in counter-clockwise order (bit
// 3k + 2, the cross product's sign flips).
template <>
struct __align__(16) ElemGeo<double> {
  double x[3], y[3];
  double ex[3], ey[3];
  double inv2a;
  uint32_t code, pad;
};
// FP32 form, whose advance is bound by the instructions it issues: the nodes in ascending order
// of their ids, so that an edge's pivot needs no selection (node lo for the edges opposite mid
// and hi, node mid for the one opposite lo) and the third node's offset is not formed; the
// edges in the order of the nodes opposite them, their vectors negated where the cross
// product's sign flips; and the neighbours (ElemTopo's, in local order), which the walk then
// reads with the rest.  code: bits 2k, 2k + 1 the place of local vertex k in that order.
// 12,100-triangle channel, 3.6M particles: 1,262 warp instructions per 32 particles and 166 us
// with the nodes in local order (a selection per edge) and an event's own counter in every
// thread, 1,073 and 155 us so; at 25M particles 1,050 us and 930.
struct GeoNode {
  float xh, yh, xl, yl;
};
template <>
struct __align__(16) ElemGeo<float> {
  GeoNode lo, mid;
  float ex[3], ey[3];
  float inv2a;
  uint32_t code;
  int32_t nb[3], pad;
  GeoNode hi;
};

// Per-element topology: node ids, neighbour across the edge opposite each vertex (-1 = a
// boundary edge; -2 - j = a free-slip boundary edge whose own line is entry j of the
// free-slip edge table), index into the no-slip and free-slip line tables (-1 = none).
struct __align__(16) ElemTopo {
  int n0, n1, n2, wall;
  int nb0, nb1, nb2, fslip;
};

// A boundary line: a point on it and the unit normal pointing into the domain (FP32 form:
// the point as hi + lo pairs).
template <typename T>
struct Line;
template <>
struct __align__(32) Line<double> {
  double px, py, nx, ny;
};
template <>
struct __align__(16) Line<float> {
  float px, py, nx, ny, pxl, pyl, pad0, pad1;
};

// A particle position: FP64, or (FP32 form) each coordinate as hi + lo.
template <typename T>
struct Pos;
template <>
struct Pos<double> {
  double x, y;
};
template <>
struct Pos<float> {
  float xh, xl, yh, yl;
};

// ---------------------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11).  Counter = (particle id, step,
// purpose, block); key = (seed low word, seed high word ^ instance).
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    const uint64_t p0 = static_cast<uint64_t>(0xD2511F53u) * c.x;
    const uint64_t p1 = static_cast<uint64_t>(0xCD9E8D57u) * c.z;
    c = make_uint4(static_cast<uint32_t>(p1 >> 32) ^ c.y ^ k0, static_cast<uint32_t>(p1),
                   static_cast<uint32_t>(p0 >> 32) ^ c.w ^ k1, static_cast<uint32_t>(p0));
  }
  return c;
}

// Uniform on (0, 1) from one 32-bit word: (w + 1/2) 2^-32.  The FP32 form keeps relative
// precision for small words (the Gaussian tail) and may round the top words up to 1.
__device__ __forceinline__ double uniform01(uint32_t w, double) {
  return (static_cast<double>(w) + 0.5) * 2.3283064365386963e-10;
}
__device__ __forceinline__ float uniform01(uint32_t w, float) {
  return fmaf(__uint2float_rn(w), 2.3283064365386963e-10f, 1.1641532182693481e-10f);
}

// Box & Muller (1958): two independent N(0, 1) from two uniform words.
__device__ __forceinline__ void box_muller(uint32_t w1, uint32_t w2, double& g1, double& g2) {
  const double r = sqrt(-2.0 * log(uniform01(w1, 0.0)));
  double s, c;
  sincospi(2.0 * uniform01(w2, 0.0), &s, &c);
  g1 = r * c;
  g2 = r * s;
}
__device__ __forceinline__ void box_muller(uint32_t w1, uint32_t w2, float& g1, float& g2) {
  const float r = sqrtf(-2.0f * logf(uniform01(w1, 0.0f)));
  float s, c;
  sincospif(2.0f * uniform01(w2, 0.0f), &s, &c);
  g1 = r * c;
  g2 = r * s;
}

template <typename T>
__device__ __forceinline__ T dlog(T x);
template <>
__device__ __forceinline__ double dlog<double>(double x) { return log(x); }
template <>
__device__ __forceinline__ float dlog<float>(float x) { return logf(x); }

// Gamma(shape >= 1, scale) by Marsaglia & Tsang (2000).  Attempt j uses Philox block j:
// one Gaussian from words 0-1 (cosine branch) and one uniform from word 2.  After
// kGammaAttempts rejections the mean is returned and *exhausted is set.
template <typename T>
__device__ T gamma_draw(uint32_t k0, uint32_t k1, uint32_t pid, uint32_t step, uint32_t purpose,
                        T shape, T scale, int* exhausted) {
  const T d = shape - T(1) / T(3);
  const T c = T(1) / sqrt(T(9) * d);
  for (uint32_t j = 0; j < kGammaAttempts; ++j) {
    const uint4 r = philox(make_uint4(pid, step, purpose, j), k0, k1);
    T xg, dummy;
    box_muller(r.x, r.y, xg, dummy);
    const T uu = uniform01(r.z, T(0));
    const T t = T(1) + c * xg;
    if (t <= T(0)) continue;
    const T vv = t * t * t;
    if (dlog(uu) < T(0.5) * xg * xg + d - d * vv + d * dlog(vv)) return d * vv * scale;
  }
  *exhausted = 1;
  return shape * scale;
}

template <typename T>
__host__ __device__ __forceinline__ T min_image(T d, T L) {
  if (L > T(0)) {
    if (d > T(0.5) * L) return d - L;
    if (d < T(-0.5) * L) return d + L;
  }
  return d;
}

template <typename T>
__device__ __forceinline__ T wrap_period(T x, T L) {
  if (L > T(0)) {
    if (x < T(0)) x += L;
    if (x >= L) x -= L;
  }
  return x;
}

// (h, l) += d for an FP32 pair: an exact two-sum of the leading parts (Knuth), the error
// added to the trailing part, then renormalised (Dekker's fast two-sum), every operation
// rounded on its own.
__device__ __forceinline__ void pair_add(float& h, float& l, float d) {
  const float s = __fadd_rn(h, d);
  const float bb = __fsub_rn(s, h);
  const float e = __fadd_rn(__fsub_rn(h, __fsub_rn(s, bb)), __fsub_rn(d, bb));
  const float t = __fadd_rn(l, e);
  h = __fadd_rn(s, t);
  l = __fsub_rn(t, __fsub_rn(h, s));
}
// The FP32 pair nearest a double (hi = its FP32 rounding, lo = the FP32 rounding of the rest).
__host__ __device__ __forceinline__ void pair_of(double v, float& h, float& l) {
  h = static_cast<float>(v);
  l = static_cast<float>(v - static_cast<double>(h));
}
__host__ __device__ __forceinline__ double pair_value(float h, float l) {
  return static_cast<double>(h) + static_cast<double>(l);
}

// Node k's coordinates as FP64 (the FP32 form's pairs summed).
__device__ __forceinline__ double node_x(const ElemGeo<double>& g, int k) { return g.x[k]; }
__device__ __forceinline__ double node_y(const ElemGeo<double>& g, int k) { return g.y[k]; }
__device__ __forceinline__ GeoNode local_node(const ElemGeo<float>& g, int k) {
  const uint32_t r = (g.code >> (2 * k)) & 3u;
  return r == 0u ? g.lo : (r == 1u ? g.mid : g.hi);
}
__device__ __forceinline__ double node_x(const ElemGeo<float>& g, int k) {
  const GeoNode n = local_node(g, k);
  return pair_value(n.xh, n.xl);
}
__device__ __forceinline__ double node_y(const ElemGeo<float>& g, int k) {
  const GeoNode n = local_node(g, k);
  return pair_value(n.yh, n.yl);
}

// min_image and wrap_period of the FP64 form, their tests on the bits (a comparison takes the
// FP64 pipe like any other operation): d stays while its high word is below L / 2's, which a
// particle near its element's nodes meets unless the seam lies between.
__device__ __forceinline__ double near_image(double d, double L) {
  const int32_t hl = m64::hi_word(L);
  if (hl > 0 && (m64::hi_word(d) & 0x7fffffff) >= hl - 0x100000) return min_image(d, L);
  return d;
}
__device__ __forceinline__ double near_period(double x, double L) {
  const int64_t bx = m64::bits(x), bl = m64::bits(L);
  return bl > 0 && (bx < 0 || bx >= bl) ? wrap_period(x, L) : x;
}

// The FP32 form's: one comparison decides (the same differences as min_image's).
__device__ __forceinline__ float near_image(float d, float L) {
  if (L > 0.0f && fabsf(d) > 0.5f * L) return min_image(d, L);
  return d;
}

// Node b minus node a (minimum image in x), in the working precision.
__device__ __forceinline__ void node_vec(const GeoNode& a, const GeoNode& b, float L, float& ex, float& ey) {
  ex = __fadd_rn(min_image(__fsub_rn(b.xh, a.xh), L), __fsub_rn(b.xl, a.xl));
  ey = __fadd_rn(__fsub_rn(b.yh, a.yh), __fsub_rn(b.yl, a.yl));
}
// Particle minus node k (minimum image in x), in the working precision.
__device__ __forceinline__ void node_rel(const ElemGeo<double>& g, int k, const Pos<double>& P, double L,
                                         double& dx, double& dy) {
  dx = near_image(P.x - g.x[k], L);
  dy = P.y - g.y[k];
}
__device__ __forceinline__ void node_rel(const GeoNode& n, const Pos<float>& P, float L, float& dx, float& dy) {
  dx = __fadd_rn(near_image(__fsub_rn(P.xh, n.xh), L), __fsub_rn(P.xl, n.xl));
  dy = __fadd_rn(__fsub_rn(P.yh, n.yh), __fsub_rn(P.yl, n.yl));
}

// Particle minus a point given in FP64 (FP32 form: as the pair (ph, pl)), minimum image in x.
__device__ __forceinline__ double rel_x(const Pos<double>& P, double px, double, double L) {
  return near_image(P.x - px, L);
}
__device__ __forceinline__ double rel_y(const Pos<double>& P, double py, double) { return P.y - py; }
__device__ __forceinline__ float rel_x(const Pos<float>& P, float ph, float pl, float L) {
  return __fadd_rn(near_image(__fsub_rn(P.xh, ph), L), __fsub_rn(P.xl, pl));
}
__device__ __forceinline__ float rel_y(const Pos<float>& P, float ph, float pl) {
  return __fadd_rn(__fsub_rn(P.yh, ph), __fsub_rn(P.yl, pl));
}

// Signed distance of a particle from a boundary line (positive on the domain side).
__device__ __forceinline__ double line_dist(const Line<double>& ln, const Pos<double>& P, double L) {
  return min_image(P.x - ln.px, L) * ln.nx + (P.y - ln.py) * ln.ny;
}
__device__ __forceinline__ float line_dist(const Line<float>& ln, const Pos<float>& P, float L) {
  return rel_x(P, ln.px, ln.pxl, L) * ln.nx + rel_y(P, ln.py, ln.pyl) * ln.ny;
}

// P += (dx, dy): plain FP64, or pair additions.
__device__ __forceinline__ void pos_add(Pos<double>& P, double dx, double dy) {
  P.x += dx;
  P.y += dy;
}
__device__ __forceinline__ void pos_add(Pos<float>& P, float dx, float dy) {
  pair_add(P.xh, P.xl, dx);
  pair_add(P.yh, P.yl, dy);
}
// Eq. 7's move X + U dt + sqrt(2 nu) dW per coordinate (FP64: one expression, as the
// oracle writes it; FP32: the increment added to the pair).
__device__ __forceinline__ void pos_move(Pos<double>& P, double ux, double uy, double dt, double s2nu,
                                         double dWx, double dWy) {
  P.x = P.x + ux * dt + s2nu * dWx;
  P.y = P.y + uy * dt + s2nu * dWy;
}
__device__ __forceinline__ void pos_move(Pos<float>& P, float ux, float uy, float dt, float s2nu,
                                         float dWx, float dWy) {
  pair_add(P.xh, P.xl, ux * dt + s2nu * dWx);
  pair_add(P.yh, P.yl, uy * dt + s2nu * dWy);
}
// Reflection across a line at signed distance d < 0: P -= 2 d n.
__device__ __forceinline__ void pos_reflect(Pos<double>& P, double d, double nx, double ny) {
  P.x -= 2.0 * d * nx;
  P.y -= 2.0 * d * ny;
}
__device__ __forceinline__ void pos_reflect(Pos<float>& P, float d, float nx, float ny) {
  pair_add(P.xh, P.xl, -(2.0f * d * nx));
  pair_add(P.yh, P.yl, -(2.0f * d * ny));
}
// Periodic wrap of x into [0, L).
__device__ __forceinline__ void pos_wrap(Pos<double>& P, double L) { P.x = near_period(P.x, L); }
__device__ __forceinline__ void pos_wrap(Pos<float>& P, float L) {
  if (L > 0.0f) {
    if (P.xh < 0.0f) pair_add(P.xh, P.xl, L);
    if (P.xh >= L) pair_add(P.xh, P.xl, -L);
  }
}
__device__ __forceinline__ double pos_x(const Pos<double>& P) { return P.x; }
__device__ __forceinline__ double pos_y(const Pos<double>& P) { return P.y; }
__device__ __forceinline__ double pos_x(const Pos<float>& P) { return pair_value(P.xh, P.xl); }
__device__ __forceinline__ double pos_y(const Pos<float>& P) { return pair_value(P.yh, P.yl); }
__device__ __forceinline__ Pos<double> pos_of(double x, double y, double) { return {x, y}; }
__device__ __forceinline__ Pos<float> pos_of(double x, double y, float) {
  Pos<float> P;
  pair_of(x, P.xh, P.xl);
  pair_of(y, P.yh, P.yl);
  return P;
}

// Separately rounded products (no fused multiply-add).  Every evaluation of an edge's
// cross product then rounds identically, whichever element and slot it is computed for,
// so the two elements sharing an edge always see exactly opposite values (a point on the
// edge is in both), and the FP64 form matches host arithmetic bit for bit.
__device__ __forceinline__ double xmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float xmul(float a, float b) { return __fmul_rn(a, b); }

// Twice the signed areas N^A, N^B, N^C (Eqs. 44-45, Fig. 1): for each vertex, the cross
// product of the opposite edge with the vector from one end of that edge to the particle.
// Each edge is pivoted at its lower-numbered node, so the two elements sharing an edge
// evaluate it with identical rounding and opposite signs (watertight point location).
// The particle's offsets from the three nodes, formed from the nodes' own coordinates and the
// particle's alone, then each edge's stored vector crossed with the offset from its pivot.
__device__ __forceinline__ void area_cross(const ElemGeo<double>& g, const Pos<double>& P, double L, double (&n)[3]) {
  double dx[3], dy[3];
#pragma unroll
  for (int m = 0; m < 3; ++m) node_rel(g, m, P, L, dx[m], dy[m]);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const uint32_t c = g.code >> (3 * k);
    const int pv = static_cast<int>(c & 3u);
    const double px = pv == 0 ? dx[0] : (pv == 1 ? dx[1] : dx[2]);
    const double py = pv == 0 ? dy[0] : (pv == 1 ? dy[1] : dy[2]);
    const double cr = xmul(g.ex[k], py) - xmul(g.ey[k], px);
    n[k] = (c & 4u) ? -cr : cr;
  }
}
// FP32 form: in the order of the nodes' ids (local_order puts them back).
__device__ __forceinline__ void area_cross(const ElemGeo<float>& g, const Pos<float>& P, float L, float (&n)[3]) {
  float ax, ay, bx, by;
  node_rel(g.lo, P, L, ax, ay);
  node_rel(g.mid, P, L, bx, by);
  n[0] = xmul(g.ex[0], by) - xmul(g.ey[0], bx);
  n[1] = xmul(g.ex[1], ay) - xmul(g.ey[1], ax);
  n[2] = xmul(g.ex[2], ay) - xmul(g.ey[2], ax);
}
__device__ __forceinline__ void local_order(const ElemGeo<double>&, double (&)[3]) {}
__device__ __forceinline__ void local_order(const ElemGeo<float>& g, float (&n)[3]) {
  const float v[3] = {n[0], n[1], n[2]};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const uint32_t r = (g.code >> (2 * k)) & 3u;
    n[k] = r == 0u ? v[0] : (r == 1u ? v[1] : v[2]);
  }
}

// Area coordinates lambda_k = N^k / A_e (Eqs. 37-38 shapefunction values at the particle).
template <typename T>
__device__ __forceinline__ void area_coords(const ElemGeo<T>& g, const Pos<T>& P, T L, T& la, T& lb, T& lc) {
  T n[3];
  area_cross(g, P, L, n);
  local_order(g, n);
  la = n[0] * g.inv2a;
  lb = n[1] * g.inv2a;
  lc = n[2] * g.inv2a;
}

// Point in the triangle with weights (1 - s) A + s (1 - t) B + s t C (Osada et al.).
__device__ __forceinline__ Pos<double> triangle_point(const ElemGeo<double>& g, double s, double t, double L) {
  Pos<double> P;
  P.x = g.x[0] + s * (1.0 - t) * min_image(g.x[1] - g.x[0], L) + s * t * min_image(g.x[2] - g.x[0], L);
  P.y = g.y[0] + s * (1.0 - t) * (g.y[1] - g.y[0]) + s * t * (g.y[2] - g.y[0]);
  return P;
}
__device__ __forceinline__ Pos<float> triangle_point(const ElemGeo<float>& g, float s, float t, float L) {
  float bx, by, cx, cy;
  const GeoNode n0 = local_node(g, 0);
  node_vec(n0, local_node(g, 1), L, bx, by);
  node_vec(n0, local_node(g, 2), L, cx, cy);
  Pos<float> P{n0.xh, n0.xl, n0.yh, n0.yl};
  pos_add(P, s * (1.0f - t) * bx + s * t * cx, s * (1.0f - t) * by + s * t * cy);
  return P;
}

}  // namespace pdfx

namespace pdfx {

// Fox's projection (Eqs. 64-66): from the element's moments em (layout of the element
// statistics: 4-6 variances, 7-9 <uv>, <uw>, <vw>, 12 scalar variance) and its scalar-
// velocity covariances uphi[3], the factors f_a = alpha_a / s_a of the projected velocity
// U_rho = sum_a f_a (U_a - <U_a>), alpha solving rho_ab alpha_b = rho_a by Cramer's rule;
// all zero when the scalar or a velocity component has no variance or |det| <= 1e-12.
__host__ __device__ inline void fox_factors(const double* em, const double* uphi, double f[3]) {
  f[0] = f[1] = f[2] = 0.0;
  const double var0 = em[4], var1 = em[5], var2 = em[6], vphi = em[12];
  if (!(vphi > 0.0) || !(var0 > 0.0) || !(var1 > 0.0) || !(var2 > 0.0)) return;
  const double s[3] = {sqrt(var0), sqrt(var1), sqrt(var2)}, sphi = sqrt(vphi);
  const double cuv = em[7], cuw = em[8], cvw = em[9];
  const double A[3][3] = {{1.0, cuv / (s[0] * s[1]), cuw / (s[0] * s[2])},
                          {cuv / (s[0] * s[1]), 1.0, cvw / (s[1] * s[2])},
                          {cuw / (s[0] * s[2]), cvw / (s[1] * s[2]), 1.0}};
  const double b[3] = {uphi[0] / (s[0] * sphi), uphi[1] / (s[1] * sphi), uphi[2] / (s[2] * sphi)};
  auto det3 = [](const double M[3][3]) {
    return M[0][0] * (M[1][1] * M[2][2] - M[1][2] * M[2][1]) -
           M[0][1] * (M[1][0] * M[2][2] - M[1][2] * M[2][0]) +
           M[0][2] * (M[1][0] * M[2][1] - M[1][1] * M[2][0]);
  };
  const double det = det3(A);
  if (!(fabs(det) > 1e-12)) return;
  for (int i = 0; i < 3; ++i) {
    double M[3][3];
    for (int r = 0; r < 3; ++r)
      for (int c = 0; c < 3; ++c) M[r][c] = c == i ? b[r] : A[r][c];
    f[i] = (det3(M) / det) / s[i];
  }
}

}  // namespace pdfx
