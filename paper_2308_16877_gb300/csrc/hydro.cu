// Hexahedral Lagrangian hydro whose equation-of-state call is the approximated
// region (the paper approximates kernels of the LULESH proxy application,
// Table 1, Section 4.1; the scheme itself is a textbook staggered-grid update,
// the same one the CPU oracle restates).
//
// Per time step, on the EOS region's stream:
//   node kernel     forces from the stored volume gradients and the stored
//                   p + q, velocity and position update (1 / (12 m) stored at
//                   init), symmetry planes x = 0, y = 0, z = 0;
//   element kernel  exact trilinear-hexahedron volume and its gradient at the
//                   new positions, relative volume, artificial viscosity, the
//                   EOS inputs (e, v_{n+1}, dv, q_{n+1});
//   EOS region      exact, TAF, iACT or perforation through the region API;
//   finalize        e = p v / (gamma - 1), v = v_{n+1}, pq = p + q.
// With the exact EOS the last three are one kernel.
//
// Volume of a trilinear hexahedron and its gradient. With corners P_c in
// lexicographic order (c = a + 2b + 4d for offsets a, b, d), the integral of
// det J over the reference cube equals Grandy's sum of three triple products
// (J. Grandy, "Efficient computation of volume of hexahedral cells", LLNL
// UCRL-ID-128886, 1997), one per pair of faces meeting at corner 7 and at
// corner 0:
//   12 V = s1 . (c1 x d1) + s2 . (c2 x d2) + s3 . (c3 x d3),
//   s1 = (P2 - P1) + (P6 - P3), c1 = P7 - P2, d1 = P3 - P0,
//   s2 = (P4 - P2) + (P5 - P6), c2 = P7 - P4, d2 = P6 - P0,
//   s3 = (P1 - P4) + (P3 - P5) = -(s1 + s2), c3 = P7 - P1, d3 = P5 - P0.
// V is a cubic polynomial of the corners, so its gradient follows by the
// product rule: with A_i = c_i x d_i, B_i = d_i x s_i, C_i = s_i x c_i (the
// derivatives of the i-th triple product with respect to s_i, c_i and d_i),
// each corner collects the terms of the differences it appears in:
//   12 dV/dP0 = -(C1 + C2 + C3)        12 dV/dP7 = B1 + B2 + B3
//   12 dV/dP1 = (A3 - A1) - B3         12 dV/dP3 = (A3 - A1) + C1
//   12 dV/dP2 = (A1 - A2) - B1         12 dV/dP6 = (A1 - A2) + C2
//   12 dV/dP4 = (A2 - A3) - B2         12 dV/dP5 = (A2 - A3) + C3
// Since p31 + p12 + p23 = 0 (p31 = A3 - A1, p12 = A1 - A2, p23 = A2 - A3), the
// two sums are those of the other corners, and s3 = -(s1 + s2) takes A2 and A1
// out of the volume:
//   12 dV/dP7 = -(g1 + g2 + g4), 12 dV/dP0 = -(g3 + g5 + g6),
//   12 V = s2 . p23 - s1 . p31;
// each of g1..g6 adds its cross product to p31, p12 or p23.
// Every difference is of two corners of one element, so it carries the
// rounding of the element's size, not of its position. The kernel stores
// 12 dV/dP_c (the 1/12 is applied where the gradient is used).
// All of it runs in 64-bit fixed point: per element and axis the coordinates
// relative to corner 0 are placed on a grid six bits finer than the largest
// coordinate's significand (exact for every coordinate within six binades of
// it, else rounded to that grid) and shifted up to 60 bits; differences and
// their sums are exact, a product keeps its upper 64 bits from three 32-bit
// partial products, and each output is rounded once to FP64. GB300 issues two
// FP64 operations per SM and clock against 16 to 18 32 x 32 -> 64-bit
// multiply-adds and 64 other integer operations, and the fixed-point form is
// the more accurate one: against the exact gradient of jittered elements 0.31
// units of 2^-53 (rms, of the area terms) against 0.47 to 0.82, the volume 0.5
// against 0.95. FP64 instructions per element: 260 for the plain sum over the
// trilinear form's 24 corner triples, 104 with FP64 cross products of exact
// integer differences, 80 with those fused into the corner sums, 25
// conversions now; a step at 64^3 with the exact EOS 107.8, 95.6 and 43.4 us
// for the last three (with the fused EOS, 78.9 for the second), 20 steps at
// 256^3 with iACT 98.2, 83.8 and 56.8 ms. Coordinates that are infinite or NaN,
// elements smaller than 2^-27 of their coordinates and results outside the
// normal FP64 range take the same form in FP64.
#include <math.h>

#include "hpac_internal.cuh"
#include "regions.cuh"

namespace hpac {
namespace {

constexpr double kCq = 2.0;   // quadratic viscosity coefficient
constexpr double kCl = 0.5;   // linear viscosity coefficient

// The differences of Grandy's form, per axis: s1, s2, t = s1 + s2 = -s3,
// c1..c3, d1..d3 (component 0 x, 1 y, 2 z).
struct HexDiffs {
  double s1[3], s2[3], t[3], c1[3], c2[3], c3[3], d1[3], d2[3], d3[3];
};

// The differences in FP64 (the fallback for non-finite coordinates).
__device__ __forceinline__ void hex_diffs_fp64(const double (&X)[8], const double (&Y)[8], const double (&Z)[8],
                                               HexDiffs &D) {
  const double *P[3] = {X, Y, Z};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const double *p = P[a];
    D.s1[a] = (p[2] - p[1]) + (p[6] - p[3]);
    D.s2[a] = (p[4] - p[2]) + (p[5] - p[6]);
    D.t[a] = D.s1[a] + D.s2[a];
    D.c1[a] = p[7] - p[2];
    D.c2[a] = p[7] - p[4];
    D.c3[a] = p[7] - p[1];
    D.d1[a] = p[3] - p[0];
    D.d2[a] = p[6] - p[0];
    D.d3[a] = p[5] - p[0];
  }
}

// base + component a of x cross y, (b, c) the two axes after a.
__device__ __forceinline__ double add_cross(const double (&x)[3], const double (&y)[3], int b, int c, double base) {
  return fma(x[b], y[c], fma(-x[c], y[b], base));
}

// 12 dV/dP_c for the eight corners (absolute positions) and the volume V, in
// the form above, in FP64.
__device__ __noinline__ double hex_grad12_fp64(const double (&X)[8], const double (&Y)[8], const double (&Z)[8],
                                               double (&gx)[8], double (&gy)[8], double (&gz)[8]) {
  HexDiffs D;
  hex_diffs_fp64(X, Y, Z, D);
  double v12 = 0.0, w12 = 0.0;
  double *g[3] = {gx, gy, gz};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int b = (a + 1) % 3, c = (a + 2) % 3;
    const double A3 = fma(D.c3[b], D.d3[c], -__dmul_rn(D.c3[c], D.d3[b]));
    const double p31 = add_cross(D.d1, D.c1, b, c, A3);    // A3 - A1
    const double p23 = add_cross(D.c2, D.d2, b, c, -A3);   // A2 - A3
    const double p12 = -__dadd_rn(p31, p23);               // A1 - A2
    const double g1 = add_cross(D.d3, D.t, b, c, p31), g3 = add_cross(D.s1, D.c1, b, c, p31);
    const double g2 = add_cross(D.s1, D.d1, b, c, p12), g6 = add_cross(D.s2, D.c2, b, c, p12);
    const double g4 = add_cross(D.s2, D.d2, b, c, p23), g5 = add_cross(D.c3, D.t, b, c, p23);
    g[a][0] = -__dadd_rn(__dadd_rn(g3, g6), g5);
    g[a][1] = g1;
    g[a][2] = g2;
    g[a][3] = g3;
    g[a][4] = g4;
    g[a][5] = g5;
    g[a][6] = g6;
    g[a][7] = -__dadd_rn(__dadd_rn(g1, g2), g4);
    v12 = a == 0 ? __dmul_rn(D.s1[a], p31) : fma(D.s1[a], p31, v12);
    w12 = a == 0 ? __dmul_rn(D.s2[a], p23) : fma(D.s2[a], p23, w12);
  }
  return __dsub_rn(w12, v12) * (1.0 / 12.0);
}

constexpr int kFixedGuard = 6;  // grid bits below the largest coordinate's significand

// A coordinate whose exponent lies more than kFixedGuard binades below the
// element's largest, rounded to the grid (half away from zero).
__device__ __forceinline__ int64_t to_fixed_small(double x, int sh) {
  const uint64_t bits = (uint64_t)__double_as_longlong(x);
  const uint64_t m = (bits & 0xfffffffffffffull) | 1ull << 52;
  const int r = min(-sh, 63);
  const uint64_t M = (m + (1ull << (r - 1))) >> r;
  return (int64_t)bits < 0 ? -(int64_t)M : (int64_t)M;
}

// x << s for 0 <= s < 32: a funnel shift and a shift, where the general 64-bit
// shift also handles 32 to 63 (20 steps at 256^3: 61.7 -> 59.8 ms).
__device__ __forceinline__ uint64_t shl_below_32(uint64_t x, int s) {
  const uint32_t lo = (uint32_t)x, hi = (uint32_t)(x >> 32);
  return ((uint64_t)__funnelshift_l(lo, hi, s) << 32) | (lo << s);
}

// Coordinates of one axis relative to corner 0, R[c] = (P_c - P_0) / 2^S (R[0]
// unused), exactly for coordinates within kFixedGuard binades of the largest
// one, scaled so that the largest |R| lies in [2^59, 2^60) (less for an element
// smaller than 2^-27 of its coordinates). `bad` is set for an infinite or NaN
// coordinate, and where all corners coincide to that measure. Returns S.
__device__ __forceinline__ int to_relative(const double *P, int64_t (&R)[8], bool &bad) {
  uint32_t emax = 1;
#pragma unroll
  for (int c = 0; c < 8; ++c) emax = max(emax, ((uint32_t)__double2hiint(P[c]) >> 20) & 0x7ffu);
  bad |= emax == 0x7ffu;
  int64_t F[8];  // P / 2^(emax - 1075 - kFixedGuard), |F| < 2^59
  int below = 0;  // negative: a coordinate needs rounding to the grid
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const uint32_t hi = (uint32_t)__double2hiint(P[c]), lo = (uint32_t)__double2loint(P[c]);
    const uint32_t ec = (hi >> 20) & 0x7ffu;
    const int sh = (int)ec - (int)emax + kFixedGuard;  // <= kFixedGuard
    below |= ec ? sh : 0;
    // zeros, and subnormals, which are nothing on the grid of normal
    // coordinates of this size
    const uint64_t m = ec ? ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32) | lo : 0;
    const int64_t sign = (int64_t)(int32_t)hi >> 31;
    F[c] = ((int64_t)shl_below_32(m, sh & 31) ^ sign) - sign;
  }
  bad |= emax < 64u;
  // one branch for the eight: a branch for each kept their instructions apart
  // (64^3, 100 steps: 4.65 -> 4.34 ms; 256^3, 20 steps: 59.8 -> 56.8 ms)
  if (below < 0) {
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const uint32_t ec = ((uint32_t)__double2hiint(P[c]) >> 20) & 0x7ffu;
      const int sh = (int)ec - (int)emax + kFixedGuard;
      if (ec && sh < 0) F[c] = to_fixed_small(P[c], sh);
    }
  }
  uint32_t m = 0;
#pragma unroll
  for (int c = 1; c < 8; ++c) {
    R[c] = F[c] - F[0];
    const int32_t h = (int32_t)(R[c] >> 32);
    m |= (uint32_t)(h ^ (h >> 31));
  }
  bad |= m == 0u;
  const int sh = __clz(m) - 4;  // 0..28: |R| < 2^60, the magnitude's high word is below 2^28
#pragma unroll
  for (int c = 1; c < 8; ++c) R[c] = (int64_t)shl_below_32((uint64_t)R[c], sh);
  return (int)emax - 1075 - kFixedGuard - sh;
}

// A 64-bit integer as h 2^32 + l with signed 32-bit parts (|x| < 2^62).
struct Parts {
  int32_t h, l;
};

__device__ __forceinline__ Parts parts(int64_t x) {
  Parts p;
  p.l = (int32_t)x;
  p.h = (int32_t)(x >> 32) + (int32_t)((uint32_t)x >> 31);
  return p;
}

__device__ __forceinline__ int64_t wide(int32_t a, int32_t b) { return (int64_t)a * b; }

// base + (x_b y_c - x_c y_b) 2^-64, component a of a cross product, from the
// three upper partial products of each term (each a 32 x 32 -> 64-bit
// multiply-add), rounded: within 1 of the exact value.
__device__ __forceinline__ int64_t add_cross(const Parts (&x)[3], const Parts (&y)[3], int b, int c, int64_t base) {
  const int64_t up = wide(x[b].h, y[c].h) + base, un = wide(x[c].h, y[b].h);
  int64_t mp = wide(x[b].h, y[c].l) + 0x80000000ll;
  mp += wide(x[b].l, y[c].h);
  int64_t mn = wide(x[c].h, y[b].l);
  mn += wide(x[c].l, y[b].h);
  return (up - un) + ((mp - mn) >> 32);
}

// (x y - z w) 2^-64, likewise.
__device__ __forceinline__ int64_t sub_products(const Parts &x, const Parts &y, const Parts &z, const Parts &w) {
  const int64_t up = wide(x.h, y.h), un = wide(z.h, w.h);
  int64_t mp = wide(x.h, y.l) + 0x80000000ll;
  mp += wide(x.l, y.h);
  int64_t mn = wide(z.h, w.l);
  mn += wide(z.l, w.h);
  return (up - un) + ((mp - mn) >> 32);
}

// v 2^k for v = 0 or |v| >= 1/16, by its exponent field (the caller has checked
// that the result is normal).
__device__ __forceinline__ double scaled(double v, int k) {
  const int hi = __double2hiint(v);
  return __hiloint2double(hi ? hi + (k << 20) : 0, __double2loint(v));
}

// 12 dV/dP_c and V in 64-bit fixed point: with |R| < 2^60 the differences of
// two corners lie below 2^61, s1, s2 and t below 2^62; a cross product keeps the
// upper 64 bits (below 2^60), the corner sums below 2^63. One unit is about
// 2^-56 of an element's area terms, so with one rounding to FP64 per output the
// errors stay below those of the FP64 form (0.65 ulp and more per output).
__device__ __forceinline__ double hex_grad12(const double (&X)[8], const double (&Y)[8],
                                             const double (&Z)[8], double (&gx)[8], double (&gy)[8],
                                             double (&gz)[8]) {
  const double *P[3] = {X, Y, Z};
  double *g[3] = {gx, gy, gz};
  Parts s1[3], s2[3], t[3], c1[3], c2[3], c3[3], d1[3], d2[3], d3[3];
  int S[3];
  bool bad = false;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    int64_t R[8];
    S[a] = to_relative(P[a], R, bad);
    const int64_t u1 = (R[2] - R[1]) + (R[6] - R[3]), u2 = (R[4] - R[2]) + (R[5] - R[6]);
    s1[a] = parts(u1);
    s2[a] = parts(u2);
    t[a] = parts(u1 + u2);
    c1[a] = parts(R[7] - R[2]);
    c2[a] = parts(R[7] - R[4]);
    c3[a] = parts(R[7] - R[1]);
    d1[a] = parts(R[3]);
    d2[a] = parts(R[6]);
    d3[a] = parts(R[5]);
  }
  const int kv = S[0] + S[1] + S[2] + 125;  // 12 V: 2^64 2^64 2^-3
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int k = S[(a + 1) % 3] + S[(a + 2) % 3] + 64;
    bad |= k < -1000 || k > 900;
  }
  bad |= kv < -1000 || kv > 900;
  if (bad) {  // copies: only these need addresses
    double x[8], y[8], z[8], hx[8], hy[8], hz[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) x[c] = X[c], y[c] = Y[c], z[c] = Z[c];
    const double V = hex_grad12_fp64(x, y, z, hx, hy, hz);
#pragma unroll
    for (int c = 0; c < 8; ++c) gx[c] = hx[c], gy[c] = hy[c], gz[c] = hz[c];
    return V;
  }
  int64_t v12 = 0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int b = (a + 1) % 3, c = (a + 2) % 3, k = S[b] + S[c] + 64;
    const int64_t A3 = add_cross(c3, d3, b, c, 0);
    const int64_t p31 = add_cross(d1, c1, b, c, A3);    // A3 - A1
    const int64_t p23 = add_cross(c2, d2, b, c, -A3);   // A2 - A3
    const int64_t p12 = -(p31 + p23);                   // A1 - A2
    const int64_t g1 = add_cross(d3, t, b, c, p31), g3 = add_cross(s1, c1, b, c, p31);
    const int64_t g2 = add_cross(s1, d1, b, c, p12), g6 = add_cross(s2, c2, b, c, p12);
    const int64_t g4 = add_cross(s2, d2, b, c, p23), g5 = add_cross(c3, t, b, c, p23);
    g[a][0] = scaled(__ll2double_rn(-(g3 + g6 + g5)), k);
    g[a][1] = scaled(__ll2double_rn(g1), k);
    g[a][2] = scaled(__ll2double_rn(g2), k);
    g[a][3] = scaled(__ll2double_rn(g3), k);
    g[a][4] = scaled(__ll2double_rn(g4), k);
    g[a][5] = scaled(__ll2double_rn(g5), k);
    g[a][6] = scaled(__ll2double_rn(g6), k);
    g[a][7] = scaled(__ll2double_rn(-(g1 + g2 + g4)), k);
    v12 += sub_products(s2[a], parts(p23 * 8), s1[a], parts(p31 * 8));
  }
  return scaled(__ll2double_rn(__mul64hi(v12, 0x5555555555555556ll)), kv - 2);  // v12 / 3, then / 4
}

// Division of a 32-bit index by a fixed divisor with one multiply-high, an
// add and two shifts (Granlund and Montgomery, "Division by invariant
// integers using multiplication", PLDI 1994): with l = ceil(log2 d) and
// m = floor(2^32 (2^l - d) / d) + 1, x / d = (t + ((x - t) >> s1)) >> s2,
// t = umulhi(m, x), s1 = min(l, 1), s2 = max(l - 1, 0), for every 32-bit x
// and d >= 1. Mesh indices stay below 2^31 (n <= 1024: (n + 1)^3 < 1.1e9), so
// the kernels split them with it instead of 64-bit divisions.
struct FastDiv {
  uint32_t d, m, s1, s2;
};

FastDiv make_fastdiv(uint32_t d) {
  uint32_t l = 0;
  while ((1ull << l) < d) ++l;
  FastDiv f;
  f.d = d;
  f.m = (uint32_t)((((1ull << l) - d) << 32) / d + 1);
  f.s1 = l > 0 ? 1 : 0;
  f.s2 = l > 0 ? l - 1 : 0;
  return f;
}

__device__ __forceinline__ uint32_t fdiv(uint32_t x, const FastDiv &f) {
  const uint32_t t = __umulhi(f.m, x);
  return (t + ((x - t) >> f.s1)) >> f.s2;
}

// Corner positions of element e (lexicographic corner order).
__device__ __forceinline__ void gather(int n, int64_t e, const double *__restrict__ x,
                                       const double *__restrict__ y, const double *__restrict__ z,
                                       double (&X)[8], double (&Y)[8], double (&Z)[8]) {
  const int64_t n1 = n + 1;
  const int64_t i = e % n, j = (e / n) % n, k = e / ((int64_t)n * n);
  const int64_t base = (k * n1 + j) * n1 + i;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int64_t nd = base + ((c >> 2) & 1) * n1 * n1 + ((c >> 1) & 1) * n1 + (c & 1);
    X[c] = x[nd];
    Y[c] = y[nd];
    Z[c] = z[nd];
  }
}

// The same gather for the time-step kernel: element e split by the fixed
// divisor n, node offsets in 32 bits.
__device__ __forceinline__ void gather32(uint32_t e, const FastDiv &fn, const double *__restrict__ x,
                                         const double *__restrict__ y, const double *__restrict__ z,
                                         double (&X)[8], double (&Y)[8], double (&Z)[8]) {
  const uint32_t n = fn.d, n1 = n + 1;
  const uint32_t jk = fdiv(e, fn), i = e - jk * n;
  const uint32_t k = fdiv(jk, fn), j = jk - k * n;
  const uint32_t base = (k * n1 + j) * n1 + i;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int64_t nd = base + ((c >> 2) & 1) * n1 * n1 + ((c >> 1) & 1) * n1 + (c & 1);
    X[c] = x[nd];
    Y[c] = y[nd];
    Z[c] = z[nd];
  }
}

__global__ void __launch_bounds__(128) init_elem_kernel(hpac_hydro_state s) {
  const int n = s.n;
  const int64_t E = (int64_t)n * n * n;
  const double gm1 = s.gamma - 1.0;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < E;
       e += (int64_t)gridDim.x * blockDim.x) {
    double X[8], Y[8], Z[8], gx[8], gy[8], gz[8];
    gather(n, e, s.x, s.y, s.z, X, Y, Z);
    const double V = hex_grad12(X, Y, Z, gx, gy, gz);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      s.grad[(0 * 8 + c) * E + e] = gx[c];
      s.grad[(1 * 8 + c) * E + e] = gy[c];
      s.grad[(2 * 8 + c) * E + e] = gz[c];
    }
    s.V0[e] = V;
    s.rV0[e] = 1.0 / V;
    s.vrel[e] = 1.0;
    s.p[e] = gm1 * s.e[e];
    s.q[e] = 0.0;
    s.pq[e] = s.p[e];
  }
}

__global__ void __launch_bounds__(256) init_node_kernel(hpac_hydro_state s) {
  const int n = s.n;
  const int64_t n1 = n + 1, Nn = n1 * n1 * n1;
  for (int64_t nd = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; nd < Nn;
       nd += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = nd % n1, j = (nd / n1) % n1, k = nd / (n1 * n1);
    double m = 0.0;
    for (int64_t ek = k - 1; ek <= k; ++ek)
      for (int64_t ej = j - 1; ej <= j; ++ej)
        for (int64_t ei = i - 1; ei <= i; ++ei) {
          if (ei < 0 || ej < 0 || ek < 0 || ei >= n || ej >= n || ek >= n) continue;
          m += 0.125 * s.V0[(ek * n + ej) * n + ei];
        }
    s.mnode[nd] = m;
    s.rmass[nd] = 1.0 / (12.0 * m);
    s.u[nd] = s.v[nd] = s.w[nd] = 0.0;
  }
}

// Forces at x^n from (p + q) and the stored gradients; velocity and position.
// Node indices are split by the fixed divisor n + 1 (fn1) in 32 bits.
// An element outside the mesh contributes zeros (predicated loads), so that every
// node runs the same straight-line code with its 32 loads in flight together (80
// registers; with a branch per element the loads went in small groups).
__global__ void __launch_bounds__(256, 3) node_kernel(hpac_hydro_state s, FastDiv fn1) {
  const int n = s.n;
  grid_wait();
  const uint32_t n1 = fn1.d, Nn = n1 * n1 * n1;
  const int64_t E = (int64_t)n * n * n;
  const double dt = s.dt;
  for (uint32_t nd = blockIdx.x * blockDim.x + threadIdx.x; nd < Nn; nd += gridDim.x * blockDim.x) {
    const uint32_t jk = fdiv(nd, fn1), i_ = nd - jk * n1;
    const uint32_t k_ = fdiv(jk, fn1), j_ = jk - k_ * n1;
    const int i = (int)i_, j = (int)j_, k = (int)k_;
    double pq[8], g[8][3];
#pragma unroll
    for (int c = 7; c >= 0; --c) {  // c: corner of this node in the element
      const int ei = i - (c & 1), ej = j - ((c >> 1) & 1), ek = k - (c >> 2);
      const bool in = (unsigned)ei < (unsigned)n && (unsigned)ej < (unsigned)n && (unsigned)ek < (unsigned)n;
      const int64_t el = (int64_t)(((uint32_t)ek * n + (uint32_t)ej) * n + (uint32_t)ei);
      pq[c] = in ? s.pq[el] : 0.0;
#pragma unroll
      for (int d = 0; d < 3; ++d) g[c][d] = in ? s.grad[(d * 8 + c) * E + el] : 0.0;
    }
    // zero pressures (material ahead of a shock) give zero forces whatever the
    // finite gradients are: a warp without any other node skips the FP64 sums,
    // which kept the pipe 87% busy (64^3, 100 steps: 5.47 -> 4.80 ms; 256^3, 20
    // steps with iACT: 64.3 -> 61.7; a warp with such a node pays 60 integer
    // instructions)
    uint32_t live = 0, top = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      live |= ((uint32_t)__double2hiint(pq[c]) << 1) | (uint32_t)__double2loint(pq[c]);
#pragma unroll
      for (int d = 0; d < 3; ++d) top = max(top, (uint32_t)__double2hiint(g[c][d]) & 0x7ff00000u);
    }
    double fx = 0.0, fy = 0.0, fz = 0.0;
    if (__any_sync(__activemask(), live != 0u || top == 0x7ff00000u)) {
#pragma unroll
      for (int c = 7; c >= 0; --c) {
        fx = fma(pq[c], g[c][0], fx);
        fy = fma(pq[c], g[c][1], fy);
        fz = fma(pq[c], g[c][2], fz);
      }
    }
    // the stored gradients are 12 dV/dx: rmass = 1 / (12 m), formed once at
    // init (a double division per node and step would cost a fifth of the
    // kernel's FP64 work)
    const double sc = dt * s.rmass[nd];
    double un = fma(fx, sc, s.u[nd]);
    double vn = fma(fy, sc, s.v[nd]);
    double wn = fma(fz, sc, s.w[nd]);
    if (i == 0) un = 0.0;
    if (j == 0) vn = 0.0;
    if (k == 0) wn = 0.0;
    s.u[nd] = un;
    s.v[nd] = vn;
    s.w[nd] = wn;
    s.x[nd] += dt * un;
    s.y[nd] += dt * vn;
    s.z[nd] += dt * wn;
  }
}

// New volume and gradient, viscosity, and the EOS region's inputs. Element
// indices are split by the fixed divisor n (fn) in 32 bits.
// EXACT: the step evaluates the EOS exactly, so the element's pressure and the
// finalize kernel's updates follow here from registers (as separate launches
// the two took 24 us of a 64^3 step: their loads and stores, and a launch whose
// FP64 work nothing overlaps). With the node kernel's loads in flight together,
// a 64^3 step went from 95.6 to 78.9 us.
template <bool EXACT>
__global__ void __launch_bounds__(128, 4) elem_kernel(hpac_hydro_state s, FastDiv fn, double inv_gm1) {
  const int n = s.n;
  const int64_t E = (int64_t)n * n * n;
  grid_wait();
  const double dt = s.dt, gamma = s.gamma;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < E;
       e += (int64_t)gridDim.x * blockDim.x) {
    double X[8], Y[8], Z[8], gx[8], gy[8], gz[8];
    gather32((uint32_t)e, fn, s.x, s.y, s.z, X, Y, Z);
    const double V = hex_grad12(X, Y, Z, gx, gy, gz);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      s.grad[(0 * 8 + c) * E + e] = gx[c];
      s.grad[(1 * 8 + c) * E + e] = gy[c];
      s.grad[(2 * 8 + c) * E + e] = gz[c];
    }
    // v1 = V / V0 without a division per element and step: exactly 1 for an
    // element at its reference volume (so an unmoved element keeps dv = 0),
    // else V times the stored 1 / V0 (within a rounding of the quotient)
    const double V0e = s.V0[e];
    const double v1 = V == V0e ? 1.0 : V * s.rV0[e];
    const double dv = v1 - s.vrel[e];
    double qn = 0.0;
    if (dv < 0.0) {
      const double L = cbrt(V);
      const double rho = 1.0 / v1;
      const double pp = s.p[e] > 0.0 ? s.p[e] : 0.0;
      const double cs = sqrt(gamma * pp * v1);
      const double du = L * dv / (v1 * dt);
      qn = rho * (kCq * kCq * du * du + kCl * cs * fabs(du));
    }
    const double x[4] = {s.e[e], v1, dv, qn};
#pragma unroll
    for (int d = 0; d < 4; ++d) s.eos_in[d * E + e] = x[d];
    s.q[e] = qn;
    if (EXACT) {
      const double p = Eos64{gamma}(x);
      s.p[e] = p;
      s.e[e] = p * v1 * inv_gm1;
      s.vrel[e] = v1;
      s.pq[e] = p + qn;
    }
  }
}

// inv_gm1 = 1 / (gamma - 1), formed once on the host: a double division per
// thread would cost more than the element update itself.
__global__ void __launch_bounds__(256) finalize_kernel(hpac_hydro_state s, double inv_gm1) {
  grid_wait();
  const int64_t E = (int64_t)s.n * s.n * s.n;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < E;
       e += (int64_t)gridDim.x * blockDim.x) {
    const double v1 = s.eos_in[E + e];
    s.e[e] = s.p[e] * v1 * inv_gm1;
    s.vrel[e] = v1;
    s.pq[e] = s.p[e] + s.q[e];  // the next step's nodal forces use p + q
  }
}

// The derived arrays from the state: pq = p + q and rV0 = 1 / V0 per element,
// rmass = 1 / (12 m) per node.
__global__ void __launch_bounds__(256) derive_kernel(hpac_hydro_state s) {
  const int64_t E = (int64_t)s.n * s.n * s.n, n1 = s.n + 1, Nn = n1 * n1 * n1;
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < (E > Nn ? E : Nn);
       j += (int64_t)gridDim.x * blockDim.x) {
    if (j < E) {
      s.pq[j] = s.p[j] + s.q[j];
      s.rV0[j] = 1.0 / s.V0[j];
    }
    if (j < Nn) s.rmass[j] = 1.0 / (12.0 * s.mnode[j]);
  }
}

unsigned grid_for(int64_t work, int threads, int device) {
  int sms = 148;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  const int64_t want = (work + threads - 1) / threads;
  const int64_t cap = (int64_t)sms * 16;
  return (unsigned)(want < 1 ? 1 : (want > cap ? cap : want));
}

hpac_status check_state(const hpac_hydro_state *s) {
  if (!s) return set_error(HPAC_EINVAL, "hydro state is NULL");
  if (s->n < 1 || s->n > 1024) return set_error(HPAC_EINVAL, "hydro n = %d not in 1..1024", s->n);
  if (s->reserved0 != 0) return set_error(HPAC_EINVAL, "reserved field not zero");
  if (!(s->dt > 0.0) || !isfinite(s->dt)) return set_error(HPAC_EINVAL, "hydro dt must be > 0");
  if (!(s->gamma > 1.0) || !isfinite(s->gamma)) return set_error(HPAC_EINVAL, "gamma must be > 1");
  const void *ptrs[] = {s->x, s->y, s->z, s->u, s->v, s->w, s->mnode, s->e, s->p, s->q, s->vrel,
                        s->V0, s->grad, s->eos_in, s->pq, s->rmass, s->rV0};
  for (const void *p : ptrs)
    if (!p) return set_error(HPAC_EINVAL, "a hydro state array is NULL");
  return HPAC_OK;
}

}  // namespace
}  // namespace hpac

using namespace hpac;

extern "C" hpac_status hpac_hydro_init(const hpac_hydro_state *s, void *cuda_stream) {
  TraceRange trace_("hpac_hydro_init");
  hpac_status st = check_state(s);
  if (st != HPAC_OK) return st;
  int dev = 0;
  HPAC_CUDA_TRY(cudaGetDevice(&dev));
  cudaStream_t stream = (cudaStream_t)cuda_stream;
  const int64_t E = (int64_t)s->n * s->n * s->n, Nn = (int64_t)(s->n + 1) * (s->n + 1) * (s->n + 1);
  init_elem_kernel<<<grid_for(E, 128, dev), 128, 0, stream>>>(*s);
  HPAC_CUDA_TRY(cudaGetLastError());
  init_node_kernel<<<grid_for(Nn, 256, dev), 256, 0, stream>>>(*s);
  HPAC_CUDA_TRY(cudaGetLastError());
  return HPAC_OK;
}

extern "C" hpac_status hpac_hydro_derive(const hpac_hydro_state *s, void *cuda_stream) {
  TraceRange trace_("hpac_hydro_derive");
  hpac_status st = check_state(s);
  if (st != HPAC_OK) return st;
  int dev = 0;
  HPAC_CUDA_TRY(cudaGetDevice(&dev));
  const int64_t Nn = (int64_t)(s->n + 1) * (s->n + 1) * (s->n + 1);
  derive_kernel<<<grid_for(Nn, 256, dev), 256, 0, (cudaStream_t)cuda_stream>>>(*s);
  HPAC_CUDA_TRY(cudaGetLastError());
  return HPAC_OK;
}

extern "C" hpac_status hpac_hydro_nodes(const hpac_hydro_state *s, void *cuda_stream) {
  TraceRange trace_("hpac_hydro_nodes");
  hpac_status st = check_state(s);
  if (st != HPAC_OK) return st;
  int dev = 0;
  HPAC_CUDA_TRY(cudaGetDevice(&dev));
  const int64_t Nn = (int64_t)(s->n + 1) * (s->n + 1) * (s->n + 1);
  HPAC_CUDA_TRY(launch_chained(node_kernel, grid_for(Nn, 256, dev), 256, 0, (cudaStream_t)cuda_stream, *s,
                               make_fastdiv(s->n + 1)));
  return HPAC_OK;
}

template <bool EXACT>
static hpac_status launch_elements(const hpac_hydro_state *s, cudaStream_t stream) {
  const int64_t E = (int64_t)s->n * s->n * s->n;
  // 128 threads, four blocks (16 warps) per SM at 128 registers (4% faster
  // than 136 registers at 96 threads, 15 warps); one element per thread
  const int64_t blocks = (E + 127) / 128;
  HPAC_CUDA_TRY(launch_chained(elem_kernel<EXACT>, (unsigned)(blocks < 0x7fffffffLL ? blocks : 0x7fffffffLL), 128, 0,
                               stream, *s, make_fastdiv(s->n), 1.0 / (s->gamma - 1.0)));
  return HPAC_OK;
}

extern "C" hpac_status hpac_hydro_elements(const hpac_hydro_state *s, void *cuda_stream) {
  TraceRange trace_("hpac_hydro_elements");
  hpac_status st = check_state(s);
  if (st != HPAC_OK) return st;
  return launch_elements<false>(s, (cudaStream_t)cuda_stream);
}

extern "C" hpac_status hpac_hydro_finalize(const hpac_hydro_state *s, void *cuda_stream) {
  TraceRange trace_("hpac_hydro_finalize");
  hpac_status st = check_state(s);
  if (st != HPAC_OK) return st;
  int dev = 0;
  HPAC_CUDA_TRY(cudaGetDevice(&dev));
  const int64_t E = (int64_t)s->n * s->n * s->n;
  HPAC_CUDA_TRY(launch_chained(finalize_kernel, grid_for(E, 256, dev), 256, 0, (cudaStream_t)cuda_stream, *s,
                               1.0 / (s->gamma - 1.0)));
  return HPAC_OK;
}

extern "C" hpac_status hpac_hydro_step(const hpac_hydro_state *s, hpac_region *eos,
                                       int32_t technique, const void *knobs, uint8_t *d_mask,
                                       hpac_stats *h_stats) {
  TraceRange trace_("hpac_hydro_step");
  hpac_status st = check_state(s);
  if (st != HPAC_OK) return st;
  if (!eos) return set_error(HPAC_EINVAL, "EOS region is NULL");
  const int64_t E = (int64_t)s->n * s->n * s->n;
  const hpac_region_desc &d = eos->d;
  if (d.kind != HPAC_REGION_EOS || d.dtype != HPAC_F64 || d.n != E || d.in_stride != E)
    return set_error(HPAC_EINVAL, "EOS region must be kind EOS, F64, n = in_stride = n^3 = %lld",
                     (long long)E);
  if (d.param != s->gamma) return set_error(HPAC_EINVAL, "EOS gamma differs from the hydro gamma");
  if (technique < 0 || technique > 3) return set_error(HPAC_EINVAL, "technique %d", technique);
  if (technique > 0 && !knobs) return set_error(HPAC_EINVAL, "knobs are NULL");
  cudaStream_t stream = eos->stream;
  st = hpac_hydro_nodes(s, stream);
  if (st != HPAC_OK) return st;
  if (technique == 0) {  // elements, exact EOS and finalize in one kernel
    int dev = -1;
    HPAC_CUDA_TRY(cudaGetDevice(&dev));
    if (dev != eos->device)
      return set_error(HPAC_EINVAL, "current device %d differs from the region's device %d", dev, eos->device);
    st = launch_elements<true>(s, stream);
    if (st == HPAC_OK && h_stats) {
      HPAC_CUDA_TRY(cudaStreamSynchronize(stream));
      *h_stats = hpac_stats{E, 0, 0, 0};
    }
    return st;
  }
  st = hpac_hydro_elements(s, stream);
  if (st != HPAC_OK) return st;
  switch (technique) {
    case 1:
      st = hpac_run_taf(eos, static_cast<const hpac_taf_knobs *>(knobs), s->eos_in, s->p, d_mask,
                        nullptr, h_stats);
      break;
    case 2:
      st = hpac_run_iact(eos, static_cast<const hpac_iact_knobs *>(knobs), s->eos_in, s->p, d_mask,
                         nullptr, h_stats);
      break;
    default:
      st = hpac_run_perfo(eos, static_cast<const hpac_perfo_knobs *>(knobs), s->eos_in, s->p,
                          d_mask, h_stats);
      break;
  }
  if (st != HPAC_OK) return st;
  return hpac_hydro_finalize(s, stream);
}

extern "C" hpac_status hpac_hydro_run(const hpac_hydro_state *s, hpac_region *eos, int32_t steps,
                                      int32_t technique, const void *knobs) {
  TraceRange trace_("hpac_hydro_run");
  if (steps < 0) return set_error(HPAC_EINVAL, "steps < 0");
  for (int32_t k = 0; k < steps; ++k) {
    hpac_status st = hpac_hydro_step(s, eos, technique, knobs, nullptr, nullptr);
    if (st != HPAC_OK) return st;
  }
  return HPAC_OK;
}
