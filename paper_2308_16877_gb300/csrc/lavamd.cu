// LavaMD-style neighbour-box forces (Table 1, LavaMD: particle potential and
// forces from the particles of the neighbouring boxes). Section 5 approximates
// the force calculation for a neighbouring box with TAF and iACT and compares
// thread- and warp-level decisions (Figure 9).
//
// One block per home box, one thread per particle of the box (NP of
// ceil(NP / 32) * 32 threads). The block walks the box's neighbour sequence
// (the home box, then the touching boxes in the order dz, dy, dx); at each
// step the neighbour's NP particles are staged in shared memory once for the
// whole block. Each warp then sums the pair terms of its computing lanes'
// particles, four lanes to a particle (box_force), so its cost follows the
// number of particles it computes rather than the slowest lane. A step in
// which no thread of the block computes stages nothing, so decisions taken
// per block drop the step's loads as well as its arithmetic.
//
// TAF: per particle, a window of the last hsize accurate outputs (four
// components) in shared memory, column per thread; the statistic is the RSD
// of the window's potentials; a prediction repeats the newest output.
// iACT: the inputs are the particle's coordinates scaled to single precision;
// tables of tsize slots (scaled coordinates, four outputs) shared by
// 32 / tperwarp lanes; read, decide, execute and write phases with the write
// by the farthest exact lane of each table (a butterfly over its lanes).
// Decisions at warp and block level use the majority rules of the other
// regions (ballots, or block-wide counts at a barrier).
#include <math.h>

#include "exp_fixed.cuh"
#include "hpac_internal.cuh"
#include "regions.cuh"

namespace hpac {
namespace {

enum { LMD_EXACT = 0, LMD_TAF = 1, LMD_IACT = 2 };
constexpr int kMaxParPerBox = 1024;
constexpr int kMaxBoxes1d = 1290;  // B^3 blocks stay below 2^31

struct LmdArgs {
  const double *rq;
  double *fv;
  uint8_t *mask;
  unsigned long long *counters;  // [0] approximated, [1] borderline
  int64_t P;
  int B, NP;
  double na2;  // -a2
  // TAF
  int h, p, reset, thr_inf;
  double thr;
  // iACT
  int tsize, g, L;
  float thr_f;
  double sc[3];
  ExpFixed ex;  // the exponential's tables and constants
};

// Shared memory of a block of NL threads: the staged box (x, y, z, q rows of
// NP doubles), then the TAF windows (h x 4 x NL doubles) or the iACT tables
// (ntab x tsize x 4 output doubles, ntab x tsize x 3 key floats, ntab fill
// counts and ntab round-robin pointers).
__host__ __device__ inline size_t lmd_smem(int tech, int NP, int NL, int h, int tsize, int g) {
  size_t b = (size_t)32 * NP;
  if (tech == LMD_TAF) b += (size_t)32 * h * NL;
  if (tech == LMD_IACT) {
    const size_t ntab = (size_t)(NL / 32) * g;
    b += ntab * tsize * 32 + ((ntab * tsize * 12 + 7) & ~(size_t)7) + ntab * 8;
  }
  return b;
}

// Coordinates on a block's fixed-point grid: F = x 2^(61 - X), |x| < 2^X, where
// X is one binade above the home box's largest coordinate (the touching boxes
// lie within a box side of it; a box with a larger coordinate takes FP64). A
// coordinate down to 2^(X - 9) is exact, a smaller one is rounded to 2^(X - 62)
// unless its last bits are zero. Where FP64 would keep the difference of two such
// coordinates, the grid loses it (thin sheets of particles, clusters beside one
// far particle), so box_force corrects the terms of rounded particles, and a box
// with more than one in eight of them takes FP64.
struct PairGrid {
  int X;
  bool ok;  // the grid and the exponential's scale are in range
};

// X from the largest biased exponent among the home box's coordinates. The
// squared distances in fixed point have an absolute error (below 6 2^(2X - 60),
// zero on average), so the grid is for exponentials that it leaves within half an
// ulp of those of exact distances, a tenth on average: a2 log2(e) < 2^ex,
// ex + 2 X <= 4.
__device__ __forceinline__ PairGrid pair_grid(int emax, int ex) {
  PairGrid g;
  g.X = emax + 1 - 1022;
  g.ok = emax >= 122 && emax <= 1900 && ex + 2 * g.X <= 4;
  return g;
}

__device__ __forceinline__ int biased_exponent(double x) {
  return (int)(((uint32_t)__double2hiint(x) >> 20) & 0x7ffu);
}

// x on the grid; rounds: whether bits of it are lost there.
__device__ __forceinline__ int64_t to_grid(double x, int X, bool &rounds) {
  const uint64_t bits = (uint64_t)__double_as_longlong(x);
  int e = (int)(bits >> 52) & 0x7ff;
  uint64_t m = bits & 0xfffffffffffffull;
  if (e) m |= 1ull << 52;
  else e = 1;
  const int sh = e - 1014 - X;  // (e - 1075) + (61 - X), at most 8
  uint64_t M;
  if (sh >= 0) {
    M = m << sh;
  } else {
    const int r = min(-sh, 63);
    M = (m + (1ull << (r - 1))) >> r;
    rounds |= (m & ((1ull << r) - 1ull)) != 0ull;
  }
  return (int64_t)bits < 0 ? -(int64_t)M : (int64_t)M;
}

__device__ __forceinline__ int64_t to_grid(double x, int X) {
  bool unused = false;
  return to_grid(x, X, unused);
}

// x less its grid value, exact where to_grid rounds x (|x| < 2^(X - 9)).
__device__ __forceinline__ double grid_rest(double x, int X) {
  return x - (double)to_grid(x, X) * __hiloint2double((X - 61 + 1023) << 20, 0);
}

// a 2^(X - 62) with the sign of neg, rounded to nearest even, for a < 2^63
// (twice a grid difference's magnitude).
__device__ __forceinline__ double from_grid(uint64_t a, uint32_t neg, int X) {
  const int lz = __clzll((long long)a);   // 1..64
  const uint64_t m = a << (lz - 1);       // leading one at bit 62
  const uint64_t r = (m + 0x1ffull + ((m >> 10) & 1ull)) >> 10;
  const uint64_t d = r + ((uint64_t)(uint32_t)(1023 + X - lz) << 52);
  return __longlong_as_double((long long)(a ? d | ((uint64_t)neg << 32) : 0ull));
}

// The high 64 bits of a a, at most 3 below the exact value.
__device__ __forceinline__ uint64_t square_hi64(uint64_t a) {
  const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a;
  return (uint64_t)ah * ah + 2ull * __umulhi(ah, al);
}

// What the three squares of a pair lose on average. Without it the exponentials
// of close pairs came out 0.4 units of 2^-53 low on average at the largest scale
// taken (rms 0.50; 0.31 with it, 0.30 with FP64 differences). At r2 = 0 the
// product with the scale is at most 3 and the exponential still 1.
constexpr uint64_t kSquaresLoss = 4;

struct PairExp {  // the exponential's tables (shared memory) and constants
  const uint64_t *ta, *tb;
  uint64_t c;
  int ex;
  uint32_t limit;
};

// exp(-a2 r2) of the grid point at and the staged point m, and the differences dd
// (shift: a2 log2(e) r2 = h 2^(shift - 64)).
__device__ __forceinline__ double grid_pair(const int64_t (&at)[3], const double *sx, const double *sy,
                                            const double *sz, int m, const PairExp &pe, int X, int shift,
                                            double (&dd)[3]) {
  const double *const rows[3] = {sx, sy, sz};
  uint64_t r2 = kSquaresLoss;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int64_t d = at[a] - __double_as_longlong(rows[a][m]);
    const uint32_t neg = (uint32_t)((uint64_t)d >> 32) & 0x80000000u;
    const uint64_t twice = (uint64_t)(d < 0 ? -d : d) << 1;
    r2 += square_hi64(twice);  // in 2^(2X - 60)
    dd[a] = from_grid(twice, neg, X);
  }
  const uint64_t h = mul_hi64(r2, pe.c);
  uint32_t n = 0;
  uint64_t f;
  if (shift > 0) {
    n = (uint32_t)(h >> 32) >> (32 - shift);
    f = h << shift;
  } else {
    f = shift > -64 ? h >> -shift : 0ull;
  }
  return exp_fixed_tail(n, f, pe.ta, pe.tb);
}

// The staged box's particles (rows of stride P at xj), a bit set where the grid
// rounds a coordinate.
struct Rounded {
  const uint32_t *bits;
  const double *xj;
  int64_t P;
};

// The contribution of the staged box to every computing lane's particle,
// computed by the whole warp. The computing lanes' particles go in groups of
// eight; within a group four lanes share a particle, each sums the pair terms
// j = quarter + 4 t, and the four partial sums meet by two shuffle levels. So
// c computing lanes cost the warp ceil(c / 8) ceil(NP / 4) rounds of the pair
// loop, where one lane per particle would cost NP rounds whatever c is: a
// warp with a few computing lanes (thread-level decisions, or the last,
// partly filled warp of a box) is not held for a full pass. Called by all lanes
// of the warp; y is written on the computing lanes only.
// GB300 issues two FP64 operations per SM and clock, so the loop keeps five of
// them per pair: q v and the four sums (the forces' factor 2 is applied to the
// sums). FIXED: the staged coordinates and the particle's are on the block's
// grid, the differences are exact 64-bit integers, rounded once to FP64 for the
// sums; their squares and the exponential stay in fixed point. ROUNDED: a
// particle of the home or the staged box is rounded there, and its rests are
// added. Else the
// differences and r2 are FP64 too (11 operations), and the exponential the
// fixed-point one while the arguments are in its range, the library's otherwise.
// 16^3 boxes of 100 particles under block-level TAF: 34.1 ms with a table-driven
// exponential in FP64 (24 operations per pair), 16.1 with the exponential in
// fixed point (11), 8.5 with the differences too (5).
template <bool FIXED, bool ROUNDED>
__device__ __forceinline__ void box_force(const double *__restrict__ sx, const double *__restrict__ sy,
                                          const double *__restrict__ sz, const double *__restrict__ sq,
                                          int NP, double na2, bool compute, double xp, double yp,
                                          double zp, const PairExp &pe, int X, const Rounded &rounded,
                                          double (&y)[4]) {
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31, sub = lane >> 2, quarter = lane & 3;
  const int shift = pe.ex + 4 + 2 * X;  // FIXED: a2 log2(e) r2 = h 2^(shift - 64)
  unsigned rest = __ballot_sync(kAll, compute);
  while (rest) {
    // this group: the next (up to) eight computing lanes, the s-th on sub-group s
    unsigned group = 0;
    int src = -1;
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      const unsigned low = rest & (0u - rest);
      if (s == sub && low) src = __ffs(low) - 1;
      group |= low;
      rest ^= low;
    }
    const int from = src >= 0 ? src : lane;
    const double px = __shfl_sync(kAll, xp, from), py = __shfl_sync(kAll, yp, from),
                 pz = __shfl_sync(kAll, zp, from);
    double pot = 0.0, fx = 0.0, fy = 0.0, fz = 0.0;
    if (src >= 0 && FIXED) {
      const int64_t at[3] = {to_grid(px, X), to_grid(py, X), to_grid(pz, X)};
#pragma unroll 2
      for (int m = quarter; m < NP; m += 4) {
        double dd[3];
        const double qv = sq[m] * grid_pair(at, sx, sy, sz, m, pe, X, shift, dd);
        pot += qv;
        fx = fma(qv, dd[0], fx);
        fy = fma(qv, dd[1], fy);
        fz = fma(qv, dd[2], fz);
      }
    }
    if (FIXED && ROUNDED) {
      // a difference is that of the grid points plus that of the rests:
      // sum_j q v (rest_i - rest_j) = rest_i pot - sum over rounded j of q v rest_j
      const double at_x[3] = {__shfl_sync(kAll, xp, from), __shfl_sync(kAll, yp, from),
                              __shfl_sync(kAll, zp, from)};
      if (src >= 0) {
        const double rest[3] = {grid_rest(at_x[0], X), grid_rest(at_x[1], X), grid_rest(at_x[2], X)};
        if (rest[0] != 0.0) fx = fma(rest[0], pot, fx);
        if (rest[1] != 0.0) fy = fma(rest[1], pot, fy);
        if (rest[2] != 0.0) fz = fma(rest[2], pot, fz);
        const int64_t at[3] = {to_grid(at_x[0], X), to_grid(at_x[1], X), to_grid(at_x[2], X)};
        for (int w = 0; w < (NP + 31) / 32; ++w)
          for (uint32_t b = rounded.bits[w] & (0x11111111u << quarter); b; b &= b - 1) {
            const int m = 32 * w + __ffs(b) - 1;
            double dd[3];
            const double qv = sq[m] * grid_pair(at, sx, sy, sz, m, pe, X, shift, dd);
            fx = fma(-qv, grid_rest(rounded.xj[m], X), fx);
            fy = fma(-qv, grid_rest(rounded.xj[rounded.P + m], X), fy);
            fz = fma(-qv, grid_rest(rounded.xj[2 * rounded.P + m], X), fz);
          }
      }
    }
    if (src >= 0 && !FIXED) {
#pragma unroll 4
      for (int m = quarter; m < NP; m += 4) {
        const double dx = px - sx[m], dy = py - sy[m], dz = pz - sz[m];
        const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
        double v = exp_fixed(r2, pe.ta, pe.tb, pe.c, pe.ex);
        const bool far = !exp_fixed_in_range(r2, pe.limit);
        if (__any_sync(__activemask(), far)) {
          if (far) v = exp(na2 * r2);
        }
        const double qv = sq[m] * v;
        pot += qv;
        fx = fma(qv, dx, fx);
        fy = fma(qv, dy, fy);
        fz = fma(qv, dz, fz);
      }
    }
#pragma unroll
    for (int off = 1; off < 4; off <<= 1) {
      pot += __shfl_xor_sync(kAll, pot, off);
      fx += __shfl_xor_sync(kAll, fx, off);
      fy += __shfl_xor_sync(kAll, fy, off);
      fz += __shfl_xor_sync(kAll, fz, off);
    }
    fx += fx;  // the pair's force is 2 q v d
    fy += fy;
    fz += fz;
    // each computing lane of the group takes its sub-group's sums
    const bool mine = (group >> lane) & 1u;
    const int at = mine ? 4 * __popc(group & ((1u << lane) - 1u)) : lane;
    const double r0 = __shfl_sync(kAll, pot, at), r1 = __shfl_sync(kAll, fx, at),
                 r2 = __shfl_sync(kAll, fy, at), r3 = __shfl_sync(kAll, fz, at);
    if (mine) {
      y[0] = r0;
      y[1] = r1;
      y[2] = r2;
      y[3] = r3;
    }
  }
}

// Up to 256 particles: 80 registers, so that six blocks of 128 threads share an
// SM instead of five (8.56 -> 8.45 ms under TAF at 16^3 x 100); iACT, which would
// spill half of its decision state, 128 for four blocks. The static shared memory
// is at most the 1 KB that max_dyn_smem() leaves.
template <int TECH, int LEVEL, int MAXT>
__global__ void __launch_bounds__(MAXT, MAXT != 256 ? 1 : TECH != LMD_IACT ? 3 : 2) lavamd_kernel(LmdArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint8_t s_nb[27];  // neighbours: 16 (dz + 1) + 4 (dy + 1) + dx + 1
  __shared__ uint64_t s_ta[32], s_tb[64];
  __shared__ int s_nn, s_emax, s_off[3];
  __shared__ uint32_t s_rounded[32];
  __shared__ unsigned long long s_cnt[2];
  const int tid = threadIdx.x, lane = tid & 31, NL = blockDim.x, NP = a.NP;
  const int64_t hb = blockIdx.x, P = a.P;
  double *sx = reinterpret_cast<double *>(smem_raw);
  double *sy = sx + NP, *sz = sy + NP, *sq = sz + NP;
  double *win = sq + NP;  // TAF windows / iACT table outputs
  const int ntab = TECH == LMD_IACT ? (NL / 32) * a.g : 0;
  float *tkey = reinterpret_cast<float *>(win + (size_t)ntab * a.tsize * 4);
  int *tfill = reinterpret_cast<int *>(
      reinterpret_cast<unsigned char *>(win + (size_t)ntab * a.tsize * 4) +
      (((size_t)ntab * a.tsize * 12 + 7) & ~(size_t)7));
  int *trr = tfill + ntab;

  if (tid == 0) {
    const int B = a.B;
    const int hx = (int)(hb % B), hy = (int)((hb / B) % B), hz = (int)(hb / ((int64_t)B * B));
    int nn = 0;
    s_nb[nn++] = 21;  // the home box
    for (int dz = -1; dz <= 1; ++dz)
      for (int dy = -1; dy <= 1; ++dy)
        for (int dx = -1; dx <= 1; ++dx) {
          if (dx == 0 && dy == 0 && dz == 0) continue;
          const int x = hx + dx, y = hy + dy, z = hz + dz;
          if (x < 0 || y < 0 || z < 0 || x >= B || y >= B || z >= B) continue;
          s_nb[nn++] = (uint8_t)(16 * dz + 4 * dy + dx + 21);
        }
    s_nn = nn;
    s_cnt[0] = s_cnt[1] = 0;
    s_emax = s_off[0] = s_off[1] = s_off[2] = 0;
  }
  if (TECH == LMD_IACT)
    for (int t = tid; t < ntab; t += NL) tfill[t] = trr[t] = 0;
  for (int t = tid; t < 64; t += NL) {
    if (t < 32) s_ta[t] = a.ex.a[t];
    s_tb[t] = a.ex.b[t];
  }
  __syncthreads();

  const bool act = tid < NP;
  const int64_t pidx = hb * NP + tid;
  double xp = 0.0, yp = 0.0, zp = 0.0;
  if (act) {
    xp = a.rq[pidx];
    yp = a.rq[P + pidx];
    zp = a.rq[2 * P + pidx];
  }
  {
    int e = max(max(biased_exponent(xp), biased_exponent(yp)), biased_exponent(zp));
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) atomicMax(&s_emax, e);
  }
  __syncthreads();
  PairGrid grid = pair_grid(s_emax, a.ex.ex);
  bool home_rounds = false;
  to_grid(xp, grid.X, home_rounds);
  to_grid(yp, grid.X, home_rounds);
  to_grid(zp, grid.X, home_rounds);
  const int home_rounded = __syncthreads_count(home_rounds);
  if (8 * home_rounded > NP) grid.ok = false;
  const PairExp pe{s_ta, s_tb, a.ex.c, a.ex.ex, a.ex.limit};
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  unsigned long long n_apx = 0, n_border = 0;
  // TAF state
  int head = 0, cnt = 0, pred = 0;
  const double inv_h = TECH == LMD_TAF ? 1.0 / (double)a.h : 1.0;
  // iACT state: the lane's scaled coordinates and its table
  float z[3] = {0.0f, 0.0f, 0.0f};
  int tab = 0;
  if (TECH == LMD_IACT) {
    tab = (tid >> 5) * a.g + lane / a.L;
    z[0] = __double2float_rn(__dmul_rn(a.sc[0], xp));
    z[1] = __double2float_rn(__dmul_rn(a.sc[1], yp));
    z[2] = __double2float_rn(__dmul_rn(a.sc[2], zp));
  }

  const int nn = s_nn;
  for (int k = 0; k < nn; ++k) {
    const int code = s_nb[k];
    const int b = (int)hb + (((code >> 4) - 1) * a.B + (code >> 2 & 3) - 1) * a.B + (code & 3) - 1;
    double y[4] = {0.0, 0.0, 0.0, 0.0};
    bool compute = act, apx = false;
    // iACT read phase and decision
    float dmin = INFINITY;
    int near = -1;
    if (TECH == LMD_IACT) {
      bool has = false, wants = false;
      if (act) {
        const int f = tfill[tab];
        const float *kt = tkey + (size_t)tab * a.tsize * 3;
        float best = INFINITY;
        for (int j = 0; j < f; ++j) {
          float s = 0.0f;
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const float df = __fsub_rn(z[d], kt[3 * j + d]);
            s = __fadd_rn(s, __fmul_rn(df, df));
          }
          if (near < 0 || s < best) {
            best = s;
            near = j;
          }
        }
        has = f > 0;
        if (has) {
          dmin = __fsqrt_rn(best);
          wants = dmin < a.thr_f;
          if (a.counters && borderline((double)dmin, a.thr)) ++n_border;
        }
      }
      if (LEVEL == HPAC_LEVEL_THREAD) {
        apx = act && wants;
      } else if (LEVEL == HPAC_LEVEL_WARP) {
        const int na = __popc(__ballot_sync(0xffffffffu, act));
        const int nw = __popc(__ballot_sync(0xffffffffu, act && wants));
        apx = 2 * nw > na && act && has;
      } else {
        const int na = __syncthreads_count(act);
        const int nw = __syncthreads_count(act && wants);
        apx = 2 * nw > na && act && has;
      }
      compute = act && !apx;
    }
    const bool predict = TECH == LMD_TAF && act && pred > 0;
    if (TECH == LMD_TAF) compute = act && !predict;

    // execute: stage the neighbour box if any thread computes, on the block's
    // grid unless one of its coordinates lies outside. s_off[k % 3] says so; a
    // slot is cleared two barriers after its last reader.
    bool fixed = grid.ok;
    int box_rounded = 0;
    const bool any = __syncthreads_or(compute);
    if (tid == 0) s_off[(k + 1) % 3] = 0;
    if (any) {
      const int64_t j0 = (int64_t)b * NP;
      double c[3] = {0.0, 0.0, 0.0};
      bool rounds = false;
      if (act) {  // a block has a thread per particle
#pragma unroll
        for (int d = 0; d < 3; ++d) c[d] = a.rq[d * P + j0 + tid];
        const double q = a.rq[3 * P + j0 + tid];
        sq[tid] = q;
        if (grid.ok) {
          // infinite charges, or any that could overflow the potential: the rests'
          // terms would turn infinities into NaN
          if (biased_exponent(q) > 2000) s_off[k % 3] = 1;
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            if (biased_exponent(c[d]) > grid.X + 1022) s_off[k % 3] = 1;
            sx[d * NP + tid] = __longlong_as_double(to_grid(c[d], grid.X, rounds));
          }
        } else {
#pragma unroll
          for (int d = 0; d < 3; ++d) sx[d * NP + tid] = c[d];
        }
      }
      const unsigned word = __ballot_sync(0xffffffffu, rounds);
      if (lane == 0) s_rounded[tid >> 5] = word;
      box_rounded = __syncthreads_count(rounds);
      fixed = grid.ok && s_off[k % 3] == 0 && 8 * box_rounded <= NP;
      if (grid.ok && !fixed) {
        __syncthreads();
        if (act) {
#pragma unroll
          for (int d = 0; d < 3; ++d) sx[d * NP + tid] = c[d];
        }
        __syncthreads();
      }
    }
    const Rounded rounded{s_rounded, a.rq + (int64_t)b * NP, P};
    if (fixed && home_rounded + box_rounded == 0)
      box_force<true, false>(sx, sy, sz, sq, NP, a.na2, compute, xp, yp, zp, pe, grid.X, rounded, y);
    else if (fixed)
      box_force<true, true>(sx, sy, sz, sq, NP, a.na2, compute, xp, yp, zp, pe, grid.X, rounded, y);
    else
      box_force<false, false>(sx, sy, sz, sq, NP, a.na2, compute, xp, yp, zp, pe, grid.X, rounded, y);
    bool decided = false, wants = false;
    if (compute) {
      if (a.mask) a.mask[(int64_t)k * P + pidx] = HPAC_MASK_EXACT;
      if (TECH == LMD_TAF) {
        int slot;
        if (cnt < a.h) {
          slot = head + cnt;
          if (slot >= a.h) slot -= a.h;
          ++cnt;
        } else {
          slot = head;
          head = head + 1 == a.h ? 0 : head + 1;
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) win[(size_t)(slot * 4 + c) * NL + tid] = y[c];
        decided = true;
        if (cnt == a.h) {
          const double s = window_rsd<double>(win + tid, 4 * NL, head, a.h, inv_h);
          if (a.counters && borderline(s, a.thr)) ++n_border;
          wants = a.thr_inf || s < a.thr;
        }
      }
    } else if (predict) {
      int newest = head + cnt - 1;
      if (newest >= a.h) newest -= a.h;
#pragma unroll
      for (int c = 0; c < 4; ++c) y[c] = win[(size_t)(newest * 4 + c) * NL + tid];
      if (a.mask) a.mask[(int64_t)k * P + pidx] = HPAC_MASK_APPROX;
      ++n_apx;
      if (--pred == 0 && a.reset) cnt = 0;
    } else if (apx) {
      const double *yt = win + ((size_t)tab * a.tsize + near) * 4;
#pragma unroll
      for (int c = 0; c < 4; ++c) y[c] = yt[c];
      if (a.mask) a.mask[(int64_t)k * P + pidx] = HPAC_MASK_APPROX;
      ++n_apx;
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[c] += y[c];

    if (TECH == LMD_TAF) {
      // decision at the requested level
      if (LEVEL == HPAC_LEVEL_THREAD) {
        if (decided && wants) pred = a.p;
      } else if (LEVEL == HPAC_LEVEL_WARP) {
        const int nd = __popc(__ballot_sync(0xffffffffu, decided));
        const int nw = __popc(__ballot_sync(0xffffffffu, decided && wants));
        if (2 * nw > nd && decided && cnt == a.h) pred = a.p;
      } else {
        const int nd = __syncthreads_count(decided);
        const int nw = __syncthreads_count(decided && wants);
        if (2 * nw > nd && decided && cnt == a.h) pred = a.p;
      }
    }
    if (TECH == LMD_IACT) {
      // write phase: per table, the exact lane farthest from it (lowest lane
      // on ties) stores its coordinates and outputs in the round-robin slot
      float key = writer_key(compute, dmin, lane, a.L);
      int who = lane;
      for (int off = 1; off < a.L; off <<= 1) {
        const float ok = __shfl_xor_sync(0xffffffffu, key, off);
        const int ow = __shfl_xor_sync(0xffffffffu, who, off);
        if (ok > key || (ok == key && ow < who)) {
          key = ok;
          who = ow;
        }
      }
      if (key >= 0.0f && who == lane) {
        const int s = trr[tab];
        double *yt = win + ((size_t)tab * a.tsize + s) * 4;
        float *kt = tkey + ((size_t)tab * a.tsize + s) * 3;
#pragma unroll
        for (int c = 0; c < 4; ++c) yt[c] = y[c];
#pragma unroll
        for (int d = 0; d < 3; ++d) kt[d] = z[d];
        trr[tab] = s + 1 == a.tsize ? 0 : s + 1;
        if (tfill[tab] < a.tsize) tfill[tab] = tfill[tab] + 1;
      }
      __syncwarp();
    }
  }
  if (act) {
#pragma unroll
    for (int c = 0; c < 4; ++c) a.fv[(int64_t)c * P + pidx] = acc[c];
  }
  if (a.counters) {
    warp_count(s_cnt, n_apx, n_border);
    __syncthreads();
    if (tid == 0) {
      if (s_cnt[0]) atomicAdd(&a.counters[0], s_cnt[0]);
      if (s_cnt[1]) atomicAdd(&a.counters[1], s_cnt[1]);
    }
  }
}

template <int TECH, int LEVEL, int MAXT>
hpac_status launch_one(const LmdArgs &a, int64_t nbox, int NL, size_t smem, cudaStream_t st) {
  auto fn = lavamd_kernel<TECH, LEVEL, MAXT>;
  HPAC_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  fn<<<(unsigned)nbox, NL, smem, st>>>(a);
  HPAC_CUDA_TRY(cudaGetLastError());
  return HPAC_OK;
}

template <int TECH, int MAXT>
hpac_status launch_level(int level, const LmdArgs &a, int64_t nbox, int NL, size_t smem, cudaStream_t st) {
  switch (level) {
    case HPAC_LEVEL_WARP: return launch_one<TECH, HPAC_LEVEL_WARP, MAXT>(a, nbox, NL, smem, st);
    case HPAC_LEVEL_BLOCK: return launch_one<TECH, HPAC_LEVEL_BLOCK, MAXT>(a, nbox, NL, smem, st);
    default: return launch_one<TECH, HPAC_LEVEL_THREAD, MAXT>(a, nbox, NL, smem, st);
  }
}

template <int MAXT>
hpac_status launch_tech(int tech, int level, const LmdArgs &a, int64_t nbox, int NL, size_t smem,
                        cudaStream_t st) {
  if (tech == LMD_TAF) return launch_level<LMD_TAF, MAXT>(level, a, nbox, NL, smem, st);
  if (tech == LMD_IACT) return launch_level<LMD_IACT, MAXT>(level, a, nbox, NL, smem, st);
  return launch_one<LMD_EXACT, HPAC_LEVEL_THREAD, MAXT>(a, nbox, NL, smem, st);
}

}  // namespace
}  // namespace hpac

extern "C" hpac_status hpac_lavamd_run(const hpac_lavamd_desc *desc, int32_t technique,
                                       const void *knobs, const double *d_rq, double *d_fv,
                                       uint8_t *d_mask, hpac_stats *h_stats, void *cuda_stream) {
  using namespace hpac;
  TraceRange trace_("hpac_lavamd_run");
  if (!desc) return set_error(HPAC_EINVAL, "desc is NULL");
  const int B = desc->boxes1d, NP = desc->par_per_box;
  if (B < 0 || B > kMaxBoxes1d) return set_error(HPAC_EINVAL, "boxes1d %d outside 0..%d", B, kMaxBoxes1d);
  if (NP < 1 || NP > kMaxParPerBox)
    return set_error(HPAC_EINVAL, "par_per_box %d outside 1..%d", NP, kMaxParPerBox);
  if (!(desc->a2 >= 0.0) || isinf(desc->a2)) return set_error(HPAC_EINVAL, "a2 must be finite and >= 0");
  if (technique < LMD_EXACT || technique > LMD_IACT) return set_error(HPAC_EINVAL, "technique %d", technique);
  if (technique != LMD_EXACT && !knobs) return set_error(HPAC_EINVAL, "knobs are NULL");
  const int64_t nbox = (int64_t)B * B * B, P = nbox * NP;
  const int NL = (NP + 31) / 32 * 32;
  LmdArgs a{};
  a.ex = exp_fixed_constants(desc->a2);
  a.P = P;
  a.B = B;
  a.NP = NP;
  a.na2 = -desc->a2;
  a.mask = d_mask;
  int level = HPAC_LEVEL_THREAD;
  if (technique == LMD_TAF) {
    const hpac_taf_knobs *k = static_cast<const hpac_taf_knobs *>(knobs);
    if (k->hsize < 1 || k->hsize > kMaxHsize) return set_error(HPAC_EINVAL, "hsize %d", k->hsize);
    if (k->psize < 0) return set_error(HPAC_EINVAL, "psize %d", k->psize);
    if (!(k->thresh >= 0.0)) return set_error(HPAC_EINVAL, "thresh must be >= 0");
    if (k->reset_on_exit != 0 && k->reset_on_exit != 1) return set_error(HPAC_EINVAL, "reset_on_exit");
    level = k->level;
    a.h = k->hsize;
    a.p = k->psize;
    a.reset = k->reset_on_exit;
    a.thr = k->thresh;
    a.thr_inf = isinf(k->thresh) ? 1 : 0;
  } else if (technique == LMD_IACT) {
    const hpac_iact_knobs *k = static_cast<const hpac_iact_knobs *>(knobs);
    if (k->tsize < 1 || k->tsize > kMaxTsize) return set_error(HPAC_EINVAL, "tsize %d", k->tsize);
    const int g = k->tperwarp;
    if (g < 1 || g > 32 || (g & (g - 1)) != 0) return set_error(HPAC_EINVAL, "tperwarp %d", g);
    if (!(k->thresh >= 0.0)) return set_error(HPAC_EINVAL, "thresh must be >= 0");
    level = k->level;
    a.tsize = k->tsize;
    a.g = g;
    a.L = 32 / g;
    a.thr = k->thresh;
    a.thr_f = (float)k->thresh;
    for (int d = 0; d < 3; ++d) a.sc[d] = k->in_scale ? k->in_scale[d] : 1.0;
  }
  if (level < HPAC_LEVEL_THREAD || level > HPAC_LEVEL_BLOCK) return set_error(HPAC_EINVAL, "level %d", level);
  if (h_stats) *h_stats = hpac_stats{0, 0, 0, 0};
  if (P == 0) return HPAC_OK;
  if (!d_rq || !d_fv) return set_error(HPAC_EINVAL, "d_rq or d_fv is NULL");
  if (((uintptr_t)d_rq | (uintptr_t)d_fv) & 7) return set_error(HPAC_EINVAL, "d_rq and d_fv must be 8-byte aligned");
  int dev = 0;
  HPAC_CUDA_TRY(cudaGetDevice(&dev));
  const size_t smem = lmd_smem(technique, NP, NL, a.h, a.tsize, a.g);
  if (smem > (size_t)max_dyn_smem(dev))
    return set_error(HPAC_EINVAL, "the configuration needs %zu bytes of shared memory per block (limit %d)",
                     smem, max_dyn_smem(dev));
  cudaStream_t st = (cudaStream_t)cuda_stream;
  unsigned long long *d_cnt = nullptr;
  if (h_stats) {
    HPAC_CUDA_TRY(cudaMallocAsync((void **)&d_cnt, 2 * sizeof(unsigned long long), st));
    HPAC_CUDA_TRY(cudaMemsetAsync(d_cnt, 0, 2 * sizeof(unsigned long long), st));
  }
  a.counters = d_cnt;
  a.rq = d_rq;
  a.fv = d_fv;
  hpac_status s = NL <= 256 ? launch_tech<256>(technique, level, a, nbox, NL, smem, st)
                            : launch_tech<1024>(technique, level, a, nbox, NL, smem, st);
  if (h_stats) {
    unsigned long long c[2] = {0, 0};
    if (s == HPAC_OK) {
      HPAC_CUDA_TRY(cudaMemcpyAsync(c, d_cnt, sizeof(c), cudaMemcpyDeviceToHost, st));
    }
    HPAC_CUDA_TRY(cudaFreeAsync(d_cnt, st));
    HPAC_CUDA_TRY(cudaStreamSynchronize(st));
    const int64_t per = 3 * (int64_t)B - 2;
    *h_stats = hpac_stats{per * per * per * NP, (int64_t)c[0], 0, (int64_t)c[1]};
  }
  return s;
}
