// Batched knob sweep: many approximation configurations over many
// Black-Scholes regions of uneven sizes in one persistent, graph-captured
// launch (the paper's design-space exploration of Section 2.4 / Section 4,
// Table 2, which builds and runs every configuration separately).
//
// A run first evaluates the region once per option of its regions
// (price_options): the exact output does not depend on the configuration. (One
// configuration over more options than L2 holds evaluates it where needed.) Work
// is then the cross product (region tile, group of configurations). A tile is `tile_blocks` x
// blockDim.x consecutive logical threads of one region, each walking its
// grid-stride invocations i = t + k T_r (Section 3.1.3). Items go band
// by band of tiles, so that the groups of one tile run close together in time
// and reuse its options from L2. A persistent grid takes items from
// one atomic counter (no waits between blocks). For every invocation the
// kernel takes the output under each of the group's configurations - TAF at
// thread level or a perforation pattern - and folds its error against the
// double-precision exact price into per-(configuration, region) sums; no
// per-configuration output array exists.
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "hpac_internal.cuh"
#include "perfo_rule.cuh"
#include "regions.cuh"

struct hpac_sweep {
  int device;
  cudaStream_t user_stream;
  cudaStream_t cap_stream;
  cudaGraph_t graph;
  cudaGraphExec_t exec;
  int n_cfg, n_reg, n_grp;
  void *d_cfg, *d_grp, *d_reg, *d_tile_prefix;
  float4 *d_x4;    // the inputs packed per option: S, K, T, sigma
  float4 *d_ref4;  // the exact prices split: hi, lo, 1/|a|, and the run's region output
  float4 *d_tiny, *d_tiny_terms;
  hpac_sweep_stats *d_stats;
  unsigned long long *d_counter;
};

namespace hpac {
namespace {

struct SweepCfg {
  int tech;      // HPAC_SWEEP_TAF or HPAC_SWEEP_PERFO
  int hsize, psize;
  int thr_inf;
  float thr_f;
  double thr_d;
  DropRule rule;  // lo/hi/T are filled per region on the device
  int m_or_percent;
  int cls;  // configuration class (CLS_*)
  int out;  // the caller's index of this configuration
};

// Consecutive configurations of one class that a work item runs together.
struct SweepGroup {
  int first, count, cls;
};

struct SweepReg {
  int64_t n, off, T;
  int64_t tiles;
};

// The exact price a is held as two floats, hi = fl(a) and lo = fl(a - hi), so
// that the error a - y of a single-precision output comes out in single
// precision as (hi - y) + lo. Prices with |fl(a)| < 1e-30 (deep out-of-the-money
// options) are "tiny": their relative error needs an exponent range single
// precision lacks, so lo instead holds (as integer bits) an index into a
// compact table of {m_hi, m_lo, k} with a = (m_hi + m_lo) 2^k, m_hi in [1, 2)
// (index -1 where a = 0, which carries no relative term). The squared error of
// a tiny price uses d = hi - y, whose square differs from (a - y)^2 only below
// the single-precision range.
__device__ __forceinline__ bool is_tiny(float hi) { return !(fabsf(hi) >= 1e-30f); }

__global__ void count_tiny(const double *__restrict__ ref, int64_t n, unsigned long long *count) {
  unsigned c = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double a = ref[i];
    if (is_tiny((float)a) && a != 0.0) ++c;
  }
  c = __reduce_add_sync(0xffffffffu, c);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(count, (unsigned long long)c);
}

__global__ void split_ref(const double *__restrict__ ref, float4 *__restrict__ ref4,
                          float4 *__restrict__ tiny, unsigned long long *__restrict__ slot,
                          int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double a = ref[i];
    const float h = (float)a;
    const float inv = (float)(1.0 / fabs(a));  // 1/|a| rounded once: the relative term is one multiply
    if (!is_tiny(h)) {
      ref4[i] = make_float4(h, (float)(a - (double)h), inv, 0.0f);
    } else if (a == 0.0) {
      ref4[i] = make_float4(h, __int_as_float(-1), inv, 0.0f);
    } else {
      const unsigned long long j = atomicAdd(slot, 1ull);
      // NaN keeps k = -100 so that its term stays NaN, as in double precision
      const int k = isnan(a) ? -100 : ilogb(a);
      const double m = isnan(a) ? a : ldexp(a, -k);
      const float mh = (float)m;
      tiny[j] = make_float4(mh, (float)(m - (double)mh), __int_as_float(k), 0.0f);
      ref4[i] = make_float4(h, __int_as_float((int)j), inv, 0.0f);
    }
  }
}

// Packs the four input rows into one 16-byte vector per option, so that an
// invocation issues one load for its inputs.
__global__ void pack_inputs(const float *__restrict__ in, int64_t stride, float4 *__restrict__ x4,
                            int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    x4[i] = make_float4(in[i], in[stride + i], in[2 * stride + i], in[3 * stride + i]);
}

// y 2^s for s >= 0, exact whenever representable; +-inf past the float range.
// Integer exponent arithmetic (subnormal y normalised first), no rounding.
__device__ __forceinline__ float scale_up_pow2(float y, int s) {
  unsigned b = __float_as_uint(y);
  const unsigned sign = b & 0x80000000u;
  b &= 0x7fffffffu;
  if (b == 0u || b >= 0x7f800000u) return y;  // zero, inf, NaN
  int e = (int)(b >> 23);
  unsigned m = b & 0x7fffffu;
  if (e == 0) {
    const int lz = __clz((int)m) - 8;  // bring the leading one to bit 23
    m = (m << lz) & 0x7fffffu;
    e = 1 - lz;
  }
  e += s;
  if (e >= 255) return __uint_as_float(sign | 0x7f800000u);
  return __uint_as_float(sign | ((unsigned)e << 23) | m);
}

// (hi, lo) += x with an error-free two-sum: the float pair keeps about 48 bits.
__device__ __forceinline__ void ff_add(float &hi, float &lo, float x) {
  const float s = __fadd_rn(hi, x);
  const float bp = __fsub_rn(s, hi);
  const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(x, bp));
  hi = s;
  lo = __fadd_rn(lo, e);
}

__device__ __forceinline__ void ff_warp_sum(float &hi, float &lo) {
  for (int off = 16; off > 0; off >>= 1) {
    const float oh = __shfl_down_sync(0xffffffffu, hi, off);
    const float ol = __shfl_down_sync(0xffffffffu, lo, off);
    lo = __fadd_rn(lo, ol);
    ff_add(hi, lo, oh);
  }
}

struct ItemSums {
  float rel_hi, rel_lo, sq_hi, sq_lo;
  double rel_wide;  // terms beyond the single-precision range
  unsigned n_alt;
};

// The decision RSD(window) < thr of the TAF kernel on a window stored twice
// over (slot s and s + h hold the same value), so that the h values oldest ..
// newest are the contiguous slots p[0], p[BT], ..., p[(h-1) BT]: the same IEEE
// two-pass moments in the same order, the same guard-banded fast test, and
// the correctly rounded statistic from those moments inside the band.
template <int BT>
__device__ __forceinline__ bool rsd_below_contig(const float *p, int h, float thr, float inv_h) {
  float sum = 0.f;
#pragma unroll 4
  for (int j = 0; j < h; ++j) sum = __fadd_rn(sum, p[j * BT]);
  const float mu = div_count(sum, h, inv_h);
  float acc = 0.f;
#pragma unroll 4
  for (int j = 0; j < h; ++j) {
    const float d = __fsub_rn(p[j * BT], mu);
    acc = __fadd_rn(acc, __fmul_rn(d, d));
  }
  return rsd_below_moments(mu, acc, h, thr, inv_h);
}

// The relative term of output y against a tiny exact price (table entry e):
// |a - y| / |a| = |(m_hi - y 2^-k) + m_lo| / |m_hi| to float precision, or
// `wide` when the ratio needs the double-precision range (the term is then 0).
// Rare, and out of line like wide_term: the sweep kernel's loops are then a
// few hundred instructions each (inlined into every loop they overran the
// instruction cache, and 13 of 20 stalled warps waited for instructions).
__device__ __noinline__ float tiny_term(const float4 &e, float y, bool &wide) {
  const float ys = scale_up_pow2(y, -__float_as_int(e.z));
  wide = !(fabsf(ys) < 1e30f || isnan(ys));
  return wide ? 0.0f : __fdiv_rn(fabsf((e.x - ys) + e.y), fabsf(e.x));
}

// |a - y| / |a| in double precision.
__device__ __noinline__ double wide_term(const double *a_, float y) {
  const double a = *a_;
  return fabs(a - (double)y) / fabs(a);
}

// The region's output of every option, once per run: the exact output depends
// on the option alone, so the configurations share it instead of evaluating
// the region again (110 of the ~180 instructions a configuration spent on an
// option). It goes into the spare fourth word of the option's reference
// record, so that a configuration reads one 16-byte vector per option instead
// of two. A tiny price's relative terms of the accurate output and of a
// dropped one (0) are formed here as well. About 0.17 ms for 21M options, HBM
// bound (48 B per option). Launched over the ranges of options that lie in a
// region: over everything up to the last region's end, 1M options behind a gap of
// 16M took 0.20 ms for one to four configurations.
__global__ void __launch_bounds__(256) price_options(BlackScholes32 reg, const float4 *__restrict__ x4,
                                                     float4 *__restrict__ ref4,
                                                     const float4 *__restrict__ tiny,
                                                     float4 *__restrict__ tiny_terms, int64_t first, int64_t end) {
  for (int64_t i = first + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < end;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float4 v = __ldcs(x4 + i);
    float4 r = ref4[i];
    const float x[4] = {v.x, v.y, v.z, v.w};
    r.w = reg(x);
    ref4[i] = r;
    const int j = __float_as_int(r.y);
    if (is_tiny(r.x) && j >= 0) {
      bool wide, none;
      const float4 e = tiny[j];
      const float exact = tiny_term(e, r.w, wide), dropped = tiny_term(e, 0.0f, none);
      tiny_terms[j] = make_float4(exact, dropped, wide ? 1.0f : 0.0f, 0.0f);
    }
  }
}

// One option as the configurations of a group see it: the difference from the
// exact price (whose square is the squared error) and the factors b c of the
// relative term, for the accurate output (a) and for a dropped one (d).
struct Option {
  float hi, lo, inv, y;
  float da, ba, ca, dd, bd, cd;
  int j;      // tiny prices: table entry, -1 where the exact price is 0
  bool tiny, wide;
};

__device__ __forceinline__ Option read_option(const float4 &r, const float4 *__restrict__ tiny_terms) {
  Option o;
  o.hi = r.x, o.lo = r.y, o.inv = r.z, o.y = r.w;
  o.tiny = is_tiny(r.x);
  o.wide = false;
  o.j = -1;
  o.da = (r.x - r.w) + r.y;
  o.dd = r.x + r.y;
  o.ba = fabsf(o.da), o.bd = fabsf(o.dd);
  o.ca = o.cd = r.z;
  if (o.tiny) {
    o.j = __float_as_int(r.y);
    o.da = r.x - r.w;
    o.dd = r.x;
    o.ba = o.ca = o.bd = o.cd = 0.0f;
    if (o.j >= 0) {
      const float4 t = tiny_terms[o.j];
      o.ba = o.bd = 1.0f;  // fma(1, term, sum) is the rounded sum
      o.ca = t.x, o.cd = t.y;
      o.wide = t.z != 0.0f;
    }
  }
  return o;
}

// How a sweep runs: configurations in groups, or one at a time, from the options
// priced beforehand (FORM_GROUPS, FORM_SINGLES) or pricing them itself (FORM_ONE).
enum { FORM_GROUPS = 0, FORM_SINGLES, FORM_ONE };

// The option of record r without a price (FORM_ONE; with the factors that a
// predicted output takes over), and with it.
__device__ __forceinline__ Option read_reference(const float4 &r) {
  Option o{};
  o.hi = r.x, o.lo = r.y, o.inv = r.z;
  o.tiny = is_tiny(r.x);
  o.j = o.tiny ? __float_as_int(r.y) : -1;
  o.ca = o.tiny ? 0.0f : r.z;
  o.ba = o.j >= 0 ? 1.0f : 0.0f;
  return o;
}

__device__ __forceinline__ void set_price(Option &o, float y, const float4 *__restrict__ tiny) {
  o.y = y;
  if (!o.tiny) {
    o.da = (o.hi - y) + o.lo;
    o.ba = fabsf(o.da);
    o.ca = o.inv;
  } else {
    o.da = o.hi - y;
    o.ba = o.ca = 0.0f;
    if (o.j >= 0) {
      o.ba = 1.0f;
      o.ca = tiny_term(tiny[o.j], y, o.wide);
    }
  }
}

__device__ __forceinline__ void set_dropped(Option &o, const float4 *__restrict__ tiny) {
  o.dd = o.tiny ? o.hi : o.hi + o.lo;
  o.bd = o.tiny ? 0.0f : fabsf(o.dd);
  o.cd = o.tiny ? 0.0f : o.inv;
  if (o.tiny && o.j >= 0) {
    bool none;
    o.bd = 1.0f;
    o.cd = tiny_term(tiny[o.j], 0.0f, none);
  }
}

struct ItemArgs {
  BlackScholes32 reg;
  const float4 *xr, *rr, *tiny, *tiny_terms;  // the region's inputs and records, the tiny table
  const double *r64;                     // the region's exact prices
  int64_t tile;
  int tile_blocks;
};

__device__ __forceinline__ float evaluate(const ItemArgs &A, const float4 &v) {
  const float x[4] = {v.x, v.y, v.z, v.w};
  return A.reg(x);
}

// Errors of C configurations in single precision: sums of 16 terms, each then
// folded into an error-free pair.
template <int C>
struct Errors {
  float rel[C], sq[C];
  int in_chunk;
  __device__ __forceinline__ void init() {
    in_chunk = 0;
#pragma unroll
    for (int c = 0; c < C; ++c) rel[c] = sq[c] = 0.f;
  }
  __device__ __forceinline__ void add(int c, float d, float b, float f) {
    sq[c] = fmaf(d, d, sq[c]);
    rel[c] = fmaf(b, f, rel[c]);
  }
  __device__ __forceinline__ void flush(ItemSums (&acc)[C]) {
#pragma unroll
    for (int c = 0; c < C; ++c) {
      ff_add(acc[c].rel_hi, acc[c].rel_lo, rel[c]);
      ff_add(acc[c].sq_hi, acc[c].sq_lo, sq[c]);
      rel[c] = sq[c] = 0.f;
    }
    in_chunk = 0;
  }
  __device__ __forceinline__ void step(ItemSums (&acc)[C]) {
    if (++in_chunk == 16) flush(acc);
  }
};

// Configuration classes. The configurations of a group share a class, so a
// group runs one specialised loop.
enum { CLS_TAF = 0, CLS_TAF2, CLS_TAF4, CLS_TAF8, CLS_RANGE, CLS_MOD, CLS_RANDOM };
constexpr int kMaxGroup = 4;

// C TAF configurations over `tile_blocks` x BT logical threads of region R.
// KH > 0: their history size, the windows in registers; KH = 0 (C = 1): a
// window in shared memory, stored twice over. Idx is the index type (32-bit
// when every offset fits). A region whose threads have fewer invocations than
// the history size never fills a window, so no window is kept there.
template <int BT, int KH, int C, bool PRICED, typename Idx>
__device__ __forceinline__ void taf_item(const SweepCfg *__restrict__ cfg, int count, const SweepReg &R,
                                         const ItemArgs &A, float *win, ItemSums (&acc)[C],
                                         unsigned &n_inv, unsigned &n_used) {
  const Idx n = (Idx)R.n, T = (Idx)R.T;
  const int h = KH > 0 ? KH : cfg[0].hsize;
  const float inv_h = 1.0f / (float)h;
  const bool fills = (R.n + R.T - 1) / R.T >= h;
  float thr[C];
  int thr_inf[C], psize[C];
#pragma unroll
  for (int c = 0; c < C; ++c) {
    const SweepCfg &K = cfg[c < count ? c : 0];
    thr[c] = K.thr_f, thr_inf[c] = K.thr_inf, psize[c] = K.psize;
  }
  Errors<C> err;
  err.init();
  for (int lb = 0; lb < A.tile_blocks; ++lb) {
    const int64_t t64 = (A.tile * A.tile_blocks + lb) * (int64_t)BT + threadIdx.x;
    if (t64 >= R.T) break;  // later logical blocks of this tile are past T too
    float w[C][KH > 0 ? KH : 1];
    int pos = 0, cnt[C], pred[C];
#pragma unroll
    for (int c = 0; c < C; ++c) {
      cnt[c] = pred[c] = 0;
#pragma unroll
      for (int j = 0; j < (KH > 0 ? KH : 1); ++j) w[c][j] = 0.f;
    }
    const Idx t = (Idx)t64;
    float4 next = make_float4(0.f, 0.f, 0.f, 0.f), next_x = next;
    if (t < n) next = A.rr[t];
    if (!PRICED && t < n) next_x = A.xr[t];
    for (Idx i = t; i < n; i += T) {
      const float4 r = next, x = next_x;
      if (i + T < n) next = A.rr[i + T];
      if (!PRICED && i + T < n && pred[0] < 2) next_x = A.xr[i + T];
      Option o = PRICED ? read_option(r, A.tiny_terms) : read_reference(r);
      ++n_inv;
      n_used += !o.tiny || o.j >= 0;
#pragma unroll
      for (int c = 0; c < C; ++c) {
        float d = o.da, b = o.ba, f = o.ca;
        if (pred[c] > 0) {  // the newest window value
          const float y = KH > 0 ? w[c][KH > 0 ? KH - 1 : 0] : win[(pos + h - 1) * BT + threadIdx.x];
          --pred[c];
          ++acc[c].n_alt;
          if (!o.tiny) {
            d = (o.hi - y) + o.lo;
            b = fabsf(d);
          } else {
            d = o.hi - y;
            if (o.j >= 0) {
              bool wide;
              f = tiny_term(A.tiny[o.j], y, wide);
              if (wide) acc[c].rel_wide += wide_term(A.r64 + i, y);  // a ratio past 1e30
            }
          }
        } else {
          if (!PRICED) {  // one configuration
            set_price(o, evaluate(A, x), A.tiny);
            d = o.da, b = o.ba, f = o.ca;
          }
          if (fills) {
            if (KH > 0) {
#pragma unroll
              for (int j = 0; j + 1 < KH; ++j) w[c][j] = w[c][j + 1];
              w[c][KH > 0 ? KH - 1 : 0] = o.y;
            } else {
              win[pos * BT + threadIdx.x] = o.y;
              win[(pos + h) * BT + threadIdx.x] = o.y;
              pos = (pos + 1 == h) ? 0 : pos + 1;
            }
            cnt[c] = cnt[c] < h ? cnt[c] + 1 : h;
            if (cnt[c] == h) {
              bool wants = thr_inf[c] != 0;
              if (!wants) {
                if constexpr (KH > 0) {
                  float mu, dev;
                  reg_window_moments(w[c], inv_h, mu, dev);
                  wants = rsd_below_moments(mu, dev, KH, thr[c], inv_h);
                } else {
                  wants = rsd_below_contig<BT>(win + pos * BT + threadIdx.x, h, thr[c], inv_h);
                }
              }
              if (wants) pred[c] = psize[c];
            }
          }
          if (o.wide) acc[c].rel_wide += wide_term(A.r64 + i, o.y);
        }
        err.add(c, d, b, f);
      }
      err.step(acc);
    }
  }
  err.flush(acc);
}

// C perforation configurations of one class over the same logical threads.
template <int BT, int CLS, int C, bool PRICED, typename Idx>
__device__ __forceinline__ void perfo_item(const SweepCfg *__restrict__ cfg, int count, const SweepReg &R,
                                           const ItemArgs &A, ItemSums (&acc)[C], unsigned &n_inv,
                                           unsigned &n_used) {
  const Idx n = (Idx)R.n, T = (Idx)R.T;
  // ini / fini: kept range; small / large: residues of the key modulo M
  // advanced incrementally (key k with step 1 when herded, i with step T
  // otherwise)
  Idx keep_lo[C], keep_hi[C];
  unsigned m[C], inc[C];
  bool herded[C], small[C];
  // random: a herded pattern's decisions for the first 64 steps, hashed once
  // per item by the lanes of the warp; later steps and per-invocation
  // patterns hash their key
  uint64_t seed[C], bits[C];
  uint32_t cut[C];
#pragma unroll
  for (int c = 0; c < C; ++c) {
    const SweepCfg &K = cfg[c < count ? c : 0];
    keep_lo[c] = 0, keep_hi[c] = n;
    m[c] = 1, inc[c] = 0;
    seed[c] = bits[c] = 0;
    cut[c] = 0;
    herded[c] = K.rule.herded != 0;
    small[c] = K.rule.kind == HPAC_PERFO_SMALL;
    if (CLS == CLS_RANGE) {
      const int64_t range = (R.n * (int64_t)K.m_or_percent) / 100;
      if (K.rule.kind == HPAC_PERFO_INI) keep_lo[c] = (Idx)range;
      if (K.rule.kind == HPAC_PERFO_FINI) keep_hi[c] = (Idx)(R.n - range);
    }
    if (CLS == CLS_RANDOM) {
      seed[c] = K.rule.seed;
      cut[c] = K.rule.cut;
      if (herded[c]) {
        const uint64_t l = threadIdx.x & 31;
        const unsigned b0 = __ballot_sync(0xffffffffu, (uint32_t)(splitmix64(seed[c] ^ l) >> 40) < cut[c]);
        const unsigned b1 =
            __ballot_sync(0xffffffffu, (uint32_t)(splitmix64(seed[c] ^ (l + 32)) >> 40) < cut[c]);
        bits[c] = (uint64_t)b1 << 32 | b0;
      }
    }
    if (CLS == CLS_MOD) {
      m[c] = (unsigned)K.rule.m;
      inc[c] = herded[c] ? 1u % m[c] : (unsigned)(R.T % (int64_t)m[c]);
    }
  }
  Errors<C> err;
  err.init();
  for (int lb = 0; lb < A.tile_blocks; ++lb) {
    const int64_t t64 = (A.tile * A.tile_blocks + lb) * (int64_t)BT + threadIdx.x;
    if (t64 >= R.T) break;
    const Idx t = (Idx)t64;
    unsigned res[C];
#pragma unroll
    for (int c = 0; c < C; ++c) res[c] = CLS != CLS_MOD || herded[c] ? 0u : (unsigned)(t64 % (int64_t)m[c]);
    auto dropped = [&](int c, Idx i, Idx k) {  // once per step, in order
      if (CLS == CLS_RANGE) return (i < keep_lo[c]) || (i >= keep_hi[c]);
      if (CLS == CLS_MOD) {
        const bool drop = small[c] ? res[c] == m[c] - 1u : res[c] != 0u;
        res[c] += inc[c];
        res[c] = res[c] >= m[c] ? res[c] - m[c] : res[c];
        return drop;
      }
      if (herded[c] && k < 64) return ((bits[c] >> k) & 1ull) != 0;
      return (uint32_t)(splitmix64(seed[c] ^ (uint64_t)(herded[c] ? k : i)) >> 40) < cut[c];
    };
    float4 next = make_float4(0.f, 0.f, 0.f, 0.f), next_x = next;
    bool next_drop = true;
    if (t < n) next = A.rr[t];
    if (!PRICED && t < n) {
      next_drop = dropped(0, t, 0);
      if (!next_drop) next_x = A.xr[t];
    }
    Idx k = 0;
    for (Idx i = t; i < n; i += T, ++k) {
      const float4 r = next, x = next_x;
      const bool drop0 = next_drop;
      if (i + T < n) next = A.rr[i + T];
      if (!PRICED && i + T < n) {
        next_drop = dropped(0, i + T, k + 1);
        if (!next_drop) next_x = A.xr[i + T];
      }
      Option o = PRICED ? read_option(r, A.tiny_terms) : read_reference(r);
      ++n_inv;
      n_used += !o.tiny || o.j >= 0;
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const bool drop = PRICED ? dropped(c, i, k) : drop0;
        acc[c].n_alt += drop;
        if (!PRICED) {  // one configuration
          if (drop)
            set_dropped(o, A.tiny);
          else
            set_price(o, evaluate(A, x), A.tiny);
        }
        // a dropped output keeps the (zero) prefill
        err.add(c, drop ? o.dd : o.da, drop ? o.bd : o.ba, drop ? o.cd : o.ca);
        if (o.wide && !drop) acc[c].rel_wide += wide_term(A.r64 + i, o.y);
      }
      err.step(acc);
    }
  }
  err.flush(acc);
}

// Warp sums of an item's C configurations into s_warp[c][warp].
template <int C, int W>
__device__ __forceinline__ void warp_sums(ItemSums (&acc)[C], ItemSums (&s_warp)[kMaxGroup][W]) {
#pragma unroll
  for (int c = 0; c < C; ++c) {
    ff_warp_sum(acc[c].rel_hi, acc[c].rel_lo);
    ff_warp_sum(acc[c].sq_hi, acc[c].sq_lo);
    acc[c].n_alt = __reduce_add_sync(0xffffffffu, acc[c].n_alt);
    if (__any_sync(0xffffffffu, acc[c].rel_wide != 0.0))
      for (int off = 16; off > 0; off >>= 1)
        acc[c].rel_wide += __shfl_down_sync(0xffffffffu, acc[c].rel_wide, off);
    if ((threadIdx.x & 31) == 0) s_warp[c][threadIdx.x >> 5] = acc[c];
  }
}

// Bound by instruction issue (66% of the cycles issue, the integer and select
// pipe 62% busy): about 73 warp instructions per 32 (configuration, option)
// pairs against 220 when every configuration evaluated the region. 256
// configurations x 21M options: 12.85 ms (37.6 ms before). 64 registers, 1024
// threads per SM: 12.8 ms, against 12.9 at 896, 13.8 at 768, 15.0 at 640 and
// 17.3 ms at 512 threads per SM, although the smaller ones spill nothing.
// FORM_SINGLES: every group has one configuration, whose loop runs no copies of
// it. 21M options, two, three and four configurations of different classes: 433, 570
// and 747 us when each evaluated the region, 464, 579 and 725 with copies, 375, 440
// and 494 now; 256K options 56, 53 and 54, 46, 46 and 51, 33, 34 and 33.
template <int BT, typename Idx, int FORM>
__global__ void __launch_bounds__(BT, 1024 / BT) sweep_kernel(
    const SweepCfg *__restrict__ cfgs, const SweepGroup *__restrict__ groups, int n_grp,
    const SweepReg *__restrict__ regs, int n_reg, const int64_t *__restrict__ tile_prefix, int64_t n_tiles,
    int band, int tile_blocks, BlackScholes32 reg, const float4 *__restrict__ x4, const float4 *__restrict__ ref4,
    const float4 *__restrict__ tiny, const float4 *__restrict__ tiny_terms, const double *__restrict__ ref64,
    hpac_sweep_stats *__restrict__ stats, unsigned long long *__restrict__ counter) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float *win = reinterpret_cast<float *>(smem_raw);
  constexpr int W = BT / 32;
  __shared__ long long s_item, s_tile;
  __shared__ int s_reg, s_grp;
  __shared__ ItemSums s_warp[kMaxGroup][W];
  __shared__ unsigned s_inv[W], s_used[W];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t n_items = n_tiles * n_grp;
  for (;;) {
    __syncthreads();  // everyone has read the previous item and its sums
    if (threadIdx.x == 0) {
      const long long item = (long long)atomicAdd(counter, 1ull);
      int r = 0;
      if (item < n_items) {
        // band of `band` tiles, then group, then tile (the last band is short)
        const int64_t per = (int64_t)band * n_grp, b = item / per, rest = item - b * per;
        const int64_t in_band = n_tiles - b * band < band ? n_tiles - b * band : band;
        const int64_t g = b * band + rest % in_band;
        s_grp = (int)(rest / in_band);
        s_tile = g;
        int lo = 0, hi = n_reg - 1;  // last r with tile_prefix[r] <= g
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if (tile_prefix[mid] <= g) lo = mid; else hi = mid - 1;
        }
        r = lo;
      }
      s_item = item;
      s_reg = r;
    }
    __syncthreads();
    const long long item = s_item;
    if (item >= n_items) break;
    const SweepGroup G = groups[s_grp];
    const int r = s_reg;
    const SweepReg R = regs[r];
    const ItemArgs A{reg, x4 + R.off, ref4 + R.off, tiny, tiny_terms, ref64 + R.off, s_tile - tile_prefix[r], tile_blocks};
    const SweepCfg *cfg = cfgs + G.first;
    unsigned n_inv = 0, n_used = 0;
    constexpr bool kPriced = FORM != FORM_ONE;
    constexpr int kTaf = FORM == FORM_GROUPS ? 2 : 1, kPerfo = FORM == FORM_GROUPS ? 4 : 1;
    switch (G.cls) {
      case CLS_TAF2: {
        ItemSums acc[kTaf] = {};
        taf_item<BT, 2, kTaf, kPriced, Idx>(cfg, G.count, R, A, win, acc, n_inv, n_used);
        warp_sums(acc, s_warp);
        break;
      }
      case CLS_TAF4: {
        ItemSums acc[kTaf] = {};
        taf_item<BT, 4, kTaf, kPriced, Idx>(cfg, G.count, R, A, win, acc, n_inv, n_used);
        warp_sums(acc, s_warp);
        break;
      }
      case CLS_TAF8: {
        ItemSums acc[kTaf] = {};
        taf_item<BT, 8, kTaf, kPriced, Idx>(cfg, G.count, R, A, win, acc, n_inv, n_used);
        warp_sums(acc, s_warp);
        break;
      }
      case CLS_RANGE: {
        ItemSums acc[kPerfo] = {};
        perfo_item<BT, CLS_RANGE, kPerfo, kPriced, Idx>(cfg, G.count, R, A, acc, n_inv, n_used);
        warp_sums(acc, s_warp);
        break;
      }
      case CLS_MOD: {
        ItemSums acc[kPerfo] = {};
        perfo_item<BT, CLS_MOD, kPerfo, kPriced, Idx>(cfg, G.count, R, A, acc, n_inv, n_used);
        warp_sums(acc, s_warp);
        break;
      }
      case CLS_RANDOM: {
        ItemSums acc[kPerfo] = {};
        perfo_item<BT, CLS_RANDOM, kPerfo, kPriced, Idx>(cfg, G.count, R, A, acc, n_inv, n_used);
        warp_sums(acc, s_warp);
        break;
      }
      default: {
        ItemSums acc[1] = {};
        taf_item<BT, 0, 1, kPriced, Idx>(cfg, G.count, R, A, win, acc, n_inv, n_used);
        warp_sums(acc, s_warp);
      }
    }
    n_inv = __reduce_add_sync(0xffffffffu, n_inv);
    n_used = __reduce_add_sync(0xffffffffu, n_used);
    if (lane == 0) {
      s_inv[wid] = n_inv;
      s_used[wid] = n_used;
    }
    __syncthreads();
    // one atomic set per configuration of the item
    if ((int)threadIdx.x < G.count) {
      const int c = threadIdx.x;
      ItemSums a = s_warp[c][0];
      n_inv = s_inv[0];
      n_used = s_used[0];
      for (int w = 1; w < W; ++w) {
        const ItemSums &b = s_warp[c][w];
        a.rel_lo = __fadd_rn(a.rel_lo, b.rel_lo);
        ff_add(a.rel_hi, a.rel_lo, b.rel_hi);
        a.sq_lo = __fadd_rn(a.sq_lo, b.sq_lo);
        ff_add(a.sq_hi, a.sq_lo, b.sq_hi);
        a.rel_wide += b.rel_wide;  // zero unless some term needed double range
        a.n_alt += b.n_alt;
        n_inv += s_inv[w];
        n_used += s_used[w];
      }
      hpac_sweep_stats *o = stats + (size_t)cfg[c].out * n_reg + r;
      atomicAdd(&o->sum_abs_rel, ((double)a.rel_hi + (double)a.rel_lo) + a.rel_wide);
      atomicAdd(&o->sum_sq, (double)a.sq_hi + (double)a.sq_lo);
      atomicAdd((unsigned long long *)&o->invocations, (unsigned long long)n_inv);
      atomicAdd((unsigned long long *)(G.cls <= CLS_TAF8 ? &o->approximated : &o->skipped),
                (unsigned long long)a.n_alt);
      atomicAdd((unsigned long long *)&o->mape_terms, (unsigned long long)n_used);
    }
  }
}

// set_only: raise the kernel's dynamic shared memory limit (outside capture);
// otherwise launch it on the capture stream.
template <int BT, typename Idx, int FORM>
cudaError_t launch_form(bool set_only, hpac_sweep *p, unsigned grid, size_t smem, int64_t n_tiles,
                        int band, int tile_blocks, const double *d_ref, BlackScholes32 reg) {
  auto fn = sweep_kernel<BT, Idx, FORM>;
  if (set_only) return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  fn<<<grid, BT, smem, p->cap_stream>>>(
      (const SweepCfg *)p->d_cfg, (const SweepGroup *)p->d_grp, p->n_grp, (const SweepReg *)p->d_reg,
      p->n_reg, (const int64_t *)p->d_tile_prefix, n_tiles, band, tile_blocks, reg, p->d_x4, p->d_ref4, p->d_tiny,
      p->d_tiny_terms, d_ref, p->d_stats, p->d_counter);
  return cudaGetLastError();
}

template <int BT, typename Idx, class... A>
cudaError_t launch_sweep(int form, A... args) {
  return form == FORM_ONE       ? launch_form<BT, Idx, FORM_ONE>(args...)
         : form == FORM_SINGLES ? launch_form<BT, Idx, FORM_SINGLES>(args...)
                                : launch_form<BT, Idx, FORM_GROUPS>(args...);
}

void free_plan(hpac_sweep *p) {
  if (!p) return;
  if (p->exec) cudaGraphExecDestroy(p->exec);
  if (p->graph) cudaGraphDestroy(p->graph);
  if (p->cap_stream) cudaStreamDestroy(p->cap_stream);
  cudaFree(p->d_cfg);
  cudaFree(p->d_grp);
  cudaFree(p->d_reg);
  cudaFree(p->d_tile_prefix);
  cudaFree(p->d_x4);
  cudaFree(p->d_ref4);
  cudaFree(p->d_tiny);
  cudaFree(p->d_tiny_terms);
  cudaFree(p->d_stats);
  cudaFree(p->d_counter);
  free(p);
}

}  // namespace
}  // namespace hpac

using namespace hpac;

extern "C" hpac_status hpac_sweep_create(int32_t n_configs, const hpac_sweep_config *h_configs,
                                         int32_t n_regions, const hpac_sweep_region *h_regions,
                                         const float *d_in, int64_t in_stride,
                                         const double *d_ref, double rate, int32_t block_threads,
                                         int32_t blocks_per_sm, int32_t tile_blocks,
                                         void *cuda_stream, hpac_sweep **out) {
  if (!out) return set_error(HPAC_EINVAL, "out is NULL");
  *out = nullptr;
  if (n_configs < 1 || n_regions < 1 || !h_configs || !h_regions || !d_in || !d_ref)
    return set_error(HPAC_EINVAL, "empty sweep or NULL pointer");
  if (block_threads != 64 && block_threads != 128 && block_threads != 256)
    return set_error(HPAC_EINVAL, "block_threads must be 64, 128 or 256");
  if (blocks_per_sm < 1 || blocks_per_sm > 32 || tile_blocks < 1 || tile_blocks > 64)
    return set_error(HPAC_EINVAL, "blocks_per_sm in 1..32, tile_blocks in 1..64");
  if (!isfinite(rate)) return set_error(HPAC_EINVAL, "rate is not finite");
  std::vector<SweepCfg> cfg(n_configs);
  int hmax = 0;  // largest history size whose window is in shared memory
  for (int c = 0; c < n_configs; ++c) {
    const hpac_sweep_config &k = h_configs[c];
    SweepCfg &s = cfg[c];
    memset(&s, 0, sizeof(s));
    s.tech = k.technique;
    s.out = c;
    if (k.technique == HPAC_SWEEP_TAF) {
      if (k.hsize < 1 || k.hsize > kMaxHsize || k.psize < 0 || !(k.thresh >= 0.0))
        return set_error(HPAC_EINVAL, "config %d: bad TAF knobs", c);
      if (k.level != HPAC_LEVEL_THREAD)
        return set_error(HPAC_EUNSUPPORTED, "config %d: the sweep runs TAF at thread level", c);
      s.hsize = k.hsize;
      s.psize = k.psize;
      s.thr_f = (float)k.thresh;
      s.thr_d = k.thresh;
      s.thr_inf = isinf(k.thresh) ? 1 : 0;
      s.cls = k.hsize == 2 ? CLS_TAF2 : k.hsize == 4 ? CLS_TAF4 : k.hsize == 8 ? CLS_TAF8 : CLS_TAF;
      if (s.cls == CLS_TAF) hmax = k.hsize > hmax ? k.hsize : hmax;
    } else if (k.technique == HPAC_SWEEP_PERFO) {
      const int pk = k.perfo_kind;
      if (pk < HPAC_PERFO_SMALL || pk > HPAC_PERFO_RANDOM)
        return set_error(HPAC_EINVAL, "config %d: perforation kind %d", c, pk);
      if ((pk == HPAC_PERFO_SMALL || pk == HPAC_PERFO_LARGE) && k.m_or_percent < 1)
        return set_error(HPAC_EINVAL, "config %d: M < 1", c);
      if ((pk == HPAC_PERFO_INI || pk == HPAC_PERFO_FINI) &&
          (k.m_or_percent < 0 || k.m_or_percent > 100))
        return set_error(HPAC_EINVAL, "config %d: percent not in 0..100", c);
      if (pk == HPAC_PERFO_RANDOM && !(k.rate >= 0.0 && k.rate <= 1.0))
        return set_error(HPAC_EINVAL, "config %d: rate not in [0,1]", c);
      s.rule.kind = pk;
      s.rule.herded = k.herded ? 1 : 0;
      s.rule.m = k.m_or_percent;
      s.rule.seed = k.seed;
      s.rule.cut = (uint32_t)floor(k.rate * 16777216.0);
      s.m_or_percent = k.m_or_percent;
      s.cls = pk == HPAC_PERFO_RANDOM                           ? CLS_RANDOM
              : pk == HPAC_PERFO_INI || pk == HPAC_PERFO_FINI ? CLS_RANGE
                                                              : CLS_MOD;
    } else {
      return set_error(HPAC_EINVAL, "config %d: technique %d", c, k.technique);
    }
  }
  // Configurations of a class run in groups: an option's record is read once
  // per group (one 16-byte vector from L2 per option and configuration would
  // need 9.6 TB/s at the speed the arithmetic reaches), and the independent
  // configurations hide each other's latency. Four perforation configurations
  // or two TAF windows in registers; a window in shared memory runs alone, so
  // that the shared memory of a block stays what one window needs.
  std::stable_sort(cfg.begin(), cfg.end(), [](const SweepCfg &a, const SweepCfg &b) {
    return a.cls != b.cls ? a.cls < b.cls : a.rule.herded < b.rule.herded;
  });
  std::vector<SweepGroup> grp;
  for (int c = 0; c < n_configs; ++c) {
    const int cls = cfg[c].cls, most = cls == CLS_TAF ? 1 : cls <= CLS_TAF8 ? 2 : kMaxGroup;
    if (grp.empty() || grp.back().cls != cls || grp.back().count == most)
      grp.push_back(SweepGroup{c, 0, cls});
    ++grp.back().count;
  }
  bool singles = true;
  for (const SweepGroup &g : grp) singles = singles && g.count == 1;
  std::vector<SweepReg> reg(n_regions);
  std::vector<int64_t> prefix(n_regions + 1, 0);
  int64_t total = 0;
  const int64_t lt = (int64_t)block_threads * tile_blocks;
  for (int r = 0; r < n_regions; ++r) {
    const hpac_sweep_region &g = h_regions[r];
    if (g.n < 1 || g.offset < 0 || g.offset + g.n > in_stride || g.logical_threads < 0)
      return set_error(HPAC_EINVAL, "region %d: bad size, offset or logical threads", r);
    reg[r].n = g.n;
    reg[r].off = g.offset;
    reg[r].T = g.logical_threads > 0 ? g.logical_threads : g.n;
    reg[r].tiles = (reg[r].T + lt - 1) / lt;
    // per-item counts are 32-bit: a work item covers fewer than 2^32 invocations
    if ((double)lt * (double)((g.n + reg[r].T - 1) / reg[r].T) >= 4294967295.0)
      return set_error(HPAC_EUNSUPPORTED, "region %d: a work item would exceed 2^32 invocations", r);
    prefix[r + 1] = prefix[r] + reg[r].tiles;
    total = total > g.offset + g.n ? total : g.offset + g.n;
  }
  const int64_t n_tiles = prefix[n_regions];
  // The ranges of options that lie in a region, to be priced in a launch each: a
  // gap of less than 64K options is priced along (0.5 us), and where more than
  // eight ranges are left, larger ones.
  std::vector<std::pair<int64_t, int64_t>> used, ranges;
  for (const SweepReg &g : reg) used.emplace_back(g.off, g.off + g.n);
  std::sort(used.begin(), used.end());
  for (int64_t gap = 65536; ranges.empty() || ranges.size() > 8; gap *= 2) {
    ranges.clear();
    for (const auto &u : used) {
      if (!ranges.empty() && u.first - ranges.back().second < gap)
        ranges.back().second = std::max(ranges.back().second, u.second);
      else
        ranges.push_back(u);
    }
  }
  // Items go band by band of tiles, and within a band group by group: the
  // blocks of an SM then run the same class's loop most of the time (with the
  // groups innermost they ran all classes at once), while the band's records,
  // at most 32 MB, stay in L2 for the next group.
  int64_t tile_bytes = 1;
  for (int r = 0; r < n_regions; ++r) {
    const int64_t b = 16 * lt * ((reg[r].n + reg[r].T - 1) / reg[r].T);
    tile_bytes = tile_bytes > b ? tile_bytes : b;
  }
  int64_t band = (32ll << 20) / tile_bytes;
  band = band < 64 ? 64 : band > 65536 ? 65536 : band;
  hpac_sweep *p = (hpac_sweep *)calloc(1, sizeof(hpac_sweep));
  if (!p) return set_error(HPAC_ENOMEM, "host allocation failed");
  p->n_cfg = n_configs;
  p->n_reg = n_regions;
  p->n_grp = (int)grp.size();
  p->user_stream = (cudaStream_t)cuda_stream;
  cudaError_t e = cudaGetDevice(&p->device);
#define SW_TRY(call)                          \
  do {                                        \
    e = (call);                               \
    if (e != cudaSuccess) {                   \
      free_plan(p);                           \
      return cuda_error(e, #call);            \
    }                                         \
  } while (0)
  SW_TRY(e);
  SW_TRY(cudaMalloc(&p->d_cfg, sizeof(SweepCfg) * n_configs));
  SW_TRY(cudaMalloc(&p->d_grp, sizeof(SweepGroup) * grp.size()));
  SW_TRY(cudaMalloc(&p->d_reg, sizeof(SweepReg) * n_regions));
  SW_TRY(cudaMalloc(&p->d_tile_prefix, sizeof(int64_t) * (n_regions + 1)));
  SW_TRY(cudaMalloc(&p->d_x4, sizeof(float4) * total));
  SW_TRY(cudaMalloc(&p->d_ref4, sizeof(float4) * total));
  SW_TRY(cudaMalloc(&p->d_stats, sizeof(hpac_sweep_stats) * n_configs * n_regions));
  SW_TRY(cudaMalloc(&p->d_counter, sizeof(unsigned long long)));
  SW_TRY(cudaStreamCreateWithFlags(&p->cap_stream, cudaStreamNonBlocking));
  SW_TRY(cudaMemcpyAsync(p->d_cfg, cfg.data(), sizeof(SweepCfg) * n_configs, cudaMemcpyHostToDevice,
                         p->cap_stream));
  SW_TRY(cudaMemcpyAsync(p->d_grp, grp.data(), sizeof(SweepGroup) * grp.size(), cudaMemcpyHostToDevice,
                         p->cap_stream));
  SW_TRY(cudaMemcpyAsync(p->d_reg, reg.data(), sizeof(SweepReg) * n_regions, cudaMemcpyHostToDevice,
                         p->cap_stream));
  SW_TRY(cudaMemcpyAsync(p->d_tile_prefix, prefix.data(), sizeof(int64_t) * (n_regions + 1),
                         cudaMemcpyHostToDevice, p->cap_stream));
  // the inputs and reference come from the caller's stream
  cudaEvent_t ready;
  SW_TRY(cudaEventCreateWithFlags(&ready, cudaEventDisableTiming));
  SW_TRY(cudaEventRecord(ready, p->user_stream));
  SW_TRY(cudaStreamWaitEvent(p->cap_stream, ready, 0));
  cudaEventDestroy(ready);
  // the tiny-price table: count, size it, then split (slots in any order)
  SW_TRY(cudaMemsetAsync(p->d_counter, 0, sizeof(unsigned long long), p->cap_stream));
  count_tiny<<<1024, 256, 0, p->cap_stream>>>(d_ref, total, p->d_counter);
  SW_TRY(cudaGetLastError());
  unsigned long long n_tiny = 0;
  SW_TRY(cudaMemcpyAsync(&n_tiny, p->d_counter, sizeof(n_tiny), cudaMemcpyDeviceToHost, p->cap_stream));
  SW_TRY(cudaStreamSynchronize(p->cap_stream));
  if (n_tiny >= (1ull << 31)) {
    free_plan(p);
    return set_error(HPAC_EUNSUPPORTED, "more than 2^31 exact prices below 1e-30");
  }
  SW_TRY(cudaMalloc(&p->d_tiny, sizeof(float4) * (n_tiny ? n_tiny : 1)));
  SW_TRY(cudaMalloc(&p->d_tiny_terms, sizeof(float4) * (n_tiny ? n_tiny : 1)));
  SW_TRY(cudaMemsetAsync(p->d_counter, 0, sizeof(unsigned long long), p->cap_stream));
  split_ref<<<1024, 256, 0, p->cap_stream>>>(d_ref, p->d_ref4, p->d_tiny, p->d_counter, total);
  SW_TRY(cudaGetLastError());
  pack_inputs<<<1024, 256, 0, p->cap_stream>>>(d_in, in_stride, p->d_x4, total);
  SW_TRY(cudaGetLastError());
  SW_TRY(cudaStreamSynchronize(p->cap_stream));
  int sms = 148;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p->device);
  // the TAF window is stored twice over (2 hsize slots per lane)
  const size_t smem = (size_t)2 * hmax * block_threads * sizeof(float);
  const bool idx32 = 2 * total < (int64_t)INT32_MAX;  // i + T stays below 2 total
  const unsigned grid = (unsigned)(sms * blocks_per_sm);
  const int bandi = (int)band;
  const BlackScholes32 bs{(float)rate};
  // One configuration prices the options itself where their inputs and records
  // (32 B each) exceed L2: 21M options 227..262 us (246..327 when every
  // configuration did, 312..388 from priced options with copies), while 1M options
  // take 57..67 us that way and 44..55 priced beforehand. A pattern hashed per
  // invocation is drawn ahead of the loads there and gains nothing: 326 us, 310
  // priced beforehand.
  int l2 = 0;
  cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, p->device);
  int64_t priced = 0;
  for (const auto &u : ranges) priced += u.second - u.first;
  const bool hashes = cfg[0].cls == CLS_RANDOM && !cfg[0].rule.herded;
  const int form = n_configs == 1 && 32 * priced > l2 && !hashes ? FORM_ONE : singles ? FORM_SINGLES : FORM_GROUPS;
  auto launch = [&](bool set_only) -> cudaError_t {
    if (block_threads == 64)
      return idx32 ? launch_sweep<64, int>(form, set_only, p, grid, smem, n_tiles, bandi, tile_blocks, d_ref, bs)
                   : launch_sweep<64, int64_t>(form, set_only, p, grid, smem, n_tiles, bandi, tile_blocks, d_ref, bs);
    if (block_threads == 128)
      return idx32 ? launch_sweep<128, int>(form, set_only, p, grid, smem, n_tiles, bandi, tile_blocks, d_ref, bs)
                   : launch_sweep<128, int64_t>(form, set_only, p, grid, smem, n_tiles, bandi, tile_blocks, d_ref, bs);
    return idx32 ? launch_sweep<256, int>(form, set_only, p, grid, smem, n_tiles, bandi, tile_blocks, d_ref, bs)
                 : launch_sweep<256, int64_t>(form, set_only, p, grid, smem, n_tiles, bandi, tile_blocks, d_ref, bs);
  };
  SW_TRY(launch(true));
  // capture: clear the counter and the sums, price the options, then the
  // persistent kernel
  SW_TRY(cudaStreamBeginCapture(p->cap_stream, cudaStreamCaptureModeThreadLocal));
  cudaMemsetAsync(p->d_counter, 0, sizeof(unsigned long long), p->cap_stream);
  cudaMemsetAsync(p->d_stats, 0, sizeof(hpac_sweep_stats) * n_configs * n_regions, p->cap_stream);
  if (form != FORM_ONE)
    for (const auto &u : ranges)
      price_options<<<(unsigned)(sms * 8), 256, 0, p->cap_stream>>>(bs, p->d_x4, p->d_ref4, p->d_tiny,
                                                                   p->d_tiny_terms, u.first, u.second);
  cudaError_t launch_err = cudaGetLastError();
  if (launch_err == cudaSuccess) launch_err = launch(false);
  e = cudaStreamEndCapture(p->cap_stream, &p->graph);
  if (launch_err != cudaSuccess) e = launch_err;
  SW_TRY(e);
  SW_TRY(cudaGraphInstantiate(&p->exec, p->graph, 0));
#undef SW_TRY
  *out = p;
  return HPAC_OK;
}

extern "C" hpac_status hpac_sweep_run(hpac_sweep *p) {
  TraceRange trace_("hpac_sweep_run");
  if (!p) return set_error(HPAC_EINVAL, "sweep is NULL");
  HPAC_CUDA_TRY(cudaGraphLaunch(p->exec, p->user_stream));
  return HPAC_OK;
}

extern "C" hpac_status hpac_sweep_results(hpac_sweep *p, hpac_sweep_stats *h_stats) {
  if (!p || !h_stats) return set_error(HPAC_EINVAL, "NULL argument");
  HPAC_CUDA_TRY(cudaMemcpyAsync(h_stats, p->d_stats,
                                sizeof(hpac_sweep_stats) * p->n_cfg * p->n_reg,
                                cudaMemcpyDeviceToHost, p->user_stream));
  HPAC_CUDA_TRY(cudaStreamSynchronize(p->user_stream));
  return HPAC_OK;
}

extern "C" hpac_status hpac_sweep_destroy(hpac_sweep *p) {
  if (!p) return HPAC_OK;
  cudaStreamSynchronize(p->user_stream);
  free_plan(p);
  return HPAC_OK;
}
