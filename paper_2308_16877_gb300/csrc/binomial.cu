// Binomial Options region (Table 1): an American call priced on a
// Cox-Ross-Rubinstein tree, one option per team of 32 lanes (the paper gives a
// whole block to one option and decides per block, Section 4.2). The logical
// schedule counts teams: team t prices options i = t + k T in turn, and TAF /
// iACT / perforation decide per team at each of its steps k, exactly as the
// other regions' logical threads do at thread level.
//
// Tree layout: node j of the current level lives in group j / 128, lane
// (j % 128) / 4 and there in register slot j % 4, so every lane keeps working
// while the level shrinks from N + 1 nodes to one, and only the last of a
// lane's four nodes has its upper neighbour j + 1 on another lane: one shuffle
// per 128 nodes and level. The slots are held as packed single-precision pairs
// (0, 2) and (1, 3): the upper neighbours of the first pair are the second
// pair as it stands. No block barrier: a team is one warp. Four teams share a
// block.
#include <math.h>

#include "convert.cuh"
#include "hpac_internal.cuh"
#include "perfo_rule.cuh"
#include "regions.cuh"

namespace hpac {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kTeams = 4;  // teams (warps) per block

struct TreeC {
  float puA, pdA, uf;
  double v, u2, u256;  // v = sigma sqrt(dt), e^{2 v}, e^{256 v}
};

// Per-option constants in double, rounded once: dt = T/N, v = sigma sqrt(dt),
// u = e^v, d = 1/u, a = e^{r dt}, pu = (a - d)/(u - d), weights pu/a, (1-pu)/a.
// The whole warp prices one option, so the four exponentials are one call with
// the lane's argument, and the two weights one division (FP64 is GB300's
// narrow pipe; with every lane evaluating every exponential the constants took
// longer than a 255-step tree).
__device__ __forceinline__ TreeC tree_constants(float Tm, float sig, double r, int N) {
  const int lane = threadIdx.x & 31;
  const double dt = (double)Tm / N;
  const double v = (double)sig * sqrt(dt);
  const double arg = lane == 0 ? v : lane == 1 ? r * dt : lane == 2 ? 2.0 * v : 256.0 * v;
  const double e = exp(arg);
  const double u = __shfl_sync(kFull, e, 0), a = __shfl_sync(kFull, e, 1);
  const double u2 = __shfl_sync(kFull, e, 2), u256 = __shfl_sync(kFull, e, 3);
  const double d = 1.0 / u;
  const double pu = (a - d) / (u - d), pd = 1.0 - pu;
  const double w = (lane == 0 ? pu : pd) / a;
  return TreeC{(float)__shfl_sync(kFull, w, 0), (float)__shfl_sync(kFull, w, 1), (float)u, v, u2, u256};
}

// S0 e^{v k}.
__device__ __noinline__ double leaf_price(float S0, double v, int k) { return (double)S0 * exp(v * (double)k); }

// One backward step over the first A groups: V <- max(fma(pu/a, V_up, pd/a V),
// S u - X), S <- S u, two nodes per packed instruction (each half rounded as
// the scalar operation would be). `top` is the node above the last group.
template <int G, int A>
__device__ __forceinline__ void tree_step(unsigned long long (&V)[G][2], unsigned long long (&S)[G][2],
                                          float top, unsigned long long pu2, unsigned long long pd2,
                                          unsigned long long uf2, unsigned long long x2, int lane, int next) {
#pragma unroll
  for (int g = 0; g < A; ++g) {
    float v0, v2, above, none;
    f32x2_unpack(V[g][0], v0, v2);
    if (g + 1 < G)
      f32x2_unpack(V[g + 1 < G ? g + 1 : 0][0], above, none);
    else
      above = top;
    const float v4 = __shfl_sync(kFull, lane == 0 ? above : v0, next);
    const unsigned long long up[2] = {V[g][1], f32x2_pack(v2, v4)};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const unsigned long long cont = f32x2_fma(pu2, up[h], f32x2_mul(pd2, V[g][h]));
      S[g][h] = f32x2_mul(S[g][h], uf2);
      float c0, c1, e0, e1;
      f32x2_unpack(cont, c0, c1);
      f32x2_unpack(f32x2_sub(S[g][h], x2), e0, e1);
      V[g][h] = f32x2_pack(fmaxf(c0, e0), fmaxf(c1, e1));  // early exercise
    }
  }
}

// The steps to the levels n >= 128 (A - 1) with A groups, then with A - 1, ...:
// the number of groups is fixed within a segment, so its loop has no test per
// group.
template <int G, int A>
__device__ __forceinline__ void tree_segments(unsigned long long (&V)[G][2], unsigned long long (&S)[G][2],
                                              float top, unsigned long long pu2, unsigned long long pd2,
                                              unsigned long long uf2, unsigned long long x2, int lane, int next,
                                              int n) {
  if constexpr (A > 0) {
#pragma unroll 1
    for (; n >= 128 * (A - 1); --n) tree_step<G, A>(V, S, top, pu2, pd2, uf2, x2, lane, next);
    tree_segments<G, A - 1>(V, S, top, pu2, pd2, uf2, x2, lane, next, n);
  }
}

// Price of one option by the whole warp (all lanes return it); N <= 128 G.
// Bound by the single-precision pipe: per 128 nodes and level 8 packed
// operations (16 issue cycles of a quarter-SM), 4 maxima, one shuffle, one
// select and one move: 17.1 warp instructions against 28. 16,384 options of
// 1024 steps in teams of four took 1.68 ms (2.23 ms with one node per lane and slot: a shuffle,
// a select and a repacking per 32 nodes), 12,000 of 255 steps 164 us (175).
// ncu: issue 63%, that pipe 69% of the cycles, its throttle the first stall.
// 123 registers, four blocks per SM; five at 96 registers took 1.73 ms, and
// scalar instead of packed operations for any of the four gained nothing.
template <int G>
__device__ __forceinline__ float team_price(float S0, float X, float Tm, float sig, double r, int N) {
  const int lane = threadIdx.x & 31;
  const TreeC c = tree_constants(Tm, sig, r, N);
  unsigned long long V[G][2], S[G][2];
  // leaves S_j = S0 e^{v (2j - N)}: the lane's first by exp, the next ones by
  // the factors e^{2v} and e^{256v}, in double (a few double ulps from each
  // leaf's own exp)
  double first = leaf_price(S0, c.v, 8 * lane - N);
  double Sd = first;
  // e^{256v} out of range, or the lowest leaf e^{-vN} (S0 >= e^-104) below the
  // normal range, from where the factors would lead to wrong leaves: each leaf's
  // own exp
  const bool far = !(256.0 * c.v < 700.0 && c.v * N < 600.0);
#pragma unroll
  for (int g = 0; g < G; ++g) {
    float s[4], p[4];
    Sd = first;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int j = 128 * g + 4 * lane + i;
      if (far) Sd = leaf_price(S0, c.v, 2 * j - N);
      s[i] = j <= N ? double_to_float_rn_novote(Sd) : 0.0f;
      p[i] = fmaxf(__fsub_rn(s[i], X), 0.0f);
      Sd *= c.u2;
    }
    first *= c.u256;
    S[g][0] = f32x2_pack(s[0], s[2]);
    S[g][1] = f32x2_pack(s[1], s[3]);
    V[g][0] = f32x2_pack(p[0], p[2]);
    V[g][1] = f32x2_pack(p[1], p[3]);
  }
  // N = 128 G: the top leaf lies past the last group; lane 31's next one
  if (far) Sd = leaf_price(S0, c.v, 256 * (G - 1) + 8 * (lane + 1) - N);
  const float top = __shfl_sync(kFull, fmaxf(__fsub_rn((float)Sd, X), 0.0f), 31);
  tree_segments<G, G>(V, S, top, f32x2_pack(c.puA, c.puA), f32x2_pack(c.pdA, c.pdA),
                      f32x2_pack(c.uf, c.uf), f32x2_pack(X, X), lane, (lane + 1) & 31, N - 1);
  float v0, v2;
  f32x2_unpack(V[0][0], v0, v2);
  return __shfl_sync(kFull, v0, 0);
}

enum { TECH_EXACT = 0, TECH_TAF = 1, TECH_IACT = 2, TECH_PERFO = 3 };

struct BinoArgs {
  const float *in;
  int64_t stride, n, T;
  float *out;
  uint8_t *mask;
  float *stat;
  double r;
  int N;
  // TAF
  int h, p, thr_inf, reset;
  float thr;
  double thr_d;
  // iACT
  int tsize;
  float scale[4];
  // perforation
  DropRule rule;
  unsigned long long *counters;
};

// Shared memory per team: TAF window (h floats) or iACT table (tsize x 4
// scaled inputs, then tsize outputs).
template <int G, int TECH>
__global__ void __launch_bounds__(32 * kTeams, G == 8 ? 4 : 7) binomial_kernel(BinoArgs a) {
  extern __shared__ __align__(16) float sm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t team = (int64_t)blockIdx.x * kTeams + warp;
  const int per = TECH == TECH_TAF ? a.h : TECH == TECH_IACT ? 5 * a.tsize : 0;
  float *mine = sm + warp * per;
  unsigned long long n_alt = 0, n_border = 0;
  if (team < a.T) {
    // TAF state (uniform across the team's lanes)
    int pos = 0, cnt = 0, pred = 0;
    const float inv_h = TECH == TECH_TAF ? 1.0f / (float)a.h : 1.0f;
    // iACT state
    int filled = 0, rr = 0;
    for (int64_t k = 0, i = team; i < a.n; ++k, i += a.T) {
      if (TECH == TECH_PERFO) {
        bool drop;
        if (a.rule.kind == HPAC_PERFO_INI || a.rule.kind == HPAC_PERFO_FINI)
          drop = i < a.rule.lo || i >= a.rule.hi;
        else
          drop = a.rule.drop_key(a.rule.herded ? k : i);
        if (drop) {
          if (lane == 0 && a.mask) a.mask[i] = HPAC_MASK_SKIPPED;
          ++n_alt;
          continue;  // the output keeps the caller's value
        }
      }
      const float S0 = a.in[i], X = a.in[a.stride + i], Tm = a.in[2 * a.stride + i],
                  sig = a.in[3 * a.stride + i];
      if (TECH == TECH_TAF) {
        if (pred > 0) {
          const float y = mine[pos == 0 ? a.h - 1 : pos - 1];
          if (lane == 0) {
            a.out[i] = y;
            if (a.mask) a.mask[i] = HPAC_MASK_APPROX;
            if (a.stat) a.stat[i] = nan_v<float>();
          }
          --pred;
          ++n_alt;
          if (a.reset && pred == 0) cnt = 0;
          continue;
        }
        const float y = team_price<G>(S0, X, Tm, sig, a.r, a.N);
        __syncwarp();
        if (lane == 0) {
          a.out[i] = y;
          if (a.mask) a.mask[i] = HPAC_MASK_EXACT;
          mine[pos] = y;
        }
        __syncwarp();
        pos = pos + 1 == a.h ? 0 : pos + 1;
        cnt = cnt < a.h ? cnt + 1 : a.h;
        if (cnt == a.h) {
          bool wants;
          if (a.stat == nullptr && a.counters == nullptr && !a.thr_inf) {
            wants = rsd_below_fast<float>(mine, 1, pos, a.h, a.thr, inv_h);
          } else {
            const float s = window_rsd<float>(mine, 1, pos, a.h, inv_h);
            if (lane == 0 && a.stat) a.stat[i] = s;
            if (a.counters && borderline((double)s, a.thr_d)) ++n_border;
            wants = a.thr_inf || s < a.thr;
          }
          if (wants) pred = a.p;
        } else if (lane == 0 && a.stat) {
          a.stat[i] = nan_v<float>();
        }
        continue;
      }
      if (TECH == TECH_IACT) {
        const float z[4] = {__fmul_rn(a.scale[0], S0), __fmul_rn(a.scale[1], X),
                            __fmul_rn(a.scale[2], Tm), __fmul_rn(a.scale[3], sig)};
        // distances to the valid slots, two per lane, then the lowest-index minimum
        float best = INFINITY;
        int near = -1;
        for (int j = lane; j < filled; j += 32) {
          float acc = 0.0f;
#pragma unroll
          for (int d = 0; d < 4; ++d) {
            const float df = __fsub_rn(z[d], mine[4 * j + d]);
            acc = __fadd_rn(acc, __fmul_rn(df, df));
          }
          if (near < 0 || acc < best) {
            best = acc;
            near = j;
          }
        }
        for (int off = 16; off > 0; off >>= 1) {
          const float ob = __shfl_xor_sync(kFull, best, off);
          const int on = __shfl_xor_sync(kFull, near, off);
          if (on >= 0 && (near < 0 || ob < best || (ob == best && on < near))) {
            best = ob;
            near = on;
          }
        }
        const bool has = filled > 0;
        const float dmin = has ? __fsqrt_rn(best) : INFINITY;
        if (lane == 0 && a.stat) a.stat[i] = dmin;
        if (a.counters && has && borderline((double)dmin, a.thr_d)) ++n_border;
        if (has && dmin < a.thr) {
          if (lane == 0) {
            a.out[i] = mine[4 * a.tsize + near];
            if (a.mask) a.mask[i] = HPAC_MASK_APPROX;
          }
          ++n_alt;
          continue;
        }
        const float y = team_price<G>(S0, X, Tm, sig, a.r, a.N);
        __syncwarp();
        if (lane == 0) {
          a.out[i] = y;
          if (a.mask) a.mask[i] = HPAC_MASK_EXACT;
#pragma unroll
          for (int d = 0; d < 4; ++d) mine[4 * rr + d] = z[d];
          mine[4 * a.tsize + rr] = y;
        }
        __syncwarp();
        rr = rr + 1 == a.tsize ? 0 : rr + 1;
        filled = filled < a.tsize ? filled + 1 : a.tsize;
        continue;
      }
      const float y = team_price<G>(S0, X, Tm, sig, a.r, a.N);
      if (lane == 0) {
        a.out[i] = y;
        if (a.mask) a.mask[i] = HPAC_MASK_EXACT;
      }
    }
  }
  if (a.counters && lane == 0) {
    if (n_alt) atomicAdd(&a.counters[0], n_alt);
    if (n_border) atomicAdd(&a.counters[1], n_border);
  }
}

template <int G>
hpac_status launch_groups(const hpac_region *r, int tech, const BinoArgs &a, size_t smem) {
  const int64_t blocks = (a.T + kTeams - 1) / kTeams;
  if (blocks > 0x7fffffffLL) return set_error(HPAC_EINVAL, "too many logical teams");
  const dim3 grid((unsigned)blocks), block(32 * kTeams);
  switch (tech) {
    case TECH_TAF: binomial_kernel<G, TECH_TAF><<<grid, block, smem, r->stream>>>(a); break;
    case TECH_IACT: binomial_kernel<G, TECH_IACT><<<grid, block, smem, r->stream>>>(a); break;
    case TECH_PERFO: binomial_kernel<G, TECH_PERFO><<<grid, block, smem, r->stream>>>(a); break;
    default: binomial_kernel<G, TECH_EXACT><<<grid, block, smem, r->stream>>>(a); break;
  }
  HPAC_CUDA_TRY(cudaGetLastError());
  return HPAC_OK;
}

}  // namespace

hpac_status launch_binomial(hpac_region *r, int technique, const void *knobs, const void *in,
                            void *out, uint8_t *mask, void *stat, unsigned long long *counters) {
  const hpac_region_desc &d = r->d;
  if (d.n == 0) return HPAC_OK;
  BinoArgs a{};
  a.in = static_cast<const float *>(in);
  a.stride = d.in_stride;
  a.n = d.n;
  a.T = logical_threads(d);
  a.out = static_cast<float *>(out);
  a.mask = mask;
  a.stat = static_cast<float *>(stat);
  a.r = d.param;
  a.N = d.arg;
  a.counters = counters;
  a.rule.kind = -1;
  size_t smem = 0;
  if (technique == TECH_TAF) {
    const hpac_taf_knobs *k = static_cast<const hpac_taf_knobs *>(knobs);
    a.h = k->hsize;
    a.p = k->psize;
    a.thr = (float)k->thresh;
    a.thr_d = k->thresh;
    a.thr_inf = isinf(k->thresh) ? 1 : 0;
    a.reset = k->reset_on_exit;
    smem = (size_t)kTeams * a.h * sizeof(float);
  } else if (technique == TECH_IACT) {
    const hpac_iact_knobs *k = static_cast<const hpac_iact_knobs *>(knobs);
    a.tsize = k->tsize;
    a.thr = (float)k->thresh;
    a.thr_d = k->thresh;
    for (int j = 0; j < 4; ++j) a.scale[j] = k->in_scale ? (float)k->in_scale[j] : 1.0f;
    smem = (size_t)kTeams * 5 * a.tsize * sizeof(float);
  } else if (technique == TECH_PERFO) {
    const hpac_perfo_knobs *k = static_cast<const hpac_perfo_knobs *>(knobs);
    a.rule.kind = k->kind;
    a.rule.herded = k->herded ? 1 : 0;
    a.rule.m = k->m_or_percent;
    a.rule.seed = k->seed;
    a.rule.cut = (uint32_t)floor(k->rate * 16777216.0);
    a.rule.T = a.T;
    const int64_t cut = (d.n * (int64_t)k->m_or_percent) / 100;
    a.rule.lo = k->kind == HPAC_PERFO_INI ? cut : 0;
    a.rule.hi = k->kind == HPAC_PERFO_FINI ? d.n - cut : d.n;
  }
  // Exact prices do not depend on the teams: a team per option, so that the
  // last wave of blocks is a small part of many (4096 teams of 4 options are
  // 1.7 waves at 1024 steps: 1.69 -> 1.59 ms).
  constexpr int64_t kMaxTeams = 0x7fffffffLL * kTeams;  // a grid's
  if (technique == TECH_EXACT && a.T < a.n) a.T = a.n < kMaxTeams ? a.n : kMaxTeams;
  // the registers of a lane hold 4 nodes of each group of 128
  if (a.N <= 256) return launch_groups<2>(r, technique, a, smem);
  if (a.N <= 512) return launch_groups<4>(r, technique, a, smem);
  return launch_groups<8>(r, technique, a, smem);
}

}  // namespace hpac
