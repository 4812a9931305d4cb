// Quality loss against an exact reference (Section 4): MAPE (Eq. 1), RMSE and
// the misclassification rate MCR (Eq. 2), accumulated in double precision.
//
// One deterministic pass: a grid of blocks reduces grid-stride slices to
// per-block partials (a tree inside each block), and the last block to finish
// reduces the partials in index order (as a second launch that took 4.5 us and
// its gap). Two entry points differ only in where the partials live:
//  - hpac_quality: a device buffer of kBlocks + 2 partials (the last one holds
//    the ticket), allocated with cudaMalloc on a device's first call and kept
//    for the life of the process, with a page-locked host result that the
//    kernel writes; a host mutex serializes calls, which wait for their result.
//  - hpac_quality_noalloc: a fixed static __device__ array of kStaticPartials
//    + 2 partials compiled into the library, addressed through a per-device
//    cache of its device address; no lock (callers serialize overlapping
//    calls themselves, see hpac.h).
// Both per-device caches hold device addresses of the primary context: they
// assume that context is not reset (cudaDeviceReset) while the process uses
// the library.
#include <math.h>
#include <mutex>

#include "hpac_internal.cuh"
#include "convert.cuh"

namespace hpac {
namespace {

constexpr int kBlocks = 1216;  // 8 x 152 SMs
constexpr int kThreads = 256;

struct Partial {
  double sum;
  double zmax;
  unsigned long long used;
  unsigned long long zeros;
  unsigned long long zbad;
};

// |x| (its bits) rounded to single precision, ties to even, then scaled by
// 2^-sub: exponent fields only, so valid wherever the scaled result is a
// normal single.
__device__ __forceinline__ float round_scaled(uint64_t abs_bits, int sub) {
  const uint64_t t = abs_bits + 0x0fffffffull + ((abs_bits >> 29) & 1ull);
  return __uint_as_float((uint32_t)(t >> 29) - ((uint32_t)(sub + (1023 - 127)) << 23));
}

// The term of an element that the straight-line code of quality_partial does
// not cover (its conversions, and for MAPE the range of its ratio), a != 0 for
// MAPE, as bits; bit 32 set: the ratio needs the double-precision division.
template <typename B, int METRIC>
__device__ __noinline__ uint64_t odd_term(double a, B braw) {
  const double b = (double)braw, d = a - b;
  if (METRIC == HPAC_METRIC_MCR) return __float_as_uint(a != b ? 1.0f : 0.0f);
  if (METRIC == HPAC_METRIC_RMSE) {
    const float f = __double2float_rn(d);
    return __float_as_uint(f * f);
  }
  const uint64_t aabs = (uint64_t)__double_as_longlong(a) & 0x7fffffffffffffffull;
  const uint64_t dabs = (uint64_t)__double_as_longlong(d) & 0x7fffffffffffffffull;
  const int ea = (int)(aabs >> 52), ed = (int)(dabs >> 52), rel = ed - ea;
  if (ea == 0 || ea == 0x7ff || ed == 0x7ff || (ed == 0 && dabs != 0ull) || rel > 126) return 1ull << 32;
  // a ratio below 2^-1021 rounds to zero
  float fd = 0.0f;
  if (dabs != 0ull && rel >= -1022)
    fd = __double2float_rn(
        __longlong_as_double((long long)((dabs & 0xfffffffffffffull) | ((uint64_t)(rel + 1023) << 52))));
  return __float_as_uint(__fdiv_rn(fd, round_scaled(aabs, ea - 1023)));
}

__device__ __noinline__ double wide_ratio(double a, double b) { return fabs(a - b) / fabs(a); }

// Adds a block's partials (the sum in a fixed order, a tree over the threads)
// into thread 0's. MAPE alone counts zeros.
template <bool ZEROS>
__device__ __forceinline__ void reduce_block(Partial &v) {
  __shared__ double s_sum[kThreads];
  __shared__ unsigned long long s_cnt[4][kThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31;
  s_sum[tid] = v.sum;
  unsigned long long c[4] = {v.used, v.zeros, v.zbad, (unsigned long long)__double_as_longlong(v.zmax)};
#pragma unroll
  for (int q = 0; q < (ZEROS ? 4 : 1); ++q) {
    for (int off = 16; off > 0; off >>= 1) {
      const unsigned long long o = __shfl_down_sync(0xffffffffu, c[q], off);
      c[q] = q == 3 ? (o > c[q] ? o : c[q]) : c[q] + o;  // zmax >= 0: its bits order as it does
    }
    if (lane == 0) s_cnt[q][tid >> 5] = c[q];
  }
  __syncthreads();
  for (int w = kThreads / 2; w >= 32; w >>= 1) {
    if (tid < w) s_sum[tid] += s_sum[tid + w];
    __syncthreads();
  }
  if (tid < 32) {
    double sum = s_sum[tid];
    for (int off = 16; off > 0; off >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, off);
    if (tid == 0) {
#pragma unroll
      for (int q = 0; q < (ZEROS ? 4 : 1); ++q)
        for (int w = 1; w < kThreads / 32; ++w) {
          const unsigned long long o = s_cnt[q][w];
          c[q] = q == 3 ? (o > c[q] ? o : c[q]) : c[q] + o;
        }
      v = Partial{sum, __longlong_as_double((long long)c[3]), c[0], c[1], c[2]};
    }
  }
  __syncthreads();  // the shared arrays are free again
}

// Resident blocks per SM (the grid is one wave, so they also fix which
// elements a thread sums).
template <typename B, int METRIC>
constexpr int resident() {
  return METRIC == HPAC_METRIC_MAPE ? 4 : METRIC == HPAC_METRIC_RMSE && sizeof(B) == 8 ? 5 : 6;
}

// GB300 issues one double-precision warp instruction per 16 cycles per SM, so
// the per-element work keeps a single FP64 operation (the difference a - b,
// exact for the single-precision approximations; for MCR the comparison). The
// conversions between the precisions and the range tests of the exact value run
// on the integer pipes (the same bits as the hardware conversions and
// comparisons), the ratio or square is formed in single precision, and the terms
// are summed in groups of 16 before entering the double-precision accumulator.
// For MAPE the exact value and the difference are first scaled by the power of
// two that puts |a| in [1, 2) (an exact change of their exponent fields), so the
// single-precision ratio covers every finite exact value; only ratios above
// 2^126 and subnormal operands take the double-precision division.
// Each thread walks its grid-stride sequence four elements at a time, for MAPE
// with the next four in flight. Operands and results in the normal range (b may be
// subnormal or zero, the difference zero) take straight-line code; the other
// elements (0.1% of a book of option prices) go out of line in their turn.
// 2^24 options: MAPE 98 us with every element's case distinctions in line (150
// instructions each, a warp vote among them), 86 with the straight-line groups
// and the general code inlined behind them, 79 as it stands (TAF and its MAPE
// 213, 187 and 181 us); 5,000,011 options, iACT and its RMSE 114, 96 and 90 us.
template <typename B, int METRIC>
__global__ void __launch_bounds__(kThreads, resident<B, METRIC>()) quality_partial(const double *__restrict__ a,
                                                            const void *__restrict__ bv_, int64_t n,
                                                            Partial *part, unsigned *ticket,
                                                            Partial *res) {
  const B *__restrict__ b = static_cast<const B *>(bv_);
  constexpr int metric = METRIC;
  double sum = 0.0;
  unsigned long long zmax = 0;  // bits of the largest |b| where a == 0 (NaN skipped, as fmax does)
  unsigned used = 0, zeros = 0, zbad = 0;  // one thread's elements: memory holds far fewer than 2^32
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  float chunk = 0.0f;
  int in_chunk = 0;
  auto add = [&](float term) {
    chunk += term;
    ++used;
    if (++in_chunk == 16) {
      sum += float_to_double(chunk);
      chunk = 0.0f;
      in_chunk = 0;
    }
  };
  int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  double an[4];
  B bn[4];
  auto load = [&](int64_t at) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      an[k] = 1.0;
      bn[k] = (B)1;
      if (at + k * stride < n) {
        an[k] = __ldcs(a + at + k * stride);
        bn[k] = __ldcs(b + at + k * stride);
      }
    }
  };
  // (40 registers, 48 warps per SM, without MAPE's division: nothing ahead)
  constexpr bool kAhead = METRIC == HPAC_METRIC_MAPE;
  if (kAhead) load(i0);
  for (; i0 < n; i0 += 4 * stride) {
    double av[4];
    B bv[4];
    if (!kAhead) load(i0);
#pragma unroll
    for (int k = 0; k < 4; ++k) av[k] = an[k], bv[k] = bn[k];
    if (kAhead) load(i0 + 4 * stride);
    const int have = i0 + 3 * stride < n ? 4 : i0 + 2 * stride < n ? 3 : i0 + stride < n ? 2 : 1;
    float term[4];
    unsigned odd = 0u;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      double bi;
      bool plain = true;
      if (sizeof(B) == 4) {
        // exponent and fraction moved to their places; a subnormal is scaled
        // by 2^64 first (exact) and its exponent taken back
        uint32_t u = __float_as_uint((float)bv[k]);
        const uint32_t low = u << 1;  // without the sign
        plain = low < 0xff000000u;    // finite
        const bool tiny = low < 0x01000000u;
        if (tiny) u = __float_as_uint((float)bv[k] * 18446744073709551616.0f);
        const uint32_t hi = ((uint32_t)((int)u >> 3) & 0x8fffffffu) + (tiny ? 0x34000000u : 0x38000000u);
        bi = __hiloint2double((int)(low ? hi : u), (int)(u << 29));
      } else {
        bi = (double)bv[k];
      }
      if (metric == HPAC_METRIC_MCR) {
        term[k] = av[k] != bi ? 1.0f : 0.0f;
      } else {
        // the one FP64 operation; the opaque move keeps the compiler from
        // recomputing it where its bits are used
        uint64_t dbits;
        asm volatile("mov.b64 %0, %1;" : "=l"(dbits) : "d"(av[k] - bi));
        const uint64_t dabs = dbits & 0x7fffffffffffffffull;
        const int ed = (int)(dabs >> 52);
        if (metric == HPAC_METRIC_MAPE) {
          const bool same = dabs == 0ull;
          const uint64_t aabs = (uint64_t)__double_as_longlong(av[k]) & 0x7fffffffffffffffull;
          const int ea = (int)(aabs >> 52);
          plain = plain && (unsigned)(ea - 1) < 0x7feu && ed != 0x7ff &&
                  ((ed != 0 && (unsigned)(ed - ea + 125) <= 251u) || same);
          const float fd = same ? 0.0f : round_scaled(dabs, ea - 1023);
          term[k] = __fdiv_rn(fd, round_scaled(aabs, ea - 1023));
        } else {
          // below 2^-126 the square underflows to zero
          plain = plain && ed < 1150;
          const float fd = ed < 897 ? 0.0f : round_scaled(dabs, 0);
          term[k] = fd * fd;
        }
      }
      if (!plain) odd |= 1u << k;
    }
    if (odd == 0u && have == 4 && (in_chunk & 3) == 0) {
#pragma unroll
      for (int k = 0; k < 4; ++k) chunk += term[k];
      used += 4;
      in_chunk += 4;
      if (in_chunk == 16) {
        sum += float_to_double(chunk);
        chunk = 0.0f;
        in_chunk = 0;
      }
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (k >= have) break;
        if (!(odd >> k & 1u)) {
          add(term[k]);
          continue;
        }
        if (metric == HPAC_METRIC_MAPE && av[k] == 0.0) {
          const uint64_t babs = (uint64_t)__double_as_longlong((double)bv[k]) & 0x7fffffffffffffffull;
          ++zeros;
          if (babs != 0ull) ++zbad;
          if (babs <= 0x7ff0000000000000ull && babs > zmax) zmax = babs;
          continue;
        }
        const uint64_t t = odd_term<B, METRIC>(av[k], bv[k]);
        if (t >> 32) {
          sum += wide_ratio(av[k], (double)bv[k]);
          ++used;
        } else {
          add(__uint_as_float((uint32_t)t));
        }
      }
    }
  }
  sum += float_to_double(chunk);
  constexpr bool kZeros = METRIC == HPAC_METRIC_MAPE;
  Partial acc{sum, __longlong_as_double((long long)zmax), used, zeros, zbad};
  reduce_block<kZeros>(acc);
  __shared__ bool s_last;
  if (threadIdx.x == 0) {
    part[blockIdx.x] = acc;
    __threadfence();  // the partial before the ticket
    s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();  // the ticket before the other blocks' partials
  acc = Partial{0.0, 0.0, 0, 0, 0};
  for (int j = threadIdx.x; j < (int)gridDim.x; j += blockDim.x) {
    const Partial *p = part + j;
    acc.sum += __ldcg(&p->sum);
    acc.used += __ldcg(&p->used);
    if (kZeros) {
      acc.zmax = fmax(acc.zmax, __ldcg(&p->zmax));
      acc.zeros += __ldcg(&p->zeros);
      acc.zbad += __ldcg(&p->zbad);
    }
  }
  reduce_block<kZeros>(acc);
  if (threadIdx.x == 0) {
    *ticket = 0;  // for the next call on this scratch
    *res = acc;
  }
}

// The partial-sum kernel for an approximation type and a metric (one
// instantiation each, so a metric's unused paths are not compiled in).
using PartialKernel = void (*)(const double *, const void *, int64_t, Partial *, unsigned *, Partial *);
PartialKernel partial_kernel(int32_t approx_dtype, int32_t metric) {
  if (approx_dtype == HPAC_F32) {
    if (metric == HPAC_METRIC_MAPE) return quality_partial<float, HPAC_METRIC_MAPE>;
    if (metric == HPAC_METRIC_RMSE) return quality_partial<float, HPAC_METRIC_RMSE>;
    return quality_partial<float, HPAC_METRIC_MCR>;
  }
  if (metric == HPAC_METRIC_MAPE) return quality_partial<double, HPAC_METRIC_MAPE>;
  if (metric == HPAC_METRIC_RMSE) return quality_partial<double, HPAC_METRIC_RMSE>;
  return quality_partial<double, HPAC_METRIC_MCR>;
}

// Per-device scratch: kBlocks partials, a result and the ticket (0 between
// calls); the page-locked host result, NULL where it could not be had.
Partial *g_scratch[64] = {nullptr};
Partial *g_host_result[64] = {nullptr};
std::mutex g_mu;

// Callers hold g_mu for the whole call: the scratch is shared by every call
// on the device and the call waits for its result before releasing it.
hpac_status scratch_for(int dev, cudaStream_t st, Partial **out) {
  if (dev < 0 || dev >= 64) return set_error(HPAC_EUNSUPPORTED, "device ordinal %d", dev);
  if (!g_scratch[dev]) {
    Partial *p = nullptr;
    cudaError_t e = cudaMalloc(&p, (kBlocks + 2) * sizeof(Partial));
    // on the call's stream (the legacy stream would break captures of blocking
    // streams on other threads), and done before calls on other streams
    if (e == cudaSuccess) e = cudaMemsetAsync(p + kBlocks + 1, 0, sizeof(Partial), st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
      cudaFree(p);
      return cuda_error(e, "hpac_quality scratch");
    }
    if (cudaHostAlloc(&g_host_result[dev], sizeof(Partial), cudaHostAllocDefault) != cudaSuccess) {
      cudaGetLastError();
      g_host_result[dev] = nullptr;
    }
    g_scratch[dev] = p;
  }
  *out = g_scratch[dev];
  return HPAC_OK;
}

}  // namespace
}  // namespace hpac

using namespace hpac;

extern "C" hpac_status hpac_quality(int32_t approx_dtype, int64_t n, const double *d_exact,
                                    const void *d_approx, int32_t metric,
                                    hpac_quality_result *h_result, void *cuda_stream) {
  TraceRange trace_("hpac_quality");
  if (!h_result) return set_error(HPAC_EINVAL, "h_result is NULL");
  if (n < 0) return set_error(HPAC_EINVAL, "n < 0");
  if (metric < HPAC_METRIC_MAPE || metric > HPAC_METRIC_MCR)
    return set_error(HPAC_EINVAL, "metric %d", metric);
  if (approx_dtype != HPAC_F32 && approx_dtype != HPAC_F64)
    return set_error(HPAC_EINVAL, "dtype %d", approx_dtype);
  if (n > 0 && (!d_exact || !d_approx)) return set_error(HPAC_EINVAL, "NULL data pointer");
  *h_result = hpac_quality_result{0.0, 0.0, 0, 0, 0};
  if (n == 0) return HPAC_OK;
  int dev = 0;
  HPAC_CUDA_TRY(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(g_mu);
  cudaStream_t st = (cudaStream_t)cuda_stream;
  Partial *scr = nullptr;
  hpac_status s = scratch_for(dev, st, &scr);
  if (s != HPAC_OK) return s;
  // one wave of resident blocks (at most kBlocks): every thread's sequence
  // runs to the end without a second, partly filled wave
  const PartialKernel fn = partial_kernel(approx_dtype, metric);
  int per_sm = 0, sms = 0;
  HPAC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kThreads, 0));
  HPAC_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int64_t wave = (int64_t)(per_sm > 0 ? per_sm : 1) * sms;
  int64_t blocks = (n + kThreads - 1) / kThreads;
  if (blocks > wave) blocks = wave;
  if (blocks > kBlocks) blocks = kBlocks;
  // page-locked host memory has one address for host and device (unified
  // addressing), so the kernel's result needs no copy
  Partial *host = g_host_result[dev];
  fn<<<(unsigned)blocks, kThreads, 0, st>>>(d_exact, d_approx, n, scr,
                                            reinterpret_cast<unsigned *>(scr + kBlocks + 1),
                                            host ? host : scr + kBlocks);
  HPAC_CUDA_TRY(cudaGetLastError());
  Partial res;
  if (!host) HPAC_CUDA_TRY(cudaMemcpyAsync(&res, scr + kBlocks, sizeof(Partial), cudaMemcpyDeviceToHost, st));
  HPAC_CUDA_TRY(cudaStreamSynchronize(st));
  if (host) res = *host;
  double v = res.used ? res.sum / (double)res.used : 0.0;
  if (metric == HPAC_METRIC_RMSE) v = sqrt(v);
  h_result->value = v;
  h_result->zero_max_abs = res.zmax;
  h_result->used = (int64_t)res.used;
  h_result->zeros = (int64_t)res.zeros;
  h_result->zeros_mismatch = (int64_t)res.zbad;
  return HPAC_OK;
}

// ---------------------------------------------------------------------------
// Allocation-free variant of hpac_quality.
//
// Its scratch is a fixed array compiled into the library instead of a buffer
// obtained from cudaMalloc: every GPU that loads the library holds these
// 16,386 partials (about 656 KB) until the process exits. The reduction runs
// ceil(n / 8192) blocks of the same kernel (each thread reduces at most
// 32 elements), so n may not exceed 16,384 * 8,192 = 134,217,728 elements.
// ---------------------------------------------------------------------------
namespace hpac {
namespace {

constexpr int64_t kStaticTile = (int64_t)kThreads * 32;          // elements per block
constexpr int kStaticPartials = 16384;                            // blocks at most
constexpr int64_t kStaticMaxN = kStaticTile * kStaticPartials;    // 134,217,728

static __device__ __align__(256) Partial g_static_scratch[kStaticPartials + 2];

// Device address of g_static_scratch per device ordinal, looked up once with
// that device current (host code may not use the symbol itself as a pointer).
Partial *g_static_addr[64] = {nullptr};
std::mutex g_static_mu;

hpac_status static_scratch(int dev, Partial **out) {
  if (dev < 0 || dev >= 64) return set_error(HPAC_EUNSUPPORTED, "device ordinal %d", dev);
  std::lock_guard<std::mutex> lk(g_static_mu);
  if (!g_static_addr[dev]) {
    void *p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess) return cuda_error(e, "cudaGetSymbolAddress(g_static_scratch)");
    g_static_addr[dev] = static_cast<Partial *>(p);
  }
  *out = g_static_addr[dev];
  return HPAC_OK;
}

}  // namespace
}  // namespace hpac

extern "C" hpac_status hpac_quality_noalloc(int32_t approx_dtype, int64_t n, const double *d_exact,
                                            const void *d_approx, int32_t metric,
                                            hpac_quality_result *h_result, void *cuda_stream) {
  TraceRange trace_("hpac_quality_noalloc");
  if (!h_result) return set_error(HPAC_EINVAL, "h_result is NULL");
  if (n < 0) return set_error(HPAC_EINVAL, "n < 0");
  if (n > kStaticMaxN)
    return set_error(HPAC_EINVAL,
                     "hpac_quality_noalloc: n = %lld exceeds the %lld-element limit of its fixed "
                     "scratch; use hpac_quality for larger inputs",
                     (long long)n, (long long)kStaticMaxN);
  if (metric < HPAC_METRIC_MAPE || metric > HPAC_METRIC_MCR)
    return set_error(HPAC_EINVAL, "metric %d", metric);
  if (approx_dtype != HPAC_F32 && approx_dtype != HPAC_F64)
    return set_error(HPAC_EINVAL, "dtype %d", approx_dtype);
  if (n > 0 && (!d_exact || !d_approx)) return set_error(HPAC_EINVAL, "NULL data pointer");
  *h_result = hpac_quality_result{0.0, 0.0, 0, 0, 0};
  int dev = 0;
  HPAC_CUDA_TRY(cudaGetDevice(&dev));
  Partial *scr = nullptr;
  hpac_status s = static_scratch(dev, &scr);
  if (s != HPAC_OK) return s;
  if (n == 0) {
    // The warm-up call: besides the address lookup above, make the runtime
    // load the kernels now (with lazy module loading they would load, and
    // allocate device memory for their code, at their first launch).
    cudaFuncAttributes fa;
    for (int32_t dt : {HPAC_F32, HPAC_F64})
      for (int32_t m : {HPAC_METRIC_MAPE, HPAC_METRIC_RMSE, HPAC_METRIC_MCR})
        HPAC_CUDA_TRY(cudaFuncGetAttributes(&fa, partial_kernel(dt, m)));
    return HPAC_OK;
  }
  cudaStream_t st = (cudaStream_t)cuda_stream;
  // Every partial slot the last block reads is written earlier in this call,
  // and the ticket is cleared first: overlapping calls (which spoil one another's
  // results) can leave it at any count.
  HPAC_CUDA_TRY(cudaMemsetAsync(scr + kStaticPartials + 1, 0, sizeof(unsigned), st));
  const int64_t blocks = (n + kStaticTile - 1) / kStaticTile;
  partial_kernel(approx_dtype, metric)<<<(unsigned)blocks, kThreads, 0, st>>>(
      d_exact, d_approx, n, scr, reinterpret_cast<unsigned *>(scr + kStaticPartials + 1),
      scr + kStaticPartials);
  HPAC_CUDA_TRY(cudaGetLastError());
  Partial res;
  HPAC_CUDA_TRY(
      cudaMemcpyAsync(&res, scr + kStaticPartials, sizeof(Partial), cudaMemcpyDeviceToHost, st));
  HPAC_CUDA_TRY(cudaStreamSynchronize(st));
  double v = res.used ? res.sum / (double)res.used : 0.0;
  if (metric == HPAC_METRIC_RMSE) v = sqrt(v);
  h_result->value = v;
  h_result->zero_max_abs = res.zmax;
  h_result->used = (int64_t)res.used;
  h_result->zeros = (int64_t)res.zeros;
  h_result->zeros_mismatch = (int64_t)res.zbad;
  return HPAC_OK;
}
