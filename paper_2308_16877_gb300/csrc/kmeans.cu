// K-Means centroid update, the exact step between two (approximated)
// assignments (Table 1, K-Means: iterate until no observation changes
// cluster). One pass over the observations accumulates the per-cluster
// feature sums and counts in shared memory: one column per thread up to 32
// clusters (fixed point), one copy per warp beyond (double); each block adds its
// columns or copies and then the workspace with one double-precision atomic per
// value; a second tiny kernel divides. Changed assignments are counted in the same pass.
#include "hpac_internal.cuh"

namespace hpac {
namespace {

constexpr int kThreads = 256;

// Each warp accumulates into its own copy of the per-cluster sums, so the
// shared-memory double-precision atomics of one instruction collide only among
// lanes of the same warp and cluster; the copies are then added once per block.
constexpr int kWarps = kThreads / 32;

__global__ void __launch_bounds__(kThreads) kmeans_sums(const float *__restrict__ x, int64_t stride,
                                                        int64_t n, int K,
                                                        const float *__restrict__ assign,
                                                        const float *__restrict__ prev,
                                                        double *__restrict__ sum,
                                                        unsigned long long *__restrict__ cnt,
                                                        unsigned long long *__restrict__ changed) {
  __shared__ double s_sum[kWarps][kMaxClusters * 8];
  __shared__ unsigned s_cnt[kWarps][kMaxClusters];
  const int warp = threadIdx.x >> 5;
  for (int j = threadIdx.x; j < kWarps * K * 8; j += blockDim.x) s_sum[j / (K * 8)][j % (K * 8)] = 0.0;
  for (int j = threadIdx.x; j < kWarps * K; j += blockDim.x) s_cnt[j / K][j % K] = 0;
  __syncthreads();
  double *ws = s_sum[warp];
  unsigned *wc = s_cnt[warp];
  unsigned ch = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float a = assign[i];
    const int k = (int)a;
    if (k >= 0 && k < K) {  // ids are produced in range; anything else is left out
      atomicAdd(&wc[k], 1u);
#pragma unroll
      for (int d = 0; d < 8; ++d) atomicAdd(&ws[k * 8 + d], (double)x[d * stride + i]);
    }
    if (prev && prev[i] != a) ++ch;
  }
  ch = __reduce_add_sync(0xffffffffu, ch);
  if ((threadIdx.x & 31) == 0 && ch) atomicAdd(changed, (unsigned long long)ch);
  __syncthreads();
  for (int j = threadIdx.x; j < K * 8; j += blockDim.x) {
    double v = 0.0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) v += s_sum[w][j];
    if (v != 0.0) atomicAdd(&sum[j], v);
  }
  for (int j = threadIdx.x; j < K; j += blockDim.x) {
    unsigned long long c = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) c += s_cnt[w][j];
    if (c) atomicAdd(&cnt[j], c);
  }
}

// For up to 32 clusters: L observations at a time, each on kParts threads that
// take 8 / kParts features each and keep their own column of per-cluster sums
// (and counts, the first part) in shared memory ([cluster * 8 + d][column],
// conflict-free), so the pass needs no atomics; the block then adds its columns
// (each thread starting at its own column, so the reads spread over the banks)
// and the workspace gets one atomic per value.
//
// The sums are 64-bit integers on a fixed-point grid per block and feature: a
// single-precision value with biased exponent e in [low, low + win] is its
// 24-bit significand shifted left by e - low, so every addition is exact.
// `low` comes from the block's first observations (win - 2 binades below the
// largest exponent seen there); a value outside the window (and every infinity
// and NaN) is added in double precision to a block total instead. A warp of
// which a thread has more than kFar + 1 in 8 such values (data sorted by
// magnitude, blocks that begin with zeros, widely spread values) turns its
// columns into double precision and goes on in that: 4M observations 174 to 198
// us, where the additions to the block total took 355 to 780 (columns in double
// throughout 160 to 253, values on the grid 65 to 105). win is at most
// 24 and leaves room for the thread's number of additions in 63 bits. Sums in
// double took a conversion and an addition per value, 16 operations per
// observation on a pipe that issues two per SM and clock: 107 us for 4M
// observations, where reading them takes 25.
//
// The columns leave room for about 200 observations at a time per SM at 16
// clusters, so two threads share one (13 warps per SM instead of 6), and each
// keeps four observations in flight and four more ahead, 16 bytes per load
// where rows and pointers are aligned (VEC), else four coalesced loads.
// One iteration over 4M observations (assignment and update): 216 us with sums
// in double, 139 with one thread per observation, 120 with two.
constexpr int kObs = 4;   // observations per thread and step
constexpr int kParts = 2; // threads per observation
constexpr int kOwn = 8 / kParts;  // features per thread
constexpr int kWin = 24;  // widest exponent window
constexpr int kFar = 4;   // values off the grid a thread may have anyway

template <int L, bool VEC>
__global__ void __launch_bounds__(L * kParts) kmeans_sums_private(const float *__restrict__ x, int64_t stride,
                                                         int64_t n, int K, int win,
                                                         const float *__restrict__ assign,
                                                         const float *__restrict__ prev,
                                                         double *__restrict__ sum,
                                                         unsigned long long *__restrict__ cnt,
                                                         unsigned long long *__restrict__ changed) {
  extern __shared__ __align__(16) long long s_acc[];                  // [K * 8][L]
  double *s_far = reinterpret_cast<double *>(s_acc + K * 8 * L);      // [K * 8]: values off the grid
  unsigned *s_n = reinterpret_cast<unsigned *>(s_far + K * 8);        // [K][L]
  __shared__ unsigned s_top[8];
  constexpr int NT = L * kParts;
  __shared__ bool s_double[NT / 32];  // the warp's columns are in double precision
  const int tid = threadIdx.x, part = tid / L, col = tid % L, d0 = part * kOwn;
  for (int j = tid; j < K * 8 * L; j += NT) s_acc[j] = 0;
  for (int j = tid; j < K * 8; j += NT) s_far[j] = 0.0;
  for (int j = tid; j < K * L; j += NT) s_n[j] = 0;
  if (tid < 8) s_top[tid] = 0;
  if (tid < NT / 32) s_double[tid] = false;
  __syncthreads();
  // observation j of the group based at g
  auto at = [&](int64_t g, int j) { return VEC ? g + (int64_t)col * kObs + j : g + (int64_t)j * L + col; };
  auto load = [&](const float *row, int64_t g, float (&v)[kObs]) {
    if (VEC && at(g, kObs - 1) < n) {
      const float4 q = *reinterpret_cast<const float4 *>(row + at(g, 0));
      v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
    } else {
#pragma unroll
      for (int j = 0; j < kObs; ++j) v[j] = at(g, j) < n ? row[at(g, j)] : 0.0f;
    }
  };
  const int64_t step = (int64_t)gridDim.x * L * kObs;
  int64_t g = (int64_t)blockIdx.x * L * kObs;
  float a[kObs], pa[kObs], xv[kOwn][kObs];
  auto fetch = [&](int64_t from, float (&fa)[kObs], float (&fp)[kObs], float (&fx)[kOwn][kObs]) {
    load(assign, from, fa);
    if (prev && part == 0) load(prev, from, fp);
#pragma unroll
    for (int d = 0; d < kOwn; ++d) load(x + (d0 + d) * stride, from, fx[d]);
  };
  fetch(g, a, pa, xv);
#pragma unroll
  for (int d = 0; d < kOwn; ++d) {
    unsigned e = 0;
#pragma unroll
    for (int j = 0; j < kObs; ++j) {
      const unsigned ej = (__float_as_uint(xv[d][j]) >> 23) & 0xffu;
      if (ej < 255u) e = max(e, ej);
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if ((tid & 31) == 0) atomicMax(&s_top[d0 + d], e);
  }
  __syncthreads();
  int low[kOwn];
#pragma unroll
  for (int d = 0; d < kOwn; ++d) low[d] = min(max((int)s_top[d0 + d] + 2, win + 1), 254) - win;
  unsigned ch = 0;
  auto unit_of = [](int lo) { return __hiloint2double((lo - 150 + 1023) << 20, 0); };  // 2^(lo - 150)
  int n_far = 0, allowed = kFar;
  bool on_grid = true;
  for (; g < n && on_grid; g += step) {
    float an[kObs], pn[kObs], xn[kOwn][kObs];
    if (g + step < n) fetch(g + step, an, pn, xn);
#pragma unroll
    for (int j = 0; j < kObs; ++j) {
      if (at(g, j) >= n) continue;
      const int k = (int)a[j];
      if (k >= 0 && k < K) {  // ids are produced in range; anything else is left out
        if (part == 0) s_n[k * L + col] += 1;
        long long v[kOwn];
        unsigned far = 0;
#pragma unroll
        for (int d = 0; d < kOwn; ++d) {
          const unsigned bits = __float_as_uint(xv[d][j]);
          const int m = (int)((bits & 0x7fffffu) | 0x800000u);
          const unsigned sh = ((bits >> 23) & 0xffu) - (unsigned)low[d];
          v[d] = (long long)((int)bits < 0 ? -m : m) << (sh & 31u);
          far |= (sh > (unsigned)win ? 1u : 0u) << d;
        }
        if (far) {
#pragma unroll
          for (int d = 0; d < kOwn; ++d)
            if (far >> d & 1u) {
              v[d] = 0;
              if (xv[d][j] != 0.0f) {
                atomicAdd(&s_far[k * 8 + d0 + d], (double)xv[d][j]);
                ++n_far;
              }
            }
        }
        long long *acc = s_acc + (size_t)(k * 8 + d0) * L + col;
#pragma unroll
        for (int d = 0; d < kOwn; ++d) acc[d * L] += v[d];
      }
      if (prev && part == 0 && pa[j] != a[j]) ++ch;
    }
#pragma unroll
    for (int j = 0; j < kObs; ++j) {
      a[j] = an[j];
      pa[j] = pn[j];
#pragma unroll
      for (int d = 0; d < kOwn; ++d) xv[d][j] = xn[d][j];
    }
    allowed += kOwn * kObs / 8;
    on_grid = !__any_sync(0xffffffffu, n_far > allowed);
  }
  if (!on_grid) {  // the same on every lane of a warp
    if ((tid & 31) == 0) s_double[tid >> 5] = true;
    for (int k = 0; k < K; ++k)
#pragma unroll
      for (int d = 0; d < kOwn; ++d) {
        long long *acc = s_acc + (size_t)(k * 8 + d0 + d) * L + col;
        *acc = __double_as_longlong((double)*acc * unit_of(low[d]));
      }
    for (; g < n; g += step) {
      float an[kObs], pn[kObs], xn[kOwn][kObs];
      if (g + step < n) fetch(g + step, an, pn, xn);
#pragma unroll
      for (int j = 0; j < kObs; ++j) {
        if (at(g, j) < n) {
          const int k = (int)a[j];
          if (k >= 0 && k < K) {
            if (part == 0) s_n[k * L + col] += 1;
            long long *acc = s_acc + (size_t)(k * 8 + d0) * L + col;
#pragma unroll
            for (int d = 0; d < kOwn; ++d)
              acc[d * L] = __double_as_longlong(__longlong_as_double(acc[d * L]) + (double)xv[d][j]);
          }
          if (prev && part == 0 && pa[j] != a[j]) ++ch;
        }
        a[j] = an[j];
        pa[j] = pn[j];
#pragma unroll
        for (int d = 0; d < kOwn; ++d) xv[d][j] = xn[d][j];
      }
    }
  }
  ch = __reduce_add_sync(0xffffffffu, ch);
  if ((tid & 31) == 0 && ch) atomicAdd(changed, (unsigned long long)ch);
  const bool mixed = __syncthreads_or(!on_grid);
  for (int j = tid; j < K * 8; j += NT) {
    // the columns' high and low words summed apart (no overflow), joined in
    // double with one rounding
    long long hi = 0;
    unsigned long long lo = 0;
    double far = s_far[j];
    if (!mixed) {
      for (int l = 0; l < L; ++l) {
        const long long v = s_acc[j * L + ((l + tid) & (L - 1))];
        hi += (int)(v >> 32);
        lo += (unsigned)v;
      }
    } else {
      for (int l = 0; l < L; ++l) {
        const int c = (l + tid) & (L - 1);
        const long long v = s_acc[j * L + c];
        if (s_double[((j & 7) / kOwn * L + c) >> 5]) {
          far += __longlong_as_double(v);
        } else {
          hi += (int)(v >> 32);
          lo += (unsigned)v;
        }
      }
    }
    const int lowj = min(max((int)s_top[j & 7] + 2, win + 1), 254) - win;
    const double v = fma((double)hi, 4294967296.0, (double)lo) * unit_of(lowj) + far;
    if (v != 0.0) atomicAdd(&sum[j], v);
  }
  for (int j = tid; j < K; j += NT) {
    unsigned long long c = 0;
    for (int l = 0; l < L; ++l) c += s_n[j * L + ((l + tid) & (L - 1))];
    if (c) atomicAdd(&cnt[j], c);
  }
}

__global__ void kmeans_divide(int K, const double *__restrict__ sum,
                              const unsigned long long *__restrict__ cnt, float *__restrict__ cent) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= K * 8) return;
  const unsigned long long c = cnt[j / 8];
  if (c) cent[j] = (float)(sum[j] / (double)c);  // an empty cluster keeps its centroid
}

}  // namespace
}  // namespace hpac

using namespace hpac;

extern "C" size_t hpac_kmeans_workspace_bytes(int32_t clusters) {
  if (clusters < 1 || clusters > kMaxClusters) return 0;
  return (size_t)(clusters * 8 + clusters + 1) * 8;
}

extern "C" hpac_status hpac_kmeans_update(int64_t n, int32_t clusters, const float *d_x,
                                          int64_t stride, const float *d_assign,
                                          const float *d_prev, float *d_cent, void *d_work,
                                          int64_t *h_changed, void *cuda_stream) {
  TraceRange trace_("hpac_kmeans_update");
  if (n < 0 || clusters < 1 || clusters > kMaxClusters || stride < n)
    return set_error(HPAC_EINVAL, "K-Means update: bad n, clusters or stride");
  if (!d_cent || !d_work || (n > 0 && (!d_x || !d_assign)))
    return set_error(HPAC_EINVAL, "K-Means update: NULL pointer");
  if ((uintptr_t)d_work % 8) return set_error(HPAC_EINVAL, "workspace not 8-byte aligned");
  cudaStream_t s = (cudaStream_t)cuda_stream;
  double *sum = static_cast<double *>(d_work);
  unsigned long long *cnt = reinterpret_cast<unsigned long long *>(sum + clusters * 8);
  unsigned long long *changed = cnt + clusters;
  HPAC_CUDA_TRY(cudaMemsetAsync(d_work, 0, hpac_kmeans_workspace_bytes(clusters), s));
  int dev = 0, sms = 148;
  HPAC_CUDA_TRY(cudaGetDevice(&dev));
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (clusters <= 32) {
    // thread-private columns: 64 observations at a time per block up to 16
    // clusters, 32 up to 32
    const int L = clusters <= 16 ? 64 : 32;
    const size_t smem = (size_t)clusters * 8 * (L + 1) * 8 + (size_t)clusters * L * sizeof(unsigned);
    // 16-byte loads where every row starts on a 16-byte boundary
    const uintptr_t low_bits = (uintptr_t)d_x | (uintptr_t)d_assign | (uintptr_t)d_prev | (uintptr_t)stride * 4;
    const bool vec = low_bits % 16 == 0;
    auto fn = L == 64 ? (vec ? kmeans_sums_private<64, true> : kmeans_sums_private<64, false>)
                      : (vec ? kmeans_sums_private<32, true> : kmeans_sums_private<32, false>);
    HPAC_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 1;
    HPAC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, L * kParts, smem));
    const int64_t group = (int64_t)L * kObs;
    int64_t blocks = (n + group - 1) / group;
    const int64_t cap = (int64_t)sms * (per_sm < 1 ? 1 : per_sm);
    blocks = blocks < 1 ? 1 : blocks > cap ? cap : blocks;
    // a thread's sum stays below 2^62: 24 + win bits per value, 2^(38 - win) values
    const int64_t per_thread = ((n + group - 1) / group + blocks - 1) / blocks * kObs;
    int win = kWin;
    while (win > 0 && per_thread > (int64_t)1 << (38 - win)) --win;
    fn<<<(unsigned)blocks, L * kParts, smem, s>>>(d_x, stride, n, clusters, win, d_assign, d_prev, sum, cnt, changed);
  } else {
    int64_t blocks = (n + kThreads - 1) / kThreads;
    const int64_t cap = (int64_t)sms * 4;
    blocks = blocks < 1 ? 1 : blocks > cap ? cap : blocks;
    kmeans_sums<<<(unsigned)blocks, kThreads, 0, s>>>(d_x, stride, n, clusters, d_assign, d_prev, sum,
                                                        cnt, changed);
  }
  HPAC_CUDA_TRY(cudaGetLastError());
  kmeans_divide<<<(clusters * 8 + 255) / 256, 256, 0, s>>>(clusters, sum, cnt, d_cent);
  HPAC_CUDA_TRY(cudaGetLastError());
  if (h_changed) {
    unsigned long long c = 0;
    HPAC_CUDA_TRY(cudaMemcpyAsync(&c, changed, sizeof(c), cudaMemcpyDeviceToHost, s));
    HPAC_CUDA_TRY(cudaStreamSynchronize(s));
    *h_changed = (int64_t)c;
  }
  return HPAC_OK;
}
