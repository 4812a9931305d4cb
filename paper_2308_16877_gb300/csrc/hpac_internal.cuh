// Internal declarations shared by the translation units of libhpac.
#pragma once

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>
#include <math.h>
#include <stdint.h>

#include "hpac.h"

struct hpac_region {
  hpac_region_desc d;
  cudaStream_t stream;
  int device;
  unsigned long long *d_counters;  // [0] approximated, [1] borderline
  int persist;                     // TAF windows / iACT tables kept across calls
  void *d_state;                   // their device copy (region-owned)
  size_t state_bytes;
  int64_t state_key[6];            // technique and shape the copy holds
  const void *aux;                 // K-Means: the caller's centroids (device)
};

namespace hpac {

constexpr int kWarp = 32;
constexpr int kMaxIn = 8;
constexpr int kMaxHsize = 64;
constexpr int kMaxTsize = 64;
constexpr int kMaxBinomialSteps = 1024;
constexpr int kMaxClusters = 64;
constexpr double kBorderRel = 1e-6;

// Thread-local error reporting (hpac_last_error).
hpac_status set_error(hpac_status s, const char *fmt, ...);
hpac_status cuda_error(cudaError_t e, const char *what);

inline int64_t logical_threads(const hpac_region_desc &d) {
  return d.logical_threads > 0 ? d.logical_threads : (d.n > 0 ? d.n : 1);
}

// Launchers (one translation unit each). All validate nothing: the C ABI layer
// has checked the descriptor and knobs before calling them.
hpac_status launch_exact(const hpac_region *r, const void *in, void *out);
hpac_status launch_perfo(const hpac_region *r, const hpac_perfo_knobs *k, const void *in, void *out,
                         uint8_t *mask, unsigned long long *counters);
hpac_status launch_taf(hpac_region *r, const hpac_taf_knobs *k, const void *in, void *out,
                       uint8_t *mask, void *stat, unsigned long long *counters);
hpac_status launch_iact(hpac_region *r, const hpac_iact_knobs *k, const void *in, void *out,
                        uint8_t *mask, void *stat, unsigned long long *counters);

// The Binomial region: every technique runs in binomial.cu's team kernels
// (technique 0 exact, 1 TAF, 2 iACT, 3 perforation; knobs of that technique).
hpac_status launch_binomial(hpac_region *r, int technique, const void *knobs, const void *in,
                            void *out, uint8_t *mask, void *stat, unsigned long long *counters);

// The persistent state buffer of a TAF or iACT run: nullptr when the region
// keeps no state; otherwise a zeroed buffer of `bytes` the first time a shape
// (key) is seen, the previous run's buffer when the key repeats.
hpac_status region_state(hpac_region *r, const int64_t (&key)[6], size_t bytes, void **out);

inline size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

// A named NVTX range around a library call, for timeline tools (Nsight
// Systems, ncu --nvtx); without a tool attached the push and pop return at
// once.
struct TraceRange {
  explicit TraceRange(const char *name) { nvtxRangePushA(name); }
  ~TraceRange() { nvtxRangePop(); }
  TraceRange(const TraceRange &) = delete;
  TraceRange &operator=(const TraceRange &) = delete;
};

// Largest dynamic shared memory a block of this device may use.
int max_dyn_smem(int device);

// Number of SMs of the device.
int sm_count(int device);

// Physical block size (a multiple of 32, at most b) for a launch of `threads`
// threads whose block is not part of the semantics (plain maps, thread- and
// warp-level decisions): small enough to give every SM about eight blocks.
// The work of a region is often uneven along the invocation index (a shock
// front, a run of approximations), and double-precision work runs at a small
// fraction of the single-precision rate, so a few large blocks left on a few
// SMs would set the kernel time.
int balanced_block(int64_t threads, int b, int device);

// Launch with programmatic stream serialization: the kernel may be scheduled
// while the launch before it in the stream drains. Every thread of a kernel
// launched this way calls grid_wait() before its first access to global memory,
// which returns when everything before it in the stream is complete and visible.
// Inputs are read with coherent loads: the kernel may have started before they
// were written. Between launches of a few microseconds the gap is a third of the
// time: exact, TAF and perforated prices of 65,536 options 14.3 -> 12.1 us, a 64^3
// hydro step 58.2 -> 54.7, a training batch of 8192 19.4 -> 17.5.
// No kernel lets its successor be scheduled earlier than its own blocks end
// (griddepcontrol.launch_dependents at its start): the successor's blocks then take
// the places that are free while this one runs, many on few SMs, and stay there.
// Ten steps at 32^3 under TAF took 484 us that way, 231 without (400 with
// launches one after another), at 64^3 1011 and 837, 64 training batches 1138 and
// 1117; no call gained by it.
template <class... P, class... A>
inline cudaError_t launch_chained(void (*kernel)(P...), unsigned blocks, unsigned threads, size_t smem,
                                  cudaStream_t stream, A... args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

#ifdef __CUDACC__
// An exactly computing lane's key for the choice of its table's writer (the largest
// key, ties to the lowest lane; -1 for the other lanes), L lanes to a table. A
// distance that is NaN is farther than none and none is farther than it, so the
// table's first exact lane keeps the entry if its distance is NaN and no other does.
// (As keys NaN would leave lanes with different winners, all of which would write.)
__device__ __forceinline__ float writer_key(bool exact, float dmin, int lane, int L) {
  const float key = exact ? dmin : -1.0f;
  if (!__any_sync(0xffffffffu, key != key)) return key;
  const unsigned lanes = (L == 32 ? 0xffffffffu : (1u << L) - 1u) << (lane & ~(L - 1));
  const unsigned table = __ballot_sync(0xffffffffu, exact) & lanes;
  return key == key ? key : __ffs(table) - 1 == lane ? INFINITY : -1.0f;
}

__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
#endif

}  // namespace hpac

#define HPAC_CUDA_TRY(call)                                   \
  do {                                                        \
    cudaError_t e_ = (call);                                  \
    if (e_ != cudaSuccess) return hpac::cuda_error(e_, #call); \
  } while (0)
