// Host-side helpers shared by the entry points: argument checks and the launch counter.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "unstep.h"

namespace unstep {

constexpr int kHeadDim = 128;
constexpr int kPairs = 64;
constexpr int kMaxStreamsPerLaunch = 32;  // per-stream host scalars travel as kernel parameters

extern std::atomic<int64_t> g_launches;

// Device address of the status word on the current device (null if it cannot be found).
int* status_word();

// A checking build (-DUNSTEP_CHECK) tests every global store of the kernels against the extent of
// the buffer it belongs to; a store outside is skipped and recorded in the status word (no trap),
// so that a wrong index shows up as UNSTEP_ERR_BOUNDS instead of silent corruption.  This stands
// in for a memory checker where none can be run.  In a normal build the macros are the plain stores.
// UNSTEP_STORE_32 stores 32 bytes, two 16-byte vectors of `base` from vector `idx` on.
#ifdef UNSTEP_CHECK
#define UNSTEP_STORE(base, idx, extent, value, status)                                  \
  do {                                                                                  \
    const long long idx_ = static_cast<long long>(idx);                                 \
    if (idx_ >= 0 && idx_ < static_cast<long long>(extent)) (base)[idx_] = (value);     \
    else atomicExch((status), static_cast<int>(UNSTEP_ERR_BOUNDS));                     \
  } while (0)
#define UNSTEP_STORE_32(base, idx, extent, words, status)                               \
  do {                                                                                  \
    const long long idx_ = static_cast<long long>(idx);                                 \
    if (idx_ >= 0 && idx_ + 2 <= static_cast<long long>(extent)) ptx::st_global_32((base) + idx_, (words)); \
    else atomicExch((status), static_cast<int>(UNSTEP_ERR_BOUNDS));                     \
  } while (0)
#else
#define UNSTEP_STORE(base, idx, extent, value, status) ((base)[idx] = (value))
#define UNSTEP_STORE_32(base, idx, extent, words, status) ptx::st_global_32((base) + (idx), (words))
#endif

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Shape checks common to every call.  `need_ring` also checks batch/heads/ring_frames.
inline int check_shape(const unstep_shape_t* s, bool need_ring) {
  if (s == nullptr) return UNSTEP_ERR_INVALID_ARG;
  if (s->head_dim != kHeadDim) return s->head_dim > 0 ? UNSTEP_ERR_UNSUPPORTED : UNSTEP_ERR_INVALID_ARG;
  if (s->chunk_frames <= 0 || s->grid_h <= 0 || s->grid_w <= 0) return UNSTEP_ERR_INVALID_ARG;
  if (s->band_t <= 0 || s->band_h <= 0 || s->band_w <= 0) return UNSTEP_ERR_INVALID_ARG;
  if ((s->band_t | s->band_h | s->band_w) & 1) return UNSTEP_ERR_INVALID_ARG;
  if (s->band_t + s->band_h + s->band_w != s->head_dim) return UNSTEP_ERR_INVALID_ARG;
  if (!(s->rope_base > 0.0)) return UNSTEP_ERR_INVALID_ARG;
  const int64_t T = static_cast<int64_t>(s->grid_h) * s->grid_w;
  const int64_t L = T * s->chunk_frames;
  if (T > (1 << 24) || L > (1 << 26)) return UNSTEP_ERR_INVALID_ARG;
  if (need_ring) {
    if (s->batch <= 0 || s->heads <= 0 || s->ring_frames <= 0) return UNSTEP_ERR_INVALID_ARG;
    if (s->ring_frames < s->chunk_frames) return UNSTEP_ERR_INVALID_ARG;
    if (s->heads > 4096 || s->batch > (1 << 20)) return UNSTEP_ERR_INVALID_ARG;
    // element offsets inside one stream's ring must fit comfortably in 63 bits / TMA strides in 40
    const int64_t ring_elems = static_cast<int64_t>(s->ring_frames) * T * s->heads * kHeadDim;
    if (ring_elems > (int64_t(1) << 38)) return UNSTEP_ERR_INVALID_ARG;
  }
  return UNSTEP_OK;
}

// Launch whose set-up may, with `overlap`, run while the kernel before it on the stream finishes
// (programmatic dependent launch).  Every kernel launched this way passes grid_wait(), which returns
// when all earlier work of the stream is complete and visible, before it touches global memory; so
// it also completes only after that work, and the kernel behind it may rely on the same.  Between
// kernels of one stream this hides the 2-3 us of launch, scheduling and prologue: back to back, the
// append of four streams 57.4 -> 55.5 us, the append behind the norm 18.7 -> 17.7, the table of
// 3 x 45 x 80 tokens 6.1 -> 4.6, append and attention of a toy layer 22.5 -> 16.8.
// With `cluster` > 1, that many neighbouring blocks form a cluster.
template <typename... KernelArgs, typename... Args>
inline cudaError_t launch_clusters(bool overlap, unsigned cluster, void (*kernel)(KernelArgs...), dim3 grid, dim3 block,
                                   size_t smem, cudaStream_t stream, const Args&... args) {
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (overlap) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = cluster;
    attr[n].val.clusterDim.y = 1;
    attr[n++].val.clusterDim.z = 1;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = n;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<KernelArgs>(args)...);
  return cudaGetLastError();
}
template <typename... KernelArgs, typename... Args>
inline cudaError_t launch_overlapped(bool overlap, void (*kernel)(KernelArgs...), dim3 grid, dim3 block,
                                     size_t smem, cudaStream_t stream, const Args&... args) {
  return launch_clusters(overlap, 1, kernel, grid, block, smem, stream, args...);
}

#if defined(__CUDACC__)
// Returns 0, as a value that only exists behind the wait.  What a kernel reads may be written while it is
// already running, so no load may move above the wait, as the compiler may move __ldcs and its like,
// which clobber nothing: their addresses take this 0 in.  Nor may such a load be an __ldg or go
// through a `const __restrict__` pointer: those become ld.global.nc, which is for data that nobody
// writes during the kernel's lifetime, and that began before the wait.  __ldca and __ldcs are coherent.
__device__ __forceinline__ int grid_wait() {
  int zero;
  asm volatile("griddepcontrol.wait;\nmov.u32 %0, 0;" : "=r"(zero)::"memory");
  return zero;
}
// The next kernel of the stream may be set up once every block has called this or has ended.  The
// append and the table call it first thing: their blocks are short, and the attention behind them
// needs a whole SM, which it only gets when their blocks there are done.  The attention does not:
// blocks of the next kernel that wait on SMs it leaves idle would keep other streams' work from them.
__device__ __forceinline__ void grid_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
#endif

// The device the call will run on must be sm_100.
inline int check_device() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return UNSTEP_ERR_CUDA;
  static thread_local int cached_dev = -1, cached_major = 0;
  if (cached_dev != dev) {
    int major = 0;
    if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess)
      return UNSTEP_ERR_CUDA;
    cached_dev = dev;
    cached_major = major;
  }
  return cached_major == 10 ? UNSTEP_OK : UNSTEP_ERR_UNSUPPORTED;
}

}  // namespace unstep
