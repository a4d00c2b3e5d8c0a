// Shared host/device helpers of libsao: status handling, launch bookkeeping,
// the device error word and small device utilities.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/sao.h"

namespace sao {

// ----------------------------------------------------------------------------
// host side
// ----------------------------------------------------------------------------

// Records `msg` as the calling thread's last error and returns `st`.
sao_status fail(sao_status st, const char *fmt, ...);
const char *last_error();
void set_checked(int on);
void profile_enable(int on);
void profile_reset();
int profile_read(const char **names, int64_t *launches, double *total_ms, int cap);

// Wraps a CUDA runtime call: on failure records the error and returns SAO_ERR_CUDA.
#define SAO_CUDA_TRY(expr)                                                       \
  do {                                                                           \
    cudaError_t e_ = (expr);                                                     \
    if (e_ != cudaSuccess)                                                       \
      return ::sao::fail(SAO_ERR_CUDA, "%s: %s (%s:%d)", #expr,                  \
                         cudaGetErrorString(e_), __FILE__, __LINE__);            \
  } while (0)

#define SAO_TRY(expr)                                                            \
  do {                                                                           \
    sao_status s_ = (expr);                                                      \
    if (s_ != SAO_OK) return s_;                                                 \
  } while (0)

// Called after every kernel launch: picks up launch errors and, when kernel
// profiling is on, closes the event pair opened by launch_begin.
int launch_begin(const char *kind, cudaStream_t s);
sao_status launch_end(int slot, cudaStream_t s);

// A launch that may begin while the kernel before it in the stream still runs
// (programmatic dependent launch): pdl(kernel, grid, block, smem, stream)(args).
// The kernel starts with grid_wait(), which returns once everything before it
// in the stream is done and visible, so the order of (coherent) memory accesses is
// that of ordinary launches; what overlaps is the launch itself, 1-2 us for each of
// the 5 to 15 launches of a call. Every CTA of such a kernel has to pass grid_wait(),
// also one with nothing to do, or the kernel after it could start too early.
template <class... P>
struct PdlLaunch {
  void (*kernel)(P...);
  dim3 grid, block;
  size_t smem;
  cudaStream_t stream;
  template <class... A>
  void operator()(A &&...args) const {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<A &&>(args)...);  // errors: launch_end reads the last one
  }
};
template <class... P>
PdlLaunch<P...> pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s) {
  return PdlLaunch<P...>{kernel, grid, block, smem, s};
}

// Zeros `bytes` (a multiple of 4) of a 16-byte aligned scratch buffer with a launch
// of its own kind: a memset keeps the kernels on both sides of it apart, which
// cost 1-2 us of the idle GPU in a call of three launches.
sao_status clear_scratch(void *p, size_t bytes, cudaStream_t s);

// Device properties of the current device (cached per device).
struct DeviceInfo {
  int device;
  int sm_count;
  int cc_major, cc_minor;
  size_t smem_optin;
};
sao_status device_info(DeviceInfo *out);

// Every workspace starts with a 256-byte header whose first word is the
// device error word of the calls that use it. begin_call clears it in checked
// mode; finish_call (checked mode) synchronises, reads and reports it.
constexpr size_t kWsHeader = 256;
sao_status begin_call(void *ws, cudaStream_t s);
sao_status finish_call(void *ws, cudaStream_t s);
bool checked_mode();

bool aligned16(const void *p);

// Workspace carving: hands out 256-byte aligned slices of the caller's buffer.
struct Carver {
  char *base;
  size_t cap;
  size_t off = 0;
  Carver(void *b, size_t c) : base(static_cast<char *>(b)), cap(c) {}
  template <class T>
  T *take(size_t count) {
    size_t bytes = (count * sizeof(T) + 255) & ~size_t(255);
    T *p = reinterpret_cast<T *>(base + off);
    off += bytes;
    return p;
  }
  bool ok() const { return off <= cap; }
};

inline size_t round256(size_t b) { return (b + 255) & ~size_t(255); }

// ----------------------------------------------------------------------------
// device side
// ----------------------------------------------------------------------------

// First statement of a kernel launched with pdl(): waits for everything before
// it in the stream. A small grid then lets the next kernel be launched as soon as
// every CTA of this one has started (it waits in its own grid_wait()); a large
// one, and a GEMM (grid_wait_long), only as its CTAs exit: CTAs that wait on the
// SMs for a long kernel slowed it (forward GEMM of the large head 2.86 -> 3.05 ms).
constexpr unsigned kEarlyGrid = 304;
__device__ __forceinline__ void grid_wait_long() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_wait() {
  grid_wait_long();
  if (gridDim.x <= kEarlyGrid) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// A load of global memory. The lifetime of a kernel launched with pdl() overlaps that
// of the kernel before it, which may have written any of its inputs, so nothing is
// read-only during it and the non-coherent path (ld.global.nc: __ldg, const
// __restrict__) is not defined. This is an ordinary load; the clobber in grid_wait()
// keeps it behind the wait. (As volatile __ldca() loads, which may pass the stores
// before them, the running mean and the scan were slower: 1,048,909 tokens 37.4 us
// against 33.3 for the calls of the running-mean arm.)
template <class T>
__device__ __forceinline__ T ld(const T *p) {
  return *p;
}

// Kernels OR SAO_DEVERR_* bits into the workspace's error word.
__device__ __forceinline__ void raise_device_error(unsigned int *err, unsigned int bits) {
  atomicOr(err, bits);
}

__device__ __forceinline__ uint64_t globaltimer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Every wait on another CTA or on an mbarrier gives up after this long (or
// after kSpinLimit polls), raises an error bit and lets the kernel finish.
constexpr uint64_t kWaitLimitNs = 2000000000ull;  // 2 s
constexpr uint32_t kSpinLimit = 1u << 28;

}  // namespace sao
