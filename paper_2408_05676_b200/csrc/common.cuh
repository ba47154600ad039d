// Shared host-side helpers of the library: error reporting, argument checks, the
// per-device scratch buffers and small utilities.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/laser.h"

#define LASER_API extern "C" __attribute__((visibility("default")))

namespace laser {

void set_error(const char* fmt, ...);

#define LASER_CUDA(expr)                                                                  \
  do {                                                                                    \
    cudaError_t e_ = (expr);                                                              \
    if (e_ != cudaSuccess) {                                                              \
      ::laser::set_error("%s: %s (%s:%d)", #expr, cudaGetErrorString(e_), __FILE__, __LINE__); \
      return e_ == cudaErrorMemoryAllocation ? LASER_ERR_OOM : LASER_ERR_CUDA;            \
    }                                                                                     \
  } while (0)

#define LASER_REQUIRE(cond, ...)                                                          \
  do {                                                                                    \
    if (!(cond)) {                                                                        \
      ::laser::set_error(__VA_ARGS__);                                                    \
      return LASER_ERR_INVALID_ARG;                                                       \
    }                                                                                     \
  } while (0)

#define LASER_TRY(expr)                                                                   \
  do {                                                                                    \
    laser_status s_ = (expr);                                                             \
    if (s_ != LASER_OK) return s_;                                                        \
  } while (0)

// Scratch of at least `bytes` on the current device for one subsystem (`slot`), 256-byte
// aligned, zero-filled when (re)allocated.  Grows by reallocation (synchronising the
// device), so a pointer is only valid until the next call that asks for more.  Contents
// persist between calls.
enum { SCRATCH_ACCEPT = 0, SCRATCH_DRAFT = 1, SCRATCH_ACCEPT_TREE = 2, SCRATCH_GROUPING = 3, SCRATCH_SLOTS = 4 };
laser_status scratch_get(int slot, size_t bytes, void** out);

// Stream-ordered device memory from a pool of the library's own (one per device, any thread and stream).  Memory given back
// stays with the pool up to 2 GB, so that building and dropping retrieval pools does not go through the driver each time (a
// gigabyte takes it 4 .. 100 ms to hand out and 4 to take back); what is above goes back to the device at the next
// synchronisation, and all of it at laser_trim or when one of the library's allocations finds no memory (device_malloc,
// pooled_alloc).
laser_status pooled_alloc(void** p, size_t bytes, cudaStream_t stream);
void pooled_free(void* p, cudaStream_t stream);
// cudaMalloc for the library's long-lived buffers
cudaError_t device_malloc(void** p, size_t bytes);

// Kernel launch counter (per process) for the statistics.
extern long long g_launches;
inline void count_launch(int n = 1) { g_launches += n; }

inline cudaStream_t as_stream(void* s) { return reinterpret_cast<cudaStream_t>(s); }

template <typename T>
inline T ceil_div(T a, T b) { return (a + b - 1) / b; }

#ifdef __CUDACC__
// The small kernels of a step overlap their launches: each is launched while the one before still runs (launch_overlapped),
// lets the next one be launched from its first instruction on (next_may_launch), and waits for everything before it in the
// stream before it reads or writes global memory (wait_for_earlier; all of a grid's blocks that do work call it, so that a
// kernel's end implies the end of every kernel before it).  What a kernel reads after the wait must not be `const
// __restrict__`: such loads count as invariant and may be moved ahead of it.
__device__ __forceinline__ void next_may_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_earlier() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Device clock in ns, the same on all SMs: the generation loop's stage times are taken by its kernels, since an event between two
// kernels stops them from overlapping.
__device__ __forceinline__ unsigned long long device_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t)::"memory");
  return t;
}

template <typename... P, typename... A>
inline cudaError_t launch_overlapped(void (*kernel)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t stream, A&&... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
#endif

}  // namespace laser
