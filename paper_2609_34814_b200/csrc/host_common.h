// Host-side helpers shared by the entry points: thread-local error text and launch counter.
#pragma once
#include <cstdarg>
#include <cstdio>
#include <cuda_runtime.h>
#include "waveal.h"

namespace waveal {

char* last_error_buffer();          // thread-local, 512 bytes
int32_t& launch_counter();          // thread-local

inline waveal_status fail(waveal_status s, const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(last_error_buffer(), 512, fmt, ap);
  va_end(ap);
  return s;
}

inline bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

#ifdef __CUDACC__
// The kernels of one call that follow each other on the stream: each is launched while the one before it
// drains (programmatic dependent launch), sets itself up, and waits before it touches what that one
// writes.  Every kernel launched this way waits, so whoever follows the last one follows all of them.
// The first kernel of a call is launched the ordinary way: it starts when all earlier work has ended.
__device__ __forceinline__ void wait_for_previous_kernel() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next_kernel_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... Params, class... Args>
inline cudaError_t launch_chained(void (*kernel)(Params...), dim3 grid, int threads, size_t smem, cudaStream_t stream,
                                  Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}
#endif

#define WAVEAL_CUDA_OK(expr)                                                                 \
  do {                                                                                       \
    cudaError_t e__ = (expr);                                                                \
    if (e__ != cudaSuccess)                                                                  \
      return ::waveal::fail(WAVEAL_ERR_CUDA, "%s failed: %s", #expr, cudaGetErrorString(e__)); \
  } while (0)

}  // namespace waveal
