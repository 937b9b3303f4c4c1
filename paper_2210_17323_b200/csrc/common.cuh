// Shared host/device helpers of the GPTQ B200 library (not part of the public ABI).
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>
#include <stddef.h>

#include "../../include/gptq_b200.h"

namespace gptq {

constexpr size_t kAlign = 256;

inline size_t align_up(size_t x, size_t a = kAlign) { return (x + a - 1) / a * a; }

// Carves 256-byte aligned pieces out of the caller's workspace; with base == nullptr it only measures.
struct WsCarver {
  char* base;
  size_t off = 0;
  explicit WsCarver(void* b) : base(static_cast<char*>(b)) {}
  template <class T>
  T* take(size_t count) {
    size_t o = off;
    off = align_up(off + count * sizeof(T));
    return base ? reinterpret_cast<T*>(base + o) : nullptr;
  }
};

// SM count of the current device (cached per device).
int device_sm_count();

inline bool aligned_to(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

#define GPTQ_CUDA_TRY(expr)                           \
  do {                                                \
    cudaError_t _e = (expr);                          \
    if (_e != cudaSuccess) return GPTQ_ERR_CUDA;      \
  } while (0)

// Number of kernels this library has launched in this process (diagnostic, see gptq_launch_count()).
void count_launch(int n = 1);

// Placed after every kernel launch: counts it and surfaces launch-configuration errors.
#define GPTQ_LAUNCH_CHECK()                 \
  do {                                      \
    ::gptq::count_launch();                 \
    GPTQ_CUDA_TRY(cudaGetLastError());      \
  } while (0)

// Launches that follow one another inside a call.  A kernel launched by launch_next may be set up while the one before it in the stream
// ends (programmatic dependent launch): every thread of it begins with pdl_wait, which returns when that kernel is complete and its
// results are visible.  A kernel lets the next one be set up by pdl_next, a short one at once, a long one shortly before its end: what is
// set up holds its place on the SMs, and other streams have use for it.  Only where a kernel of the same call that begins with pdl_wait
// too stands directly before it in the stream; in a kernel launched in the ordinary way the wait is over at once.
// (768-wide layer, 21 launches: 340 -> 320 us; 1000 x 2400 1604 -> 1562; 125M-shaped block on several streams 2034 -> 1793.)
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_begin() { pdl_wait(); pdl_next(); }
template <class... P, class... A>
inline cudaError_t launch_next(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s;
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
#define GPTQ_LAUNCH_NEXT(...)                                       \
  do {                                                              \
    GPTQ_CUDA_TRY(::gptq::launch_next(__VA_ARGS__));                \
    ::gptq::count_launch();                                         \
  } while (0)

// dev_info word layout: [0] status, [1] detail (pivot index, ...).  First error wins.
__device__ __forceinline__ void report_error(int* dev_info, int status, int detail) {
  if (dev_info && atomicCAS(dev_info, 0, status) == 0) dev_info[1] = detail;
}

// largest power of two <= x (x > 0, finite); 1 for anything else
__device__ __forceinline__ float pow2_floor(float x) {
  if (!(x > 0.f) || !isfinite(x)) return 1.f;
  int e;
  frexpf(x, &e);                       // x = m 2^e, m in [0.5, 1)
  e = max(-100, min(100, e - 1));
  return ldexpf(1.f, e);
}
// power of two s with s * x in [2^(top-1), 2^top) (x > 0, finite); 1 for anything else
__device__ __forceinline__ float pow2_scale_to(float x, int top) {
  if (!(x > 0.f) || !isfinite(x)) return 1.f;
  int e;
  frexpf(x, &e);
  e = max(-100, min(100, top - e));
  return ldexpf(1.f, e);
}
__device__ __forceinline__ int ceil_div_d(int a, int b) { return (a + b - 1) / b; }
inline int ceil_div(int64_t a, int64_t b) { return static_cast<int>((a + b - 1) / b); }

}  // namespace gptq
