// Shared host-side plumbing of the library: status codes, CUDA error capture, argument checks.
#pragma once
#include <cuda_runtime.h>
#include <utility>
#include <cuda_bf16.h>
#include <stdint.h>
#include <stddef.h>
#include "../../include/shadowsync.h"

namespace ss {

extern thread_local int g_last_cuda_error;

inline ss_status cuda_fail(cudaError_t e) {
  g_last_cuda_error = (int)e;
  return SS_ERR_CUDA;
}

#define SS_CUDA(expr)                                  \
  do {                                                 \
    cudaError_t e__ = (expr);                          \
    if (e__ != cudaSuccess) return ss::cuda_fail(e__); \
  } while (0)

// Launch check: picks up a failed launch without synchronising.
#define SS_LAUNCH_OK()                                  \
  do {                                                  \
    cudaError_t e__ = ss::g_step_sink ? cudaSuccess : cudaGetLastError(); \
    if (e__ != cudaSuccess) return ss::cuda_fail(e__);  \
  } while (0)

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
inline cudaStream_t as_stream(ss_stream s) { return reinterpret_cast<cudaStream_t>(s); }

// What the calls of a training step enqueue.  While a step plan records a step or brings its graph up to date with one
// (step.cu), their kernels and events go to it; otherwise g_step_sink is null and they go to the streams.
struct LaunchShape {
  const void* kernel;
  dim3 grid, block;
  size_t smem;
  int cluster;
};
struct StepSink {
  virtual cudaError_t kernel(const LaunchShape& shape, cudaStream_t st, void** params, const size_t* sizes, int n) = 0;
  virtual cudaError_t record(cudaEvent_t e, cudaStream_t st) = 0;
  virtual cudaError_t wait(cudaStream_t st, cudaEvent_t e) = 0;
  virtual void ctas(int n) = 0;                            // how many CTAs a tensor-core launch was given
  int device = 0;
 protected:
  ~StepSink() = default;
};
extern thread_local StepSink* g_step_sink;
cudaError_t launch_now(const LaunchShape& shape, cudaStream_t st, void** params);   // a programmatic dependent launch
inline cudaError_t current_device(int* dev) {              // (a step asks two to four dozen times)
  if (!g_step_sink) return cudaGetDevice(dev);
  *dev = g_step_sink->device;
  return cudaSuccess;
}
inline cudaError_t step_record(cudaEvent_t e, cudaStream_t st) { return g_step_sink ? g_step_sink->record(e, st) : cudaEventRecord(e, st); }
inline cudaError_t step_wait(cudaStream_t st, cudaEvent_t e) { return g_step_sink ? g_step_sink->wait(st, e) : cudaStreamWaitEvent(st, e, 0); }

#ifdef __CUDACC__
// Two independent fused multiply-adds in one instruction (sm_100); each rounds like fmaf.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(d)
      : "l"(*reinterpret_cast<const uint64_t*>(&a)), "l"(*reinterpret_cast<const uint64_t*>(&b)), "l"(*reinterpret_cast<const uint64_t*>(&c)));
  return *reinterpret_cast<const float2*>(&d);
}
#endif

#ifdef __CUDACC__
// Programmatic dependent launch: the kernel may be brought onto the device while the one before it on the stream drains,
// and waits, as the first thing every one of its threads does, until that kernel is complete and its stores are visible.
// The gap between dependent kernels of a few microseconds all but closes (from about 2.4 us).
__device__ __forceinline__ void wait_for_previous_kernel() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <typename... P>
inline cudaError_t launch_params(const LaunchShape& shape, cudaStream_t st, const P&... args) {
  void* ptr[] = {const_cast<void*>(static_cast<const void*>(&args))...};
  const size_t size[] = {sizeof(P)...};
  return g_step_sink ? g_step_sink->kernel(shape, st, ptr, size, (int)sizeof...(P)) : launch_now(shape, st, ptr);
}
template <typename... P, typename... A>
inline cudaError_t launch_cluster_dependent(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, int cluster, cudaStream_t st, A&&... args) {
  const LaunchShape shape{reinterpret_cast<const void*>(kernel), grid, block, smem, cluster};
  return launch_params<P...>(shape, st, std::forward<A>(args)...);
}
template <typename... P, typename... A>
inline cudaError_t launch_dependent(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  return launch_cluster_dependent(kernel, grid, block, smem, 1, st, std::forward<A>(args)...);
}
#endif

// SS_OK when the current device is compute capability 10.x, cached per device.
ss_status check_arch();
int num_sms();

// Sets n words to zero by a kernel of one block: it starts as the kernel before it ends, and the next one as it ends (a
// memset would break that chain).
ss_status clear_words(int* p, int n, cudaStream_t st);

}  // namespace ss
