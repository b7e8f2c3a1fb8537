// Shared host/device helpers of libdabnn_b200 (CUDA path only).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdlib.h>

#include "dabnn.h"

namespace dabnn {

inline cudaStream_t as_stream(void* s) { return reinterpret_cast<cudaStream_t>(s); }

inline dabnn_status launch_status() {
  return cudaGetLastError() == cudaSuccess ? DABNN_OK : DABNN_ERR_CUDA;
}

inline bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

inline int ceil_div(long long a, long long b) { return static_cast<int>((a + b - 1) / b); }

// Estimated time, in microseconds, of a layer on the integer pipes (epi: 0 int32, 1 sign words, 2 residual stream; vec: the fp32 or
// int32 rows start on 16 bytes; sms: sm_count(), which asks the runtime and is asked once per call).
double int_pipes_us(dabnn_shape in, int O, dabnn_conv cv, int epi, bool out_nchw, bool vec, int sms);

// The three output forms on the tensor-core engine from the caller's packed weights (16-byte aligned).  Arguments as of the
// entry points of the same form, already checked; DABNN_ERR_UNSUPPORTED where the engine does not cover the layer or is estimated
// to take longer than limit_us.
dabnn_status tc_bits_bconv2d(const uint64_t* a_packed, dabnn_shape in, const uint64_t* w_packed, int O, dabnn_conv cv, int32_t* out,
                             bool out_nchw, double limit_us, int sms, cudaStream_t st);
dabnn_status tc_bits_bn_sign_pack(const uint64_t* a_packed, dabnn_shape in, const uint64_t* w_packed, int O, dabnn_conv cv,
                                  const float* scale, const float* shift, uint64_t* out_packed, double limit_us, int sms, cudaStream_t st);
dabnn_status tc_bits_bn_add_sign_pack(const uint64_t* a_packed, dabnn_shape in, const uint64_t* w_packed, int O, dabnn_conv cv,
                                      const float* scale, const float* shift, const float* residual, float* y_out,
                                      uint64_t* out_packed, double limit_us, int sms, cudaStream_t st);

// dabnn_bconv2d_bn_add_sign_pack on the integer pipes whatever the size: a forward's block whose caller gave no prepared weights.
dabnn_status int_pipes_bn_add_sign_pack(const uint64_t* a_packed, dabnn_shape in, const uint64_t* w_packed, int O, dabnn_conv cv,
                                        const float* scale, const float* shift, const float* residual, float* y_out,
                                        uint64_t* out_packed, cudaStream_t st);

// The Bi-Real block on the tensor-core engine as the forward launches it.  chained: with programmatic stream serialization
// (the kernel sets itself up under its predecessor's tail; its weights and BN vectors must be constants of the stream).
// limit_us as above.
dabnn_status tc_bireal_block(const uint64_t* a_packed, dabnn_shape in, const void* w_tc, int O, dabnn_conv cv,
                             const float* scale, const float* shift, const float* residual, float* y_out,
                             uint64_t* out_packed, bool chained, double limit_us, int sms, cudaStream_t st);

// Chained launches for forwards of a few images, where every kernel is shorter than the time it takes to start one.  A
// kernel started by launch_chain() while g_chain_launch is set may begin before its predecessor in the stream has
// finished: it may do what does not depend on the predecessor (index set-up, fetching weights) and must call
// chain_wait() -- which returns once the predecessor has completed and its writes are visible -- before it touches
// anything else.  chain_trigger(), called by every CTA once its main work is done, lets the successor start.  In a
// kernel launched the ordinary way both are no-ops.
extern thread_local bool g_chain_launch;  // per host thread: set by a forward call for the launches it makes itself

// The calls of the C ABI are chained too (launch_next), but know nothing of what ran before: the caller may have packed the weights
// a moment ago.  Their kernels touch no global memory before the wait -- they only get themselves onto the SMs, set up tensor
// memory, barriers and indices while the previous kernel drains.  A kernel lets its successor in early (chain_trigger) only behind
// its main work, and where every SM has room for it then: the CTAs of a successor that come in as SMs empty one by one settle on the first of them (1x1,
// 512 -> 2048, batch 256: a pack of 392 CTAs, let in by the convolution before it at its start or end, made the pair take 124 or 76 us,
// 58.5 when it came in at the end of that convolution; 63 with ordinary launches).
// A kernel that does not take part sees ordinary stream order on both sides.  DABNN_NO_CHAIN in the environment (read once) keeps
// ordinary launches, for measurements.
inline bool chain_enabled() {
  static const bool on = getenv("DABNN_NO_CHAIN") == nullptr;
  return on;
}
#ifdef __CUDACC__
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// The same for a pointer to what the previous kernel wrote: loads through the result cannot be moved above the wait, not even those
// that count as invariant (__ldg, and any through a const __restrict__ pointer, whose cache hint keeps them in place only where the
// intrinsic is a volatile asm).
template <typename T>
__device__ __forceinline__ const T* chain_wait_for(const T* p) {
  size_t g = __cvta_generic_to_global(p);  // (so that the result is known to point to global memory: int32 pack of 119 x 56 x 56 x 70, NHWC,
                                           // 27.9 us, 30.4 with generic loads)
  asm volatile("griddepcontrol.wait;" : "+l"(g)::"memory");
  return static_cast<const T*>(__cvta_global_to_generic(g));
}
// ... and for further pointers, behind a wait.
template <typename T>
__device__ __forceinline__ const T* after_wait(const T* p) {
  asm volatile("" : "+l"(p)::"memory");
  return p;
}
__device__ __forceinline__ void chain_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Read-only-path 16-byte load for data that the PREVIOUS kernel of a chain wrote.  Volatile asm, so that it stays behind
// chain_wait(): __ldg and loads through const __restrict__ pointers count as invariant, and the compiler may move those
// above the wait, before which the data may not have been written.
__device__ __forceinline__ float4 ld_nc_f4(const float* p) {
  float4 v;
  asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}

// Two fp32 fused multiply-adds in one instruction (fma.rn.f32x2): each lane of the pair is the same correctly rounded
// fmaf as the scalar instruction, so results do not change; it halves the issue slots of an FMA-bound loop.
__device__ __forceinline__ unsigned long long pack_f32x2(float lo, float hi) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack_f32x2(unsigned long long v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ void fma_f32x2(unsigned long long& acc, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}

template <typename... KArgs, typename... Args>
inline void launch_next(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
  if (!chain_enabled()) {
    kern<<<grid, block, smem, st>>>(args...);
    return;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}
template <typename... KArgs, typename... Args>
inline void launch_chain(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
  if (g_chain_launch) launch_next(kern, grid, block, smem, st, args...);
  else kern<<<grid, block, smem, st>>>(args...);
}
#endif

// The STEM module front end of Bi-Real Net 18 (stem_module.cu): fp32 [N][56][56][64] and its packed signs from the images.
dabnn_status launch_stem_module(const dabnn_stem_module_params* sm, const float* images, int N, float* a1, float* cat,
                                float* out, uint64_t* bits, cudaStream_t st);

// Per-device host caches (function attributes set, SM counts, symbol addresses) are arrays over the device ordinal.
constexpr int kMaxDevices = 64;
// Ordinal of the calling thread's current device, or -1 (no device, or an ordinal beyond kMaxDevices).
inline int current_device() {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return -1;
  }
  return (dev >= 0 && dev < kMaxDevices) ? dev : -1;
}

// Number of SMs of the current device (cached per device).
int sm_count();

}  // namespace dabnn
