// Shared device/host helpers of the ctof library (complex arithmetic, error
// plumbing).  Internal header: not part of the C ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/ctof.h"

#define CTOF_CUDA_TRY(expr)                                  \
  do {                                                       \
    cudaError_t _e = (expr);                                 \
    if (_e != cudaSuccess) {                                 \
      ctof_set_last_cuda_error(_e, #expr, __FILE__, __LINE__); \
      return CTOF_ECUDA;                                     \
    }                                                        \
  } while (0)

#define CTOF_TRY(expr)              \
  do {                              \
    ctof_status _s = (expr);        \
    if (_s != CTOF_OK) return _s;   \
  } while (0)

void ctof_set_last_cuda_error(cudaError_t e, const char* what, const char* file, int line);
void ctof_set_last_error_text(const char* msg);

__host__ __device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__host__ __device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__host__ __device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__host__ __device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }
__host__ __device__ __forceinline__ float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }

// Programmatic dependent launch: a kernel started with ctof_launch may begin
// while the kernel before it in the stream is still running.  Every such kernel
// calls pdl_trigger() at its start (its own successor may then be set up) and
// pdl_wait() before it touches anything that earlier work in the stream reads
// or writes; only its set-up (barriers, tables made at build time) goes before
// the wait.  A kernel completes only after its wait, so the order of the whole
// chain is kept.
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... P, typename... A>
cudaError_t ctof_launch(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}
#endif

// Soft threshold (proximal map of thr |.|).
#ifdef __CUDACC__
__device__ __forceinline__ float soft(float a, float thr) {
  const float m = fabsf(a) - thr;
  return m > 0.f ? copysignf(m, a) : 0.f;
}
#endif

static inline int ctof_round_up(int x, int m) { return (x + m - 1) / m * m; }
static inline int ctof_div_up(long long x, long long m) { return (int)((x + m - 1) / m); }
