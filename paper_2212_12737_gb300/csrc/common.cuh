// Shared helpers for the libgdml CUDA sources (sm_103a).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <cstdio>
#include <string>

#include "../../include/gdml.h"

namespace gdml {

// Streaming multiprocessors of the current device (152 on GB300: 2 dies x 76), queried once per
// device; grids are sized in multiples of it.
int num_sms();

// Lets launches of `fn` on the current device take `bytes` of dynamic shared memory; false if CUDA refuses.
// Per device, and raised only: a thread whose call needs less leaves what another one's launch relies on.
bool allow_smem_of(const void* fn, size_t bytes);
template <typename F>
bool allow_smem(F* fn, size_t bytes) {
  return allow_smem_of(reinterpret_cast<const void*>(fn), bytes);
}

// Host-side error carrier: every internal call returns a gdml_status and
// writes a message into the context.
struct Err {
  gdml_status st = GDML_OK;
  std::string msg;
};

#define GDML_CUDA_TRY(expr)                                                              \
  do {                                                                                   \
    cudaError_t _e = (expr);                                                             \
    if (_e != cudaSuccess) {                                                             \
      return ::gdml::fail(GDML_ERR_CUDA, std::string(#expr " -> ") + cudaGetErrorString(_e)); \
    }                                                                                    \
  } while (0)

// thread-local last error (used when no context exists yet)
gdml_status fail(gdml_status st, const std::string& msg);
const std::string& last_msg();
void clear_msg();

// host-side count of kernel launches issued by this library (inside CUDA
// graphs a captured launch counts once per replay; see count_graph_launches)
void count_launch(int64_t n = 1);
int64_t launch_count();

inline int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }
__device__ __forceinline__ int64_t cdiv_dev(int64_t a, int64_t b) { return (a + b - 1) / b; }

// (sh, sl) += a * (bh + bl) in double-float: a * bh formed exactly by FMA
// (TwoProduct), the a * bl term folded into the low part, summed by TwoSum.
__device__ __forceinline__ void df_add_prod(float& sh, float& sl, float a, float bh, float bl) {
  const float ph = a * bh;
  float pl = fmaf(a, bh, -ph);
  pl = fmaf(a, bl, pl);
  const float t = sh + ph;
  const float v = t - sh;
  float e = (sh - (t - v)) + (ph - v);
  e += sl + pl;
  sh = t + e;
  sl = e - (sh - t);
}

// Deterministic block reduction of one double (fixed tree order).
template <int THREADS>
__device__ __forceinline__ double block_sum(double v, double* sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  double r = 0.0;
  if (warp == 0) {
    r = lane < THREADS / 32 ? sh[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  }
  __syncthreads();
  return r;  // valid in thread 0
}

// p = i(i-1)/2 + j with i > j  ->  (i, j)
__device__ __forceinline__ void pair_of(int p, int& i, int& j) {
  // FP32 estimate (GB300's FP64 pipe is slow), then exact integer correction
  int ii = (int)((1.f + sqrtf(1.f + 8.f * (float)p)) * 0.5f);
  while (ii * (ii - 1) / 2 > p) --ii;
  while ((ii + 1) * ii / 2 <= p) ++ii;
  i = ii;
  j = p - ii * (ii - 1) / 2;
}
// Programmatic dependent launch: grid_wait returns once the kernels before this one in the stream have
// completed, grid_trigger lets the next one start (when every CTA has called it or has ended)
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// whether launches into the stream are not being captured (early starts gained nothing in captured loops)
inline bool not_capturing(cudaStream_t st) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) {
    (void)cudaGetLastError();
    return false;
  }
  return cap == cudaStreamCaptureStatusNone;
}
// launches a kernel that with `early` may start before the one ahead of it in the stream has ended (it
// calls grid_wait)
template <typename... P, typename... A>
void launch_after(bool early, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = early ? 1 : 0;
  (void)cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

__device__ __forceinline__ int pair_idx(int i, int j) {  // requires i != j
  return i > j ? i * (i - 1) / 2 + j : j * (j - 1) / 2 + i;
}


}  // namespace gdml
