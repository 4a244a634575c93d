// Shared host/device helpers of the GRASS B200 library (not part of the ABI).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>

#include "grass.h"

namespace grass {

// Status word layout on the device: [0] first error code, [1] detail.
// Kernels record with record_status(); the first error wins.
__device__ __forceinline__ void record_status(int* status, int code, int detail) {
  if (atomicCAS(&status[0], 0, code) == 0) status[1] = detail;
}

// Device address of the current device's status word (host function, common.cu).
int* status_word(cudaError_t* err);

// grass_select (select.cu).
int select_rows(const float* norms, int64_t m, int32_t r, int method, uint64_t seed,
                uint32_t layer_id, uint32_t epoch, int32_t* idx, float* rho, void* ws, size_t ws_bytes,
                cudaStream_t s);

// Brackets one kernel launch with events while a profile is active (common.cu).
void profile_mark_begin(int kernel_id, cudaStream_t s);
void profile_mark_end(cudaStream_t s);
struct ProfileScope {
  cudaStream_t s;
  ProfileScope(int kernel_id, cudaStream_t stream) : s(stream) { profile_mark_begin(kernel_id, s); }
  ~ProfileScope() { profile_mark_end(s); }
};

#define GRASS_CUDA_TRY(expr)                                                             \
  do {                                                                                   \
    cudaError_t e__ = (expr);                                                            \
    if (e__ != cudaSuccess) {                                                            \
      fprintf(stderr, "grass: %s failed: %s (%s:%d)\n", #expr, cudaGetErrorString(e__),  \
              __FILE__, __LINE__);                                                       \
      return GRASS_ERR_CUDA;                                                             \
    }                                                                                    \
  } while (0)

#define GRASS_LAUNCH_CHECK() GRASS_CUDA_TRY(cudaGetLastError())

// Programmatic dependent launch.  A library call is a chain of short kernels.  They are launched with this
// attribute, the first one too, so that their blocks are placed and run their prologue while the kernel before drains, and
// wait in grid_dep_wait() for its results.  Each waits before it writes memory or reads what an earlier kernel of the
// call or of the stream writes, so completion is transitive along the chain and along the stream.  There is no exception for
// what a kernel further back wrote: the wait makes visible what the grids before it wrote, and nothing is said of a
// read ahead of it.  (An update that read M, V, W and idx before its wait took 10.7 us instead of 11.3 a step of
// T = 2048, 512 x 512, r = 128, 170.0 instead of 171.5 of T = 4096, 5120 x 13824, r = 1024.)  Eagerly launched steps gained 1
// to 2.7 us from the attribute on their first kernel (T = 4096, 1024 x 1024, r = 128: 16.4 -> 13.7).
// A kernel that something may follow in its call lets it in with grid_dep_launch(), late enough that what is left is short.
// It does so too where it is its call's last (selections, row norms, an unsplit projection), so the next call's first kernel
// may be resident while this one still writes, and a projection then holds its SMs.  Another stream does not miss them: 60 x
// (selection of 13824 rows, projection of T = 4096) beside 60 steps of 1B down take 5.49 ms, and 5.61 if last
// kernels let nothing in; refreshes of 60M, 350M, 1B and 7B layers on two streams take 0 to 3 % longer so.
// What an earlier kernel writes (inputs made by the program's last kernel, G_C, partials, norms, idx, rho, the gathered
// operand) is still being written when a dependent kernel becomes resident, so it is not constant for that kernel's
// lifetime: such a kernel reads it with ordinary loads (also ptx::ld_s32, ld_f32, ld_na_u16), through pointers
// without __restrict__ and without __ldg, which the compiler could move above grid_dep_wait().
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_launch() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
inline cudaLaunchAttribute dependent_launch_attr() {
  cudaLaunchAttribute a = {};
  a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a.val.programmaticStreamSerializationAllowed = 1;
  return a;
}
// For kernels that call grid_dep_wait().
template <typename... P, typename... A>
cudaError_t launch_kernel(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                          A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr = dependent_launch_attr();
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

inline bool aligned_to(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }
inline size_t round_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

__device__ __forceinline__ float to_float(float v) { return v; }
__device__ __forceinline__ float to_float(__nv_bfloat16 v) { return __bfloat162float(v); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

}  // namespace grass
