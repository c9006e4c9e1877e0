// Shared host/device helpers of the Lynx CUDA library (sm_100a).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>

#include "lynx.h"
#include "workspace_layout.cuh"

#define LYNX_D 128

namespace lynx {

__host__ inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Status of the launch just made.  With LYNX_DEBUG set in the environment the CUDA error text
// goes to stderr.
__host__ inline lynx_status launch_status() {
  const cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) return LYNX_OK;
  if (getenv("LYNX_DEBUG")) fprintf(stderr, "lynx: CUDA error at launch: %s\n", cudaGetErrorString(e));
  return LYNX_ERR_CUDA;
}

// Programmatic dependent launch: a kernel launched this way may become resident while the last CTAs of the kernel before it
// in the stream are still running, and must call pdl_wait() before it touches global memory.  pdl_trigger() lets the kernel
// after it do the same; pdl_wait() waits until everything before it in the stream has completed and is visible; pdl_begin()
// is both, for kernels whose CTAs are short.  It takes the launch gap and the ramp of a grid off chains of kernels (planes to
// pages and attention on them, four kernels: 41.0 -> 35.1 us for 4096 tokens, 75.3 -> 73.7 us for 32768, 247.3 -> 243.3 us
// for 131072, equal at 524288; two small quantisations 10.9 -> 9.9 us).  Where a grid's CTAs run long, the trigger belongs
// behind their work: see hier_quantize.cu.
template <class... P, class... A>
__host__ inline lynx_status launch_cluster(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, unsigned cluster, void* stream,
                                           A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = static_cast<cudaStream_t>(stream);
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  if (cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...) != cudaSuccess) {
    launch_status();
    return LYNX_ERR_CUDA;
  }
  return launch_status();
}
template <class... P, class... A>
__host__ inline lynx_status launch_pdl(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, void* stream, A... args) {
  return launch_cluster(kernel, grid, block, smem, 1u, stream, args...);
}
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_begin() {
  pdl_trigger();
  pdl_wait();
}
// What a kernel launched this way reads of earlier kernels' results goes through ordinary (coherent) loads: such a kernel is
// alive while they still write, and the read-only path (__ldg, const __restrict__ parameters) is defined only for data that
// does not change during the kernel's whole life.  ld_dep is volatile, so it also stays behind the wait.  Any of 4, 8 or 16
// bytes, at an address aligned to as many.
template <class T>
__device__ __forceinline__ T ld_dep(const T* p) {
  static_assert(sizeof(T) == 4 || sizeof(T) == 8 || sizeof(T) == 16, "a register, a pair or four");
  union { uint32_t r[sizeof(T) / 4]; T v; } u;
  if constexpr (sizeof(T) == 4)
    asm volatile("ld.global.b32 %0, [%1];" : "=r"(u.r[0]) : "l"(p));
  else if constexpr (sizeof(T) == 8)
    asm volatile("ld.global.v2.b32 {%0,%1}, [%2];" : "=r"(u.r[0]), "=r"(u.r[1]) : "l"(p));
  else
    asm volatile("ld.global.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(u.r[0]), "=r"(u.r[1]), "=r"(u.r[2]), "=r"(u.r[3]) : "l"(p));
  return u.v;
}

// Number of SMs of the current device (cached per device id).
__host__ int sm_count();

// Status flags, word 0 of a workspace.
constexpr uint32_t kFlagBadBlock = 1u;
constexpr uint32_t kFlagTimeout = 2u;
constexpr uint32_t kFlagRange = 4u;

}  // namespace lynx
