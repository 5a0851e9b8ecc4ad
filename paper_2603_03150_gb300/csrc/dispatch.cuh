// Launch helpers shared by the translation units that launch tile kernels.
#pragma once
#include "common.cuh"
#include <cuda_runtime.h>

// SpMV variant of a schedule -> template instantiation: segmented with
// E = 8, 16, 32 nonzeros per thread, or vector with 4 / 8 lanes per row
// (E_ = -4, -8); PDHG_DISPATCH_S also the slices of single LPs in float64.
#define PDHG_DISPATCH_E(e, ...)                 \
  switch (e) {                                  \
    case -4: {                                  \
      constexpr int E_ = -4;                    \
      __VA_ARGS__;                              \
    } break;                                    \
    case -8: {                                  \
      constexpr int E_ = -8;                    \
      __VA_ARGS__;                              \
    } break;                                    \
    case 32: {                                  \
      constexpr int E_ = 32;                    \
      __VA_ARGS__;                              \
    } break;                                    \
    case 16: {                                  \
      constexpr int E_ = 16;                    \
      __VA_ARGS__;                              \
    } break;                                    \
    default: {                                  \
      constexpr int E_ = 8;                     \
      __VA_ARGS__;                              \
    } break;                                    \
  }

#define PDHG_DISPATCH_S(T, e, ...)              \
  if (sizeof(T) == 8 && (e) == kSliced) {       \
    constexpr int E_ = sliced_or_8<T>();        \
    __VA_ARGS__;                                \
  } else {                                      \
    PDHG_DISPATCH_E(e, __VA_ARGS__)             \
  }
// the float64 report, Algorithm 1 and power iteration: E = 8 tiles or slices
#define PDHG_DISPATCH_FIXED(e, ...)             \
  if ((e) == kSliced) {                         \
    constexpr int E_ = kSliced;                 \
    __VA_ARGS__;                                \
  } else {                                      \
    constexpr int E_ = kFixedE;                 \
    __VA_ARGS__;                                \
  }

namespace pdhg {

// (float32 half-steps have no slices: no kernels of that kind are built)
template <typename T>
constexpr int sliced_or_8() {
  return sizeof(T) == 8 ? kSliced : 8;
}

// Launch with programmatic stream serialization (the kernel must start with
// pdl_enter(): it may begin while the previous kernel on the stream drains).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), int grid, int block, size_t smem,
                              cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// raises a kernel's dynamic shared-memory limit to what the device allows
// next to its static shared memory
inline cudaError_t set_max_dyn_smem(const void* f, size_t max_smem) {
  cudaFuncAttributes a;
  cudaError_t r = cudaFuncGetAttributes(&a, f);
  if (r == cudaSuccess)
    r = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(max_smem - a.sharedSizeBytes));
  return r;
}

}  // namespace pdhg
