// Programmatic dependent launch: a kernel of the explicit path may start while
// its predecessor in the stream drains.  pdl_trigger lets the successor's blocks
// take the room that the last blocks of this grid leave free; pdl_wait holds a
// thread until every earlier kernel of the chain has completed and its writes
// are visible.  Every kernel launched with launch_after calls pdl_wait before it
// reads or writes anything that another kernel touches (only its parameters,
// operator tables among them, may come first), so completion is transitive along
// the stream.
#pragma once
#include <cuda_runtime.h>

namespace dgswe {

__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename T>
__device__ __forceinline__ void hide_pointer(T& p) {
  asm volatile("" : "+l"(p)::"memory");
}
template <typename... T>
__device__ __forceinline__ void after_wait(T&... p) {
  (hide_pointer(p), ...);
}

// Grids beyond the chip's room for threads (152 SMs of 2,048) start the plain
// way: their last blocks gain nothing from company, and the successor's waiting
// blocks cost them 1 % (2,097,152 FP32 triangles, p = 2), where 73,728 gain 6 %.
constexpr size_t kPdlThreads = 152 * 2048;

template <typename... KA, typename... A>
inline void launch_after(void (*kernel)(KA...), unsigned grid, unsigned block, size_t smem, cudaStream_t s, A&&... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = (size_t)grid * block <= kPdlThreads ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<KA>(args)...);
}

}  // namespace dgswe
