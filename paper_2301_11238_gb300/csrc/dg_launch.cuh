// Programmatic dependent launch: a kernel of the explicit path may start while
// its predecessor in the stream drains.  pdl_wait holds a thread until every
// earlier kernel of the chain has completed and its writes are visible; only then
// pdl_trigger lets the successor's blocks take the room that this grid leaves
// free, so at most one grid waits (with the trigger first, three or four wait,
// and the places they hold spread a grid's blocks unevenly over the SMs: 1D FP64,
// 11,726 intervals, p = 2, 77 -> 173 us a step).  Every kernel launched with
// launch_after calls pdl_wait before it reads or writes anything that another
// kernel touches (only its parameters, operator tables among them, may come
// first), so completion is transitive along the stream.
#pragma once
#include <cuda_runtime.h>
#include <type_traits>

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

// Threads of the largest grid that starts this way.  A grid whose blocks take
// their places while its predecessor drains is spread unevenly: two on one SM,
// none on another.  An FP64 pass of about a block an SM is one long chain of
// instructions and then takes up to twice as long (19,208 triangles, two steps,
// no programmatic launch against all: p = 2 0.81 / 1.15 ms, wet/dry mode 0.37 /
// 0.54 ms), so FP64 grids start this way up to a warp an SM (200 intervals, 16
// steps: 0.81 / 0.85 ms).  FP32 passes are short, and the launch is a larger part
// of them: four warps an SM (11,726 intervals, 16 steps, 0.455 ms against 0.492;
// 19,602 triangles, four steps, 0.50 / 0.55 ms; 1 % slower at 2,097,152).
template <typename T>
constexpr bool is_fp32_data = std::is_same_v<std::remove_cv_t<std::remove_pointer_t<T>>, float>;
template <typename... KA>
constexpr size_t kPdlThreads = (is_fp32_data<KA> || ...) ? 152 * 128 : 152 * 32;

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
  cfg.numAttrs = (size_t)grid * block <= kPdlThreads<KA...> ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<KA>(args)...);
}

}  // namespace dgswe
