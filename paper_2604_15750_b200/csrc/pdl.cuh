// Programmatic dependent launch between the kernels of a step.  A kernel launched with launch_chained may
// start while the one before it in the stream still runs: its blocks take the SMs that become free, set
// up barriers, TMEM and tensor maps, and wait in pdl_wait() until everything before has completed and is
// visible.  Every kernel launched this way calls pdl_wait() in all of its blocks before it touches global
// memory that a kernel of the step writes (so that completion is transitive).  k_gemm_tc loads weights before: no kernel of a
// sequence writes them, and a sequence starts with k_step_begin, a launch without the attribute, which runs after all that
// was in the stream before it (weights written there included).  pdl_trigger() only allows the next kernel's blocks to be scheduled,
// once every block has called it or ended; a kernel without it counts as triggered when it ends.  A kernel that
// allocates TMEM triggers behind the allocation: a block of the next kernel that fitted beside one of these
// would take the columns first and hold them in pdl_wait(), whose end is behind the allocation that waits for
// them.  Two kernels of a layer were 2.1 us apart; the 224 launches of a 1024-token LLaDA-8B prefill took 15.37 ms
// and take 14.84 ms.
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

namespace dc {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// The same for a kernel that reads what earlier kernels wrote through __restrict__ pointers, which it passes here: the
// compiler may move a load through such a pointer in front of a statement that cannot change what it points to.
template <typename P0, typename... P>
__device__ __forceinline__ void pdl_wait(P0& p0, P&... p) {
  pdl_wait();
  auto behind = [](auto& q) { asm volatile("" : "+l"(q) : : "memory"); };
  behind(p0);
  (behind(p), ...);
}
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// (the arguments by reference: a step's lengths alone are 900 bytes, and the typed launch function copies them twice)
template <typename... P>
inline cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                  const std::common_type_t<P>&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr; cfg.numAttrs = 1;
  void* a[] = {const_cast<void*>(static_cast<const void*>(&args))...};
  return cudaLaunchKernelExC(&cfg, reinterpret_cast<const void*>(kernel), a);
}

}  // namespace dc
