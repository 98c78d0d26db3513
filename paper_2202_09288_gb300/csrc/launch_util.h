// launch_util.h -- grid sizing of the task kernels, and programmatic dependent launch.
#pragma once

#include <cuda_runtime.h>

namespace chol {

// Grid of a task launch: one CTA per task.  The kernels it is used for also take further tasks
// from the launch's work queue when their grid is smaller than the task list, so any grid size is
// correct; measured on GB300, one CTA per task (the hardware block scheduler refills SMs as
// CTAs finish) balances the uneven task costs of a level better than a single resident wave
// of CTAs taking tasks from the queue.
template <typename K>
inline int task_grid(K kernel, int threads, size_t smem, int ntasks) {
  (void)kernel;
  (void)threads;
  (void)smem;
  return ntasks;
}

// Launches k so that its CTAs may start while the kernel before it in the stream still runs
// (programmatic dependent launch), as soon as every CTA of that kernel has started and called
// pdl_launch_dependents (or, without that call, has ended).  k may read what no kernel since the last
// ordinary launch writes; for everything else it calls pdl_wait first, which returns when the
// kernel before has ended and its writes are visible -- and with it every earlier one, since a
// kernel that calls pdl_wait in all its CTAs cannot end before the one before it.
// What an earlier kernel of such a chain writes is not read-only while k runs: k's parameters for it are
// not __restrict__ (the compiler could take its loads through the read-only path, or before the wait).
// Only kernels of a few CTAs, whose successor has something to fetch meanwhile, call
// pdl_launch_dependents (the solves, POTRF and the blocked TRSM): from a kernel that fills the GPU the
// next one's CTAs go to whichever SMs are free first, several to one FP64 unit (with the call
// in every factorization kernel the 48^3 27-point step took 111.7 ms instead of 102.5; with ordinary
// launches throughout, 104.7).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*k)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, KArgs(args)...);
}

#ifdef __CUDACC__
__device__ __forceinline__ void pdl_launch_dependents() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
#endif

}  // namespace chol
