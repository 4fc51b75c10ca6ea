// Programmatic stream serialisation: a kernel's blocks may be set up while the kernel before
// drains, which takes the launch latency between short kernels out of a chain.
#pragma once

#include <cuda_runtime.h>

#include "cpm_internal.cuh"

namespace cpm {
namespace {

// Waits until the kernel before has completed and its writes are visible; a kernel launched by
// launch_next touches nothing that another kernel of its chain writes or reads before that.
__device__ __forceinline__ void wait_previous(bool set_up_next = true) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (set_up_next) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// The kernel after this one may be set up once every block has come here (or has ended).  Not
// where that kernel is a short grid of long blocks: set up in the places that happen to be free,
// they crowd some SMs and leave others idle (FP64 structure factors of 512 points: 26 -> 87 us).
__device__ __forceinline__ void set_up_next() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// A kernel that needs nothing of the one before (late) may run beside it, once all blocks of that
// one have passed their own wait.  It ends after it all the same (the grid's first thread calls
// this at its end), so that whatever waits for this kernel has waited for both.
__device__ __forceinline__ void end_after_previous(bool late) {
  if (late && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) wait_previous(false);
}

// p, for what another kernel of the chain writes: nothing is read through the result before the
// point of the call (after the wait).  Through a const __restrict__ parameter, or a __restrict__
// one that the wait does not name, the compiler may move a load above the wait, and may take the
// non-coherent path, which is for data that nothing writes while this kernel is resident; these
// are still being written while it waits.  For the same reason such data are read by plain loads or
// __ldca, never __ldg, which is for the constant operands (E, P, the tables).
template <typename T>
__device__ __forceinline__ T* fresh(T* p) {
  size_t g = __cvta_generic_to_global(p);  // (stays a global address for the compiler)
  asm volatile("" : "+l"(g)::"memory");
  return (T*)__cvta_global_to_generic(g);
}

template <typename... P, typename... A>
void launch_next(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s,
                 A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, P(args)...);
  note_launch();
}

__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// The time into *t (if not null), by the grid's first thread.
__device__ __forceinline__ void stamp_time(unsigned long long* t) {
  if (t && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0) *t = now_ns();
}

}  // namespace
}  // namespace cpm
