// lc_step.cuh — launches of one step that run into one another.
#pragma once

#include "lc_internal.cuh"

namespace lc {

// The kernels of a step (one per bin group) are independent of one another:
// what any of them reads was complete before the first, and what they share
// they only add to by atomics.  So each may start while the one before it
// runs out: it lets its successor in as soon as its own blocks have all
// started (step_begin), and its last block ends only once its predecessor
// has ended (step_end), so that the end of the last kernel is the end of the
// step.  The first kernel of a step, and whatever follows it, are launched
// plainly and wait for all before them.
//
// What it is for: a step has up to ten kernels, of 2 us upwards, and each
// gap (2 us) and each tail (the last blocks of long rows) left SMs idle.
// Measured (ms, plain launches / this): local move of a 1 M-vertex SBM 2.39 /
// 2.08, pLeiden of R-MAT scale 18 30.7 / 26.4, R-MAT scale 20 level 6.76 /
// 6.06, 512-graph batch 64.7 / 59.5, R-MAT scale 22 70.0 / 65.1.
__device__ __forceinline__ void step_begin() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void step_end() {
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

class Step {
 public:
  explicit Step(cudaStream_t s) : s_(s) {}
  int launches = 0;
  // plain: a kernel that reads what its predecessors of the step wrote, or
  // that has no step_begin and step_end
  template <typename... P, typename... A>
  void run(bool plain, void (*k)(P...), unsigned grid, unsigned threads, size_t smem, A... args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s_;
    cfg.attrs = &at;
    cfg.numAttrs = plain || launches == 0 ? 0 : 1;
    cudaLaunchKernelEx(&cfg, k, args...);  // an error shows in launch_check()
    launches++;
  }

 private:
  cudaStream_t s_;
};

}  // namespace lc
