// launch_util.cuh -- kernel launches with programmatic dependent launch.
//
// A time loop is a chain of kernels, each reading what the previous one
// wrote.  Launched with programmatic stream serialisation, kernel j+1 is set
// up while kernel j runs; its blocks wait in `griddepcontrol.wait` (chain_entry:
// a hardware wait for the previous grid to complete and its memory to be
// visible) before touching anything a step writes.  Before it they read the
// first of the tables that no step writes (geometry, neighbours, tiles).
//
// The one-wave tile kernel also signals `griddepcontrol.launch_dependents`
// (chain_next) right after that wait, so that the next grid's blocks start
// beside its own and read their tables while it computes: 65,536 cells on
// tiles of 128 take 2.5 us per step, against 3.2 without.  (Signalled before the
// wait, several grids queue up on the SMs and spread the running one unevenly:
// 3.2 us.)  Elsewhere the signal costs more than it hides: the persistent
// shape 1 ran 5-10 % slower on 160,000 to 1M cells (4.07 -> 4.65, 9.2 -> 9.8 us),
// the others within 3 % either way.  The implicit signal at grid completion
// still hides most of the launch gap.  Without a programmatic predecessor the
// wait returns at once, so the kernels are correct under any launch.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace fv {
namespace {

// In every kernel launched in a programmatic chain, before it touches what a
// step writes.
__device__ __forceinline__ void chain_entry() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Lets the next kernel of the chain start (its blocks take what this grid
// leaves free and wait in chain_entry).
__device__ __forceinline__ void chain_next() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... KArgs, typename... Args>
cudaError_t launch_chained(void (*kernel)(KArgs...), unsigned grid, unsigned block, size_t smem,
                           cudaStream_t s, bool programmatic, Args&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  if (programmatic) {
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
  }
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

}  // namespace
}  // namespace fv
