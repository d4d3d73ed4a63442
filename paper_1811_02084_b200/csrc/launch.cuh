// Launches chained on their stream: a kernel launched with launch_chained may be set up while the launch before it still
// drains, calls chain_wait() before it touches memory, and from there on lets the launch behind it do the same.  (About 1.5
// us a launch on a stream of short ones.)
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

namespace mtf {

// A driver call that wants a current context, which a thread has only once a runtime call that needs the device was made on it
// (cuTensorMapEncodeTiled as a thread's first call: CUDA_ERROR_INVALID_CONTEXT).
template <typename F>
CUresult in_context(F call) {
  CUresult r = call();
  int dev = 0;
  if (r == CUDA_ERROR_INVALID_CONTEXT && cudaGetDevice(&dev) == cudaSuccess && cudaSetDevice(dev) == cudaSuccess) r = call();
  return r;
}

// One lane of the (converged) warp; the compiler then knows the branch for a single thread's and keeps addresses and descriptors in
// uniform registers: an M = 128, N = 64 MMA issues in 48 cycles, behind `lane == 0` in 64.  With it in every thread that issues loads or MMAs the attention
// block of 16 x 512 positions took 409 us instead of 449, the decoder layer 4668 instead of 4891, the feed-forward block on 128 tokens 48.2 instead of 49.3.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}

__device__ __forceinline__ void chain_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// The wait alone, for a kernel of one short block per row: a launch let in at the start takes the free block slots of whichever
// SM has them, and when that launch is another such kernel its blocks then lie unevenly.  This way it is let in as the blocks end.
__device__ __forceinline__ void chain_wait_only() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The error is left for the caller's cudaGetLastError.
template <typename... P, typename... A>
void launch_chained(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3(grid, 1, 1); cfg.blockDim = dim3(block, 1, 1); cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cfg.attrs = at; cfg.numAttrs = 1;
  (void)cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace mtf
