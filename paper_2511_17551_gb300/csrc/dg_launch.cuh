// Launches that overlap with the end of the kernel before them in the stream (programmatic
// dependent launch).  A kernel started this way may begin once every CTA of its predecessor has
// called pdl_trigger or ended; before pdl_wait, which returns when the predecessor has completed
// and its writes are visible, it reads nothing that a kernel writes and writes nothing.  Every
// kernel launched with launch_pdl calls pdl_wait in each CTA that does any work and pdl_trigger
// only behind it, so completion is transitive along the stream; behind a copy, a memset, an
// event or a kernel that does not trigger, the kernel starts when that has completed.
//
// The time steps are chains of kernels of 10 to 200 us, each of which used to wait for the last
// CTA of the one before, its memory flush and its own launch.  10 steps of the 12 x 10 x 9 N = 4
// Navier-Stokes mesh: 1394 -> 1122 us; 32^3 N = 3: 8.89 -> 8.51 ms; five of the 131 k element cylinder:
// 3.24 -> 3.09 ms (each with the state set and read back); meshes of a few elements: 15 to 30 % less.  The trigger of the two long
// kernels (right-hand side, gradients) stands before their last phase: at their start it cost 3 to
// 14 % against there, since the next kernel's CTAs then take the places that their own CTAs leave
// and lie unevenly on the SMs.  In FP64, where the FP64 pipe of an SM bounds its CTAs, that weighs
// more than the overlap (8^3: 2.61 -> 3.13 ms), so FP64 kernels do not trigger at all: only
// the launch itself is hidden (2.61 -> 2.49 ms).  Nor do the training kernels, one wave of CTAs each: an
// iteration of gathers, gradient and Adam 36 -> 25 us.
#pragma once
#include <cuda_runtime.h>

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// apart: an ordinary launch, behind the whole kernel before it (a context whose kernels are being timed)
template <typename... P, typename... A>
inline cudaError_t launch_pdl(bool apart, void (*k)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, A... a) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = apart ? 0 : 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k, static_cast<P>(a)...);
  if (e != cudaSuccess) cudaGetLastError();  // reported here: not to the next call that asks
  return e;
}
