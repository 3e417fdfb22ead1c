// Steps launched one behind the other without the gap between two kernels.
//
// A step reads what the step before it wrote, so its blocks wait for all of the
// predecessor; but the launch itself (block scheduling, parameters, the first
// instructions) need not.  Such a kernel begins with follow_predecessor() and is
// launched by launch_step_kernel(): the blocks come up while the predecessor's last
// ones finish and wait there until it is complete and its writes are visible.
//
// Measured, before -> after (us a step): a step of the adjoint at 256^2 FP32 6.3 -> 5.1;
// D2Q9 FP32 1003 x 517 11.5 -> 11.2; rows layout FP32, 20 launches, 1024^2 18.7 -> 17.1,
// 2048^2 54.5 -> 52.5, 4096^2 192.6 -> 190.5 (by graph 16.6 -> 16.4, 51.6 -> 51.5, 189.5 ->
// 189.7; these three before follow_predecessor_only); D3Q19 FP32 64^3 14.4 -> 14.2, 256^3 469 -> 458; 48 lattices of a batch
// 76.6 -> 75.6.  It costs nothing anywhere that was tried, so every step kernel is
// launched so, except into a caller's own capture.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace lbm {

// All threads, before the first access to global memory.  Every block of a kernel that
// is launched with launch_step_kernel waits here, whatever it does later, so that
// "complete" includes all earlier steps.  The successor's blocks may come up as soon as
// every block of this kernel has passed here.  (Nothing to wait for in an ordinary launch.)
__device__ __forceinline__ void follow_predecessor() {
  asm volatile("griddepcontrol.wait;\n griddepcontrol.launch_dependents;" ::: "memory");
}

// The same without the early start of the successor, whose blocks then come up as this
// kernel's exit: for persistent kernels, where they would hold the SMs' free slots while
// tiles are left (20 steps, against an ordinary launch and an early start: FP32 4096^2 3738,
// 3704 -> 3689 us; FP16 4096 x 2048 2009, 1972 -> 1962).
__device__ __forceinline__ void follow_predecessor_only() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// overlap = false: an ordinary launch (a caller's stream capture records plain edges).
template <typename... P, typename... A>
cudaError_t launch_step_kernel(bool overlap, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                               cudaStream_t stream, A&&... args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = &attr;
  cfg.numAttrs = overlap ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

inline bool stream_captured(cudaStream_t s) {
  cudaStreamCaptureStatus c = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &c) == cudaSuccess) return c != cudaStreamCaptureStatusNone;
  cudaGetLastError();
  return true;  // unknown
}

}  // namespace lbm
