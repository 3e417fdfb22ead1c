// Steps launched one behind the other without the gap between two kernels.
//
// A step reads what the step before it wrote, so its blocks wait for all of the
// predecessor; but the launch itself (block scheduling, parameters, the first
// instructions) need not.  Such a kernel begins with follow_predecessor() and is
// launched by launch_step_kernel(): its blocks come up as the predecessor's blocks exit
// and wait there until all of it is complete and its writes are visible.
//
// Measured, ordinary launch -> this (us a step): adjoint FP32 256^2 6.9 -> 5.0, 400^2 11.0 ->
// 8.6; D2Q9 by graph FP32 256^2 2.61 -> 2.37, 1003 x 517 7.95 -> 7.74, FP16 450^2 4.80 -> 4.45,
// FP64 256^2 30.7 -> 30.4, one launch a call FP32 512^2 6.3 -> 4.9; FP32 4096^2 187 -> 184.5; D3Q19
// FP32 24 x 72 x 32 5.55 -> 5.3, 64^3 14.35 -> 14.07, 160^3 133.8 -> 133.4.  Nowhere that was
// tried slower, so every step kernel is launched so, except into a caller's own capture.
//
// Measured and not kept: griddepcontrol.launch_dependents right after the wait, so that the
// successor comes up while its predecessor runs.  Its blocks then take places next to the
// running ones, several to an SM, and keep them, so the next step runs with its blocks
// heaped: FP64 301 x 299 45.2 -> 59.2, adjoint 400^2 8.6 -> 9.8, D3Q19 48 x 32 x 32 5.35 -> 6.24
// (slower than ordinary launches), 160^3 133.4 -> 140.4; at best 1% faster (52 x 50 x 219).
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace lbm {

// All threads, before the first access to global memory.  Every block of a kernel that
// is launched with launch_step_kernel waits here, whatever it does later, so that
// "complete" includes all earlier steps.  (Nothing to wait for in an ordinary launch.)
__device__ __forceinline__ void follow_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

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
