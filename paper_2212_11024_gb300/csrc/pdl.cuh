// pdl.cuh -- programmatic dependent launch: a kernel of a chain on one stream is
// brought to the SMs while the last blocks of the one before still run, and
// waits there for its completion, so that the launch's latency passes beside it.
//
// 20 steps launched one by one on a stream, us per step without and with it:
// one-site kernel FP32 64^3 14.4 -> 12.3, 128^3 128.5 -> 126.0, FP16 129 x 127 x
// 131 101.4 -> 99.2; row kernel FP16 64^3 11.4 -> 9.7, 128^3 69.6 -> 67.2, 256^3
// 514.0 -> 510.9, 512 x 256 x 256 1059.6 -> 1057.3; window kernel BF16 250 x 124
// x 132 147.9 -> 146.4.  A graph launches its kernel nodes as fast by its plain
// edges (all of the row and window kernel's cases the same either way; FP32 32^3
// 3.4 us, with programmatic edges 4.9), so a launch that is being captured is a
// plain one.
#pragma once

#include <cuda_runtime.h>

#include <utility>

#include "flame_internal.h"

namespace flame {

// The step kernels of a variant are chained this way.  Not those of the
// finite-difference current: they read the B field that the kernel before them
// writes through read-only loads, which take no notice of the wait.
template <int VAR>
constexpr bool kChained = VAR != kVarFdCurrent;

// The next kernel of the chain may come as soon as every block of this one has
// called this or ended; it then takes the places that ending blocks leave.
__device__ __forceinline__ void next_kernel_may_come() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// At the start of a chained kernel, before it reads or writes global memory:
// waits until every kernel before this one has completed and its writes are
// visible.  After a plain launch both do nothing.
__device__ __forceinline__ void after_previous_kernel() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// kern<<<grid, block, smem, s>>>(args...) as such a kernel.
template <class... P, class... A>
cudaError_t launch_chained(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  const bool asked = cudaStreamIsCapturing(s, &cap) == cudaSuccess;
  if (!asked) (void)cudaGetLastError();  // the launch below reports what is wrong
  const bool plain = !asked || cap != cudaStreamCaptureStatusNone;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = plain ? 0 : 1;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);
}

}  // namespace flame
