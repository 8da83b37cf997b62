// pdl.cuh -- launching a kernel under the end of the one before it in its stream.
//
// A chain of kernels of a few microseconds loses ~1.5 us a launch between the last block of
// one and the first instruction of the next.  A kernel launched here may have its blocks
// started once every block of its predecessor has passed pdl_enter (or ended); each block
// first sets up what depends on no other kernel (barriers, tensor memory) and then enters:
// it waits until the predecessor has ended and its writes are visible, and only then lets its own
// successor start.  So at most two kernels of a stream are on the GPU at once, no kernel can end
// before its predecessors, and nothing that a block reads after entering can have been cached
// before it was written.  Every block has to enter; a kernel launched the ordinary way may
// enter as well (nothing to wait for).
// Reads behind the wait: plain loads by pointers without __restrict__ (or ld_stream).  A const
// __restrict__ pointer promises that nobody writes its data while the kernel runs, which does
// not hold here: the compiler may take the read-only path, or move the load up over the wait.  The
// load intrinsics with a cache hint say nothing about their order either.  Constant tables may
// go by way of __ldg.
// (Flow gradients of 4096 windows, 28 launches, 510 -> 449 us; ResNet stem and two blocks, 54
// launches, 1477 -> 1398; 4096 x 1968 x 512 dense forward and backward, 6 launches, 75 -> 65;
// 20,000 posterior draws 185 -> 171.)
#pragma once

#include <utility>

#include <cuda_runtime.h>

namespace gwx {

__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// A read that is not needed again (evicted first), in its place behind the wait.
__device__ __forceinline__ float4 ld_stream(const float4* p) {
  float4 v;
  asm volatile("ld.global.cs.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p)
               : "memory");
  return v;
}

template <class... P, class... A>
cudaError_t pdl_launch(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);
}

}  // namespace gwx
