// Kernel launch with programmatic stream serialisation: the grid may be set up while the last blocks of the kernel before
// it in the stream still run.  Every kernel launched this way begins with stream_order_begin() or stream_order_wait(), before it
// touches any memory: the wait holds until all earlier work of the stream has completed and its writes are visible, so the
// order on the stream is the usual one, and only launch latency (1 to 2 us on B200, a quarter of the smallest calls) overlaps.
//
// A kernel launched this way is on the GPU while the one before it still writes, so what that one may write (states, pools,
// streams, index arrays) is not read-only for the kernel's lifetime, which is what the non-coherent path (ld.global.nc, __ldg,
// and plain loads through a const __restrict__ parameter, which the compiler may turn into it) is specified for.  Such data
// is read by ordinary loads behind stream_order_wait(); only the tables of a plan, written once before any launch
// can name them, take the non-coherent path.
#pragma once
#include <cuda_runtime.h>

__device__ __forceinline__ void stream_order_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void stream_order_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// Once every block of a kernel has released or ended, the next kernel's blocks are placed wherever there is room, and hold their
// registers, shared memory and threads there while they wait: on this stream that delays nothing, but work of OTHER streams
// cannot have that room meanwhile.  So only kernels that end soon after their last block has started release at once (the
// copies, the kernel in front of a refresh).  The refresh kernels, which can run for milliseconds on a few SMs, wait first
// and release a few microseconds before they end, enough to hide the launch.  With a release at once, a Store beside a
// refresh of one long request (2 of 148 SMs) ended behind it, at 1.05 of its time; now at 0.08.
__device__ __forceinline__ void stream_order_begin() {
  stream_order_release();
  stream_order_wait();
}

template <typename... P, typename... A>
cudaError_t launch_in_order(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, void *stream, const A &...args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = static_cast<cudaStream_t>(stream);
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
