// Launches of kernels that follow one another in a stream.
#pragma once

#include <cuda_runtime.h>

namespace fockx {

// A kernel's launch overlaps the end of the kernel before it in its stream: the
// launch says so (launch_after), and the kernel's first statement waits for that
// one to be complete and its writes to be visible, so nothing of it but the launch
// itself runs early.  Every thread waits, so what came before the previous kernel
// is over too.  Nine launches of an FP64 apply of 8 bands at 24^3: 154 -> 133 us;
// a Sternheimer solve of 32 bands at 48^3: 4.80 -> 4.45 ms.  (Letting the next
// kernel's blocks in as soon as the last of this one have started, by
// griddepcontrol.launch_dependents, costs more than it gives: 159 us, 5.35 ms; they take
// their places on the multiprocessors before those are evenly free.)
__device__ __forceinline__ void after_previous() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
template <class... P, class... A>
cudaError_t launch_after(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s, A&&... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = dim3(threads);
  c.dynamicSmemBytes = smem;
  c.stream = s;
  c.attrs = &at;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
  return cudaGetLastError();
}

}  // namespace fockx
