// Kernel launches with programmatic stream serialisation.
//
// A solve is a chain of dependent kernels of a few microseconds.  Launched plainly, each starts
// only when its predecessor has drained and its writes are flushed (4.1 us from one small kernel to
// the next in a stream).  Here the next kernel's launch, its tables and index arithmetic overlap the
// end of its predecessor; pdl_wait then waits for the predecessor's completion.  192 x 192 mixed_dd
// solve 2.85 -> 2.37 ms, 512 x 1024 double step 16.8 -> 15.8 ms, 256^3 mixed_dd solve 13.59 -> 13.27 ms.
// The predecessor's blocks release it by exiting: an explicit launch_dependents right after
// pdl_wait starts it sooner (96 x 96 float transform 10.1 -> 7.0 us) but places its blocks on the SMs
// that have room then, unevenly (256^3 solve 15.2 ms, 512 x 1024 step 20.3 ms).
//
// Every kernel launched by pdl_launch executes pdl_wait in every thread before it touches memory
// that a kernel may write, and before it returns: a kernel's completion then implies that of all
// its predecessors in the stream.
#pragma once

#include <cuda_runtime.h>

namespace vd {

__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <typename... K, typename... A>
inline void pdl_launch(void (*kernel)(K...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<K>(args)...);
}

}  // namespace vd
