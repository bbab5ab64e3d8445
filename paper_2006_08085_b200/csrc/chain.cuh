// Steps follow one another on a stream: a launch may begin while the one before it is still finishing (programmatic dependent
// launch), does what needs none of its results - barriers, tables of the workspace, tensor memory - and waits for its end and its
// writes before it touches the state arrays.  What this hides is the way from one launch to the next and the set-up, 1 .. 6 us.
#ifndef DETAG_CHAIN_CUH
#define DETAG_CHAIN_CUH

#include <cuda_runtime.h>

namespace detag {

// The launches before this one are complete.  Every thread that reads or writes state passes it.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// The next launch may begin (once every block has said so).  After chain_wait(): what it finds running is this launch alone.
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Launch with that attribute; a cudaError_t value.  The caller reports a failure, so it is not left behind as the runtime's last
// error for whoever asks next.
template <typename... P>
int launch_chained(void (*kernel)(P...), unsigned grid, unsigned threads, size_t smem, cudaStream_t stream, const P&... args) {
  cudaLaunchConfig_t config = {};
  config.gridDim = dim3(grid);
  config.blockDim = dim3(threads);
  config.dynamicSmemBytes = smem;
  config.stream = stream;
  cudaLaunchAttribute chained = {};
  chained.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  chained.val.programmaticStreamSerializationAllowed = 1;
  config.attrs = &chained;
  config.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&config, kernel, args...);
  if (e != cudaSuccess) cudaGetLastError();
  return static_cast<int>(e);
}

}  // namespace detag
#endif  // DETAG_CHAIN_CUH
