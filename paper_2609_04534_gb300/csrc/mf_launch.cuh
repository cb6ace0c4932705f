// mf_launch.cuh -- launches whose start overlaps the end of the kernel before them
// (programmatic dependent launch).
//
// The kernels of an apply or a CG iteration follow one another on one stream, and on a small mesh
// each runs for a few microseconds, about as long as its launch, its CTAs' placement and the
// drain of its predecessor.  Each of them therefore starts with pdl_enter(): it lets the next
// kernel's CTAs be placed as soon as all of its own have started, and then waits until the kernel
// before it has finished and its writes are visible.  Every kernel of the chain waits before it
// touches memory, so each one's completion implies that of all before it.  A launch without the
// attribute, or a predecessor that never lets go early, behaves as before.
//
// Such a kernel's lifetime begins before the wait, while its predecessors still write.  So in these
// kernels no pointer to data that a kernel of the chain writes (vectors, partial sums, CG state)
// is __restrict__: the qualifier tells the compiler that nothing else changes the data during
// the kernel, and lets it move a load above the wait or serve it from the read-only cache.  Without
// it, the wait's memory clobber orders every load behind it.  Only what is written before the chain
// begins keeps the qualifier: the curved geometry, the Jacobi diagonal, a batch's descriptors.
// Measured on one GB300, back-to-back mf_apply calls: Q2 8^3 FP64 14.3 -> 9.5 us, Q6 21x17x25 FP32
// 30.7 -> 26.3, Q2 123^3 538 -> 531.  A launch under stream capture is left plain: graphs with
// such edges ran CG iterations no faster (Q2 8^3 17.3 and 17.4 us) and their instantiation cost a
// serving burst a fifth of its time (22.5 -> 27.5 ms).
#pragma once
#include <utility>

#include <cuda_runtime.h>

namespace mf {

// First statement of every kernel launched by launch_pdl that touches memory.
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <typename... Params, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(Params...), unsigned blocks, int threads, size_t smem, cudaStream_t s,
                              Args&&... args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  cfg.attrs = &attr;
  const cudaError_t asked = cudaStreamIsCapturing(s, &cap);
  cfg.numAttrs = asked == cudaSuccess && cap == cudaStreamCaptureStatusNone ? 1 : 0;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, Params(std::forward<Args>(args))...);
  if (e != cudaSuccess || asked != cudaSuccess) (void)cudaGetLastError(); // reported here, not by the next check as well
  return e;
}

} // namespace mf
