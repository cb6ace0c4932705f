// A launch that the runtime refuses (more threads than a block can have)
// through launch_pdl (mf_launch.cuh): the error is returned, and not left behind as CUDA's last
// error for the next check to report as its own.  Prints "ok" and exits 0.
#include <cstdio>

#include "mf_launch.cuh"

__global__ void nothing(int) { mf::pdl_enter(); }

int main() {
  const cudaError_t e = mf::launch_pdl(nothing, 1, 2048, 0, nullptr, 0);
  const cudaError_t left = cudaPeekAtLastError();
  if (e == cudaSuccess || left != cudaSuccess) {
    std::printf("FAIL returned %s, left %s\n", cudaGetErrorName(e), cudaGetErrorName(left));
    return 1;
  }
  std::printf("ok\n");
  return 0;
}
