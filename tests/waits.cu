// Kernels for tests of the bounded waits of csrc/tma.cuh: a wait runs out on a barrier at which nobody arrives, after a second.
#include <cuda_runtime.h>

#include "tma.cuh"

using namespace pact;

// Every warp waits for a barrier of its own choice: the late one for a barrier that is never complete.
__global__ void k_late_warp(int late, int32_t *status, int32_t *ok) {
  __shared__ uint64_t bar[2];
  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_arrive(&bar[0]);
  }
  __syncthreads();
  const int w = threadIdx.x >> 5;
  const bool landed = mbar_wait_warp_or_report(&bar[w == late], 0, status);
  if ((threadIdx.x & 31) == 0) ok[w] = landed;
}

extern "C" int late_warp(int late, int warps, int32_t *status, int32_t *ok, void *stream) {
  k_late_warp<<<1, 32 * warps, 0, (cudaStream_t)stream>>>(late, status, ok);
  return (int)cudaGetLastError();
}
