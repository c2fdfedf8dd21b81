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

// Every warp waits `waits` times for a barrier that is never complete, and remembers in s_abort that it gave up.
__global__ void k_many_waits(int waits, int32_t *failed) {
  __shared__ uint64_t bar;
  __shared__ int s_abort;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    s_abort = 0;
  }
  __syncthreads();
  int n = 0;
  for (int i = 0; i < waits; ++i)
    if (!mbar_wait_warp_unless(&s_abort, &bar, 0)) {
      s_abort = 1;
      ++n;
    }
  if ((threadIdx.x & 31) == 0) failed[threadIdx.x >> 5] = n;
}

extern "C" int many_waits(int waits, int warps, int32_t *failed, void *stream) {
  k_many_waits<<<1, 32 * warps, 0, (cudaStream_t)stream>>>(waits, failed);
  return (int)cudaGetLastError();
}
extern "C" int late_warp(int late, int warps, int32_t *status, int32_t *ok, void *stream) {
  k_late_warp<<<1, 32 * warps, 0, (cudaStream_t)stream>>>(late, status, ok);
  return (int)cudaGetLastError();
}
