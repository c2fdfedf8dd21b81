// pact_prune_static: the percentile split (Eq. 3-4) for callers that must not allocate.
//
// pact_prune needs a caller-provided workspace, and somebody has to cudaMalloc that workspace.
// Some hosts of this library cannot: code that runs inside another framework's stream callback or
// between the iterations of a latency-critical decode loop, plugins that are handed tensors but no
// allocator, and processes whose memory pool is already carved up and closed.  The split itself needs
// none: its keys are in registers or shared memory, and beyond that it reads the scores again.
#include <math.h>
#include <string.h>

#include "kernels.cuh"

using namespace pact;

extern "C" pact_status pact_prune_static(const float *score, int N, const pact_params *p, uint8_t *keep,
                                         int32_t *kept_idx, int32_t *pruned_idx, int32_t *counts,
                                         void *stream) {
  if (!score || !keep || !kept_idx || !pruned_idx || !counts || !p || N < 1) return PACT_ERR_INVALID_ARG;
  if (N > PACT_PRUNE_STATIC_MAX_N) return PACT_ERR_UNSUPPORTED;
  if (!(p->lambda >= 0.0 && p->lambda <= 1.0)) return PACT_ERR_INVALID_ARG;
  DeviceCfg cfg;
  if (select_configure(&cfg) != cudaSuccess) return PACT_ERR_CUDA;   // (of the current device; no context has done it)
  cudaStream_t st = (cudaStream_t)stream;
  Batch bt;
  memset(&bt, 0, sizeof(bt));
  bt.B = 1;
  ImgDesc &m = bt.img[0];
  m.N = N;
  long long mt = p->n_prune >= 0 ? (long long)p->n_prune : (long long)floor(p->lambda * (double)N + 1e-6);
  if (mt > N - 1) mt = N - 1;
  if (mt < 0) mt = 0;
  m.m_target = (int)mt;
  m.score = const_cast<float *>(score);
  m.keep = keep;
  m.kept_idx = kept_idx;
  m.pruned_idx = pruned_idx;
  m.counts_user = counts;
  return launch_split(bt, N, cfg, st) == cudaSuccess ? PACT_OK : PACT_ERR_CUDA;
}
