// Labels and member counts of a group of 32 tokens, for the kernels that form them from the nearest-centre pass or are given them.
#pragma once
#include "common.cuh"

namespace pact {

// lab: the cluster of token i (lane = token) or -1.  The group's members per cluster are added to the table of its 128-token block and to the
// cluster sizes (integer adds: the sums do not depend on the order in which groups finish).
__device__ __forceinline__ void count_group(const ImgDesc &im, int i, int lane, int lab) {
  const unsigned same = __match_any_sync(0xffffffffu, lab);
  if (lab >= 0 && lane == __ffs(same) - 1) {
    const int len = __popc(same), b = i / kListBlock;
    // 16-bit cell (c, b) of the table, added to through the 32-bit word that holds it (a cell stays <= 128)
    uint32_t *word = reinterpret_cast<uint32_t *>(im.cnt_cb) + (((size_t)lab * im.nbp + b) >> 1);
    atomicAdd(word, (uint32_t)len << (16 * (b & 1)));
    atomicAdd(&im.csize[lab], len);
  }
}

// Labels of a group whose nearest centres are final: a survivor takes its nearest centre's cluster (a centre its own), a pruned token
// that cluster iff the distance is strictly below alpha * d_c (Eq. 8-9), else -1.
// r: the token's position among the survivors (< 0: pruned); own_cid: its cluster id if it is a centre, else -1
// (both known before the pass, so that only the nearest centre has to be fetched here).
template <typename D>
__device__ __forceinline__ void label_group(const ImgDesc &im, int i, int lane, int C, int r, int own_cid) {
  int lab = -1, joined = 0, dropped = 0, band = 0;
  if (i < im.N) {
    const unsigned long long pk = __ldcg(im.best + i);
    lab = (int)(pk & 0xFFFFFFFFull);
    const float dd = __uint_as_float((uint32_t)(pk >> 32));
    if (r >= 0) {
      if (own_cid >= 0) lab = own_cid;
    } else {
      if (D::in_band_t(dd, im)) ++band;
      if (D::below_t(dd, im)) ++joined; else { lab = -1; ++dropped; }
    }
    if (lab >= C || lab < -1) lab = -1;             // only after a failed earlier stage
    im.label[i] = lab;
    if (im.label_user) im.label_user[i] = lab;
  }
  count_group(im, i, lane, lab);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    joined += __shfl_xor_sync(0xffffffffu, joined, o);
    dropped += __shfl_xor_sync(0xffffffffu, dropped, o);
    band += __shfl_xor_sync(0xffffffffu, band, o);
  }
  if (lane == 0) {
    if (joined) atomicAdd(&im.cnt[PACT_CNT_R], joined);
    if (dropped) atomicAdd(&im.cnt[PACT_CNT_DISCARDED], dropped);
    if (band) atomicAdd(&im.cnt[PACT_CNT_BAND_ADC], band);
  }
}

}  // namespace pact
