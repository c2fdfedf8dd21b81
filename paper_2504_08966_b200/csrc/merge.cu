// Merge (Eq. 10, Algorithm 3 step 4): one hidden state per cluster = mean of its members in
// float accumulation and ascending token order; position id of the centre; cluster sizes;
// text rows copied around the merged span.
//
//   k_label_counts   labels (reincorporation test of Eq. 8) and members per cluster, in all and by block of 128 tokens; the rows x
//                    centres pass on single CTAs (gram_umma.cu) does this itself
//   k_members        a stable counting sort of the tokens by cluster id: every token writes one 16-byte record {token, cluster, first
//                    member position, cluster size} at its place in the cluster-sorted member array.  Also P', sizes and log sizes.
//   k_lists          both in one kernel with an image-wide barrier, for few tokens
//   k_merge  the member array (followed by the text rows) is cut into contiguous ranges;
//            a CTA streams its columns of the rows of a range with many loads in flight and no look-ups, keeps
//            the running cluster in registers and writes a row out whenever the cluster id changes.
//            Large clusters cut by a range boundary leave partial sums; the last CTA to arrive adds them in
//            range order, so the result does not depend on timing.
#include "kernels.cuh"
#include "labels.cuh"
#include "merge_ranges.h"
#include "tma.cuh"

namespace pact {

__device__ __forceinline__ int ld_cg_i32(const int *p) {
  int v;
  asm volatile("ld.global.cg.s32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ int ld_acquire_i32(const int *p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ float4 ld_cg_f4(const float *p) {
  float4 v;
  asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}

// ---- member lists --------------------------------------------------------------------------------
// grid (ceil(maxN / 128), B), 128 threads.
// Part 1: block b sorts its 128 tokens by (cluster id, token), discarded tokens last; the first token of
//   every run writes the run length to cnt_cb[c][b] (a table that is zero before the kernel) and adds it
//   to csize[c].
// Part 2 (after every block of the image has finished part 1): the member in sorted position t of block b
//   belongs at  member_off[c] + (members of c in the blocks before b) + (its place in the run),  where
//   member_off is the exclusive prefix sum of csize.  It writes its record there; the first member of a
//   cluster also writes P', the size and its logarithm for the cluster's output row.
// The parts are separated by a barrier over the blocks of the image (all blocks must be resident: cooperative launch).
// For the whole step of up to kListsMaxN tokens on the double-precision tiles, which has ten kernels with it and eleven without; that number is
// what it is kept for.  k_label_counts and k_members do the same for all others, and would be faster here too: one fp32 image of 680 tokens (d_k 128) 49.7 us
// with k_lists and 45.7 with these two, of 1024 56.6 and 52.4, four of 800 72.4 and 68.4, bf16 with d_k 160, 1000 tokens, 65.1 and 62.0.  (Here a token
// looks up its cluster in the sorted block, and the counts of the blocks before its own come in one trip to the L2 after the other.)
// The labels are first formed here from the nearest-centre pass (survivors: cluster id of the nearest centre, a centre its own
// id; pruned tokens: that id iff the distance is strictly below alpha * d_c, else -1) and written out.
constexpr int kScanTile = kListBlock * 8;   // cluster sizes scanned per step of part 2
constexpr int kNoLabel = 0x7fffffff;
constexpr int kListsMaxN = 1024;

template <typename T>
__global__ void __launch_bounds__(kListBlock) k_lists(const __grid_constant__ Batch bt, int spin_limit) {
  using D = typename DistOf<T>::type;
  const ImgDesc &im = bt.img[blockIdx.y];
  TL_SCOPE(im, 8);
  pdl_wait();
  pdl_trigger();
  const int N = im.N;
  const int nblk = (N + kListBlock - 1) / kListBlock;
  const int b = blockIdx.x, t = threadIdx.x, lane = t & 31, w = t >> 5;
  if (b >= nblk) return;
  __shared__ int slab[kListBlock], s_lab[kListBlock], s_tok[kListBlock];
  __shared__ int excl[kScanTile];
  __shared__ int wsum[kListBlock / 32];
  __shared__ int s_carry;
  const int C = min(*im.C_ptr, im.Np);
  const int i = b * kListBlock + t;

  int lab = -1;
  int joined = 0, dropped = 0, band = 0;
  if (i < N) {
    const int r = im.slot[i];                     // >= 0: survivor position; < 0: pruned
    const unsigned long long pk = im.best[i];
    lab = (int)(pk & 0xFFFFFFFFull);
    const float dd = __uint_as_float((uint32_t)(pk >> 32));
    if (r >= 0) {
      if ((im.cmask[r >> 5] >> (r & 31)) & 1u) lab = im.cid[r];
    } else {
      if (D::in_band_t(dd, im)) ++band;
      if (D::below_t(dd, im)) ++joined; else { lab = -1; ++dropped; }
    }
    if (lab >= C) lab = -1;                       // only after a failed earlier stage
    im.label[i] = lab;
    if (im.label_user) im.label_user[i] = lab;
  }
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
  const int key = lab < 0 ? kNoLabel : lab;
  slab[t] = key;
  __syncthreads();
  int rank = 0;
#pragma unroll 8
  for (int u = 0; u < kListBlock; ++u) {
    const int o = slab[u];
    rank += (o < key) || (o == key && u < t);
  }
  s_lab[rank] = key;
  s_tok[rank] = i;
  __syncthreads();
  // first position whose cluster id is >= c
  auto lower = [&](int c) {
    int lo = 0, hi = kListBlock;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (s_lab[mid] < c) lo = mid + 1; else hi = mid;
    }
    return lo;
  };
  const int c = s_lab[t];
  const bool valid = c != kNoLabel;
  const int run0 = valid ? lower(c) : t;
  if (valid && run0 == t) {
    const int len = lower(c + 1) - t;
    im.cnt_cb[(size_t)c * im.nbp + b] = (uint16_t)len;
    atomicAdd(&im.csize[c], len);
  }
  TL_POINT(im, 13);
  // every block of the image has published its run lengths before anyone reads them
  __threadfence();
  __syncthreads();
  if (t == 0) {
    atomicAdd(&im.cnt[19], 1);
    int spins = 0;
    while (ld_acquire_i32(&im.cnt[19]) < nblk) {
      if (++spins > spin_limit) { atomicMin(&im.cnt[PACT_CNT_STATUS], (int)PACT_ERR_TIMEOUT); break; }
      __nanosleep(40);
    }
  }
  __syncthreads();
  __threadfence();
  TL_POINT(im, 14);

  // part 2
  int before = 0, size = 0;                          // members of c in earlier blocks; members of c
  if (valid) {
    const uint4 *row = reinterpret_cast<const uint4 *>(im.cnt_cb + (size_t)c * im.nbp);
    for (int v = 0; v * 8 < b; ++v) {
      const uint4 x = __ldcg(row + v);
      const uint32_t xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int cntk = (int)((xs[k >> 1] >> ((k & 1) * 16)) & 0xFFFFu);
        if (v * 8 + k < b) before += cntk;
      }
    }
    size = ld_cg_i32(&im.csize[c]);
  }
  // member_off[c] = cluster sizes below c, scanned kScanTile at a time
  if (t == 0) s_carry = 0;
  __syncthreads();
  int moff = 0;
  for (int base = 0; base < C; base += kScanTile) {
    int v8[8], s = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int cc = base + t * 8 + k;
      v8[k] = cc < C ? ld_cg_i32(&im.csize[cc]) : 0;
      s += v8[k];
    }
    int x = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    int off = s_carry;
    for (int k = 0; k < w; ++k) off += wsum[k];
    int run = off + x - s;
#pragma unroll
    for (int k = 0; k < 8; ++k) { excl[t * 8 + k] = run; run += v8[k]; }
    __syncthreads();
    if (valid && c >= base && c < base + kScanTile) moff = excl[c - base];
    if (t == kListBlock - 1) s_carry = run;
    __syncthreads();
  }
  if (b == 0 && t == 0) im.cnt[20] = s_carry;        // members in all clusters
  if (!valid) return;
  int pos = moff + before + (t - run0);
  pos = max(0, min(pos, N - 1));                     // in bounds whatever an aborted stage left behind
  const int tok = s_tok[t];
  im.members[pos] = make_int4(tok, c, moff, size);
  if (before == 0 && t == run0) {                    // first member of the cluster: the row's bookkeeping
    const int dst = im.vis_start + c;
    if (im.P_out) im.P_out[dst] = im.P[im.vis_start + min(max(im.cidx_ptr[c], 0), N - 1)];
    if (im.size_out) im.size_out[dst] = size;
    if (im.logw_out) im.logw_out[dst] = logf((float)size);   // Eq. 11: log of the token weight
  }
}

// ---- labels and member counts ----------------------------------------------------------------------
// grid (ceil(maxN / 128), B), 128 threads, a group of 32 tokens per warp.  FROM_BEST: the labels are formed from the nearest-centre pass,
// as in k_lists (what does not come from that pass is read before the wait for it); otherwise label[] is given, and an id
// outside [-1, C) is dropped like -1 and reported through the status word.
template <typename T, bool FROM_BEST>
__global__ void __launch_bounds__(kListBlock) k_label_counts(const __grid_constant__ Batch bt) {
  using D = typename DistOf<T>::type;
  const ImgDesc &im = bt.img[blockIdx.y];
  const int i = blockIdx.x * kListBlock + threadIdx.x, lane = threadIdx.x & 31;
  int r = -1, own = -1;
  const int C = min(ld_cg_i32(im.C_ptr), im.Np);
  if (FROM_BEST && i < im.N) {
    r = ld_cg_i32(&im.slot[i]);
    if (r >= 0 && ((__ldcg(&im.cmask[r >> 5]) >> (r & 31)) & 1u)) own = ld_cg_i32(&im.cid[r]);
  }
  pdl_wait();
  pdl_trigger();
  if (i - lane >= im.N) return;
  if (FROM_BEST) {
    label_group<D>(im, i, lane, C, r, own);
  } else {
    int lab = i < im.N ? im.label[i] : -1;
    if (lab >= C || lab < -1) {                        // a label the caller should not have passed
      lab = -1;
      atomicMin(&im.cnt[PACT_CNT_STATUS], (int)PACT_ERR_INVALID_ARG);
    }
    count_group(im, i, lane, lab);
  }
}

// ---- member records from finished labels ----------------------------------------------------------
// grid (ceil(maxN / 128), B), 128 threads.  The rows x centres pass on single CTAs, as its groups of rows finished, or
// k_label_counts has already written the labels, the cluster sizes and cnt_cb (members of cluster c in token block b); what
// is left is the second part of k_lists: the member of cluster c that is token i of block b
// belongs at  member_off[c] + (members of c in the blocks before b) + (members of c before i in block b).
__global__ void __launch_bounds__(kListBlock) k_members(const __grid_constant__ Batch bt, int label_none) {
  const ImgDesc &im = bt.img[blockIdx.y];
  TL_SCOPE(im, 8);
  // the number of clusters was final before the kernel ahead of this one began, and this kernel cannot start before
  // every CTA of that has begun: it may be read ahead of the wait
  const int C = min(ld_cg_i32(im.C_ptr), im.Np);
  pdl_wait();
  pdl_trigger();
  const int N = im.N;
  const int nblk = (N + kListBlock - 1) / kListBlock;
  const int b = blockIdx.x, t = threadIdx.x, lane = t & 31, w = t >> 5;
  if (b >= nblk) return;
  __shared__ __align__(16) int slab[kListBlock];
  __shared__ int excl[kScanTile];
  __shared__ int wsum[kListBlock / 32];
  __shared__ int s_carry;
  const int i = b * kListBlock + t;
  int c = -1;
  if (i < N) {
    if (C > 0) c = ld_cg_i32(&im.label[i]);
    else if (label_none) {                           // no centre at all (a failed earlier stage): nothing was labelled
      im.label[i] = -1;
      if (im.label_user) im.label_user[i] = -1;
    }
    if (c >= C || c < -1) c = -1;
  }
  const bool valid = c >= 0;
  slab[t] = c;
  // in flight while the block is searched: the counts of the earlier blocks, the cluster's size, the sizes to scan
  constexpr int kCbRegs = 8;                         // rows of cnt_cb of up to 64 token blocks are read at once
  uint4 cb[kCbRegs];
  int size = 0;
  const uint4 *row = reinterpret_cast<const uint4 *>(im.cnt_cb + (size_t)(valid ? c : 0) * im.nbp);
#pragma unroll
  for (int v = 0; v < kCbRegs; ++v) cb[v] = (valid && v * 8 < b) ? __ldcg(row + v) : make_uint4(0u, 0u, 0u, 0u);
  if (valid) size = ld_cg_i32(&im.csize[c]);
  int v8[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int cc = t * 8 + k;
    v8[k] = cc < C ? ld_cg_i32(&im.csize[cc]) : 0;
  }
  __syncthreads();
  TL_POINT(im, 13);
  int place = 0;                                     // members of c before token i in this block
  if (valid) {
    const int4 *s4 = reinterpret_cast<const int4 *>(slab);
    const int full = t >> 2;
    for (int u = 0; u < full; ++u) {
      const int4 x = s4[u];
      place += (x.x == c) + (x.y == c) + (x.z == c) + (x.w == c);
    }
    const int4 x = s4[full];
    place += ((t & 3) > 0 && x.x == c) + ((t & 3) > 1 && x.y == c) + ((t & 3) > 2 && x.z == c);
  }
  int before = 0;
#pragma unroll
  for (int v = 0; v < kCbRegs; ++v) {
    const uint32_t xs[4] = {cb[v].x, cb[v].y, cb[v].z, cb[v].w};
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (v * 8 + k < b) before += (int)((xs[k >> 1] >> ((k & 1) * 16)) & 0xFFFFu);
  }
  for (int v0 = kCbRegs; v0 * 8 < b; v0 += kCbRegs) {   // more token blocks than that
#pragma unroll
    for (int v = 0; v < kCbRegs; ++v) cb[v] = (valid && (v0 + v) * 8 < b) ? __ldcg(row + v0 + v) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int v = 0; v < kCbRegs; ++v) {
      const uint32_t xs[4] = {cb[v].x, cb[v].y, cb[v].z, cb[v].w};
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if ((v0 + v) * 8 + k < b) before += (int)((xs[k >> 1] >> ((k & 1) * 16)) & 0xFFFFu);
    }
  }
  // member_off[c] = cluster sizes below c, scanned kScanTile at a time
  if (t == 0) s_carry = 0;
  __syncthreads();
  int moff = 0;
  for (int base = 0; base < C; base += kScanTile) {
    int s = 0;
    if (base > 0) {
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int cc = base + t * 8 + k;
        v8[k] = cc < C ? ld_cg_i32(&im.csize[cc]) : 0;
      }
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) s += v8[k];
    int x = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    int off = s_carry;
    for (int k = 0; k < w; ++k) off += wsum[k];
    int run = off + x - s;
#pragma unroll
    for (int k = 0; k < 8; ++k) { excl[t * 8 + k] = run; run += v8[k]; }
    __syncthreads();
    if (valid && c >= base && c < base + kScanTile) moff = excl[c - base];
    if (t == kListBlock - 1) s_carry = run;
    __syncthreads();
  }
  if (b == 0 && t == 0) im.cnt[20] = s_carry;        // members in all clusters
  TL_POINT(im, 14);
  if (!valid) return;
  int pos = moff + before + place;
  pos = max(0, min(pos, N - 1));                     // in bounds whatever an aborted stage left behind
  im.members[pos] = make_int4(i, c, moff, size);
  if (before == 0 && place == 0) {                   // first member of the cluster: the row's bookkeeping
    const int dst = im.vis_start + c;
    if (im.P_out) im.P_out[dst] = im.P[im.vis_start + min(max(im.cidx_ptr[c], 0), N - 1)];
    if (im.size_out) im.size_out[dst] = size;
    if (im.logw_out) im.logw_out[dst] = logf((float)size);   // Eq. 11: log of the token weight
  }
}

// What k_label_counts and k_merge accumulate into, and the counters (pact_merge; in the whole step k_tokens clears them).
__global__ void __launch_bounds__(256) k_list_clear(const __grid_constant__ Batch bt) {
  pdl_wait();
  pdl_trigger();
  const ImgDesc &im = bt.img[blockIdx.y];
  const int gt = blockIdx.x * 256 + threadIdx.x, gs = gridDim.x * 256;
  if (gt < kCntInts) im.cnt[gt] = 0;
  for (int r = gt; r < im.Np; r += gs) { im.csize[r] = 0; im.cticket[r] = 0; }
  uint4 *tab = reinterpret_cast<uint4 *>(im.cnt_cb);
  const int nq = im.Np * (im.nbp / 8);
  for (int i = gt; i < nq; i += gs) tab[i] = make_uint4(0u, 0u, 0u, 0u);
}

// ---- Eq. 10 ------------------------------------------------------------------------------------------
// Grid (ranges x slices, B), 128 threads, eight CTAs per SM.  Work items are the member records in cluster order
// followed by the text rows; a CTA takes one range of `per` of them and one slice of the columns, a thread VPL groups of
// eight columns, and adds the rows of the running cluster in float.  The rows arrive through two half rings in shared
// memory, one bulk copy per row and one barrier per half: while one half is added the other is on its way.
//
// A cluster of at most `whole` members is done by the range it begins in, however far it reaches past the range's
// end: a cut costs a chain of three trips through the L2 at the end of a CTA (about 2.5 us).  Larger clusters are cut at
// the range boundaries: their sums go to scratch with a ticket, and the CTA that draws a cluster's last ticket adds the
// sums in range order and stores the row, so the result does not depend on which CTA that is.
//
// Instructions count here: 45000 rows of 7 KB (324 MB in, 52 MB out) through 16-byte copies of every thread's own took 85
// warp instructions per 512 bytes and with them 83 us; with bulk copies a thread only adds, and from the end of the lists to
// the end of the last CTA it is 75 us, 5.0 TB/s.  One image of 7290 tokens, 53 MB that mostly lie in the L2: 17 us.
constexpr int kMrgThreads = 128;
constexpr int kMrgRingBytes = 24 * 1024;            // rows in flight per CTA when an SM has eight, more when it has fewer
constexpr int kMrgRingMost = 192 * 1024;
constexpr int kMrgMaxHalf = 32;                     // rows in a half ring

template <typename T, typename O, int VPL>
__global__ void __launch_bounds__(kMrgThreads, kMrgCtasPerSm) k_merge(const __grid_constant__ Batch bt, int per, int whole, int slices, int ring_bytes) {
  const ImgDesc &im = bt.img[blockIdx.y];
  TL_SCOPE(im, 9);
  extern __shared__ uint4 ring[];
  __shared__ uint64_t s_bar[2];
  __shared__ int s_abort;
  if (threadIdx.x == 0) {
    mbar_init(&s_bar[0], 1);
    mbar_init(&s_bar[1], 1);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // (No early trigger: with one the next call's first kernel is placed while this one still fills most SMs, all on the few
  // that are free, and takes 4 to 12 us more from there.)
  pdl_wait();
  const int t = threadIdx.x;
  __shared__ int s_row[kMrgThreads], s_cluster[kMrgThreads], s_dst[kMrgThreads];   // row of H, cluster, output row of an item
  __shared__ float s_inv[kMrgThreads];              // 1 / size (1 for text rows and centre-only merging)
  __shared__ int s_last;
  const int n_text = im.n_total - im.N, d = bt.d, ng = d / 8;
  const bool center_only = (im.flags & PACT_FLAG_CENTER_ONLY) != 0;
  const int x = blockIdx.x / slices, sl = blockIdx.x - x * slices;
  // this slice's groups of eight columns: gn from g0 on; thread t takes g0 + t, g0 + t + nth
  const int gps = (ng + slices - 1) / slices, g0 = sl * gps, gn = min(ng, g0 + gps) - g0, nth = (gn + VPL - 1) / VPL;
  bool mine[VPL];
#pragma unroll
  for (int v = 0; v < VPL; ++v) mine[v] = t < nth && t + v * nth < gn;
  const int lo = x * per;
  // everything the range needs to know in one trip to the L2: the counts, the records of its first items and of its last
  auto fetch = [&](int p) { return center_only ? make_int4(__ldcg(im.cidx_ptr + min(p, im.N - 1)), p, p, 1) : __ldcg(im.members + min(p, im.N - 1)); };
  const int C_raw = ld_cg_i32(im.C_ptr), n_all = ld_cg_i32(&im.cnt[20]);
  const int4 rec_lo = fetch(lo), rec_hi = fetch(lo + per - 1), rec_t = fetch(lo + t);
  const int C = min(C_raw, im.Np), n_mem = center_only ? C : min(max(n_all, 0), im.N);
  const int hi = min(n_mem + n_text, lo + per);
  // every other counter is final: this is the last kernel of the call
  if (blockIdx.x == 0 && t < PACT_N_COUNTERS) im.counters_user[t] = t == PACT_CNT_N_OUT ? n_text + C : ld_cg_i32(&im.cnt[t]);
  if (lo >= hi) return;
  // {token, cluster, first member, size} of a member; in bounds whatever an aborted earlier stage left in the records
  auto checked = [&](int4 r, int p) {
    r.x = min(max(r.x, 0), im.N - 1);
    r.y = min(max(r.y, 0), C - 1);
    r.z = min(max(r.z, 0), p);
    r.w = min(max(r.w, p - r.z + 1), n_mem - r.z);
    return r;
  };
  int start = lo, stop = hi;
  int cut_head = -1, cut_tail = -1;                 // first member of the cut cluster the range begins / ends with
  int cut_head_n = 0, cut_tail_n = 0;
  if (lo < n_mem) {
    const int4 a = checked(rec_lo, lo);
    if (a.z < lo) {
      if (a.w <= whole) start = a.z + a.w;          // done by the range it begins in
      else { cut_head = a.z; cut_head_n = a.w; }
    }
    if (hi < n_mem) {
      const int4 b = checked(rec_hi, hi - 1);
      if (b.z + b.w > hi) {
        if (b.w > whole) { cut_tail = b.z; cut_tail_n = b.w; }
        else if (b.z >= lo) stop = b.z + b.w;       // the last cluster of the range goes on a little
        else stop = lo;                             // (the whole range belongs to a cluster that began before it)
      }
    }
    if (start >= stop) return;
  }

  const T *H = reinterpret_cast<const T *>(im.H) + (size_t)g0 * 8;
  O *Ho = reinterpret_cast<O *>(im.H_out) + (size_t)(g0 + t) * 8;
  float acc[VPL][8];
  auto zero = [&]() {
#pragma unroll
    for (int v = 0; v < VPL; ++v)
#pragma unroll
      for (int e = 0; e < 8; ++e) acc[v][e] = 0.f;
  };
  auto store_row = [&](float inv, int dst) {
    O *o = Ho + (size_t)dst * im.ldHo;
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
      float y[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) y[e] = acc[v][e] * inv;
      if (mine[v]) store_vec8<O>(o + (size_t)v * nth * 8, y);
    }
  };
  // a cluster cut by a range boundary: sum to scratch, ticket, and the last one adds the sums in range order
  auto cut = [&](int first, int size, float inv, int dst, int slot) {
    float *part = im.mpart + (size_t)(g0 + t) * 8;
#pragma unroll
    for (int v = 0; v < VPL; ++v)
      if (mine[v]) {
        float4 *p = reinterpret_cast<float4 *>(part + ((size_t)x * 2 + slot) * d + (size_t)v * nth * 8);
        p[0] = make_float4(acc[v][0], acc[v][1], acc[v][2], acc[v][3]);
        p[1] = make_float4(acc[v][4], acc[v][5], acc[v][6], acc[v][7]);
      }
    const int x0 = first / per, x1 = (first + size - 1) / per;
    int32_t *ticket = &im.cticket[x0 * 8 + sl];     // (at most one cluster goes on after a range; a range has kMrgLeast places or more)
    __threadfence();
    __syncthreads();
    if (t == 0) s_last = (atomicAdd(ticket, 1) == x1 - x0);
    __syncthreads();
    const bool last = s_last != 0;
    __syncthreads();                                 // s_last may be rewritten by the second cut cluster
    if (!last) return;
    __threadfence();
    zero();
#pragma unroll
    for (int v = 0; v < VPL; ++v)
      if (mine[v])
#pragma unroll 4
        for (int xx = x0; xx <= x1; ++xx) {
          const float *p = part + ((size_t)xx * 2 + (xx == x0 ? 1 : 0)) * d + (size_t)v * nth * 8;
          const float4 u = ld_cg_f4(p), w = ld_cg_f4(p + 4);
          acc[v][0] += u.x; acc[v][1] += u.y; acc[v][2] += u.z; acc[v][3] += u.w;
          acc[v][4] += w.x; acc[v][5] += w.y; acc[v][6] += w.z; acc[v][7] += w.w;
        }
    if (t == 0) *ticket = 0;
    store_row(inv, dst);
  };

  const uint32_t rowb = (uint32_t)gn * 8 * (uint32_t)sizeof(T);
  const int half = min(kMrgMaxHalf, ring_bytes / 2 / (int)rowb);   // rows in a half ring (at least three)
  int h = 0, cur = -1, cur_dst = 0;                   // h: the half that is next
  uint32_t par = 0;
  bool first_cut = cut_head >= 0;                     // the running cluster is the one the range begins with
  float cur_inv = 1.f;
  for (int t0 = lo; t0 < stop; t0 += kMrgThreads) {
    const int tn = min(kMrgThreads, stop - t0);
    if (t0 > lo) __syncthreads();                     // the previous tile's records are no longer needed
    if (t < tn) {
      const int p = t0 + t;
      if (p < n_mem) {
        const int4 r = checked(t0 == lo ? rec_t : fetch(p), p);
        s_row[t] = im.vis_start + r.x;
        s_cluster[t] = r.y;
        s_dst[t] = im.vis_start + r.y;
        s_inv[t] = 1.0f / (float)r.w;
      } else {                                        // a text row: a cluster of its own, numbered after the real ones
        const int tr = p - n_mem, src = tr < im.vis_start ? tr : tr + im.N, dst = tr < im.vis_start ? tr : tr + C;
        s_row[t] = src;
        s_cluster[t] = C + tr;
        s_dst[t] = dst;
        s_inv[t] = 1.f;
        if (sl == 0) {
          im.P_out[dst] = im.P[src];
          im.size_out[dst] = 1;
          if (im.logw_out) im.logw_out[dst] = 0.f;
        }
      }
    }
    __syncthreads();
    TL_POINT(im, 15);
    // rows j .. of the tile into half hh (the rows shared out among the warps: issuing one takes a warp about 90 ns)
    // nothing reads them again: their lines leave the L2 first (one image of 7290 tokens 0.5 us, three of 2309 0.9)
    auto issue = [&](int j, int hh) {
      const int n = min(half, tn - j);
      if (n <= 0) return;
      if ((t & 31) != 0 || *const_cast<volatile int *>(&s_abort)) return;   // (nothing is asked for after a wait that ran out)
      if (t == 0) mbar_arrive_expect_tx(&s_bar[hh], (uint32_t)n * rowb);
      for (int k = t >> 5; k < n; k += kMrgThreads / 32)
        bulk_load_hint(reinterpret_cast<uint8_t *>(ring) + (size_t)(hh * half + k) * rowb, H + (size_t)s_row[j + k] * im.ldH, rowb, &s_bar[hh], kEvictFirst);
    };
    const int j0 = max(start - t0, 0);                // (a first tile may begin with items of the range before)
    issue(j0, h);
    issue(j0 + half, h ^ 1);
#pragma unroll 1
    for (int jh = j0; jh < tn; jh += half) {
      // (after a wait that ran out the CTA goes on through its barriers and tickets, but without copies and without waiting)
      if (!mbar_wait_warp_unless(&s_abort, &s_bar[h], (par >> h) & 1)) s_abort = 1;
      par ^= 1u << h;
      const uint8_t *buf = reinterpret_cast<const uint8_t *>(ring) + (size_t)(h * half) * rowb + (size_t)t * 8 * sizeof(T);
      const int je = min(jh + half, tn);
#pragma unroll 1
      for (int j = jh; j < je; ++j, buf += rowb) {
        const int c = s_cluster[j];
        if (c != cur) {                               // the next cluster begins (the same for all threads)
          if (cur >= 0) {
            if (first_cut) cut(cut_head, cut_head_n, cur_inv, cur_dst, 0);
            else store_row(cur_inv, cur_dst);
            first_cut = false;
          }
          zero();
          cur = c; cur_dst = s_dst[j]; cur_inv = s_inv[j];
        }
#pragma unroll
        for (int v = 0; v < VPL; ++v)
          if (mine[v]) {
            Raw8<T> xr;
            xr.from_ring(reinterpret_cast<const uint4 *>(buf + (size_t)v * nth * 8 * sizeof(T)));
            xr.add_to(acc[v]);
          }
      }
      __syncthreads();                                // this half has been read
      issue(jh + 2 * half, h);
      h ^= 1;
    }
  }
  if (first_cut) cut(cut_head, cut_head_n, cur_inv, cur_dst, 0);
  else if (cut_tail >= 0) cut(cut_tail, cut_tail_n, cur_inv, cur_dst, 1);
  else store_row(cur_inv, cur_dst);
  if (t >= 32 || !s_abort) return;
  land_copies(s_bar, 2);
  if (t == 0) atomicMin(&im.counters_user[PACT_CNT_STATUS], (int)PACT_ERR_TIMEOUT);
}

// ---- launchers -----------------------------------------------------------------------------------

static bool lists_in_one(int maxN, int B, const DeviceCfg &cfg) {
  return maxN <= kListsMaxN && (long long)((maxN + kListBlock - 1) / kListBlock) * B <= cfg.lists_resident;
}
int lists_kernels(int maxN, int B, bool from_best, const DeviceCfg &cfg) { return from_best && lists_in_one(maxN, B, cfg) ? 1 : 2; }

cudaError_t launch_members(const Batch &bt, int maxN, bool label_none, cudaStream_t st) {
  const dim3 grid((maxN + kListBlock - 1) / kListBlock, bt.B);
  return launch_k(k_members, grid, dim3(kListBlock), 0, st, true, bt, label_none ? 1 : 0);
}

cudaError_t launch_lists(const Batch &bt, int maxN, bool bf16, bool from_best, int spin_limit, const DeviceCfg &cfg, cudaStream_t st) {
  const dim3 grid((maxN + kListBlock - 1) / kListBlock, bt.B), block(kListBlock);
  if (from_best && lists_in_one(maxN, bt.B, cfg))
    return bf16 ? launch_coop(k_lists<__nv_bfloat16>, grid, block, 0, st, true, bt, spin_limit) : launch_coop(k_lists<float>, grid, block, 0, st, true, bt, spin_limit);
  const auto counts = !from_best ? k_label_counts<float, false> : bf16 ? k_label_counts<__nv_bfloat16, true> : k_label_counts<float, true>;
  const cudaError_t e = launch_k(counts, grid, block, 0, st, true, bt);
  return e != cudaSuccess ? e : launch_members(bt, maxN, false, st);
}

size_t merge_scratch_rows() { return 2 * kMrgRanges; }

template <typename T, typename O, int VPL>
static cudaError_t launch_merge_v(const Batch &bt, int n_items, int slices, const DeviceCfg &cfg, cudaStream_t st) {
  const int per = merge_per(n_items, slices, bt.B, cfg.sm_count), ranges = (n_items + per - 1) / per;
  const long long per_sm = ((long long)ranges * slices * bt.B + cfg.sm_count - 1) / cfg.sm_count;
  int ring = per_sm >= kMrgCtasPerSm ? kMrgRingBytes : (int)(kMrgCtasPerSm * kMrgRingBytes / per_sm);
  if (ring > kMrgRingMost) ring = kMrgRingMost;
  const int row = ((bt.d / 8 + slices - 1) / slices) * 8 * (int)sizeof(T), most = 2 * kMrgMaxHalf, room = (ring / row < most ? ring / row : most) - per;
  const int whole = merge_whole(per, per_sm, room);
  return launch_k(k_merge<T, O, VPL>, dim3(ranges * slices, bt.B), dim3(kMrgThreads), (size_t)ring, st, true, bt, per, whole, slices, ring);
}

template <typename T, typename O>
static cudaError_t launch_merge_t(const Batch &bt, const DeviceCfg &cfg, cudaStream_t st) {
  int n_items = 1;
  for (int b = 0; b < bt.B; ++b) n_items = bt.img[b].n_total > n_items ? bt.img[b].n_total : n_items;
  const int s1 = (bt.d / 8 + kMrgThreads - 1) / kMrgThreads, s2 = (bt.d / 8 + 2 * kMrgThreads - 1) / (2 * kMrgThreads);
  // Two groups of columns per thread halve the instructions per byte, which counts when the GPU has several rounds of
  // CTAs to do (46000 rows of 7 KB: 4 us of 75); with less, narrower slices spread the rows over more CTAs (7300 rows:
  // 2 us of 20 the other way).  Rows of fp32 stay at one group: 4 KB per row and slice.
  if constexpr (sizeof(T) == 2)
    if ((long long)n_items * s1 * bt.B >= 64LL * kMrgCtasPerSm * cfg.sm_count) return launch_merge_v<T, O, 2>(bt, n_items, s2, cfg, st);
  return launch_merge_v<T, O, 1>(bt, n_items, s1, cfg, st);
}

template <typename T, typename O> static cudaError_t merge_attr() {
  cudaError_t e = cudaFuncSetAttribute(k_merge<T, O, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMrgRingMost);
  if constexpr (sizeof(T) == 2)
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_merge<T, O, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMrgRingMost);
  return e;
}

cudaError_t merge_configure(DeviceCfg *cfg) {
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_lists<__nv_bfloat16>, kListBlock, 0);
  if (e != cudaSuccess) return e;
  int m = per_sm;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_lists<float>, kListBlock, 0);
  if (e != cudaSuccess) return e;
  m = per_sm < m ? per_sm : m;
  cfg->lists_resident = m * cfg->sm_count;
  e = merge_attr<__nv_bfloat16, __nv_bfloat16>();
  if (e == cudaSuccess) e = merge_attr<__nv_bfloat16, float>();
  if (e == cudaSuccess) e = merge_attr<float, __nv_bfloat16>();
  if (e == cudaSuccess) e = merge_attr<float, float>();
  return e;
}

cudaError_t launch_list_clear(const Batch &bt, cudaStream_t st) {
  const long long words = (long long)bt.img[0].Np * (bt.img[0].nbp / 8);
  const long long X = (words + 2047) / 2048;          // eight 16-byte stores per thread
  return launch_k(k_list_clear, dim3((unsigned)(X < 1 ? 1 : (X > 1184 ? 1184 : X)), bt.B), dim3(256), 0, st, true, bt);
}

cudaError_t launch_merge(const Batch &bt, bool in_bf16, bool out_bf16, const DeviceCfg &cfg, cudaStream_t st) {
  if (in_bf16) return out_bf16 ? launch_merge_t<__nv_bfloat16, __nv_bfloat16>(bt, cfg, st)
                               : launch_merge_t<__nv_bfloat16, float>(bt, cfg, st);
  return out_bf16 ? launch_merge_t<float, __nv_bfloat16>(bt, cfg, st) : launch_merge_t<float, float>(bt, cfg, st);
}

}  // namespace pact
