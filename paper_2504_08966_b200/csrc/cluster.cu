// DBDPC (Algorithm 2) and reincorporation (Eq. 8-9): key gather and inverse norms, all-pairs
// distance tiles with the density and the d <= d_c adjacency fused into their epilogue, density
// rank, centre selection, tokens-by-centres nearest-centre pass, labels.
//
// This file holds the double-precision tile kernels (any element type and key width); the tcgen05 tile
// kernels for bf16 keys live in gram_umma.cu and share the epilogue arithmetic of common.cuh.
#include "f64_tiles.cuh"
#include "kernels.cuh"
#include "tma.cuh"

namespace pact {

__device__ __forceinline__ uint32_t ld_relaxed_u32(const uint32_t *p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// ---- inverse key norms, survivor gather, per-call initialisation (stage calls) ------------------------
// grid (ceil(maxN / 8), B), 256 threads, one warp per list position r (token kept_idx[r]).
template <typename T>
__global__ void __launch_bounds__(256) k_keynorm_gather(const __grid_constant__ Batch bt) {
  using D = typename DistOf<T>::type;
  using rn_t = typename D::rn_t;
  constexpr int V = Vec<T>::N;
  pdl_wait();
  pdl_trigger();
  const ImgDesc &im = bt.img[blockIdx.y];
  const int lane = threadIdx.x & 31;
  const int r = blockIdx.x * 8 + (threadIdx.x >> 5);
  const int q = *im.q_ptr;
  // arrays later kernels accumulate into
  {
    const int gt = blockIdx.x * 256 + threadIdx.x, gs = gridDim.x * 256;
    for (int k = gt; k < im.Np; k += gs) im.rho_fix[k] = 0ull;
    for (int wd = gt; wd < im.Wp; wd += gs) { im.cmask[wd] = 0u; im.rmask[wd] = 0u; }
    for (int i = gt; i < im.N; i += gs) {
      im.best[i] = kBestInit;
      if (im.label_user) im.label_user[i] = -1;
    }
    if (gt < kCntInts) im.cnt[gt] = 0;
  }
  if (r >= q) return;
  const int i = im.kept_idx[r];
  const T *row = reinterpret_cast<const T *>(im.Kc) + (size_t)i * im.ldKc;
  const double ss = row_sumsq<T>(row, bt.d_k, lane);
  const rn_t rn = (rn_t)inv_norm(ss);
  if (lane == 0) {
    rn_tok<D>(im)[i] = rn;
    rn_kept<D>(im)[r] = rn;
  }
  T *dst = reinterpret_cast<T *>(im.Kp) + (size_t)r * bt.d_k;
  for (int v = lane; v * V < bt.d_k; v += 32)
    reinterpret_cast<uint4 *>(dst)[v] = reinterpret_cast<const uint4 *>(row)[v];
}

// Centre keys from a list of token indices (reincorporation as a stage of its own), inverse norms of all rows
// (all_rows) or of the listed pruned rows, per-call initialisation.  One warp per centre and row.
template <typename T>
__global__ void __launch_bounds__(256) k_center_key_gather(const __grid_constant__ Batch bt, int all_rows) {
  using D = typename DistOf<T>::type;
  using rn_t = typename D::rn_t;
  constexpr int V = Vec<T>::N;
  pdl_wait();
  pdl_trigger();
  const ImgDesc &im = bt.img[blockIdx.y];
  const int lane = threadIdx.x & 31;
  const int c = blockIdx.x * 8 + (threadIdx.x >> 5);
  {
    const int gt = blockIdx.x * 256 + threadIdx.x, gs = gridDim.x * 256;
    for (int i = gt; i < im.N; i += gs) im.best[i] = kBestInit;
    if (gt < kCntInts) im.cnt[gt] = 0;
    if (gt == 0) *im.r_user = 0;
  }
  if (c < (all_rows ? im.N : *im.m_ptr)) {   // inverse norm of row c, or of the c-th pruned row
    const int i = all_rows ? c : im.pruned_idx[c];
    const double ss = row_sumsq<T>(reinterpret_cast<const T *>(im.Kc) + (size_t)i * im.ldKc, bt.d_k, lane);
    if (lane == 0) rn_tok<D>(im)[i] = (rn_t)inv_norm(ss);
  }
  if (c >= *im.C_ptr) return;
  const int i = im.cidx_ptr[c];
  const T *row = reinterpret_cast<const T *>(im.Kc) + (size_t)i * im.ldKc;
  const double ss = row_sumsq<T>(row, bt.d_k, lane);
  if (lane == 0) rn_cen<D>(im)[c] = (rn_t)inv_norm(ss);
  T *dst = reinterpret_cast<T *>(im.Kcen) + (size_t)c * bt.d_k;
  for (int v = lane; v * V < bt.d_k; v += 32)
    reinterpret_cast<uint4 *>(dst)[v] = reinterpret_cast<const uint4 *>(row)[v];
}

// ---- Eq. 5-6: all pairs of survivors; density and adjacency in the epilogue --------------------
// grid (n_ctas, B) persistent over the tiles on and above the diagonal of the q x q matrix; nothing of it is stored
// except one bit per pair (d <= d_c) and one integer density per row.  A tile above the diagonal serves its rows and
// its columns; the two inverse norms are multiplied first, so that a pair has the same distance from both sides and
// duplicate keys keep exactly equal densities.
template <typename T>
__global__ void __launch_bounds__(kTileThreads) k_gram_f64(const __grid_constant__ Batch bt) {
  using D = typename DistOf<T>::type;
  pdl_wait();
  pdl_trigger();
  const ImgDesc &im = bt.img[blockIdx.y];
  TL_SCOPE(im, 4);
  const int q = *im.q_ptr;
  const int nt = (q + TS - 1) / TS;
  const int t = threadIdx.x;
  __shared__ __align__(16) double As[TS][KST];
  __shared__ __align__(16) double Bs[TS][KST];
  __shared__ F64Sums sums;
  const T *Kp = reinterpret_cast<const T *>(im.Kp);
  const auto *rnk = rn_kept<D>(im);
  int band = 0;
  for (int tile = blockIdx.x; tile < nt * (nt + 1) / 2; tile += gridDim.x) {
    int tm, tn;
    upper_tile(tile, nt, tm, tn);
    double acc[2][2][2];
    tile_dots<T>(
        t, [&](int r) { const int g = tm * TS + r; return g < q ? Kp + (size_t)g * bt.d_k : (const T *)nullptr; },
        [&](int r) { const int g = tn * TS + r; return g < q ? Kp + (size_t)g * bt.d_k : (const T *)nullptr; },
        bt.d_k, As, Bs, acc, []() { __syncthreads(); });
    gram_epilogue_f64<D>(t, tm, tn, q, acc, [&](int g) { return (double)rnk[g]; }, im, sums, band, []() { __syncthreads(); });
  }
  if (band) atomicAdd(&im.cnt[PACT_CNT_BAND_DC], band);
}

// ---- choice of the reduction layer: largest distance between two keys of a layer ---------------
// Each image of the batch is one layer's key matrix (Kc, N rows).  Inverse norms first (one warp per
// key), then the tiles on and above the diagonal with a max-epilogue; the result accumulates in
// cnt[kCntSpread] as the bit pattern of a non-negative float.
template <typename T>
__global__ void __launch_bounds__(256) k_key_rnorm(const __grid_constant__ Batch bt) {
  using D = typename DistOf<T>::type;
  using rn_t = typename D::rn_t;
  pdl_wait();
  pdl_trigger();
  const ImgDesc &im = bt.img[blockIdx.y];
  const int lane = threadIdx.x & 31;
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i == 0 && lane == 0) im.cnt[kCntSpread] = 0;
  if (i >= im.N) return;
  const T *row = reinterpret_cast<const T *>(im.Kc) + (size_t)i * im.ldKc;
  const double ss = row_sumsq<T>(row, bt.d_k, lane);
  if (lane == 0) rn_tok<D>(im)[i] = (rn_t)inv_norm(ss);
}

template <typename T>
__global__ void __launch_bounds__(kTileThreads) k_spread_f64(const __grid_constant__ Batch bt) {
  using D = typename DistOf<T>::type;
  using acc_t = typename D::acc_t;
  pdl_wait();
  pdl_trigger();
  const ImgDesc &im = bt.img[blockIdx.y];
  const int N = im.N;
  const int nt = (N + TS - 1) / TS;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5, wy = w >> 1, wx = w & 1;
  __shared__ __align__(16) double As[TS][KST];
  __shared__ __align__(16) double Bs[TS][KST];
  const T *K = reinterpret_cast<const T *>(im.Kc);
  const auto *rn = rn_tok<D>(im);
  float mx = 0.f;
  for (int tile = blockIdx.x; tile < nt * (nt + 1) / 2; tile += gridDim.x) {   // every unordered pair once
    int tm, tn;
    upper_tile(tile, nt, tm, tn);
    double acc[2][2][2];
    tile_dots<T>(
        t, [&](int r) { const int g = tm * TS + r; return g < N ? K + (size_t)g * im.ldKc : (const T *)nullptr; },
        [&](int r) { const int g = tn * TS + r; return g < N ? K + (size_t)g * im.ldKc : (const T *)nullptr; },
        bt.d_k, As, Bs, acc, []() { __syncthreads(); });
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      const int gi = tm * TS + wy * 16 + a * 8 + (lane >> 2);
      if (gi >= N) continue;
      const auto rni = rn[gi];
#pragma unroll
      for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int gj = tn * TS + wx * 16 + b * 8 + 2 * (lane & 3) + e;
          if (gj >= N || gj == gi) continue;
          mx = fmaxf(mx, (float)D::dist((acc_t)acc[a][b][e], rni, rn[gj]));
        }
    }
  }
  const unsigned wmx = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));   // distances are >= 0
  if (lane == 0 && wmx) atomicMax(reinterpret_cast<unsigned *>(&im.cnt[kCntSpread]), wmx);
}

// one warp: max_dist[l] of the layers of this batch, and the earliest layer at or above the threshold
__global__ void k_spread_finish(const __grid_constant__ Batch bt, float *max_dist, int32_t *layer_out,
                                int layer_base, float threshold) {
  pdl_wait();
  pdl_trigger();
  const int l = threadIdx.x;
  float v = -1.f;
  if (l < bt.B) {
    v = __int_as_float(bt.img[l].cnt[kCntSpread]);
    max_dist[layer_base + l] = v;
  }
  const unsigned hit = __ballot_sync(0xffffffffu, l < bt.B && v >= threshold);
  if (l == 0 && layer_out) {
    if (layer_base == 0) *layer_out = -1;
    if (hit && *layer_out < 0) *layer_out = layer_base + (__ffs(hit) - 1);
  }
}

// ---- centre selection -------------------------------------------------------------------------
// The sequential loop of Algorithm 2 picks the lexicographically first maximal independent set of
// the graph {d_ij <= d_c} in density order (ties: lower index first); that set is unique, so any
// schedule that only takes final decisions reproduces it (the argument of Appendix D.2).  A row becomes
//   removed  once an earlier neighbour is a centre,
//   a centre once every earlier neighbour is removed.
// Both facts are monotone bits of two masks in global memory, so rows are resolved asynchronously and a decision may reach
// others late.  A new centre removes its neighbours itself: it sets its adjacency words in the mask of removed rows (an
// earlier neighbour is in it already).  A row keeps one earlier neighbour that is not removed as its witness and looks at
// its adjacency words again only when the witness has been removed; without another one it is a centre.  (A row whose
// witness is a centre waits for its own bit.)  Most rows are looked at once or twice; with every row's earlier neighbours
// filtered first and every open row tested against both masks in every sweep, 16 images of 1458 survivors took 23 us for
// the same decisions.
//
// k_centers: one CTA of 1024 threads per SM, the CTAs shared out evenly among the images (the last image also takes the
// remainder).  A CTA has a block of rows, their adjacency words and all densities of its image in shared memory (what does
// not fit stays in the L2); lane k of warp w keeps the state of row w + 32 k.  In a sweep the CTA copies the mask of removed
// rows to shared memory once (thousands of warps polling the same few L2 lines queue up there), and its warps decide what
// they can from the copy.  Bound by latency, a trip to the L2 per sweep: 8 us for one image of 3645 survivors, 11 us for 16
// of 1458, 14 us for 4 of 4916.
// CTAs wait for one another's decisions but need not be resident together: after kCenIdle sweeps in which no row of the image
// was removed a CTA leaves its open rows to k_center_keys, where every CTA resolves what is open by itself.  (Progress is
// what counts, not the number of sweeps: 2600 rows whose decisions hang on one another in a chain of 1300 take 1300 sweeps
// and more, and left to k_center_keys after 512 they took 175 ms.)  (As a cooperative launch the kernel could not
// begin beside the one before, which cost a call on a stream 4 us.  One cluster of 16 CTAs per image, with masks in each
// other's shared memory, was no faster with 16 images and 18 us slower with one: 16 SMs are too few to take in the rows.)
//
// k_center_keys: cluster ids (number of centres with a lower index), centre list, centre keys and inverse norms.
constexpr int kCenThreads = 1024;
constexpr int kCenWarps = kCenThreads / 32;
static_assert(kCenWarps == 32, "lane k of warp w has row w + 32 k");
constexpr int kCenIdle = 512;                            // sweeps of k_centers without a removed row (about a microsecond each)

// One row against the removed rows, by a warp: an earlier neighbour that is not removed, or -1.
__device__ __forceinline__ int open_earlier(const uint32_t *row, const uint32_t *removed, const unsigned long long *keys, int r, int nw, int lane) {
  const unsigned long long mine = keys[r];
  for (int base = 0; base < nw; base += 32) {
    const int wd = base + lane;
    uint32_t bits = wd < nw ? row[wd] & ~removed[wd] : 0u;
    if (wd == (r >> 5)) bits &= ~(1u << (r & 31));
    while (__any_sync(0xffffffffu, bits != 0u)) {        // a bit per lane at a time: nearly always the first will do
      int found = -1;
      if (bits) {
        const int j = wd * 32 + __ffs(bits) - 1;
        bits &= bits - 1;
        const unsigned long long o = keys[j];
        if (o > mine || (o == mine && j < r)) found = j;
      }
      const unsigned hits = __ballot_sync(0xffffffffu, found >= 0);
      if (hits) return __shfl_sync(0xffffffffu, found, __ffs(hits) - 1);
    }
  }
  return -1;
}

__global__ void __launch_bounds__(kCenThreads, 1) k_centers(const __grid_constant__ Batch bt, int mask_cap, int keys_cap, int adj_bytes,
                                                            int sweep_limit) {
  TL_SCOPE(bt.img[0], 5);
  extern __shared__ __align__(16) uint8_t cen_smem[];
  uint32_t *rm = reinterpret_cast<uint32_t *>(cen_smem);              // [mask_cap] copy of the removed rows
  unsigned long long *skeys = reinterpret_cast<unsigned long long *>(rm + mask_cap);   // [keys_cap] densities
  uint4 *sadj = reinterpret_cast<uint4 *>(skeys + keys_cap);          // adjacency words of the first rows of the CTA
  __shared__ uint64_t s_bar;
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const int per = max(1, (int)gridDim.x / bt.B);
  const int b = min((int)blockIdx.x / per, bt.B - 1);
  const int ncta = b == bt.B - 1 ? (int)gridDim.x - per * (bt.B - 1) : per, rank = (int)blockIdx.x - b * per;
  const ImgDesc &im = bt.img[b];
  if (t == 0) {
    mbar_init(&s_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // the number of survivors comes from a kernel before the all-pairs pass, and this kernel begins when every CTA of that pass is
  // past its wait (pdl_trigger() never comes first): it may be read ahead of the wait (DBDPC and merge of 7290 tokens 113.9 -> 112.9 us with that here and in k_center_keys)
  const int q = (int)ld_relaxed_u32(reinterpret_cast<const uint32_t *>(im.q_ptr)), nw = (q + 31) >> 5, nv = (nw + 3) >> 2;
  const int rows = (q + ncta - 1) / ncta, r0 = min(q, rank * rows), n = min(q, r0 + rows) - r0;
  for (int wd = t; wd < nw; wd += kCenThreads) rm[wd] = 0u;
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  if (n <= 0) return;
  const bool in_smem = q <= keys_cap;
  if (in_smem && t == 0) {
    const uint32_t bytes = ((uint32_t)q * 8 + 15) & ~15u;
    mbar_arrive_expect_tx(&s_bar, bytes);
    bulk_load(skeys, im.rho_fix, bytes, &s_bar);
  }
  const unsigned long long *keys = in_smem ? skeys : im.rho_fix;
  const int nsm = min(n, adj_bytes / (nv * 16));
  for (int l = wid; l < nsm; l += 4 * kCenWarps)
    for (int v = lane; v < nv; v += 32) {
      uint4 x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (l + u * kCenWarps < nsm) x[u] = __ldcg(reinterpret_cast<const uint4 *>(im.adj + (size_t)(r0 + l + u * kCenWarps) * im.Wp) + v);
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (l + u * kCenWarps < nsm) sadj[(size_t)(l + u * kCenWarps) * nv + v] = x[u];
    }
  if (in_smem) mbar_wait_warp_or_report(&s_bar, 0, &im.cnt[PACT_CNT_STATUS]);
  __syncthreads();
  TL_POINT(bt.img[0], 10);

  int wit = -1;                                          // witness of row wid + 32 lane
  bool done = false;                                     // that row is a centre
  int sweeps = 0, idle = 0;
  for (;;) {
    int pending = 0;
    ++sweeps;
    for (int m = 0; m * kCenThreads < n; ++m) {
      const int l = wid + 32 * (m * 32 + lane), r = r0 + l;
      bool open = l < n && !(m == 0 && done) && !((rm[r >> 5] >> (r & 31)) & 1u);
      if (m > 0 && open) open = !((ld_relaxed_u32(&im.cmask[r >> 5]) >> (r & 31)) & 1u);   // (blocks of more than 1024 rows)
      const bool look = open && (m > 0 || wit < 0 || ((rm[wit >> 5] >> (wit & 31)) & 1u));
      pending |= open && !look;
      unsigned todo = __ballot_sync(0xffffffffu, look);
      while (todo) {
        const int k = __ffs(todo) - 1, ll = wid + 32 * (m * 32 + k), rr = r0 + ll;
        todo &= todo - 1;
        const uint32_t *row = ll < nsm ? reinterpret_cast<const uint32_t *>(sadj + (size_t)ll * nv) : im.adj + (size_t)rr * im.Wp;
        const int f = open_earlier(row, rm, keys, rr, nw, lane);
        if (f >= 0) {
          pending = 1;
          if (m == 0 && lane == k) wit = f;
          continue;
        }
        for (int wd = lane; wd < nw; wd += 32) {
          uint32_t e = row[wd];
          if (wd == (rr >> 5)) {
            e &= ~(1u << (rr & 31));
            atomicOr(&im.cmask[wd], 1u << (rr & 31));
          }
          if (e) atomicOr(&im.rmask[wd], e);
        }
        if (m == 0 && lane == k) done = true;
      }
    }
    if (!__syncthreads_or(pending)) break;               // no row of this CTA is open
    if (sweeps >= sweep_limit || idle >= kCenIdle) {
      if (t == 0 && sweeps >= sweep_limit) atomicMin(&im.cnt[PACT_CNT_STATUS], (int)PACT_ERR_TIMEOUT);
      break;
    }
    int moved = 0;
    for (int wd = t; wd < nw; wd += kCenThreads) {
      const uint32_t x = ld_relaxed_u32(&im.rmask[wd]);
      moved |= x != rm[wd];
      rm[wd] = x;
    }
    idle = __syncthreads_or(moved) ? 0 : idle + 1;
  }
  TL_POINT(bt.img[0], 11);
  if (in_smem && !mbar_try_wait(&s_bar, 0)) land_copies(&s_bar, 1);   // (only after a wait that ran out)
  if (t == 0) atomicMax(&im.cnt[PACT_CNT_SWEEPS], sweeps);
}

// grid (X, B), 256 threads, dynamic smem: three words per 32 survivors.
constexpr int kCenKeyThreads = 256;

template <typename T>
__global__ void __launch_bounds__(kCenKeyThreads) k_center_keys(const __grid_constant__ Batch bt, int mask_cap) {
  using D = typename DistOf<T>::type;
  constexpr int V = Vec<T>::N, kWarps = kCenKeyThreads / 32;
  const ImgDesc &im = bt.img[blockIdx.y];
  extern __shared__ __align__(16) uint8_t cen_smem[];
  uint32_t *cm = reinterpret_cast<uint32_t *>(cen_smem), *rm = cm + mask_cap;   // [mask_cap] centres, removed rows
  int *pref = reinterpret_cast<int *>(rm + mask_cap);                 // [mask_cap] centres before the word
  __shared__ int wsum[kWarps], s_carry;
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  if (t == 0) s_carry = 0;
  const int q = (int)ld_relaxed_u32(reinterpret_cast<const uint32_t *>(im.q_ptr));   // (ahead of the wait, as in k_centers)
  pdl_wait();
  pdl_trigger();
  TL_POINT(bt.img[0], 12);
  const int nw = (q + 31) >> 5, gw = blockIdx.x * kWarps + wid, nwarps = gridDim.x * kWarps;
  int open = 0;
  for (int wd = t; wd < nw; wd += kCenKeyThreads) {
    const uint32_t c = __ldcg(&im.cmask[wd]), r = __ldcg(&im.rmask[wd]);
    cm[wd] = c;
    rm[wd] = r;
    open |= (c | r) != (wd * 32 + 32 <= q ? 0xffffffffu : (1u << (q & 31)) - 1u);
  }
  if (__syncthreads_or(open)) {
    // Rows that k_centers left: every CTA resolves them, to the same end (the set is unique), against its own copies;
    // the first CTA also writes the centres for later kernels.  The earliest open row is decided in every pass, so q passes
    // are enough.
    int passes = 0;
    do {
      open = 0;
      for (int r = wid; r < q; r += kWarps) {
        const uint32_t bit = 1u << (r & 31);
        const volatile uint32_t *vc = cm + (r >> 5), *vr = rm + (r >> 5);
        if ((*vc | *vr) & bit) continue;
        const uint32_t *row = im.adj + (size_t)r * im.Wp;
        // (the neighbour of a centre is removed here as well: should an earlier stage have failed, the words need not be
        // symmetric, and the earliest open row must still be decided)
        int hit = 0;
        for (int wd = lane; wd < nw; wd += 32) hit |= (row[wd] & *const_cast<volatile uint32_t *>(cm + wd)) != 0u;
        if (__any_sync(0xffffffffu, hit)) {
          if (lane == 0) atomicOr(&rm[r >> 5], bit);
          continue;
        }
        if (open_earlier(row, rm, im.rho_fix, r, nw, lane) >= 0) { open = 1; continue; }
        for (int wd = lane; wd < nw; wd += 32) {
          uint32_t e = row[wd];
          if (wd == (r >> 5)) {
            e &= ~bit;
            atomicOr(&cm[wd], bit);
            if (blockIdx.x == 0) atomicOr(&im.cmask[wd], bit);
          }
          if (e) atomicOr(&rm[wd], e);
        }
      }
      if (++passes > q) {
        if (t == 0) atomicMin(&im.cnt[PACT_CNT_STATUS], (int)PACT_ERR_TIMEOUT);
        open = 0;
      }
    } while (__syncthreads_or(open));
    if (blockIdx.x == 0 && t == 0) im.cnt[PACT_CNT_SWEEPS] += passes;
  }
  for (int base = 0; base < nw; base += kCenKeyThreads) {
    const int wd = base + t, pc = wd < nw ? __popc(cm[wd]) : 0;
    int x = pc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) wsum[wid] = x;
    __syncthreads();
    int off = s_carry;
    for (int k = 0; k < wid; ++k) off += wsum[k];
    if (wd < nw) pref[wd] = off + x - pc;
    __syncthreads();
    if (t == kCenKeyThreads - 1) s_carry = off + x;
    __syncthreads();
  }
  if (blockIdx.x == 0 && t == 0) {
    im.cnt[PACT_CNT_C] = s_carry;
    if (im.C_user) *im.C_user = s_carry;
  }
  for (int r = gw; r < q; r += nwarps) {
    if (lane == 0 && im.rho_user) im.rho_user[r] = (float)((double)__ldcg(&im.rho_fix[r]) * (1.0 / (double)(1u << kRhoShift)));
    const uint32_t m = cm[r >> 5];
    if (!((m >> (r & 31)) & 1u)) continue;
    const int c = pref[r >> 5] + __popc(m & ((1u << (r & 31)) - 1u));
    const T *src = reinterpret_cast<const T *>(im.Kp) + (size_t)r * bt.d_k;
    const int nvk = bt.d_k / V;
    uint4 buf[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (lane + 32 * u < nvk) buf[u] = __ldcg(reinterpret_cast<const uint4 *>(src) + lane + 32 * u);
    if (lane == 0) {
      const int tok = im.kept_idx[r];
      im.cid[r] = c;
      im.center_idx[c] = tok;
      if (im.center_idx_user) im.center_idx_user[c] = tok;
      rn_cen<D>(im)[c] = rn_kept<D>(im)[r];
    }
    uint4 *dst = reinterpret_cast<uint4 *>(reinterpret_cast<T *>(im.Kcen) + (size_t)c * bt.d_k);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (lane + 32 * u < nvk) dst[lane + 32 * u] = buf[u];
    for (int v = lane + 128; v < nvk; v += 32) dst[v] = __ldcg(reinterpret_cast<const uint4 *>(src) + v);
  }
}

// ---- nearest centre of every row (Algorithm 2 assignment; Eq. 8 argmin) ---------------------------
// grid (n_ctas, B) persistent over 32 x 32 tiles of rows x centres; the running minimum of a row
// is one 64-bit word (distance bits, cluster id) reduced with atomicMin, so ties go to the lower id.
template <typename T>
__global__ void __launch_bounds__(kTileThreads) k_assign_f64(const __grid_constant__ Batch bt, int mode) {
  using D = typename DistOf<T>::type;
  pdl_wait();
  pdl_trigger();
  const ImgDesc &im = bt.img[blockIdx.y];
  TL_SCOPE(im, 6);
  const int C = *im.C_ptr;
  const int nrows = mode == ROWS_ALL ? im.N : (mode == ROWS_KEPT_LIST ? *im.q_ptr : *im.m_ptr);
  const int32_t *list = mode == ROWS_KEPT_LIST ? im.kept_idx : im.pruned_idx;
  const int ntm = (nrows + TS - 1) / TS, ntn = (C + TS - 1) / TS;
  const int t = threadIdx.x;
  __shared__ __align__(16) double As[TS][KST];
  __shared__ __align__(16) double Bs[TS][KST];
  __shared__ unsigned long long rowbest[2][TS];
  __shared__ int rowtok[TS];
  const T *Kc = reinterpret_cast<const T *>(im.Kc);
  const T *Kcen = reinterpret_cast<const T *>(im.Kcen);
  const auto *rnt = rn_tok<D>(im);
  const auto *rnc = rn_cen<D>(im);
  for (int tile = blockIdx.x; tile < ntm * ntn; tile += gridDim.x) {
    const int tm = tile / ntn, tn = tile % ntn;
    __syncthreads();                                   // the tile before has written its minima
    if (t < TS) {
      const int g = tm * TS + t;
      rowtok[t] = g < nrows ? (mode == ROWS_ALL ? g : list[g]) : -1;
    }
    __syncthreads();
    double acc[2][2][2];
    tile_dots<T>(
        t, [&](int r) { const int tok = rowtok[r]; return tok >= 0 ? Kc + (size_t)tok * im.ldKc : (const T *)nullptr; },
        [&](int r) { const int g = tn * TS + r; return g < C ? Kcen + (size_t)g * bt.d_k : (const T *)nullptr; },
        bt.d_k, As, Bs, acc, []() { __syncthreads(); });
    assign_epilogue_f64<D>(t, tn * TS, C, acc, [&](int l) { return rowtok[l] >= 0 ? rnt[rowtok[l]] : (typename D::rn_t)0; },
                           [&](int c) { return rnc[c]; }, rowbest);
    __syncthreads();
    if (t < TS && rowtok[t] >= 0) atomicMin(&im.best[rowtok[t]], rowbest[0][t] < rowbest[1][t] ? rowbest[0][t] : rowbest[1][t]);
  }
}

// ---- labels -----------------------------------------------------------------------------------
// survivors: cluster id of the nearest centre (a centre: its own id); pruned tokens: that id iff
// the distance is strictly below alpha * d_c, else -1.
template <typename T>
__global__ void __launch_bounds__(256) k_label(const __grid_constant__ Batch bt, int mode) {
  using D = typename DistOf<T>::type;
  const ImgDesc &im = bt.img[blockIdx.y];
  TL_SCOPE(im, 7);
  pdl_wait();
  pdl_trigger();
  const int nrows = mode == ROWS_ALL ? im.N : (mode == ROWS_KEPT_LIST ? *im.q_ptr : *im.m_ptr);
  int joined = 0, dropped = 0, band = 0;
  for (int g = blockIdx.x * 256 + threadIdx.x; g < nrows; g += gridDim.x * 256) {
    int tok, r;                                   // r >= 0: survivor position; < 0: pruned
    if (mode == ROWS_ALL) { tok = g; r = im.slot[g]; }
    else if (mode == ROWS_KEPT_LIST) { tok = im.kept_idx[g]; r = g; }
    else { tok = im.pruned_idx[g]; r = -1; }
    const unsigned long long pk = im.best[tok];
    int lab = (int)(pk & 0xFFFFFFFFull);
    const float dd = __uint_as_float((uint32_t)(pk >> 32));
    if (r >= 0) {
      if ((im.cmask[r >> 5] >> (r & 31)) & 1u) lab = im.cid[r];
    } else {
      if (D::in_band_t(dd, im)) ++band;
      if (D::below_t(dd, im)) ++joined; else { lab = -1; ++dropped; }
    }
    im.label[tok] = lab;
    if (im.label_user) im.label_user[tok] = lab;
  }
  // warp-aggregated counters
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    joined += __shfl_xor_sync(0xffffffffu, joined, o);
    dropped += __shfl_xor_sync(0xffffffffu, dropped, o);
    band += __shfl_xor_sync(0xffffffffu, band, o);
  }
  if ((threadIdx.x & 31) == 0) {
    if (joined) {
      atomicAdd(&im.cnt[PACT_CNT_R], joined);
      if (im.r_user) atomicAdd(im.r_user, joined);
    }
    if (dropped) atomicAdd(&im.cnt[PACT_CNT_DISCARDED], dropped);
    if (band) atomicAdd(&im.cnt[PACT_CNT_BAND_ADC], band);
  }
}

// ---- launchers ---------------------------------------------------------------------------------

cudaError_t cluster_configure(DeviceCfg *cfg) {
  cfg->centers_smem_max = (int)cfg->smem_optin - 1024;
  cudaError_t e = cudaFuncSetAttribute(k_centers, cudaFuncAttributeMaxDynamicSharedMemorySize, cfg->centers_smem_max);
  constexpr int masks = (kMaxTokens / 32 + 4) * 12;
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_center_keys<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, masks);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_center_keys<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, masks);
  return e;
}

#define PACT_DISPATCH(bf16, KERNEL, grid, block, st, ...)                                      \
  ((bf16) ? launch_k(KERNEL<__nv_bfloat16>, grid, dim3(block), 0, st, true, __VA_ARGS__)       \
          : launch_k(KERNEL<float>, grid, dim3(block), 0, st, true, __VA_ARGS__))

cudaError_t launch_keynorm_gather(const Batch &bt, int maxN, bool bf16, cudaStream_t st) {
  return PACT_DISPATCH(bf16, k_keynorm_gather, dim3((maxN + 7) / 8, bt.B), 256, st, bt);
}

cudaError_t launch_center_key_gather(const Batch &bt, int maxN, bool bf16, bool all_rows, cudaStream_t st) {
  return PACT_DISPATCH(bf16, k_center_key_gather, dim3((maxN + 7) / 8, bt.B), 256, st, bt, all_rows ? 1 : 0);
}

static int tile_grid(long long tiles, int cap) { return (int)(tiles < 1 ? 1 : (tiles > cap ? cap : tiles)); }

cudaError_t launch_gram(const Batch &bt, int maxN, bool bf16, const DeviceCfg &cfg, cudaStream_t st) {
  const long long nt = (maxN + TS - 1) / TS;
  dim3 grid(tile_grid(nt * (nt + 1) / 2, cfg.sm_count * 5), bt.B);
  return PACT_DISPATCH(bf16, k_gram_f64, grid, kTileThreads, st, bt);
}

cudaError_t launch_centers(const Batch &bt, int maxQ, bool bf16, const DeviceCfg &cfg, int sweep_limit, cudaStream_t st) {
  // maxQ is an estimate of the largest survivor count (ties can exceed it): the masks are sized for every token, densities
  // and adjacency by the estimate, and what does not fit is read from global memory.
  int maxN = 1;
  for (int b = 0; b < bt.B; ++b) maxN = bt.img[b].N > maxN ? bt.img[b].N : maxN;
  const int mask_cap = ((maxN + 31) / 32 + 3) & ~3, ncta = cfg.sm_count / bt.B > 1 ? cfg.sm_count / bt.B : 1;
  const size_t room = (size_t)cfg.centers_smem_max - (size_t)mask_cap * 4;
  const int keys_cap = (size_t)maxQ * 8 + 16 <= room / 2 ? (maxQ + 1) & ~1 : 0;
  size_t adj = (size_t)((maxQ + ncta - 1) / ncta) * ((maxQ + 127) / 128) * 16;
  if (adj > room - (size_t)keys_cap * 8) adj = room - (size_t)keys_cap * 8;
  const size_t smem = (size_t)mask_cap * 4 + (size_t)keys_cap * 8 + adj;
  const cudaError_t e = launch_k(k_centers, dim3(cfg.sm_count > bt.B ? cfg.sm_count : bt.B), dim3(kCenThreads), smem, st, true, bt, mask_cap, keys_cap, (int)adj, sweep_limit);
  if (e != cudaSuccess) return e;
  // a warp for a row (two rows: 1 us more of one image), but no more than four CTAs per SM in all: each reads the masks of
  // its image (with eight: 2 us more of 16 images)
  const int most = 4 * cfg.sm_count / bt.B, want = (maxQ + kCenKeyThreads / 32 - 1) / (kCenKeyThreads / 32), X = want < most ? want : most;
  const dim3 grid(X > 0 ? X : 1, bt.B), block(kCenKeyThreads);
  return bf16 ? launch_k(k_center_keys<__nv_bfloat16>, grid, block, (size_t)mask_cap * 12, st, true, bt, mask_cap)
              : launch_k(k_center_keys<float>, grid, block, (size_t)mask_cap * 12, st, true, bt, mask_cap);
}

cudaError_t launch_assign(const Batch &bt, int maxN, bool bf16, RowMode mode, const DeviceCfg &cfg, cudaStream_t st) {
  const long long nt = (maxN + TS - 1) / TS;
  dim3 grid(tile_grid(nt * nt, cfg.sm_count * 5), bt.B);
  return PACT_DISPATCH(bf16, k_assign_f64, grid, kTileThreads, st, bt, (int)mode);
}

cudaError_t launch_key_rnorm(const Batch &bt, int maxN, bool bf16, cudaStream_t st) {
  dim3 grid((maxN + 7) / 8, bt.B);
  return PACT_DISPATCH(bf16, k_key_rnorm, grid, 256, st, bt);
}

cudaError_t launch_spread(const Batch &bt, int maxN, bool bf16, const DeviceCfg &cfg, cudaStream_t st) {
  const long long nt = (maxN + TS - 1) / TS;
  dim3 grid(tile_grid(nt * (nt + 1) / 2, cfg.sm_count * 5), bt.B);
  return PACT_DISPATCH(bf16, k_spread_f64, grid, kTileThreads, st, bt);
}

cudaError_t launch_spread_finish(const Batch &bt, float *max_dist, int32_t *layer_out, int layer_base, float threshold,
                          cudaStream_t st) {
  return launch_k(k_spread_finish, dim3(1), dim3(32), 0, st, true, bt, max_dist, layer_out, layer_base, threshold);
}

cudaError_t launch_label(const Batch &bt, int maxN, bool bf16, RowMode mode, cudaStream_t st) {
  dim3 grid(tile_grid((maxN + 255) / 256, 1 << 16), bt.B);
  return PACT_DISPATCH(bf16, k_label, grid, 256, st, bt, (int)mode);
}

}  // namespace pact
