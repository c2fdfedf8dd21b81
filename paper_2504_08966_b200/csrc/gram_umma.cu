// tcgen05 tile kernels for bf16 keys (sm_100a): the all-pairs distance pass of DBDPC (Eq. 5) with
// the density (Eq. 6) and the d <= d_c adjacency fused into the epilogue, the rows x centres
// nearest-centre pass (Algorithm 2 assignment, Eq. 8), and the largest distance between two keys of a
// layer (the quantity that decides the reduction layer L) as a max-epilogue over the tiles on and above
// the diagonal.  Nothing of the distance matrix reaches memory: accumulators live in tensor memory
// and are consumed from there.
//
// One persistent CTA per SM, 576 threads:
//   warp 0      TMA producer: 128-byte-swizzled K-slabs of the two operands into a shared-memory ring
//   warp 1      allocates tensor memory, issues tcgen05.mma (128 x BN x 16, bf16 -> fp32)
//   warps 2-17  epilogue: tcgen05.ld of their 32-lane quadrant (four warps per quadrant, a quarter of the
//               columns each), distance arithmetic of common.cuh
// Several accumulators (512 / BN of them share the tensor memory) let the epilogue of tile t overlap
// the MMAs of the next tiles.  The all-pairs pass computes every unordered pair of survivors once: a
// 128 x 128 block above the diagonal serves its rows (density sums, adjacency words) and, through a
// shared-memory exchange of the terms and a warp transpose of the adjacency bits, its columns as well;
// blocks on the diagonal serve their rows only.  Every mbarrier wait is bounded; when one runs out the
// CTA raises the image's status word, drains what it armed, frees its tensor memory and returns.
#include <cuda.h>

#include "kernels.cuh"
#include "labels.cuh"
#include "umma.cuh"

namespace pact {

namespace {

constexpr int BM = 128;           // rows per tile (UMMA M)
constexpr int BK = 64;            // bf16 elements per K-slab = one 128-byte swizzle row
constexpr int A_BYTES = BM * BK * 2;
constexpr int TMEM_COLS = 512;    // all of an SM's tensor memory
constexpr int MAX_STAGES = 6;
constexpr int EPI_WARPS = 16;      // per tensor-memory lane quadrant EPI_WARPS / 4 warps share the columns
                                  // (16 measured 0.35 us per step faster than 8 once a stage held two K-slabs)
constexpr int THREADS = 64 + EPI_WARPS * 32;
constexpr int MAX_ACC = 4;

// Per tile width BN (UMMA N): 256 columns for the rows x centres and the largest-distance passes,
// 128 for the all-pairs pass, whose tiles are the 128 x 128 blocks on and above the diagonal.
template <int BN> struct TileCfg {
  static constexpr int B_BYTES = BN * BK * 2;
  // a stage holds two K-slabs of both operands: half as many barrier waits per tile as with one (measured
  // 0.4 us per step faster at equal bytes in flight)
  static constexpr int SLABS = 2;
  static constexpr int STAGE_BYTES = SLABS * (A_BYTES + B_BYTES);
  static constexpr int STAGES = 2;
  static constexpr int NACC = TMEM_COLS / BN;      // accumulators in tensor memory
  static constexpr int HALF = BN / (EPI_WARPS / 4); // columns per epilogue warp
  // BN = 128 (all-pairs pass): one 32 x 32 exchange buffer per epilogue warp behind the ring
  static constexpr size_t RING = 1024 + (size_t)STAGES * STAGE_BYTES;
  static constexpr size_t SMEM = RING + (BN == 128 ? (size_t)EPI_WARPS * 32 * 36 * 4 : 0);
  // kind::f16 instruction descriptor: fp32 accumulate, bf16 x bf16, both operands K-major.
  static constexpr uint32_t IDESC =
      (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
};

struct TmapSet {
  CUtensorMap a[kMaxBatchPerLaunch];
  CUtensorMap b[kMaxBatchPerLaunch];
};
struct AssignMaps {
  CUtensorMap a[kMaxBatchPerLaunch], b[kMaxBatchPerLaunch];
  CUtensorMap b32[kMaxBatchPerLaunch];             // the centres in boxes of 32 rows
};

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, uint64_t *bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(x), "r"(y) : "memory");
}

struct Shared {
  uint64_t full[MAX_STAGES], empty[MAX_STAGES], acc_full[MAX_ACC], acc_empty[MAX_ACC];
  uint64_t done;                                   // every MMA this CTA has issued is complete
  uint32_t tmem_base;
  int abort;
  __align__(16) float rn_col[EPI_WARPS][128];    // inverse norms of this warp's columns
};

enum { MODE_GRAM = 0, MODE_ASSIGN = 1, MODE_SPREAD = 2 };
// The largest-distance pass runs into the power limit: its warps sleep while they wait.  Ten layers of 7290 keys, awake and asleep: one pass after
// another for 0.3 s 228 and 221 us, for 2 ms 193 and 187, a pass by itself after a pause of 5 ms 209 and 198; three layers 72 and 69, one 32.4 and
// 31.6 by themselves.  The other passes are bound by how soon a wait ends (16 images of 2916 tokens 247 -> 256 us with all waits asleep).
constexpr bool sleeps(int mode) { return mode == MODE_SPREAD; }

// The largest-distance pass needs every unordered pair once: tiles that lie wholly below the diagonal
// are left out (by the producer, the MMA issuer and the epilogue alike).
template <int MODE, int BN> __device__ __forceinline__ bool tile_wanted(int tmi, int tni) {
  return MODE != MODE_SPREAD || (tni + 1) * BN > tmi * BM;
}

// Tile `t` of the pass -> block row and block column.  The all-pairs pass walks the nb (nb + 1) / 2
// blocks with column >= row, row by row; the other passes walk the full grid.
template <int MODE> __device__ __forceinline__ int tile_count(int ntm, int ntn) {
  return MODE == MODE_GRAM ? ntm * (ntm + 1) / 2 : ntm * ntn;
}
template <int MODE> __device__ __forceinline__ void tile_at(int t, int ntm, int ntn, int &tmi, int &tni) {
  if (MODE == MODE_GRAM) {
    // row i starts at i * ntm - i (i - 1) / 2
    const float b = 2.f * (float)ntm + 1.f;
    int i = (int)((b - sqrtf(fmaxf(b * b - 8.f * (float)t, 0.f))) * 0.5f);
    i = max(0, min(i, ntm - 1));
    while (i > 0 && i * ntm - i * (i - 1) / 2 > t) --i;
    while (i + 1 < ntm && (i + 1) * ntm - (i + 1) * i / 2 <= t) ++i;
    tmi = i;
    tni = i + (t - (i * ntm - i * (i - 1) / 2));
  } else if (MODE == MODE_ASSIGN) {
    // full-width column tiles first, the (usually narrow) last column last: the CTAs that take a second
    // tile then take a cheap one
    const int fullc = ntn - 1, nfull = ntm * fullc;
    if (t < nfull) { tmi = t / fullc; tni = t % fullc; }
    else { tmi = t - nfull; tni = fullc; }
  } else {
    tmi = t / ntn;
    tni = t % ntn;
  }
}
// The epilogue of one accumulator tile for one warp: the warp's 32 rows (tensor-memory lanes) of the 128-row
// block tmi against HALF columns from cbase on.  Waits for the accumulator, reads it 32 columns at a time and
// applies the mode's arithmetic; arrive() is called once the accumulator has been read.  skip: the warp only
// waits and releases (a block below the diagonal of the all-pairs pass).  Returns false when the wait ran out.
template <int MODE, int HALF, typename Arrive>
__device__ __forceinline__ bool epi_tile(const ImgDesc &im, int tmi, int cbase, bool skip, int nrows,
                                         int ncols, uint32_t taddr, uint64_t *acc_full, uint32_t parity, float *rn_col,
                                         uint32_t *tr, int lane, int qd, int &band, float &mx, Arrive arrive) {
  // inverse norms of this warp's columns and of this lane's row (in flight while the MMAs run)
  const float *rn_src = MODE == MODE_GRAM ? im.rnk : (MODE == MODE_SPREAD ? im.rn : im.rnc);
  float4 r4;
  {
    const int gj = cbase + lane * 4;
    r4.x = gj + 0 < ncols ? rn_src[gj + 0] : 0.f;
    r4.y = gj + 1 < ncols ? rn_src[gj + 1] : 0.f;
    r4.z = gj + 2 < ncols ? rn_src[gj + 2] : 0.f;
    r4.w = gj + 3 < ncols ? rn_src[gj + 3] : 0.f;
  }
  const int row = tmi * BM + qd * 32 + lane;
  const bool row_ok = row < nrows;
  float rni = row_ok ? (MODE == MODE_GRAM ? im.rnk[row] : im.rn[row]) : 0.f;
  if (MODE == MODE_GRAM) {
    // the all-pairs pass multiplies the two inverse norms first; a vanishing key (inverse norm at
    // its clamp, 1e20) takes 0 here so that the product stays finite: dot product 0, distance 1
    constexpr float kHuge = 1e19f;
    if (rni > kHuge) rni = 0.f;
    if (r4.x > kHuge) r4.x = 0.f;
    if (r4.y > kHuge) r4.y = 0.f;
    if (r4.z > kHuge) r4.z = 0.f;
    if (r4.w > kHuge) r4.w = 0.f;
    r4.x *= -0.5f; r4.y *= -0.5f; r4.z *= -0.5f; r4.w *= -0.5f;   // see gram_chunk
  }
  __syncwarp();
  if (lane * 4 < HALF) reinterpret_cast<float4 *>(rn_col)[lane] = r4;
  __syncwarp();
  if (!mbar_wait_warp<sleeps(MODE)>(acc_full, parity)) return false;
  tc_fence_after();
  unsigned long long rowsum = 0ull;
  float bd = 3.0f, bc = -4.0f;                  // distance to the nearest centre of the tile (<= 2) and its cosine
  int bi = 0;
  const float d_c = im.d_c, neg_k = -im.inv_dn_log2e;
  const int r0 = tmi * BM + qd * 32;
  uint32_t first_bits = 0u;
  const bool above = MODE == MODE_GRAM && cbase / BM > tmi;   // block above the diagonal: rows and columns
#pragma unroll 1
  for (int ch = 0; ch < HALF / 32; ++ch) {
    const int c0 = cbase + ch * 32;
    if (skip || c0 >= ncols) break;              // uniform
    uint32_t v[32];
    tmem_ld32(taddr + ch * 32, v);
    tmem_ld_wait();
    if (MODE == MODE_GRAM) {
      uint32_t bits, colbits = 0u;
      float nearest;
      unsigned long long colsum = 0ull;
      if (above) {
        // every row of this block is a survivor (only the last block row is ragged, and it has no
        // block to its right); each pair (row, column) is also the pair (column, row)
        if (c0 + 32 > ncols)
          gram_chunk<true, true>(v, rn_col + ch * 32, rni, row, c0, ncols, d_c, neg_k, lane, tr, rowsum, bits, nearest, colsum, colbits);
        else
          gram_chunk<false, true>(v, rn_col + ch * 32, rni, row, c0, ncols, d_c, neg_k, lane, tr, rowsum, bits, nearest, colsum, colbits);
        const int gj = c0 + lane;
        if (gj < ncols) {
          atomicAdd(&im.rho_fix[gj], colsum);
          im.adj[(size_t)gj * im.Wp + (r0 >> 5)] = colbits;
        }
      } else {
        const bool edge = (c0 + 32 > ncols) || (c0 < r0 + 32 && c0 + 32 > r0);
        if (edge) gram_chunk<true, false>(v, rn_col + ch * 32, rni, row, c0, ncols, d_c, neg_k, lane, tr, rowsum, bits, nearest, colsum, colbits);
        else gram_chunk<false, false>(v, rn_col + ch * 32, rni, row, c0, ncols, d_c, neg_k, lane, tr, rowsum, bits, nearest, colsum, colbits);
      }
      if (__any_sync(0xffffffffu, nearest <= kNear)) {   // rare
        tmem_ld32(taddr + ch * 32, v);
        tmem_ld_wait();
        band += gram_band(v, rn_col + ch * 32, rni, row, c0, ncols, d_c);
      }
      // Two words of a row in one store, where a warp has them: a sector of the L2 is written once instead of twice.  (Adjacency
      // words are four bytes in a sector each and were 5 us of the 43 over 7290 keys; DBDPC of those 115.1 -> 113.3 us.)
      if constexpr (HALF == 64) {
        if (ch == 0) first_bits = bits;
        if (row_ok) {
          uint32_t *at = im.adj + (size_t)row * im.Wp + (cbase >> 5);
          if (ch == 1) *reinterpret_cast<uint2 *>(at) = make_uint2(first_bits, bits);
          else if (cbase + 32 >= ncols) *at = bits;
        }
      } else if (row_ok) im.adj[(size_t)row * im.Wp + (c0 >> 5)] = bits;
    } else if (MODE == MODE_SPREAD) {
      // The largest distance of the chunk belongs to its smallest cosine: d = clamp(1 - c) does not increase
      // with c, in floating point either, so the products dot * rn_j are compared and one cosine and distance is
      // formed per chunk from the smallest (the row's inverse norm is positive).  Rows and columns past the end hold zero dot products,
      // i.e. distance 1, and the pair (i, i) is not a pair: chunks that hold either take the checked loop.
      constexpr float kNone = 3.0e38f;
      float cmin = kNone;
      const bool plain = c0 + 32 <= ncols && r0 + 32 <= nrows && (c0 + 32 <= r0 || c0 >= r0 + 32);   // uniform
      if (plain) {
#pragma unroll
        for (int k4 = 0; k4 < 32; k4 += 4) {
          const float4 rn4 = *reinterpret_cast<const float4 *>(rn_col + ch * 32 + k4);
          const float rnj[4] = {rn4.x, rn4.y, rn4.z, rn4.w};
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) cmin = fminf(cmin, __uint_as_float(v[k4 + kk]) * rnj[kk]);
        }
      } else {
        const int lim = row_ok ? min(32, ncols - c0) : 0;
        const int self = row - c0;
#pragma unroll
        for (int k4 = 0; k4 < 32; k4 += 4) {
          const float4 rn4 = *reinterpret_cast<const float4 *>(rn_col + ch * 32 + k4);
          const float rnj[4] = {rn4.x, rn4.y, rn4.z, rn4.w};
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            const int k = k4 + kk;
            const float c = __uint_as_float(v[k]) * rnj[kk];
            if (k < lim && k != self) cmin = fminf(cmin, c);
          }
        }
      }
      if (cmin < kNone) mx = fmaxf(mx, fminf(fmaxf(1.0f - cmin * rni, 0.0f), 2.0f));
    } else {
      // the nearest centre of the chunk is the one with the largest cosine (dot * rn_i) * rn_j; the first of
      // equal cosines wins, i.e. the centre with the lowest index; the distance is formed once per tile
      const int lim = min(32, ncols - c0);
#pragma unroll
      for (int k4 = 0; k4 < 32; k4 += 4) {
        const float4 rn4 = *reinterpret_cast<const float4 *>(rn_col + ch * 32 + k4);
        const float rnj[4] = {rn4.x, rn4.y, rn4.z, rn4.w};
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          const int k = k4 + kk;
          const float c = (__uint_as_float(v[k]) * rni) * rnj[kk];
          if (k < lim && c > bc) { bc = c; bi = c0 + k; }
        }
      }
    }
  }
  if (MODE == MODE_ASSIGN && bc > -3.0f) bd = fminf(fmaxf(1.0f - bc, 0.0f), 2.0f);
  // the accumulator may be overwritten once all epilogue warps have read it
  tc_fence_before();
  __syncwarp();
  if (lane == 0) arrive();
  if (row_ok && !skip) {
    if (MODE == MODE_GRAM) atomicAdd(&im.rho_fix[row], rowsum);
    else if (MODE == MODE_ASSIGN && bd <= 2.0f) {
      const unsigned long long pk = ((unsigned long long)__float_as_uint(bd) << 32) | (unsigned)bi;
      atomicMin(&im.best[row], pk);
    }
  }
  return true;
}

}  // namespace

// grid (X, B), 64 + 32 EPI_WARPS threads, dynamic smem = TileCfg<BN>::SMEM.
template <int MODE, int BN>
__global__ void __launch_bounds__(THREADS, 1) k_tiles_umma(const __grid_constant__ Batch bt,
                                                           const __grid_constant__ TmapSet tm) {
  using Cfg = TileCfg<BN>;
  constexpr int STAGES = Cfg::STAGES, NACC = Cfg::NACC, HALF = Cfg::HALF, SLABS = Cfg::SLABS;
  constexpr int STAGE_BYTES = Cfg::STAGE_BYTES, B_BYTES = Cfg::B_BYTES;
  const ImgDesc &im = bt.img[blockIdx.y];
  TL_SCOPE(im, MODE == MODE_GRAM ? 4 : 6);
  extern __shared__ uint8_t smem_raw[];
  __shared__ Shared sh;
  uint8_t *ring = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  // set-up that does not depend on the kernels before this one
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(&sh.full[s], 1); mbar_init(&sh.empty[s], 1); }
    for (int a = 0; a < NACC; ++a) { mbar_init(&sh.acc_full[a], 1); mbar_init(&sh.acc_empty[a], EPI_WARPS); }
    mbar_init(&sh.done, 1);
    sh.abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(&sh.tmem_base, TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = sh.tmem_base;
  pdl_wait();
  pdl_trigger();

  int nrows, ncols;
  if (MODE == MODE_GRAM) { nrows = *im.q_ptr; ncols = nrows; }
  else { nrows = im.N; ncols = im.N; }
  const int ntm = (nrows + BM - 1) / BM, ntn = (ncols + BN - 1) / BN;
  const int ntiles = tile_count<MODE>(ntm, ntn);
  const bool active = (int)blockIdx.x < ntiles;       // CTAs without a tile only give their tensor memory back
  const int nslab = bt.d_k / BK;

  if (!active) {
  } else if (warp == 0) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      const CUtensorMap *ma = &tm.a[blockIdx.y], *mb = &tm.b[blockIdx.y];
      uint32_t it = 0;
      bool ok = true;
      for (int tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x) {
        int tmi, tni;
        tile_at<MODE>(tile, ntm, ntn, tmi, tni);
        if (!tile_wanted<MODE, BN>(tmi, tni)) continue;
        for (int ks = 0; ks < nslab; ks += SLABS, ++it) {
          const int s = it % STAGES;
          const int n = min(SLABS, nslab - ks);
          if (!mbar_wait(&sh.empty[s], ((it / STAGES) & 1) ^ 1)) { ok = false; break; }
          uint8_t *a_dst = ring + (size_t)s * STAGE_BYTES, *b_dst = a_dst + SLABS * A_BYTES;
          mbar_arrive_expect_tx(&sh.full[s], (uint32_t)n * (A_BYTES + B_BYTES));
          for (int h = 0; h < n; ++h) {
            tma_load_2d(a_dst + h * A_BYTES, ma, &sh.full[s], (ks + h) * BK, tmi * BM);
            tma_load_2d(b_dst + h * B_BYTES, mb, &sh.full[s], (ks + h) * BK, tni * BN);
            if (BN == 256) tma_load_2d(b_dst + h * B_BYTES + B_BYTES / 2, mb, &sh.full[s], (ks + h) * BK, tni * BN + BN / 2);
          }
        }
      }
      if (!ok) atomicExch(&sh.abort, 1);
      // drain: every armed stage completes before the CTA may exit (its copies target this smem)
      const uint32_t armed = it < (uint32_t)STAGES ? it : (uint32_t)STAGES;
      for (uint32_t k = 0; k < armed; ++k) {
        const uint32_t j = it - 1 - k;
        mbar_wait(&sh.full[j % STAGES], (j / STAGES) & 1);
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    if (lane == 0) {
      uint32_t it = 0, tcount = 0;
      bool ok = true;
      for (int tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x) {
        int tmi, tni;
        tile_at<MODE>(tile, ntm, ntn, tmi, tni);
        if (!tile_wanted<MODE, BN>(tmi, tni)) continue;
        const uint32_t a = tcount % NACC;
        if (!mbar_wait(&sh.acc_empty[a], ((tcount / NACC) & 1) ^ 1)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + a * BN;
        for (int ks = 0; ks < nslab; ks += SLABS, ++it) {
          const int s = it % STAGES;
          const int n = min(SLABS, nslab - ks);
          if (!mbar_wait(&sh.full[s], (it / STAGES) & 1)) { ok = false; break; }
          tc_fence_after();
          const uint32_t a_addr = smem_u32(ring + (size_t)s * STAGE_BYTES);
          const uint64_t da = smem_desc(a_addr), db = smem_desc(a_addr + SLABS * A_BYTES);
#pragma unroll
          for (int h = 0; h < SLABS; ++h) {
            if (h < n) {
#pragma unroll
              for (int k = 0; k < BK / 16; ++k)
                umma_bf16(d_tmem, desc_at(da, h * A_BYTES + k * 32), desc_at(db, h * B_BYTES + k * 32), Cfg::IDESC, (ks | h | k) != 0);
            }
          }
          umma_commit(&sh.empty[s]);               // frees the slab once these MMAs have read it
        }
        if (ok) umma_commit(&sh.acc_full[a]);      // accumulator complete
        ++tcount;
      }
      // whatever way the loop ended, no MMA may still be running when the tensor memory is given back
      umma_commit(&sh.done);
      if (!mbar_wait(&sh.done, 0)) ok = false;
      if (!ok) atomicExch(&sh.abort, 1);
    }
  } else {
    // ---------------- epilogue ----------------
    const int ew = warp - 2;
    const int qd = warp & 3;                        // tensor-memory lane quadrant this warp may read
    const int half = ew >> 2;                       // which half of the tile's columns
    float *rn_col = sh.rn_col[ew];
    uint32_t *tr = reinterpret_cast<uint32_t *>(ring + Cfg::RING - 1024) + ew * (32 * 36);   // BN = 128 only
    uint32_t tcount = 0;
    int band = 0;
    bool ok = true;
    float mx = 0.f;                                 // largest distance seen by this lane (MODE_SPREAD)
    for (int tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x) {
      int tmi, tni;
      tile_at<MODE>(tile, ntm, ntn, tmi, tni);
      if (!tile_wanted<MODE, BN>(tmi, tni)) continue;
      const uint32_t a = tcount % NACC;
      const int cbase = tni * BN + half * HALF;     // first column of this warp
      const uint32_t taddr = tmem_base + a * BN + half * HALF + ((uint32_t)(qd * 32) << 16);
      ok = epi_tile<MODE, HALF>(im, tmi, cbase, false, nrows, ncols, taddr, &sh.acc_full[a], (tcount / NACC) & 1,
                                rn_col, tr, lane, qd, band, mx, [&]() { mbar_arrive(&sh.acc_empty[a]); });
      if (!ok) break;
      ++tcount;
    }
    if (!ok) atomicExch(&sh.abort, 1);
    if (MODE == MODE_GRAM && band) atomicAdd(&im.cnt[PACT_CNT_BAND_DC], band);
    if (MODE == MODE_SPREAD) {
      // distances are clamped to [0, 2]: their bit patterns order like unsigned integers
      const unsigned w = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));
      if (lane == 0 && w) atomicMax(reinterpret_cast<unsigned *>(&im.cnt[kCntSpread]), w);
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem_base, TMEM_COLS);
  if (threadIdx.x == 0 && sh.abort) atomicMin(&im.cnt[PACT_CNT_STATUS], (int)PACT_ERR_TIMEOUT);
}

// ---- rows x centres on single CTAs ---------------------------------------------------------------------------------
// grid (X, B), 64 + 32 EPI_WARPS threads, one CTA per SM with the roles of k_tiles_umma.  Tiles are 128 rows x W centres.
// kept_rows, bit 0: rows are the gathered survivors (Kp, rnk) instead of all tokens; bit 1: the labels, cluster sizes and
// per-block member counts are formed here as groups of rows finish.
//
// For the stage calls and the whole step of a few images; that of batches and long images takes pairs of CTAs.
// Where the row blocks are few enough that every CTA needs one tile only, the centres are shared out among as many columns of tiles
// as give every CTA one, all of the same width: up to 512 columns, i.e. the whole tensor memory, in two instructions per
// step (DBDPC and merge of 2977 keys 61.5 -> 60.0 us against columns of 256 whatever C is; where some CTAs had a second, narrow tile,
// 7290 rows and 535 centres, the pass ended 1.7 us earlier).  More row blocks: tiles of 256 in rounds, two accumulators, the (usually
// narrow) last column last.  Bound by latency: of 12 us with 7290 rows 2.0 pass until the first operands are there, 3.7 until the last,
// 1.1 until the accumulator is complete, 2.0 in the epilogue, 1.1 for the tickets.
constexpr int kAsnRing = 192 * 1024;                 // (with more of it the next kernels' CTAs find no room beside this one and crowd on a few SMs)
constexpr int kAsnSmem = 1024 + kAsnRing;
constexpr int kAsnMostCols = TMEM_COLS, kAsnLeastCols = 128;   // (with 64 as least, DBDPC and merge of 2977 keys 60.3 us, 59.6 with 128, 61.3 with 256)

// a / b for a below 2^22 and b > 0 (the compiler's division is three times as long, from a cold instruction cache)
__device__ __forceinline__ int div_small(int a, int b) {
  int q = (int)__fdividef((float)a, (float)b);
  q -= q * b > a;
  return q + ((q + 1) * b <= a);
}
struct AsnTiles {
  int ntm, ntn, W, slabs, stages, nacc, stage_bytes;
  __device__ __forceinline__ AsnTiles(int nrows, int C, int ctas) {
    ntm = (nrows + BM - 1) / BM;
    W = 256;
    if (ntm * ((C + kAsnMostCols - 1) / kAsnMostCols) <= ctas && ntm > 0) {
      const int n = min(div_small(ctas, ntm), (C + kAsnLeastCols - 1) / kAsnLeastCols);
      W = n > 0 ? (div_small(C + n - 1, n) + 31) & ~31 : kAsnLeastCols;
    }
    ntn = div_small(C + W - 1, W);
    nacc = W <= 256 ? 2 : 1;
    const int slab = A_BYTES + W * BK * 2;
    slabs = 4 * slab <= kAsnRing ? 2 : 1;              // two K-slabs per stage where two stages fit
    stage_bytes = slabs * slab;
    stages = 4 * stage_bytes <= kAsnRing ? 4 : 3 * stage_bytes <= kAsnRing ? 3 : 2;
  }
  // columns of tile column tni that the MMA has to produce, in steps of 32
  __device__ __forceinline__ int width(int tni, int C) const { return min(W, (C - tni * W + 31) & ~31); }
};

// (80 registers: with 94 no CTA of k_merge finds room beside one of this kernel before it ends, and the calls took 3 to 4 us more)
__global__ void __maxnreg__(80) k_assign(const __grid_constant__ Batch bt, const __grid_constant__ AssignMaps tm, int kept_rows) {
  const ImgDesc &im = bt.img[blockIdx.y];
  TL_SCOPE(im, 6);
  extern __shared__ uint8_t smem_raw[];
  __shared__ Shared sh;
  uint8_t *ring = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < MAX_STAGES; ++s) { mbar_init(&sh.full[s], 1); mbar_init(&sh.empty[s], 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(&sh.acc_full[a], 1); mbar_init(&sh.acc_empty[a], EPI_WARPS); }
    mbar_init(&sh.done, 1);
    sh.abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(&sh.tmem_base, TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = sh.tmem_base;
  pdl_wait();
  pdl_trigger();

  const int nrows = (kept_rows & 1) ? *im.q_ptr : im.N, C = *im.C_ptr;
  const AsnTiles tl(nrows, C, gridDim.x);
  const int ntiles = tl.ntm * tl.ntn, nslab = bt.d_k / BK;
  const bool active = (int)blockIdx.x < ntiles;       // CTAs without a tile only give their tensor memory back

  if (!active) {
  } else if (warp == 0) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      const CUtensorMap *ma = &tm.a[blockIdx.y], *mb = &tm.b[blockIdx.y], *mc = &tm.b32[blockIdx.y];
      uint32_t it = 0;
      int s = 0;
      uint32_t par = 1;
      bool ok = true;
      for (int tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x) {
        int tmi, tni;
        tile_at<MODE_ASSIGN>(tile, tl.ntm, tl.ntn, tmi, tni);
        const int wd = tl.width(tni, C);
        for (int ks = 0; ks < nslab; ks += tl.slabs, ++it) {
          const int n = min(tl.slabs, nslab - ks);
          if (!mbar_wait(&sh.empty[s], par)) { ok = false; break; }
          uint8_t *a_dst = ring + (size_t)s * tl.stage_bytes, *b_dst = a_dst + tl.slabs * A_BYTES;
          mbar_arrive_expect_tx(&sh.full[s], (uint32_t)n * (A_BYTES + wd * BK * 2));
          for (int h = 0; h < n; ++h, b_dst += tl.W * BK * 2) {
            tma_load_2d(a_dst + h * A_BYTES, ma, &sh.full[s], (ks + h) * BK, tmi * BM);
            int r = 0;
            for (; r + BM <= wd; r += BM) tma_load_2d(b_dst + r * BK * 2, mb, &sh.full[s], (ks + h) * BK, tni * tl.W + r);
            for (; r < wd; r += 32) tma_load_2d(b_dst + r * BK * 2, mc, &sh.full[s], (ks + h) * BK, tni * tl.W + r);
          }
          if (++s == tl.stages) { s = 0; par ^= 1; }
        }
      }
      if (!ok) atomicExch(&sh.abort, 1);
      // drain: every armed stage completes before the CTA may exit (its copies target this smem)
      const uint32_t armed = min(it, (uint32_t)tl.stages);
      for (uint32_t k = 0; k < armed; ++k) {
        const uint32_t j = it - 1 - k;
        mbar_wait(&sh.full[j % tl.stages], (j / tl.stages) & 1);
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    if (lane == 0) {
      uint32_t tcount = 0;
      int s = 0;
      uint32_t par = 0;
      bool ok = true;
      for (int tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x, ++tcount) {
        int tmi, tni;
        tile_at<MODE_ASSIGN>(tile, tl.ntm, tl.ntn, tmi, tni);
        const int wd = tl.width(tni, C);
        const uint32_t a = tl.nacc == 2 ? tcount & 1 : 0, ph = tl.nacc == 2 ? tcount >> 1 : tcount;
        if (!mbar_wait(&sh.acc_empty[a], (ph & 1) ^ 1)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + a * 256;
        // kind::f16, fp32 accumulate, bf16 x bf16, both operands K-major, M = 128, N = the first 256 columns and the others
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BM >> 4) << 24);
        const uint32_t first = idesc | ((uint32_t)(min(wd, 256) >> 3) << 17), second = idesc | ((uint32_t)(max(wd - 256, 0) >> 3) << 17);
        for (int ks = 0; ks < nslab; ks += tl.slabs) {
          const int n = min(tl.slabs, nslab - ks);
          if (!mbar_wait(&sh.full[s], par)) { ok = false; break; }
          tc_fence_after();
          const uint32_t a_addr = smem_u32(ring + (size_t)s * tl.stage_bytes);
          const uint64_t da = smem_desc(a_addr), db = smem_desc(a_addr + tl.slabs * A_BYTES);
#pragma unroll
          for (int h = 0; h < 2; ++h)
            if (h < n) {
              const uint64_t ah = desc_at(da, h * A_BYTES), bh = desc_at(db, h * tl.W * BK * 2);
#pragma unroll
              for (int k = 0; k < BK / 16; ++k) umma_bf16(d_tmem, desc_at(ah, k * 32), desc_at(bh, k * 32), first, (ks | h | k) != 0);
              if (wd > 256) {
#pragma unroll
                for (int k = 0; k < BK / 16; ++k) umma_bf16(d_tmem + 256, desc_at(ah, k * 32), desc_at(bh, 256 * BK * 2 + k * 32), second, (ks | h | k) != 0);
              }
            }
          umma_commit(&sh.empty[s]);                 // frees the stage once these MMAs have read it
          if (++s == tl.stages) { s = 0; par ^= 1; }
        }
        if (ok) umma_commit(&sh.acc_full[a]);        // accumulator complete
      }
      // whatever way the loop ended, no MMA may still be running when the tensor memory is given back
      umma_commit(&sh.done);
      if (!mbar_wait(&sh.done, 0)) ok = false;
      if (!ok) atomicExch(&sh.abort, 1);
    }
  } else {
    // ---------------- epilogue ----------------
    const int ew = warp - 2;
    const int qd = warp & 3;                          // tensor-memory lane quadrant this warp may read
    const int part = ew >> 2;                         // which quarter of the tile's columns
    float *rn_col = sh.rn_col[ew];
    uint32_t tcount = 0;
    bool ok = true;
    // Labels: a group of 32 tokens is final once `need` warps (every column tile, every quarter of the columns) have put their
    // nearest centres in place; each warp draws a ticket per group and the one that draws the last labels the group.  The
    // tickets of up to kPend tiles are drawn together, so that a warp waits for its atomics to land once, not once per tile.
    constexpr int kPend = 4;
    const int need = (kept_rows & 2) ? tl.ntn * (EPI_WARPS / 4) : 0;
    int pend_tmi[kPend] = {}, pend_r[kPend] = {}, pend_cid[kPend] = {}, npend = 0;
    unsigned long long seen = 0ull;                   // previous values of the minima this lane has updated
    auto flush_labels = [&]() {
      // Every lane's atomic minima have returned, i.e. are in place, once their return values have been used:
      // the fence then has nothing left to wait for.  (No stored value has distance bits above 2.0f.)
      const unsigned odd = __ballot_sync(0xffffffffu, seen == 0xFFFFFFFE00000001ull);
      seen = 0ull;
      __threadfence();
      int mine = 0;
      if (lane < npend && odd == 0u) {
        int tmi_l = pend_tmi[0];
#pragma unroll
        for (int k = 1; k < kPend; ++k) if (lane == k) tmi_l = pend_tmi[k];
        mine = atomicAdd(&im.rtick[tmi_l * (BM / 32) + qd], 1) == need - 1;
      }
      const unsigned lastmask = __ballot_sync(0xffffffffu, mine);
      if (lastmask) __threadfence();
#pragma unroll
      for (int k = 0; k < kPend; ++k)
        if (k < npend && ((lastmask >> k) & 1u))
          label_group<DistF>(im, pend_tmi[k] * BM + qd * 32 + lane, lane, C, pend_r[k], pend_cid[k]);
      npend = 0;
    };
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
      int tmi, tni;
      tile_at<MODE_ASSIGN>(tile, tl.ntm, tl.ntn, tmi, tni);
      const int wd = tl.width(tni, C);
      const uint32_t a = tl.nacc == 2 ? tcount & 1 : 0, ph = tl.nacc == 2 ? tcount >> 1 : tcount;
      // this warp's columns of the tile
      const int cw = ((wd >> 2) + 15) & ~15, c_lo = tni * tl.W + part * cw, c_hi = min(min(c_lo + cw, tni * tl.W + wd), C);
      const int row = tmi * BM + qd * 32 + lane;
      const bool row_ok = row < nrows;
      // inverse norms of the warp's columns and of the lane's row, and what the labels need besides the nearest centre (known before the pass)
      float4 r4;
      {
        const int gj = c_lo + lane * 4;
        r4.x = gj + 0 < c_hi ? im.rnc[gj + 0] : 0.f;
        r4.y = gj + 1 < c_hi ? im.rnc[gj + 1] : 0.f;
        r4.z = gj + 2 < c_hi ? im.rnc[gj + 2] : 0.f;
        r4.w = gj + 3 < c_hi ? im.rnc[gj + 3] : 0.f;
      }
      const float rni = row_ok ? ((kept_rows & 1) ? im.rnk[row] : im.rn[row]) : 0.f;
      if (need > 0) {
        int r = -1, own = -1;
        if (row_ok) {
          r = im.slot[row];
          if (r >= 0 && ((im.cmask[r >> 5] >> (r & 31)) & 1u)) own = im.cid[r];
        }
        pend_tmi[npend] = tmi; pend_r[npend] = r; pend_cid[npend] = own;
      }
      __syncwarp();
      reinterpret_cast<float4 *>(rn_col)[lane] = r4;
      __syncwarp();
      if (!mbar_wait_warp(&sh.acc_full[a], ph & 1)) { ok = false; break; }
      tc_fence_after();
      // the nearest centre is the one with the largest cosine (dot * rn_i) * rn_j; the first of equal cosines wins, i.e. the
      // centre with the lowest index; the distance is formed once per tile
      float bc = -4.0f;
      int bi = 0;
#pragma unroll 1
      for (int c0 = c_lo; c0 < c_hi; c0 += 32) {
        uint32_t v[32];
        tmem_ld32(tmem_base + a * 256 + (uint32_t)(c0 - tni * tl.W) + ((uint32_t)(qd * 32) << 16), v);
        tmem_ld_wait();
        const int lim = c_hi - c0;
#pragma unroll
        for (int k4 = 0; k4 < 32; k4 += 4) {
          const float4 rn4 = *reinterpret_cast<const float4 *>(rn_col + (c0 - c_lo) + k4);
          const float rnj[4] = {rn4.x, rn4.y, rn4.z, rn4.w};
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            const float c = (__uint_as_float(v[k4 + kk]) * rni) * rnj[kk];
            if (k4 + kk < lim && c > bc) { bc = c; bi = c0 + k4 + kk; }
          }
        }
      }
      // the accumulator may be overwritten once all epilogue warps have read it
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.acc_empty[a]);
      if (row_ok && bc > -3.0f) {
        const float bd = fminf(fmaxf(1.0f - bc, 0.0f), 2.0f);
        const unsigned long long pk = ((unsigned long long)__float_as_uint(bd) << 32) | (unsigned)bi;
        unsigned long long *best = &im.best[(kept_rows & 1) ? im.kept_idx[row] : row];
        if (need > 0) seen |= atomicMin(best, pk);   // the labels wait for the value: the minimum is then in place
        else atomicMin(best, pk);
      }
      ++tcount;
      if (need > 0 && ++npend == kPend) flush_labels();
    }
    if (need > 0 && ok && npend > 0) flush_labels();
    if (!ok) atomicExch(&sh.abort, 1);
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem_base, TMEM_COLS);
  if (threadIdx.x == 0 && sh.abort) atomicMin(&im.cnt[PACT_CNT_STATUS], (int)PACT_ERR_TIMEOUT);
}

// ---- tiles on pairs of CTAs (cta_group::2) ----------------------------------------------------------------------
// Two CTAs of a cluster share one 256 x 256 tile: each holds 128 of its rows (operand A) and 128 of its
// columns (half of operand B), CTA 0 issues tcgen05.mma.cta_group::2 for both, and each CTA finds its
// 128 x 256 part of the product in its own tensor memory.  A CTA therefore fetches half as many operand
// bytes from the L2 per output element as it does alone.  The largest-distance pass always runs this way, the
// all-pairs pass when an SM has six or more 128 x 128 blocks to do and the rows x centres pass of the whole step when it has two
// or more 128-row blocks (with fewer, the coarser tiles cost a round).
//   full[s]      in CTA 0: both CTAs' copies of stage s report their bytes there
//   empty[s]     in each CTA: tcgen05.commit (multicast to both CTAs) once the MMAs have read stage s
//   acc_full[a]  in each CTA: tcgen05.commit (multicast) once accumulator a is complete
//   acc_empty[a] in CTA 0: the epilogue warps of both CTAs arrive there
// Every mbarrier wait is bounded as in the single-CTA kernel.  Without a bound are the cluster barriers (both CTAs of a cluster run at once, and every
// way through the kernel passes all four) and the allocation and deallocation, which are the pair's together: each lies between two cluster barriers,
// so that neither CTA asks before the other one runs and neither leaves, and its SM goes to another stream's kernel, before
// both have their tensor memory back.  The allocation finds it free: no SM has two CTAs with tensor memory (kAloneOnSm).
constexpr int PBN = 256;                              // tile width of the pair kernel
constexpr int PNACC = TMEM_COLS / PBN;
constexpr int PMAX_STAGES = 5;
// EW epilogue warps per CTA (8 or 16).  The all-pairs pass runs with 16: its epilogue is heavy, and its exchange
// buffers (one per epilogue warp) leave room for four stages of one K-slab; the others run with 8 and three
// stages of two K-slabs each: a stage costs a barrier round trip between the two CTAs whatever it holds, and
// with half as many stages per tile the MMA issuer waits half as often.
template <int MODE, int EW> struct PairCfg {
  static constexpr int SLABS = (MODE == MODE_GRAM && EW > 8) ? 1 : 2;   // K-slabs per stage
  static constexpr int STAGES = (MODE == MODE_GRAM && EW > 8) ? 4 : 3;
  static constexpr int STAGE_BYTES = SLABS * 2 * A_BYTES;   // per CTA: SLABS x (128 rows of A, 128 rows of B)
  static constexpr size_t RING = 1024 + (size_t)STAGES * STAGE_BYTES;
  static constexpr size_t SMEM = RING + (MODE == MODE_GRAM ? (size_t)EW * 32 * 36 * 4 : 0);
  static constexpr int THREADS = 64 + EW * 32;
  static constexpr int COLS = PBN / (EW / 4);      // columns of the tile per epilogue warp
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// address of the same shared-memory location in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void mbar_arrive_remote(uint32_t cluster_addr) {
  // relaxed: the warp has nothing to publish through memory, its reads of the accumulator are complete
  // (tcgen05.wait::ld) before the arrive is issued, and a release at cluster scope would cost a memory fence
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_alloc2(uint32_t *slot, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc2(uint32_t addr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols) : "memory");
}
// tiled copy whose bytes are reported to a barrier that may live in the other CTA of the pair (no multicast:
// the data go to this CTA's shared memory only)
__device__ __forceinline__ void tma_load_2d_pair(void *dst, const CUtensorMap *map, uint32_t bar_cluster_addr, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(smem_u32(dst)), "l"(map), "r"(bar_cluster_addr), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void umma_bf16_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum) : "memory");
}
// arrives on the barrier at this shared-memory offset in both CTAs of the pair once the MMAs issued so far are done
__device__ __forceinline__ void umma_commit_pair(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(smem_u32(bar)), "h"((unsigned short)3) : "memory");
}

// A CTA that holds tensor memory must not wait for another one that wants some on its SM, which clusters would: every kernel with tensor memory takes
// more than half of an SM's 228 KB of shared memory, so that there is no other.
static_assert(PairCfg<MODE_GRAM, 16>::SMEM > kAloneOnSm && PairCfg<MODE_ASSIGN, 8>::SMEM > kAloneOnSm && PairCfg<MODE_SPREAD, 8>::SMEM > kAloneOnSm &&
              TileCfg<128>::SMEM > kAloneOnSm && TileCfg<256>::SMEM > kAloneOnSm && kAsnSmem > kAloneOnSm, "one CTA with tensor memory per SM");

template <int EW> struct SharedPair {
  uint64_t full[PMAX_STAGES], empty[PMAX_STAGES], acc_full[PNACC], acc_empty[PNACC];
  uint64_t done;                                   // every MMA of the pair is complete (signalled in both CTAs)
  uint32_t tmem_base;
  int abort;
  __align__(16) float rn_col[EW][128];
};

// grid (2 P) in clusters of two CTAs, 64 + 32 EW threads, dynamic smem = PairCfg<MODE, EW>::SMEM.
// The 256 x 256 tiles of all images (or layers) of the batch form one list, image after image; pair p takes the
// items p, p + P, ... of it, so that the pairs stay equally loaded whatever the number of images.  CTA r of the
// pair owns the 128-row block 2 I + r of tile (I, J).  In the all-pairs and largest-distance passes the tiles
// with J >= I are listed, and of the tile (I, I) the block (2 I + 1, 2 I) lies below the diagonal: computed, not used.
template <int MODE, int EW>
__global__ void __launch_bounds__(PairCfg<MODE, EW>::THREADS, 1) k_tiles_pair(const __grid_constant__ Batch bt,
                                                                              const __grid_constant__ TmapSet tm) {
  using PC = PairCfg<MODE, EW>;
  constexpr int PSTAGES = PC::STAGES, SLABS = PC::SLABS, PSTAGE_BYTES = PC::STAGE_BYTES;
  constexpr size_t PRING = PC::RING;
  constexpr bool ASLEEP = sleeps(MODE);
  constexpr int LIST = MODE == MODE_ASSIGN ? MODE_ASSIGN : MODE_GRAM;   // how the tiles of an image are listed
  TL_SCOPE(bt.img[0], MODE == MODE_GRAM ? 4 : 6);
  extern __shared__ uint8_t smem_raw[];
  __shared__ SharedPair<EW> sh;
  __shared__ int s_first[kMaxBatchPerLaunch + 1], s_rows[kMaxBatchPerLaunch], s_cols[kMaxBatchPerLaunch];
  uint8_t *ring = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const bool leader = rank == 0;

  cluster_arrive();                                   // this CTA runs
  if (threadIdx.x == 0) {
    for (int s = 0; s < PSTAGES; ++s) { mbar_init(&sh.full[s], 1); mbar_init(&sh.empty[s], 1); }
    for (int a = 0; a < PNACC; ++a) { mbar_init(&sh.acc_full[a], 1); mbar_init(&sh.acc_empty[a], 2 * EW); }
    mbar_init(&sh.done, 1);
    sh.abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  // The allocation takes tensor memory of both SMs: it may only be asked for once the other CTA is known to run there.  (Without
  // this barrier, and with an exit that did not wait for the other CTA's deallocation, calls on four streams did not come to an end;
  // within one stream no other kernel with tensor memory is next to this one.)
  cluster_wait();
  if (warp == 1) tmem_alloc2(&sh.tmem_base, TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  cluster_arrive();                                   // this CTA's barriers and tensor memory exist
  tc_fence_after();
  const uint32_t tmem_base = sh.tmem_base;
  pdl_wait();
  pdl_trigger();

  // rows, columns and first list position of every image
  if (threadIdx.x == 0) {
    int first = 0;
    for (int b = 0; b < bt.B; ++b) {
      const ImgDesc &ib = bt.img[b];
      int nr, nc;
      if (MODE == MODE_GRAM) { nr = *ib.q_ptr; nc = nr; }
      else if (MODE == MODE_SPREAD) { nr = ib.N; nc = ib.N; }
      else { nr = ib.N; nc = *ib.C_ptr; }
      s_rows[b] = nr;
      s_cols[b] = nc;
      s_first[b] = first;
      first += tile_count<LIST>((nr + 2 * BM - 1) / (2 * BM), (nc + PBN - 1) / PBN);
    }
    s_first[bt.B] = first;
  }
  __syncthreads();
  cluster_wait();                                     // the other CTA's too: from here on either may signal and write there
  tc_fence_after();
  const int total = s_first[bt.B];
  const int P = gridDim.x >> 1, pr = blockIdx.x >> 1;
  const int nslab = bt.d_k / BK;
  // item -> image b (items only grow, so b only moves forward), tile (I, J), rows and columns of the image
  auto locate = [&](int item, int &b, int &I, int &J, int &nrows, int &ncols) {
    while (item >= s_first[b + 1]) ++b;
    nrows = s_rows[b];
    ncols = s_cols[b];
    tile_at<LIST>(item - s_first[b], (nrows + 2 * BM - 1) / (2 * BM), (ncols + PBN - 1) / PBN, I, J);
  };
  // columns the MMA has to produce: the rows x centres pass stops at the last centre, in steps of 32
  auto width = [&](int J, int ncols) {
    if (MODE != MODE_ASSIGN) return PBN;
    const int left = ncols - J * PBN;
    return left >= PBN ? PBN : ((left + 31) & ~31);
  };

  if (pr >= total) {
  } else if (warp == 0) {
    // ---------------- TMA producer (each CTA for its own shared memory) ----------------
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      int b = 0;
      for (int item = pr; ok && item < total; item += P) {
        int I, J, nrows, ncols;
        locate(item, b, I, J, nrows, ncols);
        const CUtensorMap *ma = &tm.a[b], *mb = &tm.b[b];
        const int bw = width(J, ncols);
        for (int ks = 0; ks < nslab; ks += SLABS, ++it) {
          const int s = it % PSTAGES;
          const int n = min(SLABS, nslab - ks);      // K-slabs of this stage
          if (!mbar_wait<ASLEEP>(&sh.empty[s], ((it / PSTAGES) & 1) ^ 1)) { ok = false; break; }
          uint8_t *a_dst = ring + (size_t)s * PSTAGE_BYTES, *b_dst = a_dst + SLABS * A_BYTES;
          if (leader) mbar_arrive_expect_tx(&sh.full[s], (uint32_t)n * 4u * A_BYTES);   // the bytes of both CTAs
          const uint32_t bar = map_to_rank(smem_u32(&sh.full[s]), 0);
          for (int h = 0; h < n; ++h) {
            tma_load_2d_pair(a_dst + h * A_BYTES, ma, bar, (ks + h) * BK, (2 * I + (int)rank) * BM);
            tma_load_2d_pair(b_dst + h * A_BYTES, mb, bar, (ks + h) * BK, J * PBN + (int)rank * (bw >> 1));
          }
        }
      }
      if (!ok) atomicExch(&sh.abort, 1);
      // drain: the copies of both CTAs into every armed stage complete before either may exit
      const uint32_t armed = leader ? min(it, (uint32_t)PSTAGES) : 0u;
      for (uint32_t k = 0; k < armed; ++k) {
        const uint32_t j = it - 1 - k;
        mbar_wait(&sh.full[j % PSTAGES], (j / PSTAGES) & 1);
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (CTA 0 for both) ----------------
    if (lane == 0 && leader) {
      uint32_t it = 0, tcount = 0;
      bool ok = true;
      int b = 0;
      for (int item = pr; ok && item < total; item += P) {
        int I, J, nrows, ncols;
        locate(item, b, I, J, nrows, ncols);
        const uint32_t a = tcount % PNACC;
        if (!mbar_wait<ASLEEP>(&sh.acc_empty[a], ((tcount / PNACC) & 1) ^ 1)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + a * PBN;
        // kind::f16, fp32 accumulate, bf16 x bf16, both operands K-major, M = 256 over the pair, N = this tile's width
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(width(J, ncols) >> 3) << 17) | ((uint32_t)((2 * BM) >> 4) << 24);
        for (int ks = 0; ks < nslab; ks += SLABS, ++it) {
          const int s = it % PSTAGES;
          const int n = min(SLABS, nslab - ks);
          if (!mbar_wait<ASLEEP>(&sh.full[s], (it / PSTAGES) & 1)) { ok = false; break; }
          tc_fence_after();
          const uint32_t a_addr = smem_u32(ring + (size_t)s * PSTAGE_BYTES);
          const uint64_t da = smem_desc(a_addr), db = smem_desc(a_addr + SLABS * A_BYTES);
#pragma unroll
          for (int h = 0; h < SLABS; ++h) {
            if (h < n) {
#pragma unroll
              for (int k = 0; k < BK / 16; ++k)
                umma_bf16_pair(d_tmem, desc_at(da, h * A_BYTES + k * 32), desc_at(db, h * A_BYTES + k * 32), idesc, (ks | h | k) != 0);
            }
          }
          umma_commit_pair(&sh.empty[s]);          // frees the stage in both CTAs once these MMAs have read it
        }
        if (ok) umma_commit_pair(&sh.acc_full[a]); // accumulator complete, in both CTAs
        ++tcount;
      }
      umma_commit_pair(&sh.done);                  // both CTAs learn that no MMA is running any more
      if (!ok) atomicExch(&sh.abort, 1);
    }
    // whatever way the loop ended, no MMA may still be running when the tensor memory is given back
    if (lane == 0 && !mbar_wait<ASLEEP>(&sh.done, 0)) atomicExch(&sh.abort, 1);
  } else {
    // ---------------- epilogue (each CTA for its 128 rows) ----------------
    const int ew = warp - 2;
    const int qd = warp & 3;                        // tensor-memory lane quadrant this warp may read
    const int half = ew >> 2;                       // which part of the tile's columns
    float *rn_col = sh.rn_col[ew];
    uint32_t *tr = reinterpret_cast<uint32_t *>(ring + PRING - 1024) + ew * (32 * 36);   // all-pairs pass only
    uint32_t tcount = 0;
    bool ok = true;
    float mx = 0.f;                                 // largest distance of the current image (layer)
    int b = 0, b_mx = 0;
    auto flush_mx = [&](int bb) {
      const unsigned w = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));
      if (lane == 0 && w) atomicMax(reinterpret_cast<unsigned *>(&bt.img[bb].cnt[kCntSpread]), w);
      mx = 0.f;
    };
    for (int item = pr; ok && item < total; item += P) {
      int I, J, nrows, ncols;
      locate(item, b, I, J, nrows, ncols);
      if (MODE == MODE_SPREAD && b != b_mx) { flush_mx(b_mx); b_mx = b; }
      const ImgDesc &im = bt.img[b];
      const uint32_t a = tcount % PNACC;
      const int R = 2 * I + (int)rank;              // this CTA's 128-row block
      const int cbase = J * PBN + half * PC::COLS;  // this warp's columns
      const bool skip = MODE != MODE_ASSIGN && cbase / BM < R;   // below the diagonal
      const uint32_t taddr = tmem_base + a * PBN + half * PC::COLS + ((uint32_t)(qd * 32) << 16);
      const uint32_t rel = map_to_rank(smem_u32(&sh.acc_empty[a]), 0);
      int band = 0;
      ok = epi_tile<MODE, PC::COLS>(im, R, cbase, skip, nrows, ncols, taddr, &sh.acc_full[a], (tcount / PNACC) & 1,
                                    rn_col, tr, lane, qd, band, mx, [&]() { mbar_arrive_remote(rel); });
      if (MODE == MODE_GRAM && band) atomicAdd(&im.cnt[PACT_CNT_BAND_DC], band);
      if (!ok) break;
      ++tcount;
    }
    if (!ok) atomicExch(&sh.abort, 1);
    if (MODE == MODE_SPREAD) flush_mx(b_mx);
  }

  tc_fence_before();
  __syncthreads();
  cluster_barrier();                                  // nothing is in flight towards the other CTA any more
  tc_fence_after();
  if (warp == 1) tmem_dealloc2(tmem_base, TMEM_COLS);
  __syncthreads();
  cluster_barrier();                                  // neither SM goes to another kernel's CTA before both have given their tensor memory back
  if (threadIdx.x == 0 && sh.abort)
    for (int b = 0; b < bt.B; ++b) atomicMin(&bt.img[b].cnt[PACT_CNT_STATUS], (int)PACT_ERR_TIMEOUT);
}

// ---- host side -----------------------------------------------------------------------------------

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

bool encode_rows(const DeviceCfg &cfg, CUtensorMap *map, const void *base, long long rows, long long ld_elems, int d_k, int box_rows = BM) {
  const cuuint64_t dims[2] = {(cuuint64_t)d_k, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)ld_elems * 2};
  const cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return reinterpret_cast<EncodeTiledFn>(cfg.encode_tiled)(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

constexpr int kGramBN = 128, kWideBN = 256;

}  // namespace

bool umma_supported(int d_k) { return d_k % BK == 0; }

namespace {
template <int MODE, int EW>
cudaError_t launch_pair(const Batch &bt, const TmapSet &tm, long long tiles, const DeviceCfg &cfg, cudaStream_t st) {
  using PC = PairCfg<MODE, EW>;
  long long P = cfg.sm_count / 2;                     // one pair per two SMs
  if (P > tiles * bt.B) P = tiles * bt.B;
  if (P < 1) P = 1;
  LaunchOpt opt;
  opt.cluster = 2;
  return launch_opt(opt, k_tiles_pair<MODE, EW>, dim3((unsigned)(2 * P)), dim3(PC::THREADS), PC::SMEM, st, bt, tm);
}

// can clusters of two CTAs of this kernel be launched at all?
template <int MODE, int EW> cudaError_t pair_configure(bool &ok) {
  using PC = PairCfg<MODE, EW>;
  ok = false;
  cudaError_t e = cudaFuncSetAttribute(k_tiles_pair<MODE, EW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PC::SMEM);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(2);
  lc.blockDim = dim3(PC::THREADS);
  lc.dynamicSmemBytes = PC::SMEM;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  lc.attrs = attr;
  lc.numAttrs = 1;
  int n = 0;
  e = cudaOccupancyMaxActiveClusters(&n, k_tiles_pair<MODE, EW>, &lc);
  if (e != cudaSuccess || n < 1) (void)cudaGetLastError();
  else ok = true;
  return cudaSuccess;
}
}  // namespace

cudaError_t umma_configure(DeviceCfg *cfg) {
  void *fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres);
  if (e != cudaSuccess) return e;
  if (qres != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
  cfg->encode_tiled = fn;
  e = cudaFuncSetAttribute(k_tiles_umma<MODE_GRAM, kGramBN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)TileCfg<kGramBN>::SMEM);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_tiles_umma<MODE_SPREAD, kWideBN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)TileCfg<kWideBN>::SMEM);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_assign, cudaFuncAttributeMaxDynamicSharedMemorySize, kAsnSmem);
  if (e != cudaSuccess) return e;
  e = pair_configure<MODE_ASSIGN, 8>(cfg->pair_assign);
  if (e != cudaSuccess) return e;
  e = pair_configure<MODE_GRAM, 16>(cfg->pair_gram);
  if (e != cudaSuccess) return e;
  return pair_configure<MODE_SPREAD, 8>(cfg->pair_spread);
}

static int umma_grid_x(long long tiles, int B, int sms) {
  long long x = sms / B;                            // one CTA per SM: all CTAs of the batch run at once
  if (x < 1) x = 1;
  if (x > tiles) x = tiles;
  return (int)(x < 1 ? 1 : x);
}

cudaError_t launch_gram_umma(const Batch &bt, int maxN, const DeviceCfg &cfg, cudaStream_t st, int est_rows) {
  TmapSet tm;
  for (int b = 0; b < bt.B; ++b) {
    const ImgDesc &im = bt.img[b];
    if (!encode_rows(cfg, &tm.a[b], im.Kp, im.Np, bt.d_k, bt.d_k)) return cudaErrorInvalidValue;
    tm.b[b] = tm.a[b];
  }
  // With many blocks per SM (batches, long images) pairs of CTAs on 256 x 256 tiles with 16 epilogue warps each are
  // faster: half the operand bytes per pair of blocks and a shorter epilogue.  With few (three per SM on one
  // 7290-token image) the coarser tiles cost a round, and single CTAs on 128 x 128 blocks are.
  if (est_rows < 1 || est_rows > maxN) est_rows = maxN;
  const long long nq = (est_rows + BM - 1) / BM;
  if (cfg.pair_gram && nq * (nq + 1) / 2 * bt.B >= 6LL * cfg.sm_count) {
    const long long n2 = (maxN + 2 * BM - 1) / (2 * BM);
    return launch_pair<MODE_GRAM, 16>(bt, tm, n2 * (n2 + 1) / 2, cfg, st);
  }
  const long long nb = (maxN + BM - 1) / BM;
  dim3 grid(umma_grid_x(nb * (nb + 1) / 2, bt.B, cfg.sm_count), bt.B);
  return launch_k(k_tiles_umma<MODE_GRAM, kGramBN>, grid, dim3(THREADS), TileCfg<kGramBN>::SMEM, st, true, bt, tm);
}

bool umma_pairs_for_assign(int maxN, int B, const DeviceCfg &cfg) {
  // With two or more 128-row blocks per SM (batches, long images) pairs of CTAs on 256 x 256 tiles are faster: a pair fetches two thirds
  // of the operand bytes.  (From 1025 tokens on a call by itself is faster with them too, one image of 7290 tokens by 2 us; but four such
  // calls on four streams did not come to an end while a pair asked for tensor memory before both of its CTAs ran and left one by one.)
  return cfg.pair_assign && (long long)((maxN + BM - 1) / BM) * B >= 2LL * cfg.sm_count;
}

// labels: the single-CTA kernel also forms labels and member counts (all-token rows only); pairs: the pair kernel
// (all-token rows, no labels)
cudaError_t launch_assign_umma(const Batch &bt, int maxN, bool kept_rows, const DeviceCfg &cfg, cudaStream_t st, bool labels,
                               bool pairs) {
  const auto rows_map = [&](const ImgDesc &im, CUtensorMap *m) {
    return kept_rows ? encode_rows(cfg, m, im.Kp, im.Np, bt.d_k, bt.d_k) : encode_rows(cfg, m, im.Kc, im.N, im.ldKc, bt.d_k);
  };
  if (pairs && !kept_rows && cfg.pair_assign) {
    TmapSet tm;
    for (int b = 0; b < bt.B; ++b)
      if (!rows_map(bt.img[b], &tm.a[b]) || !encode_rows(cfg, &tm.b[b], bt.img[b].Kcen, bt.img[b].Np, bt.d_k, bt.d_k)) return cudaErrorInvalidValue;
    const long long pt = (long long)((maxN + 2 * BM - 1) / (2 * BM)) * ((maxN + PBN - 1) / PBN);
    return launch_pair<MODE_ASSIGN, 8>(bt, tm, pt, cfg, st);
  }
  AssignMaps tm;
  for (int b = 0; b < bt.B; ++b) {
    const ImgDesc &im = bt.img[b];
    if (!rows_map(im, &tm.a[b]) || !encode_rows(cfg, &tm.b[b], im.Kcen, im.Np, bt.d_k, bt.d_k) ||
        !encode_rows(cfg, &tm.b32[b], im.Kcen, im.Np, bt.d_k, bt.d_k, 32))
      return cudaErrorInvalidValue;
  }
  const long long tiles = (long long)((maxN + BM - 1) / BM) * ((maxN + kAsnLeastCols - 1) / kAsnLeastCols);
  dim3 grid(umma_grid_x(tiles, bt.B, cfg.sm_count), bt.B);
  return launch_k(k_assign, grid, dim3(THREADS), kAsnSmem, st, true, bt, tm, (kept_rows ? 1 : 0) | (labels && !kept_rows ? 2 : 0));
}

// every layer of the batch is one "image": rows and columns are all N keys of K_clu
cudaError_t launch_spread_umma(const Batch &bt, int maxN, const DeviceCfg &cfg, cudaStream_t st) {
  TmapSet tm;
  for (int b = 0; b < bt.B; ++b) {
    const ImgDesc &im = bt.img[b];
    if (!encode_rows(cfg, &tm.a[b], im.Kc, im.N, im.ldKc, bt.d_k)) return cudaErrorInvalidValue;
    tm.b[b] = tm.a[b];
  }
  if (cfg.pair_spread) {
    const long long ptiles = (long long)((maxN + 2 * BM - 1) / (2 * BM)) * ((maxN + PBN - 1) / PBN);
    return launch_pair<MODE_SPREAD, 8>(bt, tm, ptiles, cfg, st);
  }
  const long long tiles = (long long)((maxN + BM - 1) / BM) * ((maxN + kWideBN - 1) / kWideBN);
  dim3 grid(umma_grid_x(tiles, bt.B, cfg.sm_count), bt.B);
  return launch_k(k_tiles_umma<MODE_SPREAD, kWideBN>, grid, dim3(THREADS), TileCfg<kWideBN>::SMEM, st, true, bt, tm);
}

}  // namespace pact
