// The middle of the step for small images in one kernel: scores, split, DBDPC, reincorporation and member lists by one
// thread-block cluster per image, between k_tokens and k_merge.
//
// A small image leaves the chain of kernels bound by latency: with 729 tokens the seven kernels from the scores to the
// member lists took 40 us, 4 to 10 us each, almost all of it launches, the first reads of what the kernel before left
// in the L2, and cold instructions.  Here the 16 CTAs of a cluster own a slice of the tokens each, hand keys, flags and
// labels to one another by stores into each other's shared memory, and meet at cluster barriers of about a third of a
// microsecond instead of at kernel boundaries.  Only densities, adjacency bits and nearest centres, which tiles of
// different CTAs contribute to, go through global memory (the L2).  The two passes over the hidden states before and
// after stay kernels of the whole GPU: 16 SMs take in 2 TB/s.  The arithmetic of every stage is that of the wide kernels
// (euti.cu, gram_umma.cu, cluster.cu, merge.cu).  Much of the code runs once per launch, from a cold instruction
// cache, so loops are kept rolled where the wide kernels unroll them.
//
//   1  scores and sort keys of the own tokens, to all                    | barrier
//   2  keep flags of the own tokens by counting keys, to all             | barrier
//   3  survivor list; tiles of the all-pairs pass                        | barrier
//   4  centres (every CTA resolves them itself); tiles of rows x centres | barrier
//   5  labels of the own tokens, to all                                  | barrier
//   6  cluster sizes (every CTA itself), records of the own tokens
#include "f64_tiles.cuh"
#include "kernels.cuh"
#include "umma.cuh"

namespace pact {

namespace {

constexpr int kSmThreads = 512;
constexpr int kSmWarps = kSmThreads / 32;
constexpr int CL = 16;                                 // CTAs of a cluster
constexpr int kSmMaxW = kSmallMaxN / 32;
constexpr int kSmMaxHeads = 32;
constexpr int kSmallMaxF64 = 672;                      // most tokens without the tensor cores (see small_fits)

// tcgen05 tiles: 128 rows against 64 others, or 128 rows against themselves, 512 key elements at a time: a chunk of
// both operands is resident at once, so that a tile of keys of up to that width waits for memory and for the tensor
// core once each (as a ring of 128-element stages it was four trips of a microsecond).
constexpr int kSmBM = 128, kSmBN = 64, kSmBK = 64, kSmSlabs = 8;
constexpr int kSmABytes = kSmBM * kSmBK * 2, kSmBBytes = kSmBN * kSmBK * 2;
constexpr int kSmTileBytes = kSmSlabs * (kSmABytes + kSmBBytes);
// double-precision tiles: four groups of 128 threads with a tile each
constexpr size_t kSmDynUmma = 1024 + kSmTileBytes;
constexpr size_t kSmDynF64 = 1024 + 186 * 1024;
struct F64Group {
  double As[TS][KST], Bs[TS][KST];
  F64Sums sums;
  unsigned long long rowbest[2][TS];
};

template <typename T> struct SmallShared {
  using rn_t = typename DistOf<T>::type::rn_t;
  __align__(16) uint32_t key[kSmallMaxN];              // sort keys of all tokens
  rn_t rn[kSmallMaxN];                                 // inverse norms of all clustering keys
  float rn_col[kSmWarps][32];
  short lab[kSmallMaxN];                               // labels of all tokens
  short own_cid[kSmallMaxN];                           // cluster id of a token that is a centre, else -1
  unsigned short kept[kSmallMaxN];                     // token of survivor r
  unsigned short cen[kSmallMaxN];                      // token of centre c
  int off[kSmallMaxN + 1], size[kSmallMaxN];           // first member and number of members of a cluster
  unsigned char keep8[kSmallMaxN];
  __align__(16) uint32_t cm[kSmMaxW], rm[kSmMaxW];                   // centres, removed
  int pref[kSmMaxW];
  int wsum[kSmWarps];
  int C;
  uint64_t acc_bar;
  uint64_t done;                                       // after a wait that ran out: every MMA this CTA has issued is complete
  uint32_t tmem_base;
  int abort;
};

// stores to this shared-memory location of CTA `rank` of the cluster
__device__ __forceinline__ uint32_t at_rank(const void *p, int rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void put(uint32_t *p, int rank, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(at_rank(p, rank)), "r"(v) : "memory");
}
__device__ __forceinline__ void put(short *p, int rank, short v) {
  asm volatile("st.shared::cluster.u16 [%0], %1;" ::"r"(at_rank(p, rank)), "h"(v) : "memory");
}
__device__ __forceinline__ void put(unsigned char *p, int rank, unsigned char v) {
  asm volatile("st.shared::cluster.u8 [%0], %1;" ::"r"(at_rank(p, rank)), "r"((uint32_t)v) : "memory");
}

__device__ __forceinline__ uint4 ld_volatile_smem4(const uint32_t *p) {
  uint4 v;
  asm volatile("ld.volatile.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(smem_u32(p)) : "memory");
  return v;
}
__device__ __forceinline__ int pow2_ceil(int x) { return x <= 1 ? 1 : 1 << (32 - __clz(x - 1)); }

// One tile of dot products on the tensor core, rows of both operands gathered from K by token (a negative token gives
// a row of zeros).  tokA: tokens of the rows t / 8 and t / 8 + 64 that this thread copies, tokB: token of row t / 8 of
// the other operand (nB rows); same: the 128 rows against themselves.  The accumulator (tensor-memory columns 0 ..)
// is complete when the calling warp gets true; false: the wait for it ran out.  The CTA then goes on through its few tiles
// (every wait is bounded, and the status word says that the results are not valid, whatever operands an MMA still read) and
// finish_mmas() comes before it gives its tensor memory back.  (To leave the loops together takes an or-barrier or a flag per tile, 0.6 to 0.9 us
// of an image of 729 tokens.)
template <typename Sh>
__device__ __forceinline__ bool small_tile(Sh &sh, uint8_t *buf, uint32_t &phase, const __nv_bfloat16 *K, long long ldK, int d_k,
                                           const int (&tokA)[2], int tokB, int nB, bool same) {
  const int t = threadIdx.x, piece = t & 7, row0 = t >> 3;
  const uint32_t a0 = smem_u32(buf), b0 = same ? a0 : a0 + kSmSlabs * kSmABytes;
  const uint32_t at = row0 * 128 + ((piece ^ (row0 & 7)) << 4);          // 128-byte swizzle (rows + 64: the same)
  const __nv_bfloat16 *srcA0 = K + (long long)max(tokA[0], 0) * ldK + piece * 8, *srcA1 = K + (long long)max(tokA[1], 0) * ldK + piece * 8;
  const __nv_bfloat16 *srcB = K + (long long)max(tokB, 0) * ldK + piece * 8;
  bool ok = true;
  for (int k0 = 0; k0 < d_k; k0 += kSmSlabs * kSmBK) {
    const int n = min(kSmSlabs, (d_k - k0) / kSmBK);
    // (through registers: twice the rate of 16-byte asynchronous copies, see bulk_load in tma.cuh)
    constexpr int UH = 4;
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 1
    for (int h0 = 0; h0 < n; h0 += UH) {
      uint4 x[UH], y[UH], b[UH];
#pragma unroll
      for (int u = 0; u < UH; ++u) {
        const int o = k0 + (h0 + u) * kSmBK;
        const bool in = h0 + u < n;
        x[u] = in && tokA[0] >= 0 ? __ldg(reinterpret_cast<const uint4 *>(srcA0 + o)) : z;
        y[u] = in && tokA[1] >= 0 ? __ldg(reinterpret_cast<const uint4 *>(srcA1 + o)) : z;
        b[u] = in && !same && tokB >= 0 ? __ldg(reinterpret_cast<const uint4 *>(srcB + o)) : z;
      }
#pragma unroll
      for (int u = 0; u < UH; ++u)
        if (h0 + u < n) {
          *reinterpret_cast<uint4 *>(buf + (h0 + u) * kSmABytes + at) = x[u];
          *reinterpret_cast<uint4 *>(buf + (h0 + u) * kSmABytes + at + 64 * 128) = y[u];
          if (!same && row0 < nB) *reinterpret_cast<uint4 *>(buf + kSmSlabs * kSmABytes + (h0 + u) * kSmBBytes + at) = b[u];
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (t == 0) {
      tc_fence_after();
      const int N = same ? kSmBM : nB;
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(kSmBM >> 4) << 24);
      const int bstep = same ? kSmABytes : kSmBBytes;
#pragma unroll 1
      for (int h = 0; h < n; ++h)
#pragma unroll
        for (int k = 0; k < kSmBK / 16; ++k)
          umma_bf16(sh.tmem_base, smem_desc(a0 + h * kSmABytes + k * 32), smem_desc(b0 + h * bstep + k * 32), idesc, (k0 | h | k) != 0);
      umma_commit(&sh.acc_bar);
    }
    ok = mbar_wait_warp(&sh.acc_bar, phase);
    if (!ok) sh.abort = 1;
    phase ^= 1;
  }
  tc_fence_after();
  return ok;
}

// No MMA may still be running when the tensor memory is given back.  (A call: code that hardly ever runs costs its place in
// the instruction stream, 0.5 us of an image of 729 tokens.)
__device__ __noinline__ void finish_mmas(uint64_t *done) {
  umma_commit(done);
  mbar_wait(done, 0);
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr) : "memory");
}
// 32 columns of one row (= lane) of the all-pairs pass: the arithmetic of gram_chunk (umma.cuh) eight columns at a time,
// one copy of the code for all kinds of blocks.  colsum and colbits are those of column c0 + lane.
__device__ __forceinline__ void small_gram_chunk(uint32_t taddr, const float *rn_col, float rni, int row, int c0, int ncols, float d_c,
                                                 float neg_k, int lane, uint32_t *tr, unsigned long long &rowsum, uint32_t &bits,
                                                 int &band, unsigned long long &colsum, uint32_t &colbits) {
  unsigned long long s = 0ull;
  uint32_t b = 0u;
#pragma unroll 1
  for (int k8 = 0; k8 < 32; k8 += 8) {
    uint32_t v[8];
    tmem_ld8(taddr + k8, v);
    tmem_ld_wait();
    uint32_t b8 = 0u;
#pragma unroll
    for (int kk = 0; kk < 8; ++kk) {
      const int gj = c0 + k8 + kk;
      float dd = fminf(fmaxf(1.0f - __uint_as_float(v[kk]) * (rni * rn_col[k8 + kk]), 0.0f), 2.0f);
      if (gj == row) dd = 0.f;
      const bool ok = gj < ncols;
      const uint32_t term = ok ? __float2uint_rn(ex2_approx(dd * neg_k) * (float)(1u << kRhoShift)) : 0u;
      s += term;
      if (ok && dd <= d_c) b8 |= 1u << kk;
      if (ok && row < gj && fabsf(dd - d_c) <= 1e-6f) ++band;
      tr[(k8 + kk) * 36 + lane] = row < ncols ? term : 0u;
    }
    b |= b8 << k8;
  }
  rowsum = s;
  bits = b;
  __syncwarp();
  unsigned long long cs = 0ull;
  const uint4 *src = reinterpret_cast<const uint4 *>(tr + lane * 36);
#pragma unroll 2
  for (int j = 0; j < 8; ++j) {
    const uint4 x = src[j];
    cs += ((unsigned long long)x.x + x.y) + ((unsigned long long)x.z + x.w);
  }
  colsum = cs;
  uint32_t w = row < ncols ? b : 0u;
#pragma unroll
  for (int sft = 16; sft >= 1; sft >>= 1) {            // transpose of the 32 x 32 bits
    const uint32_t m = sft == 16 ? 0x0000FFFFu : sft == 8 ? 0x00FF00FFu : sft == 4 ? 0x0F0F0F0Fu : sft == 2 ? 0x33333333u : 0x55555555u;
    const uint32_t y = __shfl_xor_sync(0xffffffffu, w, sft);
    w = (lane & sft) ? ((w & ~m) | ((y >> sft) & m)) : ((w & m) | ((y << sft) & ~m));
  }
  colbits = w;
  __syncwarp();
}

// tile `t` of the nt (nt + 1) / 2 tiles on and above the diagonal (a few rows of tiles: no root needed)
__device__ __forceinline__ void upper_tile_scan(int t, int nt, int &tm, int &tn) {
  int i = 0;
  while (t >= nt - i) { t -= nt - i; ++i; }
  tm = i;
  tn = i + t;
}

__device__ __forceinline__ void group_sync(int g) { asm volatile("bar.sync %0, 128;" ::"r"(1 + g) : "memory"); }

}  // namespace

// grid (CL, B) in clusters of CL CTAs, 512 threads, dynamic smem = kSmDynUmma or kSmDynF64.
template <typename T, bool UMMA>
__global__ void __launch_bounds__(kSmThreads, 1) k_small(const __grid_constant__ Batch bt, int rpp, int sweep_limit) {
  using D = typename DistOf<T>::type;
  using rn_t = typename D::rn_t;
  const ImgDesc &im = bt.img[blockIdx.y];
  TL_SCOPE(im, 2);
  extern __shared__ uint8_t smem_raw[];
  __shared__ SmallShared<T> sh;
  uint8_t *dyn = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int t = threadIdx.x, lane = t & 31, w = t >> 5, rank = blockIdx.x;
  const int N = im.N, n_qh = bt.n_qh;
  const int R = (N + CL - 1) / CL, own0 = min(N, rank * R), nown = min(N, own0 + R) - own0;
  if constexpr (UMMA) { if (w == 0) tmem_alloc(&sh.tmem_base, 128); }
  if (t == 0) {
    mbar_init(&sh.acc_bar, 1);
    mbar_init(&sh.done, 1);
    sh.abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (UMMA) tc_fence_before();
  __syncthreads();
  if (UMMA) tc_fence_after();
  cluster_arrive();                                    // (every CTA of the cluster runs before one stores to another)
  pdl_wait();
  pdl_trigger();

  // ---- 1: scores and sort keys of the own tokens (see k_scores) ---------------------------------------------------------
  // G softmax pieces: a warp per head merges them, lane = piece
  constexpr int PL = kSmallMaxN / kMinPiece / 32;                // pieces per lane
  const int G = (N + rpp - 1) / rpp;
  double *s_fac = reinterpret_cast<double *>(dyn);               // [n_qh][G] what turns a term of piece g into a share
  double e_own[4], nrm_own = 0.0;
  if (t < nown) {                                                // on their way while the pieces are merged
    nrm_own = im.nrm[own0 + t];
#pragma unroll
    for (int j = 0; j < 4; ++j) e_own[j] = j < n_qh ? im.E[(size_t)j * N + own0 + t] : 0.0;
  }
  for (int i = t; i < N; i += kSmThreads) sh.rn[i] = rn_tok<D>(im)[i];
  for (int j = w; j < n_qh; j += kSmWarps) {
    double m[PL], z[PL], M = -1.0e300, Z = 0.0;
#pragma unroll
    for (int k = 0; k < PL; ++k) {
      const int g = lane + 32 * k;
      m[k] = g < G ? *piece_at(im, j, g) : -1.0e300;
      z[k] = g < G ? piece_at(im, j, g)[1] : 0.0;
    }
#pragma unroll
    for (int k = 0; k < PL; ++k) M = m[k] > M ? m[k] : M;
    M = warp_max(M);
#pragma unroll
    for (int k = 0; k < PL; ++k)
      if (32 * k < G) {
        m[k] = exp(m[k] - M);
        Z += z[k] * m[k];
      }
    Z = warp_sum(Z);
    const double inv = 1.0 / (Z * (double)n_qh);
#pragma unroll
    for (int k = 0; k < PL; ++k)
      if (lane + 32 * k < G) s_fac[j * G + lane + 32 * k] = m[k] * inv;
  }
  __syncthreads();
  if (t < nown) {
    const int g = (own0 + t) / rpp;
    double s = 0.0;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j < n_qh) s = fma(e_own[j], s_fac[j * G + g], s);
    for (int j = 4; j < n_qh; ++j) s = fma(im.E[(size_t)j * N + own0 + t], s_fac[j * G + g], s);
    const float sf = (float)(s * nrm_own);
    if (im.score_user) im.score_user[own0 + t] = sf;
    sh.key[own0 + t] = score_key(sf);
  }
  __syncthreads();
  cluster_wait();
  for (int e = t; e < nown * CL; e += kSmThreads) {
    const int dst = e / nown, i = own0 + (e - dst * nown);
    if (dst != rank) put(&sh.key[i], dst, sh.key[i]);
  }
  cluster_sync();
  TL_POINT(im, 4);

  // ---- 2: a token survives iff more than m tokens have a score no larger than its own (tau is the (m + 1)-th smallest) --
  {
    const int tpt = min(32, kSmThreads / pow2_ceil(max(1, R)));   // threads per token
    const int li = t / tpt, part = t % tpt;
    const uint32_t mine = li < nown ? sh.key[own0 + li] : 0u;
    int cnt = 0;
    const uint4 *k4 = reinterpret_cast<const uint4 *>(sh.key);
#pragma unroll 2
    for (int j = part; j < N >> 2; j += tpt) {
      const uint4 k = k4[j];
      cnt += (k.x <= mine) + (k.y <= mine) + (k.z <= mine) + (k.w <= mine);
    }
    if (part < (N & 3)) cnt += sh.key[(N & ~3) + part] <= mine;   // (at least eight threads per token)
    for (int o = tpt >> 1; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    if (li < nown) {
      const unsigned char kp = cnt > im.m_target;
      if (part == 0 && im.keep_user) im.keep_user[own0 + li] = kp;
      for (int u = part; u < CL; u += tpt) put(&sh.keep8[own0 + li], u, kp);
    }
  }
  cluster_sync();
  TL_POINT(im, 5);

  // ---- 3: survivor list ---------------------------------------------------------------------------------------------
  int q = 0;
  for (int base = 0; base < N; base += kSmThreads) {
    const int i = base + t;
    const bool kp = i < N && sh.keep8[i];
    const unsigned bal = __ballot_sync(0xffffffffu, kp);
    if (lane == 0) sh.wsum[w] = __popc(bal);
    __syncthreads();
    int pos = q + __popc(bal & ((1u << lane) - 1u)), tot = 0;
#pragma unroll
    for (int k = 0; k < kSmWarps; ++k) { if (k < w) pos += sh.wsum[k]; tot += sh.wsum[k]; }
    if (kp) sh.kept[pos] = (unsigned short)i;
    if (i < N) sh.own_cid[i] = -1;
    q += tot;
    __syncthreads();
  }
  // ---- all pairs of survivors (Eq. 5-6) -------------------------------------------------------------------------------
  const T *Kc = reinterpret_cast<const T *>(im.Kc);
  const int nw = (q + 31) >> 5;
  uint32_t phase = 0;
  int band = 0;
  if constexpr (UMMA) {
    // units: the blocks of 128 rows against themselves, then every block against the 64-row halves of those after it
    const int nb = (q + kSmBM - 1) / kSmBM;
    for (int unit = rank; unit < nb * nb; unit += CL) {
      int tm = unit, c00 = unit * kSmBM;
      const bool diag = unit < nb;
      if (!diag) {
        int tn;
        upper_tile_scan((unit - nb) >> 1, nb - 1, tm, tn);
        c00 = (tn + 1) * kSmBM + ((unit - nb) & 1) * kSmBN;
      }
      if (c00 >= q) continue;                          // the same for the whole CTA
      int tokA[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int ra = tm * kSmBM + (t >> 3) + 64 * k;
        tokA[k] = ra < q ? sh.kept[ra] : -1;
      }
      const int rb = c00 + (t >> 3);
      const bool ok = small_tile(sh, dyn, phase, Kc, im.ldKc, bt.d_k, tokA, rb < q ? (int)sh.kept[rb] : -1, kSmBN, diag);
      const int qd = w & 3, k0 = (w >> 2) * 32, c0 = c00 + k0, r0 = tm * kSmBM + qd * 32, row = r0 + lane;
      if (ok && c0 < q && (diag || k0 < kSmBN)) {
        constexpr float kHuge = 1e19f;                 // a vanishing key: see epi_tile
        float rnj = c0 + lane < q ? (float)sh.rn[sh.kept[c0 + lane]] : 0.f, rni = row < q ? (float)sh.rn[sh.kept[row]] : 0.f;
        if (rnj > kHuge) rnj = 0.f;
        if (rni > kHuge) rni = 0.f;
        sh.rn_col[w][lane] = rnj;
        __syncwarp();
        uint32_t *tr = reinterpret_cast<uint32_t *>(dyn) + w * (32 * 36);
        unsigned long long rowsum, colsum;
        uint32_t bits, colbits;
        small_gram_chunk(sh.tmem_base + k0 + ((uint32_t)(qd * 32) << 16), sh.rn_col[w], rni, row, c0, q, im.d_c, -im.inv_dn_log2e, lane, tr,
                         rowsum, bits, band, colsum, colbits);
        if (!diag && c0 + lane < q) {
          atomicAdd(&im.rho_fix[c0 + lane], colsum);
          im.adj[(size_t)(c0 + lane) * im.Wp + (r0 >> 5)] = colbits;
        }
        if (row < q) {
          atomicAdd(&im.rho_fix[row], rowsum);
          im.adj[(size_t)row * im.Wp + (c0 >> 5)] = bits;
        }
      }
      tc_fence_before();
      __syncthreads();                                 // the operands and the accumulator may be used again
    }
  } else {
    const int g = t >> 7, tg = t & 127, nt = (q + TS - 1) / TS;
    F64Group &fg = reinterpret_cast<F64Group *>(dyn)[g];
    for (int tile = g * CL + rank; tile < nt * (nt + 1) / 2; tile += 4 * CL) {
      int tm, tn;
      upper_tile_scan(tile, nt, tm, tn);
      double acc[2][2][2];
      tile_dots<T>(
          tg, [&](int r) { const int x = tm * TS + r; return x < q ? Kc + (size_t)sh.kept[x] * im.ldKc : (const T *)nullptr; },
          [&](int r) { const int x = tn * TS + r; return x < q ? Kc + (size_t)sh.kept[x] * im.ldKc : (const T *)nullptr; },
          bt.d_k, fg.As, fg.Bs, acc, [&]() { group_sync(g); });
      gram_epilogue_f64<D>(tg, tm, tn, q, acc, [&](int x) { return (double)sh.rn[sh.kept[x]]; }, im, fg.sums, band, [&]() { group_sync(g); });
    }
  }
  band = __reduce_add_sync(0xffffffffu, band);
  if (lane == 0 && band) atomicAdd(&im.cnt[PACT_CNT_BAND_DC], band);
  cluster_sync();
  TL_POINT(im, 6);

  // ---- 4: centres, resolved from shared memory by every CTA for itself -------------------------------------------------
  // A row is removed once a neighbour is a centre (an undecided row's neighbour that is a centre comes before it: had
  // the row come first, the neighbour could not have become one) and becomes a centre once no undecided neighbour
  // comes before it in density order.  Both facts are final, so any order of looking gives Algorithm 2's result.
  // Rows of adjacency words are a whole odd number of 16-byte pieces long: eight rows read by a quarter warp meet no bank
  // twice.
  uint4 *s_adj = reinterpret_cast<uint4 *>(dyn);                             // [q][ns]
  const int nw4 = (nw + 3) >> 2, ns = nw4 | 1;
  unsigned long long *s_rho = reinterpret_cast<unsigned long long *>(s_adj + q * ns);   // [q]
  {
    constexpr int UL = 4;
    const int last = nw - (nw4 - 1) * 4;               // words in the last piece of a row
#pragma unroll 1
    for (int e0 = t; e0 < q * nw4; e0 += kSmThreads * UL) {
      uint4 x[UL];
#pragma unroll
      for (int u = 0; u < UL; ++u) {
        const int e = e0 + u * kSmThreads, r = e / nw4;
        if (e < q * nw4) x[u] = __ldcg(reinterpret_cast<const uint4 *>(im.adj + (size_t)r * im.Wp) + (e - r * nw4));
      }
#pragma unroll
      for (int u = 0; u < UL; ++u) {
        const int e = e0 + u * kSmThreads, r = e / nw4, k = e - r * nw4;
        if (k == nw4 - 1) {                            // words past the last survivor were never written
          if (last < 2) x[u].y = 0u;
          if (last < 3) x[u].z = 0u;
          if (last < 4) x[u].w = 0u;
        }
        if (e < q * nw4) s_adj[r * ns + k] = x[u];
      }
    }
    for (int r = t; r < q; r += kSmThreads) s_rho[r] = __ldcg(im.rho_fix + r);
    if (t < kSmMaxW) { sh.cm[t] = 0u; sh.rm[t] = 0u; }
  }
  __syncthreads();
  {
    constexpr int RPT = kSmallMaxN / kSmThreads;       // rows per thread
    bool done[RPT];
#pragma unroll
    for (int k = 0; k < RPT; ++k) done[k] = t + k * kSmThreads >= q;
    int sweeps = 0;
    for (;;) {
      ++sweeps;
      int pending = 0;
#pragma unroll
      for (int k = 0; k < RPT; ++k) {
        const int r = t + k * kSmThreads;
        if (done[k]) continue;
        const uint4 *row = s_adj + r * ns;
        uint32_t hit = 0u;
#pragma unroll 4
        for (int v = 0; v < nw4; ++v) {
          const uint4 a = row[v], c = ld_volatile_smem4(&sh.cm[4 * v]);
          hit |= (a.x & c.x) | (a.y & c.y) | (a.z & c.z) | (a.w & c.w);
        }
        bool alive = false;
        if (!hit) {                                    // (a neighbour that has become a centre since counts as undecided)
          const unsigned long long mine = s_rho[r];
          for (int wd = 0; wd < nw && !alive; ++wd) {
            uint32_t a = reinterpret_cast<const uint32_t *>(row)[wd];
            if (!a) continue;
            a &= ~*const_cast<volatile uint32_t *>(&sh.rm[wd]);
            if (wd == (r >> 5)) a &= ~(1u << (r & 31));
            while (a) {
              const int b = __ffs(a) - 1, j = wd * 32 + b;
              a &= a - 1;
              const unsigned long long o = s_rho[j];
              if (o > mine || (o == mine && j < r)) { alive = true; break; }
            }
          }
        }
        if (hit) { atomicOr(&sh.rm[r >> 5], 1u << (r & 31)); done[k] = true; }
        else if (!alive) { atomicOr(&sh.cm[r >> 5], 1u << (r & 31)); done[k] = true; }
        else pending = 1;
      }
      if (!__syncthreads_or(pending)) break;
      if (sweeps >= sweep_limit) {
        if (t == 0) atomicMin(&im.cnt[PACT_CNT_STATUS], (int)PACT_ERR_TIMEOUT);
        break;
      }
    }
    if (rank == 0 && t == 0) im.cnt[PACT_CNT_SWEEPS] = sweeps;
  }
  if (w == 0) {                                        // cluster ids: centres by ascending token
    const int pc = lane < nw ? __popc(sh.cm[lane]) : 0;
    int x = pc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    sh.pref[lane] = x - pc;
    if (lane == 31) sh.C = x;
  }
  __syncthreads();
  const int C = sh.C;
  for (int r = t; r < q; r += kSmThreads) {
    const uint32_t m = sh.cm[r >> 5];
    if ((m >> (r & 31)) & 1u) {
      const int c = sh.pref[r >> 5] + __popc(m & ((1u << (r & 31)) - 1u));
      sh.cen[c] = sh.kept[r];
      sh.own_cid[sh.kept[r]] = (short)c;
    }
  }
  __syncthreads();
  TL_POINT(im, 7);

  // ---- rows x centres -----------------------------------------------------------------------------------------------
  if constexpr (UMMA) {
    // blocks of 128 tokens; the centres in column tiles of at most 64, more of them where that gives idle CTAs work
    const int nbN = (N + kSmBM - 1) / kSmBM;
    int ntn = max((C + kSmBN - 1) / kSmBN, min((C + 15) / 16, CL / nbN));
    const int CW = max(16, ((C + ntn - 1) / max(1, ntn) + 15) & ~15);
    ntn = (C + CW - 1) / CW;
    for (int unit = rank; unit < nbN * ntn; unit += CL) {
      const int blk = unit / ntn, cb = (unit - blk * ntn) * CW;
      int tokA[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int ra = blk * kSmBM + (t >> 3) + 64 * k;
        tokA[k] = ra < N ? ra : -1;
      }
      const int rb = cb + (t >> 3);
      const bool ok = small_tile(sh, dyn, phase, Kc, im.ldKc, bt.d_k, tokA, rb < C ? (int)sh.cen[rb] : -1, CW, false);
      const int qd = w & 3, row = blk * kSmBM + qd * 32 + lane, k0 = (w >> 2) * 32, c0 = cb + k0;
      const int lim = ok ? min(min(32, CW - k0), C - c0) : 0;
      if (lim > 0) {
        sh.rn_col[w][lane] = lane < lim ? (float)sh.rn[sh.cen[c0 + lane]] : 0.f;
        __syncwarp();
        const float rni = row < N ? (float)sh.rn[row] : 0.f;
        float bc = -4.0f;
        int bi = 0;
#pragma unroll 1
        for (int k8 = 0; k8 < lim; k8 += 8) {
          uint32_t v[8];
          tmem_ld8(sh.tmem_base + k0 + k8 + ((uint32_t)(qd * 32) << 16), v);
          tmem_ld_wait();
#pragma unroll
          for (int kk = 0; kk < 8; ++kk) {
            const float c = (__uint_as_float(v[kk]) * rni) * sh.rn_col[w][k8 + kk];
            if (k8 + kk < lim && c > bc) { bc = c; bi = c0 + k8 + kk; }
          }
        }
        if (row < N && bc > -3.0f) {
          const float bd = fminf(fmaxf(1.0f - bc, 0.0f), 2.0f);
          atomicMin(&im.best[row], ((unsigned long long)__float_as_uint(bd) << 32) | (unsigned)bi);
        }
      }
      tc_fence_before();
      __syncthreads();
    }
  } else {
    const int g = t >> 7, tg = t & 127, ntm = (N + TS - 1) / TS, ntn = (C + TS - 1) / TS;
    F64Group &fg = reinterpret_cast<F64Group *>(dyn)[g];
    for (int tile = g * CL + rank; tile < ntm * ntn; tile += 4 * CL) {
      const int tm = tile / ntn, tn = tile % ntn;
      double acc[2][2][2];
      tile_dots<T>(
          tg, [&](int r) { const int x = tm * TS + r; return x < N ? Kc + (size_t)x * im.ldKc : (const T *)nullptr; },
          [&](int r) { const int x = tn * TS + r; return x < C ? Kc + (size_t)sh.cen[x] * im.ldKc : (const T *)nullptr; },
          bt.d_k, fg.As, fg.Bs, acc, [&]() { group_sync(g); });
      assign_epilogue_f64<D>(tg, tn * TS, C, acc, [&](int l) { return tm * TS + l < N ? sh.rn[tm * TS + l] : (rn_t)0; },
                             [&](int c) { return sh.rn[sh.cen[c]]; }, fg.rowbest);
      group_sync(g);
      if (tg < TS && tm * TS + tg < N)
        atomicMin(&im.best[tm * TS + tg], fg.rowbest[0][tg] < fg.rowbest[1][tg] ? fg.rowbest[0][tg] : fg.rowbest[1][tg]);
    }
  }
  cluster_sync();
  TL_POINT(im, 8);

  // ---- 5: labels of the own tokens (Eq. 8-9) ---------------------------------------------------------------------------
  {
    const int wn = (nown + 31) / 32;                   // warps with tokens
    if (w < wn) {
      int joined = 0, dropped = 0, bnd = 0;
      const int i = own0 + t;
      if (t < nown) {
        const unsigned long long pk = __ldcg(im.best + i);
        int lab = (int)(pk & 0xFFFFFFFFull);
        const float dd = __uint_as_float((uint32_t)(pk >> 32));
        if (sh.keep8[i]) {
          if (sh.own_cid[i] >= 0) lab = sh.own_cid[i];
        } else {
          if (D::in_band_t(dd, im)) ++bnd;
          if (D::below_t(dd, im)) ++joined; else { lab = -1; ++dropped; }
        }
        if (lab >= C || lab < -1) lab = -1;            // only after a failed earlier stage
        if (im.label_user) im.label_user[i] = lab;
        for (int u = 0; u < CL; ++u) put(&sh.lab[i], u, (short)lab);
      }
      joined = __reduce_add_sync(0xffffffffu, joined);
      dropped = __reduce_add_sync(0xffffffffu, dropped);
      bnd = __reduce_add_sync(0xffffffffu, bnd);
      if (lane == 0) {
        if (joined) atomicAdd(&im.cnt[PACT_CNT_R], joined);
        if (dropped) atomicAdd(&im.cnt[PACT_CNT_DISCARDED], dropped);
        if (bnd) atomicAdd(&im.cnt[PACT_CNT_BAND_ADC], bnd);
      }
    }
    if (t == 0 && sh.abort) atomicMin(&im.cnt[PACT_CNT_STATUS], (int)PACT_ERR_TIMEOUT);
  }
  if constexpr (UMMA) {
    if (w == 0) {
      if (lane == 0 && sh.abort) finish_mmas(&sh.done);
      __syncwarp();
      tmem_dealloc(sh.tmem_base, 128);
    }
  }
  cluster_sync();
  TL_POINT(im, 10);

  // ---- 6: a stable counting sort of the tokens by cluster: sizes and offsets by every CTA for itself, records of the own ---
  const int nchunk = (N + 31) / 32;
  unsigned char *s_tab = dyn;                          // [nchunk][C] members of cluster c in chunk of 32 tokens
  if (rank == 0 && t == 0) {
    im.cnt[PACT_CNT_Q] = q;
    im.cnt[PACT_CNT_M] = N - q;
    im.cnt[PACT_CNT_C] = C;
  }
  for (int c = rank * kSmThreads + t; c < C; c += CL * kSmThreads) im.center_idx[c] = sh.cen[c];   // (centre-only merging)
  for (int e = t; e < (nchunk * C + 15) / 16; e += kSmThreads) reinterpret_cast<uint4 *>(s_tab)[e] = make_uint4(0u, 0u, 0u, 0u);
  for (int c = t; c < C; c += kSmThreads) sh.size[c] = 0;
  __syncthreads();
  for (int ch = w; ch < nchunk; ch += kSmWarps) {
    const int i = ch * 32 + lane, lab = i < N ? sh.lab[i] : -1;
    const unsigned same = __match_any_sync(0xffffffffu, lab);
    if (lab >= 0 && lane == __ffs(same) - 1) {
      s_tab[ch * C + lab] = (unsigned char)__popc(same);
      atomicAdd(&sh.size[lab], __popc(same));
    }
  }
  __syncthreads();
  {
    constexpr int SPT = kSmallMaxN / kSmThreads;       // sizes per thread
    int v[SPT], s = 0;
#pragma unroll
    for (int k = 0; k < SPT; ++k) { v[k] = t * SPT + k < C ? sh.size[t * SPT + k] : 0; s += v[k]; }
    int x = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) sh.wsum[w] = x;
    __syncthreads();
    int run = x - s, tot = 0;
#pragma unroll
    for (int k = 0; k < kSmWarps; ++k) { if (k < w) run += sh.wsum[k]; tot += sh.wsum[k]; }
#pragma unroll
    for (int k = 0; k < SPT; ++k) {
      if (t * SPT + k < C) sh.off[t * SPT + k] = run;
      run += v[k];
    }
    if (t == 0) sh.off[C] = tot;
  }
  __syncthreads();
  if (rank == 0 && t == 0) im.cnt[20] = sh.off[C];
  // place of an own token among its cluster's members: eight threads share the chunks before it
  {
    const int li = t >> 3, part = t & 7, i = own0 + li;
    const int lab = li < nown ? sh.lab[i] : -1;
    int before = 0;
    if (lab >= 0) {
      const int ch = i >> 5;
      for (int u = part; u < ch; u += 8) before += s_tab[u * C + lab];
      for (int k = (ch << 5) + part; k < i; k += 8) before += sh.lab[k] == lab;
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
    if (lab >= 0 && part == 0) {
      im.members[sh.off[lab] + before] = make_int4(i, lab, sh.off[lab], sh.size[lab]);
      if (before == 0) {                               // first member of the cluster: the row's bookkeeping
        const int dst = im.vis_start + lab;
        im.P_out[dst] = im.P[im.vis_start + sh.cen[lab]];
        im.size_out[dst] = sh.size[lab];
        if (im.logw_out) im.logw_out[dst] = logf((float)sh.size[lab]);
      }
    }
  }
}

// ---- host side ---------------------------------------------------------------------------------------------------

namespace {

static_assert(sizeof(SmallShared<__nv_bfloat16>) + kSmDynUmma <= 227 * 1024 && sizeof(SmallShared<float>) + kSmDynF64 <= 227 * 1024, "shared memory of an SM");
static_assert(kSmDynUmma > kAloneOnSm, "one CTA with tensor memory per SM");
static_assert(4 * sizeof(F64Group) <= kSmDynF64 - 1024, "double-precision tiles");
static_assert((size_t)kSmallMaxN * (kSmMaxW / 4 + 1) * 16 + kSmallMaxN * 8 <= kSmDynF64 - 1024, "adjacency of the survivors");
static_assert(kSmMaxHeads * (kSmallMaxN / kMinPiece) * 8 <= kSmDynF64 - 1024 && kSmMaxW * kSmallMaxN <= kSmDynF64 - 1024, "softmax pieces, member table");

template <typename T, bool UMMA> cudaError_t small_attr() {
  constexpr int dyn = (int)(UMMA ? kSmDynUmma : kSmDynF64);
  cudaError_t e = cudaFuncSetAttribute(k_small<T, UMMA>, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_small<T, UMMA>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return e;
}

template <typename T, bool UMMA>
cudaError_t launch_small_t(const Batch &bt, int rpp, int sweep_limit, cudaStream_t st) {
  LaunchOpt opt;
  opt.cluster = CL;
  return launch_opt(opt, k_small<T, UMMA>, dim3(CL, bt.B), dim3(kSmThreads), UMMA ? kSmDynUmma : kSmDynF64, st, bt, rpp, sweep_limit);
}

}  // namespace

cudaError_t small_configure(DeviceCfg *cfg) {
  cudaError_t e = small_attr<__nv_bfloat16, true>();
  if (e == cudaSuccess) e = small_attr<__nv_bfloat16, false>();
  if (e == cudaSuccess) e = small_attr<float, false>();
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(CL);
  lc.blockDim = dim3(kSmThreads);
  lc.dynamicSmemBytes = kSmDynUmma;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CL;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  lc.attrs = attr;
  lc.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, k_small<__nv_bfloat16, true>, &lc) != cudaSuccess) {
    (void)cudaGetLastError();
    n = 0;
  }
  cfg->small_clusters = n;
  return cudaSuccess;
}

// Up to as many images as clusters fit on the GPU at once (with a second round the wide kernels are as fast), and as long as
// the chain of kernels that the cluster saves (about 10 us) is worth more than the SMs it leaves idle.  Calls of one image in
// us, cluster against wide kernels, C = N / 16:
//   tensor-core tiles   One round of the all-pairs pass, i.e. 512 survivors (d_k 512: 512 survivors of 1024 tokens 51 against
//                       53, 538 of 768 tokens 65 against 53), and not too many operands for 16 SMs to take in (d_k 1024: 768
//                       tokens 58 against 60, 1024 tokens 62 against 60).
//   double precision    32 x 32 tiles of survivors and of tokens x centres (a twentieth of the tokens), each with a fixed part
//                       of about 256 key elements' time (fp32, d_k 128: 512 tokens, half pruned, 43 against 49, nothing pruned
//                       64 against 50; d_k 512: 256 tokens 57 against 66 and 70 against 64; d_k 1024, 512 tokens, nothing
//                       pruned 200 against 97).
// With more images the idle share is smaller (d_k 512, two and four images of 512 half-pruned tokens: 70 against 76, 73
// against 102).  Of 340 calls of one to four images measured, d_k 64 to 2048 and pruning 0 to 0.8, the rule takes 0.4 % more
// than the better form of each would, the sizes alone took 9 %.
bool small_fits(const Batch &bt, int maxN, bool umma, const DeviceCfg &cfg) {
  if (maxN > (umma ? kSmallMaxN : kSmallMaxF64) || bt.n_qh > kSmMaxHeads || bt.B > cfg.small_clusters) return false;
  const double idle = 1.0 - (double)(CL * bt.B) / cfg.sm_count;
  for (int b = 0; b < bt.B; ++b) {
    const int N = bt.img[b].N, q = N - bt.img[b].m_target;
    if (umma) {
      const int nb = (q + kSmBM - 1) / kSmBM;
      if (nb * nb > CL || (double)N * bt.d_k * idle > 710e3) return false;
    } else {
      const int nq = (q + TS - 1) / TS, tiles = nq * (nq + 1) / 2 + (N + TS - 1) / TS * ((N / 20 + TS - 1) / TS);
      if (tiles > 160 || (double)tiles * (bt.d_k + 256) * idle * idle > 26700.0) return false;
    }
  }
  return true;
}

cudaError_t launch_small(const Batch &bt, bool in_bf16, bool umma, int rpp, int sweep_limit, cudaStream_t st) {
  if (in_bf16) return umma ? launch_small_t<__nv_bfloat16, true>(bt, rpp, sweep_limit, st) : launch_small_t<__nv_bfloat16, false>(bt, rpp, sweep_limit, st);
  return launch_small_t<float, false>(bt, rpp, sweep_limit, st);
}

}  // namespace pact
