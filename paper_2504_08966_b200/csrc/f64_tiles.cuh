// Tiles of dot products in double precision (m8n8k4 tensor instruction) and their epilogue for the all-pairs pass,
// shared by the kernels for fp32 keys and the one-kernel step for small images.
#pragma once
#include "common.cuh"

namespace pact {

// ---- 32 x 32 tile of dot products in double, 128 threads -----------------------------------------
// fp32 keys (and bf16 keys of a width the tcgen05 tiles do not take) get their dot products from the double-precision
// tensor instruction (m8n8k4): the products of fp32 values are exact in double and the sums carry its full precision.
// Warp (wy, wx) owns the 16 x 16 quarter at rows 16 wy, columns 16 wx as 2 x 2 fragments; lane l holds of fragment
// (a, b) the row 8 a + l / 4 and the columns 8 b + 2 (l % 4) + {0, 1}.  Small tiles on purpose: these matrices are
// small (a thumbnail has 138 survivors), so the tiles have to be many for the SMs to share them.  The operands are
// widened once when they are staged; the next slab is on its way from the L2 while this one is multiplied.
// One scalar FMA per product with 64 x 64 tiles, widening at every use, took 23 us for 138 x 138 x 128.
constexpr int TS = 32;        // tile side
constexpr int KC = 64;        // key elements staged per step
constexpr int KST = KC + 4;   // row stride of a staged slab in doubles: fragment loads meet no bank twice
constexpr int kTileThreads = 128;

// t: thread within the group of 128 that shares the tile; sync: barrier of that group.
template <typename T, typename RowA, typename RowB, typename Sync>
__device__ __forceinline__ void tile_dots(int t, RowA rowA, RowB rowB, int d_k, double (*As)[KST], double (*Bs)[KST],
                                          double (&acc)[2][2][2], Sync sync) {
  constexpr int V = Vec<T>::N;
  constexpr int VPR = KC / V;                          // vectors per row of a slab
  constexpr int NV = 2 * TS * VPR / kTileThreads;      // vectors per thread: the first half A, the second half B
  const int lane = t & 31, w = t >> 5, wy = w >> 1, wx = w & 1;
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) acc[a][b][0] = acc[a][b][1] = 0.0;
  uint4 buf[NV];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int u = 0; u < NV; ++u) {
      const int v = (u % (NV / 2)) * kTileThreads + t, row = v / VPR, k = k0 + (v % VPR) * V;
      const T *p = u < NV / 2 ? rowA(row) : rowB(row);
      buf[u] = p && k < d_k ? *reinterpret_cast<const uint4 *>(p + k) : make_uint4(0u, 0u, 0u, 0u);
    }
  };
  fetch(0);
  for (int k0 = 0; k0 < d_k; k0 += KC) {
    sync();                                            // the slab before has been read
#pragma unroll
    for (int u = 0; u < NV; ++u) {
      const int v = (u % (NV / 2)) * kTileThreads + t, row = v / VPR, k = (v % VPR) * V;
      double *dst = (u < NV / 2 ? As[row] : Bs[row]) + k;
      float x[V];
      widen_vec<T>(buf[u], x);
#pragma unroll
      for (int e = 0; e < V; e += 2) *reinterpret_cast<double2 *>(dst + e) = make_double2((double)x[e], (double)x[e + 1]);
    }
    sync();
    if (k0 + KC < d_k) fetch(k0 + KC);
#pragma unroll 8
    for (int k = 0; k < KC; k += 4) {
      double a[2], b[2];
#pragma unroll
      for (int f = 0; f < 2; ++f) {
        a[f] = As[wy * 16 + f * 8 + (lane >> 2)][k + (lane & 3)];
        b[f] = Bs[wx * 16 + f * 8 + (lane >> 2)][k + (lane & 3)];
      }
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j)
          asm("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
              : "+d"(acc[i][j][0]), "+d"(acc[i][j][1]) : "d"(a[i]), "d"(b[j]));
    }
  }
}

// tile `t` of the nt (nt + 1) / 2 tiles on and above the diagonal, row by row
__device__ __forceinline__ void upper_tile(int t, int nt, int &tm, int &tn) {
  const double b = 2.0 * nt + 1.0;
  int i = (int)((b - sqrt(fmax(b * b - 8.0 * t, 0.0))) * 0.5);
  i = max(0, min(i, nt - 1));
  while (i > 0 && i * nt - i * (i - 1) / 2 > t) --i;
  while (i + 1 < nt && (i + 1) * nt - (i + 1) * i / 2 <= t) ++i;
  tm = i;
  tn = i + (t - (i * nt - i * (i - 1) / 2));
}

// Epilogue of one tile of the all-pairs pass (Eq. 5-6): density terms, adjacency bits and the band count of the pairs
// of rows tm * 32 .. and columns tn * 32 ..; a tile above the diagonal serves its rows and its columns.  rn(g): inverse
// norm of survivor g.  sh may be reused once the group has passed its next barrier.
struct F64Sums {
  unsigned long long rsum[2][TS], csum[2][TS];         // by column half of the rows, by row half of the columns
  uint32_t rbits[2][TS], cbits[2][TS];
};
template <typename D, typename Rn, typename Sync>
__device__ __forceinline__ void gram_epilogue_f64(int t, int tm, int tn, int q, const double (&acc)[2][2][2], Rn rn,
                                                  const ImgDesc &im, F64Sums &sh, int &band, Sync sync) {
  using dist_t = typename D::acc_t;
  const int lane = t & 31, w = t >> 5, wy = w >> 1, wx = w & 1;
  unsigned long long rs[2] = {0ull, 0ull}, cs[2][2] = {};
  uint32_t rb[2] = {0u, 0u}, cb[2][2] = {};
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const int li = wy * 16 + a * 8 + (lane >> 2), gi = tm * TS + li;
    const double rni = gi < q ? rn(gi) : 0.0;
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int lj = wx * 16 + b * 8 + 2 * (lane & 3) + e, gj = tn * TS + lj;
        if (gi >= q || gj >= q) continue;
        dist_t dd = (dist_t)fmin(fmax(1.0 - acc[a][b][e] * (rni * rn(gj)), 0.0), 2.0);
        if (gi == gj) dd = 0;
        const unsigned long long term = D::term(dd, im);
        rs[a] += term;
        cs[b][e] += term;
        if (D::within(dd, im)) { rb[a] |= 1u << lj; cb[b][e] |= 1u << li; }
        if (gi < gj && D::in_band(dd, im)) ++band;
      }
  }
#pragma unroll
  for (int a = 0; a < 2; ++a) {                      // rows: the four lanes that hold parts of one
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
      rs[a] += __shfl_xor_sync(0xffffffffu, rs[a], o);
      rb[a] |= __shfl_xor_sync(0xffffffffu, rb[a], o);
    }
    if ((lane & 3) == 0) { sh.rsum[wx][wy * 16 + a * 8 + (lane >> 2)] = rs[a]; sh.rbits[wx][wy * 16 + a * 8 + (lane >> 2)] = rb[a]; }
#pragma unroll
    for (int e = 0; e < 2; ++e) {                    // columns: the eight lanes
#pragma unroll
      for (int o = 4; o < 32; o <<= 1) {
        cs[a][e] += __shfl_xor_sync(0xffffffffu, cs[a][e], o);
        cb[a][e] |= __shfl_xor_sync(0xffffffffu, cb[a][e], o);
      }
      if (lane < 4) { sh.csum[wy][wx * 16 + a * 8 + 2 * lane + e] = cs[a][e]; sh.cbits[wy][wx * 16 + a * 8 + 2 * lane + e] = cb[a][e]; }
    }
  }
  sync();
  if (t < 2 * TS) {                                  // (the barrier inside the next tile_dots comes before these are rewritten)
    const int l = t & (TS - 1), side = t / TS;       // 0: rows, 1: columns (above the diagonal only)
    const int g = (side ? tn : tm) * TS + l;
    if (g < q && !(side && tm == tn)) {
      atomicAdd(&im.rho_fix[g], side ? sh.csum[0][l] + sh.csum[1][l] : sh.rsum[0][l] + sh.rsum[1][l]);
      im.adj[(size_t)g * im.Wp + (side ? tm : tn)] = side ? (sh.cbits[0][l] | sh.cbits[1][l]) : (sh.rbits[0][l] | sh.rbits[1][l]);
    }
  }
}

// Epilogue of one tile of the rows x centres pass: the nearest of the centres c0 .. of each of the 32 rows as a packed
// (distance bits, cluster id) word, one per column half.  rnt(l), rnc(c): inverse norms of local row l and centre c.
template <typename D, typename RnT, typename RnC>
__device__ __forceinline__ void assign_epilogue_f64(int t, int c0, int C, const double (&acc)[2][2][2], RnT rnt, RnC rnc,
                                                    unsigned long long (*rowbest)[TS]) {
  using acc_t = typename D::acc_t;
  const int lane = t & 31, w = t >> 5, wy = w >> 1, wx = w & 1;
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const int l = wy * 16 + a * 8 + (lane >> 2);
    const auto rni = rnt(l);
    unsigned long long bestv = kBestInit;
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int c = c0 + wx * 16 + b * 8 + 2 * (lane & 3) + e;
        if (c >= C) continue;
        const float dd = (float)D::dist((acc_t)acc[a][b][e], rni, rnc(c));
        const unsigned long long pk = ((unsigned long long)__float_as_uint(dd) << 32) | (unsigned)c;
        bestv = pk < bestv ? pk : bestv;
      }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
      const unsigned long long y = __shfl_xor_sync(0xffffffffu, bestv, o);
      bestv = y < bestv ? y : bestv;
    }
    if ((lane & 3) == 0) rowbest[wx][l] = bestv;
  }
}

}  // namespace pact
