// tcgen05 primitives of a single CTA (tensor memory, MMA, commit, loads) and the epilogue arithmetic of the all-pairs
// pass, shared by the tile kernels and the one-kernel step for small images.
#pragma once
#include "common.cuh"
#include "tma.cuh"

namespace pact {

constexpr size_t kAloneOnSm = 114 * 1024;   // a CTA with more dynamic shared memory than this has its SM to itself among its like

__device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t addr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum) : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory operand descriptor: K-major rows of 128 bytes, 128-byte swizzle, 8-row groups
// 1024 bytes apart, descriptor version 1.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// The descriptor of an operand `bytes` (a multiple of 16) after the one of d.  One addition: the thread that issues the MMAs has
// about 180 clocks for each of a 128 x 256 x 16 step, and a descriptor formed anew for every one takes a good part of them
// (rows x centres pass of one image of 12935 tokens in rounds of tiles: 4 us of a call of 163).
__device__ __forceinline__ uint64_t desc_at(uint64_t d, uint32_t bytes) { return d + (bytes >> 4); }

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float fma_sat(float a, float b, float c) {   // clamped to [0, 1]
  float y;
  asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
  return y;
}

// One 32-column chunk of the epilogue of the all-pairs pass for one row (= one lane): distance
// (Eq. 5), density term (Eq. 6) as an integer multiple of 2^-30, adjacency bit d <= d_c, band count.
// EDGE adds the per-element checks that only edge chunks need (diagonal, columns past the end).
// COLS (blocks above the diagonal) also hands every pair to its column: the warp's 32 x 32 terms go
// through a shared-memory buffer `tr` (row stride 36 words: conflict-free stores, 16-byte loads), lane k
// adds the 32 terms of column k, and a 32 x 32 bit transpose gives it the column's adjacency word.
//
// This pass is bound by its epilogue: 7290 keys on pairs of CTAs take 46 us by themselves with 20 instructions per pair, the
// issue slots 45 % busy, the special functions and the tensor pipe 36 %; four epilogue warps per scheduler wait for shuffles,
// conversions and shared memory as often as they issue.  Fewer instructions shorten those chains, so the arithmetic of DistF
// (common.cuh) is written for few of them, with the same results: all of it on half the distance, whose clamp to
// [0, 1] is part of the multiply-add and whose scaling by two is exact (rn_col holds -1/2 of the columns' inverse norms);
// the adjacency bit is the sign of h minus the number after d_c / 2; `nearest`, the smallest magnitude of that, tells whether
// a pair may be within the band (see gram_band); three terms are summed in 32 bits.  DBDPC of 7290 tokens as a call:
// 120 -> 116 us; the pass over four images of 4916 survivors: 84 -> 78 us.
template <bool EDGE, bool COLS>
__device__ __forceinline__ void gram_chunk(const uint32_t (&v)[32], const float *rn_col, float rni, int row, int c0,
                                           int ncols, float d_c, float neg_k, int lane, uint32_t *tr,
                                           unsigned long long &rowsum, uint32_t &bits, float &nearest,
                                           unsigned long long &colsum, uint32_t &colbits) {
  uint32_t b = 0u;
  unsigned long long s = 0ull;
  uint32_t s3 = 0u;                                 // three terms, each at most 2^30, fit in 32 bits
  const float after = __uint_as_float(__float_as_uint(0.5f * d_c) + 1u), k2 = 2.0f * neg_k;   // (d_c is not negative)
  float closest = 4.0f;
  // rn_i * rn_j first: a pair must get the same distance whichever of the two is the row, so that
  // duplicate keys keep exactly equal densities
#pragma unroll
  for (int k4 = 0; k4 < 32; k4 += 4) {
    const float4 rn4 = *reinterpret_cast<const float4 *>(rn_col + k4);
    const float rnj[4] = {rn4.x, rn4.y, rn4.z, rn4.w};
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      const int k = k4 + kk;
      const float h = EDGE && c0 + k == row ? 0.f : fma_sat(__uint_as_float(v[k]), rni * rnj[kk], 0.5f), t = h - after;
      uint32_t term = __float2uint_rn(ex2_approx(h * k2) * (float)(1u << kRhoShift));
      if (EDGE && c0 + k >= ncols) term = 0u;
      b = __funnelshift_l(__float_as_uint(t), b, 1);
      closest = fminf(closest, fabsf(t));
      s3 += term;
      if (k % 3 == 2 || k == 31) { s += s3; s3 = 0u; }   // a run of keys at distance 0 adds 2^30 each
      if (COLS) tr[k * 36 + lane] = term;
    }
  }
  b = __brev(b);                                    // (column 0 went in first)
  if (EDGE && c0 + 32 > ncols) b &= ncols > c0 ? (1u << (ncols - c0)) - 1u : 0u;
  rowsum += s;
  bits = b;
  nearest = closest;
  if (COLS) {
    __syncwarp();
    // lane k: the 32 terms of column k, three to a 32-bit partial sum as above
    unsigned long long cs = 0ull;
    uint32_t c3 = 0u;
    const uint4 *src = reinterpret_cast<const uint4 *>(tr + lane * 36);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint4 x = src[j];
      const uint32_t xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        c3 += xs[i];
        if ((j * 4 + i) % 3 == 2 || j * 4 + i == 31) { cs += c3; c3 = 0u; }
      }
    }
    colsum = cs;
    // transpose the 32 x 32 bit matrix (lane l holds row l): five exchange steps
    uint32_t w = b;
#pragma unroll
    for (int sft = 16; sft >= 1; sft >>= 1) {
      const uint32_t m = sft == 16 ? 0x0000FFFFu : sft == 8 ? 0x00FF00FFu : sft == 4 ? 0x0F0F0F0Fu
                         : sft == 2 ? 0x33333333u : 0x55555555u;
      const uint32_t y = __shfl_xor_sync(0xffffffffu, w, sft);
      w = (lane & sft) ? ((w & ~m) | ((y >> sft) & m)) : ((w & m) | ((y << sft) & ~m));
    }
    colbits = w;
    __syncwarp();                                   // tr may be rewritten by the next chunk
  }
}

// Pairs (row, column after it) of the chunk within 1e-6 of d_c; called where the chunk's `nearest` is at most kNear.
constexpr float kNear = 1e-6f;                      // half of the band, and the step to the number after d_c / 2
__device__ __forceinline__ int gram_band(const uint32_t (&v)[32], const float *rn_col, float rni, int row, int c0, int ncols, float d_c) {
  int n = 0;
#pragma unroll
  for (int k = 0; k < 32; ++k)
    n += row < c0 + k && c0 + k < ncols && fabsf(2.0f * fma_sat(__uint_as_float(v[k]), rni * rn_col[k], 0.5f) - d_c) <= 1e-6f;
  return n;
}

}  // namespace pact
