// EUTI (Algorithm 1): global query (Eq. 1), per-head softmax over the visual tokens and hidden-state
// norm (Eq. 2), percentile split (Eq. 3-4).  Every accumulation that decides an ordering is carried
// in double so that the float32 score the library returns is the correctly rounded value in all but
// rare double-rounding cases.
//
//   k_qsum           column sums of Q -> global query
//   k_tokens         one pass over the hidden states and the keys: |h_i|, 1 / |k_i|, k_i . Qglobal per head,
//                    softmax pieces of up to 32 tokens (HBM-bound, the first of two reads of H); also clears what later
//                    kernels accumulate into
//   k_scores         merges the pieces, writes the float32 scores and the histogram of their top key bits
//   k_select         every CTA selects the threshold (histogram bin, then one pass inside it that mostly leaves the key
//                    itself, else a few that are ranked; radix passes for many equal scores) and counts the survivors
//                    before its tokens, then writes its share of the lists and gathers its share of the survivor keys
//   k_split_regs, k_split   the split for the stage call pact_prune (scores given, no histogram): radix select
//
// The kernels are short chains of dependent memory round trips; each issues all the loads it can
// before it consumes the first.
#include <string.h>

#include <type_traits>

#include "kernels.cuh"
#include "tma.cuh"

namespace pact {

__device__ __forceinline__ double ld_cg_f64(const double *p) {
  double v;
  asm volatile("ld.global.cg.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ void ld_cg_f64x2(const double *p, double &a, double &b) {
  asm volatile("ld.global.cg.v2.f64 {%0, %1}, [%2];" : "=d"(a), "=d"(b) : "l"(p));
}

// Widening to double by moving bits: the exponent field of the element becomes the low bits of the double's, i.e. the
// double is the element times 2^-896, exactly, zeros and subnormal numbers included (the sum is multiplied by 2^896 at
// the end).  The conversion unit takes 16 elements per clock and SM and was what bounded the sums over Q.  An infinity or a
// NaN would come out as an ordinary number near 2^128: NonFinite finds them.
constexpr double kWidenScale = 0x1p896;
template <typename T> __device__ __forceinline__ void widen_scaled(const uint4 &v, double (&x)[Vec<T>::N]);
__device__ __forceinline__ double scaled_hi(uint32_t w) { return __hiloint2double((int)w >> 3 & (int)0x8FFFE000, 0); }   // bf16 in the upper half
template <> __device__ __forceinline__ void widen_scaled<__nv_bfloat16>(const uint4 &v, double (&x)[8]) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) { x[2 * i] = scaled_hi(w[i] << 16); x[2 * i + 1] = scaled_hi(w[i]); }
}
__device__ __forceinline__ double scaled_f32(uint32_t w) { return __hiloint2double((int)w >> 3 & (int)0x8FFFFFFF, (int)(w << 29)); }
template <> __device__ __forceinline__ void widen_scaled<float>(const uint4 &v, double (&x)[4]) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) x[i] = scaled_f32(w[i]);
}
// NaN once one of the elements seen was not finite, else 0: x * 0 is NaN for an infinity and for a NaN.  CH chains: four
// multiply-adds per vector in one are longer than the column sums beside them.
template <int CH> __device__ __forceinline__ void see_finite(__nv_bfloat162 (&z)[CH], const uint4 &v) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) z[i % CH] = __hfma2(*reinterpret_cast<const __nv_bfloat162 *>(&w[i]), __floats2bfloat162_rn(0.f, 0.f), z[i % CH]);
}
template <int CH> __device__ __forceinline__ void see_finite(float (&z)[CH], const uint4 &v) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) z[i % CH] = fmaf(__uint_as_float(w[i]), 0.f, z[i % CH]);
}
template <typename T, int CH> struct NonFinite {
  using Z = typename std::conditional<sizeof(T) == 2, __nv_bfloat162, float>::type;
  Z z[CH];
  __device__ __forceinline__ NonFinite() { memset(z, 0, sizeof(z)); }
  __device__ __forceinline__ void see(const uint4 &v) { see_finite<CH>(z, v); }
  __device__ __forceinline__ float value() const {
    float s = 0.f;
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      if constexpr (sizeof(T) == 2) s += __low2float(z[c]) + __high2float(z[c]);
      else s += z[c];
    }
    return s;
  }
};
// Sum of the 32 parts of each of n <= 4 rows of this warp: eight lanes per row.
template <typename F>
__device__ __forceinline__ void finish_row_sums(const double (*acc)[32], int n, F put_sum) {
  const int lane = threadIdx.x & 31, j = lane >> 3;
  double s = 0.0;
  if (j < n) {
#pragma unroll
    for (int k = 0; k < 4; ++k) s += acc[j][(lane & 7) * 4 + k];
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (j < n && (lane & 7) == 0) put_sum(j, s);
  __syncwarp();
}

// ---- Eq. 1: column sums of Q -----------------------------------------------------------------------------
// grid (ncg RP, B) in clusters of RP CTAs, 256 threads at no more than 64 registers, two CTAs per SM or three, which
// leave room for k_tokens beside them.  Work item (column group of GV 16-byte vectors, block of rows): thread t takes
// vector t % GV of the group and the rows r0 + t / GV, + 256 / GV, ...; the row lanes of a warp are added with shuffles, the
// warps through shared memory.  The RP row blocks of a column group are one cluster: the CTAs store their sums into the
// first one's shared memory, which adds them in block order (the others leave at once: fetching the sums took a second
// barrier and 2 us more).  Bound by memory: 7.5 MB of one image's Q take 9 us with the start of the call, 48 MB of 16 images
// 25 us beside the row stream of k_tokens.  (Partial sums in global memory behind a ticket cost 2.6 us from the last row to
// the global query; with a conversion instruction per element instead of widen_scaled an SM took in 30 GB/s.)
constexpr int kQsumThreads = 256;
constexpr int kQsumWarps = kQsumThreads / 32;

template <typename T, int GV>
__global__ void __launch_bounds__(kQsumThreads, 4) k_qsum(const __grid_constant__ Batch bt, int RP, uint64_t policy) {
  constexpr int V = Vec<T>::N, LANES = kQsumThreads / GV;
  const ImgDesc &im = bt.img[blockIdx.y];
  TL_SCOPE(im, 0);
  pdl_wait();                                           // the work before this call, which may still use the workspace
  pdl_trigger();                                        // k_tokens may start: much of it does not need the query
  const int t = threadIdx.x, lane = t & 31, w = t >> 5, N = im.N, n_qcols = bt.n_qcols;
  if (!im.Q || (im.flags & PACT_FLAG_NORM_ONLY)) return;
  if (RP > 1) cluster_arrive();                         // (every CTA of the cluster runs before one stores to another)
  const int nvq = n_qcols / V;
  const int cg = blockIdx.x / RP, rp = blockIdx.x % RP; // rp = rank of the CTA in its cluster
  __shared__ double sm[kQsumWarps * GV * V];
  __shared__ double s_part[kQPartRows][GV * V];
  const int rchunk = (N + RP - 1) / RP;
  const int r0 = min(N, rp * rchunk), r1 = min(N, r0 + rchunk);
  const int v = cg * GV + (t % GV);
  double acc[V];
#pragma unroll
  for (int k = 0; k < V; ++k) acc[k] = 0.0;
  if (v < nvq) {
    constexpr int UQ = 8;
    NonFinite<T, 2> odd;
    const T *Q = reinterpret_cast<const T *>(im.Q) + (size_t)v * V;
    for (int r = r0 + t / GV; r < r1; r += LANES * UQ) {
      uint4 buf[UQ];
#pragma unroll
      for (int u = 0; u < UQ; ++u)
        if (r + u * LANES < r1) buf[u] = ld_hint(Q + (size_t)(r + u * LANES) * im.ldQ, policy);
#pragma unroll
      for (int u = 0; u < UQ; ++u) {
        if (r + u * LANES < r1) {
          double x[V];
          widen_scaled<T>(buf[u], x);
          odd.see(buf[u]);
#pragma unroll
          for (int k = 0; k < V; ++k) acc[k] += x[k];
        }
      }
    }
    // one column for all of the vector's: with a column that is NaN every score is
    acc[0] += (double)odd.value();
  }
#pragma unroll
  for (int o = GV; o < 32; o <<= 1)
#pragma unroll
    for (int k = 0; k < V; ++k) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
  if (lane < GV) {
#pragma unroll
    for (int k = 0; k < V; ++k) sm[(w * GV + lane) * V + k] = acc[k];
  }
  __syncthreads();
  const bool col_ok = t < GV * V && cg * GV + t / V < nvq;
  const size_t col = (size_t)cg * GV * V + t;
  double mine = 0.0;
  if (col_ok) {
#pragma unroll
    for (int ww = 0; ww < kQsumWarps; ++ww) mine += sm[ww * GV * V + t];
    if (RP == 1) im.qg[col] = mine * kWidenScale / (double)N;
  }
  if (RP == 1) return;
  cluster_wait();
  if (t < GV * V) st_cluster_f64(&s_part[rp][t], 0, mine);   // to the first CTA of the cluster
  cluster_arrive();
  if (rp != 0) return;
  cluster_wait();
  if (col_ok) {
    double s = 0.0;
    for (int u = 0; u < RP; ++u) s += s_part[u][t];
    im.qg[col] = s * kWidenScale / (double)N;
  }
}

// ---- Eq. 2, token pass: hidden-state norm, inverse key norm, logits, softmax pieces --------------------------------
// Persistent: one CTA of 512 threads and at most 64 registers per SM (beside it a CTA of k_qsum still fits), units of
// at most 32 tokens shared out over all images of the call (cut on the host: divisions from a cold instruction cache, before
// the first row was asked for, took 0.4 us).  Two groups of warps work side by side:
//   norms    Every warp takes each eighth token of the CTA's units (of each unit by itself, units of 25 tokens cost a round of
//            rows: one image of 7290 0.7 us).  The hidden-state rows run through two buffers of the warp's
//            own in shared memory, one bulk copy per row (or per 8 KB of it), so that copies never wait for arithmetic.
//            Sums of squares in float over a 16-byte vector and in double across.  Nothing here needs the global query.
//   logits   Two teams of four warps take the units in turn; a team's scoring keys come through a buffer of its own, in
//            flight before the global query is known: inverse key norms (of the first unit of either team before the wait for it); k_i . Qglobal per head in double; per head the
//            largest logit of the unit, exp(l - that) per token and their sum.  Up to two
//            query heads per key head a lane is a token (with few tokens a part of its elements), and the global query
//            comes from shared memory at one address per warp: with the lanes spread over the row the loads of the
//            query were what took the time, and with the double-precision tensor instruction (m8n8k4, whose rate is
//            that of the ordinary one) the seven idle heads of eight: 16 tokens of four heads took 4100 clocks a team.
//            With more heads per key head that instruction is the better form, see group_piece.
// `what` names the parts of the work (kTok...): hidden states that arrive from the host piece by piece have their norms
// formed by launches of their own.
// As 16-byte loads of four tokens per warp, one token's row at a time and the logits between them, the pass took 4.2 TB/s
// of HBM, and with 28 query heads on 4 key heads 31 us of 40 for a few hundred tokens.  Now 46656 tokens of 3584 (382 MB)
// end 77 us after the call began, against 100 us; bound by memory, 5.6 TB/s with the queries.
constexpr int kTokInit = 1, kTokNorms = 2, kTokLogits = 4;
constexpr int kTokThreads = 512;
constexpr int kTokGroup = 256;                          // threads of the norms group and of the logits group
constexpr int kTokTeam = kTokGroup / 2;                 // threads of a logits team
static_assert(kTokWarps == kTokGroup / 32, "a row buffer for each warp of the norms");
constexpr int kTeamWarps = kTokTeam / 32;

// Logits of this lane's token (its vectors p, p + P, ... of nv) with RB heads of a key head, q at one address per part.
// NaN if an element is not finite (even where the sum would be minus infinity and the token's share zero: to sum such keys again
// by ordinary conversions took the call of an image of 729 tokens 0.5 to 0.9 us just by being in the kernel).
template <typename T, int RB>
__device__ __forceinline__ void head_dots(const uint8_t *krow, const double *q, int d_h, int p, int P, double (&l)[RB]) {
  constexpr int V = Vec<T>::N, CH = 4 / RB;             // CH chains per head: an FMA takes nine clocks, two per warp can start
  const int nv = d_h / V;
  double acc[RB][CH];
#pragma unroll
  for (int j = 0; j < RB; ++j)
#pragma unroll
    for (int c = 0; c < CH; ++c) acc[j][c] = 0.0;
  NonFinite<T, 1> odd;
#pragma unroll 2
  for (int v = p; v < nv; v += P) {
    const uint4 raw = *(reinterpret_cast<const uint4 *>(krow) + v);
    double a[V];
    widen_scaled<T>(raw, a);
    odd.see(raw);
#pragma unroll
    for (int j = 0; j < RB; ++j) {
      const double2 *qj = reinterpret_cast<const double2 *>(q + (size_t)j * d_h + v * V);
#pragma unroll
      for (int e = 0; e < V; e += 2) {
        const double2 x = qj[e / 2];
        acc[j][e % CH] = fma(a[e], x.x, acc[j][e % CH]);
        acc[j][(e + 1) % CH] = fma(a[e + 1], x.y, acc[j][(e + 1) % CH]);
      }
    }
  }
#pragma unroll
  for (int j = 0; j < RB; ++j) {
    l[j] = acc[j][0];
#pragma unroll
    for (int c = 1; c < CH; ++c) l[j] += acc[j][c];
    l[j] *= kWidenScale;
  }
  l[0] = __hiloint2double(__double2hiint(l[0]) | __float_as_int(odd.value()), __double2loint(l[0]));   // (one head is enough: a score is their mean)
  for (int o = 32 / P; o < 32; o <<= 1)
#pragma unroll
    for (int j = 0; j < RB; ++j) l[j] += __shfl_xor_sync(0xffffffffu, l[j], o);
}

// The same heads j0, j0 + 1, ...: logits (zero without a query), the piece's largest, exp and sum.  tl = 32 / P lanes are
// the tokens of the unit, n of them real.
template <typename T, int RB>
__device__ __forceinline__ void head_piece(const Batch &bt, const ImgDesc &im, const uint8_t *krow, const double *q, bool use_query, int P, int j0,
                                           int r0, int n, int g) {
  const int lane = threadIdx.x & 31, tl = 32 / P, r = lane & (tl - 1), p = lane / tl;
  double l[RB];
  if (use_query) head_dots<T, RB>(krow, q, bt.d_h, p, P, l);
  else {
#pragma unroll
    for (int j = 0; j < RB; ++j) l[j] = 0.0;
  }
  double m[RB], e[RB], sum[RB];
#pragma unroll
  for (int j = 0; j < RB; ++j) {
    m[j] = warp_max(r < n ? l[j] : -1.0e300);
    e[j] = r < n ? exp(l[j] - m[j]) : 0.0;
    sum[j] = e[j];
  }
  for (int o = tl >> 1; o > 0; o >>= 1)
#pragma unroll
    for (int j = 0; j < RB; ++j) sum[j] += __shfl_xor_sync(0xffffffffu, sum[j], o);
#pragma unroll
  for (int j = 0; j < RB; ++j) {
    if (r < n && p == 0) im.E[(size_t)(j0 + j) * im.N + r0 + r] = e[j];
    if (lane == 0) *reinterpret_cast<double2 *>(piece_at(im, j0 + j, g)) = make_double2(m[j], sum[j]);
  }
}

// Two at a time, as a call: one chain of dependent steps takes 180 clocks, and every copy of the code is fetched from a cold
// instruction cache.
__device__ __noinline__ double2 exp_two(double a, double b) { return make_double2(exp(a), exp(b)); }
// Two elements of a key row, widened as widen_scaled does.
template <typename T> struct Pair;
template <> struct Pair<__nv_bfloat16> {
  uint32_t w;
  __device__ __forceinline__ void load(const uint8_t *p) { w = *reinterpret_cast<const uint32_t *>(p); }
  __device__ __forceinline__ void widen(double &a, double &b) const { a = scaled_hi(w << 16); b = scaled_hi(w); }
  __device__ __forceinline__ void see(float &z) const {     // (an infinity or a NaN times zero is a NaN)
    z = fmaf(__uint_as_float(w << 16), 0.f, z);
    z = fmaf(__uint_as_float(w & 0xFFFF0000u), 0.f, z);
  }
};
template <> struct Pair<float> {
  uint2 w;
  __device__ __forceinline__ void load(const uint8_t *p) { w = *reinterpret_cast<const uint2 *>(p); }
  __device__ __forceinline__ void widen(double &a, double &b) const { a = scaled_f32(w.x); b = scaled_f32(w.y); }
  __device__ __forceinline__ void see(float &z) const {
    z = fmaf(__uint_as_float(w.x), 0.f, z);
    z = fmaf(__uint_as_float(w.y), 0.f, z);
  }
};
// The larger of two doubles by their bits as integers, as warp_max orders them.
__device__ __forceinline__ double max_by_bits(double a, double b) {
  const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
  const long long kx = x ^ ((x >> 63) & 0x7fffffffffffffffll), ky = y ^ ((y >> 63) & 0x7fffffffffffffffll);
  return kx > ky ? a : b;
}

// The same for nr <= 8 heads of a key head at once, on the double-precision tensor instruction (m8n8k4: 8 tokens x 4 elements
// by 4 elements x 8 heads).  Lane 4 m + c holds of the keys the elements 2 c, 2 c + 1 of each eight of token m of a block,
// of the query the same elements of head m, and of the product the heads 2 c, 2 c + 1 of token m; the order in which the
// elements of a sum meet is free.  The query is read once for up to four blocks of eight tokens.
// With a token per lane every multiply-add takes eight bytes of the query per lane from shared memory, which hands out 128
// bytes a clock: 32 tokens of one head of 128 cost 256 clocks of it, against 512 clocks of the double-precision unit for up
// to eight heads here.  So heads come here from three per key head on: three images, 5190 tokens, 28 heads on 4 key heads:
// 13 us from the query to the pieces with a token per lane, 5 here; one of 7426 tokens 14 and 9.
// NB: blocks of eight tokens.  SMEM: keys and query are in shared memory (else a unit is one block).
template <typename T, int NB, bool SMEM>
__device__ __forceinline__ void group_piece(const Batch &bt, const ImgDesc &im, const uint8_t *kh, size_t kstride, const double *q,
                                            bool use_query, int nr, int j0, int r0, int n, int g) {
  constexpr int CH = NB <= 2 ? 2 : 1;                    // chains per block: a multiply takes 27 clocks, one can start every 16
  if constexpr (SMEM) {
    __builtin_assume(__isShared(kh));
    __builtin_assume(__isShared(q));
  }
  const int lane = threadIdx.x & 31, m = lane >> 2, c = lane & 3;
  double l[NB][2];
#pragma unroll
  for (int b = 0; b < NB; ++b) l[b][0] = l[b][1] = 0.0;
  if (use_query) {
    float odd[NB];
    double acc[NB][CH][2];
    const uint8_t *kr[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      odd[b] = 0.f;
#pragma unroll
      for (int h = 0; h < CH; ++h) acc[b][h][0] = acc[b][h][1] = 0.0;
      kr[b] = kh + (size_t)min(b * 8 + m, n - 1) * kstride + 2 * c * sizeof(T);
    }
    const double *qr = q + (size_t)min(m, nr - 1) * bt.d_h + 2 * c;
#pragma unroll 2
    for (int k0 = 0; k0 < bt.d_h; k0 += 8) {
      const bool in = sizeof(T) == 2 || k0 + 2 * c < bt.d_h;       // (fp32 head widths are multiples of four)
      const double2 x = in ? *reinterpret_cast<const double2 *>(qr + k0) : make_double2(0.0, 0.0);
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        Pair<T> k = {};
        if (in) k.load(kr[b] + (size_t)k0 * sizeof(T));
        double a0, a1;
        k.widen(a0, a1);
        k.see(odd[b]);
        asm("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(acc[b][0][0]), "+d"(acc[b][0][1]) : "d"(a0), "d"(x.x));
        asm("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(acc[b][CH - 1][0]), "+d"(acc[b][CH - 1][1]) : "d"(a1), "d"(x.y));
      }
    }
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      odd[b] += __shfl_xor_sync(0xffffffffu, odd[b], 1);
      odd[b] += __shfl_xor_sync(0xffffffffu, odd[b], 2);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const double v = (CH == 2 ? acc[b][0][e] + acc[b][CH - 1][e] : acc[b][0][e]) * kWidenScale;
        l[b][e] = __hiloint2double(__double2hiint(v) | __float_as_int(odd[b]), __double2loint(v));
      }
    }
  }
  double mx[2] = {-1.0e300, -1.0e300}, sum[2] = {0.0, 0.0};
#pragma unroll
  for (int b = 0; b < NB; ++b)
    if (b * 8 + m < n) {
#pragma unroll
      for (int e = 0; e < 2; ++e) mx[e] = max_by_bits(mx[e], l[b][e]);
    }
#pragma unroll
  for (int o = 4; o < 32; o <<= 1)
#pragma unroll
    for (int e = 0; e < 2; ++e) mx[e] = max_by_bits(mx[e], __shfl_xor_sync(0xffffffffu, mx[e], o));
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const double2 x = exp_two(l[b][0] - mx[0], l[b][1] - mx[1]);
    if (b * 8 + m < n) {
      double *E = im.E + (size_t)(j0 + 2 * c) * im.N + r0 + b * 8 + m;
      sum[0] += x.x;
      sum[1] += x.y;
      if (2 * c < nr) E[0] = x.x;
      if (2 * c + 1 < nr) E[im.N] = x.y;
    }
  }
#pragma unroll
  for (int o = 4; o < 32; o <<= 1)
#pragma unroll
    for (int e = 0; e < 2; ++e) sum[e] += __shfl_xor_sync(0xffffffffu, sum[e], o);
#pragma unroll
  for (int e = 0; e < 2; ++e)
    if (m == 0 && 2 * c + e < nr) *reinterpret_cast<double2 *>(piece_at(im, j0 + 2 * c + e, g)) = make_double2(mx[e], sum[e]);
}

// QUERY: the global query in shared memory; GROUP: heads through group_piece (a kernel of its own: in one, either path has
// fewer registers).
template <typename T, bool QUERY, bool GROUP>
__global__ void __launch_bounds__(kTokThreads, 2) k_tokens(const __grid_constant__ Batch bt, const TokCfg cfg, const __grid_constant__ TokUnits un, uint64_t row_policy, int what) {
  using D = typename DistOf<T>::type;
  using rn_t = typename D::rn_t;
  constexpr int V = Vec<T>::N;
  TL_SCOPE(bt.img[0], 1);
  const int lane = threadIdx.x & 31;
  const bool norms = threadIdx.x < kTokGroup;
  const int n_kvh = bt.n_kvh, d_h = bt.d_h, n_rep = bt.n_qh / n_kvh, rpp = cfg.rpp;
  extern __shared__ __align__(16) uint8_t smem[];
  const int ks = tok_key_stride(bt.d_k * (int)sizeof(T));
  uint8_t *s_key = smem + (size_t)kTokWarps * cfg.nbuf * cfg.chunk;   // [2][rpp][ks], behind the row buffers
  double *s_q = reinterpret_cast<double *>(s_key + (size_t)2 * cfg.keys * rpp * ks);     // [n_qh][d_h] global query
  double(*s_acc)[32] = reinterpret_cast<double(*)[32]>(s_q + (QUERY ? bt.n_qcols : 0));  // [kTokWarps tok_warp_rows(rpp)][32] parts of the sums of squares
  __shared__ uint64_t s_rbar[kTokWarps][kTokMaxBuf], s_kbar[2];
  __shared__ int s_abort, s_query;                                    // s_query: the global queries are complete
  if (lane == 0) {
    const int w = threadIdx.x >> 5;
    if (w < kTokWarps) {
      for (int i = 0; i < kTokMaxBuf; ++i) mbar_init(&s_rbar[w][i], 1);
    } else if (w < kTokWarps + 2) mbar_init(&s_kbar[w - kTokWarps], 1);
    else if (w == kTokWarps + 2) { s_query = 0; s_abort = 0; }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // units of this CTA: neighbours, so that it meets few images (each brings another query)
  const int cta = blockIdx.x, u0 = cta * un.per + min(cta, un.extra), u1 = u0 + un.per + (cta < un.extra);
  auto image_of = [&](int u, int b) { while (u >= un.first[b + 1]) ++b; return b; };

  if (norms) {
    const int w = threadIdx.x >> 5, t = threadIdx.x;
    uint8_t *s_rows = smem + (size_t)w * cfg.nbuf * cfg.chunk;        // this warp's row buffers
    double(*s_part)[32] = s_acc + tok_warp_rows(rpp) * w;   // parts of the sums of squares of its rows of a unit
    // the stream of this warp's row chunks, ahead of their use: unit, next row, rows left of the unit, chunk of the row
    int lu = u0 - 1, lb = 0, lrows = 0, lc = 0, islot = 0, ldealt = 0;
    const uint8_t *lsrc = nullptr;
    size_t lstep = 0;
    const int last = bt.d * (int)sizeof(T) - (cfg.nchunk - 1) * cfg.chunk;   // bytes of a row's last chunk
    auto issue_row = [&]() {                            // lane 0: the next chunk of the stream into its buffer
      while (lrows == 0) {
        if (++lu >= u1) { lu = u1; return; }
        lb = image_of(lu, lb);
        const ImgDesc &im = bt.img[lb];
        const int r0 = (lu - un.first[lb]) * rpp, n = min(rpp, im.N - r0);
        if (im.flags & PACT_FLAG_NO_NORM) continue;
        const int first = (w - ldealt) & (kTokWarps - 1);   // this warp's first row of the unit
        ldealt += n;
        if (n <= first) continue;
        lrows = (n - first + kTokWarps - 1) / kTokWarps;
        lsrc = reinterpret_cast<const uint8_t *>(reinterpret_cast<const T *>(im.H) + (size_t)(im.vis_start + r0 + first) * im.ldH);
        lstep = (size_t)im.ldH * kTokWarps * sizeof(T);
      }
      const int bytes = lc == cfg.nchunk - 1 ? last : cfg.chunk;
      mbar_arrive_expect_tx(&s_rbar[w][islot], bytes);
      bulk_load_hint(s_rows + (size_t)islot * cfg.chunk, lsrc + (size_t)lc * cfg.chunk, bytes, &s_rbar[w][islot], row_policy);
      if (++islot == cfg.nbuf) islot = 0;
      if (++lc == cfg.nchunk) { lc = 0; lsrc += lstep; --lrows; }
    };
    // One buffer per warp until k_qsum is done, all of them from then on: with more from the start this stream leaves k_qsum a
    // third of the memory rate and the logits begin late (16 images of 2916 tokens: at 37 us), with none the memory
    // idles towards the end of k_qsum.
    // (A launch without norms asks for no row: nobody would wait for it, and the CTA could end with the copy under way.)
    if (lane == 0 && (what & kTokNorms)) issue_row();
    bool all = false;
    int slot = 0, b = 0, dealt = 0;                     // buffer that is next; rows of the units before
    uint32_t par = 0;                                   // parity of each buffer's barrier
    for (int u = u0; u < u1 && (what & kTokNorms); ++u) {
      b = image_of(u, b);
      const ImgDesc &im = bt.img[b];
      const int r0 = (u - un.first[b]) * rpp, n = min(rpp, im.N - r0);
      if (im.flags & PACT_FLAG_NO_NORM) {
        for (int r = t; r < n; r += kTokGroup) im.nrm[r0 + r] = 1.0;
        continue;
      }
      const int first = (w - dealt) & (kTokWarps - 1);
      dealt += n;
      int mine = 0;
      for (int r = first; r < n; r += kTokWarps, ++mine) {
        double a0 = 0.0, a1 = 0.0;
        for (int c = 0; c < cfg.nchunk; ++c) {
          if (!mbar_wait_warp(&s_rbar[w][slot], (par >> slot) & 1)) {
            s_abort = 1;
            goto norms_end;
          }
          par ^= 1u << slot;
          const uint4 *row = reinterpret_cast<const uint4 *>(s_rows + (size_t)slot * cfg.chunk);
          const int nv = min(cfg.chunk, bt.d * (int)sizeof(T) - c * cfg.chunk) / 16;
          int v = lane;
          for (; v + 96 < nv; v += 128) {
            uint4 x[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) x[k] = row[v + 32 * k];
            sumsq_accumulate<T>(x[0], a0); sumsq_accumulate<T>(x[1], a1);
            sumsq_accumulate<T>(x[2], a0); sumsq_accumulate<T>(x[3], a1);
          }
          for (; v < nv; v += 32) sumsq_accumulate<T>(row[v], a0);
          __syncwarp();
          if (lane == 0) {
            issue_row();
            if (!all && *const_cast<volatile int *>(&s_query)) {
              all = true;
              for (int k = 1; k < cfg.nbuf; ++k) issue_row();
            }
          }
          if (++slot == cfg.nbuf) slot = 0;
        }
        s_part[mine][lane] = a0 + a1;
      }
      __syncwarp();
      finish_row_sums(s_part, mine, [&](int j, double s) { im.nrm[r0 + first + j * kTokWarps] = sqrt(s); });
    }
norms_end:
    pdl_wait();
  } else {
    const int team = threadIdx.x >= kTokGroup + kTokTeam, t = threadIdx.x & (kTokTeam - 1), w = t >> 5;   // within the team
    const int P = rpp <= 8 ? 4 : rpp <= 16 ? 2 : 1;     // lanes per token
    uint8_t *s_mine = s_key + (size_t)team * rpp * ks;
    auto issue_keys = [&](int u) {                      // lane 0 of every warp: its share of the scoring keys of unit u
      if (u >= u1 || *const_cast<volatile int *>(&s_abort)) return;
      const int b = image_of(u, 0);
      const ImgDesc &im = bt.img[b];
      const int r0 = (u - un.first[b]) * rpp, n = min(rpp, im.N - r0);
      if (w == 0) mbar_arrive_expect_tx(&s_kbar[team], n * bt.d_k * (int)sizeof(T));
      for (int r = w; r < n; r += kTeamWarps)
        bulk_load(s_mine + (size_t)r * ks, reinterpret_cast<const T *>(im.Ke) + (size_t)(r0 + r) * im.ldKe, bt.d_k * (int)sizeof(T), &s_kbar[team]);
    };
    if (cfg.keys && (what & kTokLogits) && lane == 0) issue_keys(u0 + team);
    auto sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "n"(kTokTeam) : "memory"); };
    auto sync_both = []() { asm volatile("bar.sync 3, %0;" ::"n"(kTokGroup) : "memory"); };
    if (what & kTokInit) {                                      // what later kernels accumulate into
      const int gt = blockIdx.x * kTokGroup + threadIdx.x - kTokGroup, gs = gridDim.x * kTokGroup;
      for (int i = 0; i < bt.B; ++i) {
        const ImgDesc &im = bt.img[i];
        for (int r = gt; r < im.Np; r += gs) { im.rho_fix[r] = 0ull; im.csize[r] = 0; im.cticket[r] = 0; }
        for (int wd = gt; wd < im.Wp; wd += gs) { im.cmask[wd] = 0u; im.rmask[wd] = 0u; im.rtick[wd] = 0; }
        for (int r = gt; r < im.N; r += gs) im.best[r] = kBestInit;
        uint4 *tab = reinterpret_cast<uint4 *>(im.cnt_cb);
        for (int r = gt; r < im.Np * (im.nbp / 8); r += gs) tab[r] = make_uint4(0u, 0u, 0u, 0u);
        for (int r = gt; r < kHistBins; r += gs) im.ghist[r] = 0;
        if (gt < kCntInts) im.cnt[gt] = 0;
      }
    }
    int b = 0, loaded = -1;                             // loaded: image whose query is in s_q
    uint32_t par = 0;
    if (!(what & kTokLogits)) {
      pdl_wait();
      s_query = 1;
      pdl_trigger();
    }
    const auto has_query = [&](int i) { return !(bt.img[i].flags & PACT_FLAG_NORM_ONLY) && bt.img[i].Q != nullptr; };
    for (int p0 = u0; p0 < u1 && (what & kTokLogits); p0 += 2) {   // a unit for each team, of the images b and b2
      b = image_of(p0, b);
      const int b2 = p0 + 1 < u1 ? image_of(p0 + 1, b) : b, mu = p0 + team, mb = team ? b2 : b;
      const ImgDesc &im = bt.img[mb];
      const int g = mu - un.first[mb], r0 = g * rpp, n = mu < u1 ? min(rpp, im.N - r0) : 0;
      const bool use_query = has_query(mb), need_b = QUERY && has_query(b), need_b2 = QUERY && has_query(b2);
      const double *qg_b = bt.img[b].qg, *qg_b2 = bt.img[b2].qg;
      const uint8_t *keys = cfg.keys ? s_mine : reinterpret_cast<const uint8_t *>(reinterpret_cast<const T *>(im.Ke) + (size_t)r0 * im.ldKe);
      const size_t kstride = cfg.keys ? (size_t)ks : (size_t)im.ldKe * sizeof(T);
      if (n > 0) {
        if (cfg.keys && !mbar_wait_warp_unless(&s_abort, &s_kbar[team], par)) s_abort = 1;   // (on through the teams' barriers, but without copies)
        par ^= 1u;
        if (im.Kc) {                                     // inverse norms: eight lanes per row, four rows at a time
          const bool same = cfg.keys && im.Kc == im.Ke;
          const uint8_t *kc = same ? keys : reinterpret_cast<const uint8_t *>(reinterpret_cast<const T *>(im.Kc) + (size_t)r0 * im.ldKc);
          const size_t cs = same ? kstride : (size_t)im.ldKc * sizeof(T);
          const int nv = bt.d_k / V;
          for (int rb = w * 4; rb < n; rb += kTeamWarps * 4) {
            const int r = rb + lane / 8;
            double a = 0.0;
            if (r < n) {
#pragma unroll 4
              for (int v = lane & 7; v < nv; v += 8) sumsq_accumulate<T>(*(reinterpret_cast<const uint4 *>(kc + (size_t)r * cs) + v), a);
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            if (r < n && (lane & 7) == 0) rn_tok<D>(im)[r0 + r] = (rn_t)inv_norm(a);
          }
        }
      }
      if (p0 == u0) {
        pdl_wait();                                      // the global queries are complete
        s_query = 1;
        pdl_trigger();
      }
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {
        if (h ? need_b2 && loaded != b2 : need_b && loaded != b) {   // (the same for both teams)
          if (loaded >= 0) sync_both();
          loaded = h ? b2 : b;
          const double *qg = h ? qg_b2 : qg_b;
#pragma unroll 4
          for (int c = 2 * (threadIdx.x - kTokGroup); c < bt.n_qcols; c += 2 * kTokGroup) {
            double2 x;
            ld_cg_f64x2(qg + c, x.x, x.y);
            *reinterpret_cast<double2 *>(s_q + c) = x;
          }
          sync_both();
        }
        if (h != team || n == 0) continue;
        const double *q = QUERY ? s_q : im.qg;
        if constexpr (GROUP) {
          const int nblk = (n_rep + 7) / 8;              // blocks of up to eight query heads per key head
          const bool in_smem = QUERY && cfg.keys;
          for (int it = w; it < n_kvh * nblk; it += kTeamWarps) {
            const int kv = it / nblk, j = (it - kv * nblk) * 8, j0 = kv * n_rep + j, nr = min(8, n_rep - j);
            const uint8_t *kh = keys + (size_t)kv * d_h * sizeof(T);
            if (!in_smem) group_piece<T, 1, false>(bt, im, kh, kstride, q + (size_t)j0 * d_h, use_query, nr, j0, r0, n, g);   // (n <= kMinPiece)
            else if (n <= 8) group_piece<T, 1, true>(bt, im, kh, kstride, q + (size_t)j0 * d_h, use_query, nr, j0, r0, n, g);
            else if (n <= 16) group_piece<T, 2, true>(bt, im, kh, kstride, q + (size_t)j0 * d_h, use_query, nr, j0, r0, n, g);
            else if (n <= 24) group_piece<T, 3, true>(bt, im, kh, kstride, q + (size_t)j0 * d_h, use_query, nr, j0, r0, n, g);
            else group_piece<T, 4, true>(bt, im, kh, kstride, q + (size_t)j0 * d_h, use_query, nr, j0, r0, n, g);
          }
        } else {
          const uint8_t *krow = keys + (size_t)min(lane & (32 / P - 1), n - 1) * kstride;
          for (int kv = w; kv < n_kvh; kv += kTeamWarps) {
            const uint8_t *kh = krow + (size_t)kv * d_h * sizeof(T);
            if (n_rep == 2) head_piece<T, 2>(bt, im, kh, q + (size_t)2 * kv * d_h, use_query, P, 2 * kv, r0, n, g);
            else head_piece<T, 1>(bt, im, kh, q + (size_t)kv * d_h, use_query, P, kv, r0, n, g);
          }
        }
      }
      if (cfg.keys && mu + 2 < u1) {
        sync();                                          // the keys have been read
        if (lane == 0) issue_keys(mu + 2);
      }
    }
  }
  __syncthreads();
  if (threadIdx.x < 32 && s_abort) {
    land_copies(&s_rbar[0][0], kTokWarps * kTokMaxBuf);
    land_copies(s_kbar, 2);
    if (threadIdx.x == 0)
      for (int i = 0; i < bt.B; ++i) atomicMin(&bt.img[i].cnt[PACT_CNT_STATUS], (int)PACT_ERR_TIMEOUT);
  }
}

// ---- Eq. 2, second half: merge the pieces (M = max, Z = sum S_g exp(M_g - M), fixed order), scores --------
// grid (ceil(maxN / 256) rounded up to CL, B) in clusters of CL CTAs, 512 threads: two per token, each with half of the heads.
// A cluster merges all G pieces for itself: its CTAs share out the heads (four or fewer per CTA up to 32 heads), the warps of a
// CTA the heads and the pieces of a head, four loads per lane in flight; the results go to every CTA of the cluster.  What
// turns a term into a share, exp(M_g - M) / (Z n_qh), is formed once per piece and head of the CTA's tokens.  with_hist:
// every score also counts in the histogram of its top key bits, the first level of the threshold selection.
// EP: terms of a token that a thread asks for before the merge (all of its half up to four heads, else eight, with 128 registers:
// at 64 some are spilled, 1 us of a call with 28 heads, although the CTA could then begin beside k_tokens).
// Bound by latency and by the instructions it takes: what does not depend on k_tokens comes before the wait for it (a microsecond of
// divisions), a value that has to be spilled while it is loaded costs its whole latency, and two exponentials at a time come
// from one copy of the code.  With every CTA merging all heads, 286 pieces of 28 heads took 22 us, 9 now; three images with
// 28 heads (5190 tokens) 13 us, 9 now; four heads 4.9 us, 4.1 now.  (Going through the code once before the wait, to have the
// instructions in the cache, halved the time behind the wait and cost as much before it.)
constexpr int kScoreTok = 256;                          // tokens per CTA
constexpr int kScoreThreads = 2 * kScoreTok;
constexpr int kScoreWarps = kScoreThreads / 32;
constexpr int kScoreHeads = 32;                         // heads whose factors are in shared memory at a time
constexpr int kScorePieces = kScoreTok / kMinPiece + 1; // most pieces that a CTA's tokens belong to
constexpr int kScoreMaxCl = 8;

template <int EP>
__global__ void __launch_bounds__(kScoreThreads, EP > 2 ? 1 : 2) k_scores(const __grid_constant__ Batch bt, int rpp, int with_hist, int CL) {
  const ImgDesc &im = bt.img[blockIdx.y];
  TL_SCOPE(im, 2);
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int N = im.N, n_qh = bt.n_qh, i0 = blockIdx.x * kScoreTok, rank = blockIdx.x % CL;
  if (i0 - rank * kScoreTok >= N) {                     // no CTA of the cluster has tokens
    pdl_wait();
    return;
  }
  __shared__ double sM[256], sInv[256];
  __shared__ double pmx[kScoreWarps], pz[kScoreWarps];
  __shared__ double s_fac[kScorePieces * kScoreHeads], s_half[kScoreTok];
  // pieces of the CTA's tokens: np from g0 on; this thread's token, its half of the heads and its factor of the first 32 heads
  const int G = (N + rpp - 1) / rpp, g0 = i0 / rpp, np = i0 < N ? (min(N, i0 + kScoreTok) - 1) / rpp - g0 + 1 : 0;
  const int tok = t & (kScoreTok - 1), half = t / kScoreTok, i = i0 + tok, tok_piece = i / rpp - g0;
  const int nh0 = min(n_qh, kScoreHeads), per0 = (nh0 + 1) >> 1, jb = half * per0, je = i < N ? min(nh0, jb + per0) : jb;
  const double *e_src = im.E + (size_t)jb * N + i;
  const int f_head = t / max(np, 1), f_piece = t - f_head * np;
  const double *m_src = t < np * nh0 ? piece_at(im, f_head, g0 + f_piece) : im.part;
  const double *nrm_src = i < N ? im.nrm + i : im.nrm;
  // heads of this CTA, warps per head, pieces of this warp: 32 sub + lane, + step, ...
  const int hpc = (n_qh + CL - 1) / CL, j_lo = rank * hpc, nh = max(0, min(hpc, n_qh - j_lo));
  int wph = 1;
  while (wph < kScoreWarps && hpc * wph * 2 <= kScoreWarps) wph *= 2;
  const int hpp = kScoreWarps / wph, wh = w / wph, sub = w - wh * wph, step = 32 * wph;   // heads per pass
  constexpr int U = 4;
  const int nbatch = (G + U * step - 1) / (U * step);
  if (CL > 1) cluster_sync();                           // every CTA of the cluster runs before one stores to another
  double e_pre[EP], nrm_i = 0.0, m_pre = 0.0, s = 0.0;
  pdl_wait();
  pdl_trigger();
  for (int p = 0; p < hpc; p += hpp) {
    const bool mine = p + wh < nh;
    const int j = j_lo + p + wh;
    auto load = [&](int b, double (&pm)[U], double (&ps)[U]) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int h = sub * 32 + lane + step * (U * b + u);
        pm[u] = -1.0e300;
        ps[u] = 0.0;
        if (mine && h < G) ld_cg_f64x2(piece_at(im, j, h), pm[u], ps[u]);
      }
    };
    double pm0[U], ps0[U], m = -1.0e300;
    load(0, pm0, ps0);
    if (p == 0) {                                       // the token's terms and the first factor's piece arrive during the merge
#pragma unroll
      for (int u = 0; u < EP; ++u) e_pre[u] = ld_cg_f64(jb + u < je ? e_src + (size_t)u * N : im.E);
      nrm_i = ld_cg_f64(nrm_src);
      m_pre = ld_cg_f64(m_src);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) m = pm0[u] > m ? pm0[u] : m;
    for (int b = 1; b < nbatch; ++b) {
      double pm[U], ps[U];
      load(b, pm, ps);
#pragma unroll
      for (int u = 0; u < U; ++u) m = pm[u] > m ? pm[u] : m;
    }
    m = warp_max(m);
    if (wph > 1) {
      if (lane == 0) pmx[w] = m;                        // (then all heads of the CTA are in one pass)
      __syncthreads();
      if (mine)
        for (int k = 0; k < wph; ++k) { const double o = pmx[w - sub + k]; m = o > m ? o : m; }
    }
    double z = 0.0;
#pragma unroll
    for (int u = 0; u < U; u += 2)
      if (step * u < G) {                               // (an empty slot adds 0 * exp(-huge) = 0)
        const double2 x = exp_two(pm0[u] - m, pm0[u + 1] - m);
        z += ps0[u] * x.x;
        z += ps0[u + 1] * x.y;
      }
    for (int b = 1; b < nbatch; ++b) {
      double pm[U], ps[U];
      load(b, pm, ps);
#pragma unroll
      for (int u = 0; u < U; u += 2) {
        const double2 x = exp_two(pm[u] - m, pm[u + 1] - m);
        z += ps[u] * x.x;
        z += ps[u + 1] * x.y;
      }
    }
    z = warp_sum(z);
    if (wph > 1) {
      if (lane == 0) pz[w] = z;
      __syncthreads();
      z = 0.0;
      for (int k = 0; k < wph; ++k) z += pz[w - sub + k];
    }
    if (mine && sub == 0 && lane < CL) {                // to every CTA of the cluster
      const double inv = 1.0 / (z * (double)n_qh);
      if (CL > 1) {
        st_cluster_f64(&sM[j], lane, m);
        st_cluster_f64(&sInv[j], lane, inv);
      } else {
        sM[j] = m;
        sInv[j] = inv;
      }
    }
  }
  if (CL > 1) cluster_sync();
  // (heads EP .. of the half; the registers are not free earlier)
  double e_more[EP];
  if (EP > 2) {
#pragma unroll
    for (int u = 0; u < EP; ++u) e_more[u] = jb + EP + u < je ? ld_cg_f64(e_src + (size_t)(EP + u) * N) : 0.0;
  }
  s = 0.0;
  for (int h0 = 0; h0 < n_qh; h0 += kScoreHeads) {
    const int nhh = min(kScoreHeads, n_qh - h0);
    __syncthreads();
    for (int f = t; f < np * nhh; f += kScoreThreads) { // factor f: head h0 + f / np, piece f % np
      const int jf = h0 + f / np;
      const double mg = h0 == 0 && f == t ? m_pre : ld_cg_f64(piece_at(im, jf, g0 + f % np));
      s_fac[f] = exp(mg - sM[jf]) * sInv[jf];
    }
    __syncthreads();
    if (i < N) {
      const double *fac = s_fac + tok_piece;
      if (h0 == 0) {
#pragma unroll
        for (int j = 0; j < EP; ++j)
          if (jb + j < je) s = fma(e_pre[j], fac[(jb + j) * np], s);
        if (EP > 2) {
#pragma unroll
          for (int j = 0; j < EP; ++j)
            if (jb + EP + j < je) s = fma(e_more[j], fac[(jb + EP + j) * np], s);
        }
      } else {
        const int per = (nhh + 1) >> 1, hi = min(nhh, half * per + per);
        for (int j = half * per; j < hi; ++j) s = fma(ld_cg_f64(im.E + (size_t)(h0 + j) * N + i), fac[j * np], s);
      }
    }
  }
  if (half == 1) s_half[tok] = s;
  __syncthreads();
  if (half == 1 || i >= N) return;
  const float sf = (float)((s + s_half[tok]) * nrm_i);
  im.score[i] = sf;
  if (im.score_user) im.score_user[i] = sf;
  if (with_hist) atomicAdd(&im.ghist[key_bin(score_key(sf))], 1);
}

// ---- Eq. 3-4 in the whole step: threshold, ordered compaction, survivor keys (Eq. 7) ------------------------
// grid (X, B), 512 threads, one CTA per SM; dynamic smem: N sort keys where a thread's share does not fit its registers.
// CTA x owns the tokens [x tpc, (x + 1) tpc).  Every CTA selects the threshold itself (identical in all of them),
// counts the survivors before its tokens, writes keep flags, lists and slots of its tokens and copies the clustering keys
// of its survivors to their rows of K'.
constexpr int kSelThreads = 512;
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kHistPerThread = kHistBins / kSelThreads;
constexpr size_t kSelKeyBytes = 96 * 1024;     // most shared memory for sort keys or rows
constexpr int kSelBits = 10;                  // key bits per pass of the selection below the first-level histogram
constexpr int kSelFew = 64;                   // candidates that are ranked one against another
static_assert((1 << kSelBits) == 2 * kSelThreads && kHistPerThread == 8 && kSelWarps <= 32, "bins per thread, a warp total per lane");

struct SelShared {
  int hist[1 << kSelBits];                     // keys of the threshold's bin by the bits below, and one key of each
  uint32_t one[1 << kSelBits];
  int wtot[kSelWarps], wtot2[kSelWarps];
  uint32_t few[kSelFew];
  uint32_t s_prefix;
  int s_k, s_bin, s_cnt, s_less, s_few;
  int own_tok[kSelThreads], own_slot[kSelThreads];
};

// Warp-inclusive sum.
__device__ __forceinline__ int warp_scan(int v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  return v;
}

// The bins of a pass are in sh.hist: the one with rank k among them, by all threads: its digit to sh.s_bin, the keys in it to
// sh.s_cnt, the rank in it to sh.s_k.  The bins are zero again afterwards.
__device__ __forceinline__ void find_digit(int k, SelShared &sh) {
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  int2 *mine = reinterpret_cast<int2 *>(sh.hist) + t;
  const int2 c = *mine;
  *mine = make_int2(0, 0);
  const int incl = warp_scan(c.x + c.y, lane);
  if (lane == 31) sh.wtot[w] = incl;
  __syncthreads();
  const int below = incl - c.x - c.y + (int)__reduce_add_sync(0xffffffffu, lane < w ? sh.wtot[lane] : 0);
  if (below <= k && k < below + c.x + c.y) {            // exactly one thread: the candidates number more than k
    const bool second = k >= below + c.x;
    sh.s_bin = 2 * t + second;
    sh.s_cnt = second ? c.y : c.x;
    sh.s_k = k - below - (second ? c.x : 0);
  }
  __syncthreads();
}

// The threshold by radix passes over the bits below `hi`, kSelBits at a time: rank k among the keys with these upper bits, `less`
// keys of the first-level bin before them.  (skey: the keys in shared memory, or null.  A call: it hardly ever runs.)
__device__ __noinline__ void radix_threshold(const float *score, const uint32_t *skey, int N, int hi, uint32_t prefix, int k, int less, SelShared &sh) {
  const int t = threadIdx.x;
  for (; hi > 0; hi -= kSelBits) {
    const int lo = hi > kSelBits ? hi - kSelBits : 0;
    const uint32_t dmask = (1u << (hi - lo)) - 1u;
    const uint32_t above = hi >= 32 ? 0u : ~((1u << hi) - 1u);          // bits already fixed
    __syncthreads();
    for (int i = t; i < N; i += kSelThreads) {
      const uint32_t kk = skey ? skey[i] : score_key(__ldcg(score + i));
      if ((kk & above) == (prefix & above)) atomicAdd(&sh.hist[(kk >> lo) & dmask], 1);
    }
    __syncthreads();
    find_digit(k, sh);
    less += k - sh.s_k;                                 // keys under the prefix that come before the digit
    k = sh.s_k;
    prefix |= (uint32_t)sh.s_bin << lo;
  }
  if (t == 0) {
    sh.s_less = less;
    sh.s_prefix = prefix;
  }
  __syncthreads();
}

// KPT > 0: thread t holds the keys t, t + 512, ... in registers (N <= 512 KPT); KPT == 0: keys from shared memory (IN_SMEM)
// or re-read from the scores.  (A kernel for each case: the code runs once, from a cold instruction cache.)
// The histogram of the keys' top bits, filled by k_scores, gives the bin of the threshold, the (m_target + 1)-th smallest
// key, and its rank in the bin (sixteen bins per factor of two: some hundred keys of 7290); a pass over the next ten bits
// of those mostly leaves one key, which has been put down beside the count, else a few, which are ranked one against another.
// Bound by latency and by the instructions of 16 warps, four clocks each, most of them run once: 1024 threads were 0.5 us slower
// (eight clocks), ranking all keys of the bin by counting 3 us, and a pass through the code before the wait, for the
// instruction cache, cost what it gave.  The rows of the own tokens wait in shared memory when it is known which survive; scores,
// histogram and norms come in one trip.  From the end of k_scores: one image of 7290 8.0 us -> 6.7, four of 16384 (16 keys per
// thread from shared memory, three passes over them) 22 -> 15.  Above 16384 tokens, with one CTA per SM where there were two (events
// around the kernel): 24577 29 us -> 18, 65536 60 -> 41, 131072 107 -> 72; the own tokens then go in rounds of 512.
template <typename T, int KPT, bool IN_SMEM>
__global__ void __launch_bounds__(kSelThreads, 1) k_select(const __grid_constant__ Batch bt, int pre) {
  using D = typename DistOf<T>::type;
  constexpr int V = Vec<T>::N, KR = KPT > 0 ? KPT : 1;
  const ImgDesc &im = bt.img[blockIdx.y];
  TL_SCOPE(im, 3);
  extern __shared__ __align__(16) uint8_t sel_smem[];
  uint32_t *skey = reinterpret_cast<uint32_t *>(sel_smem);     // KPT == 0: the keys; else (pre) the rows of the own tokens
  __shared__ SelShared sh;
  __shared__ uint64_t s_bar;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int N = im.N, X = gridDim.x, x = blockIdx.x, m_t = im.m_target;
  const int tpc = (N + X - 1) / X, tok0 = min(N, x * tpc), ntok = min(N, tok0 + tpc) - tok0;
  const int nv = bt.d_k / V, rowb = nv * 16, npre = KPT > 0 && pre ? ntok : 0;
  const T *Kc = reinterpret_cast<const T *>(im.Kc);
  T *Kp = reinterpret_cast<T *>(im.Kp);
  const float *score = im.score;
  const int4 *hist = reinterpret_cast<const int4 *>(im.ghist) + 2 * t;
  const auto key_at = [&](int i) -> uint32_t { return IN_SMEM ? skey[i] : score_key(__ldcg(score + i)); };
  reinterpret_cast<int2 *>(sh.hist)[t] = make_int2(0, 0);
  // the keys of the own tokens, before it is known which of them survive (they are an input)
  if (w == 1 && npre > 0) {
    if (lane == 0) {
      mbar_init(&s_bar, 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      mbar_arrive_expect_tx(&s_bar, npre * rowb);
    }
    __syncwarp();
    for (int r = lane; r < npre; r += 32) bulk_load(sel_smem + (size_t)r * rowb, Kc + (size_t)(tok0 + r) * im.ldKc, rowb, &s_bar);
  }
  uint32_t kreg[KR], own, tau;
  typename D::rn_t rn_own;
  int bin, rank, less;
  if (t == 0) { sh.s_bin = -1; sh.s_k = 0; sh.s_few = 0; }
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  {
    const int4 ha = __ldcg(hist), hb = __ldcg(hist + 1);   // bins [8 t, 8 t + 8)
    float sc[KR];
    if (KPT > 0) {
#pragma unroll
      for (int u = 0; u < KR; ++u) sc[u] = __ldcg(score + min(t + kSelThreads * u, N - 1));
    }
    const float so = __ldcg(score + min(tok0 + t, N - 1));
    rn_own = __ldcg(rn_tok<D>(im) + min(tok0 + t, N - 1));
    const int suma = ha.x + ha.y + ha.z + ha.w, sum = suma + (hb.x + hb.y + hb.z + hb.w), incl = warp_scan(sum, lane);
    if (lane == 31) sh.wtot[w] = incl;
    own = score_key(so);
    if (KPT > 0) {
#pragma unroll
      for (int u = 0; u < KR; ++u) kreg[u] = t + kSelThreads * u < N ? score_key(sc[u]) : 0u;   // (never in a bin but 0, never kept)
    } else if (IN_SMEM) {
#pragma unroll 8
      for (int i = t; i < N; i += kSelThreads) skey[i] = score_key(__ldcg(score + i));
    }
    __syncthreads();
    const int below = incl - sum + (int)__reduce_add_sync(0xffffffffu, lane < w ? sh.wtot[lane] : 0);   // keys in the bins before this thread's
    if (below <= m_t && m_t < below + sum) {            // exactly one thread, unless a wait ran out
      const bool upper = m_t - below >= suma;
      const int4 h = upper ? hb : ha;
      const int k = m_t - below - (upper ? suma : 0), u = (k >= h.x) + (k >= h.x + h.y) + (k >= h.x + h.y + h.z);
      sh.s_bin = 8 * t + (upper ? 4 : 0) + u;
      sh.s_k = k - (u > 0 ? h.x : 0) - (u > 1 ? h.y : 0) - (u > 2 ? h.z : 0);
    }
    __syncthreads();
    bin = sh.s_bin;
    rank = sh.s_k;
    tau = 0xffffffffu;                                  // (an inconsistent histogram: nothing is kept)
    less = 0;                                           // keys of the bin before the threshold
    if (bin > 0) {
      constexpr int lo = kHistShift - kSelBits;
      const uint32_t top = bin_first(bin) >> kHistShift;
      const auto count = [&](uint32_t key) {
        if (key >> kHistShift == top) {
          const int d = (key >> lo) & ((1 << kSelBits) - 1);
          atomicAdd(&sh.hist[d], 1);
          sh.one[d] = key;
        }
      };
      if (KPT > 0) {
#pragma unroll
        for (int u = 0; u < KR; ++u) count(kreg[u]);
      } else {
        for (int i = t; i < N; i += kSelThreads) count(key_at(i));
      }
      __syncthreads();
      find_digit(rank, sh);
      const int digit = sh.s_bin;
      less = rank - sh.s_k;
      tau = sh.one[digit];
      if (sh.s_cnt > 1) {
        const uint32_t prefix = bin_first(bin) | (uint32_t)digit << lo;
        const int k2 = sh.s_k;
        if (sh.s_cnt <= kSelFew) {
          const auto put = [&](uint32_t key) { if ((key ^ prefix) >> lo == 0u) sh.few[atomicAdd(&sh.s_few, 1)] = key; };
          if (KPT > 0) {
#pragma unroll
            for (int u = 0; u < KR; ++u) put(kreg[u]);
          } else {
            for (int i = t; i < N; i += kSelThreads) put(key_at(i));
          }
          __syncthreads();
          if (t < sh.s_cnt) {
            int l = 0, same = 0;
            for (int j = 0; j < sh.s_cnt; ++j) { l += sh.few[j] < sh.few[t]; same += sh.few[j] == sh.few[t]; }
            if (l <= k2 && k2 < l + same) { sh.s_prefix = sh.few[t]; sh.s_less = less + l; }   // (equal keys write the same)
          }
          __syncthreads();
        } else radix_threshold(score, IN_SMEM ? skey : nullptr, N, lo, prefix, k2, less, sh);
        less = sh.s_less;
        tau = sh.s_prefix;
      }
    } else if (bin == 0) {                              // the bin of all of the smallest keys, whatever their bits
      radix_threshold(score, IN_SMEM ? skey : nullptr, N, 32, 0u, rank, 0, sh);
      less = sh.s_less;
      tau = sh.s_prefix;
    }
  }
  TL_POINT(im, 7);

  // ---- survivors before the own tokens, then keep flags, lists, slots and keys of the own ones ----
  int nb = 0;
  if (KPT > 0) {
#pragma unroll
    for (int u = 0; u < KR; ++u) nb += t + kSelThreads * u < tok0 && kreg[u] >= tau;
  } else {
    for (int i = t; i < tok0; i += kSelThreads) nb += key_at(i) >= tau;
  }
  nb = __reduce_add_sync(0xffffffffu, nb);
  if (x == 0 && t == 0) {
    const int q = bin >= 0 ? N - (m_t - rank) - less : 0;   // all but the keys of lower bins and the smaller ones of its own
    im.cnt[PACT_CNT_Q] = q;
    im.cnt[PACT_CNT_M] = N - q;
  }
  int before0 = 0;                                      // survivors with a lower index than the round's tokens
  for (int c0 = 0; c0 < ntok; c0 += kSelThreads) {      // the own tokens, 512 at a time
    const int i = tok0 + c0 + t;
    const bool ok = c0 + t < ntok;
    const bool kp = ok && (c0 == 0 ? own : score_key(__ldcg(score + i))) >= tau;
    const unsigned bal = __ballot_sync(0xffffffffu, kp);
    if (lane == 0) {
      sh.wtot[w] = __popc(bal);
      if (c0 == 0) sh.wtot2[w] = nb;
    }
    __syncthreads();
    const int wt = lane < kSelWarps ? sh.wtot[lane] : 0, tot = __reduce_add_sync(0xffffffffu, wt);
    const int excl = __popc(bal & ((1u << lane) - 1u)) + (int)__reduce_add_sync(0xffffffffu, lane < w ? wt : 0);
    if (c0 == 0) before0 = __reduce_add_sync(0xffffffffu, lane < kSelWarps ? sh.wtot2[lane] : 0);
    if (ok) {
      const int pos = before0 + excl;                   // survivors with a lower index
      if (kp) { sh.own_tok[excl] = i; sh.own_slot[excl] = pos; }
      im.keep[i] = kp ? 1 : 0;
      if (im.keep_user) im.keep_user[i] = kp ? 1 : 0;
      if (kp) { im.kept_idx[pos] = i; im.slot[i] = pos; rn_kept<D>(im)[pos] = c0 == 0 ? rn_own : rn_tok<D>(im)[i]; }
      else { im.pruned_idx[i - pos] = i; im.slot[i] = -1 - (i - pos); }
    }
    __syncthreads();
    // the rows: those in shared memory by bulk copies, the others by sixteen lanes each with eight 16-byte loads in flight
    if (npre > 0) {
      const bool landed = mbar_wait_warp_or_report(&s_bar, 0, &im.cnt[PACT_CNT_STATUS]);
      if (!landed) land_copies(&s_bar, 1);              // (thread 0 waits for them, if its own wait ran out)
      if (landed && lane == 0) {
        for (int r = w; r < tot; r += kSelWarps)
          bulk_store(Kp + (size_t)sh.own_slot[r] * bt.d_k, sel_smem + (size_t)(sh.own_tok[r] - tok0) * rowb, rowb);
        bulk_store_wait();
      }
      break;                                            // (all of the own tokens are in this round)
    }
    for (int r = t >> 4; r < tot; r += kSelThreads / 8) {
      const int r2 = r + kSelThreads / 16 < tot ? r + kSelThreads / 16 : r;
      const uint4 *s0 = reinterpret_cast<const uint4 *>(Kc + (size_t)sh.own_tok[r] * im.ldKc), *s1 = reinterpret_cast<const uint4 *>(Kc + (size_t)sh.own_tok[r2] * im.ldKc);
      uint4 *d0 = reinterpret_cast<uint4 *>(Kp + (size_t)sh.own_slot[r] * bt.d_k), *d1 = reinterpret_cast<uint4 *>(Kp + (size_t)sh.own_slot[r2] * bt.d_k);
      for (int v = t & 15; v < nv; v += 64) {
        uint4 b0[4], b1[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (v + 16 * u < nv) { b0[u] = __ldg(s0 + v + 16 * u); b1[u] = __ldg(s1 + v + 16 * u); }
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (v + 16 * u < nv) { d0[v + 16 * u] = b0[u]; d1[v + 16 * u] = b1[u]; }
      }
    }
    before0 += tot;
    __syncthreads();                                    // own_tok / own_slot are rewritten by the next round
  }
}

// ---- Eq. 3-4 as a stage of its own (pact_prune): order statistic, ordered compaction ------------------

// N <= 512 KPT: grid (1), 512 threads, thread t holds the keys t, t + 512, ... in registers.  As k_select, but without a
// histogram to begin with: keys are taken relative to the smallest one, which spreads them evenly over the digits of the first
// pass (raw float bits of scores that span a few binades share most of their top bits), and the bits above the highest one in which
// two keys differ need no pass.  One CTA, bound by its instructions (four
// clocks each with 16 warps, eight with 32) and barriers: with the tokens of a thread next to one another in 1024 threads, radix passes
// until one key was left and flags and lists written thread by thread, 7290 tokens took 8.5 us from the scores, 5 now.
template <int KPT>
__global__ void __launch_bounds__(kSelThreads, 1) k_split_regs(const __grid_constant__ Batch bt) {
  const ImgDesc &im = bt.img[0];
  TL_SCOPE(im, 3);
  __shared__ SelShared sh;
  __shared__ int s_base[kSelThreads];
  static_assert(KPT * kSelWarps <= kSelThreads, "a count for each warp and key");
  const int t = threadIdx.x, lane = t & 31, w = t >> 5, N = im.N;
  const float *score = im.score;
  reinterpret_cast<int2 *>(sh.hist)[t] = make_int2(0, 0);
  if (t == 0) sh.s_few = 0;
  pdl_wait();
  pdl_trigger();
  uint32_t kreg[KPT], kmin = 0xffffffffu, kmax = 0u;
  {
    float sc[KPT];
#pragma unroll
    for (int u = 0; u < KPT; ++u) sc[u] = __ldcg(score + min(t + kSelThreads * u, N - 1));   // (the last one again past the end)
#pragma unroll
    for (int u = 0; u < KPT; ++u) {
      kreg[u] = score_key(sc[u]);
      kmin = min(kmin, kreg[u]);
      kmax = max(kmax, kreg[u]);
    }
  }
  kmin = __reduce_min_sync(0xffffffffu, kmin);
  kmax = __reduce_max_sync(0xffffffffu, kmax);
  if (lane == 0) { sh.wtot[w] = (int)kmin; sh.wtot2[w] = (int)kmax; }
  __syncthreads();
  const uint32_t kbase = __reduce_min_sync(0xffffffffu, (uint32_t)sh.wtot[lane & (kSelWarps - 1)]);
  kmax = __reduce_max_sync(0xffffffffu, (uint32_t)sh.wtot2[lane & (kSelWarps - 1)]);
  uint32_t prefix = 0u;                                 // of the threshold, relative to kbase
  int k = im.m_target;
  for (int hi = 32 - __clz(kmax - kbase); hi > 0;) {
    const int lo = hi > kSelBits ? hi - kSelBits : 0;
    const uint32_t dmask = (1u << (hi - lo)) - 1u;
    const uint32_t above = hi >= 32 ? 0u : ~((1u << hi) - 1u);
#pragma unroll
    for (int u = 0; u < KPT; ++u) {
      const uint32_t kk = kreg[u] - kbase;
      if (t + kSelThreads * u < N && (kk & above) == prefix) {
        const int d = (kk >> lo) & dmask;
        atomicAdd(&sh.hist[d], 1);
        sh.one[d] = kk;
      }
    }
    __syncthreads();
    find_digit(k, sh);
    const int cnt = sh.s_cnt;
    prefix |= (uint32_t)sh.s_bin << lo;
    k = sh.s_k;
    if (lo == 0) break;
    if (cnt == 1) {                                     // one key left under the prefix: it is the threshold
      prefix = sh.one[sh.s_bin];
      break;
    }
    if (cnt <= kSelFew) {
#pragma unroll
      for (int u = 0; u < KPT; ++u) {
        const uint32_t kk = kreg[u] - kbase;
        if (t + kSelThreads * u < N && (kk ^ prefix) >> lo == 0u) sh.few[atomicAdd(&sh.s_few, 1)] = kk;
      }
      __syncthreads();
      if (t < cnt) {
        const uint32_t mine = sh.few[t];
        int less = 0, same = 0;
        for (int j = 0; j < cnt; ++j) { less += sh.few[j] < mine; same += sh.few[j] == mine; }
        if (less <= k && k < less + same) sh.s_prefix = mine;   // (equal keys write the same)
      }
      __syncthreads();
      prefix = sh.s_prefix;
      break;
    }
    hi = lo;
  }
  const uint32_t tau = prefix + kbase;

  // ordered compaction: survivors of every 32 tokens, then before them
  unsigned bal[KPT];
#pragma unroll
  for (int u = 0; u < KPT; ++u) {
    bal[u] = __ballot_sync(0xffffffffu, t + kSelThreads * u < N && kreg[u] >= tau);
    if (lane == 0) s_base[u * kSelWarps + w] = __popc(bal[u]);
  }
  __syncthreads();
  const int mine = t < KPT * kSelWarps ? s_base[t] : 0, incl = warp_scan(mine, lane);
  if (lane == 31) sh.wtot[w] = incl;
  __syncthreads();
  const int wt = lane < kSelWarps ? sh.wtot[lane] : 0, q = __reduce_add_sync(0xffffffffu, wt);
  s_base[t] = incl - mine + (int)__reduce_add_sync(0xffffffffu, lane < w ? wt : 0);
  __syncthreads();
#pragma unroll
  for (int u = 0; u < KPT; ++u) {
    const int i = t + kSelThreads * u;
    if (i >= N) break;
    const bool kp = (bal[u] >> lane) & 1u;
    const int pos = s_base[u * kSelWarps + w] + __popc(bal[u] & ((1u << lane) - 1u));   // survivors with a lower index
    im.keep[i] = kp ? 1 : 0;
    if (kp) im.kept_idx[pos] = i;
    else im.pruned_idx[i - pos] = i;
  }
  if (t == 0) {
    im.counts_user[0] = q;
    im.counts_user[1] = N - q;
  }
}

// More tokens: grid (1), 1024 threads, thread t has the tokens [t CH, (t + 1) CH); dynamic smem: N keys when keys_in_smem, else
// they are read again from the scores.
constexpr int kSplitBits = 11;

__global__ void __launch_bounds__(1024) k_split(const __grid_constant__ Batch bt, int keys_in_smem) {
  const ImgDesc &im = bt.img[0];
  TL_SCOPE(im, 3);
  pdl_wait();
  pdl_trigger();
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int N = im.N;
  extern __shared__ uint32_t skey[];                        // [N] when keys_in_smem
  __shared__ __align__(8) int hist[1 << kSplitBits];
  __shared__ int warp_tot[32];
  __shared__ uint32_t wmin[32], wmax[32];
  __shared__ uint32_t s_prefix;
  __shared__ int s_k, s_cnt;
  const int CH = (N + 1023) / 1024;                         // tokens per thread, contiguous
  const int i0 = min(N, t * CH), cnt_mine = min(N, i0 + CH) - i0;
  if (keys_in_smem)
    for (int i = t; i < N; i += 1024) skey[i] = score_key(im.score[i]);
  if (t == 0) s_k = im.m_target;
  reinterpret_cast<int2 *>(hist)[t] = make_int2(0, 0);
  __syncthreads();
  // j-th key of this thread (j < cnt_mine)
  auto key = [&](int j) -> uint32_t { return keys_in_smem ? skey[i0 + j] : score_key(im.score[i0 + j]); };

  // keys relative to the smallest one, as in k_split_regs
  uint32_t kmin = 0xffffffffu, kmax = 0u;
  for (int j = 0; j < cnt_mine; ++j) { const uint32_t kk = key(j); kmin = min(kmin, kk); kmax = max(kmax, kk); }
  kmin = __reduce_min_sync(0xffffffffu, kmin);
  kmax = __reduce_max_sync(0xffffffffu, kmax);
  if (lane == 0) { wmin[w] = kmin; wmax[w] = kmax; }
  __syncthreads();
  kmin = __reduce_min_sync(0xffffffffu, wmin[lane]);
  kmax = __reduce_max_sync(0xffffffffu, wmax[lane]);
  const uint32_t kbase = kmin;
  const int top = 32 - __clz(kmax - kbase);                 // bits of the largest relative key (0: all keys equal)
  if (t == 0) s_prefix = 0u;
  __syncthreads();

  // Radix select of the (m_target + 1)-th smallest key over the varying bits, up to eleven bits per pass: the first pass
  // leaves a few candidates, the second nearly always one (eight bits and one warp to scan the bins: four passes, 5 us of 11).
  for (int hi = top; hi > 0; hi -= kSplitBits) {
    const int lo = hi > kSplitBits ? hi - kSplitBits : 0;
    const uint32_t dmask = (1u << (hi - lo)) - 1u;
    const uint32_t above = hi >= 32 ? 0u : ~((1u << hi) - 1u);   // bits already fixed
    const uint32_t prefix = s_prefix;
    const int k = s_k;
    for (int j = 0; j < cnt_mine; ++j) {
      const uint32_t kk = key(j) - kbase;
      if ((kk & above) == prefix) atomicAdd(&hist[(kk >> lo) & dmask], 1);
    }
    __syncthreads();
    const int2 c = reinterpret_cast<const int2 *>(hist)[t];      // every thread takes two bins
    reinterpret_cast<int2 *>(hist)[t] = make_int2(0, 0);
    int incl = c.x + c.y;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) warp_tot[w] = incl;
    __syncthreads();
    const int below = incl - c.x - c.y + __reduce_add_sync(0xffffffffu, lane < w ? warp_tot[lane] : 0);
    if (below <= k && k < below + c.x + c.y) {                   // exactly one thread: the candidates number more than k
      const bool second = k >= below + c.x;
      s_k = k - below - (second ? c.x : 0);
      s_cnt = second ? c.y : c.x;
      s_prefix = prefix | ((uint32_t)(2 * t + (second ? 1 : 0)) << lo);
    }
    __syncthreads();
    if (lo > 0 && s_cnt == 1) {                                  // one key left under the prefix: it is the threshold
      const uint32_t fixed = ~((1u << lo) - 1u), pre = s_prefix;
      __syncthreads();
      for (int j = 0; j < cnt_mine; ++j)
        if (((key(j) - kbase) & fixed) == pre) s_prefix = key(j) - kbase;
      __syncthreads();
      break;
    }
  }
  const uint32_t tau_key = s_prefix + kbase;

  // ordered compaction over the contiguous blocks of tokens
  // more than 32 tokens per thread only beyond 32768 tokens: the bits are recomputed below then
  uint32_t keptbits = 0u;
  for (int j = 0; j < cnt_mine && j < 32; ++j) if (key(j) >= tau_key) keptbits |= 1u << j;
  int mine = 0;
  if (CH <= 32) mine = __popc(keptbits);
  else for (int j = 0; j < cnt_mine; ++j) mine += key(j) >= tau_key;
  int incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) warp_tot[w] = incl;
  __syncthreads();
  if (w == 0) {
    const int v = warp_tot[lane];
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    warp_tot[lane] = x - v;                                 // exclusive
    if (lane == 31) s_k = x;                                // q
  }
  __syncthreads();
  const int q = s_k;
  int before = warp_tot[w] + incl - mine;                   // survivors with a lower index
  for (int j = 0; j < cnt_mine; ++j) {
    const int i = i0 + j;
    const bool kp = CH <= 32 ? ((keptbits >> j) & 1u) != 0u : key(j) >= tau_key;
    im.keep[i] = kp ? 1 : 0;
    if (kp) { im.kept_idx[before] = i; ++before; }
    else im.pruned_idx[i - before] = i;
  }
  if (t == 0) {
    im.counts_user[0] = q;
    im.counts_user[1] = N - q;
  }
}

// ---- launchers -----------------------------------------------------------------------------

namespace {
constexpr size_t kSplitReserve = 12288;      // static shared memory of k_split, rounded up
constexpr size_t kTokReserve = 2048;         // of k_tokens
}  // namespace

template <typename T>
static cudaError_t launch_qsum(const Batch &bt, const DeviceCfg &cfg, cudaStream_t st) {
  // column groups of four vectors where that does not take more CTAs than two per SM, else of eight; then as many row
  // blocks (CTAs of a cluster) as keep the grid within three CTAs per SM (three images with 28 query heads: 168 CTAs of
  // very different length took 26 us, twice as many take 20; with five per SM k_tokens has no room beside them)
  const int nvq = bt.n_qcols / Vec<T>::N;
  const bool narrow = (nvq + 3) / 4 * bt.B * kQPartRows <= 2 * cfg.sm_count;
  const int ncg = narrow ? (nvq + 3) / 4 : (nvq + 7) / 8;
  LaunchOpt opt;
  opt.cluster = 1;
  while (opt.cluster < kQPartRows && ncg * bt.B * opt.cluster * 2 <= 3 * cfg.sm_count) opt.cluster *= 2;
  const dim3 grid(ncg * opt.cluster, bt.B), block(kQsumThreads);
  // Nothing reads the queries again: where they are many they leave the L2 first.  Whole steps with new inputs each, kept and marked:
  // 40 MB 99.6 and 98.4 us, eight images of 48 MB together 269.8 and 267.9, of 24 MB 154.7 and 154.2, of 16 MB 116.4 and 116.3, one
  // of 6 to 30 MB the same within 0.3; scores and split alone gain 0.7 to 1.2 us from 10 MB on.
  long long rows = 0;
  for (int b = 0; b < bt.B; ++b) rows += bt.img[b].N;
  const uint64_t policy = rows * bt.n_qcols * (long long)sizeof(T) > (16ll << 20) ? kEvictFirst : kEvictNormal;
  return narrow ? launch_opt(opt, k_qsum<T, 4>, grid, block, 0, st, bt, opt.cluster, policy) : launch_opt(opt, k_qsum<T, 8>, grid, block, 0, st, bt, opt.cluster, policy);
}

template <typename T> static TokCfg tokens_config(const Batch &bt, const DeviceCfg &cfg) {
  long long total = 0;
  for (int b = 0; b < bt.B; ++b) total += bt.img[b].N;
  return tokens_config(total, bt.d * (int)sizeof(T), bt.d_k * (int)sizeof(T), bt.n_qcols, bt.n_qh / bt.n_kvh, cfg.sm_count, cfg.smem_optin - kTokReserve);
}
template <typename T>
static cudaError_t launch_tokens(const Batch &bt, bool scores_only, int what, bool pdl, const DeviceCfg &cfg, cudaStream_t st, int *rpp) {
  const TokCfg tc = tokens_config<T>(bt, cfg);
  if (rpp) *rpp = tc.rpp;
  const bool group = bt.n_qh / bt.n_kvh >= kGroupHeads;
  const auto kernel = tc.query ? (group ? k_tokens<T, true, true> : k_tokens<T, true, false>) : (group ? k_tokens<T, false, true> : k_tokens<T, false, false>);
  int N[kMaxBatchPerLaunch];
  long long tokens = 0;
  for (int b = 0; b < bt.B; ++b) tokens += N[b] = bt.img[b].N;
  TokUnits un;
  const int grid = tokens_units(N, bt.B, tc.rpp, cfg.sm_count, un);
  // Hidden states of which the merge will find too little in the L2 in any case leave it first, so that queries, keys and what the kernels
  // hand to one another stay.  Whole steps with new inputs each, kept and marked: one image of 40 MB 82.9 and 85.5 us, 75 MB 135.3 and 136.5, 82 MB 140.5
  // and 141.0, 90 MB 151.5 and 150.7, 130 MB 213.1 and 208.3; four images of 75 MB together 99.8 and 99.9, 90 MB 114.7 and 113.7.
  // Scores as a stage of their own: nobody knows whether a merge follows.  Scores and split alone, over and over on two or three buffers, gain from
  // about 32 MB on (30 MB 21.3 and 21.3 us, 38 MB 24.2 and 22.7, 52 MB 27.8 and 25.7; on new inputs the same, 52 MB 28.1 and 28.1, 100 MB 45.2 and
  // 43.0); five stages with new inputs lose (18 MB 80.8 and 82.1, 36 MB 94.4 and 97.6, 52 MB 111.6 and 114.8, 100 MB 182.9 and 180.5).
  const long long kept = scores_only ? 32ll << 20 : 80ll << 20;
  const uint64_t policy = tokens * bt.d * (long long)sizeof(T) > kept ? kEvictFirst : kEvictNormal;
  return launch_k(kernel, dim3(grid), dim3(kTokThreads), tok_smem_launch(tc, bt.d_k * (int)sizeof(T), bt.n_qcols), st, pdl, bt, tc, un, policy, what);
}

template <typename T>
static cudaError_t launch_euti_t(const Batch &bt, int maxN, int mode, const DeviceCfg &cfg, cudaStream_t st, StageMark mark, void *mark_arg, int *rpp_out,
                                 const HostFeed *feed) {
  cudaError_t e = cudaSuccess;
  if (feed && (e = cudaStreamWaitEvent(st, feed->keys, 0)) != cudaSuccess) return e;
  e = launch_qsum<T>(bt, cfg, st);
  if (e != cudaSuccess) return e;
  if (mark && (e = mark(mark_arg)) != cudaSuccess) return e;
  int rpp = 0;
  e = launch_tokens<T>(bt, mode == 1, (mode != 1 ? kTokInit : 0) | (feed ? 0 : kTokNorms) | kTokLogits, true, cfg, st, &rpp);
  if (e != cudaSuccess) return e;
  for (int k = 0, first = 0; feed && k < kFeedParts; first = feed->end[k++]) {
    // (a part without visual tokens may still bring text rows, which k_merge copies)
    if ((e = cudaStreamWaitEvent(st, feed->part[k], 0)) != cudaSuccess) return e;
    if (feed->end[k] <= first) continue;
    Batch part = bt;
    part.img[0].N = feed->end[k] - first;
    part.img[0].vis_start += first;
    part.img[0].nrm += first;
    if ((e = launch_tokens<T>(part, false, kTokNorms, false, cfg, st, nullptr)) != cudaSuccess) return e;
  }
  if (rpp_out) *rpp_out = rpp;
  if (mode == 2) return cudaSuccess;
  if (mark && (e = mark(mark_arg)) != cudaSuccess) return e;
  LaunchOpt opt;
  int CL = 1;
  while (CL < kScoreMaxCl && bt.n_qh > 4 * CL) CL *= 2;
  if (CL > 1) opt.cluster = CL;
  const int nb = (maxN + kScoreTok - 1) / kScoreTok;
  e = launch_opt(opt, bt.n_qh <= 4 ? k_scores<2> : k_scores<8>, dim3((nb + CL - 1) / CL * CL, bt.B), dim3(kScoreThreads), 0, st, bt, rpp, mode == 0 ? 1 : 0, CL);
  if (e != cudaSuccess) return e;
  if (mode == 0) {
    if (mark && (e = mark(mark_arg)) != cudaSuccess) return e;
    size_t keys = (size_t)maxN * sizeof(uint32_t);
    const bool in_smem = keys <= kSelKeyBytes;
    if (!in_smem) keys = 0;
    int X = cfg.sm_count / bt.B;
    const int want = (maxN + 15) / 16;         // at least sixteen tokens per CTA
    if (X > want) X = want;
    if (X < 1) X = 1;
    const auto kernel = maxN <= 6 * kSelThreads ? k_select<T, 6, false> : maxN <= 16 * kSelThreads ? k_select<T, 16, false>
                        : maxN <= 32 * kSelThreads ? k_select<T, 32, false> : in_smem ? k_select<T, 0, true> : k_select<T, 0, false>;
    // The rows of the own tokens wait in shared memory where all of them fit; with more per CTA (batches, long images) what
    // counts is their bytes, and the pruned ones would be read for nothing.
    int pre = 0;
    if (maxN <= 32 * kSelThreads) {
      const int rowb = bt.d_k * (int)sizeof(T), tpc = (maxN + X - 1) / X;
      pre = (size_t)tpc * rowb <= kSelKeyBytes && tpc <= kSelThreads ? tpc : 0;
      keys = (size_t)pre * rowb;
    }
    e = launch_k(kernel, dim3(X, bt.B), dim3(kSelThreads), keys, st, true, bt, pre);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

cudaError_t launch_euti(const Batch &bt, int maxN, bool bf16, int mode, const DeviceCfg &cfg, cudaStream_t st, StageMark mark, void *mark_arg, int *rpp) {
  return bf16 ? launch_euti_t<__nv_bfloat16>(bt, maxN, mode, cfg, st, mark, mark_arg, rpp, nullptr)
              : launch_euti_t<float>(bt, maxN, mode, cfg, st, mark, mark_arg, rpp, nullptr);
}
cudaError_t launch_euti_fed(const Batch &bt, int maxN, bool bf16, int mode, const DeviceCfg &cfg, cudaStream_t st, const HostFeed &feed, int *rpp) {
  return bf16 ? launch_euti_t<__nv_bfloat16>(bt, maxN, mode, cfg, st, nullptr, nullptr, rpp, &feed)
              : launch_euti_t<float>(bt, maxN, mode, cfg, st, nullptr, nullptr, rpp, &feed);
}

int euti_kernels(int mode) { return mode == 0 ? 4 : mode == 1 ? 3 : 2; }

cudaError_t launch_split(const Batch &bt, int N, const DeviceCfg &cfg, cudaStream_t st) {
  if (N <= 6 * kSelThreads) return launch_k(k_split_regs<6>, dim3(1), dim3(kSelThreads), 0, st, true, bt);
  if (N <= 16 * kSelThreads) return launch_k(k_split_regs<16>, dim3(1), dim3(kSelThreads), 0, st, true, bt);
  if (N <= 32 * kSelThreads) return launch_k(k_split_regs<32>, dim3(1), dim3(kSelThreads), 0, st, true, bt);
  const size_t sm = (size_t)N * sizeof(uint32_t);
  const bool in_smem = sm + kSplitReserve <= cfg.smem_optin;
  return launch_k(k_split, dim3(1), dim3(1024), in_smem ? sm : 0, st, true, bt, in_smem ? 1 : 0);
}

cudaError_t select_configure(DeviceCfg *cfg) {
  int dev = 0, v = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  cfg->sm_count = v;
  e = cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  cfg->smem_optin = (size_t)v;
  return cudaFuncSetAttribute(k_split, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(cfg->smem_optin - kSplitReserve));
}

cudaError_t euti_configure(const DeviceCfg &cfg, int n_qcols, int n_qh) {
  cudaError_t e = cudaSuccess;
  if ((size_t)(n_qcols + 32 * n_qh) * 8 > cfg.smem_optin - 1024) return cudaErrorInvalidConfiguration;   // the widest query
  const int tok = (int)(cfg.smem_optin - kTokReserve);
  for (const auto f : {k_tokens<__nv_bfloat16, true, true>, k_tokens<__nv_bfloat16, true, false>, k_tokens<__nv_bfloat16, false, true>, k_tokens<__nv_bfloat16, false, false>,
                       k_tokens<float, true, true>, k_tokens<float, true, false>, k_tokens<float, false, true>, k_tokens<float, false, false>})
    if ((e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, tok)) != cudaSuccess) return e;
  for (const auto f : {k_select<__nv_bfloat16, 0, true>, k_select<__nv_bfloat16, 6, false>, k_select<__nv_bfloat16, 16, false>, k_select<__nv_bfloat16, 32, false>,
                       k_select<float, 0, true>, k_select<float, 6, false>, k_select<float, 16, false>, k_select<float, 32, false>})
    if ((e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSelKeyBytes)) != cudaSuccess) return e;
  // k_tokens can only begin beside k_qsum if both run under the same split of the SM's memory (with the default it waited
  // for k_qsum to drain, 9 us at 6272 tokens); for the other kernels the default is as good or better (16384-token images: 10 us)
  return prefer_shared(k_qsum<__nv_bfloat16, 4>, k_qsum<__nv_bfloat16, 8>, k_qsum<float, 4>, k_qsum<float, 8>, k_tokens<__nv_bfloat16, true, true>,
                       k_tokens<__nv_bfloat16, true, false>, k_tokens<float, true, true>, k_tokens<float, true, false>, k_scores<2>, k_scores<8>);
}

}  // namespace pact
