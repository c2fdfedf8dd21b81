// How k_tokens (euti.cu) cuts its work: tokens per unit, bytes of a hidden-state row per copy, and what is in shared memory.
// Arithmetic on sizes alone, without CUDA, so that every size a context accepts can be gone through on the host.
#pragma once
#include <stddef.h>
#include <stdint.h>

#ifdef __CUDACC__
#define PACT_HD __host__ __device__
#else
#define PACT_HD
#endif

namespace pact {

constexpr int kMaxBatchPerLaunch = 16;   // images described by one kernel parameter block
constexpr int kMinPiece = 8;             // fewest visual tokens in a softmax piece of k_tokens (at most 32)
constexpr int kTokWarps = 8;             // warps that stream hidden-state rows
constexpr int kTokMaxBuf = 2;            // row buffers per warp
constexpr int kTokSmem = 200 * 1024;
constexpr int kGroupHeads = 3;           // query heads per key head from which they go through group_piece

struct TokCfg {
  int rpp;                               // tokens per unit (piece)
  int chunk, nchunk;                     // bytes of a hidden-state row per copy, copies per row
  int nbuf;                              // row buffers per warp
  int keys;                              // a key buffer per team (else the keys are read from global memory, and a unit has kMinPiece tokens)
  int query;                             // the global query in shared memory (else read from global memory)
};

// stride of a key row in shared memory: an odd number of 16-byte vectors, so that a vector of 8 rows is in 8 different banks
PACT_HD inline int tok_key_stride(int row_bytes) { return row_bytes | 16; }

inline size_t tok_smem(const TokCfg &c, int key_bytes, int n_qcols) {
  return (size_t)kTokWarps * c.nbuf * c.chunk + (size_t)2 * c.keys * c.rpp * tok_key_stride(key_bytes) + (size_t)c.query * n_qcols * 8 + (size_t)c.rpp * 32 * 8;
}

// What a launch asks for: the parts of the sums of squares have a row for each of a warp's tokens of a unit, so that no other warp
// writes there, up to seven rows more than the unit has tokens.  (kTokSmem leaves room for them.)
PACT_HD inline int tok_warp_rows(int rpp) { return (rpp + kTokWarps - 1) / kTokWarps; }
inline size_t tok_smem_launch(const TokCfg &c, int key_bytes, int n_qcols) {
  return tok_smem(c, key_bytes, n_qcols) + (size_t)(tok_warp_rows(c.rpp) * kTokWarps - c.rpp) * 32 * 8;
}

// total tokens of the call, rows of row_bytes, keys of key_bytes, n_rep query heads per key head, and the GPU's SMs and shared memory.
// Tokens per unit: the fewest rounds of units of `most` tokens over the SMs, then as few tokens as that many rounds allow
// (but eight), so that the rounds are full.
// Where the buffers do not fit, units of sixteen and eight tokens come first, then rows in copies of half the size, then the keys
// go without shared memory, then a part of the row buffers, at last the global query (more than 26496 columns with the largest
// rows).  Copies of 2.5 to 4 KB still take in what the memory gives, keys read from global memory do not: the token pass of 7290
// tokens of 8192 in bf16 with 64 heads on 8 takes 91 us without key buffers and 40 with rows in halves, 2916 of fp32 4096
// with 32 on 8 takes 77 and 28, 7290 of 8192 with 16 on 16 72 and 42, 2916 of 5120 with 40 on 20 (copies of 2560 bytes) 50 and 29.
inline TokCfg tokens_config(long long total, int row_bytes, int key_bytes, int n_qcols, int n_rep, int sm_count, size_t smem_optin) {
  TokCfg c;
  c.nbuf = kTokMaxBuf;
  c.keys = 1;
  c.query = 1;
  const auto cut_rows = [&](int n) {
    c.nchunk = n;
    c.chunk = ((row_bytes + n - 1) / n + 15) / 16 * 16;
  };
  const auto fits = [&]() { return tok_smem(c, key_bytes, n_qcols) <= (size_t)kTokSmem; };
  const int whole = (row_bytes + 8191) / 8192;
  for (int parts = 1; parts <= 2; ++parts) {
    cut_rows(whole * parts);
    for (int most = 32; most >= kMinPiece; most /= 2) {
      long long rounds = (total + (long long)most * sm_count - 1) / ((long long)most * sm_count);
      // (a unit for each of the two teams, where the logits are what takes the time)
      if (rounds < 2 && n_rep >= kGroupHeads) rounds = 2;
      const long long rpp = (total + rounds * sm_count - 1) / (rounds * sm_count);
      c.rpp = (int)(rpp < kMinPiece ? kMinPiece : rpp);
      if (fits()) return c;
    }
  }
  c.keys = 0;                                                             // very wide keys or queries
  c.rpp = kMinPiece;
  cut_rows(whole);
  while (!fits() && c.chunk > 1024) cut_rows(2 * c.nchunk);
  c.query = tok_smem(c, key_bytes, n_qcols) <= smem_optin;
  return c;
}

// The units of a call: those of image b begin at first[b]; CTA c takes `per` of them and one more if c < extra, in a row.
struct TokUnits {
  int first[kMaxBatchPerLaunch + 1];
  int per, extra;
};

// Units of rpp tokens of B images of N[b] tokens each, shared out; returns the number of CTAs.  (At most 16 x 2^18 / 8 units.)
inline int tokens_units(const int *N, int B, int rpp, int sm_count, TokUnits &un) {
  int units = 0;
  for (int b = 0; b <= kMaxBatchPerLaunch; ++b) {
    un.first[b] = units;
    if (b < B) units += (N[b] + rpp - 1) / rpp;
  }
  const int grid = units < sm_count ? units : sm_count;
  un.per = units / grid;
  un.extra = units - un.per * grid;
  return grid;
}

}  // namespace pact
