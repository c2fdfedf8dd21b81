// How k_merge (merge.cu) cuts the member records and text rows of an image into ranges: arithmetic on sizes alone, without CUDA, so that every
// size can be gone through on the host.
#pragma once

namespace pact {

constexpr int kMrgCtasPerSm = 8;
constexpr int kMrgRanges = 296;                     // most ranges per image (sizes the scratch)
constexpr int kMrgLeast = 8;                        // fewest items per range, see below

// items per range: 24 (with 16: 2.5 us more of 16 images of 2916 tokens, 2 us of three of 2309; with 48 as much), 12 where
// that leaves an SM less than two CTAs, 8 where 12 does: the rows of a range follow one
// another, 40 ns each where a CTA has the SM to itself.  No more than eight rounds of CTAs over the GPU, and no more ranges than
// the scratch has room for.  (16 for all small calls: 729 tokens 47.8 us, 46.3 with 8; 1300 57.4, 55.9 with 12, 57.8 with 8.)
// Never less than eight: the ticket of a cut cluster that begins in range x is at 8 x + the slice of columns (at most eight), and one that is cut
// has more than eight members, so that 8 x + 7 is still the place of a token.
inline int merge_per(int n_items, int slices, int B, int sm_count) {
  const long long most = 8LL * kMrgCtasPerSm * sm_count;
  long long r = (n_items + 23) / 24;
  if (r * slices * B < 2 * sm_count) r = (n_items + 11) / 12;
  if (r * slices * B < 2 * sm_count) r = (n_items + 7) / 8;
  if (r * slices * B > most) r = most / ((long long)slices * B);
  if (r > kMrgRanges) r = kMrgRanges;
  if (r < 1) r = 1;
  const int per = (int)((n_items + r - 1) / r);
  return per > kMrgLeast ? per : kMrgLeast;
}

// Clusters of at most this many members are done by the range they begin in, whatever its end; room: items that the ring holds beyond a range.
// One round of CTAs: the longest range counts, so only clusters that leave it within what the ring holds at once stay
// whole, and no more than kMrgWhole items past its end (as many rows as a cut costs; 900 tokens of a video 49.8 -> 45.4 us, 729 of a
// photo 46.7 -> 46.3).  Several rounds: the bytes count.
constexpr int kMrgWhole = 24;                       // items past its end that a range goes on for a cluster
inline int merge_whole(int per, long long ctas_per_sm, int room) {
  return ctas_per_sm > kMrgCtasPerSm ? per : room < kMrgLeast ? kMrgLeast : room > kMrgWhole ? kMrgWhole : room;
}

}  // namespace pact
