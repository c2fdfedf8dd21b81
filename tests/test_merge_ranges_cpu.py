"""How k_merge cuts an image into ranges (csrc/merge_ranges.h), gone through on the host."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_tickets_of_cut_clusters_are_those_of_tokens(tmp_path):
    """A cluster is cut when it has more than `whole` members and goes past its range's end.  Its ticket, 8 (range it begins in) + slice, has to lie
    below the number of tokens, and the ranges have to fit the scratch.  All sizes up to 20000 and some beyond, every number of slices and images."""
    (tmp_path / "r.cpp").write_text(r"""
#include <stdio.h>
#include "merge_ranges.h"
static bool ok(int n, int slices, int B) {
  const int per = pact::merge_per(n, slices, B, 148), ranges = (n + per - 1) / per;
  const long long ctas = ((long long)ranges * slices * B + 147) / 148;
  if (per < 8 || ranges > pact::kMrgRanges || ranges < 1) return false;
  for (int room = -64; room <= 64; ++room) {
    const int whole = pact::merge_whole(per, ctas, room);
    if (whole < 8) return false;
    // the last place a cut cluster may begin at (all items members: a text row only leaves it less room)
    const int first = n - (whole + 1);
    if (first >= 0 && first / per * 8 + slices - 1 >= n) return false;
  }
  return true;
}
int main() {
  for (int slices = 1; slices <= 8; ++slices)
    for (int B = 1; B <= 16; ++B)
      for (int n = 1; n < (1 << 18); n += n < 20000 ? 1 : 977)
        if (!ok(n, slices, B)) { printf("%d items, %d slices, %d images\n", n, slices, B); return 1; }
}
""")
    exe = str(tmp_path / "r")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-Wall", "-Werror", "-I", os.path.join(ROOT, "paper_2504_08966_b200", "csrc"), str(tmp_path / "r.cpp"), "-o", exe])
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
