"""How the token pass cuts its work (csrc/tok_units.h), over the sizes that a context accepts: compiled for the host."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SMS, OPTIN, LIMIT = 148, 227 * 1024 - 2048, 200 * 1024

SOURCE = r"""
#include <stdio.h>
#include "tok_units.h"
int main() {
  long long total; int rowb, keyb, cols, rep;
  while (scanf("%lld %d %d %d %d", &total, &rowb, &keyb, &cols, &rep) == 5) {
    pact::TokCfg c = pact::tokens_config(total, rowb, keyb, cols, rep, 148, 227 * 1024 - 2048);
    printf("%d %d %d %d %d %d %zu\n", c.rpp, c.chunk, c.nchunk, c.nbuf, c.keys, c.query, pact::tok_smem(c, keyb, cols));
  }
}
"""


@pytest.fixture(scope="module")
def configs(tmp_path_factory):
    """(total tokens, d, element bytes, n_qh, n_kvh, d_h) -> (rpp, chunk, nchunk, nbuf, keys, query, bytes of shared memory)"""
    tmp = tmp_path_factory.mktemp("units")
    (tmp / "units.cpp").write_text(SOURCE)
    subprocess.check_call(["g++", "-std=c++17", "-Wall", "-Werror", "-I", os.path.join(ROOT, "paper_2504_08966_b200", "csrc"), str(tmp / "units.cpp"), "-o", str(tmp / "units")])

    def run(cases):
        lines = [f"{n} {d * e} {kv * dh * e} {qh * dh} {qh // kv}" for n, d, e, qh, kv, dh in cases]
        out = subprocess.run([str(tmp / "units")], input="\n".join(lines), capture_output=True, text=True, check=True).stdout
        return [tuple(int(x) for x in ln.split()) for ln in out.splitlines()]

    return run


HEADS = [(1, 1, 8), (2, 2, 64), (4, 4, 128), (14, 2, 64), (28, 4, 128), (16, 16, 128), (32, 8, 96), (32, 8, 128), (32, 32, 128), (40, 20, 128), (56, 8, 128),
         (64, 8, 128), (64, 64, 128), (128, 8, 128), (32, 1, 872), (1, 1, 26496), (1, 1, 28896)]
CASES = [(n, d, e, *h) for n in (1, 8, 43, 1184, 1185, 2368, 2369, 4737, 7290, 46656, 16 << 18) for d in (8, 520, 896, 3584, 4096, 4104, 5120, 7168, 8192) for e in (2, 4) for h in HEADS]


def test_buffers_fit_and_rows_are_whole(configs):
    for (n, d, e, qh, kv, dh), (rpp, chunk, nchunk, nbuf, keys, query, smem) in zip(CASES, configs(CASES)):
        assert 8 <= rpp <= 32 and nbuf == 2
        assert chunk % 16 == 0 and chunk <= 8192 and (nchunk - 1) * chunk < d * e <= nchunk * chunk
        assert smem <= (LIMIT if keys else OPTIN)
        assert keys or rpp == 8                                     # what the forms of the kernel without key buffers rest on
        assert query or not keys


def test_rows_in_smaller_copies_before_the_keys_lose_their_buffers(configs):
    """Wide grouped-query models: 64 and 56 heads on 8 in 16 bits, 32 on 8 in fp32."""
    wide = [(n, *m) for n in (1, 729, 2916, 7290, 46656) for m in ((8192, 2, 64, 8, 128), (7168, 2, 56, 8, 128), (4096, 4, 32, 8, 128))]
    for case, (rpp, chunk, nchunk, _, keys, _, _) in zip(wide, configs(wide)):
        assert keys and 3584 <= chunk <= 4096, case


def test_what_fits_beside_whole_copies_stays_as_it_was(configs):
    """The same units as with copies of up to 8 KB alone, wherever these leave room for the keys."""
    def plain(n, d, e, qh, kv, dh):
        nchunk = -(-d * e // 8192)
        chunk = -(-(-(-d * e // nchunk)) // 16) * 16
        for most in (32, 16, 8):
            rounds = -(-n // (most * SMS))
            if rounds < 2 and qh // kv >= 3:
                rounds = 2
            rpp = max(8, -(-n // (rounds * SMS)))
            if 16 * chunk + 2 * rpp * (kv * dh * e | 16) + qh * dh * 8 + rpp * 256 <= LIMIT:
                return rpp, chunk, nchunk
        return None

    for case, got in zip(CASES, configs(CASES)):
        want = plain(*case)
        if want is not None:
            assert got[:3] == want and got[4], case


def test_every_unit_has_one_cta(tmp_path):
    """Images of any sizes: the CTAs' shares follow one another, differ by one unit at most and end with the last one."""
    (tmp_path / "share.cpp").write_text(r"""
#include <stdio.h>
#include "tok_units.h"
int main() {
  int B, rpp, N[pact::kMaxBatchPerLaunch];
  while (scanf("%d %d", &B, &rpp) == 2) {
    for (int b = 0; b < B; ++b) if (scanf("%d", N + b) != 1) return 1;
    pact::TokUnits un;
    printf("%d", pact::tokens_units(N, B, rpp, 148, un));
    for (int b = 0; b <= pact::kMaxBatchPerLaunch; ++b) printf(" %d", un.first[b]);
    printf(" %d %d\n", un.per, un.extra);
  }
}
""")
    subprocess.check_call(["g++", "-std=c++17", "-Wall", "-Werror", "-I", os.path.join(ROOT, "paper_2504_08966_b200", "csrc"), str(tmp_path / "share.cpp"), "-o", str(tmp_path / "share")])
    cases = [(rpp, N) for rpp in (8, 25, 32) for N in ([1], [8], [9], [1184], [1185], [7290], [1 << 18], [1, 262144], [2309, 1731, 1153], [33] * 16, [1 << 18] * 16)]
    out = subprocess.run([str(tmp_path / "share")], input="\n".join(f"{len(N)} {rpp} {' '.join(map(str, N))}" for rpp, N in cases), capture_output=True, text=True, check=True).stdout
    for (rpp, N), line in zip(cases, out.splitlines()):
        grid, *first, per, extra = (int(x) for x in line.split())
        want = [0]
        for n in N:
            want.append(want[-1] + -(-n // rpp))
        assert first == want + [want[-1]] * (17 - len(want))
        assert grid == min(148, want[-1]) and per >= 1 and 0 <= extra < grid and per * grid + extra == want[-1]
