"""Sizes chosen on the host (csrc/sizing.h), compiled by themselves: no GPU, no CUDA."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2111_10354_gb300", "csrc")


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    """Compiles a main() body that prints with sizing.h's functions; returns the printed lines."""
    def go(body):
        d = tmp_path_factory.mktemp("sizing")
        src, exe = d / "t.cpp", d / "t"
        src.write_text('#include <stdio.h>\n#include "sizing.h"\nusing namespace hisq;\nint main() {\n%s\n}\n' % body)
        subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
        return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n")[:-1]
    return go


def test_multishift_group_length_does_not_depend_on_earlier_solves(run):
    """Solve after solve in the memory that the one before left: every free size from nothing to plenty, in steps
    that fall between the thresholds. The length stays, is the largest that fits, and never shrinks below the buffer
    that is held."""
    out = run("""
  const size_t per = 1000, verify = 14 * 1600, taken = 14 * 1400;  // the verification takes less than is kept for it
  for (size_t room = 0; room < 40000; room += 333) {
    const int first = ms_group_length(8, per, 0, verify, 0, room);
    const size_t left = room > first * per + taken ? room - first * per - taken : 0;
    const int second = ms_group_length(8, per, first * per, verify, taken, left);
    const int third = ms_group_length(8, per, second * per, verify, taken, left);
    // a second kind of vector of half the size, as FP32 after FP64
    const int other = ms_group_length(8, per / 2, first * per, verify, taken, left);
    printf("%zu %d %d %d %d\\n", room, first, second, third, other);
  }""")
    assert len(out) > 100
    for line in out:
        room, first, second, third, other = (int(v) for v in line.split())
        fits = [s for s in (8, 4, 2, 1) if s * 1000 + 22400 <= room] or [1]
        assert first == fits[0]
        if room >= first * 1000 + 19600:  # the solve's own buffers fitted
            assert first == second == third
            assert other >= min(8, 2 * first)


def test_launch_cuts_cover_the_vectors_and_differ(run):
    """Every way to cut 1 to 64 vectors, for groups of 4 to 8: the groups add up, none exceeds its limit, the ways
    offered differ, and the full groups come first (what an untuned call takes)."""
    out = run("""
  for (int gmax = 4; gmax <= 8; ++gmax)
    for (int pow2 = 0; pow2 < 2; ++pow2)
      for (int n = 1; n <= 64; ++n) {
        int cuts[3];
        const int k = launch_cuts(n, gmax, pow2 != 0, cuts);
        for (int i = 0; i < k; ++i) {
          printf("%d %d %d %d", gmax, pow2, n, cuts[i]);
          for (int left = n; left > 0;) { const int g = next_group(cuts[i], left, gmax); printf(" %d", g); left -= g; }
          printf("\\n");
        }
      }""")
    ways = {}
    for line in out:
        gmax, pow2, n, cut, *groups = (int(v) for v in line.split())
        assert sum(groups) == n and max(groups) <= gmax and min(groups) >= 1
        if cut == 1:
            assert len(groups) == -(-n // gmax) and max(groups) - min(groups) <= 1
        if cut == 2:
            assert all(g == gmax or g & (g - 1) == 0 for g in groups)
        ways.setdefault((gmax, pow2, n), []).append((cut, groups))
    for (gmax, pow2, n), w in ways.items():
        assert w[0][0] == 0 and len(w[0][1]) == -(-n // gmax)
        assert len({tuple(g) for _, g in w}) == len(w) <= 2 + pow2
    assert [g for _, g in ways[8, 0, 12]] == [[8, 4], [6, 6]] and len(ways[8, 0, 7]) == 1
    assert [g for _, g in ways[4, 1, 3]] == [[3], [2, 1]]
