"""The adjoint's one-block tail starts on a level that fits one block, at every mesh side.

csrc/adjoint_levels.h is host code: a few lines of C++ built with it here choose the
level for every even side up to 2048 with every number of levels, and check it against
the rule in 64 bits and against the shared memory the kernel is given.
"""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "adjoint_levels.h"
#include <stdio.h>
using namespace mg;
int main() {
  long long checked = 0, tails = 0;
  for (int N = 2; N <= 2048; N += 2)
    for (int split = 0; split < 2; ++split) {
      int n[16], most = 1;
      n[0] = N;
      while (most < 16 && n[most - 1] % 2 == 0 && n[most - 1] / 2 >= 2) n[most] = n[most - 1] / 2, ++most;
      for (int nlev = 1; nlev <= most; ++nlev, ++checked) {
        int want = -1;
        for (int l = nlev - 1; l >= (split ? 1 : 0); --l)
          if (n[l] <= 16 && nlev - l <= kAdjTailLevels) want = l;
        const int got = adj_tail_level(n, nlev, split);
        if (got != want) return printf("N %d levels %d split %d: %d, not %d\n", N, nlev, split, got, want), 1;
        if (got < 0) continue;
        ++tails;
        if (adj_tail_smem(n + got, nlev - got) > (size_t)kAdjTailSmem) return printf("N %d: too large\n", N), 1;
      }
    }
  printf("%lld %lld\n", checked, tails);
  return 0;
}
"""


def test_tail_level_at_every_side(tmp_path):
    src, exe = tmp_path / "levels.cpp", tmp_path / "levels"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_2110_00328_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    checked, tails = map(int, r.stdout.split())
    assert checked > 4000 and 0 < tails < checked
