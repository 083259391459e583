"""The CTAs that a round's resident solves may take (csrc/round_share.h), compiled for the host."""
import shutil
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parents[1] / "paper_2111_11788_gb300" / "csrc"

MAIN = r"""
#include <cstdio>
#include "round_share.h"
using namespace mlmc;

int64_t slots = 0;
// a round's capture: the limit stands while it runs, also where it ends early
int64_t capture(bool fails) {
  const ScopedLimit share(slots, 114);
  if (fails) return -slots;
  return slots;
}
int main() {
  std::printf("%lld %lld", (long long)capture(false), (long long)slots);
  std::printf(" %lld %lld\n", (long long)capture(true), (long long)slots);
  // rounds on stdin: mixed, dim, jacobi, levels, then per level cells, samples, resident
  int mixed, dim, jacobi, levels;
  while (std::scanf("%d %d %d %d", &mixed, &dim, &jacobi, &levels) == 4) {
    RoundWork w;
    int below = 0, below_resident = 0;
    for (int l = 0; l < levels; ++l) {
      int n, samples, res;
      if (std::scanf("%d %d %d", &n, &samples, &res) != 3) return 1;
      w.add_level(RoundWork::of(dim, n, jacobi, samples), res, l ? RoundWork::of(dim, below, jacobi, samples) : 0.0,
                  l && below_resident);
      below = n;
      below_resident = res;
    }
    std::printf("%lld\n", (long long)resident_limit(w, mixed));
  }
}
"""

# form, dimension, solver, cells per side of level 0, samples per level, largest resident mesh; the limit
ROUNDS = [
    ("mixed", 2, "gmg", 32, (100, 100, 100, 100, 100), 128, 114),        # the finest level dominates
    ("fp64", 2, "gmg", 32, (100, 100, 100, 100, 100, 100), 128, 114),
    ("mixed", 3, "gmg", 16, (64, 32, 16, 8, 4), 16, 114),
    ("fp64", 2, "gmg", 32, (800, 400, 200, 50, 20, 7), 128, 114),        # 0.48
    ("mixed", 2, "gmg", 32, (800, 400, 200, 50, 20, 7), 128, 228),
    ("fp64", 2, "gmg", 32, (4000, 2000, 700, 50, 67), 128, 228),         # 1.3
    ("mixed", 2, "gmg", 32, (4096, 512, 64, 8, 1), 128, 0),              # resident levels carry most of it
    ("fp64", 2, "gmg", 32, (50, 50, 1000, 1), 128, 0),
    ("mixed", 2, "gmg", 32, (100, 100, 100, 100), 128, 0),               # nothing beside: 256^2 waits for its own 128^2
    ("fp64", 2, "jacobi", 50, (100, 60, 399), 170, 0),
    ("mixed", 2, "gmg", 8, (500, 200, 100), 128, 0),                     # resident meshes only
    ("mixed", 2, "gmg", 256, (20, 4), 128, 114),                         # none resident
]


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("round_share")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run([cxx, "-std=c++17", "-Wall", "-Werror", "-I", str(CSRC), str(d / "main.cpp"), "-o", str(d / "a")],
                   check=True)
    text = "\n".join(" ".join(map(str, [int(form == "mixed"), dim, int(solver == "jacobi"), len(N)] +
                                   [v for l, c in enumerate(N) for v in (n0 << l, c, int(n0 << l <= top))]))
                     for form, dim, solver, n0, N, top, _ in ROUNDS)
    return subprocess.run([str(d / "a")], input=text, check=True, capture_output=True, text=True).stdout.splitlines()


def test_the_limit_ends_with_the_capture(lines):
    assert lines[0].split() == ["114", "0", "-114", "0"]


def test_the_limit_follows_the_work_that_runs_beside(lines):
    assert [int(v) for v in lines[1:]] == [r[-1] for r in ROUNDS]
