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
}
"""


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("round_share")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run([cxx, "-std=c++17", "-Wall", "-Werror", "-I", str(CSRC), str(d / "main.cpp"), "-o", str(d / "a")],
                   check=True)
    return subprocess.run([str(d / "a")], check=True, capture_output=True, text=True).stdout.splitlines()


def test_the_limit_ends_with_the_capture(lines):
    assert lines[0].split() == ["114", "0", "-114", "0"]
