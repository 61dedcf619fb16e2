"""The remainder by a double reciprocal (csrc/mod_range.h) is exactly x % d on both
sides of its threshold, at the edges of x and d and beside multiples of d."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1612_01287_gb300", "csrc")

MAIN = """
#include <cstdio>
#include "mod_range.h"
int main() {
  const uint32_t ds[] = {1, 2, 3, 16383, 16384, 16385, 65537, 131071, 1000003, 1u << 30,
                         2147483646u, 2147483647u};
  uint64_t s = 1;
  for (uint32_t d : ds)
    for (int i = 0; i < 200000; ++i) {
      s = s * 6364136223846793005ull + 1442695040888963407ull;
      const uint64_t m = (s >> (i % 40)) / d * d;
      const uint64_t top = ~uint64_t(0) / d * d;
      const uint64_t xs[] = {s, m, m + d - 1, m - 1, ~uint64_t(0) - i, top - (i & 1)};
      for (uint64_t x : xs)
        if (rslb::mod_range(x, d) != x % d) {
          std::printf("%llu %u\\n", (unsigned long long)x, d);
          return 1;
        }
    }
  return 0;
}
"""


def test_mod_range_is_exact(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(MAIN)
    subprocess.run([cxx, "-O3", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, "x, d = " + r.stdout
