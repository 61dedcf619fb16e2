"""Classes of a batch over streams (csrc/chains.h): one chain each while there are
enough, never more than the bound, and no chain above an even share by more than
the largest item."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1612_01287_gb300", "csrc")

MAIN = """
#include <cstdio>
#include <cstdlib>
#include "chains.h"
int main() {
  for (int most : {1, 2, 16})
    for (int n = 0; n < 60; ++n) {
      std::vector<double> load;
      for (int i = 0; i < n; ++i) load.push_back(1 + (i * 7919 % 97) * (i % 5 ? 1 : 50));
      std::sort(load.rbegin(), load.rend());
      const std::vector<int> c = rslb::assign_chains(load, most);
      std::vector<double> sum(most, 0.0);
      double all = 0.0;
      bool ok = (int)c.size() == n;
      for (int i = 0; i < n && ok; ++i) {
        ok = c[i] >= 0 && c[i] < most && (n > most || c[i] == i);
        if (ok) sum[c[i]] += load[i];
        all += load[i];
      }
      const double top = *std::max_element(sum.begin(), sum.end());
      if (n && top > all / most + load[0] + 1e-9) ok = false;
      if (!ok) {
        std::printf("%d chains, %d items: %g of %g\\n", most, n, top, all);
        return 1;
      }
    }
  return 0;
}
"""


def test_chains_are_bounded_and_even(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(MAIN)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
