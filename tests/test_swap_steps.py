"""The state of a step that changes buffers (csrc/swap_steps.h) is back in buffer 0
after any number of steps and after a step that fails."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1612_01287_gb300", "csrc")

MAIN = """
#include <cstdio>
#include "swap_steps.h"
int main() {
  for (int n = 0; n <= 5; ++n)
    for (int fail = -1; fail <= n; ++fail)  // the step that fails (-1, n: none)
      for (int bad_copy = 0; bad_copy < 2; ++bad_copy) {
        int buf[2] = {0, -1}, calls = 0, copies = 0;
        const int e = rslb::swap_steps(
            n, 0,
            [&](int cur) {
              if (calls == fail) return 7;
              buf[cur ^ 1] = buf[cur] + 1;
              buf[cur] = -1;
              ++calls;
              return 0;
            },
            [&]() {
              ++copies;
              buf[0] = buf[1];
              return bad_copy ? 9 : 0;
            });
        const bool failed = fail >= 0 && fail < n;
        const int done = failed ? fail : n;
        const int want = failed ? 7 : (bad_copy && done % 2 ? 9 : 0);
        if (buf[0] != done || copies != done % 2 || e != want) {
          std::printf("%d %d %d: state %d, %d copies, error %d\\n", n, fail, bad_copy, buf[0],
                      copies, e);
          return 1;
        }
      }
  return 0;
}
"""


def test_state_returns_to_its_buffer(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(MAIN)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
