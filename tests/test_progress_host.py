"""The progress counters of the persistent kernels (csrc/progress.h), compiled for the host: waits stay right where
the 32-bit counter and its target run past 2^32, at any length of a launch."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2109_05072_gb300", "csrc")

PROBE = r"""
#include <cstdio>
#include "progress.h"
using namespace ceedgb;
int main() {
  // pieces of work per colour and iteration: one, the 64^3 mesh's, a large odd count
  const uint32_t works[3] = {1u, 32768u, 1000003u};
  for (uint32_t w : works) {
    const uint64_t wrap = ((uint64_t)1 << 32) / w;   // iterations until the counter runs past 2^32
    for (int64_t d = -3; d <= 3; ++d) {
      const uint64_t it = wrap + d;
      const uint64_t before = it * w, after = (it + 1) * w;   // exact counts around iteration `it`
      const uint32_t target = progress_target(w, (uint32_t)it);
      if (target != (uint32_t)after) return printf("target\n"), 1;
      if (progress_reached((uint32_t)before, target)) return printf("passed early: w %u d %d\n", w, (int)d), 1;
      if (progress_reached((uint32_t)(after - 1), target)) return printf("passed one early: w %u d %d\n", w, (int)d), 1;
      if (!progress_reached((uint32_t)after, target)) return printf("never passed: w %u d %d\n", w, (int)d), 1;
    }
  }
  return 0;
}
"""


def test_counters_wrap(tmp_path):
    cc = shutil.which("g++") or shutil.which("c++")
    if cc is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "probe.cpp", tmp_path / "probe"
    src.write_text(PROBE)
    subprocess.run([cc, "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
