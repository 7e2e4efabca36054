"""The batched step's work ranges (wmc_batch_ranges.cuh), checked on the host: the
sizes that are timed against each other differ, and every accepted one is among
them."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1806_00082_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "wmc_batch_ranges.cuh"
using namespace wmc;

int main() {
  int bad = 0;
  for (const int a : kTuneCandidates) {
    if (!valid_per_thread(a)) { std::printf("%d is refused\n", a); ++bad; }
    for (const int b : kTuneCandidates)
      if (a != b && batch_max_range(a) == batch_max_range(b)) { std::printf("%d and %d are the same\n", a, b); ++bad; }
  }
  for (int per = 1; per <= 512; ++per) {
    if (!valid_per_thread(per)) continue;
    bool found = false;
    for (const int a : kTuneCandidates) found |= batch_max_range(a) == batch_max_range(per);
    if (!found) { std::printf("%d is not timed\n", per); ++bad; }
  }
  return bad != 0;
}
"""


def test_the_tuner_times_every_schedule_once(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src = tmp_path / "ranges.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "ranges"
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
