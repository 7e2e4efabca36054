"""The ring of B stages of the tensor-memory row kernel (wmc_ta_ring.cuh), checked
on the host: no wait of an issuing thread can pass before its copy has landed,
whatever order the copies land in, and no stage is filled while it is read."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1806_00082_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "wmc_ta_ring.cuh"
using namespace wmc;

// A wait for a parity passes while the barrier has completed c phases iff
// parity != c % 2.
static bool passes(int c, unsigned parity) { return (unsigned)(c & 1) != parity; }

int main() {
  int bad = 0, waits = 0;
  for (int KB = 1; KB <= kTaMaxKB; ++KB)
    for (int n_my = 1; n_my <= kTaMaxTiles; ++n_my) {
      const int KP = (KB + 1) / 2, n = n_my * KP;
      if (n > kTaFills) { std::printf("KB %d, %d tiles: %d fillings\n", KB, n_my, n); ++bad; continue; }
      for (int me = 0; me < kTaIssuers; ++me)
        for (int t = 0; t < n; ++t) {
          if ((t / KP) % kTaIssuers != me) continue;
          // of the earlier fillings on this barrier, this thread knows those landed that are not
          // after the last one it has waited for; the others may or may not have
          int k = 0, seen = 0;
          for (int u = 0; u < t; ++u)
            if (ta_full_bar(u) == ta_full_bar(t)) {
              ++k;
              if ((u / KP) % kTaIssuers == me) seen = k;
            }
          ++waits;
          for (int c = seen; c <= k; ++c)
            if (passes(c, ta_full_parity(t))) {
              std::printf("KB %d, %d tiles: filling %d passes after %d of %d phases\n", KB, n_my, t, c, k);
              ++bad;
            }
          if (!passes(k + 1, ta_full_parity(t))) { std::printf("filling %d waits for ever\n", t); ++bad; }
        }
      // the copying thread waits for every phase of a stage's empty barrier in turn: one is complete
      // for each filling of the stage before t
      for (int t = kTaStages; t < n; ++t) {
        const int c = t / kTaStages - 1;
        if (ta_stage(t) != ta_stage(t - kTaStages) || passes(c, ta_empty_parity(t)) || !passes(c + 1, ta_empty_parity(t))) {
          std::printf("stage of filling %d\n", t);
          ++bad;
        }
      }
    }
  std::printf("%d waits, %d bad\n", waits, bad);
  return bad != 0;
}
"""


def test_no_wait_passes_before_its_copy(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src = tmp_path / "ring.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "ring"
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout[-2000:]
