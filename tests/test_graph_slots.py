"""The captured runs that are kept (wmc_graph_slots.cuh), checked on the host with
integers for graphs: the least recently used goes first, handles of an earlier
context are dropped and never destroyed or launched, other devices keep theirs;
and both the single and the batched form keep theirs this way."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1806_00082_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "wmc_graph_slots.cuh"

static int bad = 0;
static void check(bool ok, int line) {
  if (!ok) { std::printf("line %d\n", line); ++bad; }
}
#define CHECK(x) check(x, __LINE__)

int main() {
  wmc::GraphSlots<std::vector<int>, int, 4> g;
  std::vector<int> destroyed;
  auto kill = [&](int e) { destroyed.push_back(e); };
  auto find = [&](int dev, unsigned long long ctx, int k) {
    auto* s = g.find(dev, ctx, [&](const std::vector<int>& key) { return key == std::vector<int>{k}; });
    return s ? s->exec : -1;
  };
  auto add = [&](int dev, unsigned long long ctx, int k, int exec) { g.fill(g.take(kill), {k}, exec, dev, ctx); };
  // least recently used first
  for (int k = 0; k < 4; ++k) { CHECK(find(0, 1, k) == -1); add(0, 1, k, 100 + k); }
  CHECK(destroyed.empty());
  for (int k = 3; k >= 0; --k) CHECK(find(0, 1, k) == 100 + k);
  add(0, 1, 4, 104);
  CHECK(destroyed == std::vector<int>{103} && find(0, 1, 3) == -1 && find(0, 1, 0) == 100);
  // another device's graphs are no match and stay
  CHECK(find(1, 9, 4) == -1);
  add(1, 9, 4, 204);
  CHECK(destroyed == (std::vector<int>{103, 102}) && find(1, 9, 4) == 204 && find(0, 1, 4) == 104);
  // a new context on device 0: its handles are gone, not destroyed, and their slots come first
  CHECK(find(0, 2, 4) == -1 && find(0, 2, 0) == -1 && find(1, 9, 4) == 204);
  for (int k = 0; k < 3; ++k) add(0, 2, k, 300 + k);
  CHECK(destroyed.size() == 2 && find(1, 9, 4) == 204 && find(0, 2, 2) == 302);
  // a slot that was taken but not filled (a capture that failed) is empty
  g.take(kill);
  CHECK(destroyed.size() == 3);
  g.take(kill);
  CHECK(destroyed.size() == 3);
  return bad != 0;
}
"""


def test_kept_graphs(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src = tmp_path / "slots.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "slots"
    subprocess.run([cxx, "-std=c++17", "-Wall", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


@pytest.mark.parametrize("form", ["wmc_api.cu", "wmc_batch.cu"])
def test_graphs_are_looked_up_with_their_context(form):
    src = open(os.path.join(CSRC, form)).read()
    assert src.count("slots.find(dev, ctx,") == 1 and src.count("current_context_id();") >= 1
    launches = [line for line in src.splitlines() if "cudaGraphLaunch(" in line]
    assert launches and all("hit->exec" in line for line in launches)
