"""The 32-way search of the in-place compaction on the CPU: its interval arithmetic (csrc/warp_search.cuh), compiled for the
host, for every answer of every list length up to 4096 and around the lengths that take one more round."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "paper_2609_31395_b200", "csrc", "warp_search.cuh")

PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include "warp_search.cuh"
using namespace actkv;
// a strictly ascending list of n entries of which `answer` are below the key
static int search(int n, int answer) {
  SearchSpan s{0, n};
  int rounds = 0;
  while (s.hi - s.lo > 32) {
    int below = 0;
    for (int i = 0; i < 32; ++i) below += search_probe(s, i) < s.hi && search_probe(s, i) < answer;
    s = search_narrow(s, below);
    if (s.lo < 0 || s.hi > n || s.hi < s.lo || ++rounds > 8) return -1;
  }
  int below = 0;
  for (int i = 0; i < 32; ++i) below += s.lo + i < s.hi && s.lo + i < answer;
  return s.lo + below;
}
int main() {
  long long bad = 0;
  auto all = [&](int n, int every) {
    for (int answer = 0; answer <= n; answer += every) bad += search(n, answer) != answer;
    bad += search(n, n) != n;
  };
  for (int n = 0; n <= 4096; ++n) all(n, 1);
  for (int n : {11847, 35937}) for (int d = -34; d <= 34; ++d) all(n + d, 1);
  for (int n : {1185921, 0x7fffffff / 2}) for (int d = -1; d <= 1; ++d) all(n + d, 10007);
  std::printf("%lld\n", bad);
  return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_every_answer(tmp_path):
    src = tmp_path / "search.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "search")
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", os.path.dirname(HEADER), str(src), "-o", exe], check=True)
    res = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert res.returncode == 0 and int(res.stdout) == 0, res.stdout
