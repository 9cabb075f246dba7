"""The ring of stages on the CPU (csrc/ring.cuh, compiled for the host): after a give-up the kernel waits for exactly those of the
producers' loads that are still in flight, wherever in the ring it and the other one stopped."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "paper_2609_31395_b200", "csrc", "ring.cuh")

PROGRAM = r"""
#include <algorithm>
#include <cstdio>
#include <vector>
#include "ring.cuh"
using namespace actkv;
int main() {
  long long bad = 0;
  for (int S = 2; S <= 8; ++S)
    for (int end0 = 0; end0 <= 40; ++end0)
      for (int end1 = std::max(0, end0 - S); end1 <= end0 + S; ++end1) {
        const int ends[2] = {end0, end1};
        // an entry is issued when it is its producer's turn and the stage's previous entry has landed and been consumed
        for (int flight = 0; flight < 1 << S; ++flight) {           // stages whose last load is still in flight
          std::vector<int> last(S, -1);
          bool possible = true;
          for (int e = 0; e < std::max(end0, end1); ++e)
            if (e < ends[e % 2]) { possible = possible && (e < S || last[e % S] == e - S); last[e % S] = e; }
          if (!possible) continue;
          std::vector<int> phases(S);                               // completed phases of the stage's barrier
          for (int s = 0; s < S; ++s) phases[s] = last[s] < 0 ? 0 : last[s] / S + ((flight >> s & 1) ? 0 : 1);
          // what the producers recorded; a wait for parity x passes when the phase under way has the other parity
          std::vector<unsigned> recorded(S, RING_UNUSED);
          for (int e = 0; e < std::max(end0, end1); ++e)
            if (e < ends[e % 2]) recorded[ring_stage(e, S)] = ring_parity(e, S);
          std::vector<bool> held(S);
          for (int s = 0; s < S; ++s) held[s] = (unsigned)(phases[s] & 1) == recorded[s];
          for (int s = 0; s < S; ++s) bad += held[s] != (last[s] >= 0 && (flight >> s & 1));
        }
      }
  std::printf("%lld\n", bad);
  return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_loads_in_flight_are_waited_for(tmp_path):
    src = tmp_path / "ring.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "ring")
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", os.path.dirname(HEADER), str(src), "-o", exe], check=True)
    res = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert res.returncode == 0 and int(res.stdout) == 0, res.stdout
