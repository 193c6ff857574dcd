"""The producer's last wait for its own loads (csrc/ring.cuh), compiled for the host and run against stage barriers modelled
by the number of their completed phases, for every number of loads requested and every number of them still in flight."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include "ring.cuh"

int main() {
  for (int stages = 1; stages <= 8; ++stages)
    for (int requested = 0; requested <= 40; ++requested)
      for (int flying = 0; flying <= stages && flying <= requested; ++flying) {
        // loads 0 .. requested - flying - 1 have landed; the others land only when somebody waits for them
        int completed[8] = {0}, asked[8] = {0};
        for (int kb = 0; kb < requested; ++kb) { ++asked[kb % stages]; if (kb < requested - flying) ++completed[kb % stages]; }
        ivit::drain_ring(requested, stages, [&](int stage, unsigned parity) {
          // a wait for a parity is over as soon as the present phase has the other one
          if ((unsigned)(completed[stage] & 1) == parity) ++completed[stage];
        });
        for (int s = 0; s < stages; ++s)
          if (completed[s] != asked[s]) { std::printf("stages %d requested %d flying %d: stage %d\n", stages, requested, flying, s); return 1; }
      }
  return 0;
}
"""


def test_every_requested_load_is_waited_for(tmp_path):
    (tmp_path / "t.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_2207_01405_b200", "csrc"), str(tmp_path / "t.cpp"),
                    "-o", str(tmp_path / "t")], check=True)
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
