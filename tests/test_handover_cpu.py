"""The hand-over between the control warp of the short-row attention kernel and its Shiftmax threads, after a wait that ran
out: the kernel's own routine (csrc/handover.cuh) compiled for the host and run against hardware barriers modelled as
arrival counts.  The control warp gets as far as it can before the Shiftmax warps move."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <chrono>
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <mutex>
#include <thread>
#include <vector>
#include "handover.cuh"

// A barrier of the block: counts the arrivals of 32 threads at a time, whoever makes them; the phase ends at `total`.
struct Bar {
  std::mutex m;
  std::condition_variable cv;
  int total = 0, count = 0;
  long phase = 0;
  void arrive_locked() { count += 32; if (count >= total) { count -= total; ++phase; cv.notify_all(); } }
  void arrive() { std::lock_guard<std::mutex> l(m); arrive_locked(); }
  void sync() {
    std::unique_lock<std::mutex> l(m);
    const long p = phase;
    arrive_locked();
    if (!cv.wait_for(l, std::chrono::seconds(5), [&] { return phase > p; })) { std::puts("stuck"); std::_Exit(1); }
  }
};
Bar bars[16];
struct Barriers {
  void sync(int id) const { bars[id].sync(); }
  void arrive(int id) const { bars[id].arrive(); }
};

int main(int argc, char** argv) {
  const int warps = std::atoi(argv[1]);
  const unsigned items = std::atoi(argv[2]), done = std::atoi(argv[3]);
  const bool scores_out = std::atoi(argv[4]) != 0;
  for (Bar& b : bars) b.total = 32 * (warps + 1);
  std::vector<std::thread> all;
  all.emplace_back([&] {
    if (scores_out) bars[ivit::kBarScores].arrive();
    ivit::walk_out(Barriers{}, done, items, scores_out);
  });
  std::this_thread::sleep_for(std::chrono::milliseconds(100));
  for (int w = 0; w < warps; ++w)
    all.emplace_back([&] {
      for (unsigned n = done; n < items; ++n) { bars[ivit::kBarScores].sync(); bars[ivit::kBarOutput].sync(); }
    });
  for (std::thread& t : all) t.join();
  for (int id : {ivit::kBarScores, ivit::kBarOutput})
    if (bars[id].count != 0 || bars[id].phase != (long)(items - done)) { std::puts("phases"); return 1; }
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("handover")
    (d / "t.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I", os.path.join(ROOT, "paper_2207_01405_b200", "csrc"),
                    str(d / "t.cpp"), "-o", str(d / "t")], check=True)
    return str(d / "t")


# four, eight and sixteen Shiftmax warps: packed windows and single images; few items and more than a phase takes arrivals
@pytest.mark.parametrize("scores_out", [0, 1])
@pytest.mark.parametrize("warps,items,done", [(8, 1, 0), (8, 2, 1), (8, 40, 3), (4, 25, 0), (4, 6, 5), (16, 1, 0)])
def test_everyone_leaves_after_a_wait_that_ran_out(program, warps, items, done, scores_out):
    assert subprocess.run([program, str(warps), str(items), str(done), str(scores_out)], timeout=60).returncode == 0
