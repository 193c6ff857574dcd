"""Tensor memory is there before the next kernel may be scheduled: the end of the set-up of the Dense and the short-row
attention kernels (csrc/setup.cuh) compiled for the host, its warps as threads, the allocation as slow as it can be."""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2207_01405_b200", "csrc")

SOURCE = r"""
#include <atomic>
#include <chrono>
#include <condition_variable>
#include <cstdio>
#include <mutex>
#include <thread>
#include <vector>
#include "setup.cuh"

constexpr int kWarps = 6;
std::mutex m;
std::condition_variable cv;
int arrived = 0;
std::atomic<bool> allocated{false};
std::atomic<int> early{0}, triggers{0};

struct Cta {
  void arrive() const { std::lock_guard<std::mutex> l(m); if (++arrived == kWarps) cv.notify_all(); }
  void sync() const {
    std::unique_lock<std::mutex> l(m);
    if (++arrived == kWarps) cv.notify_all();
    cv.wait(l, [] { return arrived == kWarps; });
  }
  void trigger() const { ++triggers; if (!allocated) ++early; }
};

int main() {
  std::vector<std::thread> warps;
  for (int w = 0; w < kWarps; ++w)
    warps.emplace_back([w] {
      if (w == 1) { std::this_thread::sleep_for(std::chrono::milliseconds(200)); allocated = true; }
      ivit::end_of_setup(Cta{}, w == 0);
    });
  for (std::thread& t : warps) t.join();
  std::printf("%d triggers, %d early\n", (int)triggers, (int)early);
  return triggers > 0 && early == 0 ? 0 : 1;
}
"""


def test_no_warp_triggers_before_the_allocation(tmp_path):
    (tmp_path / "t.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I", CSRC, str(tmp_path / "t.cpp"), "-o", str(tmp_path / "t")], check=True)
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_kernels_with_tensor_memory_trigger_behind_a_barrier():
    """Every kernel that allocates tensor memory either ends its set-up through end_of_setup, or triggers after a barrier
    of the whole CTA that stands behind the allocation."""
    seen = 0
    for name in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        for body in text.split("__global__")[1:]:
            at = re.search(r"\btmem_alloc(_pair)?\(", body)
            if not at:
                continue
            seen += 1
            trigger = re.search(r"\bpdl_trigger\(\)", body)
            if "end_of_setup(" in body:
                assert not trigger, f"{name}: a trigger besides that of end_of_setup"
            elif trigger:
                assert "__syncthreads()" in body[at.start():trigger.start()], f"{name}: trigger without a barrier behind the allocation"
    assert seen >= 5
