"""A kernel's shared-memory limit is a setting of a device, and the calls that make it come from any thread: the guard
around it, without a GPU.  Every device gets its setting, whichever came first; nobody goes on before it is made; a failure
is tried again; and no kernel's limit is set past that guard."""
import glob
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1906_09108_b200", "csrc")

PROGRAM = r"""
#include <thread>
#include <vector>
#include "once_per_device.h"
int main() {
  fdg::OncePerDevice once;
  std::atomic<int> made[3] = {{0}, {0}, {0}};
  int calls = 0;
  if (once.run(0, [&]() { ++calls; return 7; }) != 7) return 1;             // a failure is reported ...
  if (once.run(0, [&]() { ++calls; return 0; }) != 0 || calls != 2) return 2;   // ... and tried again
  if (once.run(0, [&]() { ++calls; return 0; }) != 0 || calls != 2) return 3;   // a success is not
  if (once.run(1, [&]() { ++calls; return 0; }) != 0 || calls != 3) return 4;   // another device has its own
  if (once.run(64, [&]() { ++calls; return 0; }) != 0 || once.run(64, [&]() { ++calls; return 0; }) != 0 || calls != 5) return 5;
  for (int round = 0; round < 200; ++round) {
    fdg::OncePerDevice fresh;
    for (auto& m : made) m = 0;
    std::atomic<int> early{0};
    std::vector<std::thread> threads;
    for (int t = 0; t < 6; ++t)
      threads.emplace_back([&, t]() {
        const int dev = t % 3;
        if (fresh.run(dev, [&]() { std::this_thread::yield(); ++made[dev]; return 0; }) != 0 || made[dev] == 0) ++early;
      });
    for (auto& t : threads) t.join();
    if (early) return 6;
    for (auto& m : made) if (m < 1) return 7;
  }
  return 0;
}
"""


def test_once_per_device(tmp_path):
    src, exe = tmp_path / "once.cpp", str(tmp_path / "once")
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I", CSRC, "-o", exe, str(src)], check=True)
    assert subprocess.run([exe]).returncode == 0


def test_every_limit_is_set_through_the_guard():
    text = {f: open(f).read() for ext in ("*.cuh", "*.cu", "*.inc") for f in glob.glob(os.path.join(CSRC, ext))}
    assert sum(t.count("cudaFuncSetAttribute(") for t in text.values()) == 1       # set_smem_limit's own
    assert not [f for f, t in text.items() if re.search(r"static bool \w+ *(=|;)", t)]
    for f, t in text.items():
        uses = t.count("set_smem_limit(") - t.count("set_smem_limit(Kernel")
        assert uses == 0 or "static OncePerDevice once;" in t, f
