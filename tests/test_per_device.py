"""A kernel's shared-memory attribute belongs to one device: the library sets it on every device
that it launches on.  The host-side helper that keeps track is plain C++ and runs here against
a fake of the attribute call; no GPU is used."""
import glob
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2607_17572_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.cuh"

#define EXPECT(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
enum Status { ok = 0, failed = 7 };

int main() {
  {  // once on each device, in any order
    jagg::OncePerDevice once;
    int calls[80] = {};
    for (int dev : {0, 1, 0, 63, 1, 63, 5}) EXPECT(once.run(dev, [&] { ++calls[dev]; return ok; }) == ok);
    EXPECT(calls[0] == 1 && calls[1] == 1 && calls[5] == 1 && calls[63] == 1);
    for (int k = 0; k < 2; ++k) EXPECT(once.run(64, [&] { ++calls[64]; return ok; }) == ok);
    EXPECT(calls[64] == 2);  // not tracked: made each time
  }
  {  // a failure is returned and not remembered
    jagg::OncePerDevice once;
    EXPECT(once.run(2, [] { return failed; }) == failed);
    int calls = 0;
    for (int k = 0; k < 2; ++k) EXPECT(once.run(2, [&] { ++calls; return ok; }) == ok);
    EXPECT(calls == 1);
  }
  // every thread finds the attribute set on its device when run() returns
  for (int round = 0; round < 200; ++round) {
    jagg::OncePerDevice once;
    std::atomic<int> set[4] = {};
    std::atomic<int> bad{0};
    std::vector<std::thread> ts;
    for (int t = 0; t < 8; ++t)
      ts.emplace_back([&, t] {
        const int dev = t & 3;
        once.run(dev, [&] { set[dev].store(1, std::memory_order_relaxed); return ok; });
        if (!set[dev].load(std::memory_order_relaxed)) ++bad;
      });
    for (auto& t : ts) t.join();
    EXPECT(bad == 0);
  }
  return 0;
}
"""


def test_once_per_device(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "t.cc", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_attributes_are_set_through_the_helper_only():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        calls = len(re.findall(r"\bcudaFuncSetAttribute\s*\(", open(path).read()))
        assert calls == (1 if os.path.basename(path) == "common.cuh" else 0), path
