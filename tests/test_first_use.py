"""CPU: a device's first use runs alone (csrc/scw_first_use.h, which guards a process's first eigendecomposition):
once per device, with every other caller waiting, and again after a failure."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DRIVER = r"""
#include <atomic>
#include <chrono>
#include <cstdio>
#include <thread>
#include "scw_first_use.h"
int main() {
  scw::FirstUse u;
  std::atomic<int> inside{0}, calls{0}, overlaps{0}, after{0};
  std::vector<std::thread> th;
  for (int i = 0; i < 16; ++i)
    th.emplace_back([&, i] {
      bool ran = false;
      const bool ok = u.alone(i % 2, ran, [&] {
        if (inside.fetch_add(1)) ++overlaps;
        ++calls;
        std::this_thread::sleep_for(std::chrono::milliseconds(20));
        inside.fetch_sub(1);
        return calls > 1;  // the very first use fails
      });
      if (ok && !ran) ++after;
    });
  for (auto& t : th) t.join();
  bool ran = true;
  const bool ok = u.alone(0, ran, [&] { return false; });
  std::printf("%d %d %d %d %d\n", (int)calls, (int)overlaps, (int)after, (int)ok, (int)ran);
}
"""


def test_first_use_is_alone(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    (tmp_path / "t.cpp").write_text(DRIVER)
    subprocess.run([gxx, "-std=c++17", "-pthread", "-I", os.path.join(ROOT, "paper_2404_07293_gb300", "csrc"),
                    "-o", str(tmp_path / "t"), str(tmp_path / "t.cpp")], check=True)
    out = subprocess.run([str(tmp_path / "t")], check=True, capture_output=True, text=True, timeout=60).stdout.split()
    # three calls (one failed, one per device), never two at once; 13 callers found it done; a later one does not run it
    assert out == ["3", "0", "13", "1", "0"]
