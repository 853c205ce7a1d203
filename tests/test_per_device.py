"""Per-device set-up: made once on every device, by whichever thread comes first, tried again
after a failure, and refused for a device number outside the table."""
import os
import shutil
import subprocess

import pytest

SRC = r"""
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"
int main() {
  static trinity::PerDevice p;
  std::atomic<int> calls[trinity::kMaxDevices] = {};
  std::atomic<int> wrong{0};
  std::vector<std::thread> ts;
  for (int t = 0; t < 8; ++t)
    ts.emplace_back([&] {
      for (int rep = 0; rep < 200; ++rep)
        for (int dev = 0; dev < trinity::kMaxDevices; ++dev)
          if (p.get(dev, [&] { ++calls[dev]; return 100 + dev; }) != 100 + dev) ++wrong;
    });
  for (auto& t : ts) t.join();
  for (int dev = 0; dev < trinity::kMaxDevices; ++dev) wrong += calls[dev] != 1;
  static trinity::PerDevice q;
  wrong += q.get(3, [] { return 0; }) != 0;
  wrong += q.get(3, [] { return 7; }) != 7;
  wrong += q.get(2, [] { return 9; }) != 9;
  wrong += q.get(-1, [] { return 1; }) != 0;
  wrong += q.get(trinity::kMaxDevices, [] { return 1; }) != 0;
  std::printf("%d\n", wrong.load());
  return wrong.load() != 0;
}
"""


def test_every_device_is_set_up_once(tmp_path, repo_root):
    cxx = shutil.which("g++") or pytest.skip("no host compiler")
    src = tmp_path / "t.cpp"
    src.write_text(SRC)
    csrc = os.path.join(repo_root, "paper_2105_01028_gb300", "csrc")
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", csrc, str(src), "-o", str(tmp_path / "t")], check=True)
    assert subprocess.run([str(tmp_path / "t")]).returncode == 0


def test_launch_attributes_are_set_per_device(repo_root):
    """Every kernel that raises its shared-memory limit does so through the per-device table, or
    before each launch (the staged sweep)."""
    csrc = os.path.join(repo_root, "paper_2105_01028_gb300", "csrc")
    for name in sorted(os.listdir(csrc)):
        text = open(os.path.join(csrc, name)).read()
        if name.endswith(".cu") and "cudaFuncAttributeMaxDynamicSharedMemorySize" in text and name != "sweep_tma.cu":
            assert "configured_sms(" in text, name
