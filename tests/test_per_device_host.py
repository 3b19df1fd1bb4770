"""A kernel's shared-memory limit is remembered per device: the first launch on
each device sets it, a device's limit never shrinks, a failure is tried again,
and threads that raise it together leave it at the largest.  csrc/per_device.hpp
compiled for the host alone."""
import os
import shutil
import subprocess

import pytest

from tests._lib import ROOT

CSRC = os.path.join(ROOT, "paper_2307_03930_gb300", "csrc")
SOURCE = r"""
#include "per_device.hpp"
#include <cstdio>
#include <thread>
#include <vector>
int main() {
  rosko::SmemLimit a;
  int calls = 0;
  auto ok = [&](int) { ++calls; return true; };
  auto fails = [&](int) { ++calls; return false; };
  // every device once, whatever another device has
  for (int dev = 0; dev < 8; ++dev)
    for (int k = 0; k < 3; ++k)
      if (!a.ensure(dev, 1000, ok) || calls != dev + 1) return 1;
  // fewer bytes: nothing to do; more: set again, on that device only
  if (!a.ensure(3, 500, ok) || calls != 8) return 2;
  if (!a.ensure(3, 2000, ok) || calls != 9 || !a.ensure(4, 1000, ok) || calls != 9) return 3;
  // a failure is reported and not remembered
  rosko::SmemLimit b;
  calls = 0;
  if (b.ensure(1, 64, fails) || b.ensure(1, 64, fails) || calls != 2) return 4;
  if (!b.ensure(1, 64, ok) || calls != 3) return 5;
  // devices that are not remembered are set each time
  if (!b.ensure(100, 64, ok) || !b.ensure(100, 64, ok) || calls != 5) return 6;
  // together: the limit that was set last is the largest that was asked for
  rosko::SmemLimit c;
  int limit = 0;
  std::vector<std::thread> ts;
  for (int i = 1; i <= 16; ++i)
    ts.emplace_back([&, i] { c.ensure(0, 100 * i, [&](int n) { limit = n; return true; }); });
  for (auto& t : ts) t.join();
  return limit == 1600 ? 0 : 7;
}
"""


def test_limits_are_kept_per_device(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src = tmp_path / "t.cpp"
    src.write_text(SOURCE)
    exe = str(tmp_path / "t")
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0


def test_no_launch_site_keeps_its_own_flag():
    """cudaFuncSetAttribute is called in one place, which asks a SmemLimit."""
    sites = [f for f in sorted(os.listdir(CSRC))
             if "cudaFuncSetAttribute(" in open(os.path.join(CSRC, f)).read()]
    assert sites == ["common.cuh"]
