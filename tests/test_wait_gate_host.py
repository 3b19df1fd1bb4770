"""A role whose bounded wait has run out waits for nothing more, so that an error
return takes one wait limit and not one per remaining wait.  csrc/wait_gate.hpp
compiled for the host alone, walked as the tensor-core epilogue walks its ranges
and chunks."""
import os
import shutil
import subprocess

import pytest

from tests._lib import ROOT

CSRC = os.path.join(ROOT, "paper_2307_03930_gb300", "csrc")
SOURCE = r"""
#include "wait_gate.hpp"
int main() {
  const int ranges = 5, chunks = 4;
  for (int fails_at = 0; fails_at <= ranges * chunks; ++fails_at) {
    rosko::WaitGate gate;
    int waits = 0, written = 0;
    for (int r = 0; gate.open && r < ranges; ++r) {
      for (int c = 0; c < chunks; ++c)
        if (!gate([&] { return waits++ != fails_at; })) break;
      if (!gate.open) break;
      ++written;
    }
    const bool all = fails_at == ranges * chunks;
    if (waits != (all ? ranges * chunks : fails_at + 1)) return 1;
    if (written != fails_at / chunks || gate.open != all) return 2;
    // asked again, the gate neither waits nor opens
    if (!all && (gate([&] { ++waits; return true; }) || waits != fails_at + 1)) return 3;
  }
  return 0;
}
"""


def test_a_role_waits_no_more_after_an_expired_wait(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src = tmp_path / "t.cpp"
    src.write_text(SOURCE)
    exe = str(tmp_path / "t")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0


def test_the_epilogue_waits_through_the_gate():
    """Every wait for an accumulator in the epilogue goes through the gate."""
    text = open(os.path.join(CSRC, "spmm_dense_tc.cu")).read()
    epilogue = text[text.index("epilogue: TMEM -> registers -> C"):text.index("bulk_wait_all()")]
    assert epilogue.count("mbar_wait_bounded(") == 1
    assert "gate([&] {" in epilogue[:epilogue.index("mbar_wait_bounded(")]
    assert "while (gate.open && it.next(sg))" in epilogue
