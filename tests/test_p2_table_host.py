"""P2Table::holds decides whether one table of off-diagonal entries serves a
coarser level too: equal wherever the level has the coupling, whatever the
entries it lacks."""
import os
import shutil
import subprocess

import pytest

from paper_2501_11767_gb300 import build as B

PROGRAM = r"""
#include "p2stencil.h"
using namespace chnss;
int main() {
  P2Table a;
  for (int k = 0; k < kP2Slots + kP2TopSlots; ++k) {
    a.seen[k] = true;
    a.c[2 * k] = k + 0.25;
    a.c[2 * k + 1] = -k;
  }
  P2Table b = a;
  if (!b.holds(a)) return 1;
  b.seen[7] = false;                 // the level lacks a coupling
  b.c[14] = b.c[15] = 0.0;
  if (!b.holds(a)) return 2;
  if (a.holds(b)) return 3;          // ... which the other one has
  b.c[2 * 9 + 1] *= 1 + 1e-15;       // one rounding apart
  if (b.holds(a)) return 4;
  return 0;
}
"""


def test_holds(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not shutil.which("g++") or not os.path.exists(nvcc):
        pytest.skip("needs g++ and the CUDA headers")
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    subprocess.run(["g++", "-std=c++17", str(src), "-o", str(tmp_path / "t"),
                    "-I" + B.CSRC, "-I" + B.INCLUDE, "-isystem", cuda], check=True)
    assert subprocess.run([str(tmp_path / "t")]).returncode == 0
