"""Shared-memory indices of the tensor-core band sweep, enumerated on the CPU from
the arithmetic that the kernel itself is compiled with (csrc/sweep_index.h)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1906_10944_gb300", "csrc")

# For every block height B, cluster size C and half width w that one class can
# bring together (C is chosen for the class's widest matrix, the others may be as
# narrow as the block height allows): the lowest shared address that block kk
# loads for block j, and every block that holds an entry of kk's rows in band.
PROGRAM = r"""
#include <cstdio>
#include "sweep_index.h"
using namespace geneo;
int main() {
  long bad = 0, missed = 0, lowest = 0;
  for (int B = 16; B <= 64; B *= 2)
    for (int C = 1; C <= 8; C *= 2)
      for (int w = B - 1; w <= 1100; w += w < 600 ? 1 : 13) {
        const int SR = B < 32 ? B : 32, ld = (w + 4) & ~3;
        const int nb = reach_blocks(w, B, C) + C + 2;
        for (int kk = 0; kk < nb; ++kk) {
          const int first = forward_first(kk, w, B, C);
          for (int j = first; j < kk; ++j) {
            for (int r = 0; r < B; r += SR) {
              const long at = slot_lead(C) + 4L * slot_offset(kk, r, j * B, w, ld, B, SR);
              if (at < lowest) lowest = at;
              if (at < 0) ++bad;
            }
          }
          for (int j = 0; j < kk; ++j) {
            const bool holds = j * B + B - 1 >= kk * B - w;   // a column in the first row's band
            if (holds && j < first) ++missed;
          }
          // every block that arrives between two blocks of an owner is waited for
          if (kk >= C - 1 && first > kk - C + 1) ++missed;
          if (kk - first >= ring_blocks(w, B, C)) ++bad;
        }
      }
  std::printf("%ld %ld %ld\n", bad, missed, lowest);
}
"""


def test_forward_loads_stay_in_shared_memory(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("needs a host C++ compiler")
    src = tmp_path / "index.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "index")
    subprocess.run([gxx, "-O1", "-std=c++17", "-I" + CSRC, str(src), "-o", exe], check=True)
    bad, missed, lowest = map(int, subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    assert (bad, missed) == (0, 0), (bad, missed, lowest)
