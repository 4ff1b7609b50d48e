"""A parked kNN key never ties with the padding key: a boundary bucket counts as
fitting only if its largest offset, shifted over the position bits, stays below
the offset field of 0xFFFFFFFF.  (A 2^20-pattern bucket with 12 position bits has
offsets up to 0xFFFFF, the padding's own: the padding then joined the ties at the
cut.)  Host build of the kernel's header."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_10386_gb300", "csrc")

PROGRAM = r"""
#include "gd_knn_select.cuh"
#include <cstdio>
int main() {
  for (uint32_t pbits = 1; pbits < 32; ++pbits)
    for (int64_t d = -3; d <= 3; ++d) {
      const int64_t range = (1ll << (32 - pbits)) - 1 + d;
      if (range < 0 || range > 0x7FFFFFFEll) continue;
      const gd::SelCut cut{(int32_t)range, -1, 0u, 1u, 0};
      const bool fits = gd::sel_fits(cut, pbits);
      const bool apart = (uint64_t)range < (0xFFFFFFFFu >> pbits);
      if (fits != apart) { std::printf("pbits %u range %lld fits %d\n", pbits, (long long)range, (int)fits); return 1; }
    }
  return 0;
}
"""


def test_offsets_stay_below_the_padding(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not available")
    src, exe = tmp_path / "fits.cpp", tmp_path / "fits"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
