"""The aligned units from which sample rows are padded: every wanted byte of an
exactly sized buffer, and no read outside it (host build of the kernel's header)."""
import os
import shutil
import subprocess

import pytest

SOURCE = r"""
#include <stdio.h>
#include <string.h>
#include <vector>
#include "mwax_rows.h"
struct Load {
  const uint8_t *lo, *hi;
  mutable int outside = 0;
  void check(const uint8_t *p, int n) const { outside += p < lo || p + n > hi; }
  mwax::Unit16 unit(const uint8_t *p) const {
    mwax::Unit16 u;
    check(p, 16);
    memcpy(&u, p, 16);
    return u;
  }
  uint8_t byte(const uint8_t *p) const { check(p, 1); return *p; }
};
int main() {
  alignas(16) static uint8_t mem[4096];
  for (int k = 0; k < 4096; ++k) mem[k] = (uint8_t)(k * 37 + 11);
  int outside = 0, wrong = 0;
  for (int N = 1; N <= 70; ++N)
    for (int rows = 1; rows <= 20; ++rows) {
      const uint8_t *end = mem + rows * N;
      const Load load{mem, end};
      for (int r = 0; r < rows; ++r)
        for (int x = 0; x < N; x += 16) {
          const int n = N - x < 16 ? N - x : 16;
          mwax::Unit16 u[2];
          const uint8_t *at = mem + r * N + x;
          const int s = end - (at + n) >= 15 ? mwax::units_of<true>(at, n, end, load, u[0], u[1])
                                             : mwax::units_of<false>(at, n, end, load, u[0], u[1]);
          wrong += memcmp(reinterpret_cast<uint8_t *>(u) + s, mem + r * N + x, n) != 0;
        }
      outside += load.outside;
    }
  printf("%d %d\n", outside, wrong);
}
"""


def test_units_stay_inside_the_buffer(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no C++ compiler")
    csrc = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0902_0915_gb300", "csrc")
    src, exe = tmp_path / "units.cpp", tmp_path / "units"
    src.write_text(SOURCE)
    subprocess.run([gxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-I", csrc, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split() == ["0", "0"]
