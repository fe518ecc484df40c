"""The retry of launches that need all their blocks resident, with a fake launch that
refuses grids above what a partition of the GPU would take."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1310_6380_gb300", "csrc")
SRC = r"""
#include <cstdio>
#include "shrink_grid.h"
enum { OK = 0, TOO_LARGE = 720, OTHER = 700 };
int main() {
  const int room[] = {304, 303, 100, 5, 1, 0}, want[] = {304, 152, 76, 4, 1, 1};
  for (int i = 0; i < 6; ++i) {
    int calls = 0, last = 0;
    const int e = bs_shrink_grid(304, (int)TOO_LARGE, [&](int g) {
      ++calls;
      last = g;
      return g <= room[i] ? OK : TOO_LARGE;
    });
    if (last != want[i] || e != (room[i] ? OK : TOO_LARGE) || calls > 10) return 10 + i;
  }
  int calls = 0;   // any other error ends it
  if (bs_shrink_grid(304, (int)TOO_LARGE, [&](int) { ++calls; return (int)OTHER; }) != OTHER) return 20;
  return calls == 1 ? 0 : 21;
}
"""


def test_shrinks_until_it_fits(tmp_path):
    cc = shutil.which("g++") or shutil.which("c++")
    if cc is None:
        pytest.skip("no C++ compiler")
    (tmp_path / "t.cpp").write_text(SRC)
    exe = str(tmp_path / "t")
    r = subprocess.run([cc, "-std=c++17", "-I", CSRC, str(tmp_path / "t.cpp"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    assert subprocess.run([exe], timeout=60).returncode == 0


def test_the_list_reduction_uses_it():
    src = open(os.path.join(CSRC, "tridiag.cu")).read()
    body = src[src.index("int bs_launch_tridiag_list("):]
    body = body[:body.index("\n}\n")]
    assert "bs_shrink_grid(" in body
    assert body.count("cudaLaunchCooperativeKernel") == 1
