"""What a caller of the pivoted Cholesky factor makes of the kernel's report (csrc/pcholout.h), compiled
for the host: a wait that gave up is neither a zero matrix nor an empty factor."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2309_08572_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include "pcholout.h"
using namespace mpdo;
int main() {
  auto put = [](int r, double resid, int n, int rmax) {
    std::printf("%d ", (int)pchol_fit({r, 0, resid}, n, rmax, 1e-16));
  };
  put(kPcholGaveUp, 0.0, 60, 60);   // a wait gave up
  put(kPcholGaveUp, 0.0, 200, 168);
  put(0, 0.0, 60, 60);              // zero or non-finite
  put(12, 1e-17, 60, 60);           // fits
  put(60, 0.5, 60, 60);             // all columns
  put(168, 1e-17, 200, 168);        // just fits
  put(168, 1e-12, 200, 168);        // needs more
}
"""


def test_outcomes(tmp_path):
    cxx = shutil.which("g++") or pytest.skip("no host compiler")
    (tmp_path / "t.cpp").write_text(DRIVER)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(tmp_path / "t.cpp"), "-o",
                    str(tmp_path / "t")], check=True)
    out = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True, check=True).stdout
    fits, zero, full = 0, 1, 2
    assert list(map(int, out.split())) == [full, full, zero, fits, fits, fits, full]
