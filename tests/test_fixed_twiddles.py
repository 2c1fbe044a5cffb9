"""Host check of the Q61 twiddles of the fixed-point complex128 lines
(qfd::fixed_twiddle_table in csrc/qfd_launch.h): balanced limbs that add up to
cos and -sin of 2 pi e / n to half a unit of 2^-61 (long double evaluation adds
at most one more bit)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2006_16935_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "qfd_launch.h"
int main(int argc, char** argv) {
  const long n = std::atol(argv[1]);
  std::vector<double2> t(n);
  qfd::fixed_twiddle_table(n, t.data());
  std::fwrite(t.data(), sizeof(double2), n, stdout);
  return 0;
}
"""


@pytest.mark.parametrize("n", [8, 96, 192, 512, 1024])
def test_fixed_point_twiddles(tmp_path, n):
    mp = pytest.importorskip("mpmath")
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx or not os.path.isdir(CUDA_INC):
        pytest.skip("needs a host C++ compiler and the CUDA headers")
    src, exe = tmp_path / "h.cpp", tmp_path / "h"
    src.write_text(HARNESS)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I" + CUDA_INC, "-I" + CSRC, str(src), "-o", str(exe)], check=True)
    t = np.frombuffer(subprocess.run([str(exe), str(n)], check=True, capture_output=True).stdout, dtype=np.int32)
    t = t.reshape(n, 4).astype(object)
    mp.mp.prec = 120
    for e in range(n):
        a = 2 * mp.pi * e / n
        for (l, h), want in ((t[e, :2], mp.cos(a)), (t[e, 2:], -mp.sin(a))):
            assert abs(h) <= 2 ** 29
            assert abs(int(h) * 2 ** 32 + int(l) - want * 2 ** 61) <= 1
