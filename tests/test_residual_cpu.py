"""The projector's convergence measure on the host: a residual or value that
is not finite makes the round count as diverged, wherever it stands."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1808_10804_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include "residual.h"
int main() {
  const double inf = std::numeric_limits<double>::infinity(), nan = std::numeric_limits<double>::quiet_NaN();
  const double lists[][3] = {{1e-9, 3e-9, 2e-9}, {nan, 1e-9, 2e-9}, {1e-9, nan, 2e-9}, {1e-9, 2e-9, nan},
                             {nan, nan, nan},    {inf, 0, 0},       {0, -inf, 0}};
  for (auto& r : lists) std::printf("%g\n", bst::raise_worst(0.0, r, 3));
  // lists one after the other, as sector by sector
  double w = bst::raise_worst(0.0, lists[2], 3);
  std::printf("%g\n", bst::raise_worst(w, lists[0], 3));
  std::printf("%g\n", bst::raise_worst(5e-9, lists[0], 3));
  return 0;
}
"""


def test_worst_residual_sees_what_is_not_finite(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = str(tmp_path / "main")
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", CSRC, str(tmp_path / "main.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["3e-09", "inf", "inf", "inf", "inf", "inf", "inf", "inf", "5e-09"]


STEPS = r"""
#include <cstdio>
#include "residual.h"
int main() {
  const double inf = std::numeric_limits<double>::infinity(), nan = std::numeric_limits<double>::quiet_NaN();
  const double q[][3] = {// residual, tolerance, decay per step
                         {1e-6, 4e-12, 0.5}, {1e-6, 4e-12, 0.9}, {1e-6, 4e-12, 0.01}, {1e-6, 4e-12, 0.0},
                         {1e-6, 4e-12, 1.0}, {1e-6, 4e-12, 1.5}, {inf, 4e-12, 0.5},   {0.0, 4e-12, 0.5},
                         {1e-6, 4e-12, nan}, {1e-6, 4e-12, 1e-300}, {3e-12, 4e-12, 0.7}};
  for (auto& x : q) std::printf("%d\n", bst::plain_steps(9, x[0], x[1], x[2]));
  return 0;
}
"""


def test_length_of_a_plain_round(tmp_path):
    """From the decay that a plain step has, within 1 to 6 times the usual
    nine; nine where the decay is of no use.  (After a filtered round the
    decay comes from the Ritz values: its residuals fell by the filters'
    growth over another number of products.)"""
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    (tmp_path / "main.cpp").write_text(STEPS)
    exe = str(tmp_path / "main")
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", CSRC, str(tmp_path / "main.cpp"), "-o", exe], check=True)
    out = [int(x) for x in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()]
    # log(2e-12 / 1e-6) / log(0.5) = 18.9, / log(0.9) = 124.6, / log(0.01) = 2.9
    assert out == [19, 54, 9, 9, 9, 9, 9, 9, 9, 9, 9]
