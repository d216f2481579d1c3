"""Product times of a filter from one short launch in eight: the work of short launches shrinks along
a filter as columns reach their degrees, and the estimate must not lean to the long ones.  Compiled
for the host.  Bound for a linear fall: the fourth of eight is half a step above their mean; of the
last m < 8 launches, the fourth is at most 1.5 steps from their mean, and where there are fewer than
four the sample before is at most 6."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2603_10514_gb300", "csrc")

DRIVER = r"""
#include "launch_sample.h"
extern "C" double estimate(int n, const double* t, const int* few, int* timed) {
  chase::LaunchSample s;
  std::vector<double> known;
  for (int i = 0; i < n; ++i)
    if (s.next(few[i] != 0)) known.push_back(t[i]);
  *timed = (int)known.size();
  const double a = s.total(known.data(), known.size());
  s.clear();
  return s.total(nullptr, 0) == 0.0 ? a : -1.0;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("sample")
    (d / "s.cpp").write_text(DRIVER)
    so = str(d / "s.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "s.cpp"), "-o", so], check=True)
    L = ctypes.CDLL(so)
    L.estimate.restype = ctypes.c_double
    return L


def estimate(lib, t, few):
    timed = ctypes.c_int(0)
    t, few = np.ascontiguousarray(t, float), np.ascontiguousarray(few, np.int32)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    return lib.estimate(len(t), p(t), p(few), ctypes.byref(timed)), timed.value


@pytest.mark.parametrize("n", [4, 8, 16, 18, 20, 24, 36, 40])
def test_falling_work(lib, n):
    t = np.linspace(30.0, 6.0, n)
    got, timed = estimate(lib, t, np.ones(n))
    assert timed <= n // 8 + 2
    m, step = n % 8, t[0] - t[1]
    assert abs(got - t.sum()) <= step * (0.5 * (n - m) + (1.5 if m >= 4 else 6.0) * m) * (1 + 1e-12)


def test_constant_work_and_few_launches(lib):
    for n in (1, 2, 3, 4, 9):
        got, _ = estimate(lib, np.full(n, 7.0), np.ones(n))
        assert abs(got - 7.0 * n) < 1e-9
    assert estimate(lib, np.zeros(0), np.zeros(0)) == (0.0, 0)


def test_long_launches_are_all_timed(lib):
    t = np.r_[np.full(5, 200.0), np.full(10, 9.0)]
    got, timed = estimate(lib, t, np.r_[np.zeros(5), np.ones(10)])
    assert abs(got - t.sum()) < 1e-9 and timed == 5 + 2
