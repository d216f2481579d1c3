"""The steps of a divide-and-conquer merge (stedc.cuh) that the groups of one warp run together:
whatever item a group holds (a root, a deflated value), it takes part in the same collective
calls, at the same places of the code.  Compiled for the host with groups of one lane that record
where they meet."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2603_10514_gb300", "csrc")

DRIVER = r"""
#include <vector>
#include "stedc.cuh"
using namespace chase::dc;
struct One { int tid = 0, size = 1; void sync() const {} double max(double v) const { return v; } };
static std::vector<int> met;  // lines of the collective calls of one item
struct Lane {
  int lane = 0, width = 1;
  double sum(double v, int at = __builtin_LINE()) const { met.push_back(at); return v; }
  double prod(double v, int at = __builtin_LINE()) const { met.push_back(at); return v; }
  int count(int v, int at = __builtin_LINE()) const { met.push_back(at); return v; }
  bool any(bool v) const { return v; }
};
static bool same(std::vector<int>& first) {
  const bool ok = first.empty() || first == met;
  first = met;
  met.clear();
  return ok;
}
// D: eigenvalues of two halves (n1 and m - n1, ascending each), z: their coupling rows.
// Returns K, or -1 - step where two items of a step met at different places.
extern "C" int steps(int m, int n1, double rho, const double* D, const double* z, int* dest) {
  std::vector<double> f(9 * m), U((size_t)m * m);
  std::vector<int> v(9 * m);
  std::vector<unsigned char> b(3 * m);
  int cnt[4];
  Merge M;
  M.m = m; M.n1 = n1; M.rho = rho; M.sign = 1; M.D = D;
  double** fs[] = {&M.ds, &M.zs, &M.dl, &M.w, &M.mu, &M.zh, &M.lam, &M.rc, &M.rs};
  int** vs[] = {&M.perm, &M.idx, &M.defl, &M.pos, &M.gat, &M.org, &M.rp, &M.rq, &M.dest};
  for (int i = 0; i < 9; ++i) { *fs[i] = &f[i * m]; *vs[i] = &v[i * m]; }
  M.small = &b[0]; M.close = &b[m]; M.type = &b[2 * m]; M.cnt = cnt;
  setup(One(), M, z, z + n1, 1);
  const int K = cnt[0];
  for (int k = 0; k < K; ++k) root(Lane(), K, k, true, M.dl, M.w, M.rho, M.mu + k, M.org + k, M.lam + k);
  met.clear();
  std::vector<int> first;
  for (int k = 0; k < K; ++k) { zhat(Lane(), K, k, true, M.dl, M.w, M.mu, M.org, M.zh); if (!same(first)) return -1; }
  first.clear();
  for (int k = 0; k < K; ++k) {
    ucol(Lane(), K, k, true, M.dl, M.zh, M.mu, M.org, M.pos, U.data(), m);
    if (!same(first)) return -2;
  }
  first.clear();
  for (int t = 0; t < m; ++t) { place(Lane(), M, K, t, true); if (!same(first)) return -3; }
  for (int t = 0; t < m; ++t) dest[t] = M.dest[t];
  return K;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("dcsteps")
    (d / "steps.cpp").write_text(DRIVER)
    so = str(d / "steps.so")
    subprocess.run(["g++", "-O1", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, str(d / "steps.cpp"), "-o", so],
                   check=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("m,deflated", [(2, 0), (5, 2), (16, 3), (16, 16), (33, 10)])
def test_items_of_a_warp_meet_at_the_same_calls(lib, m, deflated):
    r = np.random.default_rng(m)
    n1 = m // 2
    D = np.concatenate([np.sort(r.standard_normal(n1)), np.sort(r.standard_normal(m - n1))])
    z = r.uniform(0.5, 1.0, m)
    z[r.permutation(m)[:deflated]] = 0.0
    dest = np.zeros(m, np.int32)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    K = lib.steps(m, n1, ctypes.c_double(0.7), p(D), p(z), p(dest))
    assert K == m - deflated, "items of step %d met at different calls" % -K
    assert sorted(dest) == list(range(m))
