"""The direct eigensolver of the Rayleigh-Ritz step (reduction to tridiagonal form, divide and
conquer, back-transformation).

On the CPU: the merge steps of stedc.cuh, compiled for the host, drive a whole divide and conquer
from single rows up on tridiagonals that deflate in every way.  On the GPU: solves whose search
block is the whole space, so that one Rayleigh-Ritz step must give the complete eigensystem.

Bounds: backward stability, a modest multiple of n 2^-53 times the norm; 4 n for the residual
and the orthogonality of divide and conquer (measured growth is well below n).
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2603_10514_gb300", "csrc")
U = 2.0 ** -53

DRIVER = r"""
#include <algorithm>
#include <cstring>
#include <vector>
#include "stedc.cuh"
using namespace chase::dc;
struct One { int tid = 0, size = 1; void sync() const {} double max(double v) const { return v; } };
struct Lane { int lane = 0, width = 1; double sum(double v) const { return v; }
              double prod(double v) const { return v; } int count(int v) const { return v; }
              bool any(bool v) const { return v; } };
extern "C" void dc_solve(int n, const double* d, const double* e, double* D, double* Q) {
  std::vector<double> U((size_t)n * n), out((size_t)n * n);
  for (int i = 0; i < n; ++i) {
    D[i] = d[i] - (i ? std::fabs(e[i - 1]) : 0) - (i + 1 < n ? std::fabs(e[i]) : 0);
    for (int j = 0; j < n; ++j) Q[i + (size_t)j * n] = i == j;
  }
  int L = 0;
  while ((1 << L) < n) ++L;
  for (int h = L - 1; h >= 0; --h)
    for (long q = 0; q < (1 << h); ++q) {
      const int s = (2 * q * n) >> (h + 1), mid = ((2 * q + 1) * n) >> (h + 1), m = (((2 * q + 2) * n) >> (h + 1)) - s;
      if (mid == s || mid == s + m) continue;
      std::vector<double> f(9 * m), Dm(m);
      std::vector<int> v(9 * m);
      std::vector<unsigned char> b(3 * m);
      int cnt[4];
      Merge M;
      M.m = m; M.n1 = mid - s; M.rho = 2 * std::fabs(e[mid - 1]); M.sign = e[mid - 1] < 0 ? -1 : 1; M.D = D + s;
      double** fs[] = {&M.ds, &M.zs, &M.dl, &M.w, &M.mu, &M.zh, &M.lam, &M.rc, &M.rs};
      int** vs[] = {&M.perm, &M.idx, &M.defl, &M.pos, &M.gat, &M.org, &M.rp, &M.rq, &M.dest};
      for (int i = 0; i < 9; ++i) { *fs[i] = &f[i * m]; *vs[i] = &v[i * m]; }
      M.small = &b[0]; M.close = &b[m]; M.type = &b[2 * m]; M.cnt = cnt;
      double* B = Q + s + (size_t)s * n;
      setup(One(), M, B + M.n1 - 1, B + M.n1 + (size_t)M.n1 * n, n);
      const int K = cnt[0];
      for (int k = 0; k < K; ++k) root(Lane(), K, k, true, M.dl, M.w, M.rho, M.mu + k, M.org + k, M.lam + k);
      for (int r = 0; r < cnt[3]; ++r)
        for (int i = 0; i < m; ++i) {
          double &x = B[i + (size_t)M.rp[r] * n], &y = B[i + (size_t)M.rq[r] * n], a = x;
          x = M.rc[r] * a + M.rs[r] * y;
          y = M.rc[r] * y - M.rs[r] * a;
        }
      for (int k = 0; k < K; ++k) zhat(Lane(), K, k, true, M.dl, M.w, M.mu, M.org, M.zh);
      for (int k = 0; k < K; ++k) ucol(Lane(), K, k, true, M.dl, M.zh, M.mu, M.org, M.pos, U.data(), n);
      for (int t = 0; t < m; ++t) place(Lane(), M, K, t, true);
      for (int j = 0; j < m; ++j)
        for (int i = 0; i < m; ++i) {
          double a = 0;
          if (j < K) for (int p = i < M.n1 ? 0 : cnt[1]; p < (i < M.n1 ? cnt[2] : K); ++p)
            a += B[i + (size_t)M.gat[p] * n] * U[p + (size_t)j * n];
          else a = B[i + (size_t)M.perm[M.defl[j - K]] * n];
          out[i + (size_t)M.dest[j] * m] = a;
          Dm[M.dest[j]] = j < K ? M.lam[j] : M.ds[M.defl[j - K]];
        }
      for (int j = 0; j < m; ++j) { D[s + j] = Dm[j]; std::memcpy(B + (size_t)j * n, &out[(size_t)j * m], 8 * m); }
    }
}
"""


@pytest.fixture(scope="module")
def dc(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("dc")
    (d / "dc.cpp").write_text(DRIVER)
    so = str(d / "dc.so")
    subprocess.run(["g++", "-O1", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, str(d / "dc.cpp"), "-o", so],
                   check=True)
    return ctypes.CDLL(so)


def tridiagonals(n):
    r = np.random.default_rng(n)
    i, e1 = np.arange(n, dtype=float), np.ones(max(n - 1, 0))
    yield "random", r.standard_normal(n), r.standard_normal(n - 1)
    yield "laplace", 2.0 + 0 * i, -e1
    yield "wilkinson", np.abs(i - (n - 1) / 2), e1
    yield "constant", 3.0 + 0 * i, 0 * e1
    yield "zero", 0 * i, 0 * e1
    yield "near diagonal", -2 + i / n, 1e-9 * r.standard_normal(n - 1)
    yield "cluster", 1 + 1e-14 * r.standard_normal(n), 1e-8 * r.standard_normal(n - 1)
    yield "split", r.standard_normal(n), np.where(np.arange(n - 1) % 7 == 3, 0.0, r.standard_normal(n - 1))
    yield "graded", 10.0 ** (-12 * i / n), 0.1 * 10.0 ** (-12 * (i[:-1] + 0.5) / n)


@pytest.mark.parametrize("n", [1, 2, 3, 5, 17, 32, 33, 100, 257])
def test_divide_and_conquer_steps(dc, n):
    for name, d, e in tridiagonals(n):
        D, Q = np.empty(n), np.empty((n, n), order="F")
        p = lambda a: np.ascontiguousarray(a).ctypes.data_as(ctypes.c_void_p)
        d, e = np.ascontiguousarray(d), np.ascontiguousarray(np.concatenate([e, [0.0]]))
        dc.dc_solve(n, p(d), p(e), D.ctypes.data_as(ctypes.c_void_p), Q.ctypes.data_as(ctypes.c_void_p))
        T = np.diag(d) + np.diag(e[:n - 1], 1) + np.diag(e[:n - 1], -1)
        norm = np.abs(T).sum(axis=1).max()
        assert np.all(np.diff(D) >= 0), name
        assert np.abs(T @ Q - Q * D).max() <= 4 * n * U * norm, name
        assert np.abs(Q.T @ Q - np.eye(n)).max() <= 4 * n * U, name
        assert np.abs(D - np.linalg.eigvalsh(T)).max() <= 4 * n * U * norm, name


torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def cl():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_10514_gb300 as P
    P.build()
    return P


@pytest.mark.gpu
@pytest.mark.parametrize("complex_", [False, True])
@pytest.mark.parametrize("n", [1, 2, 3, 23, 24, 31, 32, 33, 63, 64, 65, 129, 257, 601])
@pytest.mark.parametrize("spectrum", ["uniform", "multiple", "diagonal"])
def test_whole_space_rayleigh_ritz(cl, complex_, n, spectrum):
    """nev = n, nex = 0: after one iteration (degree 1, far from the damped interval) the Ritz
    pairs are the eigenpairs: eigenvalues, residuals and orthogonality to 40 n 2^-53 (the
    products before and after the eigensolver each contribute a few n 2^-53)."""
    lam = np.sort(np.random.default_rng(n).uniform(-1.0, 1.0, n))
    if spectrum == "multiple":
        lam = np.round(lam * 3) / 3
    if spectrum == "diagonal":
        A = np.diag(lam).astype(complex if complex_ else float)
    else:
        A = W.known_spectrum_matrix(lam, 7, complex_).numpy()
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(np.asarray(x).T)).cuda().mT
    V = dev(W.start_block(n, n, 8, complex_))
    h = cl.Handle(0)
    try:
        cfg = cl.config_default(prec=cl.CHASE_FP64, opt_degree=0, deg_init=1, max_iter=1, qr_force=4)
        rc, ev, res, _, _ = cl.chase_solve(h, dev(A), V, n, 0, (float(lam[0]), float(lam[-1]) + 20.0, 1000.0), cfg)
    finally:
        h.close()
    assert rc == 0
    Y, tol = V.cpu().numpy(), 40 * max(n, 4) * U
    assert np.abs(ev - lam).max() <= tol
    assert np.abs(Y.conj().T @ Y - np.eye(n)).max() <= tol
    assert np.abs(A @ Y - Y * ev).max() <= tol
