"""The direct eigensolver at every scale of the matrix: what it leaves out is small against the
matrix it is given, not against one.

Bounds as for matrices of norm about 1, relative to the norm: 4 n 2^-53 for divide and conquer
alone (on the CPU), 40 n 2^-53 for a Rayleigh-Ritz step over the whole space (on the GPU)."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import workloads as W
from test_eigh import CSRC, DRIVER, U, cl, dc, tridiagonals  # noqa: F401  (fixtures)


def ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def solve(dc, d, e):
    n = len(d)
    D, Q = np.empty(n), np.empty((n, n), order="F")
    d, e = np.ascontiguousarray(d), np.ascontiguousarray(np.concatenate([e, [0.0]]))
    dc.dc_solve(n, ptr(d), ptr(e), ptr(D), ptr(Q))
    return D, Q


def check(name, d, e, D, Q, s):
    """Against T / s, s a power of two that brings T to norm about 1."""
    n = len(d)
    d, e, D = d / s, e / s, D / s
    T = np.diag(d) + np.diag(e, 1) + np.diag(e, -1)
    norm = np.abs(T).sum(axis=1).max()
    assert np.all(np.diff(D) >= 0), name
    assert np.abs(T @ Q - Q * D).max() <= 4 * n * U * norm, name
    assert np.abs(Q.T @ Q - np.eye(n)).max() <= 4 * n * U, name
    assert np.abs(D - np.linalg.eigvalsh(T)).max() <= 4 * n * U * norm, name


@pytest.mark.parametrize("n", [2, 3, 17, 33, 100, 257])
@pytest.mark.parametrize("k", [-300, -60, -40, -27, -10, 30, 300])
def test_divide_and_conquer_is_relative_to_the_matrix(dc, n, k):
    s = 2.0 ** k
    for name, d, e in tridiagonals(n):
        check(name, s * d, s * e, *solve(dc, s * d, s * e), s)


RANGE_DRIVER = DRIVER + r"""
extern "C" void dc_solve_any(int n, const double* d, const double* e, double* D, double* Q) {
  std::vector<double> a(d, d + n), b(e, e + n);
  double x = 0;
  for (int i = 0; i < n; ++i) x = std::max(x, std::max(std::fabs(a[i]), std::fabs(b[i])));
  const int k = scale_of(x);
  for (int i = 0; i < n; ++i) { a[i] = std::ldexp(a[i], k); b[i] = std::ldexp(b[i], k); }
  dc_solve(n, a.data(), b.data(), D, Q);
  for (int i = 0; i < n; ++i) D[i] = std::ldexp(D[i], -k);
}
"""


@pytest.fixture(scope="module")
def dc_range(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("dcrange")
    (d / "dc.cpp").write_text(RANGE_DRIVER)
    so = str(d / "dc.so")
    subprocess.run(["g++", "-O1", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, str(d / "dc.cpp"), "-o", so],
                   check=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("n", [1, 2, 17, 33, 100])
@pytest.mark.parametrize("k", [-1000, -600, 0, 600, 1000])
def test_divide_and_conquer_over_the_whole_range(dc_range, n, k):
    """Scaled to its largest entry first, as the kernels do it: squares and reciprocals of the
    entries stay in range."""
    s = 2.0 ** k
    for name, d, e in tridiagonals(n):
        D, Q = np.empty(n), np.empty((n, n), order="F")
        a, b = np.ascontiguousarray(s * d), np.ascontiguousarray(np.concatenate([s * e, [0.0]]))
        dc_range.dc_solve_any(n, ptr(a), ptr(b), ptr(D), ptr(Q))
        check(name, s * d, s * e, D, Q, s)


torch = pytest.importorskip("torch")


def scaled_rayleigh_ritz(cl, complex_, n, k, prec):
    """Eigenvalues and vectors of 2^k A by one Rayleigh-Ritz step over the whole space, and A's."""
    lam = np.sort(np.random.default_rng(n).uniform(-1.0, 1.0, n))
    A = W.known_spectrum_matrix(lam, 7, complex_).numpy()
    s = 2.0 ** k
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(np.asarray(x).T)).cuda().mT
    V = dev(W.start_block(n, n, 8, complex_))
    h = cl.Handle(0)
    try:
        cfg = cl.config_default(prec=prec, opt_degree=0, deg_init=1, max_iter=1, qr_force=4, tol=1e-10 * s)
        rc, ev, _, _, _ = cl.chase_solve(h, dev(s * A), V, n, 0, (s * lam[0], s * (lam[-1] + 20.0), s * 1000.0), cfg)
    finally:
        h.close()
    assert rc == 0
    return A, lam, ev / s, V.cpu().numpy()


@pytest.mark.gpu
@pytest.mark.parametrize("complex_", [False, True])
@pytest.mark.parametrize("n,k", [(33, -40), (129, -27), (300, -40), (129, 30)])
def test_whole_space_rayleigh_ritz_at_scale(cl, complex_, n, k):
    A, lam, ev, Y = scaled_rayleigh_ritz(cl, complex_, n, k, cl.CHASE_FP64)
    tol = 40 * n * U
    assert np.abs(ev - lam).max() <= tol
    assert np.abs(Y.conj().T @ Y - np.eye(n)).max() <= tol
    assert np.abs(A @ Y - Y * ev).max() <= tol


@pytest.mark.gpu
@pytest.mark.parametrize("complex_", [False, True])
@pytest.mark.parametrize("n,k", [(1, -600), (2, 400), (33, -600), (129, -600), (129, 400), (300, -520), (601, -600)])
def test_whole_space_rayleigh_ritz_over_the_range(cl, complex_, n, k):
    """Squares of the entries leave the range of FP64 (n = 33 on one thread block, 601 on all)."""
    A, lam, ev, Y = scaled_rayleigh_ritz(cl, complex_, n, k, cl.CHASE_FP64_EMU)
    tol = 40 * max(n, 4) * U
    assert np.abs(ev - lam).max() <= tol
    assert np.abs(Y.conj().T @ Y - np.eye(n)).max() <= tol
    assert np.abs(A @ Y - Y * ev).max() <= tol


@pytest.mark.gpu
@pytest.mark.parametrize("complex_,n", [(True, 1500), (False, 2100)])
@pytest.mark.parametrize("k", [0, -600])
def test_columns_that_stay_in_global_memory(cl, complex_, n, k):
    """Orders whose columns do not fit the shared memory of one wave of thread blocks: the matrix is
    scaled where it lies."""
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    dt = torch.complex128 if complex_ else torch.float64
    rand = lambda: torch.randn(n, n, generator=g, device="cuda", dtype=dt)
    Q = torch.linalg.qr(rand())[0]
    lam = torch.sort(torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * 2 - 1)[0]
    A = (Q * lam) @ Q.mH
    A = 0.5 * (A + A.mH)
    V = cl.colmajor(rand())
    s = 2.0 ** k
    h = cl.Handle(0)
    try:
        cfg = cl.config_default(prec=cl.CHASE_FP64_EMU, opt_degree=0, deg_init=1, max_iter=1, qr_force=4, tol=1e-10 * s)
        rc, ev, _, _, _ = cl.chase_solve(h, cl.colmajor(s * A), V, n, 0, (-s, 21.0 * s, 1000.0 * s), cfg)
    finally:
        h.close()
    assert rc == 0
    ev, tol = torch.from_numpy(np.asarray(ev)).cuda() / s, 40 * n * U
    assert float((ev - lam).abs().max()) <= tol
    assert float((V.mH @ V - torch.eye(n, device="cuda", dtype=dt)).abs().max()) <= tol
    assert float((A @ V - V * ev).abs().max()) <= tol


def lanczos(cl, A, V, steps, ell):
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(np.asarray(x).T)).cuda().mT
    h = cl.Handle(0)
    try:
        return np.array(cl.chase_lanczos_bounds(h, dev(A), dev(V), steps, ell))
    finally:
        h.close()


@pytest.mark.gpu
@pytest.mark.parametrize("complex_", [False, True])
@pytest.mark.parametrize("k", [-60, -100, 100, -900, 900])
def test_lanczos_bounds_scale_with_the_matrix(cl, complex_, k):
    n, steps, ell = 600, 25, 60
    lam = W.spectrum_uniform(n, -1.0, 1.0, 5)
    A = W.known_spectrum_matrix(lam, 5, complex_).numpy()
    V = W.start_block(n, 4, 6, complex_)
    one, got = lanczos(cl, A, V, steps, ell), lanczos(cl, 2.0 ** k * A, V, steps, ell) / 2.0 ** k
    # a power of two changes no rounding; only which couplings are left out may depend on it
    assert np.abs(got - one).max() <= 100 * steps * U
    assert got[2] >= lam[-1]


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["CHASE_FP64_EMU", "CHASE_FP64"])
@pytest.mark.parametrize("complex_,k", [(False, 0), (False, -60), (True, -60), (True, 60)])
def test_solve_that_is_given_no_bounds(cl, complex_, k, prec):
    """A small or large matrix (2^-60: energies in joules) with a tolerance to match and its bounds
    from Lanczos runs, as at scale 1."""
    n, nev, nex = 400, 20, 8
    lam = W.spectrum_uniform(n, -1.0, 1.0, 5)
    A = W.known_spectrum_matrix(lam, 5, complex_).numpy()
    s = 2.0 ** k
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(np.asarray(x).T)).cuda().mT
    V = dev(W.start_block(n, nev + nex, 6, complex_))
    h = cl.Handle(0)
    try:
        cfg = cl.config_default(prec=getattr(cl, prec), opt_degree=1, tol=1e-10 * s)
        rc, ev, res, st, _ = cl.chase_solve(h, dev(s * A), V, nev, nex, None, cfg)
    finally:
        h.close()
    assert rc == 0 and st["iterations"] < 15
    assert np.abs(np.asarray(ev) / s - lam[:nev]).max() <= 1e-10
    Y = V.cpu().numpy()[:, :nev]
    assert np.linalg.norm(A @ Y - Y * (np.asarray(ev) / s), axis=0).max() <= 2e-10
