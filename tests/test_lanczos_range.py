"""Lanczos runs that end early.  A residual that vanishes beside a matrix near the lower end of FP64
would be a subnormal vector: its norm has no reciprocal in range and its inner products no digits.
c I has every Ritz value c; bound: the n roundings of the inner products.  From a start vector in
an invariant subspace a run has to see the rest of the spectrum too."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cl():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_10514_gb300 as P
    P.build()
    return P


@pytest.mark.parametrize("complex_", [False, True])
@pytest.mark.parametrize("c", [1.0, 1e-290, 1e-296, 1e-300, 1e300])
def test_multiple_of_the_identity(cl, complex_, c):
    n, steps = 64, 4
    rng = np.random.default_rng(3)
    V = rng.standard_normal((n, 2)) + (1j * rng.standard_normal((n, 2)) if complex_ else 0.0)
    A = c * np.eye(n, dtype=V.dtype)
    h = cl.Handle(0)
    try:
        got = np.array(cl.chase_lanczos_bounds(h, cl.colmajor(torch.from_numpy(A).cuda()),
                                               cl.colmajor(torch.from_numpy(V).cuda()), steps, 1))
    finally:
        h.close()
    assert np.all(np.abs(got - c) <= 8 * n * 2.0 ** -53 * c)


@pytest.mark.parametrize("complex_", [False, True])
@pytest.mark.parametrize("rotated", [False, True])
def test_start_in_an_invariant_subspace(cl, complex_, rotated):
    """One run from the eigenvector of the eigenvalue 2 (exactly, or to rounding) of a matrix with
    spectrum [2, 5], as many steps as there are: the Ritz values are eigenvalues (n steps on n = 24;
    100 n roundings), beta ends small, and the bounds are those of the whole spectrum."""
    n = 24
    rng = np.random.default_rng(9)
    lam = np.linspace(2.0, 5.0, n)
    Q = np.eye(n)
    if rotated:
        Q = np.linalg.qr(rng.standard_normal((n, n)) + (1j * rng.standard_normal((n, n)) if complex_ else 0.0))[0]
    A = (Q * lam) @ Q.conj().T
    A = (0.5 * (A + A.conj().T)).astype(complex if complex_ else float)
    v = Q[:, :1].astype(A.dtype)
    h = cl.Handle(0)
    try:
        got = cl.chase_lanczos_bounds(h, cl.colmajor(torch.from_numpy(A).cuda()),
                                      cl.colmajor(torch.from_numpy(v.copy()).cuda()), n - 1, n // 2)
    finally:
        h.close()
    assert abs(got[0] - 2.0) <= 1e-2 and got[0] >= 2.0 - 100 * n * 2.0 ** -53
    assert got[2] >= 5.0 - 100 * n * 2.0 ** -53
    assert got[2] <= 5.0 + 3.0


@pytest.mark.parametrize("complex_", [False, True])
@pytest.mark.parametrize("c", [1.0, -3.0, 1e-18])
@pytest.mark.parametrize("prec", ["CHASE_FP64", "CHASE_FP64_EMU"])
def test_solve_of_a_multiple_of_the_identity(cl, prec, c, complex_):
    """No bounds given, and none to be found but c itself."""
    n, nev, nex = 100, 6, 3
    rng = np.random.default_rng(4)
    V = rng.standard_normal((n, nev + nex)) + (1j * rng.standard_normal((n, nev + nex)) if complex_ else 0.0)
    Vd = cl.colmajor(torch.from_numpy(V).cuda())
    h = cl.Handle(0)
    try:
        cfg = cl.config_default(prec=getattr(cl, prec), opt_degree=1, tol=1e-10 * abs(c))
        rc, ev, _, _, _ = cl.chase_solve(h, cl.colmajor(torch.from_numpy(c * np.eye(n, dtype=V.dtype)).cuda()), Vd,
                                         nev, nex, None, cfg)
    finally:
        h.close()
    assert rc == 0
    np.testing.assert_allclose(ev, c, rtol=1e-12)
    Y = Vd[:, :nev]
    eye = torch.eye(nev, device="cuda", dtype=Y.dtype)
    assert float((Y.mH @ Y - eye).abs().max()) <= 1e-12


@pytest.mark.parametrize("n", [3, 4, 5, 6, 7, 8, 9, 10, 12, 16])
@pytest.mark.parametrize("c", [1.0, -2.0])
def test_solve_whose_bounds_coincide(cl, n, c):
    """One run of few steps from a unit vector: every Ritz value may round to c itself, which leaves the
    filter no interval."""
    V = np.eye(n)[:, :1]
    Vd = cl.colmajor(torch.from_numpy(V.copy()).cuda())
    h = cl.Handle(0)
    try:
        cfg = cl.config_default(prec=cl.CHASE_FP64, opt_degree=1, tol=1e-10)
        rc, ev, _, _, _ = cl.chase_solve(h, cl.colmajor(torch.from_numpy(c * np.eye(n)).cuda()), Vd, 1, 0, None, cfg)
    finally:
        h.close()
    assert rc == 0 and abs(ev[0] - c) <= 1e-12
