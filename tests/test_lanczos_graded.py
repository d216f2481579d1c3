"""Lanczos products of columns and vectors that are large at different places, where entries rounded
to their column's (vector's) largest would lose what the sum consists of: one step against sums in
extended precision, within the bound of FP64 sums of the terms themselves, u (n + 16) |A| |q| per
entry.  Beside them the matrices that the fixed-point sums are for, dense, diagonally dominant,
diagonal and sparse ones."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cl():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_10514_gb300 as P
    P.build()
    return P


def problem(kind, n, complex_, rng):
    g = lambda *s: rng.standard_normal(s) + (1j * rng.standard_normal(s) if complex_ else 0.0)
    A, v = g(n, n), g(n)
    A = A + A.conj().T
    if kind == "graded":  # d_i b_ij d_j meets v_j / d_j: every term counts the same
        d = 10.0 ** -rng.uniform(0, 7, n)
        A, v = d[:, None] * A * d, v / d
    if kind == "dominant":
        A = A + np.diag(1e6 * rng.standard_normal(n))
    if kind == "diagonal":
        A = np.diag(rng.standard_normal(n)).astype(A.dtype)
    if kind == "sparse":
        A = np.where(rng.uniform(size=(n, n)) < 3.0 / n, A, 0.0)
        A = A + A.conj().T
    if kind == "steep":  # a vector over twelve decades
        v = v * 10.0 ** -rng.uniform(0, 12, n)
    return A, v


@pytest.mark.parametrize("complex_", [False, True])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -800])
@pytest.mark.parametrize("n", [2, 33, 300, 1025])
@pytest.mark.parametrize("kind", ["dense", "graded", "dominant", "diagonal", "sparse", "steep"])
def test_one_step(cl, kind, n, scale, complex_):
    rng = np.random.default_rng(n)
    A, v = problem(kind, n, complex_, rng)
    wide = np.clongdouble if complex_ else np.longdouble
    Aw, q = A.astype(wide), v.astype(wide)
    q /= np.sqrt((np.abs(q) ** 2).sum())
    y = Aw @ q
    alpha = (q.conj() @ y).real
    beta = np.sqrt((np.abs(y - alpha * q) ** 2).sum())
    u = np.longdouble(2.0) ** -53
    f = 4 if complex_ else 2
    err = f * (n + 16) * u * (np.abs(Aw) @ np.abs(q))
    ea = f * (np.abs(q) * err).sum()
    eb = np.sqrt((err ** 2).sum()) + 2 * ea + f * (n + 16) * u * np.sqrt((np.abs(y) ** 2).sum())
    h = cl.Handle(0)
    try:
        l1, _, bsup = cl.chase_lanczos_bounds(h, cl.colmajor(torch.from_numpy(scale * A).cuda()),
                                              cl.colmajor(torch.from_numpy(v[:, None].copy()).cuda()), 1, 1)
    finally:
        h.close()
    assert abs(l1 / scale - alpha) <= ea
    assert abs(bsup / scale - (alpha + beta)) <= ea + eb


@pytest.mark.parametrize("complex_", [False, True])
@pytest.mark.parametrize("kind", ["dominant", "diagonal", "sparse", "graded"])
def test_bounds_of_several_steps(cl, kind, complex_):
    """Columns that a first step sums in FP64 stay so in the next, and for further groups of runs;
    against the oracle, tolerance as for dense matrices."""
    n, nruns, steps, ell = 300, 6, 20, 30
    rng = np.random.default_rng(5)
    A, _ = problem(kind, n, complex_, rng)
    A /= np.linalg.norm(A, 2)
    V = rng.standard_normal((n, nruns)) + (1j * rng.standard_normal((n, nruns)) if complex_ else 0.0)
    ref, _ = oracle.lanczos_bounds(A, V, steps, ell)
    h = cl.Handle(0)
    try:
        got = cl.chase_lanczos_bounds(h, cl.colmajor(torch.from_numpy(A).cuda()),
                                      cl.colmajor(torch.from_numpy(V).cuda()), steps, ell)
    finally:
        h.close()
    np.testing.assert_allclose(got, ref, rtol=0, atol=2e-9)
