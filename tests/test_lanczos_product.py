"""The Lanczos product in fixed point: one step from a given vector has alpha = q^H A q and
beta = |A q - alpha q|, compared with sums in extended precision, for counts of rows of one and
several chunks, graded and badly scaled columns, extreme scales and NaN.  Bound: every entry of A
and q is rounded to (at most) 2^-54 of its column's largest, sums in FP64 add n roundings."""
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


def one_step(cl, A, v):
    h = cl.Handle(0)
    try:
        return cl.chase_lanczos_bounds(h, cl.colmajor(torch.from_numpy(A).cuda()),
                                       cl.colmajor(torch.from_numpy(v[:, None].copy()).cuda()), 1, 1)
    finally:
        h.close()


@pytest.mark.parametrize("complex_", [False, True])
@pytest.mark.parametrize("scale", [1.0, 1e-300, 1e140])
@pytest.mark.parametrize("n,graded", [(2, False), (3, False), (31, True), (33, False), (500, True), (1025, False),
                                      (8193, False)])
def test_one_step(cl, n, graded, scale, complex_):
    if n > 8192 and (complex_ or scale != 1.0):
        pytest.skip("one large case is enough")
    rng = np.random.default_rng(n)
    A = rng.standard_normal((n, n)) + (1j * rng.standard_normal((n, n)) if complex_ else 0.0)
    if graded:
        d = 10.0 ** -rng.uniform(0, 8, n)
        A = d[:, None] * A * d
    A = scale * (A + A.conj().T)
    v = rng.standard_normal(n) + (1j * rng.standard_normal(n) if complex_ else 0.0)
    v[0] *= 1e3
    v /= np.linalg.norm(v)
    wide = np.clongdouble if complex_ else np.longdouble
    Aw, q = A.astype(wide), v.astype(wide)
    q /= np.sqrt((np.abs(q) ** 2).sum())
    y = Aw @ q
    alpha = (q.conj() @ y).real
    beta = np.sqrt((np.abs(y - alpha * q) ** 2).sum())
    u = np.longdouble(2.0) ** -53
    f = 4 if complex_ else 2
    aA, aq = np.abs(Aw), np.abs(q)
    err = f * u * (aA.max(0) * aq.sum() + aq.max() * aA.sum(0)) + 8 * u * np.abs(y)
    ea = (aq * err).sum() + f * (n + 16) * u * (aq * np.abs(y)).sum()
    eb = np.sqrt((err ** 2).sum()) + 2 * ea + f * (n + 16) * u * np.sqrt((np.abs(y) ** 2).sum())
    l1, _, bsup = one_step(cl, A, v)
    assert abs(l1 - alpha) <= ea
    assert abs(bsup - (alpha + beta)) <= ea + eb


def test_nonfinite_entry_shows(cl):
    A = np.eye(64)
    A[3, 3] = np.nan
    try:
        out = one_step(cl, A, np.full(64, 0.125))
    except cl.ChaseError:
        return
    assert not np.all(np.isfinite(out))
