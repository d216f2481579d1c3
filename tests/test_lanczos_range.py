"""Lanczos runs whose residual vanishes beside a matrix near the lower end of FP64, where it would be
a subnormal vector: its norm has no reciprocal in range and its inner products no digits.  c I has
every Ritz value c; bound: the n roundings of the inner products."""
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
