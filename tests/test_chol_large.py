"""CholeskyQR2 of blocks whose columns of the inverse factor take 46 to 48 KB of shared memory, where
a kernel has to ask for more than the 48 KB that it may use without asking (its own variables count),
and the smallest sizes that have to."""
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


@pytest.mark.parametrize("complex_,l", [(True, 2944), (True, 2945), (True, 3072), (True, 3073), (False, 5889),
                                        (False, 6145)])
def test_inverse_of_long_columns(cl, complex_, l):
    n = l + 200
    g = torch.Generator(device="cuda")
    g.manual_seed(l)
    X = cl.colmajor(torch.randn(n, l, generator=g, device="cuda", dtype=torch.complex128 if complex_ else torch.float64))
    h = cl.Handle(0)
    try:
        rc, v, info = cl.chase_qr(h, X, 1.0, qr_force=2, prec=cl.CHASE_FP64_EMU)
    finally:
        h.close()
    assert rc == 0 and v == 2 and info == 0
    eye = torch.eye(l, device="cuda", dtype=X.dtype)
    # n roundings per inner product of unit vectors
    assert float((X.mH @ X - eye).abs().max()) <= 4 * n * 2.0 ** -53
