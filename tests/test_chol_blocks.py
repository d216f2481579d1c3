"""The blocked Cholesky factor and inverse of CholeskyQR at the edges of its 32-row blocks: the
failing pivot is reported where it is (a zero column gives an exactly zero pivot) with X
unchanged, and shifted CholeskyQR2 of an ill-conditioned block is orthonormal with X = Q R."""
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


def block(cl, n, l, complex_, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    dt = torch.complex128 if complex_ else torch.float64
    return cl.colmajor(torch.randn(n, l, generator=g, device="cuda", dtype=dt))


@pytest.mark.parametrize("emulated", [False, True])
@pytest.mark.parametrize("complex_", [False, True])
@pytest.mark.parametrize("l,zero", [(1, 0), (20, 7), (32, 31), (33, 32), (70, 50), (70, 69), (200, 129)])
def test_failing_pivot_is_reported(cl, complex_, emulated, l, zero):
    X = block(cl, 300, l, complex_, l)
    X[:, zero] = 0.0
    X0 = X.clone()
    h = cl.Handle(0)
    try:
        rc, v, info = cl.chase_qr(h, X, 1.0, qr_force=1, prec=cl.CHASE_FP64_EMU if emulated else cl.CHASE_FP64)
    finally:
        h.close()
    assert rc == cl.CHASE_CHOL_FAILED and info == zero + 1
    assert torch.equal(X, X0)


@pytest.mark.parametrize("complex_", [False, True])
@pytest.mark.parametrize("l", [31, 32, 33, 64, 65, 129, 300])
def test_shifted_qr_at_block_edges(cl, complex_, l):
    n = 700
    U = torch.linalg.qr(block(cl, n, l, complex_, 1))[0]
    M = torch.linalg.qr(block(cl, l, l, complex_, 2))[0]
    X = cl.colmajor((U * torch.logspace(0.0, -9.0, l, device="cuda", dtype=torch.float64)) @ M)
    X0 = X.clone()
    h = cl.Handle(0)
    try:
        rc, v, info = cl.chase_qr(h, X, 1.0, qr_force=3, prec=cl.CHASE_FP64_EMU)
    finally:
        h.close()
    assert rc == 0 and v == 3
    eye = torch.eye(l, device="cuda", dtype=X.dtype)
    assert float(torch.linalg.norm(X.mH @ X - eye)) <= 1e-12
    R = X.mH @ X0
    assert float(torch.linalg.norm(X @ R - X0)) <= 1e-12 * float(torch.linalg.norm(X0))
    assert float(torch.linalg.norm(torch.tril(R, -1))) <= 1e-10 * float(torch.linalg.norm(X0))
