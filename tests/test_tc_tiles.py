"""BF16x3 filter products at row and column counts where the tile rule changes its answer (one
256-row block to more than a wave of CTA pairs, one column to several tiles): one step against
FP64 with the error of three BF16 products, 2^-14 of |A| |V| per entry (each operand's split
leaves 2^-16, FP32 sums the rest), plus the FP64 recurrence terms."""
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
@pytest.mark.parametrize("n,ncols", [(1, 1), (33, 2), (64, 16), (129, 47), (257, 49), (1000, 97), (2050, 257)])
def test_one_bf16x3_step(cl, complex_, n, ncols):
    ncols = min(ncols, n)
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    dt = torch.complex128 if complex_ else torch.float64
    A = torch.randn(n, n, generator=g, device="cuda", dtype=dt)
    A = A + A.mH
    V = cl.colmajor(torch.randn(n, ncols, generator=g, device="cuda", dtype=dt))
    c, e, l1 = 20.0, 21.0, -5.0
    h = cl.Handle(0)
    try:
        got = cl.chase_filter(h, cl.colmajor(A), V, [1] * ncols, c, e, l1, prec=cl.CHASE_BF16X3)
    finally:
        h.close()
    s = 1.0 / (l1 - c)
    ref = s * (A @ V - c * V)
    bound = abs(s) * (2.0 ** -14 * (A.abs() @ V.abs()) + c * V.abs() * 2.0 ** -50)
    assert float(((got - ref).abs() / bound).max()) <= 1.0
