"""Slicing of blocks whose columns are cut over several thread blocks, in single and grouped
(complex) form: one emulated filter step against FP64 at orders around multiples of 1024, with a
zero column and columns of very different size.  Bound per entry: the integers' rounding,
n 2^-55 times the row's and the column's largest magnitudes (complex: twice), plus the FP64
reference's own 2 n + 16 roundings of |A| |V|."""
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
@pytest.mark.parametrize("n,ncols", [(5, 3), (1000, 30), (1985, 9), (2048, 5), (2049, 5), (3073, 2), (4100, 700)])
def test_step_with_split_columns(cl, n, ncols, complex_):
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    dt = torch.complex128 if complex_ else torch.float64
    A = torch.randn(n, n, generator=g, device="cuda", dtype=dt)
    A = cl.colmajor(A + A.mH)
    V = torch.randn(n, ncols, generator=g, device="cuda", dtype=dt)
    V[:, 0] *= 1e-30
    V[:, 1] = 0.0
    V[-1, ncols - 1] = 1e6  # the largest entry is the last
    V = cl.colmajor(V)
    c, e, l1 = 20.0, 21.0, -5.0
    h = cl.Handle(0)
    try:
        got = cl.chase_filter(h, A, V, [1] * ncols, c, e, l1, prec=cl.CHASE_FP64_EMU)
    finally:
        h.close()
    s = 1.0 / (l1 - c)
    ref = s * (A @ V - c * V)
    f = 2 if complex_ else 1
    amax, vmax = A.abs().amax(1, keepdim=True), V.abs().amax(0, keepdim=True)
    bound = abs(s) * (f * n * 2.0 ** -55 * amax * vmax
                      + (A.abs() @ V.abs() + c * V.abs()) * (2 * n + 16) * 2.0 ** -53 * f)
    assert float(((got - ref).abs() - bound).max()) <= 0.0
