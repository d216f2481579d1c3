"""Complex emulated products in split residue rings (moduli with s^2 = -1 mod p).

On the CPU: the moduli read from the kernel source, the residues of the integer operands by the
kernel's 32-bit formula, the packed FP32 fold of the exact chunks, and the reconstruction, against
exact integers.  On the GPU: one filter step at the sizes where the product's padding, chunks and
tiles end, and one K beyond the 15-moduli range, against FP64 within the scheme's error bound.
"""
import os
import re

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_2603_10514_gb300", "csrc", "gemm_oz.cu")


def ring_moduli():
    m = re.search(r"constexpr int tr\[kRingModuli\]\s*=\s*\{([^}]*)\}", open(SRC).read())
    assert m, "ring moduli table not found"
    return [int(x) for x in m.group(1).replace("\n", " ").split(",") if x.strip()]


def root(p):
    return next(s for s in range(1, p) if (s * s + 1) % p == 0)


def test_moduli_split_and_cover_the_range():
    ps = ring_moduli()
    assert len(ps) == 16
    P = 1
    for i, p in enumerate(ps):
        root(p)
        assert 256 * (p // 2) ** 2 + p < 1 << 24  # a chunk and the folded rest are exact in FP32
        P *= p
        if i == 14:
            assert P > 2 * 2 * (1 << 15) * (1 << 114)
    assert P > 2 * 2 * (1 << 17) * (1 << 114)
    assert all(np.gcd(a, b) == 1 for i, a in enumerate(ps) for b in ps[i + 1:])


def slices(xr, xi, p):
    """write_ring4 in wrapping 32-bit arithmetic."""
    s, half = root(p), p // 2
    u32 = lambda v: np.asarray(v, dtype=np.uint32)
    k19, k38, off = u32((1 << 19) % p), u32((1 << 38) % p), u32(p - (1 << 58) % p)

    def t(x):
        X = (x + (1 << 58)).astype(np.uint64)
        return (u32(X >> np.uint64(38)) * k38 + u32((X >> np.uint64(19)) & np.uint64(0x7FFFF)) * k19
                + u32(X & np.uint64(0x7FFFF)) + off)
    tr, ti = t(xr), t(xi) % u32(p)
    u = ((tr + u32(s) * ti + u32(half)) % u32(p)).astype(np.int64) - half
    w = ((tr + u32(p - s) * ti + u32(half)) % u32(p)).astype(np.int64) - half
    return u, w


def test_operand_residues_and_reconstruction_are_exact():
    rng = np.random.default_rng(3)
    edge = [0, 1, -1, 1 << 57, -(1 << 57), (1 << 57) - 1, (1 << 38) - 1, 1 << 38, -(1 << 38), (1 << 19) - 1]
    K = 300
    x = [np.concatenate([rng.integers(-(1 << 57), (1 << 57) + 1, K - len(edge)), rng.permutation(edge)])
         for _ in range(4)]
    ar, ai, vr, vi = x
    big = lambda v: [int(z) for z in v]
    re_ = sum(a * c - b * d for a, b, c, d in zip(*map(big, x)))
    im_ = sum(a * d + b * c for a, b, c, d in zip(*map(big, x)))
    for count in (15, 16):
        ps = ring_moduli()[:count]
        P = 1
        for p in ps:
            P *= p
        R = I = 0
        for p in ps:
            s = root(p)
            ua, wa = slices(ar, ai, p)
            uv, wv = slices(vr, vi, p)
            for r, sign in ((ua, 1), (wa, -1)):
                assert np.abs(r).max() <= p // 2 and all((int(q) - int(a) - sign * s * int(b)) % p == 0
                                                         for q, a, b in zip(r, ar, ai))
            U, W = int((ua * uv).sum()) % p, int((wa * wv).sum()) % p
            M = P // p
            inv = pow(M, -1, p)
            R += (U + W) * (M * (inv * pow(2, -1, p) % p))
            I += (U + p - W) * (M * (inv * pow(2 * s, -1, p) % p))
        sym = lambda v: (v % P) - P if (v % P) > P // 2 else v % P
        assert sym(R) == re_ and sym(I) == im_


def test_packed_fold_keeps_the_class_and_the_bound():
    """fold2 in IEEE float32 over chunk sums up to the largest possible, random and extreme."""
    rng = np.random.default_rng(5)
    f = np.float32
    magic = f(12582912.0)
    for p in ring_moduli():
        top = 256 * (p // 2) ** 2
        ip = f(1) / f(p)
        acc, exact = np.zeros(4096, dtype=f), np.zeros(4096, dtype=np.int64)
        for step in range(40):
            v = rng.integers(-top, top + 1, 4096)
            v[:512] = top if step % 3 else -top
            s = acc + v.astype(f)
            # fma(s, ip, magic): the product is exact in float64, so this rounds once
            q = (s.astype(np.float64) * float(ip) + float(magic)).astype(f) - magic
            acc = (s.astype(np.float64) - q.astype(np.float64) * p).astype(f)
            exact += v
            assert np.abs(s).max() < 1 << 24 and np.abs(acc).max() <= 0.51 * p
            assert not np.any((acc.astype(np.int64) - exact) % p)


torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def cl():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_10514_gb300 as P
    P.build()
    return P


def step_error(cl, n, ncols, seed):
    """max |got - ref| / bound of one filter step on the GPU; the bound as for every emulated
    product: K 2^-53 max|A_m.| max|V_.c| and 2^-52 for the FP64 recurrence terms."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    A = torch.randn(n, n, generator=g, device="cuda", dtype=torch.complex128)
    A += A.mH.clone()
    V = cl.colmajor(torch.randn(n, ncols, generator=g, device="cuda", dtype=torch.complex128))
    c, e, l1 = 20.0, 21.0, -5.0
    h = cl.Handle(0)
    try:
        got = cl.chase_filter(h, A.conj().resolve_conj().mT, V, [1] * ncols, c,
                              e, l1, prec=cl.CHASE_FP64_EMU)
    finally:
        h.close()
    s = 1.0 / (l1 - c)
    ref = s * (A @ V - c * V)
    amax = torch.view_as_real(A).abs().amax(dim=(1, 2))
    vmax = torch.view_as_real(V).abs().amax(dim=(0, 2))
    bound = abs(s) * (2 * n * 2.0 ** -53 * 2.0 * amax[:, None] * vmax[None, :] + c * V.abs() * 2.0 ** -52)
    return float(((got - ref).abs() / bound).max())


@pytest.mark.gpu
@pytest.mark.parametrize("n,ncols", [
    (1, 1), (2, 2), (63, 3), (65, 16),             # one K block, one row pair
    (128, 17), (255, 31), (256, 32), (257, 33),    # a full row pair, one chunk and its neighbours
    (320, 48), (384, 208), (513, 209), (640, 257), # half chunks, tile edges, two column tiles
])
def test_ring_product_at_the_edges(cl, n, ncols):
    assert step_error(cl, n, min(ncols, n), 11 + n) <= 1.0


@pytest.mark.gpu
def test_ring_product_beyond_the_short_range(cl):
    """K = 32832 > 2^15: 16 moduli."""
    torch.cuda.empty_cache()
    assert step_error(cl, 32800, 3, 5) <= 1.0


@pytest.mark.gpu
@pytest.mark.parametrize("complex_", [False, True])
@pytest.mark.parametrize("n,l", [(1, 1), (31, 3), (33, 32), (64, 64), (65, 33), (257, 65), (700, 257), (1025, 321)])
def test_qr_products_at_the_edges(cl, complex_, n, l):
    """CholeskyQR2 of a well-conditioned block: both its products (X^H X and X R^-1) at the edges
    of slicing tiles (32 rows x 64 of K), row pairs and column tiles.  Q is the unique factor with
    positive diagonal R: within 64 n 2^-53 of torch's, orthonormal to the same."""
    g = torch.Generator(device="cuda")
    g.manual_seed(n + l)
    dt = torch.complex128 if complex_ else torch.float64
    U = torch.linalg.qr(torch.randn(n, l, generator=g, device="cuda", dtype=dt))[0]
    M = torch.linalg.qr(torch.randn(l, l, generator=g, device="cuda", dtype=dt))[0]
    X = cl.colmajor((U * torch.linspace(1.0, 2.0, l, device="cuda", dtype=torch.float64)) @ M)
    Q0, R0 = torch.linalg.qr(X)
    d = torch.diagonal(R0)
    Q0 = Q0 * (d / d.abs())
    h = cl.Handle(0)
    try:
        rc, v, info = cl.chase_qr(h, X, 1.0, qr_force=2, prec=cl.CHASE_FP64_EMU)
    finally:
        h.close()
    tol = 64 * max(n, 16) * 2.0 ** -53
    assert rc == 0 and v == 2 and info == 0
    assert float((X - Q0).abs().max()) <= tol
    assert float((X.mH @ X - torch.eye(l, device="cuda", dtype=dt)).abs().max()) <= tol


@pytest.mark.gpu
@pytest.mark.parametrize("complex_", [False, True])
@pytest.mark.parametrize("n,ncols", [(96, 8), (97, 9)])
@pytest.mark.parametrize("scale", [-1060, -1000, 0, 900])
def test_reconstruction_over_the_exponent_range(cl, complex_, n, ncols, scale):
    """Results from the subnormal range up to 2^900, one zero column: within the scheme's bound of
    the product of the unscaled operands (and one subnormal unit for each rounding)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    dt = torch.complex128 if complex_ else torch.float64
    A = torch.randn(n, n, generator=g, device="cuda", dtype=dt)
    A = cl.colmajor(A + A.mH)
    V = cl.colmajor(torch.randn(n, ncols, generator=g, device="cuda", dtype=dt))
    V[:, ncols // 2] = 0.0
    c, e, l1 = 0.0, 1.0, -2.0  # one step: out = A V / l1
    half = 2.0 ** (scale // 2)
    h = cl.Handle(0)
    try:
        got = cl.chase_filter(h, cl.colmajor(A * half), cl.colmajor(V * half), [1] * ncols, c, e, l1,
                              prec=cl.CHASE_FP64_EMU)
    finally:
        h.close()
    parts = lambda x: torch.view_as_real(x) if complex_ else x
    ref = (A @ V) / l1
    bound = 2 * n * 2.0 ** -53 * 2.0 * parts(A).abs().max() * parts(V).abs().max()
    err = (parts(got) / half / half if scale > -1000 else parts(got * 2.0 ** 500) * 2.0 ** (-scale - 500)) - parts(ref)
    assert float(err.abs().max()) <= float(bound) + 4 * 2.0 ** (-1074 - min(scale, 0))
    assert torch.equal(got[:, ncols // 2], torch.zeros_like(got[:, 0]))
