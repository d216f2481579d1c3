"""Lanczos bounds with every count of runs that the product kernel groups differently (1 to 4 per
pass over A, remainders, leading dimension above n), against the oracle; tolerance as for the
4-run parity test."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def cl():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_10514_gb300 as P
    P.build()
    return P


@pytest.mark.parametrize("complex_", [False, True])
@pytest.mark.parametrize("n,nruns,steps", [(3, 1, 2), (33, 2, 20), (257, 3, 25), (300, 5, 33), (301, 8, 10)])
def test_bounds_for_every_grouping_of_runs(cl, complex_, n, nruns, steps):
    lam = W.spectrum_uniform(n, -1.0, 1.0, 5)
    A = W.known_spectrum_matrix(lam, 5, complex_).numpy()
    V = W.start_block(n, nruns, 6, complex_)
    ell = max(1, n // 10)
    ref, _ = oracle.lanczos_bounds(A, V, steps, ell)
    pad = torch.zeros((n, n + 3), dtype=torch.complex128 if complex_ else torch.float64, device="cuda")
    pad[:, :n] = torch.from_numpy(np.ascontiguousarray(A.T))
    Vd = torch.from_numpy(np.ascontiguousarray(V.T)).cuda().mT
    h = cl.Handle(0)
    try:
        got = cl.chase_lanczos_bounds(h, pad[:, :n].mT, Vd, steps, ell)
    finally:
        h.close()
    np.testing.assert_allclose(got, ref, rtol=0, atol=1e-9 * (lam[-1] - lam[0]))
