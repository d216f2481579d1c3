"""The autotuner keeps the plans of real products apart from those of ring products (complex): a
complex problem that is tuned first leaves the real one of the same sizes to be measured, K splits
among its candidates."""
import re

import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cl():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_10514_gb300 as P
    P.build()
    return P


def tuned(cl, complex_):
    n, nev, nex = 600, 24, 8
    lam = W.spectrum_uniform(n, -1.0, 1.0, 5)
    A = W.known_spectrum_matrix(lam, 5, complex_, device="cuda")
    V = torch.from_numpy(np.ascontiguousarray(W.start_block(n, nev + nex, 6, complex_).T)).cuda().mT
    h = cl.Handle(0)
    try:
        cfg = cl.config_default(opt_degree=1, prec=cl.CHASE_FP64_EMU, autotune=1)
        bounds = (float(lam[0]), float(lam[nev + nex - 1]), float(lam[-1]) + 1e-3)
        rc, _, _, st, _ = cl.chase_solve(h, A, V, nev, nex, bounds, cfg)
    finally:
        h.close()
    assert rc == 0
    return st["autotune_trials"]


def buckets(cl):
    """Bucket -> splits of its plan, for each kind of product."""
    out = {}
    for line in cl.autotune_table():
        f = dict(re.findall(r"(\w+)=(\S+)", line))
        out.setdefault(int(f["ring"]), {})[f["bucket"]] = int(f["splits"])
    return out


def test_real_and_ring_products_are_tuned_apart(cl):
    cl.autotune_clear()
    try:
        assert tuned(cl, True) > 0
        first = buckets(cl)
        assert set(first) == {15} and set(first[15].values()) == {1}
        assert tuned(cl, False) > 0
        both = buckets(cl)
        assert set(both) == {0, 15} and both[15] == first[15]
        assert set(both[0]) & set(both[15])  # the same sizes, each with a plan of its own
        assert tuned(cl, True) == 0 and tuned(cl, False) == 0
    finally:
        cl.autotune_clear()
