"""Workspace of a solve whose search block is large: the blocks of the iteration and what the reduced
eigensolver keeps beside them, one real matrix of the block's order.  Sizes only: no GPU."""
import ctypes

import pytest

import paper_2603_10514_gb300 as P


@pytest.fixture(scope="module")
def lib():
    P.build()
    return P.lib()


def workspace(lib, dtype, n, l):
    b = ctypes.c_size_t(0)
    assert lib.chase_workspace_bytes(dtype, n, l, 0, P.CHASE_FP64, ctypes.byref(b)) == 0
    return b.value


@pytest.mark.parametrize("dtype,size", [(0, 8), (1, 16)])
@pytest.mark.parametrize("n,l", [(3000, 3000), (20000, 10000), (40000, 4800)])
def test_eigensolver_keeps_one_real_matrix(lib, dtype, size, n, l):
    blocks = 5 * n * l + 4 * l * l                 # V, its products and copies; reduced matrices
    fixed = workspace(lib, dtype, 8, 1)            # scratch memory and the like
    vectors = 64 * size * l + 3 * size * l * 152   # per column, and per column and SM
    assert workspace(lib, dtype, n, l) <= size * blocks + 8 * l * l + fixed + vectors + (1 << 16)
