"""The FP64 products' split into tiles and runs of K steps.

On the CPU: gemm_split.h, compiled for the host, over shapes, triangular forms, CTA counts and
scratch limits: every K step of every tile is taken once, parts of shared tiles have slots of their
own inside the scratch memory, and the owners of a tile's first and last step are right.  On the
GPU: one filter step and CholeskyQR at edges of tiles and blocks, against the same sums in another
order: 2 n + 16 roundings (complex: twice that) of |A| |V| per entry.
"""
import ctypes
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_10514_gb300", "csrc")

DRIVER = r"""
#include <vector>
#include "gemm_split.h"
using namespace chase;
extern "C" int check(int M, int N, int K, int upper, int tri, int ctas, int kmin, long long room) {
  const GemmSplit s = gemm_split(M, N, K, upper, tri, ctas, kmin, room);
  if (s.bn < 1 || s.bn > kGemmCols || !s.whole && (s.G > ctas || s.slots() * s.slot_elems() > room)) return 1;
  std::vector<char> covered((size_t)M * N, 0);
  long long w = 0;
  for (int t = 0; t < s.T; ++t) {
    const GemmTile q = s.tile(t);
    if (q.t != t || q.w0 != w || q.nb < 1 || q.nb > s.bn || q.kt != (tri && q.n0 + s.bn < s.K ? q.n0 + s.bn : s.K))
      return 2;
    w += q.kt;
    for (int j = q.n0; j < q.n0 + q.nb; ++j)
      for (int i = q.m0; i < q.m0 + kGemmRows && i < M; ++i)
        if (j >= N || covered[(size_t)j * M + i]++) return 3;
  }
  if (w != s.W) return 4;
  for (int j = 0; j < N; ++j)
    for (int i = 0; i < M; ++i)
      if (!covered[(size_t)j * M + i] && !(upper && i > j)) return 5;
  if (s.whole) return s.G == s.T ? 0 : 6;
  std::vector<char> slot(s.slots(), 0);
  std::vector<int> done(s.T, 0), lo(s.T, -1), hi(s.T, -1);
  for (int g = 0; g < s.G; ++g) {
    long long a = s.begin(g);
    const long long b = s.begin(g + 1);
    if (b <= a) return 7;
    while (a < b) {
      const GemmTile q = s.at(a);
      const int k0 = (int)(a - q.w0), k1 = (int)(q.kt < k0 + (b - a) ? q.kt : k0 + (b - a));
      if (k0 != done[q.t] || k1 <= k0) return 8;
      done[q.t] = k1;
      if (lo[q.t] < 0) lo[q.t] = g;
      hi[q.t] = g;
      if (k1 - k0 < q.kt && (g + q.t >= s.slots() || slot[g + q.t]++)) return 9;
      a += k1 - k0;
    }
  }
  for (int t = 0; t < s.T; ++t) {
    const GemmTile q = s.tile(t);
    if (done[t] != q.kt || s.owner(q.w0) != lo[t] || s.owner(q.w0 + q.kt - 1) != hi[t]) return 10;
  }
  return 0;
}
"""


def test_split_takes_every_step_once(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    (tmp_path / "s.cpp").write_text(DRIVER)
    so = str(tmp_path / "s.so")
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-I", CSRC, str(tmp_path / "s.cpp"), "-o", so], check=True)
    check = ctypes.CDLL(so).check
    check.argtypes = [ctypes.c_int] * 7 + [ctypes.c_longlong]
    for M in (1, 63, 64, 65, 300, 1531):
        for N in (1, 3, 16, 57, 64, 65, 130, 300):
            for K in (0, 1, 7, 8, 100, 1531):
                for upper, tri in ((0, 0), (1, 0), (0, 1)):
                    if upper and M != N:
                        continue
                    for room in (0, 100000, 1 << 23):
                        for ctas, kmin in ((304, 8), (304, 16), (7, 1)):
                            assert check(M, N, K, upper, tri, ctas, kmin, room) == 0, (M, N, K, upper, tri, ctas, room)


torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def cl():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_10514_gb300 as P
    P.build()
    return P


@pytest.mark.gpu
@pytest.mark.parametrize("noalloc", [False, True])
@pytest.mark.parametrize("complex_", [False, True])
@pytest.mark.parametrize("n,ncols", [(1, 1), (7, 3), (63, 2), (64, 16), (65, 57), (129, 64), (400, 1), (700, 65),
                                     (1200, 130), (2100, 299)])
def test_one_fp64_step(cl, n, ncols, complex_, noalloc):
    ncols = min(ncols, n)
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    dt = torch.complex128 if complex_ else torch.float64
    A = torch.randn(n, n, generator=g, device="cuda", dtype=dt)
    A = cl.colmajor(A + A.mH)
    V = cl.colmajor(torch.randn(n, ncols, generator=g, device="cuda", dtype=dt))
    c, e, l1 = 20.0, 21.0, -5.0
    if noalloc:
        got = cl.chase_filter_noalloc(A, V, [1] * ncols, c, e, l1)
    else:
        h = cl.Handle(0)
        try:
            got = cl.chase_filter(h, A, V, [1] * ncols, c, e, l1)
        finally:
            h.close()
    s = 1.0 / (l1 - c)
    ref = s * (A @ V - c * V)
    bound = abs(s) * (A.abs() @ V.abs() + c * V.abs()) * (2 * n + 16) * 2.0 ** -53 * (2 if complex_ else 1)
    assert float(((got - ref).abs() / bound).max()) <= 1.0


@pytest.mark.gpu
@pytest.mark.parametrize("complex_", [False, True])
@pytest.mark.parametrize("n,l", [(1, 1), (64, 64), (130, 65), (700, 33), (900, 129), (1500, 300)])
def test_fp64_qr(cl, n, l, complex_):
    g = torch.Generator(device="cuda")
    g.manual_seed(l)
    X = cl.colmajor(torch.randn(n, l, generator=g, device="cuda",
                                dtype=torch.complex128 if complex_ else torch.float64))
    X0 = X.clone()
    h = cl.Handle(0)
    try:
        rc, v, info = cl.chase_qr(h, X, 1.0, qr_force=2)
    finally:
        h.close()
    assert rc == 0 and v == 2
    eye = torch.eye(l, device="cuda", dtype=X.dtype)
    assert float(torch.linalg.norm(X.mH @ X - eye)) <= 1e-12
    R = X.mH @ X0
    assert float(torch.linalg.norm(X @ R - X0)) <= 1e-12 * float(torch.linalg.norm(X0))
    assert float(torch.linalg.norm(torch.tril(R, -1))) <= 1e-12 * float(torch.linalg.norm(X0))
