"""The calls that a user of this library has it do, with their sizes, inputs and exact results.

``listed()`` holds one case for each kind of use and ``draw(rng)`` gives more of the same
ranges; ``prepare`` makes what a program has in hand before the call, ``run`` is one call through
the public entry points, ``work`` what it cannot do without and ``exact`` its result from plain
torch in 64 bits.

Inputs are made on the GPU from the seed: A = Q diag(lambda) Q^H with Q a product of two
discrete Fourier (real: Hartley) transforms with random diagonal signs or phases, so A is dense,
its eigenvectors are known, and making it costs a few FFTs.  Spectra are those of the library's
own workloads: evenly filled [-1, 1], or a low cluster in [-2, -1] under a wide rest in [-1, 50].
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2603_10514_gb300 as P

DEV = "cuda:0"
PRECS = {"fp64": P.CHASE_FP64, "fp64_emu": P.CHASE_FP64_EMU, "bf16x3": P.CHASE_BF16X3}


# --------------------------------------------------------------------------- cases
def listed():
    return [
        # One filter call of a small real problem (n = 1000, 30 vectors, every degree 20): the
        # smallest call, bound by its launches.
        {"name": "filter_emu_r64_small", "kind": "filter", "prec": "fp64_emu", "cplx": False, "n": 1000,
         "ncols": 30, "deg_lo": 20, "deg_hi": 20, "spectrum": "even"},
        # The filter in native FP64, the default of chase_filter, at an odd order and width with
        # per-column degrees.
        {"name": "filter_fp64_c128_odd", "kind": "filter", "prec": "fp64", "cplx": True, "n": 1531,
         "ncols": 57, "deg_lo": 10, "deg_hi": 36, "spectrum": "cluster"},
        # The filter of an ordinary complex problem (n = 3000, 150 + 30 vectors).
        {"name": "filter_emu_c128", "kind": "filter", "prec": "fp64_emu", "cplx": True, "n": 3000,
         "ncols": 180, "deg_lo": 10, "deg_hi": 36, "spectrum": "cluster"},
        # A real filter at an odd order (prime) and an odd width: every padded edge is ragged.
        {"name": "filter_emu_r64_odd", "kind": "filter", "prec": "fp64_emu", "cplx": False, "n": 4999,
         "ncols": 299, "deg_lo": 10, "deg_hi": 36, "spectrum": "even"},
        # The filter of the headline problem (complex, n = 10000, 500 + 100 vectors).
        {"name": "filter_emu_c128_full", "kind": "filter", "prec": "fp64_emu", "cplx": True, "n": 10000,
         "ncols": 600, "deg_lo": 10, "deg_hi": 36, "spectrum": "cluster"},
        # The low-precision filter that mixed-precision solves start with.
        {"name": "filter_bf16x3_c128", "kind": "filter", "prec": "bf16x3", "cplx": True, "n": 4000,
         "ncols": 240, "deg_lo": 20, "deg_hi": 20, "spectrum": "cluster"},
        # Orthonormalising a filtered block: CholeskyQR2 at the headline problem's size ...
        {"name": "qr_emu_c128_full", "kind": "qr", "cplx": True, "n": 10000, "ncols": 600, "est": 1e4,
         "log_kappa": 4.0},
        # ... and shifted CholeskyQR2 (a cautious estimate, as after a solve's second filter) on a
        # small real block.
        {"name": "qr_emu_r64_small", "kind": "qr", "cplx": False, "n": 1000, "ncols": 30, "est": 1e10,
         "log_kappa": 2.0},
        # Spectral bounds before a solve that is given none: 4 Lanczos runs of 25 steps.
        {"name": "lanczos_r64", "kind": "lanczos", "cplx": False, "n": 8000, "runs": 4, "steps": 25,
         "ell": 480, "spectrum": "even"},
        # A whole solve of the small real problem (n = 1000, 20 + 10 vectors, fixed degrees).
        {"name": "solve_emu_r64_small", "kind": "solve", "cplx": False, "n": 1000, "nev": 20, "nex": 10,
         "opt": False, "spectrum": "even"},
        # The headline: a whole solve of a complex clustered problem, per-column degrees.
        {"name": "solve_emu_c128_full", "kind": "solve", "cplx": True, "n": 10000, "nev": 500, "nex": 100,
         "opt": True, "spectrum": "cluster"},
        # A batch of uneven problems, real and complex in turn, as a service holds in flight.
        {"name": "batch_emu_uneven", "kind": "batch", "count": 12, "n_lo": 505, "n_hi": 3948,
         "spread": 0.37},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["filter", "filter", "filter", "qr", "qr", "lanczos", "solve", "solve", "batch"])
    cplx = rng.random() < 0.5
    if kind == "filter":
        prec = rng.choice(["fp64_emu", "fp64_emu", "fp64_emu", "fp64", "bf16x3"])
        n = _log_uniform(rng, 500, 2000 if prec == "fp64" else 9000)
        opt = rng.random() < 0.7
        return {"kind": kind, "prec": prec, "cplx": cplx, "n": n,
                "ncols": max(1, int(n * rng.uniform(0.01, 0.08))), "deg_lo": 10 if opt else 20,
                "deg_hi": 36 if opt else 20, "spectrum": rng.choice(["even", "cluster"])}
    if kind == "qr":
        n = _log_uniform(rng, 500, 10000)
        log_kappa = rng.uniform(0.5, 5.0)
        # the estimate bounds the condition number from above, by a little or by a lot
        return {"kind": kind, "cplx": cplx, "n": n, "ncols": max(1, int(n * rng.uniform(0.01, 0.08))),
                "est": 10.0 ** (log_kappa + rng.choice([0.3, 1.5, 6.0])), "log_kappa": log_kappa}
    if kind == "lanczos":
        n = _log_uniform(rng, 500, 9000)
        return {"kind": kind, "cplx": cplx, "n": n, "runs": 4, "steps": 25, "ell": max(4, n * 6 // 100),
                "spectrum": rng.choice(["even", "cluster"])}
    if kind == "solve":
        n = _log_uniform(rng, 500, 5000)
        nev = max(2, int(n * rng.uniform(0.02, 0.05)))
        return {"kind": kind, "cplx": cplx, "n": n, "nev": nev, "nex": max(2, nev // 5),
                "opt": rng.random() < 0.7, "spectrum": rng.choice(["even", "cluster"])}
    lo = _log_uniform(rng, 500, 1000)
    return {"kind": kind, "count": rng.randint(4, 16), "n_lo": lo, "n_hi": _log_uniform(rng, 1500, 3500),
            "spread": rng.random()}


def _batch_problems(case):
    """The problems of a batch: orders log-uniform in [n_lo, n_hi] (a low-discrepancy sequence
    from `spread`), nev 5 % and nex 1 % of n, real and complex in turn."""
    out = []
    for i in range(case["count"]):
        u = (case["spread"] + i * 0.6180339887498949) % 1.0
        n = int(round(math.exp(math.log(case["n_lo"]) + u * math.log(case["n_hi"] / case["n_lo"]))))
        nev = max(2, n * 5 // 100)
        out.append({"cplx": i % 2 == 1, "n": n, "nev": nev, "nex": max(2, n // 100), "opt": True,
                    "spectrum": "even"})
    return out


# --------------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _dt(cplx):
    return torch.complex128 if cplx else torch.float64


def _transform(x, cplx, inverse=False):
    """Unitary DFT (complex) or Hartley transform (real) along dim 0."""
    if cplx:
        return (torch.fft.ifft if inverse else torch.fft.fft)(x, dim=0, norm="ortho")
    f = torch.fft.fft(x, dim=0, norm="ortho")
    return f.real - f.imag


def _signs(n, cplx, g):
    if cplx:
        a = torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * (2 * math.pi)
        return torch.polar(torch.ones_like(a), a)
    return torch.randint(0, 2, (n,), generator=g, device=DEV).to(torch.float64) * 2 - 1


def _spectrum(n, ell, kind, g):
    """Ascending eigenvalues.  even: one in each of n equal cells of [-1, 1]; cluster: ell of them
    geometric in [-2, -1], densest at the bottom, the rest one in each cell of [-1, 50]."""
    def cells(m, lo, hi):
        u = torch.rand(m, generator=g, device=DEV, dtype=torch.float64)
        i = torch.arange(m, device=DEV, dtype=torch.float64)
        return lo + (hi - lo) * (i + 0.25 + 0.5 * u) / m
    if kind == "even":
        return cells(n, -1.0, 1.0)
    i = torch.arange(ell, device=DEV, dtype=torch.float64)
    low = -2.0 + (torch.exp2(i / max(ell - 1, 1)) - 1.0)
    return torch.cat([low, cells(n - ell, -1.0, 50.0)])


class Matrix:
    """A = Q diag(lam) Q^H, Q = diag(d1) F diag(d2) F, column-major; bounds as a solve gets them."""

    def __init__(self, n, ell, spectrum, cplx, g):
        self.n, self.cplx = n, cplx
        self.lam = _spectrum(n, ell, spectrum, g)
        self.d1, self.d2 = _signs(n, cplx, g), _signs(n, cplx, g)
        lam = self.lam.cpu()
        lo, hi = float(lam[0]), float(lam[-1])
        self.bounds = (lo, float(lam[ell - 1]), hi + 1e-3 * max(1.0, hi - lo))

    def vectors(self, X):
        """Q X for a block X (n x m)."""
        Y = self.d2[:, None] * _transform(X, self.cplx)
        return self.d1[:, None] * _transform(Y, self.cplx)

    def dense(self):
        M = torch.diag(self.lam.to(_dt(self.cplx)))
        for d in (self.d2, self.d1):  # M <- D F M F^H D^H (M Hermitian)
            M = _transform(M, self.cplx)
            M = _transform(M.mH.contiguous(), self.cplx)
            M = d[:, None] * M * d.conj()[None, :]
        return P.colmajor(0.5 * (M + M.mH))


def _gauss(n, m, cplx, g):
    return P.colmajor(torch.randn(n, m, generator=g, device=DEV, dtype=_dt(cplx)) / math.sqrt(n))


def _degrees(case):
    return np.round(np.linspace(case["deg_lo"], case["deg_hi"], case["ncols"])).astype(np.int32)


_kept = {}


def _handle():
    """The program's handle: one for the process, on torch's current stream."""
    if "h" not in _kept:
        _kept["h"] = P.Handle(0, torch.cuda.current_stream().cuda_stream)
    return _kept["h"]


def _session():
    """The service's batch session, kept open between batches."""
    if "b" not in _kept:
        _kept["b"] = P.Batch(_handle())
    return _kept["b"]


def _problem(c, g):
    """Matrix, start block and a fixed vector for the phases of one eigenproblem."""
    ell = c["nev"] + c["nex"]
    M = Matrix(c["n"], ell, c["spectrum"], c["cplx"], g)
    V0 = _gauss(c["n"], ell, c["cplx"], g)
    ref = torch.randn(c["n"], generator=g, device=DEV, dtype=_dt(c["cplx"]))
    return M, V0, ref


def _filter_inputs(case, seed):
    g = _gen(seed)
    M = Matrix(case["n"], case["ncols"], case["spectrum"], case["cplx"], g)
    V = _gauss(case["n"], case["ncols"], case["cplx"], g)
    lo, mid, hi = M.bounds
    return M, V, (0.5 * (hi + mid), 0.5 * (hi - mid), lo)


def _qr_input(case, seed):
    """A block with condition number 10^log_kappa: orthonormal columns times a geometric
    spread times a unitary mix (columns of similar size, as a filter leaves them)."""
    n, l, cplx, g = case["n"], case["ncols"], case["cplx"], _gen(seed)
    s = torch.logspace(0.0, -case["log_kappa"], l, device=DEV, dtype=torch.float64)
    d = [_signs(n, cplx, g), _signs(n, cplx, g), _signs(l, cplx, g), _signs(l, cplx, g)]
    mix = torch.eye(l, device=DEV, dtype=_dt(cplx))
    for k in (2, 3):
        mix = d[k][:, None] * _transform(mix, cplx)
    X = torch.zeros(n, l, device=DEV, dtype=_dt(cplx))
    X[:l] = s[:, None] * mix
    for k in (0, 1):
        X = d[k][:, None] * _transform(X, cplx)
    return P.colmajor(X)


def prepare(case, seed):
    h, kind = _handle(), case["kind"]
    if kind == "filter":
        M, V, (c, e, lam1) = _filter_inputs(case, seed)
        return {"kind": kind, "h": h, "A": M.dense(), "V": V, "out": torch.empty_like(V), "deg": _degrees(case),
                "c": c, "e": e, "lam1": lam1, "prec": PRECS[case["prec"]]}
    if kind == "qr":
        X0 = _qr_input(case, seed)
        return {"kind": kind, "h": h, "X0": X0, "X": torch.empty_like(X0), "est": case["est"]}
    if kind == "lanczos":
        g = _gen(seed)
        M = Matrix(case["n"], case["ell"], case["spectrum"], case["cplx"], g)
        return {"kind": kind, "h": h, "A": M.dense(), "V": _gauss(case["n"], case["runs"], case["cplx"], g),
                "steps": case["steps"], "ell": case["ell"]}
    if kind == "solve":
        M, V0, ref = _problem(case, _gen(seed))
        return {"kind": kind, "h": h, "A": M.dense(), "V0": V0, "V": torch.empty_like(V0), "ref": ref,
                "nev": case["nev"], "nex": case["nex"], "bounds": M.bounds,
                "cfg": P.config_default(opt_degree=int(case["opt"]), prec=P.CHASE_FP64_EMU)}
    probs = []
    for i, c in enumerate(_batch_problems(case)):
        M, V0, ref = _problem(c, _gen(seed * 1009 + i))
        probs.append({"A": M.dense(), "V0": V0, "V": torch.empty_like(V0), "ref": ref, "nev": c["nev"],
                      "nex": c["nex"], "bounds": M.bounds,
                      "cfg": P.config_default(opt_degree=int(c["opt"]), prec=P.CHASE_FP64_EMU)})
    return {"kind": kind, "b": _session(), "probs": probs}


# --------------------------------------------------------------------------- one pass
def _phased(Y, ref):
    """Eigenvectors are defined up to a phase: the one a program fixes before it keeps them
    makes each column's inner product with a fixed vector real and positive."""
    s = ref.conj() @ Y
    return Y * (s.conj() / s.abs())


def run(s):
    kind = s["kind"]
    if kind == "filter":
        return P.chase_filter(s["h"], s["A"], s["V"], s["deg"], s["c"], s["e"], s["lam1"], out=s["out"],
                              prec=s["prec"])
    if kind == "qr":
        s["X"].copy_(s["X0"])
        P.chase_qr(s["h"], s["X"], s["est"], prec=P.CHASE_FP64_EMU)
        return s["X"]
    if kind == "lanczos":
        return list(P.chase_lanczos_bounds(s["h"], s["A"], s["V"], s["steps"], s["ell"]))
    if kind == "solve":
        # the residual norms (rounding of numbers near the tolerance) and the search block's
        # unconverged rest are not results
        s["V"].copy_(s["V0"])
        rc, evals, _, _, _ = P.chase_solve(s["h"], s["A"], s["V"], s["nev"], s["nex"], s["bounds"], s["cfg"],
                                           log_cap=0)
        return {"status": rc, "evals": evals, "vectors": _phased(s["V"][:, :s["nev"]], s["ref"])}
    probs = []
    for p in s["probs"]:
        p["V"].copy_(p["V0"])
        probs.append(s["b"].add(P.BatchProblem(p["A"], p["V"], p["nev"], p["nex"], p["bounds"], p["cfg"])))
    while s["b"].pending():
        s["b"].step()
    return [{"status": q.status, "evals": q.evals, "vectors": _phased(p["V"][:, :p["nev"]], p["ref"])}
            for p, q in zip(s["probs"], probs)]


# --------------------------------------------------------------------------- floors
def _solve_work(c):
    """A whole solve: the filter products (about 190 column products per vector with per-column
    degrees, 160 with the fixed degree, as these spectra take) and A, V0 and the vectors once."""
    ell, w = c["nev"] + c["nex"], 16 if c["cplx"] else 8
    per = (8.0 if c["cplx"] else 2.0) * c["n"] ** 2
    return {"bytes": w * (c["n"] ** 2 + 2.0 * c["n"] * ell), "flops": per * ell * (190 if c["opt"] else 160)}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        w = [_solve_work(c) for c in _batch_problems(case)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    if kind == "solve":
        return _solve_work(case)
    n, w, mac = case["n"], 16 if case["cplx"] else 8, 8.0 if case["cplx"] else 2.0
    if kind == "filter":
        return {"bytes": w * (n * n + 2.0 * n * case["ncols"]), "flops": mac * n * n * float(_degrees(case).sum())}
    if kind == "qr":
        l = case["ncols"]
        return {"bytes": w * 2.0 * n * l, "flops": 2.0 * mac * n * l * l}
    # Lanczos: A is read once per step, by all runs together
    return {"bytes": w * 1.0 * n * n * case["steps"], "flops": mac * n * n * case["runs"] * case["steps"]}


# --------------------------------------------------------------------------- exact results
def _exact_pairs(c, g):
    M, _, ref = _problem(c, g)
    E = torch.zeros(c["n"], c["nev"], device=DEV, dtype=_dt(c["cplx"]))
    E[:c["nev"]] = torch.eye(c["nev"], device=DEV, dtype=E.dtype)
    return {"status": 0, "evals": M.lam[:c["nev"]].cpu().numpy(), "vectors": _phased(M.vectors(E), ref)}


def _exact_filter(case, seed):
    M, V, (c, e, lam1) = _filter_inputs(case, seed)
    A, deg = M.dense(), torch.from_numpy(_degrees(case)).to(DEV)
    sigma1 = e / (lam1 - c)
    prev, cur, sigma = None, V, sigma1
    out = torch.where(deg[None, :] == 0, V, torch.zeros_like(V))
    for step in range(1, case["deg_hi"] + 1):
        if step == 1:
            prev, cur = cur, (A @ cur - c * cur) * (sigma1 / e)
        else:
            new = 1.0 / (2.0 / sigma1 - sigma)
            prev, cur = cur, (A @ cur - c * cur) * (2.0 * new / e) - (sigma * new) * prev
            sigma = new
        out = torch.where(deg[None, :] == step, cur, out)
    return out


def _exact_lanczos(case, seed):
    g = _gen(seed)
    M = Matrix(case["n"], case["ell"], case["spectrum"], case["cplx"], g)
    A, V = M.dense(), _gauss(case["n"], case["runs"], case["cplx"], g)
    theta, tau, top = [], [], []
    for r in range(case["runs"]):
        q = V[:, r] / torch.linalg.vector_norm(V[:, r])
        basis, al, be = [q], [], []
        for _ in range(case["steps"]):
            w = A @ basis[-1]
            al.append(float((basis[-1].conj() @ w).real))
            B = torch.stack(basis, dim=1)
            for _ in range(2):
                w = w - B @ (B.mH @ w)
            be.append(float(torch.linalg.vector_norm(w)))
            basis.append(w / be[-1])
        t, S = np.linalg.eigh(np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1))
        theta.append(t)
        tau.append(S[0] ** 2)
        top.append(t[-1] + abs(be[-1]))
    t, w = np.concatenate(theta), np.concatenate(tau)
    o = np.argsort(t)
    count = case["n"] / case["runs"] * np.cumsum(w[o])
    at = min(int(np.searchsorted(count, case["ell"] * (1.0 - 1e-10))), len(t) - 1)
    return [float(t.min()), float(t[o][at]), float(max(top))]


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        return _exact_pairs(case, _gen(seed))
    if kind == "batch":
        return [_exact_pairs(c, _gen(seed * 1009 + i)) for i, c in enumerate(_batch_problems(case))]
    if kind == "filter":
        return _exact_filter(case, seed)
    if kind == "lanczos":
        return _exact_lanczos(case, seed)
    Q, R = torch.linalg.qr(_qr_input(case, seed))
    d = torch.diagonal(R)
    return Q * (d / d.abs())
