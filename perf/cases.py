"""The work that a user of the eigensolver has it do, as measurable cases.

Whole solves in both forms (FP64 and mixed + refined) over the range of orders
the library takes, values only and partial vectors, uneven batches, the
Bethe-Salpeter driver, and the FP64-accurate product on its own.  Inputs are
the paper's random skew matrices (entries of (G - G^T)/2, G normal) and the
Bethe-Salpeter shaped ones of ``inputs.bse``, drawn on the GPU.

An eigenvector is defined up to a unit factor.  A program that compares or
combines vectors of two runs fixes that factor, and so do the passes here: a
column z is multiplied by the unit factor that makes p^H z real and positive
for a probe p that comes with the input (the transition dipole of an
absorption spectrum, say); the columns of a batch by the one that makes their
first component so.  The vectors come back whole.
"""
import math

import numpy as np
import torch

import paper_1912_04062_gb300 as sk

MODES = {"fp64": sk.SKEW_MODE_FP64, "refined": sk.SKEW_MODE_MIXED_REFINED}


def listed():
    return [
        # the smallest call of the synchronous entry point with its defaults: latency and launches
        {"name": "fp64_n48", "kind": "solve", "mode": "fp64", "n": 48, "nev": 24, "vectors": True, "matrix": "random"},
        # FP64 solves of half the spectrum: ordinary, ragged, and the largest that FP64 arithmetic does in a second
        {"name": "fp64_n500", "kind": "solve", "mode": "fp64", "n": 500, "nev": 250, "vectors": True,
         "matrix": "random"},
        {"name": "fp64_n1501", "kind": "solve", "mode": "fp64", "n": 1501, "nev": 750, "vectors": True,
         "matrix": "random"},
        {"name": "fp64_n4096", "kind": "solve", "mode": "fp64", "n": 4096, "nev": 2048, "vectors": True,
         "matrix": "bse"},
        # the mixed form with its refinement (a complete basis): the benchmark's solve at three orders
        {"name": "refined_n1000", "kind": "solve", "mode": "refined", "n": 1000, "nev": 500, "vectors": True,
         "matrix": "random"},
        {"name": "refined_n3002", "kind": "solve", "mode": "refined", "n": 3002, "nev": 1501, "vectors": True,
         "matrix": "bse"},
        {"name": "refined_n8192", "kind": "solve", "mode": "refined", "n": 8192, "nev": 4096, "vectors": True,
         "matrix": "bse"},
        # a tenth of the spectrum with vectors, odd order (nothing to refine against: double-float Q_trd)
        {"name": "partial_n6001", "kind": "solve", "mode": "refined", "n": 6001, "nev": 600, "vectors": True,
         "matrix": "random"},
        # all eigenvalues, no vectors
        {"name": "values_n4000", "kind": "solve", "mode": "refined", "n": 4000, "nev": 2000, "vectors": False,
         "matrix": "random"},
        # an uneven batch through a plan (orders log-uniform in [32, 1024], as the batched benchmark's)
        {"name": "batch_96", "kind": "batch", "count": 96, "lo": 32, "hi": 1024},
        # the Bethe-Salpeter eigenproblem with complex blocks, all positive eigenvalues
        {"name": "bse_h600", "kind": "bse", "mode": "fp64", "h": 600, "nev": 600},
        # the FP64-accurate tensor-core product that callers use by itself
        {"name": "product", "kind": "product", "m": 4096, "n": 3000, "k": 5000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fp64", "refined", "partial", "values", "batch", "bse", "product"])
    if kind == "fp64":
        n = _log(rng, 40, 4096)
        return {"kind": "solve", "mode": "fp64", "n": n, "nev": n // 2, "vectors": True, "matrix": "random"}
    if kind == "refined":
        n = 2 * _log(rng, 64, 3600)
        return {"kind": "solve", "mode": "refined", "n": n, "nev": n // 2, "vectors": True,
                "matrix": rng.choice(["random", "bse"])}
    if kind == "partial":
        n = _log(rng, 300, 6000)
        return {"kind": "solve", "mode": rng.choice(["refined", "refined", "fp64"]), "n": n,
                "nev": max(1, int(n * rng.uniform(0.02, 0.12))), "vectors": True, "matrix": "random"}
    if kind == "values":
        n = _log(rng, 100, 6000)
        return {"kind": "solve", "mode": rng.choice(["refined", "fp64"]) if n < 4000 else "refined", "n": n,
                "nev": n // 2, "vectors": False, "matrix": "random"}
    if kind == "batch":
        return {"kind": "batch", "count": _log(rng, 4, 160), "lo": rng.choice([16, 32, 48]), "hi": _log(rng, 64, 1024)}
    if kind == "bse":
        h = _log(rng, 32, 800)
        return {"kind": "bse", "mode": rng.choice(["fp64", "refined"]), "h": h,
                "nev": rng.choice([h, max(1, h // 5)])}
    return {"kind": "product", "m": _log(rng, 200, 5000), "n": _log(rng, 200, 5000), "k": _log(rng, 200, 6000)}


# ------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _sym(G):
    return 0.5 * (G + G.transpose(0, 1))


def _matrix(case, g):
    """The skew matrix of a solve."""
    n = case["n"]
    if case["matrix"] == "random":
        G = _randn(g, n, n)
        return sk.fortran(0.5 * (G - G.T))
    # K = L^T J L of M = [[Ad, B], [B, Ad]] = L L^T, the recipe of inputs.bse
    h = n // 2
    Ad = 0.05 * _sym(_randn(g, h, h)) / math.sqrt(h)
    Ad += torch.diag(2.0 + 18.0 * torch.rand(h, generator=g, device="cuda", dtype=torch.float64))
    B = 0.02 * _sym(_randn(g, h, h)) / math.sqrt(h)
    L = torch.linalg.cholesky(torch.cat([torch.cat([Ad, B], 1), torch.cat([B, Ad], 1)], 0))
    K = L.T @ torch.cat([L[h:], -L[:h]], 0)
    return sk.fortran(0.5 * (K - K.T))


def _blocks(case, g):
    """Hermitian A and complex symmetric B of a definite H_BS = [[A, B], [-conj(B), -conj(A)]]."""
    h = case["h"]
    G = torch.complex(_randn(g, h, h), _randn(g, h, h))
    A = 0.025 * (G + G.conj().T) / math.sqrt(h)
    A = A + torch.diag(2.0 + 18.0 * torch.rand(h, generator=g, device="cuda", dtype=torch.float64)).to(A.dtype)
    G = torch.complex(_randn(g, h, h), _randn(g, h, h))
    return A, 0.01 * (G + G.T) / math.sqrt(h)


def _batch(case, seed):
    """The matrices of a batch.  The orders belong to the case, and the largest is always there."""
    u = np.random.default_rng(case["count"]).uniform(math.log(case["lo"]), math.log(case["hi"]), case["count"])
    ns = [int(v) for v in np.rint(np.exp(u))]
    ns[0] = case["hi"]
    g = _gen(seed)
    out = []
    for n in ns:
        G = _randn(g, n, n)
        out.append(sk.fortran(0.5 * (G - G.T)))
    return out


def _probe(g, n):
    return _randn(g, n), _randn(g, n)


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "solve":
        A = _matrix(case, g)
        n, nev, vec = case["n"], case["nev"], case["vectors"]
        opts = sk.Options(mode=MODES[case["mode"]])
        dev = A.device
        return {"kind": kind, "A": A, "nev": nev, "probe": _probe(g, n), "opts": opts, "sync": n < 100,
                "lam": torch.empty(nev, dtype=torch.float64, device=dev),
                "Zr": sk.fortran_empty(n, nev) if vec else None, "Zi": sk.fortran_empty(n, nev) if vec else None,
                "ws": torch.empty(sk.workspace_size(n, nev, opts, vectors=vec), dtype=torch.uint8, device=dev),
                "info": torch.zeros(1, dtype=torch.int32, device=dev)}
    if kind == "batch":
        As = _batch(case, seed)
        nevs = [A.shape[0] // 2 for A in As]
        ns = torch.tensor([A.shape[0] for A in As])
        rows = torch.repeat_interleave(ns, torch.tensor(nevs))      # rows of every column of the batch
        first = torch.cumsum(rows, 0) - rows
        column = torch.repeat_interleave(torch.arange(len(rows)), rows)
        return {"kind": kind, "plan": sk.BatchedPlan(As, nevs), "first": first.cuda(), "column": column.cuda()}
    if kind == "bse":
        A, B = _blocks(case, g)
        return {"kind": kind, "A": A, "B": B, "nev": case["nev"], "opts": sk.Options(mode=MODES[case["mode"]]),
                "probe": _probe(g, 2 * case["h"])}
    return {"kind": kind, "A": _randn(g, case["m"], case["k"]), "B": _randn(g, case["n"], case["k"])}


# ------------------------------------------------------------------- passes
def _fix_phase(X, Y, probe):
    """(X, Y) times the unit factors that make p^H (X + iY) real and positive, column by column."""
    p, q = probe
    a = X.T @ p + Y.T @ q
    b = Y.T @ p - X.T @ q
    r = torch.hypot(a, b)
    c, s = a / r, b / r
    return X * c + Y * s, Y * c - X * s


def run(state):
    kind = state["kind"]
    if kind == "solve":
        if state["sync"]:
            lam, X, Y = sk.skew_eig(state["A"], state["nev"], vectors=state["Zr"] is not None)
        else:
            code = sk.skew_eig_ex(state["A"], state["nev"], state["lam"], state["Zr"], state["Zi"], state["ws"],
                                  state["info"], state["opts"])
            if code:
                raise sk.SkewError(code, "skew_eig_ex")
            lam, X, Y = state["lam"], state["Zr"], state["Zi"]
        return {"lam": lam, "z": _fix_phase(X, Y, state["probe"])} if X is not None else {"lam": lam}
    if kind == "batch":
        plan = state["plan"]
        plan.execute()
        lams, Xs, Ys = plan.results()
        x = torch.cat([X.T.reshape(-1) for X in Xs])
        y = torch.cat([Y.T.reshape(-1) for Y in Ys])
        a, b = x[state["first"]], y[state["first"]]
        r = torch.hypot(a, b)
        c, s = (a / r)[state["column"]], (b / r)[state["column"]]
        return {"lam": torch.cat(lams), "z": (x * c + y * s, y * c - x * s)}
    if kind == "bse":
        lam, psi, _ = sk.bse_solve(state["A"], state["B"], state["nev"], state["opts"])
        return {"lam": lam, "z": _fix_phase(psi.real, psi.imag, state["probe"])}
    return sk.gemm_f64acc(state["A"], state["B"])[0]


# --------------------------------------------------------------------- work
def _solve_work(n, nev, vectors):
    """One-step tridiagonalisation, and its back-transform of real and imaginary parts."""
    flops = 4.0 / 3.0 * n ** 3 + (4.0 * n * n * nev if vectors else 0.0)
    return 4.0 * n * n + 8.0 * nev + (16.0 * n * nev if vectors else 0.0), flops


def work(case):
    kind = case["kind"]
    if kind == "solve":
        b, f = _solve_work(case["n"], case["nev"], case["vectors"])
    elif kind == "batch":
        u = np.random.default_rng(case["count"]).uniform(math.log(case["lo"]), math.log(case["hi"]), case["count"])
        ns = [int(v) for v in np.rint(np.exp(u))]
        ns[0] = case["hi"]
        both = [_solve_work(n, n // 2, True) for n in ns]
        b, f = sum(x[0] for x in both), sum(x[1] for x in both)
    elif kind == "bse":
        h, nev = case["h"], case["nev"]
        n = 2 * h
        b, f = _solve_work(n, nev, True)
        b = 32.0 * h * h + 8.0 * nev + 16.0 * n * nev
        f += n ** 3 / 3.0 + n ** 3 + 2.0 * n * n * nev      # Cholesky, the skew product's triangle, L^-T z
    else:
        m, n, k = case["m"], case["n"], case["k"]
        b, f = 8.0 * (m * k + n * k + m * n), 2.0 * m * n * k
    return {"bytes": b, "flops": f}


# -------------------------------------------------------------------- exact
def _eigh(A, nev, vectors):
    """The nev largest lambda of skew A (descending) and vectors of i*lambda, from -iA's Hermitian solve."""
    H = torch.complex(torch.zeros_like(A), -A)
    if not vectors:
        return torch.linalg.eigvalsh(H).flip(0)[:nev], None
    w, V = torch.linalg.eigh(H)
    return w.flip(0)[:nev], V.flip(1)[:, :nev]


def exact(case, seed):
    kind = case["kind"]
    g = _gen(seed)
    if kind == "solve":
        if case["n"] > 4200:
            return None
        A = _matrix(case, g)
        lam, V = _eigh(0.5 * (A - A.T), case["nev"], case["vectors"])
        if V is None:
            return {"lam": lam}
        return {"lam": lam, "z": _fix_phase(V.real.contiguous(), V.imag.contiguous(), _probe(g, case["n"]))}
    if kind == "batch":
        lams, xs, ys = [], [], []
        for A in _batch(case, seed):
            lam, V = _eigh(A, A.shape[0] // 2, True)
            V = V * (V[0].conj() / V[0].abs())
            lams.append(lam)
            xs.append(V.real.T.reshape(-1))
            ys.append(V.imag.T.reshape(-1))
        return {"lam": torch.cat(lams), "z": (torch.cat(xs), torch.cat(ys))}
    if kind == "bse":
        A, B = _blocks(case, g)
        h = case["h"]
        eye = torch.eye(h, dtype=A.dtype, device=A.device)
        P, M = A + B, A - B
        S = torch.cat([torch.cat([P.real, M.imag], 1), torch.cat([-P.imag, M.real], 1)], 0)
        L = torch.linalg.cholesky(S)
        K = L.T @ torch.cat([L[h:], -L[:h]], 0)
        lam, V = _eigh(0.5 * (K - K.T), case["nev"], True)
        X = torch.linalg.solve_triangular(L.T.to(V.dtype), V, upper=True)
        Q = torch.cat([torch.cat([eye, -1j * eye], 1), torch.cat([eye, 1j * eye], 1)], 0) / math.sqrt(2.0)
        psi = (Q @ X) * torch.sqrt(lam)
        return {"lam": lam, "z": _fix_phase(psi.real.contiguous(), psi.imag.contiguous(), _probe(g, 2 * h))}
    A, B = _randn(g, case["m"], case["k"]), _randn(g, case["n"], case["k"])
    return A @ B.T
