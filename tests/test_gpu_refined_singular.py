"""The refined mode on matrices with (near-)zero eigenvalues.  Its basis [Z,
conj(Z)] needs vectors of 0 whose real and imaginary parts are of equal norm;
orders of the cluster reduction, of pairs of floats over the whole GPU and of
the lower triangle, and the two-step route (an explicit FP64 Q_trd).

Bounds: those of the other solve tests (1e-12 of the largest eigenvalue,
residual and orthogonality 50 n eps).
"""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


def _matrix(kind, n):
    rng = np.random.default_rng(9700 + n)
    A = inputs.random_skew(n, seed=9700 + n)
    if kind.startswith("zero rows"):
        z = rng.permutation(n)[: int(kind.split()[2])]
        A[z] = 0.0
        A[:, z] = 0.0
    elif kind == "odd blocks":
        h = n // 2 - (1 - (n // 2) % 2)
        A[h:, :h] = 0.0
        A[:h, h:] = 0.0
    elif kind.startswith("deficit"):
        Q = np.linalg.qr(rng.standard_normal((n, n - int(kind.split()[1]))))[0]
        A = Q @ (Q.T @ A @ Q) @ Q.T
        A = 0.5 * (A - A.T)
    elif kind == "graded":
        d = 10.0 ** np.linspace(0.0, -12.0, n)
        A = d[:, None] * A * d
    elif kind == "sparse":
        A = np.tril(A * (rng.random((n, n)) < 3.0 / n), -1)
        A = A - A.T
    return np.asfortranarray(A)


@pytest.mark.parametrize("kind", ["zero rows 2", "zero rows 4", "zero rows 20", "odd blocks", "deficit 2", "deficit 4",
                                  "deficit 40", "graded", "sparse"])
@pytest.mark.parametrize("n,two_step", [(60, False), (150, False), (400, False), (1002, False), (3300, False),
                                        (400, True)])
def test_refined_mode_with_a_null_space(kind, n, two_step):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1912_04062_gb300 as sk
    if n == 3300 and kind in ("graded", "sparse", "deficit 40"):
        pytest.skip("a cluster of hundreds of vectors takes a minute")
    A = _matrix(kind, n)
    nev = n // 2
    opts = sk.Options(mode=sk.SKEW_MODE_MIXED_REFINED, qtrd=sk.SKEW_QTRD_FP64 if two_step else sk.SKEW_QTRD_AUTO)
    dA = sk.fortran(torch.from_numpy(A).cuda())
    ws = torch.empty(sk.workspace_size(n, nev, opts), dtype=torch.uint8, device="cuda")
    lam = torch.empty(nev, dtype=torch.float64, device="cuda")
    Zr, Zi = sk.fortran_empty(n, nev), sk.fortran_empty(n, nev)
    info = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    assert sk.skew_eig_ex(dA, nev, lam, Zr, Zi, ws, info, opts) == 0
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    r, o, f = sk.metrics(dA, lam, Zr, Zi)
    assert r <= 50 * n * EPS * f and o <= 50 * n * EPS, (r / (n * EPS * f), o / (n * EPS))
    H = torch.complex(torch.zeros_like(dA), -dA)
    ref = torch.linalg.eigvalsh(H).flip(0)[:nev]
    assert float((lam - ref).abs().max()) <= 1e-12 * float(ref[0])
