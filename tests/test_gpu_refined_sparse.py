"""Very sparse matrices in the refined mode: the tridiagonal falls into many
blocks, some coupled at rounding level only, each odd one with a null vector.

Bounds: those of the other solve tests (1e-12 of the largest eigenvalue,
residual and orthogonality 50 n eps).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


@pytest.mark.parametrize("n,per_row,seed,qtrd", [
    (60, 1, 3, "AUTO"), (60, 1, 32, "AUTO"), (60, 1, 43, "AUTO"), (200, 1, 2, "AUTO"), (200, 1, 3, "AUTO"),
    (200, 1, 24, "AUTO"), (60, 2, 2, "FP32"), (60, 2, 13, "FP64"), (60, 2, 14, "FP32"), (60, 3, 38, "FP64")])
def test_refined_mode_on_very_sparse_matrices(n, per_row, seed, qtrd):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1912_04062_gb300 as sk
    rng = np.random.default_rng(100 * n + seed)
    A = np.tril(rng.standard_normal((n, n)) * (rng.random((n, n)) < per_row / n), -1)
    dA = sk.fortran(torch.from_numpy(np.asfortranarray(A - A.T)).cuda())
    nev = n // 2
    opts = sk.Options(mode=sk.SKEW_MODE_MIXED_REFINED, qtrd=getattr(sk, "SKEW_QTRD_" + qtrd))
    ws = torch.empty(sk.workspace_size(n, nev, opts), dtype=torch.uint8, device="cuda")
    lam = torch.empty(nev, dtype=torch.float64, device="cuda")
    Zr, Zi = sk.fortran_empty(n, nev), sk.fortran_empty(n, nev)
    info = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    assert sk.skew_eig_ex(dA, nev, lam, Zr, Zi, ws, info, opts) == 0
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    r, o, f = sk.metrics(dA, lam, Zr, Zi)
    assert r <= 50 * n * EPS * f and o <= 50 * n * EPS, (r / (n * EPS * f), o / (n * EPS))
    ref = torch.linalg.eigvalsh(torch.complex(torch.zeros_like(dA), -dA)).flip(0)[:nev]
    assert float((lam - ref).abs().max()) <= 1e-12 * float(ref[0])
