"""FP64 solves, single and batched, of very sparse matrices: the tridiagonal falls
into many blocks, and couplings at rounding level let one vector of a cluster
outgrow all others by more than FP64 carries.

Bounds: those of the other solve tests (1e-12 of the largest eigenvalue,
residual and orthogonality 50 n eps).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


@pytest.mark.parametrize("n,per_row,seeds", [(40, 1, [0, 1, 2, 4, 5]), (40, 2, [9, 12]), (150, 1, [2, 4, 29]),
                                             (230, 1, [0, 1, 22]), (400, 1, [1, 6, 23])])
def test_very_sparse_matrices(n, per_row, seeds):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1912_04062_gb300 as sk
    mats = []
    for seed in seeds:
        rng = np.random.default_rng(1000 * n + seed)
        A = np.tril(rng.standard_normal((n, n)) * (rng.random((n, n)) < per_row / n), -1)
        mats.append(sk.fortran(torch.from_numpy(np.asfortranarray(A - A.T)).cuda()))
    nev = n // 2
    lam, Zr, Zi, info = sk.skew_eig_batched(mats, [nev] * len(mats), info=True)
    torch.cuda.synchronize()
    assert int(info.abs().max()) == 0
    for A, l, x, y in zip(mats, lam, Zr, Zi):
        ref = torch.linalg.eigvalsh(torch.complex(torch.zeros_like(A), -A)).flip(0)[:nev]
        for v in ((l, x, y), sk.skew_eig(A, nev)):
            r, o, f = sk.metrics(A, *v)
            assert r <= 50 * n * EPS * f and o <= 50 * n * EPS, (r / (n * EPS * f), o / (n * EPS))
            assert float((v[0] - ref).abs().max()) <= 1e-12 * float(ref[0])
