"""A block far below the resolution of the eigenvalues (a decoupled block of
order 1e-140, 1e-150 beside one of order 1): its eigenvalues come out equal, its
vectors are iterated with one shift, and at odd size the same direction
outgrows all others in every one of them.  They still have to be orthonormal.

Bounds: those of the other solve tests (1e-12 of the largest eigenvalue,
residual and orthogonality 50 n eps).
"""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,h", [(40, 20), (97, 48), (100, 51), (131, 64), (301, 150)])
@pytest.mark.parametrize("t", [1e-140, 1e-150])
def test_vectors_of_a_block_below_resolution(n, h, t):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    import paper_1912_04062_gb300 as sk
    A = np.zeros((n, n))
    A[:h, :h] = inputs.random_skew(h, seed=9300 + n)
    A[h:, h:] = inputs.random_skew(n - h, seed=9301 + n) * t
    nev = n // 2
    ref = np.zeros(nev)
    ref[: h // 2] = np.sort(np.linalg.eigvalsh(1j * A[:h, :h]))[::-1][: h // 2]
    dA = sk.fortran(torch.from_numpy(np.asfortranarray(A)).cuda())
    lam, Zr, Zi = sk.skew_eig(dA, nev)
    lb, zrb, zib, info = sk.skew_eig_batched([dA], [nev], info=True)
    torch.cuda.synchronize()
    assert int(info.abs().max()) == 0
    for l, x, y in ((lam, Zr, Zi), (lb[0], zrb[0], zib[0])):
        m = oracle.scaled_metrics(A, l.cpu().numpy(), x.cpu().numpy(), y.cpu().numpy(), lam_ref=ref,
                                  norm2=float(ref[0]))
        assert m["eig_err"] <= 1e-12 and m["resid"] <= 50 and m["orth"] <= 50, m
