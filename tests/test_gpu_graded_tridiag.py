"""Tridiagonals with couplings from 1 down to 1e-300, exact zeros among them:
eigenvalues far below the norm, twisted vectors whose ratios overflow or whose
polishing solve grows without bound.  Every vector is a unit vector of small
residual, orthogonal to the others, and the status is 0.

Bounds: those of the other tridiagonal tests (residual 50 n eps ||S||,
orthogonality 50 n eps).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps

A1, A2 = 1.3150339753870934, 0.64556247  # an eigenvalue equal to a coupling, to the bit


@pytest.mark.parametrize("alpha,nev", [
    ([1e-120, 1e-30, 1, 1e-60], 2),
    ([1e-300, 1e-240, 1e-30, 1, 1e-60], 2),
    ([1e-90, 1e-90, 1e-270, 1e-30, 1, 1e-60], 2),
    ([1e-120, 0, 1e-30, 0, 1e-120, 1e-30, 1, 1e-60], 3),
    ([1e-30 * A1, A1, 1e-30 * A1, 1e-60, 1e-60, 1e-60, 1e-30 * A1, 1e-60, 1e-30 * A1], 2),
    ([1e-30 * A1, A1, 1e-30 * A1, 1e-60, 1e-60, 1e-60, 1e-30 * A1, 1e-60, 1e-30 * A1], 5),
    ([1e-60, A2, 1e-30, A2, A2, A2, A2], 2),
    ([0, 1, 0, 0, 2, 1e-100, 0, 3], 4),
])
def test_vectors_of_graded_couplings(alpha, nev):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1912_04062_gb300 as sk
    a = np.array(alpha, dtype=np.float64)
    n = a.size + 1
    lam, Q, st = sk.tridiag_eig(torch.from_numpy(a).cuda(), nev)
    torch.cuda.synchronize()
    lam, Q = lam.cpu().numpy(), Q.cpu().numpy()
    S = np.diag(a, 1) + np.diag(a, -1)
    ref = np.linalg.eigvalsh(S)[::-1][:nev]
    assert int(st.item()) == 0
    assert np.max(np.abs(lam - ref)) <= 1e-12 * ref[0]
    assert np.max(np.linalg.norm(S @ Q - Q * lam, axis=0)) <= 50 * n * EPS * ref[0]
    assert np.linalg.norm(Q.T @ Q - np.eye(nev)) <= 50 * n * EPS
