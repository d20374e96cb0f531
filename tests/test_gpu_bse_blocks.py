"""The Bethe-Salpeter driver at the edges of its 64-wide blocks (half and whole
warps of a block's entries, one row below a block, one row into the next): the
Cholesky block, the panel and the back substitution split a block's entries
over the two halves of a warp's registers and 8 rows or columns over a CTA.

Bounds: those of the driver's other test (residual 100 (2h) eps, the S-norm to
100 (2h) eps cond).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


@pytest.mark.parametrize("h,nev", [(1, 1), (2, 1), (15, 15), (16, 7), (17, 17), (31, 31), (32, 32), (33, 4),
                                   (47, 47), (49, 49), (65, 1), (95, 95), (97, 97), (161, 161)])
def test_bse_driver_at_block_edges(h, nev):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle.bse as obse
    import paper_1912_04062_gb300 as sk
    rng = np.random.default_rng(900 + h)
    G = rng.standard_normal((h, h)) + 1j * rng.standard_normal((h, h))
    A = np.diag(rng.uniform(2.0, 20.0, h)) + 0.05 * 0.5 * (G + G.conj().T) / np.sqrt(h)
    G = rng.standard_normal((h, h)) + 1j * rng.standard_normal((h, h))
    B = 0.02 * 0.5 * (G + G.T) / np.sqrt(h)
    lam, psi, st = sk.bse_solve(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), nev)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    lam, psi = lam.cpu().numpy(), psi.cpu().numpy()
    H = obse.hamiltonian(A, B)
    n2 = 2 * h
    res = np.linalg.norm(H @ psi - psi * lam, axis=0) / (np.linalg.norm(H, 2) * np.linalg.norm(psi, axis=0))
    assert np.max(res) <= 100 * n2 * EPS
    S = np.concatenate([np.ones(h), -np.ones(h)])[:, None]
    cond = np.linalg.cond(obse.symmetric_m(A, B))
    assert np.max(np.abs(psi.conj().T @ (S * psi) - np.eye(nev))) <= 100 * n2 * EPS * cond
