"""The direct (one-step) reduction with its back-transformation, and the twisted
eigenvectors of the tridiagonal, at the sizes where their tiling changes.

Orders around one row per CTA of a thread-block cluster and around the largest
that a cluster takes, around a panel of 64 reflectors, around one, two and
three rows per CTA of a 152-SM GPU, the first one whose rows do not all fit shared memory, and the
first ones of the lower-triangle form (whole and ragged blocks of 64); slabs of
one to six eigenvectors per CTA.  The two-step route (an explicit FP64 Q_trd) is
the other side of the comparison.  Bounds: those of the other solve
tests (1e-12 of the largest eigenvalue; residual and orthogonality 50 n eps).
"""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


@pytest.fixture(scope="module", autouse=True)
def _dev():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _solve(dA, nev, opts, vectors=True):
    import torch
    import paper_1912_04062_gb300 as sk
    n = dA.shape[0]
    ws = torch.empty(sk.workspace_size(n, nev, opts, vectors=vectors), dtype=torch.uint8, device="cuda")
    lam = torch.empty(nev, dtype=torch.float64, device="cuda")
    Zr = sk.fortran_empty(n, nev) if vectors else None
    Zi = sk.fortran_empty(n, nev) if vectors else None
    info = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    assert sk.skew_eig_ex(dA, nev, lam, Zr, Zi, ws, info, opts) == 0
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    return lam, Zr, Zi


@pytest.mark.parametrize("n,nev", [(2, 1), (3, 1), (15, 7), (16, 8), (17, 8), (33, 1), (49, 24), (65, 32), (66, 33),
                                   (67, 1), (130, 65), (152, 3), (153, 76), (220, 110), (221, 110), (305, 152),
                                   (306, 153), (459, 20), (610, 305), (914, 457), (1825, 912), (1826, 40), (3001, 50),
                                   (3072, 33), (3137, 1568)])
def test_direct_route_matches_two_step(n, nev):
    import torch
    import paper_1912_04062_gb300 as sk
    A = inputs.random_skew(n, seed=7000 + n)
    dA = sk.fortran(torch.from_numpy(A).cuda())
    lam2, _, _ = _solve(dA, nev, sk.Options(qtrd=sk.SKEW_QTRD_FP64))
    scale = float(lam2[0])
    lam1, Zr, Zi = _solve(dA, nev, sk.Options())
    assert float((lam1 - lam2).abs().max()) <= 1e-12 * scale
    r, o, f = sk.metrics(dA, lam1, Zr, Zi)
    assert r <= 50 * n * EPS * f and o <= 50 * n * EPS
    # values only, and a second run, give the same bits
    lam0, _, _ = _solve(dA, nev, sk.Options(), vectors=False)
    assert torch.equal(lam0, lam1)
    lam3, Zr3, Zi3 = _solve(dA, nev, sk.Options())
    assert torch.equal(lam3, lam1) and torch.equal(Zr3, Zr) and torch.equal(Zi3, Zi)


@pytest.mark.parametrize("n,scale,tiny", [(2, 1.0, 1.0), (4, 1.0, 1.0), (64, 1.0, 1.0), (220, 1.0, 1.0),
                                          (222, 1.0, 1.0), (130, 1e-120, 1.0),
                                          (306, 1e100, 1.0), (308, 1.0, 1e-5), (308, 1.0, 1e-8), (1002, 1.0, 1.0),
                                          (2070, 1.0, 1.0), (3202, 1e-40, 1.0), (3264, 1.0, 1e-5),
                                          (3266, 1.0, 1.0)])
def test_direct_route_refined_is_orthogonal(n, scale, tiny):
    # the double-float reduction and one refinement iteration have to leave
    # the orthogonality of a converged refinement (not the square of the
    # starting vectors' norm error), for any scaling of the matrix and with a
    # block far below its largest entries
    import torch
    import paper_1912_04062_gb300 as sk
    A = inputs.random_skew(n, seed=7100 + n) * scale
    if tiny != 1.0:
        h = n // 2
        A[h:, :h] = 0.0
        A[:h, h:] = 0.0
        A[h:, h:] *= tiny
    dA = sk.fortran(torch.from_numpy(np.asfortranarray(A)).cuda())
    lam, Zr, Zi = _solve(dA, n // 2, sk.Options(mode=sk.SKEW_MODE_MIXED_REFINED))
    r, o, f = sk.metrics(dA / scale, lam / scale, Zr, Zi)
    assert r <= 50 * n * EPS * f and o <= 5 * n * EPS


@pytest.mark.parametrize("glue", [1e-3, 1e-6, 1e-9, 1e-13])
@pytest.mark.parametrize("n", [62, 511])
def test_twisted_vectors_of_glued_blocks(n, glue):
    # equal blocks coupled by `glue`: pairs of eigenvalues about glue apart, so
    # loose clusters (one Gram-Schmidt pass) and tight ones (iterated)
    import torch
    import paper_1912_04062_gb300 as sk
    rng = np.random.default_rng(n)
    h = (n - 1) // 2
    half = rng.uniform(0.5, 2.0, h)
    a = np.concatenate([half, [glue], half[::-1]])[: n - 1]
    a = np.concatenate([a, rng.uniform(0.5, 2.0, n - 1 - a.size)])
    nev = n // 2
    da = torch.from_numpy(a).cuda()
    lam, Q, st = sk.tridiag_eig(da, nev)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    S = torch.diag(da, 1) + torch.diag(da, -1)
    scale = float(lam[0])
    assert float((S @ Q - Q * lam).norm(dim=0).max()) <= 50 * n * EPS * scale
    assert float((Q.T @ Q - torch.eye(nev, device="cuda", dtype=Q.dtype)).norm()) <= 50 * n * EPS


def test_batch_results_do_not_depend_on_the_cluster_size():
    # orders around the one-CTA limit, around the changes of the pass's column
    # split (72, 144 and 288 rows left) and around shared memory; alone (large
    # clusters) and in a long batch (small ones) they give the same bits
    import torch
    import paper_1912_04062_gb300 as sk
    sizes = [96, 97, 98, 145, 146, 289, 290, 500, 777, 1024]
    mats = [sk.fortran(torch.from_numpy(inputs.random_skew(n, seed=7300 + n)).cuda()) for n in sizes]
    nevs = [n // 2 if n != 500 else 33 for n in sizes]
    lam, Zr, Zi, info = sk.skew_eig_batched(mats * 12, nevs * 12, info=True)
    torch.cuda.synchronize()
    assert int(info.abs().max()) == 0
    for i, (A, nev) in enumerate(zip(mats, nevs)):
        l1, zr1, zi1 = (v[0] for v in sk.skew_eig_batched([A], [nev]))
        torch.cuda.synchronize()
        for j in (i, i + 11 * len(sizes)):
            assert torch.equal(l1, lam[j]) and torch.equal(zr1, Zr[j]) and torch.equal(zi1, Zi[j])
        n = A.shape[0]
        r, o, f = sk.metrics(A, l1, zr1, zi1)
        assert r <= 50 * n * EPS * f and o <= 50 * n * EPS
        ref, _, _ = _solve(A, nev, sk.Options(), vectors=False)
        assert float((ref - l1).abs().max()) <= 1e-12 * float(ref[0])
