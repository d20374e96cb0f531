"""Columns whose squares leave the double range, in the FP64 direct reductions.

A reflector's sigma = 2 / |u|^2 exceeds the double range below a column norm of
7.5e-155 and vanishes above 9.5e153.  Matrices at such scales, and a block of
order one beside a decoupled one far below it (whose columns the reduction meets
last): orders of a cluster, of rows over the whole GPU, of the lower triangle
and of a batch.

Bounds: those of the other solve tests (1e-12 of the largest eigenvalue,
residual and orthogonality 50 n eps).
"""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _dev():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _blocks(n, h, t):
    A = np.zeros((n, n))
    A[:h, :h] = inputs.random_skew(h, seed=9000 + n)
    A[h:, h:] = inputs.random_skew(n - h, seed=9001 + n) * t
    return A


def _ref(B, nev):
    return np.sort(np.linalg.eigvalsh(1j * B))[::-1][:nev]


def _solve(A, nev, **opts):
    import torch
    import paper_1912_04062_gb300 as sk
    n = A.shape[0]
    o = sk.Options(**opts)
    dA = sk.fortran(torch.from_numpy(np.asfortranarray(A)).cuda())
    ws = torch.empty(sk.workspace_size(n, nev, o), dtype=torch.uint8, device="cuda")
    lam = torch.empty(nev, dtype=torch.float64, device="cuda")
    Zr, Zi = sk.fortran_empty(n, nev), sk.fortran_empty(n, nev)
    info = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    assert sk.skew_eig_ex(dA, nev, lam, Zr, Zi, ws, info, o) == 0
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    return lam.cpu().numpy(), Zr.cpu().numpy(), Zi.cpu().numpy()


def _check(A, ref, lam, X, Y):
    import oracle
    m = oracle.scaled_metrics(A, lam, X, Y, lam_ref=ref, norm2=float(ref[0]))
    assert m["eig_err"] <= 1e-12 and m["resid"] <= 50 and m["orth"] <= 50, m


@pytest.mark.parametrize("n", [40, 300, 301, 3002])
@pytest.mark.parametrize("scale", [1e-155, 1e-152, 1e152])
def test_whole_matrix_at_an_extreme_scale(n, scale):
    A = inputs.random_skew(n, seed=9100 + n)
    nev = n // 2 if n < 1000 else 60
    lam, X, Y = _solve(A * scale, nev)
    _check(A, _ref(A, nev), lam / scale, X, Y)


def test_column_norms_just_below_the_square_root_of_the_range():
    # beta (x_0 - beta) overflows although the squares' sum does not: the
    # longest column first, its largest entry leading
    n, nev = 40, 20
    A = inputs.random_skew(n, seed=9200)
    c = int(np.argmax(np.linalg.norm(A, axis=0)))
    r = int(np.argmax(np.abs(A[:, c])))
    order = [c, r] + [i for i in range(n) if i not in (c, r)]
    A = A[np.ix_(order, order)]
    scale = 1.3e154 / np.linalg.norm(A[:, 0])
    b = np.linalg.norm(A[:, 0]) * scale
    with np.errstate(over="ignore"):
        assert np.isfinite(b * b) and np.isinf(b * (b + abs(A[1, 0]) * scale))
    lam, X, Y = _solve(A * scale, nev)
    _check(A, _ref(A, nev), lam / scale, X, Y)


@pytest.mark.parametrize("n", [40, 97, 300, 301, 3002])
@pytest.mark.parametrize("t", [1e-155, 1e-158, 1e-160])
def test_vectors_beside_a_tiny_block(n, t):
    h = n // 2
    nev = h // 2 if n < 1000 else 60
    A = _blocks(n, h, t)
    ref = _ref(A[:h, :h], nev)
    _check(A, ref, *_solve(A, nev))
    if n == 300:
        import paper_1912_04062_gb300 as sk
        _check(A, ref, *_solve(A, nev, mode=sk.SKEW_MODE_MIXED_REFINED))


@pytest.mark.parametrize("t", [1e-155, 1e-160])
def test_batch_beside_tiny_blocks(t):
    import torch
    import paper_1912_04062_gb300 as sk
    sizes = [97, 150, 301, 600]
    mats = [_blocks(n, n // 2, t) for n in sizes]
    nevs = [n // 4 for n in sizes]
    d = [sk.fortran(torch.from_numpy(np.asfortranarray(A)).cuda()) for A in mats]
    lam, Zr, Zi, info = sk.skew_eig_batched(d, nevs, info=True)
    torch.cuda.synchronize()
    assert int(info.abs().max()) == 0
    for A, nev, l, zr, zi in zip(mats, nevs, lam, Zr, Zi):
        h = A.shape[0] // 2
        _check(A, _ref(A[:h, :h], nev), l.cpu().numpy(), zr.cpu().numpy(), zi.cpu().numpy())
