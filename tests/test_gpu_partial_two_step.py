"""Partial vectors of the refined mode above order 4750: band reduction, chase
and double-float Q_trd (below it the direct reduction takes them), and the
direct reduction's lower triangle where it is cut into more blocks of 32 than
there are SMs (order 4865 and above on 152), in both arithmetics.

The FP64 form of the same problem (direct reduction) is the other side.  Bounds:
those of the other solve tests (1e-12 of the largest eigenvalue, residual and
orthogonality 50 n eps).
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


def _matrix(n):
    import torch
    import paper_1912_04062_gb300 as sk
    return sk.fortran(torch.from_numpy(np.asfortranarray(inputs.random_skew(n, seed=9600 + n))).cuda())


def _solve(dA, nev, kinds=None, **kw):
    import torch
    import paper_1912_04062_gb300 as sk
    n = dA.shape[0]
    opts = sk.Options(**kw)
    ws = torch.empty(sk.workspace_size(n, nev, opts), dtype=torch.uint8, device="cuda")
    lam = torch.empty(nev, dtype=torch.float64, device="cuda")
    Zr, Zi = sk.fortran_empty(n, nev), sk.fortran_empty(n, nev)
    if kinds is None:
        info = torch.full((1,), -1, dtype=torch.int32, device="cuda")
        assert sk.skew_eig_ex(dA, nev, lam, Zr, Zi, ws, info, opts) == 0
        torch.cuda.synchronize()
        assert int(info.item()) == 0
    else:
        sk.kernel_timing(True)
        assert sk.skew_eig_profile(dA, nev, lam, Zr, Zi, ws, opts)[0] == 0
        kinds.update({k: sk.kernel_timing_read(i)[2] for i, k in enumerate(sk.KERNEL_KINDS)})
        sk.kernel_timing(False)
    r, o, f = sk.metrics(dA, lam, Zr, Zi)
    assert r <= 50 * n * EPS * f and o <= 50 * n * EPS, (r / (n * EPS * f), o / (n * EPS))
    return lam, Zr, Zi


@pytest.mark.parametrize("n,nev", [(4751, 7), (4752, 300), (5001, 120)])
def test_partial_vectors_by_the_two_step_route(n, nev):
    import torch
    import paper_1912_04062_gb300 as sk
    dA = _matrix(n)
    kinds = {}
    lam, Zr, Zi = _solve(dA, nev, kinds, mode=sk.SKEW_MODE_MIXED_REFINED)
    assert kinds["qtrd"] > 0 and kinds["chase"] > 0, kinds
    direct = {}
    ref, Xr, Xi = _solve(dA, nev, direct)
    assert direct["qtrd"] == 0 and direct["chase"] == 0, direct
    assert float((lam - ref).abs().max()) <= 1e-12 * float(ref[0])
    # naming the mode's own arithmetic changes nothing
    for a, b in zip((lam, Zr, Zi), _solve(dA, nev, mode=sk.SKEW_MODE_MIXED_REFINED, qtrd=sk.SKEW_QTRD_DF)):
        assert torch.equal(a, b)


@pytest.mark.parametrize("n", [4865, 4930])
def test_triangle_with_more_blocks_than_sms(n):
    import paper_1912_04062_gb300 as sk
    nev = 40
    dA = _matrix(n)
    lam, _, _ = _solve(dA, nev)
    ref, _, _ = _solve(dA, nev, qtrd=sk.SKEW_QTRD_FP64)
    assert float((lam - ref).abs().max()) <= 1e-12 * float(ref[0])
    if n % 2 == 0:
        it = _solve(dA, n // 2, mode=sk.SKEW_MODE_MIXED_REFINED)[0]
        assert float((it[:nev] - ref).abs().max()) <= 1e-12 * float(ref[0])
