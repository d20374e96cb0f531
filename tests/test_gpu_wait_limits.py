"""Waits between CTAs that run out (SKEW_FAULT_TINY_WAIT: one poll), on each
reduction that has such waits: band reduction and chase, the pairs of floats over
the whole GPU, the lower triangle.  (The FP64 rows over the whole GPU:
test_gpu_parity.)  The kernels record SKEW_ERR_DEVICE_TIMEOUT and return, the
later ones run on what there is, and a solve with the usual limits in the same
workspace is right."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("route,n,nev", [("two-step", 400, 200), ("pairs", 400, 200), ("triangle", 3001, 10)])
def test_waits_run_out_and_the_context_survives(route, n, nev):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1912_04062_gb300 as sk
    kw = {"two-step": {"qtrd": sk.SKEW_QTRD_FP64}, "pairs": {"mode": sk.SKEW_MODE_MIXED_REFINED, "refine_iters": 1},
          "triangle": {}}[route]
    A = inputs.random_skew(n, seed=9500 + n)
    dA = sk.fortran(torch.from_numpy(np.asfortranarray(A)).cuda())
    ws = torch.zeros(sk.workspace_size(n, nev, sk.Options(**kw)), dtype=torch.uint8, device="cuda")
    lam = torch.empty(nev, dtype=torch.float64, device="cuda")
    Zr, Zi = sk.fortran_empty(n, nev), sk.fortran_empty(n, nev)
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    assert sk.skew_eig_ex(dA, nev, lam, Zr, Zi, ws, info, sk.Options(fault=sk.SKEW_FAULT_TINY_WAIT, **kw)) == 0
    torch.cuda.synchronize()
    assert int(info.item()) == sk.SKEW_ERR_DEVICE_TIMEOUT
    assert sk.skew_eig_ex(dA, nev, lam, Zr, Zi, ws, info, sk.Options(**kw)) == 0
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    r, o, f = sk.metrics(dA, lam, Zr, Zi)
    eps = np.finfo(np.float64).eps
    assert r <= 50 * n * eps * f and o <= 50 * n * eps
