"""Plans of different launch configurations that live at the same time: one
plan's creation, tuning or threshold takes nothing from another's launches, and
the results keep their bits."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


def _mats(sizes):
    import torch
    import paper_1912_04062_gb300 as sk
    return [sk.fortran(torch.from_numpy(inputs.random_skew(n, seed=9400 + n)).cuda()) for n in sizes]


@pytest.mark.parametrize("ctas", [1, 2, 3, 4])
def test_plans_of_different_thresholds_alternate(ctas):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1912_04062_gb300 as sk
    sizes = [2, 48, 64, 65, 90, 95, 96, 97]
    mats, nevs = _mats(sizes), [n // 2 for n in sizes]
    plans = [sk.BatchedPlan(mats, nevs, config=(ctas, s)) for s in (112, 0, 48, 160)]
    plans.append(sk.BatchedPlan(_mats([2, 3]), [1, 1], config=(ctas, 112)))
    ref = None
    for rep in range(2):
        for plan in plans[:4]:
            plan.execute()
            torch.cuda.synchronize()
            assert np.all(plan.info[: len(mats)].cpu().numpy() == 0)
            got = [v.clone() for part in plan.results() for v in part]
            ref = got if ref is None else ref
            assert all(torch.equal(a, b) for a, b in zip(ref, got))
        plans[4].execute()
        torch.cuda.synchronize()


def test_tuning_a_plan_without_small_orders():
    # nothing to choose but the number of CTAs, which the launch does not use
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1912_04062_gb300 as sk
    sizes = [97, 120]
    mats, nevs = _mats(sizes), [40, 60]
    plan = sk.BatchedPlan(mats, nevs, config=(2, 112))
    plan.execute()
    torch.cuda.synchronize()
    ref = [v.clone() for part in plan.results() for v in part]
    best, cands = plan.tune()
    assert best in [(c, s) for c, s, _ in cands] and all(s == 0 for _, s, _ in cands)
    plan.execute()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(ref, [v for part in plan.results() for v in part]))
