"""Tensor-core contractions whose pipeline waits give up at different places: every way of staging a sub-box, alone and in
a batch's queue.  An apply either completes with its usual bits or reports the timeout, and the next one with the default
bound is right again.  (No wait is ever left without an end: each is short here, and the kernel stops as a whole.)
"""

import pytest

from conftest import ISO
from paper_2105_08798_gb300 import inputs
from test_gpu_tensor_shapes import _sites

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [("ring", 200, 300, 1, 8, 9), ("line", 70, 130, 16, 4, 3), ("line", 70, 130, 20, 4, 17)]
LIMITS = (1, 2, 3, 5, 9, 20)


def _plan(fbc, shape, precision):
    kind, n_i, n_p, step, L, R = shape
    xy_i, xy_p = _sites(kind, n_i, n_p, step)
    plan = fbc.Plan(xy_i, xy_p, L, ISO, precision=precision, max_rhs=R)
    plan.tabulate()
    f = torch.from_numpy(inputs.forces(R, len(xy_i), L, seed=len(xy_p))).cuda()
    return plan, f, torch.zeros((R, len(xy_p), L, 3), dtype=torch.float64, device="cuda")


def _stopped(fbc, plan):
    torch.cuda.synchronize()
    try:
        plan.sync_status()
    except fbc.FBCError as e:
        assert e.status == fbc.FBC_ERR_TIMEOUT
        return True
    return False


@pytest.mark.parametrize("precision", ["tf32", "bf16x2", "bf16x3"])
@pytest.mark.parametrize("shape", SHAPES)
def test_apply(precision, shape):
    from paper_2105_08798_gb300 import fbc

    plan, f, want = _plan(fbc, shape, precision)
    with plan:
        plan.apply(f, want, project=False)
        stops = 0
        for limit in LIMITS:
            u = torch.empty_like(want)
            plan.set_wait_limit(limit)
            plan.apply(f, u, project=False)
            stopped = _stopped(fbc, plan)
            assert stopped or torch.equal(u, want)
            stops += stopped
            plan.set_wait_limit(0)
            plan.apply(f, u, project=False)
            assert not _stopped(fbc, plan) and torch.equal(u, want)
        assert stops > 0


@pytest.mark.parametrize("precision", ["tf32", "bf16x2", "bf16x3"])
def test_queue(precision):
    from paper_2105_08798_gb300 import fbc

    plans, fs, want = zip(*(_plan(fbc, s, precision) for s in SHAPES))
    for p, f, u in zip(plans, fs, want):
        p.apply(f, u, project=False)
    us = [torch.empty_like(u) for u in want]
    with fbc.Batch(list(plans), list(fs), us) as b:
        for limit in LIMITS:
            plans[0].set_wait_limit(limit)  # (a batch's launch takes its first plan's bound and status word)
            b.apply(project=False, graph=False)
            assert _stopped(fbc, plans[0]) or all(torch.equal(u, v) for u, v in zip(us, want))
            plans[0].set_wait_limit(0)
            b.apply(project=False, graph=False)
            assert not _stopped(fbc, plans[0]) and all(torch.equal(u, v) for u, v in zip(us, want))
    for p in plans:
        p.close()
