"""Kernel tables of several plans tabulated at the same time on streams of their own, from one thread and from several.

Each plan has its own medium, box, period and node count: every table has to come out with the bits it has alone.
"""

import threading

import numpy as np
import pytest

from conftest import CUBIC, ISO
from paper_2105_08798_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PLANS = [(200, 300, 64, CUBIC, "fp64", 64), (90, 130, 16, ISO, "f32x2", 64), (150, 170, 32, dict(CUBIC, C44=0.3), "fp32", 40),
         (120, 260, 128, dict(CUBIC, C12=0.7), "fp64", 96)]


@pytest.mark.parametrize("threads", [False, True])
def test_tables_of_their_own(threads):
    from paper_2105_08798_gb300 import fbc

    plans, diffs, want = [], [], []
    for n_i, n_p, L, material, precision, quad in PLANS:
        xy_i, xy_p = inputs.ring_geometry(n_i, n_p)
        plans.append(fbc.Plan(xy_i, xy_p, L, material, precision=precision, quad=quad))
        diffs.append(np.unique((xy_p[::7, None, :] - xy_i[None, ::5, :]).reshape(-1, 2), axis=0).astype(np.int32))
        plans[-1].tabulate()
        torch.cuda.synchronize()
        want.append(plans[-1].mode_table(diffs[-1]))
    streams = [torch.cuda.Stream() for _ in plans]

    def work(some):
        for _ in range(4):
            for j in some:
                plans[j].tabulate(stream=streams[j])

    if threads:
        ts = [threading.Thread(target=work, args=([j],)) for j in range(len(plans))]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
    else:
        work(range(len(plans)))
    torch.cuda.synchronize()
    for p, d, w in zip(plans, diffs, want):
        np.testing.assert_array_equal(p.mode_table(d), w)
        p.close()
