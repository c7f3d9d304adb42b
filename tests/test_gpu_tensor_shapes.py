"""Tensor-core contractions over their operand and table buffers, against the dense FP64 form at the forms' own bounds.

One to four operand buffers in tensor memory (by the rows of the force operand, 16 to 128), more than one rhs group with
a part-filled last one, table rows an even and odd number of entries apart, and every way of staging a sub-box: two
buffers or one, rows by bulk copies or (sites far apart along one line, where the rows' padding is what no longer fits)
copied by the warps that read them.
"""

import numpy as np
import pytest

from conftest import CUBIC, ISO
from paper_2105_08798_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BOUNDS = {"tf32": 5e-3, "bf16x2": 1e-4, "bf16x3": 1e-5}


def _sites(kind, n_i, n_p, step):
    if kind != "line":
        xy_i, xy_p = inputs.ring_geometry(n_i, n_p)
        if kind == "cut":  # an even number of differences along x
            xy_p = xy_p[xy_p[:, 0] > xy_p[:, 0].min()]
        return xy_i * np.array([step, 1], np.int32), xy_p * np.array([step, 1], np.int32)

    def line(n, x):
        return np.ascontiguousarray(np.stack([np.full(n, x), step * np.arange(n)], axis=1), dtype=np.int32)

    return line(n_i, 0), line(n_p, 7)


@pytest.mark.parametrize("kind,n_i,n_p,step,L,R,mat", [
    ("ring", 1, 1, 1, 4, 1, ISO), ("ring", 64, 128, 1, 8, 9, CUBIC), ("ring", 65, 129, 1, 4, 24, ISO), ("ring", 90, 140, 2, 4, 33, ISO),
    ("ring", 70, 300, 3, 4, 41, CUBIC), ("ring", 130, 150, 1, 4, 49, ISO), ("ring", 129, 257, 1, 4, 64, ISO),
    ("ring", 200, 150, 2, 8, 73, CUBIC), ("line", 70, 130, 1, 4, 3, ISO), ("line", 70, 130, 16, 4, 3, ISO),
    ("line", 70, 130, 20, 4, 17, ISO), ("line", 129, 260, 24, 4, 3, ISO), ("cut", 100, 180, 1, 8, 5, ISO)])
def test_shapes(kind, n_i, n_p, step, L, R, mat):
    from paper_2105_08798_gb300 import fbc

    xy_i, xy_p = _sites(kind, n_i, n_p, step)
    n_p = len(xy_p)
    f = torch.from_numpy(inputs.forces(R, n_i, L, seed=n_i + R)).cuda()
    with fbc.Plan(xy_i, xy_p, L, mat, max_rhs=R) as plan:
        plan.tabulate()
        out = {}
        for precision in ("fp64", *BOUNDS):
            plan.set_precision(precision)
            for r in {R, max(1, R - 1)}:
                u = torch.full((r, n_p, L, 3), float("nan"), dtype=torch.float64, device="cuda")
                try:
                    plan.apply(f[:r].contiguous(), u, project=False)
                except fbc.FBCError as e:  # a sub-box too large for this form's shared memory
                    assert precision != "fp64" and "shared memory" in str(e), e
                    continue
                torch.cuda.synchronize()
                plan.sync_status()
                out[precision, r] = u.cpu().numpy()
        for (precision, r), u in out.items():
            if precision != "fp64":
                ref = out["fp64", r]
                assert np.linalg.norm(u - ref) <= BOUNDS[precision] * np.linalg.norm(ref), (precision, r)
        assert ("bf16x2", R) in out
