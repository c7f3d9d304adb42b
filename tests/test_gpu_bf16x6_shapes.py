"""BF16X6 contraction at the edges of its tiles, row order and sub-box buffers, against the dense FP64 form.

One column, one tile exactly and one column more on each side, sites on one line (sub-boxes one cell wide or high),
sites spread out (16 instead of 12 cells per slicer thread, the shorter operand ring), one right-hand side and one more
than a group.  The bound is the form's own: six 8-bit slices and products to diagonal 8 leave 2^-47 of the largest
operand product a term, against FP64 sums of the same table and transforms: 1e-12 as for the other sizes.
"""

import numpy as np
import pytest

from conftest import CUBIC, ISO
from paper_2105_08798_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _line(n, x0, vertical):
    t = np.arange(n)
    xy = np.stack([np.full(n, x0), t] if vertical else [t, np.full(n, x0)], axis=1)
    return np.ascontiguousarray(xy, dtype=np.int32)


def _sites(kind, n_i, n_p):
    if kind == "ring":
        return inputs.ring_geometry(n_i, n_p)
    if kind in ("column", "row"):
        return _line(n_i, 0, kind == "column"), _line(n_p, 7, kind == "column")
    xy_i, xy_p = inputs.ring_geometry(n_i, n_p)  # "spread": every second site along x
    return xy_i * np.array([2, 1], np.int32), xy_p * np.array([2, 1], np.int32)


@pytest.mark.parametrize("kind,n_i,n_p,L,R,mat", [
    ("ring", 1, 1, 8, 1, ISO), ("ring", 5, 3, 2, 2, CUBIC), ("ring", 64, 128, 16, 32, ISO), ("ring", 65, 129, 4, 33, CUBIC),
    ("column", 70, 130, 8, 3, ISO), ("row", 70, 130, 8, 3, CUBIC), ("spread", 128, 200, 8, 5, ISO), ("ring", 260, 520, 4, 9, ISO)])
def test_shapes(kind, n_i, n_p, L, R, mat):
    from paper_2105_08798_gb300 import fbc

    xy_i, xy_p = _sites(kind, n_i, n_p)
    f = torch.from_numpy(inputs.forces(R, len(xy_i), L, seed=n_i + R)).cuda()
    out = {}
    with fbc.Plan(xy_i, xy_p, L, mat, precision="bf16x6", max_rhs=R) as plan:
        plan.tabulate()
        info = plan.info()
        if info["sub_w"] * info["sub_h"] > 1880:
            u = torch.zeros((R, len(xy_p), L, 3), dtype=torch.float64, device="cuda")
            with pytest.raises(fbc.FBCError) as e:
                plan.apply(f, u, project=False)
            assert e.value.status == fbc.FBC_ERR_UNSUPPORTED
            return
        for prec in ("bf16x6", "fp64"):
            plan.set_precision(prec)
            u = torch.full((R, len(xy_p), L, 3), float("nan"), dtype=torch.float64, device="cuda")
            plan.apply(f, u, project=False)
            torch.cuda.synchronize()
            plan.sync_status()
            out[prec] = u.cpu().numpy()
    assert np.linalg.norm(out["bf16x6"] - out["fp64"]) <= 1e-12 * np.linalg.norm(out["fp64"])
