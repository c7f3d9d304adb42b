"""In-plane FP64 FFT form over its butterflies, against the oracle's real-space sum at the form's 1e-12: grid lengths with
first passes of radix 2, 3, 5, 6 and 8, sites on one line along x or y (a grid of two points the other way), and interface
sites beyond the grid's lower half (a pad inside them: nothing may be left out of the first pass).
"""

import numpy as np
import pytest

from conftest import CUBIC
from paper_2105_08798_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _line(n, x0, step, along):
    t = x0 + step * np.arange(n)
    return np.ascontiguousarray(np.stack([t, 0 * t] if along == "x" else [0 * t, t], axis=1), dtype=np.int32)


@pytest.mark.parametrize("along", ["x", "y"])
@pytest.mark.parametrize("n_i,n_p,step", [(1, 1, 1), (2, 2, 1), (3, 4, 1), (5, 4, 1), (10, 8, 1), (12, 20, 1), (25, 8, 1),
                                          (40, 30, 2), (60, 90, 3), (7, 1, 40)])
def test_lines(oracle_mod, along, n_i, n_p, step):
    from paper_2105_08798_gb300 import fbc

    L, R = 4, 2
    xy_p = _line(n_p, 0, step, along)
    for x0 in (n_p * step, -(n_i // 2) * step):  # beside the pad; around it
        xy_i = _line(n_i, x0, step, along)
        xy_i = xy_i[~(xy_i[:, None] == xy_p[None]).all(-1).any(1)]
        if not len(xy_i):
            continue
        f = inputs.forces(R, len(xy_i), L, seed=n_i)
        ref = oracle_mod.pad_update(xy_i, xy_p, L, 1.0, CUBIC, f, project=False, nquad=64)
        with fbc.Plan(xy_i, xy_p, L, CUBIC, precision="fft64", max_rhs=R) as plan:
            plan.tabulate()
            u = torch.full((R, n_p, L, 3), float("nan"), dtype=torch.float64, device="cuda")
            plan.apply(torch.from_numpy(f).cuda(), u, project=False)
            torch.cuda.synchronize()
            plan.sync_status()
        assert np.linalg.norm(u.cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref)
