"""Relaxed update over the column splits of the line transforms (two columns a block up to the shape's full width), with
and without the cap (a capped one updates from the kept inverse transform) and the zero mean, against the oracle at the
FP64 forms' 1e-12.
"""

import numpy as np
import pytest

from conftest import ISO
from paper_2105_08798_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "f32x2"])
@pytest.mark.parametrize("n_i,n_p,L,R", [(1, 2, 2, 1), (3, 1, 32, 2), (129, 65, 4, 1), (40, 257, 8, 3), (260, 700, 16, 5),
                                         (150, 130, 2, 32)])
def test_relaxed_shapes(oracle_mod, precision, n_i, n_p, L, R):
    from paper_2105_08798_gb300 import fbc

    xy_i, xy_p = inputs.ring_geometry(n_i, n_p)
    f_old = inputs.forces(R, n_i, L, seed=n_i)
    f_new = 0.6 * f_old + 0.3 * inputs.forces(R, n_i, L, seed=n_i + 1)
    u0 = np.random.default_rng(n_p).normal(0, 1, (R, n_p, L, 3))
    alpha0 = np.linspace(0.5, 2.0, R)
    with fbc.Plan(xy_i, xy_p, L, ISO, precision=precision, max_rhs=R) as plan:
        plan.tabulate()
        for du_max, zero_mean in ((0.0, True), (1e-2, False), (0.3, True)):
            ref_u, ref_a = oracle_mod.relaxed_update(xy_i, xy_p, L, 1.0, ISO, f_new, f_old, u0, alpha0, du_max=du_max,
                                                     zero_mean_u=zero_mean)
            fn, fo, u = (torch.from_numpy(x.copy()).cuda() for x in (f_new, f_old, u0))
            a = torch.from_numpy(alpha0).cuda()
            plan.apply_relaxed(fn, fo, u, a, du_max=du_max, zero_mean=zero_mean)
            torch.cuda.synchronize()
            plan.sync_status()
            np.testing.assert_allclose(a.cpu().numpy(), ref_a, rtol=1e-12)
            assert np.linalg.norm(u.cpu().numpy() - ref_u) <= 1e-12 * np.linalg.norm(ref_u)
