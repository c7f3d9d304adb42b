"""Host-memory applies of the tensor-core forms whose last right-hand-side group is part filled (it goes first, in a
chunk of its own): bit for bit the device apply of all right-hand sides, in place with beta, several times.
"""

import numpy as np
import pytest

from conftest import ISO
from paper_2105_08798_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,max_rhs,R", [("bf16x6", 40, 40), ("bf16x6", 40, 33), ("bf16x6", 300, 290), ("bf16x2", 70, 65),
                                                 ("bf16x2", 70, 64), ("tf32", 9, 9)])
def test_host_equals_device(precision, max_rhs, R):
    from paper_2105_08798_gb300 import fbc

    n_i, n_p, L = 50, 70, 4
    xy_i, xy_p = inputs.ring_geometry(n_i, n_p)
    f = inputs.forces(R, n_i, L, seed=R)
    u0 = np.random.default_rng(R).normal(0, 1, (R, n_p, L, 3))
    with fbc.Plan(xy_i, xy_p, L, ISO, precision=precision, max_rhs=max_rhs) as plan:
        plan.tabulate()
        ud = torch.from_numpy(u0.copy()).cuda()
        plan.apply(torch.from_numpy(f).cuda(), ud, alpha=-0.5, beta=1.0, zero_mean=True)
        torch.cuda.synchronize()
        for _ in range(2):
            u = u0.copy()
            plan.apply_host(f, u, alpha=-0.5, beta=1.0, zero_mean=True)
            np.testing.assert_array_equal(u, ud.cpu().numpy())
