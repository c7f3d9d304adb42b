"""BF16X6 plans whose force ring leaves less than a kilobyte of the block's shared memory: the static part has to fit as
well.  Against the in-plane FP64 FFT form at the form's 1e-12.
"""

import numpy as np
import pytest

from conftest import ISO
from paper_2105_08798_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_i,n_p", [(320, 575), (323, 574), (336, 588), (1895, 3380), (3623, 5576)])
def test_full_ring(n_i, n_p):
    from paper_2105_08798_gb300 import fbc

    L, R = 4, 2
    xy_i, xy_p = inputs.ring_geometry(n_i, n_p)
    f = torch.from_numpy(inputs.forces(R, n_i, L, seed=n_i)).cuda()
    out = {}
    with fbc.Plan(xy_i, xy_p, L, ISO, max_rhs=R) as plan:
        plan.tabulate()
        for precision in ("fft64", "bf16x6"):
            plan.set_precision(precision)
            u = torch.full((R, n_p, L, 3), float("nan"), dtype=torch.float64, device="cuda")
            plan.apply(f, u)
            torch.cuda.synchronize()
            plan.sync_status()
            out[precision] = u.cpu().numpy()
    assert np.linalg.norm(out["bf16x6"] - out["fft64"]) <= 1e-12 * np.linalg.norm(out["fft64"])
