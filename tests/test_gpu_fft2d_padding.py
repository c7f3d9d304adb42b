"""In-plane FFT applies of a plan that served other precisions before, with an odd number of pad columns.

Two neighbouring columns share one complex sequence of the inverse line transform, and the last of an odd number shares
it with a padding slot of the mode buffer.  The dense forms write that slot; whatever they (or memory's former owner) left
there, an FFT apply gives the bits of a plan that never ran anything else.
"""

import numpy as np
import pytest

from conftest import CUBIC, ISO
from paper_2105_08798_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fft64", "fft32"])
@pytest.mark.parametrize("n_i,n_p,L,R,material", [(1, 1, 2, 1, ISO), (40, 61, 16, 2, ISO), (90, 129, 32, 1, CUBIC),
                                                  (90, 127, 8, 3, ISO)])
@pytest.mark.parametrize("before", [1e15, float("inf")])
def test_bits_of_a_fresh_plan(precision, n_i, n_p, L, R, material, before):
    from paper_2105_08798_gb300 import fbc

    xy_i, xy_p = inputs.ring_geometry(n_i, n_p)
    f = torch.from_numpy(inputs.forces(R, n_i, L, seed=n_p)).cuda()
    got = []
    for used in (False, True):
        with fbc.Plan(xy_i, xy_p, L, material, max_rhs=R) as plan:
            plan.tabulate()
            if used:  # fills the padding slots with values (or the NaN of inf - inf) far above the update's
                plan.apply(f * before, torch.zeros((R, n_p, L, 3), dtype=torch.float64, device="cuda"), project=False)
            plan.set_precision(precision)
            u = torch.full((R, n_p, L, 3), float("nan"), dtype=torch.float64, device="cuda")
            plan.apply(f, u, zero_mean=True)
            alpha = torch.ones(R, dtype=torch.float64, device="cuda")
            plan.apply_relaxed(f, None, u, alpha, du_max=0.01, zero_mean=True)
            torch.cuda.synchronize()
            got.append((u.cpu().numpy(), alpha.cpu().numpy()))
    assert np.isfinite(got[0][0]).all()
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)
