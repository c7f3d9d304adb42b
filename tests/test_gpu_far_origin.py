"""Geometries far from the origin: sites close to the largest accepted coordinate, where the sites' own offsets in a staged
sub-box no longer fit a signed word while their differences do.  Only differences enter the update: the bits are those of
the same geometry around the origin.
"""

import numpy as np
import pytest

from conftest import ISO
from paper_2105_08798_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FAR = 2 ** 20 - 400


@pytest.mark.parametrize("step,precisions", [(1, ("fp64", "f32x2", "fp32", "tf32", "bf16x2", "bf16x3", "bf16x6", "fft64", "fft32")),
                                             (3, ("tf32", "bf16x2", "bf16x3"))])
@pytest.mark.parametrize("shift", [(FAR, FAR), (-FAR, -FAR), (FAR, -FAR), (-FAR, FAR)])
def test_same_bits(step, precisions, shift):
    from paper_2105_08798_gb300 import fbc

    L, R = 8, 17
    xy_i, xy_p = (xy * np.array([step, 1], np.int32) for xy in inputs.ring_geometry(200, 150))
    f = torch.from_numpy(inputs.forces(R, len(xy_i), L, seed=step)).cuda()
    out = []
    for d in (np.zeros(2, np.int32), np.array(shift, np.int32)):
        with fbc.Plan(xy_i + d, xy_p + d, L, ISO, max_rhs=R) as plan:
            plan.tabulate()
            for precision in precisions:
                plan.set_precision(precision)
                u = torch.empty((R, len(xy_p), L, 3), dtype=torch.float64, device="cuda")
                plan.apply(f, u)
                torch.cuda.synchronize()
                plan.sync_status()
                out.append(u)
    for precision, a, b in zip(precisions, out, out[len(precisions):]):
        assert torch.equal(a, b), precision
