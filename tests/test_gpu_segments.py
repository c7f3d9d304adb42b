"""Plans whose interface sum is cut into segments (few tiles): one column, segments of 16 columns with a ragged last one,
of whole interface tiles, several right-hand sides, repeated applies (the segment counters are zero again), against the
oracle's real-space sum at the forms' own tolerances (1e-12 FP64-accurate, 5e-6 FP32), and each right-hand side alone
against all together, bit for bit.
"""

import numpy as np
import pytest

from conftest import CUBIC, ISO
from paper_2105_08798_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("f32x2", 1e-12), ("fp32", 5e-6)])
@pytest.mark.parametrize("n_i,n_p,L,R,mat", [(1, 1, 4, 1, ISO), (17, 130, 8, 1, CUBIC), (65, 40, 4, 5, ISO), (200, 300, 16, 2, CUBIC),
                                             (530, 129, 2, 3, ISO)])
def test_segments(oracle_mod, precision, tol, n_i, n_p, L, R, mat):
    from paper_2105_08798_gb300 import fbc

    xy_i, xy_p = inputs.ring_geometry(n_i, n_p)
    f = inputs.forces(R, n_i, L, seed=3 * n_i)
    ref = oracle_mod.pad_update(xy_i, xy_p, L, 1.0, mat, f, project=False, nquad=64)
    fd = torch.from_numpy(f).cuda()
    with fbc.Plan(xy_i, xy_p, L, mat, precision=precision, max_rhs=R) as plan:
        plan.tabulate()
        out = []
        for _ in range(3):
            u = torch.full((R, n_p, L, 3), float("nan"), dtype=torch.float64, device="cuda")
            plan.apply(fd, u, project=False)
            torch.cuda.synchronize()
            out.append(u.cpu().numpy())
        alone = torch.zeros((1, n_p, L, 3), dtype=torch.float64, device="cuda")
        plan.apply(fd[R - 1:].contiguous(), alone, project=False)
        torch.cuda.synchronize()
        plan.sync_status()
    assert np.linalg.norm(out[0] - ref) <= tol * np.linalg.norm(ref)
    np.testing.assert_array_equal(out[0], out[1])
    np.testing.assert_array_equal(out[0], out[2])
    if precision != "fp32":  # the FP32 form's one-rhs and eight-rhs tiles round alike only in the k = 0 band
        np.testing.assert_array_equal(alone.cpu().numpy()[0], out[0][R - 1])
