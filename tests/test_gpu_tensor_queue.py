"""Tensor-core batches whose instances stage their table sub-boxes differently: two buffers or one, by bulk copies or by the
warps that read them.  One persistent block runs items of all of them in turn, its barriers' parities running on, and
every instance has to give the bits of its plan's own apply.
"""

import pytest

from conftest import ISO
from paper_2105_08798_gb300 import inputs
from test_gpu_tensor_shapes import _sites, test_shapes as _test_shapes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# compact rings; sites far apart along one line, whose sub-boxes leave no room for padded rows or a second buffer
SHAPES = [("ring", 70, 130, 1, 8), ("line", 70, 130, 16, 4), ("line", 70, 130, 20, 4), ("cut", 100, 180, 1, 8),
          ("line", 129, 260, 24, 4), ("ring", 200, 150, 2, 8)]


@pytest.mark.parametrize("precision", ["tf32", "bf16x2", "bf16x3"])
@pytest.mark.parametrize("R", [3, 17])
def test_mixed_staging(precision, R):
    from paper_2105_08798_gb300 import fbc

    plans, fs, want = [], [], []
    for j, (kind, n_i, n_p, step, L) in enumerate(SHAPES):
        xy_i, xy_p = _sites(kind, n_i, n_p, step)
        plans.append(fbc.Plan(xy_i, xy_p, L, ISO, precision=precision, max_rhs=R))
        plans[-1].tabulate()
        fs.append(torch.from_numpy(inputs.forces(R, len(xy_i), L, seed=40 + j)).cuda())
        want.append(torch.zeros((R, len(xy_p), L, 3), dtype=torch.float64, device="cuda"))
        plans[-1].apply(fs[-1], want[-1], project=False)  # (every one of these shapes fits every form)
    got = [torch.full_like(u, float("nan")) for u in want]
    with fbc.Batch(plans, fs, got) as b:
        for graph in (False, True):
            b.apply(project=False, graph=graph)
            torch.cuda.synchronize()
            assert b.info()["launch_form"] == 0
            for p, u, v in zip(plans, want, got):
                p.sync_status()
                assert torch.equal(u, v)
                v.fill_(float("nan"))
    for p in plans:
        p.close()


@pytest.mark.parametrize("kind,n_i,n_p,step,L,R,mat", next(m.args[1] for m in _test_shapes.pytestmark if m.name == "parametrize"))
def test_every_form_takes_every_shape(kind, n_i, n_p, step, L, R, mat):
    """None of the geometries of those tests is too large for a form's shared memory: no form may refuse one."""
    from paper_2105_08798_gb300 import fbc

    xy_i, xy_p = _sites(kind, n_i, n_p, step)
    f = torch.from_numpy(inputs.forces(R, len(xy_i), L, seed=1)).cuda()
    with fbc.Plan(xy_i, xy_p, L, mat, max_rhs=R) as plan:
        plan.tabulate()
        for precision in ("tf32", "bf16x2", "bf16x3"):
            plan.set_precision(precision)
            plan.apply(f, torch.empty((R, len(xy_p), L, 3), dtype=torch.float64, device="cuda"))
            torch.cuda.synchronize()
            plan.sync_status()
