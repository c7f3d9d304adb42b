"""Loss gradients of the surrogate at the edges of the split weight-gradient kernel: fewer rows than one step of 32,
a last split of one row, one split (many tiles), widths that are no multiple of the 64-wide tile.

Tolerance: FP32 sums of n rows and up to H products against FP64, as the gradient tests of the other sizes.
"""

import numpy as np
import pytest

from oracle import mlp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,n", [(8, 1), (40, 31), (128, 33), (72, 64), (128, 50 * 32 + 1), (1024, 65), (96, 4097)])
def test_gradient_at_split_edges(H, n):
    from paper_2105_08798_gb300 import fbc

    rng = np.random.default_rng(7 * H + n)
    with fbc.Surrogate(width=H, seed=1) as S:
        p = rng.normal(0, 0.3 if H < 512 else 0.05, S.n_params).astype(np.float32)
        S.set_params(p)
        x = rng.normal(0, 1, (n, 4)).astype(np.float32)
        t = rng.normal(0, 1, (n, 6)).astype(np.float32)
        loss, g = S.loss_grad(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda())
        # rows that do not start on a 16-byte boundary take the scalar loads: the same sums, the same bits
        pad = torch.zeros(4 * n + 1, dtype=torch.float32, device="cuda")
        pad[1:] = torch.from_numpy(x).cuda().reshape(-1)
        loss2, g2 = S.loss_grad(pad[1:].view(n, 4), torch.from_numpy(t).cuda())
    ref_loss, ref_g = mlp.loss_grad(p, H, x, t)
    assert loss == pytest.approx(ref_loss, rel=1e-5)
    assert np.linalg.norm(g - ref_g) <= 1e-5 * np.linalg.norm(ref_g)
    assert loss2 == loss
    np.testing.assert_array_equal(g2, g)
