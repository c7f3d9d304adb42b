"""Fused BF16-weight inference with pre-activations far out in both tails of SiLU, next to each other.

The kernel evaluates neighbouring columns in pairs.  A network whose first layer puts chosen values into the columns of a
pair and whose later layers pass them on shows each: a strongly negative one has to vanish, a large positive one to come
through, whatever its neighbour is.  All parameters are exact in bf16.
"""

import numpy as np
import pytest

from oracle import mlp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

H = 32


@pytest.mark.parametrize("z0,z1", [(-2.0 ** 60, 1.0), (1.0, -2.0 ** 60), (-2.0 ** 100, -2.0 ** 80), (2.0 ** 100, -64.0),
                                   (-2.0 ** 7, 2.0 ** 90), (2.0 ** 100, 2.0 ** 100), (-41.0, -43.0), (-2.0 ** 126, 2.0 ** 126)])
@pytest.mark.parametrize("column", [0, 14, 30])
def test_pair(z0, z1, column):
    from paper_2105_08798_gb300 import fbc

    W1, W2, W3, W4 = np.zeros((4, H)), np.zeros((H, H)), np.zeros((H, H)), np.zeros((H, 6))
    b1, b2, b3, b4 = np.zeros(H), np.zeros(H), np.zeros(H), np.zeros(6)
    for j, z in enumerate((z0, z1)):
        W1[0, column + j] = z
        W2[column + j, 5 + j] = 2.0 / abs(z) if z > 8 else 2.0  # a large value scaled to 2, the others doubled
        W3[5 + j, 9 + j] = 1.0
        W4[9 + j, j] = 1.0
    p = np.concatenate([a.ravel() for a in (W1, b1, W2, b2, W3, b3, W4, b4)]).astype(np.float32)
    assert (mlp.round_bf16(p) == p).all()
    x = np.zeros((130, 4), np.float32)
    x[:, 0] = 1.0
    with fbc.Surrogate(width=H, seed=0) as S:
        S.set_params(p)
        y = S.forward(torch.from_numpy(x).cuda(), bf16_weights=True).cpu().numpy()
        S.sync_status()
    with np.errstate(over="ignore"):
        ref, _ = mlp.forward(p, H, x)
    # the activations' two bf16 pieces hold 2^-17 of a value, three layers; a vanishing one (|SiLU| < 1e-16) stays below
    # 1e-15 through a doubling and two halvings (SiLU(z) ~ z / 2)
    assert np.isfinite(y).all()
    assert (np.abs(y - ref) <= 5e-5 * np.abs(ref) + 1e-15).all()
