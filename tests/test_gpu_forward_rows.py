"""Fused BF16-weight inference at the edges of its tiles (one row, a tile of 128 and one off, both tile slots of every
SM and one row more) and with inputs whose activations reach far into both tails of SiLU, against the FP64 network with
BF16-rounded parameters: hi + lo bf16 activations carry 2^-17 per layer, 5e-5 over three layers with their sums.
"""

import numpy as np
import pytest

from oracle import mlp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H", [32, 64, 96, 128])
@pytest.mark.parametrize("n,scale", [(1, 1.0), (127, 1.0), (128, 300.0), (129, 1.0), (255, 30.0), (2 * 152 * 128 + 1, 1.0)])
def test_rows(H, n, scale):
    from paper_2105_08798_gb300 import fbc

    x = (np.random.default_rng(n + H).normal(0, scale, (n, 4))).astype(np.float32)
    with fbc.Surrogate(width=H, seed=H + 1) as S:
        y = S.forward(torch.from_numpy(x).cuda(), bf16_weights=True).cpu().numpy()
        S.sync_status()
        ref, _ = mlp.forward(mlp.round_bf16(S.params()), H, x)
    assert np.linalg.norm(y - ref) <= 5e-5 * np.linalg.norm(ref)
    assert np.abs(y - ref).max() <= 5e-5 * np.abs(ref).max()
