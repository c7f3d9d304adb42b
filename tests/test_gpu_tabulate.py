"""Kernel tables of cubic media on the GPU against the oracle's plain DFT of its own kernel.

The FP64-accurate precisions sum the quadrature through trigonometric polynomials, in pairs of node pairs
(node counts divisible by four) or node by node; the reduced precisions keep the matrix at every node.  One of
each pair of differences d, -d is evaluated; the other's entries must be the mirrored bits.
"""

import numpy as np
import pytest

from conftest import CUBIC

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ANGLE = 0.4
ROTATED = dict(CUBIC, Q=[[np.cos(ANGLE), np.sin(ANGLE), 0], [-np.sin(ANGLE), np.cos(ANGLE), 0], [0, 0, 1]])
GPA = dict(CUBIC, C11=1.5e11, C12=1.0e11, C44=0.9e11)
# interface sites and pad sites with differences both of whose signs occur, and others whose mirror does not
XI = np.array([[0, 0], [1, 0], [0, 1], [-1, 0], [0, -1], [2, 1]], np.int32)
XP = np.array([[4, 0], [-4, 0], [0, 5], [0, -5], [6, 2], [3, -7], [5, 5]], np.int32)




def _stiffness(m):
    d = np.eye(3)
    C = (m["C12"] * np.einsum("ij,kl->ijkl", d, d) + m["C44"] * (np.einsum("ik,jl->ijkl", d, d) + np.einsum("il,jk->ijkl", d, d)))
    for i in range(3):
        C[i, i, i, i] += m["C11"] - m["C12"] - 2 * m["C44"]
    Q = np.asarray(m.get("Q", np.eye(3)))
    return np.einsum("ai,bj,ck,dl,abcd->ijkl", Q, Q, Q, Q, C, optimize=True)


def _green(C, x, y, z, nquad):
    """Barnett's integral by the trapezoid rule from the in-plane direction normal to r (a sum with few nodes depends on
    where it starts), [...][3][3]."""
    x, y, z = np.broadcast_arrays(*(np.asarray(v, dtype=np.float64) for v in (x, y, z)))
    R, rho = np.sqrt(x * x + y * y + z * z), np.hypot(x, y)
    on = rho > 0
    safe = np.where(on, rho, 1.0)
    e1 = np.stack([np.where(on, -y / safe, 1.0), np.where(on, x / safe, 0.0), 0 * x], -1)
    e2 = np.cross(np.stack([x / R, y / R, z / R], -1), e1)
    S = 0.0
    for q in range(nquad):
        n = np.cos(np.pi * q / nquad) * e1 + np.sin(np.pi * q / nquad) * e2
        S = S + np.linalg.inv(np.einsum("ijkl,...j,...l->...ik", C, n, n))
    return S / (4 * np.pi * nquad * R)[..., None, None]


def _mode_table(oracle_mod, material, L, d, nquad):
    """The kernel of Eqs. 32-36 at the default order with that quadrature, and its DFT (the oracle's)."""
    C, n, N = _stiffness(material), 4, 6
    w = oracle_mod.richardson_weights(n, N)
    s = np.arange(L)
    z = np.where(s <= L // 2, s, s - L).astype(np.float64)
    x, y, z = d[:, :1].astype(np.float64), d[:, 1:].astype(np.float64), z[None, :]
    T = _green(C, x, y, z, nquad)
    for m in range(1, n + N + 1):
        t = _green(C, x, y, z + m * L, nquad) + _green(C, x, y, z - m * L, nquad) - 2 * _green(C, 0.0, 0.0, float(m * L), nquad)
        T = T + t * w[max(0, m - n):].sum()
    T[:, L // 2, 2, :2] = T[:, L // 2, :2, 2] = 0.0  # the mean of the two offsets +-L/2
    return oracle_mod.mode_table(T)


@pytest.mark.parametrize("precision", ["fp64", "f32x2", "fp32"])
@pytest.mark.parametrize("quad,material", [(64, CUBIC), (64, ROTATED), (64, GPA), (8, CUBIC), (30, ROTATED), (37, CUBIC),
                                           (512, CUBIC)])
@pytest.mark.parametrize("L", [2, 32])
def test_cubic_table_matches_oracle(oracle_mod, precision, quad, material, L):
    from paper_2105_08798_gb300 import fbc

    d = np.unique((XP[:, None, :] - XI[None, :, :]).reshape(-1, 2), axis=0)
    # converged node counts against the oracle (its sum starts elsewhere on the circle), the others node for node
    ref = (oracle_mod.mode_table(oracle_mod.kernel_table(material, L, 1.0, d, nquad=quad)) if quad >= 64
           else _mode_table(oracle_mod, material, L, d, quad))
    with fbc.Plan(XI, XP, L, material, quad=quad, precision=precision) as plan:
        plan.tabulate()
        torch.cuda.synchronize()
        got = plan.mode_table(d)
    want = np.stack([ref[..., 0, 0].real, ref[..., 0, 1].real, ref[..., 1, 1].real, ref[..., 2, 2].real,
                     ref[..., 0, 2].imag, ref[..., 1, 2].imag], axis=-1)
    # the Richardson weights amplify rounding by up to sum |w| = 1.6e4 at the default order: 1.6e4 x 2^-53 x a few
    assert np.linalg.norm(got - want) <= 1e-11 * np.linalg.norm(want)
    index = {tuple(x): t for t, x in enumerate(d)}
    pairs = [(t, index[(-x[0], -x[1])]) for t, x in enumerate(map(tuple, d)) if (-x[0], -x[1]) in index]
    assert 0 < len(pairs) < len(d)
    for a, b in pairs:
        np.testing.assert_array_equal(got[a][:, :4], got[b][:, :4])
        np.testing.assert_array_equal(got[a][:, 4:], -got[b][:, 4:])
