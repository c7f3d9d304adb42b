"""Kernel tables of cubic media from nearly isotropic to soft in shear, against extended-precision sums.

The FP64-accurate precisions have two forms of the quadrature: node by node, and through trigonometric polynomials whose
rounding is relative to the stiffest direction and not to the softest.  Whatever form a plan takes, its table must be
as exact as the node-by-node one (which the reduced precisions always take).
"""

import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

L = 16
XI = np.array([[0, 0], [1, 0], [0, 1], [-1, 0], [2, 1]], np.int32)
XP = np.array([[4, 0], [-5, 1], [6, 2], [3, -7]], np.int32)
LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288")


def _angle(v):
    """cos and sin in extended precision of pi times the rationals v."""
    return np.cos(PI * v), np.sin(PI * v)


def _green(m, x, y, z, nquad):
    """Barnett's integral by the trapezoid rule from the in-plane direction normal to r, [6][...] (11 12 22 33 13 23)."""
    x, y, z = np.broadcast_arrays(LD(x), LD(y), LD(z))
    R, rho = np.sqrt(x * x + y * y + z * z), np.sqrt(x * x + y * y)
    on = rho > 0
    safe = np.where(on, rho, LD(1))
    e1 = (np.where(on, -y / safe, LD(1)), np.where(on, x / safe, LD(0)))
    hx, hy, hz = x / R, y / R, z / R
    e2 = (-hz * e1[1], hz * e1[0], hx * e1[1] - hy * e1[0])
    c11, c12, c44 = LD(m["C11"]), LD(m["C12"]), LD(m["C44"])
    S = [0] * 6
    for q in range(nquad):
        c, s = _angle(LD(q) / nquad)
        n0, n1, n2 = c * e1[0] + s * e2[0], c * e1[1] + s * e2[1], s * e2[2]
        a, b, d = (c11 * n0 * n0 + c44 * (n1 * n1 + n2 * n2), c11 * n1 * n1 + c44 * (n0 * n0 + n2 * n2),
                   c11 * n2 * n2 + c44 * (n0 * n0 + n1 * n1))
        e, f, g = (c12 + c44) * n1 * n2, (c12 + c44) * n0 * n2, (c12 + c44) * n0 * n1
        cof = (b * d - e * e, e * f - d * g, a * d - f * f, a * b - g * g, e * g - b * f, f * g - a * e)
        det = a * cof[0] + g * cof[1] + f * cof[4]
        S = [t + v / det for t, v in zip(S, cof)]
    return np.stack(S) / (4 * PI * nquad * R)


def _mode_table(m, d, nquad):
    """The kernel of Eqs. 32-36 at the default order and its DFT, [nd][L/2 + 1][6]."""
    n, N = 4, 6
    w = [LD((n + i) ** N * (-1) ** (i + N)) / (math.factorial(i) * math.factorial(N - i)) for i in range(N + 1)]
    x, y, z = d[:, :1].astype(LD), d[:, 1:].astype(LD), np.arange(L // 2 + 1).astype(LD)[None, :]
    T = _green(m, x, y, z, nquad)
    for j in range(1, n + N + 1):
        t = (_green(m, x, y, z + j * L, nquad) + _green(m, x, y, z - j * L, nquad)
             - 2 * _green(m, 0.0, 0.0, float(j * L), nquad)[:, None, None])
        T = T + t * sum(w[max(0, j - n):])
    T[4:, :, 0] = T[4:, :, -1] = 0
    wt = np.array([1] + [2] * (L // 2 - 1) + [1], dtype=LD)
    c, s = _angle(LD(2) * np.outer(np.arange(L // 2 + 1), np.arange(L // 2 + 1)).astype(LD) / L)
    return np.stack([(T[t] * wt) @ c if t < 4 else -2 * (T[t] @ s) for t in range(6)], axis=-1)


@pytest.mark.parametrize("c11,c12,c44,quad", [
    (1.5, 1.0, 0.9, 64), (1.8, 0.4, 0.4, 64), (2.4, 1.2, 0.6, 50), (1.5, 1.0, 0.9, 48), (1.5, 1.0, 0.9, 49),
    (1.0, 0.9, 0.45, 64), (1.0, 0.2, 0.01, 64), (1.0, 0.99, 0.2, 64), (1.0, 0.99, 0.005, 64), (4.0, 0.1, 0.01, 64),
    (1.0e-3, 0.9e-3, 0.45e-3, 512)])
def test_table_as_exact_as_node_by_node(c11, c12, c44, quad):
    from paper_2105_08798_gb300 import fbc

    m = {"kind": "cubic", "C11": c11, "C12": c12, "C44": c44}
    d = np.unique((XP[:, None, :] - XI[None, :, :]).reshape(-1, 2), axis=0)
    want = _mode_table(m, d, quad)
    err = {}
    for precision in ("fp64", "fp32"):
        with fbc.Plan(XI, XP, L, m, quad=quad, precision=precision) as plan:
            plan.tabulate()
            torch.cuda.synchronize()
            err[precision] = float(np.linalg.norm((plan.mode_table(d) - want).astype(np.float64)))
    # two sums of the same length: their rounding errors over a thousand entries differ by their scatter
    assert err["fp64"] <= 2.0 * err["fp32"]
