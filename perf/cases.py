"""Performance cases of the library: the calls a user's program makes, over the sizes it makes them at.

Every case goes through the Python binding (``paper_2105_08798_gb300.fbc``), on inputs made from a seed.  The kinds:

* ``apply``      -- one pad update ``u <- beta u + alpha G f`` on device arrays, in one of the contraction forms;
* ``host``       -- the same update on pinned host arrays (copies in and out are part of the call);
* ``iteration``  -- the harmonic half of one FBC iteration: incompatibility force, relaxed update, zero mean;
* ``batch``      -- uneven instances updated together by one captured graph;
* ``geometry``   -- a new geometry: the kernel table, then the first update with it;
* ``forward``    -- the surrogate network on many rows;
* ``gradient``   -- one training step's loss and parameter gradient.

``exact`` evaluates the same quantities in 64 bits with torch and numpy alone: the kernel from its image sum, the
update as a three-dimensional circular convolution, the network by its definition.
"""

from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2105_08798_gb300 import fbc

ISO = {"kind": "isotropic", "mu": 1.0, "nu": 0.3}
CUBIC = {"kind": "cubic", "C11": 1.5, "C12": 1.0, "C44": 0.9}
K1, K2 = 1.0, 0.4  # spring model of the iteration; its long-wave medium:
SPRING = {"kind": "cubic", "C11": K1 + 2 * K2, "C12": K2, "C44": K2}
MATERIALS = {"isotropic": ISO, "cubic": CUBIC, "spring": SPRING}
RICH_N, RICH_NN = 4, 6  # default order of the image sum's extrapolation


# ---- the cases ------------------------------------------------------------------------------------------------
def _apply(name, precision, n_i, n_p, L, rhs, material="isotropic", alpha=1.0, beta=0.0, zero_mean=False):
    return {"name": name, "kind": "apply", "precision": precision, "n_i": n_i, "n_p": n_p, "L": L, "rhs": rhs,
            "material": material, "alpha": alpha, "beta": beta, "zero_mean": zero_mean}


def listed():
    return [
        # A short test slab, the smallest update in use: the call costs launches and a few idle SMs, not work.
        _apply("tiny_fp64", "fp64", 200, 300, 16, 1, alpha=-1.0, beta=1.0, zero_mean=True),
        # One step of an atomistic-continuum relaxation at a middling slab: what a coupled program repeats all day.
        {"name": "iteration_f32x2", "kind": "iteration", "precision": "f32x2", "n_i": 1000, "n_p": 1500, "L": 64,
         "rhs": 1, "material": "spring", "du_max": 0.02},
        # The paper-scale slab, anisotropic, one force vector: the dense FP64-accurate update.
        _apply("single_f32x2", "f32x2", 4000, 6000, 256, 1, material="cubic"),
        # The same slab size through the in-plane FFT form, the fast way to FP64 accuracy at one force vector.
        _apply("single_fft64", "fft64", 4000, 6000, 256, 1),
        # Many force vectors at FP64 accuracy (response of a slab to many states): the tensor-core form.
        _apply("many_bf16x6", "bf16x6", 4000, 6000, 256, 64),
        # The same form fed from a program that keeps its arrays on the host; ragged columns, a part-filled group.
        {"name": "host_bf16x6", "kind": "host", "precision": "bf16x6", "n_i": 1777, "n_p": 2666, "L": 128, "rhs": 40,
         "material": "isotropic", "alpha": -1.0, "beta": 1.0, "zero_mean": False},
        # Many vectors where 1e-5 is enough (preconditioning, screening): reduced precision on the tensor cores.
        _apply("many_bf16x2", "bf16x2", 3001, 4502, 512, 16, alpha=-1.0, beta=1.0),
        # A long, wide slab with a few vectors through the FP32 in-plane FFT form, the largest geometry in use.
        _apply("large_fft32", "fft32", 8000, 12000, 512, 8),
        # Independent dislocation segments of uneven size updated together, a few successive residuals each.
        {"name": "batch_f32x2", "kind": "batch", "precision": "f32x2", "instances": 12, "n_max": 2000, "L_max": 128,
         "rhs": 4, "pick": 7},
        # A dislocation that moved: a new table for the slab and the first update with it.
        {"name": "geometry_f32x2", "kind": "geometry", "precision": "f32x2", "n_i": 1000, "n_p": 1500, "L": 64,
         "rhs": 1, "material": "cubic"},
        # The learned far field: a mode slice's worth of rows through the network.
        {"name": "forward", "kind": "forward", "rows": 1000000, "width": 128},
        # One training step of that network at the default batch.
        {"name": "gradient", "kind": "gradient", "rows": 4096, "width": 128},
    ]


# Pair-modes per second of each form (right-hand sides counted in its groups), to keep a drawn update below the largest
# listed one.
_RATE = {"fp64": 3e10, "f32x2": 1.2e11, "fp32": 3e11, "bf16x6": 7e11, "tf32": 2e12, "bf16x2": 2e12, "bf16x3": 2e12,
         "fft64": 4e11, "fft32": 2e12}
_GROUP = {"bf16x6": 32, "tf32": 8, "bf16x2": 8, "bf16x3": 8}
_BUDGET = 0.12  # seconds


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _fit(c, rate, group):
    """Shrink a case's vectors, then its repeats, until it costs no more than the budget."""
    def cost():
        r = -(-c["rhs"] // group) * group
        return c["n_i"] * c["n_p"] * (c["L"] // 2 + 1) * r / rate

    while cost() > _BUDGET and c["rhs"] > group:
        c["rhs"] = max(group, c["rhs"] // 2)
    while cost() > _BUDGET and c["L"] > 8:
        c["L"] //= 2
    return c


def draw(rng: random.Random):
    kind = rng.choices(["apply", "host", "iteration", "batch", "geometry", "forward", "gradient"],
                       [10, 2, 2, 2, 2, 1, 1])[0]
    if kind == "forward":
        return {"kind": kind, "rows": _log(rng, 1000, 2000000), "width": rng.choice([32, 64, 96, 128])}
    if kind == "gradient":
        return {"kind": kind, "rows": _log(rng, 256, 16384), "width": rng.choice([32, 64, 96, 128])}
    if kind == "batch":
        return {"kind": kind, "precision": rng.choice(["f32x2", "fp32", "bf16x2"]), "instances": rng.randint(2, 16),
                "n_max": _log(rng, 300, 2500), "L_max": rng.choice([32, 64, 128]), "rhs": rng.randint(1, 9),
                "pick": rng.randint(0, 999)}
    n_i = _log(rng, 200, 4000 if kind != "geometry" else 1500)
    n_p = int(n_i * rng.uniform(1.2, 1.8))
    L = 1 << rng.randint(3, 9 if kind != "geometry" else 7)
    if kind == "iteration":
        c = {"kind": kind, "precision": rng.choice(["f32x2", "fft64", "fp64"]), "n_i": n_i, "n_p": n_p, "L": L,
             "rhs": rng.randint(1, 3), "material": "spring", "du_max": 0.02}
        return _fit(c, _RATE[c["precision"]], 1)
    if kind == "geometry":
        c = {"kind": kind, "precision": rng.choice(["f32x2", "fft64", "fp64"]), "n_i": n_i, "n_p": n_p, "L": L,
             "rhs": 1, "material": rng.choice(["cubic", "isotropic"])}
        return _fit(c, _RATE[c["precision"]], 1)
    if kind == "host":
        precision = rng.choice(["bf16x6", "bf16x6", "f32x2", "fft32"])
        rhs = _log(rng, 8, 64)
    else:
        precision = rng.choice(["fp64", "f32x2", "f32x2", "fft64", "fft64", "bf16x6", "bf16x6", "bf16x2", "tf32",
                                "fft32", "fp32"])
        rhs = _log(rng, 8, 64) if precision in _GROUP else _log(rng, 1, 16)
    if kind == "host":
        L = min(L, 256)
    c = _apply("", precision, n_i, n_p, L, rhs, material=rng.choice(["isotropic", "isotropic", "cubic"]) if n_i < 1500 else
               "isotropic", alpha=rng.choice([1.0, -1.0]), beta=rng.choice([0.0, 1.0]), zero_mean=rng.random() < 0.3)
    del c["name"]
    c["kind"] = kind
    return _fit(c, _RATE[precision], _GROUP.get(precision, 1))


# ---- geometry and inputs ----------------------------------------------------------------------------------------
def rings(n_i: int, n_p: int):
    """Core, interface and pad sites of a ring slab: interface = the n_i outermost sites with |x|^2 <= n_i / 2, pad =
    the n_p innermost beyond, core = the rest inside."""
    R = int(math.sqrt((n_i / 2.0) + (n_i + n_p) / math.pi * 1.4 + 64)) + 2
    ax = np.arange(-R, R + 1)
    X, Y = (a.ravel() for a in np.meshgrid(ax, ax, indexing="ij"))
    order = np.lexsort((Y, X, np.arctan2(Y.astype(float), X.astype(float)), X * X + Y * Y))
    xy = np.stack([X[order], Y[order]], axis=1).astype(np.int32)
    inner = int((2 * (X * X + Y * Y) <= n_i).sum())
    return (np.ascontiguousarray(xy[:inner - n_i]), np.ascontiguousarray(xy[inner - n_i:inner]),
            np.ascontiguousarray(xy[inner:inner + n_p]))


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _normal(seed, salt, shape, scale=1.0):
    g = torch.Generator(device=_device())
    g.manual_seed(int(seed) * 1009 + salt)
    return torch.randn(shape, generator=g, dtype=torch.float64, device=_device()) * scale


def _update_inputs(c, seed, salt=0):
    """Forces N(0, 1) and displacements of the size the update gives."""
    return (_normal(seed, salt + 1, (c["rhs"], c["n_i"], c["L"], 3)),
            _normal(seed, salt + 2, (c["rhs"], c["n_p"], c["L"], 3)))


def _instances(c):
    rng = random.Random(c["pick"])
    got = []
    for _ in range(c["instances"]):
        n_i = _log(rng, min(200, c["n_max"] // 2), c["n_max"])
        got.append({"n_i": n_i, "n_p": int(round(1.5 * n_i)), "L": 1 << rng.randint(5, c["L_max"].bit_length() - 1),
                    "rhs": c["rhs"], "material": "isotropic"})
    return got


def _iteration_inputs(c, seed):
    """Displacements of the core atoms (relaxed), the interface and the pad, and the last iteration's force."""
    core, _, _ = rings(c["n_i"], c["n_p"])
    R, L = c["rhs"], c["L"]
    return ([_normal(seed, 1, (R, len(core), L, 3), 0.05), _normal(seed, 2, (R, c["n_i"], L, 3), 0.05),
             _normal(seed, 3, (R, c["n_p"], L, 3), 0.05)], _normal(seed, 4, (R, c["n_i"], L, 3), 0.2))


def _network(c, seed):
    """Packed parameters (He-scaled weights, small biases), rows of the network's features, targets."""
    rng = np.random.default_rng([int(seed), 5])
    H, n = c["width"], c["rows"]
    parts = []
    for a, b in ((4, H), (H, H), (H, H), (H, 6)):
        parts += [rng.standard_normal(a * b) * math.sqrt(2.0 / a) * 0.8, rng.standard_normal(b) * 0.05]
    p = np.concatenate(parts).astype(np.float32)
    g = torch.Generator(device=_device())
    g.manual_seed(int(seed) * 1009 + 6)
    z = torch.rand((n, 3), generator=g, dtype=torch.float64, device=_device())
    r, qr, th = 8.0 * 12.0 ** z[:, 0], 16.0 * 1e-3 ** z[:, 1], 2 * math.pi * z[:, 2]
    x = torch.stack([qr.log() / 4, th.cos(), th.sin(), r.log() / 5], dim=1).to(torch.float32)
    t = torch.stack([0.1 * (1 + qr).rsqrt() * torch.cos(th * (j % 3)) + 0.01 * j for j in range(6)], dim=1)
    return p, x.contiguous(), t.to(torch.float32).contiguous()


# ---- what a program has in hand, and one pass ----------------------------------------------------------------------
def _plan(c):
    _, xy_i, xy_p = rings(c["n_i"], c["n_p"])
    return fbc.Plan(xy_i, xy_p, c["L"], MATERIALS[c["material"]], precision=c["precision"], max_rhs=c["rhs"])


def prepare(case, seed):
    c, s = dict(case), {"case": dict(case)}
    kind = c["kind"]
    if kind in ("forward", "gradient"):
        p, s["x"], s["t"] = _network(c, seed)
        s["net"] = fbc.Surrogate(width=c["width"], seed=0)
        s["net"].set_params(p)
        return s
    if kind == "batch":
        s["plans"], s["f"], s["u"] = [], [], []
        for j, q in enumerate(_instances(c)):
            plan = _plan(dict(q, precision=c["precision"]))
            plan.tabulate()
            f, u = _update_inputs(q, seed, 10 * j)
            s["plans"].append(plan)
            s["f"].append(f)
            s["u"].append(u)
        s["batch"] = fbc.Batch(s["plans"], s["f"], s["u"])
        return s
    s["plan"] = _plan(c)
    if kind != "geometry":
        s["plan"].tabulate()
    if kind == "iteration":
        core, xy_i, xy_p = rings(c["n_i"], c["n_p"])
        K = fbc.fbc_spring_constants(K1, K2, 1.0)
        s["stencil"] = fbc.Stencil(xy_i, [core, xy_i, xy_p], c["L"], K)
        s["u"], s["f_prev"] = _iteration_inputs(c, seed)
        s["f"] = torch.empty_like(s["f_prev"])
        s["alpha"] = torch.ones(c["rhs"], dtype=torch.float64, device=_device())
        return s
    s["f"], s["u"] = _update_inputs(c, seed)
    if kind == "host":
        for k in ("f", "u"):
            h = torch.empty(s[k].shape, dtype=torch.float64, pin_memory=True)
            h.copy_(s[k])
            s[k] = h
    return s


def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "apply":
        return s["plan"].apply(s["f"], s["u"], alpha=c["alpha"], beta=c["beta"], zero_mean=c["zero_mean"])
    if kind == "host":
        return s["plan"].apply_host(s["f"], s["u"], alpha=c["alpha"], beta=c["beta"], zero_mean=c["zero_mean"])
    if kind == "iteration":
        s["stencil"].incompat_force(s["u"], s["f"])
        s["plan"].apply_relaxed(s["f"], s["f_prev"], s["u"][2], s["alpha"], du_max=c["du_max"], zero_mean=True)
        s["f"], s["f_prev"] = s["f_prev"], s["f"]  # this iteration's force is the next one's last
        return {"f": s["f_prev"], "u": s["u"][2], "alpha": s["alpha"]}
    if kind == "batch":
        s["batch"].apply(alpha=-1.0, beta=1.0)
        return s["u"]
    if kind == "geometry":
        s["plan"].tabulate()
        return s["plan"].apply(s["f"], s["u"])
    if kind == "forward":
        return s["net"].forward(s["x"], bf16_weights=True)
    return s["net"].loss_grad(s["x"], s["t"])  # (loss, gradient)


# ---- what a pass cannot do without ------------------------------------------------------------------------------------
def _n_differences(n_i, n_p):
    """Distinct in-plane differences between pad and interface sites."""
    _, a, b = rings(n_i, n_p)
    n = int(2 * max(np.abs(a).max(), np.abs(b).max()) + 2)
    n = 1 << (n - 1).bit_length()
    A, B = np.zeros((n, n)), np.zeros((n, n))
    A[a[:, 0] % n, a[:, 1] % n] = 1
    B[b[:, 0] % n, b[:, 1] % n] = 1
    full = np.fft.irfft2(np.fft.rfft2(B, (2 * n, 2 * n)) * np.conj(np.fft.rfft2(A, (2 * n, 2 * n))), (2 * n, 2 * n))
    return int((full > 0.5).sum())


def _update_work(c, in_place):
    """One update: forces read, displacements written (and read), the used table entries read once at the width of the
    form; the dense forms' 18 multiply-adds a pair-mode, or the transforms and products of the convolution form."""
    atoms_i, atoms_p = c["rhs"] * c["n_i"] * c["L"], c["rhs"] * c["n_p"] * c["L"]
    K, p = c["L"] // 2 + 1, c["precision"]
    wide = p in ("fp64", "f32x2", "fft64", "bf16x6")
    nbytes = 24 * atoms_i + 24 * atoms_p * (2 if in_place else 1) + _n_differences(c["n_i"], c["n_p"]) * K * 6 * (8 if wide else 4)
    line = 5.0 * math.log2(c["L"]) / 2 * 3 * (atoms_i + atoms_p)
    if p.startswith("fft"):
        _, a, b = rings(c["n_i"], c["n_p"])
        m = 2 * int(np.abs(a).max() + np.abs(b).max()) + 1
        return nbytes, line + c["rhs"] * K * m * m * (2 * 3 * 5 * math.log2(m * m) / 2 + 36)
    return nbytes, line + 36.0 * c["n_i"] * c["n_p"] * K * c["rhs"]


def work(case):
    c = case
    kind = c["kind"]
    if kind in ("forward", "gradient"):
        H, n = c["width"], c["rows"]
        params, macs = 4 * H + H + 2 * (H * H + H) + 6 * H + 6, 4 * H + 2 * H * H + 6 * H
        if kind == "forward":
            return {"bytes": n * 40 + 2 * params, "flops": 2.0 * n * macs}
        return {"bytes": n * 40 + 8 * params, "flops": 6.0 * n * macs}
    if kind == "batch":
        both = [_update_work(dict(q, precision=c["precision"]), True) for q in _instances(c)]
        return {"bytes": sum(b for b, _ in both), "flops": sum(f for _, f in both)}
    nbytes, flops = _update_work(c, kind == "iteration" or c.get("beta", 0.0) != 0.0)
    if kind == "iteration":
        core, _, _ = rings(c["n_i"], c["n_p"])
        atoms = c["rhs"] * c["L"]
        nbytes += 24 * atoms * (c["n_i"] + (len(core) + c["n_i"] + c["n_p"])) + 24 * atoms * c["n_i"]
        flops += atoms * c["n_i"] * (19 * 18 + 12)
    if kind == "geometry":
        # 2 (n + N) + 1 images of every kept (difference, offset 0..L/2); a closed form, or 64 quadrature nodes each
        evals = _n_differences(c["n_i"], c["n_p"]) * (c["L"] // 2 + 1) * (2 * (RICH_N + RICH_NN) + 1)
        flops += evals * (30 if c["material"] == "isotropic" else 64 * 40)
        nbytes += _n_differences(c["n_i"], c["n_p"]) * (c["L"] // 2 + 1) * 48
    return {"bytes": float(nbytes), "flops": float(flops)}


# ---- the same in 64 bits -------------------------------------------------------------------------------------------------
def _green(m, x, y, z):
    """Continuum Green function at (x, y, z): [..., 6] in the order 11, 12, 22, 33, 13, 23."""
    if m["kind"] == "isotropic":
        r2 = x * x + y * y + z * z
        pre = 1.0 / (16.0 * math.pi * m["mu"] * (1.0 - m["nu"]) * r2.sqrt())
        q = 3.0 - 4.0 * m["nu"]
        return torch.stack([pre * (q + x * x / r2), pre * (x * y / r2), pre * (q + y * y / r2), pre * (q + z * z / r2),
                            pre * (x * z / r2), pre * (y * z / r2)], dim=-1)
    # Barnett's integral over the unit circle normal to r, by the trapezoid rule
    r = (x * x + y * y + z * z).sqrt()
    h = (x * x + y * y).sqrt()
    flat = h > 0
    hs = torch.where(flat, h, torch.ones_like(h))
    one, zero = torch.ones_like(h), torch.zeros_like(h)
    e1 = (torch.where(flat, -y / hs, one), torch.where(flat, x / hs, zero))  # no third component
    cx, cy, cz = x / r, y / r, z / r
    e2 = (-cz * e1[1], cz * e1[0], cx * e1[1] - cy * e1[0])
    c11, c44, s = m["C11"], m["C44"], m["C12"] + m["C44"]
    out = torch.zeros(r.shape + (6,), dtype=r.dtype, device=r.device)
    n = 64
    for j in range(n):
        co, si = math.cos(math.pi * j / n), math.sin(math.pi * j / n)
        n0, n1, n2 = co * e1[0] + si * e2[0], co * e1[1] + si * e2[1], si * e2[2]
        a, b, c = n0 * n0, n1 * n1, n2 * n2
        m0, m1, m2 = c11 * a + c44 * (b + c), c11 * b + c44 * (a + c), c11 * c + c44 * (a + b)
        m01, m02, m12 = s * n0 * n1, s * n0 * n2, s * n1 * n2
        k0, k01, k02 = m1 * m2 - m12 * m12, m02 * m12 - m01 * m2, m01 * m12 - m1 * m02
        det = m0 * k0 + m01 * k01 + m02 * k02
        for t, v in enumerate((k0, k01, m0 * m2 - m02 * m02, m0 * m1 - m01 * m01, k02, m01 * m02 - m0 * m12)):
            out[..., t] += v / det
    return out * (1.0 / (4.0 * math.pi * n * r))[..., None]


def _periodic(m, L, dx, dy):
    """The extrapolated image sum at every difference and offset s = 0 .. L - 1: [n][L][6]."""
    n, N, dev = RICH_N, RICH_NN, dx.device
    w = [(n + i) ** N * (-1) ** (i + N) / (math.factorial(i) * math.factorial(N - i)) for i in range(N + 1)]
    s = torch.arange(L // 2 + 1, dtype=torch.float64, device=dev)
    half = torch.empty((len(dx), L // 2 + 1, 6), dtype=torch.float64, device=dev)
    step = max(1, 20000000 // len(s))
    zero = torch.zeros(1, dtype=torch.float64, device=dev)
    for at in range(0, len(dx), step):
        x, y = dx[at:at + step, None].expand(-1, len(s)), dy[at:at + step, None].expand(-1, len(s))
        z = s[None, :].expand(x.shape[0], -1)
        acc = _green(m, x, y, z)
        for i in range(1, n + N + 1):
            # the weight of all partial sums that hold image i: the increments, not the sums, are extrapolated
            wi = sum(w[max(0, i - n):])
            acc += wi * (_green(m, x, y, z + i * L) + _green(m, x, y, z - i * L)
                         - 2.0 * _green(m, zero, zero, zero + i * L) * torch.tensor([1, 1, 1, 1, 0, 0], device=dev))
        half[at:at + step] = acc
    half[:, L // 2, 4:] = 0.0  # the mean of the two offsets +-L/2
    sign = torch.tensor([1, 1, 1, 1, -1, -1], dtype=torch.float64, device=dev)
    return torch.cat([half, half[:, 1:L // 2].flip(1) * sign], dim=1)


def _good(n):
    while True:
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1:
            return n
        n += 1


def _convolve(c, f):
    """G f at the pad atoms, with the mean force removed: a circular convolution over x, y and the line."""
    _, xy_i, xy_p = rings(c["n_i"], c["n_p"])
    dev, L = f.device, c["L"]
    D = np.abs(xy_i).max(0) + np.abs(xy_p).max(0)
    Mx, My = (_good(2 * int(d) + 1) for d in D)
    used = np.zeros((2 * D[0] + 1, 2 * D[1] + 1), dtype=bool)
    for x, y in xy_p:
        used[x - xy_i[:, 0] + D[0], y - xy_i[:, 1] + D[1]] = True
    d = torch.from_numpy(np.argwhere(used) - D).to(dev)
    T = _periodic(MATERIALS[c["material"]], L, d[:, 0].double(), d[:, 1].double())
    f = f - f.mean(dim=(1, 2), keepdim=True)
    K = L // 2 + 1
    Gk = torch.fft.fft(T, dim=1)[:, :K].contiguous()
    del T
    F = torch.fft.rfft(f, dim=2)
    R = f.shape[0]
    U = torch.empty((R, len(xy_p), K, 3), dtype=torch.complex128, device=dev)
    ii, pp = (torch.from_numpy(a.astype(np.int64)).to(dev) for a in (xy_i, xy_p))
    modes = max(1, int(2.5e8 // (Mx * My * (6 + 6 * R))))
    for k in range(0, K, modes):
        ks = slice(k, min(K, k + modes))
        nk = ks.stop - ks.start
        g = torch.zeros((Mx, My, nk, 6), dtype=torch.complex128, device=dev)
        g[d[:, 0] % Mx, d[:, 1] % My] = Gk[:, ks]
        g = torch.fft.fft2(g, dim=(0, 1))
        for r in range(R):
            a = torch.zeros((Mx, My, nk, 3), dtype=torch.complex128, device=dev)
            a[ii[:, 0] % Mx, ii[:, 1] % My] = F[r, :, ks]
            a = torch.fft.fft2(a, dim=(0, 1))
            b = torch.stack([sum(g[..., t] * a[..., j] for j, t in enumerate(row)) for row in ((0, 1, 4), (1, 2, 5), (4, 5, 3))],
                            dim=-1)
            U[r, :, ks] = torch.fft.ifft2(b, dim=(0, 1))[pp[:, 0] % Mx, pp[:, 1] % My]
    return torch.fft.irfft(U, n=L, dim=2)


def _update(c, f, u, alpha, beta, zero_mean):
    out = beta * u + alpha * _convolve(c, f)
    return out - out.mean(dim=(1, 2), keepdim=True) if zero_mean else out


def _incompat(c, u):
    """Spring forces on the interface: stiffness times the elongation of every bond."""
    sites = rings(c["n_i"], c["n_p"])
    where = {}
    for xy in sites:
        for x, y in xy:
            where[int(x), int(y)] = len(where)
    every = torch.cat(u, dim=1)
    xy_i = sites[1]
    f = torch.zeros_like(u[1])
    for nx in (-1, 0, 1):
        for ny in (-1, 0, 1):
            at = torch.tensor([where[int(x) + nx, int(y) + ny] for x, y in xy_i], device=every.device)
            col = every[:, at]
            for nz in (-1, 0, 1):
                l1 = abs(nx) + abs(ny) + abs(nz)
                if l1 not in (1, 2):
                    continue
                v = torch.tensor([nx, ny, nz], dtype=torch.float64, device=every.device)
                stretch = (u[1] - torch.roll(col, -nz, dims=2)) @ v
                f += (K1 if l1 == 1 else K2) / float(v @ v) * stretch[..., None] * v
    return f


def exact(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind in ("forward", "gradient"):
        p, x, t = _network(c, seed)
        H = c["width"]
        q = torch.from_numpy(p).to(_device())
        q = (q.to(torch.bfloat16) if kind == "forward" else q).double()
        W, o = [], 0
        for a, b in ((4, H), (H, H), (H, H), (H, 6)):
            W.append((q[o:o + a * b].view(a, b).clone(), torch.from_numpy(p).to(q)[o + a * b:o + a * b + b].clone()))
            o += a * b + b
        h = x.double()
        if kind == "gradient":
            for w, b in W:
                w.requires_grad_()
                b.requires_grad_()
        for j, (w, b) in enumerate(W):
            h = h @ w + b
            h = torch.nn.functional.silu(h) if j < 3 else h
        if kind == "forward":
            return h
        loss = ((h - t.double()) ** 2).mean()
        loss.backward()
        return float(loss.detach()), torch.cat([g.grad.reshape(-1) for pair in W for g in pair])
    if kind == "batch":
        out = []
        for j, q in enumerate(_instances(c)):
            f, u = _update_inputs(q, seed, 10 * j)
            out.append(_update(q, f, u, -1.0, 1.0, False))
        return out
    if kind == "iteration":
        u, f_prev = _iteration_inputs(c, seed)
        f = _incompat(c, u)
        g = _convolve(c, f)
        diff = f - f_prev
        alpha = -(f_prev * diff).sum(dim=(1, 2, 3)) / (diff * diff).sum(dim=(1, 2, 3))
        alpha = torch.where(alpha < 0, torch.ones_like(alpha), alpha)
        top = g.abs().amax(dim=(1, 2, 3))
        alpha = torch.where(alpha * top > c["du_max"], c["du_max"] / top, alpha)
        v = u[2] - alpha[:, None, None, None] * g
        return {"f": f, "u": v - v.mean(dim=(1, 2), keepdim=True), "alpha": alpha}
    f, u = _update_inputs(c, seed)
    return _update(c, f, u, c.get("alpha", 1.0), c.get("beta", 0.0), c.get("zero_mean", False))
