"""Workloads of the stray-field library, for measuring it.

Each case is one call (or one forward and backward pair of calls) that a micromagnetic program makes once
per step: the field of a magnetization it holds on the GPU through a plan it keeps. ``prepare`` makes
the state and the plan, ``run`` the call, ``exact`` the same result in 64 bits from plain torch.

Case values: ``kind`` "grid" (one dense state: method "dm" or "sp"), "batch" (many states of uneven
sizes) or "tg" (a CP magnetization). ``op`` of a grid case:
  field         H(M), what every stage of a time integrator needs
  field_energy  H(M) and E, a step that also logs the energy
  gradient      E(m) and dE/dm through autograd, a minimiser's or an optimiser's step
  adjoint       H(M) and the adjoint applied to an upstream gradient through autograd, the
                forward and backward of a field-matching loss
Energies of FP32 plans are logged in float32, the precision of the field that they belong to.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1204_4302_gb300 import inputs
from paper_1204_4302_gb300.autograd import DemagEnergy, DemagField
from paper_1204_4302_gb300.batch import Batch
from paper_1204_4302_gb300.plan import Plan
from paper_1204_4302_gb300.tg import TGPlan

MS = 8e5  # A/m, permalloy
MU0 = 4e-7 * math.pi
DEV = "cuda"


def _grid(name, n, op, state="random", prec="f32", method="dm", pad="pow2", tune=True, edge=2e-9, flat=1.0):
    """edge: cell edge along x and y (m); flat: the edge along z over it."""
    return {"name": name, "kind": "grid", "nx": n[0], "ny": n[1], "nz": n[2], "op": op, "state": state,
            "prec": prec, "method": method, "pad": pad, "tune": tune, "edge": edge, "flat": flat}


def listed():
    return [
        # a single small particle in a time loop, the plan as it is created: latency and launches
        _grid("cube16", (16, 16, 16), "field", tune=False, edge=1e-9),
        # a thin film with a vortex: the common geometry, a handful of layers
        _grid("film_512x128x4", (512, 128, 4), "field_energy", state="vortex"),
        # a sphere on a staircase grid (cells outside carry no moment), one minimiser step
        _grid("sphere64_gradient", (64, 64, 64), "gradient", state="sphere"),
        # a medium cube, one minimiser step over all its cells
        _grid("cube128_gradient", (128, 128, 128), "gradient"),
        # a size just above a power of two, padded to the smallest smooth lengths
        _grid("cube130_smooth", (130, 130, 130), "field_energy", pad="smooth"),
        # an uneven slab whose padding the library chooses for each axis
        _grid("slab_300x260x100", (300, 260, 100), "field_energy", state="smooth", pad="tuned"),
        # the benchmark's grid
        _grid("cube256", (256, 256, 256), "field_energy"),
        # a large film, forward and backward of a loss on the field
        _grid("film_512x512x128_adjoint", (512, 512, 128), "adjoint", state="smooth", edge=1e-9),
        # a double-precision reference run
        _grid("cube64_f64", (64, 64, 64), "field_energy", prec="f64"),
        # the benchmark's grid by the scalar potential
        _grid("cube256_sp", (256, 256, 256), "field_energy", method="sp"),
        # the benchmark's grid from a low-rank magnetization
        {"name": "tg256_rank8", "kind": "tg", "nx": 256, "ny": 256, "nz": 256, "rank": 8, "prec": "f32", "edge": 2e-9},
        # an ensemble of independent particles of uneven sizes
        {"name": "batch64", "kind": "batch", "count": 64, "sizes": 4, "edge": 3e-9},
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49))))))


def _pow2(n):
    return 1 << (2 * n - 2).bit_length() if n > 1 else 1


def draw(rng):
    what = rng.choices(("f32", "f64", "sp", "tg", "batch"), (11, 2, 3, 2, 2))[0]
    if what == "batch":
        return {"kind": "batch", "count": rng.randint(8, 64), "sizes": rng.randint(5, 10 ** 6), "edge": 3e-9}
    if what == "tg":
        return {"kind": "tg", "nx": _log(rng, 32, 256), "ny": _log(rng, 32, 256), "nz": _log(rng, 8, 256),
                "rank": _log(rng, 1, 12), "prec": "f32", "edge": 2e-9}
    most = 128 ** 3 if what == "f64" else 256 ** 3
    while True:
        top = 128 if what == "f64" else 512
        n = (_log(rng, 16, top), _log(rng, 16, top), _log(rng, 1 if what != "sp" else 4, min(top, 256)))
        if n[0] * n[1] * n[2] <= most and _pow2(n[0]) * _pow2(n[1]) * _pow2(n[2]) <= 16 * most:
            break
    op = "field_energy" if what == "sp" else rng.choice(("field", "field_energy", "gradient", "adjoint"))
    pad = rng.choice(("pow2", "pow2", "smooth")) if what == "sp" else rng.choice(("pow2", "pow2", "smooth", "tuned"))
    c = _grid("", n, op, state=rng.choice(("random", "smooth", "vortex")), prec="f64" if what == "f64" else "f32",
              method="sp" if what == "sp" else "dm", pad=pad, tune=rng.random() < 0.7,
              flat=rng.choice((1.0, 1.0, 0.5, 2.0)))
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
def _dtype(case):
    return torch.float64 if case.get("prec") == "f64" else torch.float32


def _shape(case):
    return (3, case["nz"], case["ny"], case["nx"])


def _edges(case):
    return (case["edge"], case["edge"], case["edge"] * case.get("flat", 1.0))


def _unit(m):
    return m / m.square().sum(0, keepdim=True).sqrt().clamp_min(1e-30)


def _magnetization(shape, state, g):
    """Unit vectors per cell, float64: independent directions ("random", "sphere"), a texture of some 8 cells
    ("smooth"), or a vortex about z with 5% of noise ("vortex")."""
    m = torch.randn(shape, generator=g, dtype=torch.float64, device=DEV)
    if state == "smooth":
        f = torch.fft.rfftn(m, dim=(1, 2, 3))
        for axis in (1, 2, 3):
            k = torch.fft.rfftfreq(shape[3], dtype=torch.float64, device=DEV) if axis == 3 else \
                torch.fft.fftfreq(shape[axis], dtype=torch.float64, device=DEV)
            view = [1, 1, 1, 1]
            view[axis] = -1
            f *= torch.exp(-2.0 * (math.pi * 8.0 * k) ** 2).view(view)
        m = torch.fft.irfftn(f, s=shape[1:], dim=(1, 2, 3))
    elif state == "vortex":
        y = (torch.arange(shape[2], dtype=torch.float64, device=DEV) + 0.5 - 0.5 * shape[2])[:, None]
        x = (torch.arange(shape[3], dtype=torch.float64, device=DEV) + 0.5 - 0.5 * shape[3])[None, :]
        r2 = x * x + y * y
        rc2 = (0.14 * min(shape[2], shape[3])) ** 2
        turn = torch.sqrt(1.0 - torch.exp(-4.0 * r2 / rc2)) / r2.sqrt().clamp_min(1e-9)
        m = 0.05 * m + torch.stack([-y * turn, x * turn, torch.exp(-2.0 * r2 / rc2)])[:, None]
    return _unit(m)


def _grid_inputs(case, seed):
    """(m or M, weight or None, upstream gradient or None) in the plan's precision."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    shape, dt = _shape(case), _dtype(case)
    m = _magnetization(shape, case["state"], g)
    w = None
    if case["state"] == "sphere":
        at = [torch.arange(n, dtype=torch.float64, device=DEV) + 0.5 - 0.5 * n for n in shape[1:]]
        r2 = at[0][:, None, None] ** 2 + at[1][None, :, None] ** 2 + at[2][None, None, :] ** 2
        w = (r2 < (0.5 * min(shape[1:])) ** 2).to(dt)
    up = None
    if case["op"] == "adjoint":  # the difference to a target field
        up = (MS * torch.randn(shape, generator=g, dtype=torch.float64, device=DEV)).to(dt)
    if case["op"] != "gradient":
        m = MS * m if w is None else MS * m * w
    return m.to(dt), w, up


def _batch_dims(case):
    return inputs.batch_sizes(case["count"], seed=case["sizes"])


def _batch_inputs(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return [(MS * _magnetization((3, nz, ny, nx), "random", g)).float() for nx, ny, nz in _batch_dims(case)]


def _tg_inputs(case, seed):
    """CP factors of entries of about 1, the weights falling with the term as those of a compression do."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    r, dt = case["rank"], _dtype(case)

    def columns(n):
        return torch.randn((3, r, n), generator=g, dtype=torch.float64, device=DEV).to(dt)

    lam = MS * 0.7 ** torch.arange(r, dtype=torch.float64, device=DEV)
    lam = (lam * (0.5 + torch.rand((3, r), generator=g, dtype=torch.float64, device=DEV))).to(dt)
    return lam, columns(case["nx"]), columns(case["ny"]), columns(case["nz"])


# ------------------------------------------------------------------ the calls
def prepare(case, seed):
    if case["kind"] == "tg":
        plan = TGPlan((case["nx"], case["ny"], case["nz"]), _edges(case), case["rank"], prec=case["prec"])
        return {"case": case, "plan": plan, "factors": _tg_inputs(case, seed), "log": torch.zeros((), device=DEV)}
    if case["kind"] == "batch":
        dims = _batch_dims(case)
        batch = Batch(dims, [_edges(case)] * len(dims))
        batch.autotune()
        sizes = [3 * nx * ny * nz for nx, ny, nz in dims]
        # the states' fields in one allocation, each on a 16-byte boundary
        at = np.concatenate([[0], np.cumsum([(s + 3) // 4 * 4 for s in sizes])])
        flat = torch.zeros(int(at[-1]), device=DEV)
        H = [flat[int(a):int(a) + s].view(3, nz, ny, nx) for a, s, (nx, ny, nz) in zip(at, sizes, dims)]
        return {"case": case, "batch": batch, "M": _batch_inputs(case, seed), "H": H, "flat": flat,
                "log": torch.zeros(len(dims), device=DEV)}
    M, w, up = _grid_inputs(case, seed)
    plan = Plan((case["nx"], case["ny"], case["nz"]), _edges(case), prec=case["prec"], pad=case["pad"],
                method=case["method"])
    if case["tune"]:
        plan.autotune()
    state = {"case": case, "plan": plan, "M": M, "w": w, "up": up}
    if case["op"] in ("gradient", "adjoint"):
        M.requires_grad_()
    else:
        state["H"] = torch.zeros_like(M)
    if case["prec"] == "f32":
        state["log"] = torch.zeros((), device=DEV)
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "tg":
        H, E = state["plan"].field(*state["factors"], energy=True)
        return {"H": H, "E": state["log"].copy_(E)}
    if case["kind"] == "batch":
        _, E = state["batch"].field(state["M"], state["H"], energies=True)
        return {"H": state["flat"], "E": state["log"].copy_(E)}
    plan, M = state["plan"], state["M"]
    if case["op"] == "field":
        return {"H": plan.field(M, out=state["H"])}
    if case["op"] == "field_energy":
        H, E = plan.field_energy(M, out=state["H"])
        return {"H": H, "E": state["log"].copy_(E) if "log" in state else E}
    M.grad = None
    if case["op"] == "gradient":
        E = DemagEnergy.apply(M, MS, state["w"], plan)
        E.backward()
        return {"E": state["log"].copy_(E.detach()) if "log" in state else E.detach(), "grad": M.grad}
    H = DemagField.apply(M, plan)
    H.backward(state["up"])
    return {"H": H.detach(), "grad": M.grad}


# ------------------------------------------------------------------ least work
def _field_work(n, elem, comps=6):
    """One convolution: the state read and the field written once, the kernel (comps components at every
    offset of one octant) read once; three real transforms each way of the doubled grid and the product."""
    cells = n[0] * n[1] * n[2]
    points = 8 * cells
    return (6 + comps) * elem * cells, 6 * 2.5 * points * math.log2(points) + 15 * points


def work(case):
    if case["kind"] == "batch":
        b, f = zip(*(_field_work(n, 4) for n in _batch_dims(case)))
        return {"bytes": sum(b), "flops": sum(f)}
    n = (case["nx"], case["ny"], case["nz"])
    cells = n[0] * n[1] * n[2]
    elem = 8 if case["prec"] == "f64" else 4
    if case["kind"] == "tg":
        # about 100 terms of the exponential sum, three components of `rank` terms each
        return {"bytes": 3 * elem * cells, "flops": 2.0 * cells * 300 * case["rank"]}
    b, f = _field_work(n, elem, 6 if case["method"] == "dm" else 3)
    if case["op"] in ("gradient", "adjoint"):  # two calls
        b, f = 2 * b, 2 * f
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ 64-bit results
def _tent_rule(m):
    """m-point Gauss rule of the weight 1 - |u| on [-1, 1] (Golub and Welsch)."""
    x, w = np.polynomial.legendre.leggauss(40)
    x = np.concatenate([(x - 1) / 2, (x + 1) / 2])
    w = np.concatenate([w, w]) / 2 * (1 - np.abs(x))
    prev, cur, b = np.zeros_like(x), np.ones_like(x) / math.sqrt(w.sum()), []
    for _ in range(m - 1):
        nxt = x * cur - (b[-1] * prev if b else 0.0)
        b.append(math.sqrt(np.sum(w * nxt * nxt)))
        prev, cur = cur, nxt / b[-1]
    t, v = np.linalg.eigh(np.diag(b, 1) + np.diag(b, -1))
    return t, v[0] ** 2 * w.sum()


def _newell(x, y, z):
    """Newell, Williams and Dunlop's f and g (J. Geophys. Res. 98, 1993) at points of any sign."""
    r2 = x * x + y * y + z * z
    r = torch.sqrt(r2)

    def ash(a, b2):  # asinh(a / b), with the limit 0 of its products at b = 0
        b = torch.sqrt(b2)
        return torch.where(b > 0, torch.asinh(a / torch.where(b > 0, b, 1.0)), 0.0)

    def at(a, b):
        return torch.where(b != 0, torch.atan(a / torch.where(b != 0, b, 1.0)), 0.0)

    f = (0.5 * y * (z * z - x * x) * ash(y, x * x + z * z) + 0.5 * z * (y * y - x * x) * ash(z, x * x + y * y)
         - x * y * z * at(y * z, x * r) + (2 * x * x - y * y - z * z) * r / 6)
    g = (x * y * z * ash(z, x * x + y * y) + y / 6 * (3 * z * z - y * y) * ash(x, y * y + z * z)
         + x / 6 * (3 * z * z - x * x) * ash(y, x * x + z * z) - z ** 3 / 6 * at(x * y, z * r)
         - z * y * y / 2 * at(x * z, y * r) - z * x * x / 2 * at(y * z, x * r) - x * y * r / 3)
    return f, g


_PAIRS = ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))


def _tensor_at(R, d):
    """Cell-averaged demagnetization tensor, 6 components, at the offsets R (3, k): second differences of f and
    g nearer than 6 edges, beyond it Gauss rules of the tent-weighted point dipole."""
    out = torch.zeros((6, R.shape[1]), dtype=torch.float64, device=DEV)
    dist = torch.sqrt((R * R).sum(0)) / max(d)
    near = torch.nonzero(dist < 6.0).squeeze(1)
    if near.numel():
        P = R[:, near]
        for a, wa in ((-1, 1.0), (0, -2.0), (1, 1.0)):
            for b, wb in ((-1, 1.0), (0, -2.0), (1, 1.0)):
                for c, wc in ((-1, 1.0), (0, -2.0), (1, 1.0)):
                    q = (P[0] + a * d[0], P[1] + b * d[1], P[2] + c * d[2])
                    s = -wa * wb * wc / (4 * math.pi * d[0] * d[1] * d[2])
                    for k, (i, j) in enumerate(_PAIRS):
                        o = 3 - i - j if i != j else None
                        if i == j:
                            v = _newell(q[i], q[(i + 1) % 3], q[(i + 2) % 3])[0]
                        else:
                            v = _newell(q[i], q[j], q[o])[1]
                        out[k, near] += s * v
    for lo, hi, m in ((6.0, 16.0, 8), (16.0, 64.0, 4), (64.0, math.inf, 3)):
        sel = torch.nonzero((dist >= lo) & (dist < hi)).squeeze(1)
        if not sel.numel():
            continue
        P, acc = R[:, sel], torch.zeros((6, sel.numel()), dtype=torch.float64, device=DEV)
        t, w = _tent_rule(m)
        for a in range(m):
            X = P[0] - float(t[a]) * d[0]
            for b in range(m):
                Y = P[1] - float(t[b]) * d[1]
                for c in range(m):
                    Z = P[2] - float(t[c]) * d[2]
                    q = (X, Y, Z)
                    inv2 = 1.0 / (X * X + Y * Y + Z * Z)
                    s = inv2 * torch.sqrt(inv2) * (-float(w[a] * w[b] * w[c]) * d[0] * d[1] * d[2] / (4 * math.pi))
                    t3 = 3.0 * s * inv2
                    for k, (i, j) in enumerate(_PAIRS):
                        acc[k].addcmul_(t3 * q[i], q[j])
                    acc[:3] -= s
        out[:, sel] = acc
    return out


def _cell_kernel_at(R, d):
    """S (3, k): the potential at R of a cell of unit magnetization along each axis, the difference of its two
    charged faces' potentials nearer than 6 edges, beyond it a Gauss rule over the cell."""
    out = torch.zeros((3, R.shape[1]), dtype=torch.float64, device=DEV)
    dist = torch.sqrt((R * R).sum(0)) / max(d)
    near = torch.nonzero(dist < 6.0).squeeze(1)
    if near.numel():
        P = R[:, near]
        for j in range(3):
            p, q = (j + 1) % 3, (j + 2) % 3
            for sj in (-1, 1):
                h = P[j] - sj * d[j] / 2
                for sp in (-1, 1):
                    for sq in (-1, 1):
                        a, b = sp * d[p] / 2 - P[p], sq * d[q] / 2 - P[q]
                        r = torch.sqrt(a * a + b * b + h * h)

                        def ash(u, v2):
                            v = torch.sqrt(v2)
                            return torch.where(v > 0, torch.asinh(u / torch.where(v > 0, v, 1.0)), 0.0)

                        den = h.abs() * r
                        v = (a * ash(b, a * a + h * h) + b * ash(a, b * b + h * h)
                             - h.abs() * torch.where(den > 0, torch.atan(a * b / torch.where(den > 0, den, 1.0)), 0.0))
                        out[j, near] += sj * sp * sq * v / (4 * math.pi)
    for lo, hi, m in ((6.0, 16.0, 7), (16.0, 64.0, 4), (64.0, math.inf, 3)):
        sel = torch.nonzero((dist >= lo) & (dist < hi)).squeeze(1)
        if not sel.numel():
            continue
        P, acc = R[:, sel], torch.zeros((3, sel.numel()), dtype=torch.float64, device=DEV)
        t, w = np.polynomial.legendre.leggauss(m)
        for a in range(m):
            X = P[0] - float(t[a]) * d[0] / 2
            for b in range(m):
                Y = P[1] - float(t[b]) * d[1] / 2
                for c in range(m):
                    Z = P[2] - float(t[c]) * d[2] / 2
                    inv2 = 1.0 / (X * X + Y * Y + Z * Z)
                    s = inv2 * torch.sqrt(inv2) * (float(w[a] * w[b] * w[c]) / 8 * d[0] * d[1] * d[2] / (4 * math.pi))
                    for k, q in enumerate((X, Y, Z)):
                        acc[k].addcmul_(s, q)
        out[:, sel] = acc
    return out


def _offsets(lo, n, half, d):
    """Offsets (k + half) d, lo <= k < lo + n[axis], as (3, nz ny nx)."""
    ax = [(torch.arange(n[a], dtype=torch.float64, device=DEV) + lo + half) * d[a] for a in range(3)]
    z, y, x = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
    return torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)])


def _smooth(p):
    while True:
        q = p
        for f in (2, 3, 5):
            while q % f == 0:
                q //= f
        if q == 1:
            return p
        p += 1


def _wrap(octant, sign, P):
    """A component of parity sign[axis] on the periodic grid P (z, y, x) from its values at offsets >= 0."""
    full = torch.zeros(P, dtype=torch.float64, device=DEV)
    n = octant.shape
    for fz in (0, 1):
        for fy in (0, 1):
            for fx in (0, 1):
                if (fz and n[0] < 2) or (fy and n[1] < 2) or (fx and n[2] < 2):
                    continue
                s, v, at = 1.0, octant, []
                for axis, f in enumerate((fz, fy, fx)):
                    if f:
                        s *= sign[2 - axis]
                        v = torch.flip(v.narrow(axis, 1, n[axis] - 1), (axis,))
                        at.append(slice(P[axis] - n[axis] + 1, P[axis]))
                    else:
                        at.append(slice(0, n[axis]))
                full[tuple(at)] = s * v
    return full


def _tensor_octant(n, d):
    top = max(d)
    e = tuple(v / top for v in d)
    out = torch.empty((6, n[2], n[1], n[0]), dtype=torch.float64, device=DEV)
    step = max(1, (1 << 22) // (n[0] * n[1]))
    for z in range(0, n[2], step):
        k = min(step, n[2] - z)
        R = _offsets(0, (n[0], n[1], k), 0.0, e)
        R[2] += z * e[2]
        out[:, z:z + k] = _tensor_at(R, e).view(6, k, n[1], n[0])
    return out


def _tensor_spectrum(octant, P):
    """Real spectra of the six components (they are even in all: real, or minus real times two odd axes)."""
    sign = ((1, 1, 1), (1, 1, 1), (1, 1, 1), (-1, -1, 1), (-1, 1, -1), (1, -1, -1))
    return [torch.fft.rfftn(_wrap(octant[k], sign[k], P)).real.contiguous() for k in range(6)]


def _apply_tensor(spec, M, P):
    """-N * M for M (3, nz, ny, nx) in float64."""
    f = [torch.fft.rfftn(M[c], s=P) for c in range(3)]
    at = {(i, j): k for k, (i, j) in enumerate(_PAIRS)}
    H = torch.empty_like(M)
    for i in range(3):
        h = sum(spec[at[(min(i, j), max(i, j))]] * f[j] for j in range(3))
        H[i] = -torch.fft.irfftn(h, s=P)[:M.shape[1], :M.shape[2], :M.shape[3]]
    return H


def _energy(M, H, d):
    return -0.5 * MU0 * d[0] * d[1] * d[2] * (M * H).sum()


def _potential(M, d, half):
    """S * M at the cell centres (half = 0) or at the nodes (half = 1, one more per axis)."""
    top = max(d)
    e = tuple(v / top for v in d)
    n = (M.shape[3], M.shape[2], M.shape[1])
    P = tuple(_smooth(2 * v + half) for v in reversed(n))
    total = 0
    for c in range(3):
        # offsets from -(n - 1) (or -n + 1/2 with nodes) to n - 1 (n - 1/2)
        count = tuple(2 * v - 1 + half for v in n)
        k = torch.empty((count[2], count[1], count[0]), dtype=torch.float64, device=DEV)
        step = max(1, (1 << 23) // (count[0] * count[1]))
        for z in range(0, count[2], step):
            m = min(step, count[2] - z)
            ax = [(torch.arange(count[a], dtype=torch.float64, device=DEV) - (n[a] - 1) - 0.5 * half) * e[a]
                  for a in range(3)]
            Z, Y, X = torch.meshgrid(ax[2][z:z + m], ax[1], ax[0], indexing="ij")
            R = torch.stack([X.reshape(-1), Y.reshape(-1), Z.reshape(-1)])
            k[z:z + m] = _cell_kernel_at(R, e)[c].view(m, count[1], count[0])
        total = total + torch.fft.rfftn(k, s=P) * torch.fft.rfftn(M[c], s=P)
    full = torch.fft.irfftn(total, s=P)
    at = tuple(slice(v - 1, 2 * v - 1 + half) for v in reversed(n))
    return full[at] * top


def _exact_sp(M, d):
    phi = _potential(M, d, 1)

    def mean(v, axis):
        return 0.5 * (v.narrow(axis, 0, v.shape[axis] - 1) + v.narrow(axis, 1, v.shape[axis] - 1))

    H = []
    for axis, edge in ((2, d[0]), (1, d[1]), (0, d[2])):
        v = torch.diff(phi, dim=axis) / edge
        for other in range(3):
            if other != axis:
                v = mean(v, other)
        H.append(-v)
    return torch.stack(H)


def _exact_tg(M, d):
    phi = _potential(M, d, 0)
    return torch.stack([-torch.gradient(phi, spacing=d[2 - axis], dim=axis, edge_order=2)[0] for axis in (2, 1, 0)])


def exact(case, seed):
    d = _edges(case)
    if case["kind"] == "tg":
        lam, X, Y, Z = (t.double() for t in _tg_inputs(case, seed))
        M = torch.einsum("pm,pmk,pmj,pmi->pkji", lam, Z, Y, X)
        H = _exact_tg(M, d)
        return {"H": H, "E": _energy(M, H, d)}
    if case["kind"] == "batch":
        dims, flat, E = _batch_dims(case), [], []
        top = tuple(max(n[a] for n in dims) for a in range(3))
        octant = _tensor_octant(top, d)
        for M, n in zip(_batch_inputs(case, seed), dims):
            P = tuple(_smooth(2 * v) for v in reversed(n))
            M = M.double()
            H = _apply_tensor(_tensor_spectrum(octant[:, :n[2], :n[1], :n[0]], P), M, P)
            E.append(_energy(M, H, d))
            H = H.reshape(-1)
            flat.append(torch.cat([H, H.new_zeros(-H.numel() % 4)]))
        return {"H": torch.cat(flat), "E": torch.stack(E)}
    M, w, up = _grid_inputs(case, seed)
    M = M.double()
    if case["method"] == "sp":
        H = _exact_sp(M, d)
        return {"H": H, "E": _energy(M, H, d)}
    n = (case["nx"], case["ny"], case["nz"])
    P = tuple(_smooth(2 * v) for v in reversed(n))
    spec = _tensor_spectrum(_tensor_octant(n, d), P)
    if case["op"] == "field":
        return {"H": _apply_tensor(spec, M, P)}
    if case["op"] == "field_energy":
        H = _apply_tensor(spec, M, P)
        return {"H": H, "E": _energy(M, H, d)}
    if case["op"] == "gradient":
        scale = MS if w is None else MS * w.double()
        H = _apply_tensor(spec, scale * M, P)
        return {"E": _energy(scale * M, H, d), "grad": -MU0 * d[0] * d[1] * d[2] * scale * H}
    return {"H": _apply_tensor(spec, M, P), "grad": _apply_tensor(spec, up.double(), P)}
