"""The two-stage mixed-radix passes (csrc/mix2.cuh) at the lengths where they can go
wrong: both radices above 16, the half-line column tiles of long transforms,
every z radix class, odd row lengths (no paired loads), widths that do not fill
a tile, the full half-length input and output, and the lengths of three stages
that stay with the general kernels. Fields against the oracle's to the tolerances of
the other parity tests (1e-5 FP32, 1e-12 FP64), the gradient with a cell weight
and its energy to 1e-5 / 1e-12 of the oracle's."""
import numpy as np
import pytest
import torch

import oracle
from paper_1204_4302_gb300 import inputs

pytestmark = pytest.mark.gpu

D = (1e-9, 1.2e-9, 0.9e-9)
GRIDS = [
    ((5, 270, 3), (10, 540, 6)),      # y 27 x 20, one column line per tile
    ((7, 480, 2), (14, 960, 4)),      # y 32 x 30, half-line tiles, nin = L / 2
    ((33, 300, 1), (70, 600, 1)),     # y 25 x 24, odd rows, Kx = 36
    ((500, 3, 2), (1000, 6, 4)),      # x 25 x 20, nx = L
    ((147, 5, 2), (294, 10, 4)),      # x 21 x 7, odd nx
    ((9, 4, 240), (18, 8, 480)),      # z 30 x 15 (largest middle radix class)
    ((6, 3, 135), (12, 6, 270)),      # z 27 x 10
    ((10, 9, 49), (20, 18, 98)),      # z 14 x 7
    ((17, 2, 3), (34 + 6, 4, 6)),     # z 3 x 2, x 5 x 4
    ((3, 245, 2), (6, 490, 4)),       # y 490: three stages
    ((3, 2, 252), (6, 4, 504)),       # z 504: no split with R2 <= 16
]


@pytest.mark.parametrize("prec,tol", [("f32", 1e-5), ("f64", 1e-12)])
@pytest.mark.parametrize("n,pad", GRIDS)
def test_two_stage_lengths(n, pad, prec, tol):
    from paper_1204_4302_gb300.plan import Plan
    dt = torch.float32 if prec == "f32" else torch.float64
    Ms = 8e5
    m = inputs.random_unit(n, seed=sum(n))
    rng = np.random.default_rng(7)
    w = rng.uniform(0.0, 1.0, m.shape[1:])
    plan = Plan(n, D, prec=prec, pad=pad)
    try:
        H, E = plan.field_energy(torch.tensor(Ms * m, dtype=dt, device="cuda"))
        Href = oracle.field_fft(Ms * m, D)
        assert np.max(np.abs(H.double().cpu().numpy() - Href)) <= tol * np.max(np.abs(Href))
        Eref = oracle.energy(Ms * m, Href, D)
        assert abs(E.item() - Eref) <= tol * abs(Eref)
        Eg, G = plan.energy_grad(torch.tensor(m, dtype=dt, device="cuda"), Ms,
                                 torch.tensor(w, dtype=dt, device="cuda"))
        Hw = oracle.field_fft(Ms * w * m, D)
        Gref = -oracle.MU0 * D[0] * D[1] * D[2] * Ms * w * Hw
        assert np.max(np.abs(G.double().cpu().numpy() - Gref)) <= tol * np.max(np.abs(Gref))
        Ew = oracle.energy(Ms * w * m, Hw, D)
        assert abs(Eg.item() - Ew) <= tol * abs(Ew)
    finally:
        plan.close()
