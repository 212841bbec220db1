"""The small-tile z pass (csrc/zt.cuh; z variant 8 of FP32 plans, z lengths 32, 64 and
128) and the persistent SP z pass (csrc/spws.cuh, z lengths 256 and 512): ragged column
tiles, one ky row, nz at and below half the length, the wide and the narrow tiles.
Fields to 1e-5 of the oracle's (the SP field to 4 eps log2(prod P)(1 + A), A its
amplification, as in the SP parity tests); energies by all three routes to 1e-5."""
import numpy as np
import pytest
import torch

import oracle
from paper_1204_4302_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(16, 16, 16), (9, 1, 9), (70, 33, 15), (7, 130, 16),   # L = 32 (narrow, one row, wide)
                               (12, 9, 17), (40, 20, 32),                              # L = 64
                               (5, 3, 64), (33, 17, 33), (66, 70, 40)])                # L = 128
def test_small_tile_z_pass(n):
    from paper_1204_4302_gb300.plan import Plan
    d, Ms = (2e-9, 1.5e-9, 1e-9), 8e5
    M = Ms * inputs.random_unit(n, seed=5)
    Href = oracle.field_fft(M, d)
    Eref = oracle.energy(M, Href, d)
    p = Plan(n, d, prec="f32")
    try:
        Mt = torch.tensor(M, dtype=torch.float32, device="cuda")
        for x in (0, 2):
            p.set_variants(8, 0, x)
            assert p.info()["energy_in_z"] == 1
            H, E = p.field_energy(Mt)
            assert np.max(np.abs(H.double().cpu().numpy() - Href)) <= 1e-5 * np.max(np.abs(Href))
            assert torch.equal(H, p.field(Mt))
            Es = p.energy(Mt)
            p.set_spectral_energy(False)
            _, Ex = p.field_energy(Mt)
            p.set_spectral_energy(True)
            for e in (E.item(), Es, Ex.item()):
                assert abs(e - Eref) <= 1e-5 * abs(Eref)
    finally:
        p.close()


@pytest.mark.parametrize("n", [(9, 5, 128), (3, 17, 100), (20, 1, 65), (6, 7, 256), (17, 3, 129)])
def test_persistent_sp_z_pass(n):
    from paper_1204_4302_gb300.plan import Plan
    d, Ms = (1e-9, 1.2e-9, 1e-9), 8e5
    M = Ms * inputs.random_unit(n, seed=6)
    Href = oracle.sp_field(M, d)
    p = Plan(n, d, prec="f32", method="sp")
    try:
        Mt = torch.tensor(M, dtype=torch.float32, device="cuda")
        phi = p.potential(Mt).double().cpu().numpy()
        H = p.field(Mt).double().cpu().numpy()
        A = np.max(np.abs(phi)) / (np.max(np.abs(Href)) * min(d))
        i = p.info()
        tol = 4 * np.finfo(np.float32).eps * np.log2(i["px"] * i["py"] * i["pz"]) * (1 + A)
        assert np.max(np.abs(H - Href)) <= tol * np.max(np.abs(Href))
        p.check_pipeline()
    finally:
        p.close()
