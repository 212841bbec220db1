"""The inverse x pass of 16 and 32 points in its wide form (256-thread CTAs, taken where
these are at least two per SM) with the energy taken there (M rows by
asynchronous copies, or plain loads where nx is not a multiple of 16 bytes), and
with the extra node column of scalar-potential plans, against the FP64 oracle; the
two small grids run the one-warp form."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_1204_4302_gb300 import inputs  # noqa: E402

MS = 8e5
D = (2e-9, 1.5e-9, 2.5e-9)


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1204_4302_gb300 import build
    build.build()


# rows 3 ny nz: 152 SMs x 2 wide CTAs of 64 (L = 16) or 32 (L = 32) rows in FP32,
# half of that in FP64, are 19456 and 9728 rows
@pytest.mark.parametrize("prec,tol", [("f32", 1e-5), ("f64", 1e-12)])
@pytest.mark.parametrize("n", [(16, 100, 70), (13, 100, 70), (32, 80, 50), (31, 80, 50), (16, 40, 20), (32, 40, 20)])
def test_field_energy_in_the_x_pass(n, prec, tol):
    from paper_1204_4302_gb300.plan import Plan
    M = MS * inputs.random_unit(n, seed=sum(n))
    Href = oracle.field_fft(M, D)
    Eref = oracle.energy(M, Href, D)
    p = Plan(n, D, prec=prec)
    p.set_spectral_energy(False)
    assert not p.info()["energy_in_z"]
    Mt = torch.tensor(M, dtype=p.dtype, device="cuda")
    for x in (0, 2):
        p.set_variants(*p.variants(), x)
        H, E = p.field_energy(Mt)
        rel = np.max(np.abs(H.double().cpu().numpy() - Href)) / np.max(np.abs(Href))
        assert rel <= tol, (x, rel)
        assert abs(E.item() - Eref) <= 10 * tol * abs(Eref), (x, E.item(), Eref)
    p.close()


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("n", [(16, 140, 140), (32, 100, 100)])
def test_sp_node_rows_in_the_wide_form(n, prec):
    """(nz + 1)(ny + 1) rows of nx + 1 = L + 1 values; FP32 to eight roundings per
    transform level, as the other potentials are."""
    from paper_1204_4302_gb300.plan import Plan
    M = MS * inputs.random_unit(n, seed=sum(n))
    phi_ref = oracle.sp_potential_fft(M, D)
    tol = 1e-12 if prec == "f64" else 8 * 2.0 ** -24 * math.log2(np.prod([oracle.sp_padded_size(v) for v in n]))
    p = Plan(n, D, prec=prec, method="sp")
    phi = p.potential(torch.tensor(M, dtype=p.dtype, device="cuda")).double().cpu().numpy()
    assert np.max(np.abs(phi - phi_ref)) <= tol * np.max(np.abs(phi_ref))
    p.close()
