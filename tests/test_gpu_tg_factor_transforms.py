"""Tensor-grid factor transforms at the edges of their launches: the longest row (512),
rows around a block of outputs, axes and ranks far apart, against the oracle's
potential. FP64 to 1e-12; FP32 to 16 sqrt(K) roundings, K the contraction's terms."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from oracle import tensor_grid as tg  # noqa: E402


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("n,r", [((512, 5, 3), 1), ((3, 33, 300), 9), ((16, 4, 257), 5), ((129, 128, 4), 2)])
def test_potential_matches_oracle(n, r, prec):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1204_4302_gb300 import build
    from paper_1204_4302_gb300.tg import TGPlan
    build.build()
    d = (2e-9, 1.5e-9, 2.5e-9)
    rng = np.random.default_rng(sum(n) + r)
    lam, U = 8e5 * rng.standard_normal((3, r)), [rng.standard_normal((3, r, v)) for v in n]
    M = np.stack([tg.cp_to_dense(lam[p], *(u[p].T for u in U)) for p in range(3)])
    ref = tg.cell_potential_fft(M, d, oracle.sp_kernel)
    p = TGPlan(n, d, r, prec=prec)
    dt = torch.float32 if prec == "f32" else torch.float64
    got = p.potential(*(torch.tensor(a, dtype=dt, device="cuda") for a in (lam, *U))).double().cpu().numpy()
    tol = 1e-12 if prec == "f64" else 16 * 2.0 ** -24 * math.sqrt(3 * p.info()["sinc_terms"] * r)
    assert np.max(np.abs(got - ref)) <= tol * np.max(np.abs(ref))
    p.close()
