"""Kernel forms (z, y, x) that a plan starts with: by precision and padded lengths, the
ones that were the fastest there (FP64 y form 2 at length 512 but not at 1024)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,prec,forms", [
    ((4, 300, 3), "f64", (0, 0, 1)),     # y 1024
    ((4, 512, 30), "f64", (8, 0, 1)),
    ((4, 200, 3), "f64", (0, 2, 1)),     # y 512
    ((4, 100, 3), "f64", (0, 0, 1)),
    ((4, 300, 3), "f32", (0, 0, 2)),
    ((4, 20, 100), "f32", (6, 0, 2)),
])
def test_default_forms(n, prec, forms):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1204_4302_gb300 import build
    from paper_1204_4302_gb300.plan import Plan
    build.build()
    p = Plan(n, (2e-9,) * 3, prec=prec, setup=False)
    assert (*p.variants(), p.x_variant()) == forms
    p.close()
