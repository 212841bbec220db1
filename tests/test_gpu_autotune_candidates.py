"""The autotuner times each kernel form that exists for a plan once: the launches
of a tuning run are (calls per candidate) x (candidates) x (kernels per call)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CALLS = 7  # two warm-up and five timed field + energy calls per candidate


@pytest.mark.parametrize("n,method,pad,candidates", [
    ((40, 33, 20), "dm", "smooth", 1),     # mixed-radix lengths have one form
    ((20, 20, 32), "dm", None, 2 * 6),     # z 64: forms 0, 1, 3, 4, 5, 8; two x forms
    ((20, 20, 128), "dm", None, 2 * 7),    # z 256: 0, 1, 3, 4, 5, 6, 7
    ((20, 20, 128), "sp", None, 2),        # SP at z 256: one form
    ((20, 20, 32), "sp", None, 2 * 2),     # SP at z 64: 0 and 5
])
def test_autotune_times_each_form_once(n, method, pad, candidates):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1204_4302_gb300 import build
    from paper_1204_4302_gb300.plan import Plan
    build.build()
    p = Plan(n, (2e-9,) * 3, prec="f32", method=method, pad=pad)
    M = torch.zeros(p.shape, dtype=torch.float32, device="cuda")
    c0 = p.launch_count()
    p.field_energy(M)
    per_call = p.launch_count() - c0
    c0 = p.launch_count()
    p.autotune(use_cache=False)
    assert p.launch_count() - c0 == CALLS * candidates * per_call
    p.close()
