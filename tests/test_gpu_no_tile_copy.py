"""FP32 plans without their tile-ordered tensor copy: where the device has no memory
left for it (its allocation made to fail by the host-side hook, no GPU fault), setup,
load and batches still work, and every entry point gives the results of the
complete plan within the parity tolerances of the z forms (1e-5 of the largest
field value, energies 10 times that)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1204_4302_gb300 import inputs  # noqa: E402

MS = 8e5
TOL = 1e-5
CASES = [((20, 12, 15), "dm", None),      # z 32
         ((12, 10, 30), "dm", None),      # z 64
         ((9, 17, 64), "dm", None),       # z 128
         ((12, 10, 100), "dm", None),     # z 256
         ((6, 5, 200), "dm", None),       # z 512
         ((15, 11, 20), "dm", "smooth"),  # mixed radix
         ((12, 10, 100), "sp", None)]     # SP, z 256


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1204_4302_gb300 import build
    build.build()


def _without_copy(make, full_bytes):
    """make() with its k-th allocation failing, k = 1, 2, ...: the plan that misses
    only the copy (the one allocation a plan can do without)."""
    from paper_1204_4302_gb300 import binding as B
    for k in range(1, 64):
        B.demag_debug_fail_alloc(k)
        try:
            p = make()
        except B.DemagError as e:
            assert e.name == "DEMAG_ERR_OOM"
            continue
        finally:
            B.demag_debug_fail_alloc(0)
        if p.info()["device_bytes"] < full_bytes:
            return p
        p.close()
        break
    pytest.fail("no plan without the copy")


def _rel(a, b):
    return float((a - b).abs().max() / b.abs().max())


def _compare(p, full, m):
    M = MS * m
    H, E = p.field_energy(M)
    Hf, Ef = full.field_energy(M)
    assert _rel(H, Hf) <= TOL and _rel(p.field(M), Hf) <= TOL
    assert abs(E.item() - Ef.item()) <= 10 * TOL * abs(Ef.item())
    assert abs(p.energy(M) - full.energy(M)) <= 10 * TOL * abs(Ef.item())
    if full.method == "dm":
        for grad in (False, True):
            Eg, G = p.energy_grad(m, MS, want_grad=grad)
            assert abs(Eg.item() - Ef.item()) <= 10 * TOL * abs(Ef.item())
        assert _rel(G, full.energy_grad(m, MS)[1]) <= TOL
        assert not p.info()["energy_in_z"]


@pytest.mark.parametrize("n,method,pad", CASES)
def test_plan_works_without_its_copy(n, method, pad, tmp_path):
    from paper_1204_4302_gb300.plan import Plan
    d = (2e-9, 1.5e-9, 2.5e-9)
    m = torch.tensor(inputs.random_unit(n, seed=sum(n)), dtype=torch.float32, device="cuda")
    full = Plan(n, d, method=method, pad=pad)
    p = _without_copy(lambda: Plan(n, d, method=method, pad=pad), full.info()["device_bytes"])
    _compare(p, full, m)
    p.autotune(use_cache=False)
    _compare(p, full, m)
    p.close()
    path = str(tmp_path / "plan.spec")
    full.save(path)
    q = _without_copy(lambda: Plan.load(path), full.info()["device_bytes"])
    _compare(q, full, m)
    q.close()
    full.close()


def test_tuning_without_the_copy_leaves_the_cache_alone(tmp_path, monkeypatch):
    from paper_1204_4302_gb300.plan import Plan
    cache = tmp_path / "tune.txt"
    monkeypatch.setenv("DEMAG_TUNE_CACHE", str(cache))
    n, d = (12, 10, 30), (2e-9,) * 3
    full = Plan(n, d)
    p = _without_copy(lambda: Plan(n, d), full.info()["device_bytes"])
    p.autotune()
    assert not cache.exists()
    full.autotune()
    assert cache.exists()
    p.close()
    full.close()


def test_batch_without_a_copy_runs_as_branches():
    from paper_1204_4302_gb300 import binding as B
    from paper_1204_4302_gb300.batch import Batch
    dims, cells = [(20, 12, 15), (33, 17, 5)], [(3e-9,) * 3] * 2  # z 32 (has a copy) and 16
    ms = [torch.tensor(MS * inputs.random_unit(n, seed=i), dtype=torch.float32, device="cuda") for i, n in enumerate(dims)]
    full = Batch(dims, cells)
    assert full.info()["persistent_ok"]
    Hf, Ef = full.field(ms, energies=True)
    for k in range(1, 64):
        B.demag_debug_fail_alloc(k)
        try:
            b = Batch(dims, cells)
        except B.DemagError as e:
            assert e.name == "DEMAG_ERR_OOM"
            continue
        finally:
            B.demag_debug_fail_alloc(0)
        break
    assert not b.info()["persistent_ok"] and b.info()["mode"] == Batch.BRANCHES
    with pytest.raises(B.DemagError) as err:
        b.set_mode(Batch.PASSES)
    assert err.value.name == "DEMAG_ERR_UNSUPPORTED"
    H, E = b.field(ms, energies=True)
    for a, c in zip(H, Hf):
        assert _rel(a, c) <= TOL
    assert torch.allclose(E, Ef, rtol=10 * TOL, atol=0)
    b.close()
    full.close()
