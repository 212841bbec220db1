"""The FP32 tensor-grid energy is the sum of M . H of the field that the same call
returns, to the rounding of a thread's chain of FP32 additions: the 12 terms of
four cells (each M of rank 1 from three roundings), then one addition per such
column of a thread (at least one block of 128 per SM shares them) and five of the
warp's lanes; blocks add in FP64."""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MU0 = 4e-7 * math.pi


@pytest.mark.parametrize("n", [(200, 180, 160), (40, 33, 30), (128, 9, 7), (300, 6, 5)])
def test_energy_is_the_sum_of_the_returned_field(n):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1204_4302_gb300 import build
    from paper_1204_4302_gb300.tg import TGPlan
    build.build()
    d = (2e-9, 2e-9, 2e-9)
    g = torch.Generator().manual_seed(sum(n))
    U = [1.0 + 0.25 * torch.rand((3, 1, v), generator=g) for v in n]
    lam = 8e5 * torch.tensor([[0.3], [0.5], [0.8]])
    p = TGPlan(n, d, 1, prec="f32")
    H, E = p.field(lam.cuda(), *(u.cuda() for u in U), energy=True)
    M = torch.einsum("p,pk,pj,pi->pkji", lam[:, 0].double(), U[2][:, 0].double(), U[1][:, 0].double(),
                     U[0][:, 0].double()).cuda()
    terms = M * H.double()
    scale = 0.5 * MU0 * d[0] * d[1] * d[2]
    groups = math.ceil(n[1] / 4) * n[2]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    chain = 12 + 3 + math.ceil(n[0] / 128) * math.ceil(groups / sms) + 5
    assert abs(E.item() + scale * terms.sum().item()) <= chain * 2.0 ** -24 * scale * terms.abs().sum().item()
    p.close()
