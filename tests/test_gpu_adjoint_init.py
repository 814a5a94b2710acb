"""The fused adjoint's last launch: pieces cut by the ends of time and of the
tile, and channels of one to several level-0 rows."""
import pytest

import paper_1411_5373_gb300 as FD
from paper_1411_5373_gb300 import build

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    FD.load()


@pytest.mark.parametrize("nf,nt,nd", [(64, 260, 64), (64, 1536, 64), (64, 1540, 200), (32, 3004, 150), (4, 516, 3),
                                      (2, 36, 9)])
def test_weight_gradient(nf, nt, nd):
    p = FD.Plan(1200.0, 1600.0, nf, nt, nd, "f32", schedule="fused", adjoint="fused")
    q = FD.Plan(1200.0, 1600.0, nf, nt, nd, "f32", schedule="fused", adjoint="plain")
    gen = torch.Generator(device="cuda").manual_seed(nt)
    g = torch.randn(nd, nt, device="cuda", generator=gen)
    x = torch.randn(nf, nt, device="cuda", generator=gen)
    w = torch.rand(nf, device="cuda", generator=gen) + 0.5
    gw = torch.empty(nf, device="cuda")
    got = p.adjoint(g, x=x, grad_weights=gw)
    p.device_status()
    assert torch.equal(got, p.adjoint(g))
    assert torch.equal(p.adjoint(g, x=x, weights=w, grad_weights=torch.empty_like(gw)), got * w[:, None])
    # both schedules sum a cell's nd-ish gradient samples in float32, in
    # different orders: within (terms - 1) ulp of the sum of their magnitudes
    bound = (nf + nd) * 2.0 ** -23 * q.adjoint(g.abs())
    assert bool(((got - q.adjoint(g)).abs() <= bound).all())
    # 8 products a lane, 5 + 5 butterfly steps, a piece's slots 32 apart
    terms = x.double() * got.double()
    slots = -(-nt // 64) // 32 + 1
    assert bool(((gw.double() - terms.sum(1)).abs() <= (20 + slots) * 2.0 ** -24 * terms.abs().sum(1)).all())
