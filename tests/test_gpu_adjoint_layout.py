"""The fused adjoint with rows between launches padded to whole chunks, with
and without the weight gradient, for Nf a power of two and not, on workspaces
that start as NaN bytes; with programmes in global memory; and with a launch's
cones made smaller for a second block per SM.  Gradients of small integers:
every sum is exact, so the plain schedule's result is met bit for bit."""
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


@pytest.mark.parametrize("nf,nt,nd,f_min,f_max,kw", [
    (64, 4100, 64, 1200.0, 1600.0, {}), (128, 5036, 300, 1200.0, 1600.0, {}), (100, 4108, 700, 1200.0, 1600.0, {}),
    (27, 9000, 300, 1200.0, 1600.0, {}), (8, 4132, 90, 1200.0, 1600.0, {}), (2, 4100, 40, 1200.0, 1600.0, {}),
    (45, 6256, 1756, 1100.0, 1700.0, {}),                                   # programmes in global memory
    (32, 4104, 332, 1200.0, 1600.0, {"adjoint_tile": 256}),                 # the same, Nf a power of two
    (812, 4096, 395, 1200.0, 1600.0, {}), (256, 8192, 1102, 1100.0, 1700.0, {}),  # smaller cones
])
def test_equals_plain(nf, nt, nd, f_min, f_max, kw):
    p = FD.Plan(f_min, f_max, nf, nt, nd, "f32", schedule="fused", adjoint="fused", **kw)
    q = FD.Plan(f_min, f_max, nf, nt, nd, "f32", schedule="fused", adjoint="plain")
    if kw or nf == 45:
        assert p.fused_table(15)[-1] == 0
    gen = torch.Generator(device="cuda").manual_seed(nt)
    g = torch.randint(-2, 3, (nd, nt), device="cuda", generator=gen).float()
    x = torch.randn(nf, nt, device="cuda", generator=gen)
    w = torch.rand(nf, device="cuda", generator=gen) + 0.5
    want = q.adjoint(g)
    assert float(want.abs().max()) < 2 ** 22
    gw = torch.empty(nf, device="cuda")
    for weights, grad_weights in ((None, None), (w, gw)):
        p.adjoint_workspace().fill_(255)
        got = p.adjoint(g, x=x, weights=weights, grad_weights=grad_weights)
        p.device_status()
        assert torch.equal(got, want if weights is None else want * w[:, None])
    # 8 products a lane, 5 + 5 butterfly steps, a piece's slots 32 apart
    terms = x.double() * want.double()
    slots = -(-nt // 64) // 32 + 1
    assert bool(((gw.double() - terms.sum(1)).abs() <= (20 + slots) * 2.0 ** -24 * terms.abs().sum(1)).all())
