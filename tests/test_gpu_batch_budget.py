"""Fused batches whose beams need more shared memory together than a block
has: one beam's regions with another's programme slots.  Any budget that
holds each beam by itself is accepted; results equal the oracle bit for bit."""
import numpy as np
import pytest

import filterbank_synth as fs
import oracle
import paper_1411_5373_gb300 as FD
from paper_1411_5373_gb300 import build

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

BEAMS = [(1200.0, 1600.0, 512, 8192, 512), (1200.0, 1600.0, 100, 2048, 90), (1200.0, 1600.0, 256, 16384, 256),
         (1200.0, 1600.0, 64, 1024, 64)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    FD.load()


@pytest.mark.parametrize("dtype", ["f32", "u8"])
@pytest.mark.parametrize("budget", [0, 112, 216, 224, 227])
def test_mixed_beams(dtype, budget):
    bp = FD.BatchPlan(BEAMS, dtype, schedule="fused", smem_budget=budget * 1024)
    xs = [fs.random_f32(7 + i, nf, nt) for i, (_, _, nf, nt, _) in enumerate(BEAMS)]
    if dtype == "u8":
        xs = [np.clip(128 + 16 * x, 0, 255).astype(np.uint8) for x in xs]
    outs = bp.outputs()
    bp.execute([torch.from_numpy(x).cuda() for x in xs], outs)
    for (f_min, f_max, nf, nt, nd), x, y in zip(BEAMS, xs, outs):
        want = oracle.fdmt(x, oracle.build_tables(f_min, f_max, nf, nd), "i64" if dtype == "u8" else "f32")
        assert np.array_equal(y.cpu().numpy(), want), (nf, nt, nd)
