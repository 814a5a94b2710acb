"""Fused batches whose groups keep programme slots of their own (budgets near
half an SM's shared memory, groups of different sizes): the next item's copies
go out early only where its programme's slot is clear of the item that runs.
Many small segments, so that blocks change between them often; results equal
the oracle bit for bit, repeatedly."""
import numpy as np
import pytest

import filterbank_synth as fs
import oracle
import paper_1411_5373_gb300 as FD
from paper_1411_5373_gb300 import build

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

BEAMS = [(1200.0, 1600.0, nf, nt, nd) for nf, nt, nd in (
    (256, 8192, 256), (100, 2048, 300), (64, 4096, 64), (512, 4096, 512), (27, 2048, 700), (128, 8192, 100),
    (16, 1024, 200), (200, 4096, 150), (64, 1024, 64), (333, 2048, 333))]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    FD.load()


@pytest.mark.parametrize("dtype", ["f32", "u8"])
@pytest.mark.parametrize("kib", [0, 108, 112, 113, 150, 225])
def test_results(dtype, kib):
    xs = [fs.random_u8(i, b[2], b[3]) if dtype == "u8" else fs.random_f32(i, b[2], b[3]) for i, b in enumerate(BEAMS)]
    b = FD.BatchPlan(BEAMS, dtype, schedule="fused", smem_budget=kib * 1024)
    dev = [torch.from_numpy(x).cuda() for x in xs]
    outs = b.outputs()
    want = [oracle.fdmt(x, oracle.build_tables(f0, f1, nf, nd), "i64" if dtype == "u8" else "f32")
            for x, (f0, f1, nf, nt, nd) in zip(xs, BEAMS)]
    for _ in range(4):
        for o in outs:
            o.fill_(-1)
        b.execute(dev, outs)
        for o, w in zip(outs, want):
            assert np.array_equal(o.cpu().numpy(), w)
    b.close()
