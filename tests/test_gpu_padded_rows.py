"""Layouts at their limits.  Rows of the levels between launches padded to whole chunks (nt from 4096 on
and no multiple of 64): single beams of every type and a batch in one launch,
bit-exact to the oracle, on buffers that start as NaN bytes (the columns past
nt are never written and must never reach an output); and budgets that only
the compact layout fits."""
import numpy as np
import pytest

import filterbank_synth as fs
import oracle
import paper_1411_5373_gb300 as FD
from paper_1411_5373_gb300 import build

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

MODE = {"u8": "i64", "f32": "f32", "f16state": "f16state"}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    FD.load()


@pytest.mark.parametrize("nf,nt,nd,dtype", [
    (64, 4100, 90, "f32"), (128, 4112, 300, "u8"), (64, 4104, 64, "f16state"), (100, 5036, 700, "f32"),
    (64, 4096, 64, "f32"), (64, 4092, 64, "f32"),
])
def test_beam(nf, nt, nd, dtype):
    x = fs.random_u8(nt, nf, nt) if dtype == "u8" else fs.random_f32(nt, nf, nt)
    p = FD.Plan(1200.0, 1600.0, nf, nt, nd, dtype, schedule="fused", bounds=[0, 2, 4, p_levels(nf)])
    p.workspace().fill_(255)
    got = p.execute(torch.from_numpy(x).cuda()).cpu().numpy()
    p.device_status()
    assert np.array_equal(got, oracle.fdmt(x, oracle.build_tables(1200.0, 1600.0, nf, nd), MODE[dtype]))


@pytest.mark.parametrize("nf,nt,nd,dtype,kw", [
    (128, 2064, 399, "f32", {"tile": 128, "smem_budget": 12288, "bounds": [0, 3, 5, 7]}),
    (33, 448, 156, "u8", {"tile": 512, "smem_budget": 12288, "bounds": [0, 2, 4, 6], "staging": "boxes"}),
])
def test_compact_layout(nf, nt, nd, dtype, kw):
    """Budgets that leave no room for the programmes in shared memory (they
    are read in global memory) nor for whole row pitches."""
    x = fs.random_u8(nt, nf, nt) if dtype == "u8" else fs.random_f32(nt, nf, nt)
    p = FD.Plan(1200.0, 1600.0, nf, nt, nd, dtype, schedule="fused", **kw)
    got = p.execute(torch.from_numpy(x).cuda()).cpu().numpy()
    p.device_status()
    assert np.array_equal(got, oracle.fdmt(x, oracle.build_tables(1200.0, 1600.0, nf, nd), MODE[dtype]))


def p_levels(nf):
    return (nf - 1).bit_length()


def test_batch():
    beams = [(1200.0, 1600.0, 64, 4112, 90), (1200.0, 1600.0, 100, 5040, 300), (1200.0, 1600.0, 16, 2048, 40)]
    xs = [fs.random_u8(i, b[2], b[3]) for i, b in enumerate(beams)]
    bp = FD.BatchPlan(beams, "u8", schedule="fused", fused_tile=128, smem_budget=24 * 1024)
    bp.workspace().fill_(255)
    outs = bp.execute([torch.from_numpy(x).cuda() for x in xs], bp.outputs())
    for (f0, f1, nf, nt, nd), x, y in zip(beams, xs, outs):
        assert np.array_equal(y.cpu().numpy(), oracle.fdmt(x, oracle.build_tables(f0, f1, nf, nd), "i64"))
    bp.close()
