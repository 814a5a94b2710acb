"""Walks whose upper sums move between lanes (few channels, many delays: upper
rows from 2 on): whole walks of 32 rows, pieces narrower than a strip, tiles
at both ends of time, single channels, weights, every data type; bit for bit
equal to the oracle (weighted: to the plain schedule)."""
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


@pytest.mark.parametrize("nf,nt,nd,kw", [
    (2, 2048, 1, {}), (2, 1040, 4, {}), (2, 1040, 6, {}), (2, 2048, 70, {}), (2, 4096, 300, {"tile": 64}),
    (3, 1040, 500, {}), (8, 2048, 600, {}), (8, 2064, 600, {"tile": 128, "bounds": [0, 1, 3]}),
    (27, 4112, 900, {}), (32, 4096, 1900, {}), (64, 2048, 1935, {}),
    (16, 2064, 500, {"d_min": 77, "descending": True}),
])
@pytest.mark.parametrize("dtype", ["f32", "u8", "f16state"])
def test_equals_oracle(nf, nt, nd, kw, dtype):
    x = fs.random_u8(nt, nf, nt) if dtype == "u8" else fs.random_f32(nt, nf, nt)
    p = FD.Plan(1200.0, 1600.0, nf, nt, nd, dtype, schedule="fused", **kw)
    got = p.execute(torch.from_numpy(x).cuda()).cpu().numpy()
    p.device_status()
    if "d_min" in kw:
        x = oracle.map_input(x, oracle.input_shifts(1200.0, 1600.0, nf, kw["d_min"]), kw["descending"])
    assert np.array_equal(got, oracle.fdmt(x, oracle.build_tables(1200.0, 1600.0, nf, nd), MODE[dtype]))


@pytest.mark.parametrize("nf,nt,nd", [(2, 1040, 70), (27, 4100, 900), (100, 2052, 1800)])
def test_weighted_equals_plain(nf, nt, nd):
    x = torch.from_numpy(fs.random_f32(nt, nf, nt)).cuda()
    w = torch.rand(nf, device="cuda") + 0.5
    p = FD.Plan(1200.0, 1600.0, nf, nt, nd, "f32", schedule="fused")
    q = FD.Plan(1200.0, 1600.0, nf, nt, nd, "f32", schedule="plain")
    assert torch.equal(p.execute(x, weights=w), q.execute(x, weights=w))


@pytest.mark.parametrize("dtype", ["f32", "u8"])
def test_batch_in_one_launch(dtype):
    """Few channels and many delays beside an ordinary beam."""
    beams = [(1200.0, 1600.0, 8, 2048, 600), (1200.0, 1600.0, 64, 1024, 64), (1200.0, 1600.0, 27, 4112, 900)]
    xs = [fs.random_u8(i, b[2], b[3]) if dtype == "u8" else fs.random_f32(i, b[2], b[3]) for i, b in enumerate(beams)]
    b = FD.BatchPlan(beams, dtype, schedule="fused")
    outs = b.execute([torch.from_numpy(x).cuda() for x in xs], b.outputs())
    for (f0, f1, nf, nt, nd), x, y in zip(beams, xs, outs):
        assert np.array_equal(y.cpu().numpy(), oracle.fdmt(x, oracle.build_tables(f0, f1, nf, nd), MODE[dtype]))


@pytest.mark.parametrize("nf,nt,nd,k", [(8, 1920, 600, 5), (27, 4112, 900, 8), (64, 2048, 1935, 3)])
@pytest.mark.parametrize("dtype", ["f32", "u8"])
def test_search_in_the_last_launch(nf, nt, nd, k, dtype):
    x = fs.random_u8(nt, nf, nt) if dtype == "u8" else fs.random_f32(nt, nf, nt)
    p = FD.Plan(1200.0, 1600.0, nf, nt, nd, dtype, schedule="fused", search_widths=k)
    out, peak, time = p.execute_search(torch.from_numpy(x).cuda(), k)
    p.device_status()
    want = oracle.fdmt(x, oracle.build_tables(1200.0, 1600.0, nf, nd), MODE[dtype])
    assert np.array_equal(out.cpu().numpy(), want)
    rp, rt = oracle.boxcar_search(want, k)
    assert np.array_equal(peak.cpu().numpy(), rp) and np.array_equal(time.cpu().numpy(), rt)


@pytest.mark.parametrize("nf,chunk,nd", [(2, 48, 70), (2, 512, 300), (8, 80, 600), (27, 1024, 900)])
@pytest.mark.parametrize("dtype", ["f32", "u8"])
def test_streams(nf, chunk, nd, dtype):
    """A push writes only its chunk's columns: level 1 may be the top level."""
    x = fs.random_u8(nf, nf, 4 * chunk) if dtype == "u8" else fs.random_f32(nf, nf, 4 * chunk)
    want = oracle.fdmt(x, oracle.build_tables(1200.0, 1600.0, nf, nd), MODE[dtype])
    s = FD.Stream(1200.0, 1600.0, nf, chunk, nd, dtype, "fused")
    got = [s.push(torch.from_numpy(np.ascontiguousarray(x[:, i:i + chunk])).cuda()).cpu().numpy()
           for i in range(0, 4 * chunk, chunk)]
    s.close()
    assert np.array_equal(np.concatenate(got, axis=1), want)
