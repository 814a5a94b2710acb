"""Streams over fused plans write a window's last columns straight to the
output and compute only the tiles those need: chunks from 16 samples to many
tiles, carries from none to many chunks, one-launch plans, channel counts
that are no power of two, and a reset in mid-stream.  Every push equals the
matching columns of one oracle transform, bit for bit."""
import numpy as np
import pytest

import filterbank_synth as fs
import oracle
import paper_1411_5373_gb300 as FD
from paper_1411_5373_gb300 import build

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    FD.load()


@pytest.mark.parametrize("nf,chunk,nd,pushes,dtype", [
    (2, 16, 5, 4, "f32"), (2, 1024, 1, 2, "u8"), (3, 64, 40, 5, "f32"), (16, 16, 33, 6, "u8"),
    (64, 4096, 64, 3, "f16state"), (100, 992, 300, 4, "f32"), (256, 2000, 1026, 3, "u8"), (256, 48, 700, 5, "f32"),
])
def test_pushes_equal_one_transform(nf, chunk, nd, pushes, dtype):
    nt = chunk * pushes
    x = fs.random_u8(nf + chunk, nf, nt) if dtype == "u8" else fs.random_f32(nf + chunk, nf, nt)
    T = oracle.build_tables(1200.0, 1600.0, nf, nd)
    want = oracle.fdmt(x, T, {"u8": "i64", "f32": "f32", "f16state": "f16state"}[dtype])
    st = FD.Stream(1200.0, 1600.0, nf, chunk, nd, dtype, "fused")
    parts = [torch.from_numpy(np.ascontiguousarray(x[:, i * chunk:(i + 1) * chunk])).cuda() for i in range(pushes)]
    st.push(parts[-1])  # anything; the reset forgets it
    st.reset()
    got = np.concatenate([st.push(p).cpu().numpy() for p in parts], axis=1)
    st.close()
    assert np.array_equal(got, want)


def test_captured_pushes_carry_on():
    """A reset followed by a captured pair of pushes: every replay goes on
    from the chunks before it, the first one from zeros."""
    nf, chunk, nd = 32, 512, 100
    x = fs.random_u8(7, nf, 6 * chunk)
    want = oracle.fdmt(x, oracle.build_tables(1200.0, 1600.0, nf, nd), "i64")
    parts = [torch.from_numpy(np.ascontiguousarray(x[:, i * chunk:(i + 1) * chunk])).cuda() for i in range(6)]
    st = FD.Stream(1200.0, 1600.0, nf, chunk, nd, "u8", "fused")
    a, b = parts[0].clone(), parts[1].clone()
    out = [st.push(a), st.push(b)]
    st.reset()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        st.push(a, out[0])
        st.push(b, out[1])
    got = []
    for i in range(0, 6, 2):
        a.copy_(parts[i])
        b.copy_(parts[i + 1])
        graph.replay()
        got += [o.cpu().numpy() for o in out]
    st.close()
    assert np.array_equal(np.concatenate(got, axis=1), want)
