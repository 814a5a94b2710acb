"""The filterbank's block sizes for Nf = 1024 and more: few transforms go to
blocks of 256 or 512 threads, more to larger ones; both sides of the lines, binned and
not, whole and ragged tiles, against the float64 oracle within the float32
FFT's bound, and bit for bit against each other."""
import numpy as np
import pytest

import oracle
import paper_1411_5373_gb300 as FD
from paper_1411_5373_gb300 import build

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

EPS = 2.0 ** -24


@pytest.fixture(scope="module", autouse=True)
def _lib():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    FD.load()


@pytest.mark.parametrize("nf,nbin,nt", [
    (4096, 1, 1), (4096, 1, 152), (4096, 1, 153), (4096, 1, 156), (4096, 1, 304), (4096, 1, 308), (4096, 1, 311),
    (4096, 2, 152), (4096, 2, 153), (2048, 1, 304), (2048, 1, 308), (2048, 1, 611), (2048, 1, 2432), (2048, 1, 2436),
    (2048, 2, 152), (2048, 2, 153), (2048, 3, 100), (2048, 4, 608), (2048, 4, 609), (2048, 5, 122), (2048, 5, 700),
    (1024, 1, 608), (1024, 1, 612), (1024, 4, 152), (1024, 4, 153), (1024, 7, 50),
])
def test_blocks(nf, nbin, nt):
    rng = np.random.Generator(np.random.PCG64([nf, nbin, nt]))
    more = 2600  # (times enough for the largest blocks)
    v = torch.from_numpy(rng.standard_normal((more * nf * nbin, 2)).astype(np.float32)).cuda()
    v = torch.view_as_complex(v)
    got = FD.filterbank(v[:nt * nf * nbin], nf, nbin)
    assert torch.equal(got, FD.filterbank(v, nf, nbin)[:, :nt])
    ref = oracle.stft_filterbank(v[:nt * nf * nbin].cpu().numpy().astype(np.complex128), nf, nbin)
    bound = 8 * EPS * np.log2(nf) * ref.sum(axis=0)
    assert (np.abs(got.cpu().numpy().astype(np.float64) - ref) <= bound[None, :]).all()
