"""The warp-per-window search kernel (up to 9 widths, 4-byte sums) at the
sizes where it can go wrong: rows around one lane, one window's own columns
and one walk of eight windows, unaligned rows, ties across lanes, windows and
walks, and rows of infinities, NaN and the lowest value.  Peaks bit for bit
and first times equal to the oracle's."""
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


def run(A, k, offset=0, bound=0):
    flat = torch.zeros(A.size + offset, dtype=torch.float32 if A.dtype == np.float32 else torch.int32, device="cuda")
    flat[offset:] = torch.from_numpy(A.reshape(-1)).cuda()
    peak, time = FD.search(flat[offset:].view(A.shape), k, value_bound=bound)
    return peak.cpu().numpy(), time.cpu().numpy()


@pytest.mark.parametrize("k", [2, 6, 7, 8, 9])
@pytest.mark.parametrize("nt", [31, 32, 33, 767, 768, 769, 895, 896, 897, 992, 1024, 6144, 7168, 7169, 7937])
def test_edges(nt, k):
    A = fs.random_f32(nt + k, 3, nt)
    B = np.random.default_rng(nt).integers(-1000, 1001, size=(3, nt)).astype(np.int32)
    for X, off in ((A, 0), (A, 1), (B, 0)):
        peak, time = run(X, k, off, 1000 if X is B else 0)
        rp, rt = oracle.boxcar_search(X, k)
        assert np.array_equal(peak, rp) and np.array_equal(time, rt)


@pytest.mark.parametrize("k", [5, 9])
def test_ties_take_the_first_time(k):
    A = np.zeros((4, 20000), dtype=np.float32)
    A[0, [15999, 7200, 3000, 47]] = 2.0   # equal pulses in several walks, windows and lanes
    A[1, 40:60] = 1.0
    A[2, 16::32] = 1.0
    A[3] = 1.0
    rp, rt = oracle.boxcar_search(A, k)
    peak, time = run(A, k)
    assert np.array_equal(peak, rp) and np.array_equal(time, rt)


def test_non_finite_rows():
    """A maximum of +inf keeps its first time; a row without a value above
    -inf has none (peak -inf, time 0); NaN never qualifies."""
    A = fs.random_f32(5, 4, 3000)
    A[0, [2500, 700]] = np.inf
    A[1] = -np.inf
    A[2] = np.nan
    A[3, ::2] = np.nan
    peak, time = run(A, 1)
    assert peak[0, 0] == np.inf and time[0, 0] == 700
    assert (peak[1:3, 0] == -np.inf).all() and (time[1:3, 0] == 0).all()
    assert peak[3, 0] == np.nanmax(A[3]) and time[3, 0] == int(np.nanargmax(A[3]))
