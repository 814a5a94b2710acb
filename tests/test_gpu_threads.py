"""Calls from threads that have made no CUDA call before: the tensor maps of a
launch are encoded by the driver, which needs a context that is current in the
calling thread.  Every path that encodes maps runs in a new thread with its
buffers and workspace in hand (so nothing else there binds a context), after
the main thread has run it; results equal the main thread's.  And a small
step through autograd, whose backward runs in a thread of its own."""
import threading

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


def in_new_thread(call):
    got = []

    def body():
        try:
            got.append(call())
        except BaseException as e:  # noqa: BLE001 (handed to the test)
            got.append(e)
    t = threading.Thread(target=body)
    t.start()
    t.join()
    if isinstance(got[0], BaseException):
        raise got[0]


def both(call, *outs):
    """The outputs of `call` from the main thread and from a new one."""
    call()
    torch.cuda.synchronize()
    want = [o.clone() for o in outs]
    for o in outs:
        o.zero_()
    torch.cuda.synchronize()
    in_new_thread(call)
    torch.cuda.synchronize()
    for o, w in zip(outs, want):
        assert torch.equal(o, w)


def test_transform_adjoint_and_stream():
    s = torch.cuda.current_stream()
    p = FD.Plan(1200.0, 1600.0, 64, 1024, 64, "f32", schedule="fused")
    x = torch.randn(64, 1024, device="cuda")
    w = torch.rand(64, device="cuda")
    out, g_in = torch.empty(64, 1024, device="cuda"), torch.empty(64, 1024, device="cuda")
    g_w = torch.empty(64, device="cuda")
    ws, aws = p.workspace(), p.adjoint_workspace()
    both(lambda: p.execute(x, out=out, weights=w, workspace=ws, stream=s), out)
    both(lambda: p.adjoint(x, x=x, weights=w, grad_in=g_in, grad_weights=g_w, workspace=aws, stream=s), g_in, g_w)


@pytest.mark.parametrize("nf,nt", [(1024, 64), (64, 100)])
def test_filterbank(nf, nt):
    s = torch.cuda.current_stream()
    volts = torch.randn(nf * nt, dtype=torch.complex64, device="cuda")
    out = torch.empty(nf, nt, device="cuda")
    both(lambda: FD.filterbank(volts, nf, out=out, stream=s), out)


def test_batch_in_one_launch():
    s = torch.cuda.current_stream()
    b = FD.BatchPlan([(1200.0, 1600.0, 64, 1024, 64), (1200.0, 1600.0, 32, 512, 40)], "f32", schedule="fused")
    xs = [torch.randn(64, 1024, device="cuda"), torch.randn(32, 512, device="cuda")]
    outs, ws = b.outputs(), b.workspace()
    # (the launch's graph and maps are made anew for other buffers)
    b.execute(xs, outs, workspace=ws, stream=s)
    torch.cuda.synchronize()
    other = b.outputs()
    in_new_thread(lambda: b.execute(xs, other, workspace=ws, stream=s))
    torch.cuda.synchronize()
    assert all(torch.equal(o, w) for o, w in zip(other, outs))


def test_small_step_through_autograd():
    p = FD.Plan(1200.0, 1600.0, 27, 1000, 30, "f32", schedule="fused")
    p.workspace()
    p.adjoint_workspace()
    x = torch.randn(27, 1000, device="cuda", requires_grad=True)
    w = torch.rand(27, device="cuda", requires_grad=True)
    g = torch.randn(30, 1000, device="cuda")
    gx, gw = torch.autograd.grad(FD.fdmt(x, p, w), (x, w), g)
    want = p.adjoint(g, x=x.detach(), weights=w.detach(), grad_weights=(ww := torch.empty(27, device="cuda")))
    assert torch.equal(gx, want) and torch.equal(gw, ww)
