"""A closed plan has no workspace sizes: asking for one is an error."""
import pytest

import paper_1411_5373_gb300 as F
from paper_1411_5373_gb300._native import FdmtError

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("name", ["workspace", "adjoint_workspace"])
def test_workspace_after_close_is_refused(name):
    p = F.Plan(1200.0, 1600.0, 64, 1024, 64, "f32", host_only=True)
    assert getattr(p, name)(device="cpu").numel() > 0
    p.close()
    with pytest.raises(FdmtError):
        getattr(p, name)(device="cpu")
