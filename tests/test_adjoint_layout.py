"""CPU checks of the fused adjoint's launches: rows of the levels between
launches padded to whole chunks (Nt from 4096 on and no multiple of 32), and
the shared memory a launch takes.  The emulated tables equal the float64
oracle's adjoint exactly on small integers."""
import numpy as np
import pytest

import filterbank_synth as fs
import oracle
import paper_1411_5373_gb300 as FD
from adjoint_emulator import check_adjoint_tables, emulate_adjoint, row_lengths

TWO_BLOCKS = 113 * 1024  # a block's shared memory that leaves room for a second one


def plan(f_min, f_max, nf, nt, nd, **kw):
    return FD.Plan(f_min, f_max, nf, nt, nd, "f32", schedule="fused", host_only=True, adjoint="fused", **kw)


@pytest.mark.parametrize("nf,nt,nd", [(27, 4104, 300), (32, 4100, 96), (2, 4132, 9), (100, 4108, 60)])
def test_padded_rows_equal_oracle(nf, nt, nd):
    p = plan(1200.0, 1600.0, nf, nt, nd)
    lengths = row_lengths(p, p.fused_table(10).reshape(-1, 15))
    assert lengths[0][0] == lengths[-1][1] == nt
    assert all(out == -(-nt // 32) * 32 for _, out in lengths[:-1])
    g = fs.small_ints(nt, (nd, nt)).astype(np.float32)
    got = emulate_adjoint(p, g)
    want = oracle.fdmt_adjoint(g.astype(np.float64), oracle.build_tables(1200.0, 1600.0, nf, nd))
    assert np.array_equal(got, want.astype(np.float32))
    assert check_adjoint_tables(p) > 0


@pytest.mark.parametrize("nf,nt,nd", [(27, 9000, 300), (48, 9000, 300), (32, 9000, 1000), (512, 50004, 700)])
def test_padded_rows_tables(nf, nt, nd):
    assert check_adjoint_tables(plan(1200.0, 1600.0, nf, nt, nd)) > 0


@pytest.mark.parametrize("band,nf,nt,nd,launches", [
    ((1200.0, 1600.0), 812, 65536, 395, 5),   # [10,8] 130688 and [6,4] 116096 bytes at the full budget
    ((1100.0, 1700.0), 256, 65536, 1102, 3),  # [8,6]
    ((1200.0, 1600.0), 32, 65536, 332, 1),    # [5,2]
    ((1200.0, 1600.0), 1024, 65536, 1024, 5),
])
def test_launches_leave_room_for_two_blocks(band, nf, nt, nd, launches):
    """Regions are maxima over a launch's cones; where they add up to more
    than half an SM the cones get smaller."""
    p = plan(*band, nf, nt, nd)
    smem = p.fused_table(10).reshape(-1, 15)[:, 7]
    assert (smem <= TWO_BLOCKS).sum() == launches
    assert check_adjoint_tables(p) > 0


@pytest.mark.parametrize("band,nf,nt,nd", [((1200.0, 1600.0), 32, 65536, 332), ((1100.0, 1700.0), 256, 65536, 1102),
                                           ((1200.0, 1600.0), 512, 65536, 2717), ((1200.0, 1600.0), 464, 65536, 314)])
def test_programmes_stay_in_shared_memory(band, nf, nt, nd):
    """Where a tile leaves no room for the programmes, one that is less than
    twice as narrow is taken if it does."""
    p = plan(*band, nf, nt, nd)
    assert (p.fused_table(15)[4:] > 0).all()
    assert check_adjoint_tables(p) > 0


def test_explicit_tiles_and_budgets_stand():
    """A tile or budget that the caller gives is not replaced."""
    p = plan(1200.0, 1600.0, 64, 4096, 64, adjoint_bounds=[0, 2, 4, 6], adjoint_tile=256)
    assert (p.fused_table(10).reshape(-1, 15)[:, 3] == 256).all()
    r = plan(1200.0, 1600.0, 32, 65536, 332, adjoint_tile=256)  # (whose last programmes then stay in global memory)
    assert (r.fused_table(10).reshape(-1, 15)[:, 3] == 256).all() and r.fused_table(15)[-1] == 0
    q = plan(1200.0, 1600.0, 256, 4096, 256, adjoint_smem_budget=160 * 1024)
    assert (q.fused_table(10).reshape(-1, 15)[:, 7] > TWO_BLOCKS).any()
