"""Walks whose upper sums move between lanes, on the CPU: the 32 columns kept
before a piece supply every move (a walk has at most 31), each sum that
reaches the piece is the one the row needs, and their reads stay inside the
block's shared memory."""
import numpy as np
import pytest

import paper_1411_5373_gb300 as FD

NO_UPPER, MOVES = 1, 2  # walk flags
UNDER = 128  # bytes of slack below the staged rows, behind 128 of barriers


@pytest.mark.parametrize("nf,nt,nd,dtype,kw", [
    (2, 2048, 2048, "f32", {}), (3, 1040, 500, "u8", {}), (27, 9008, 3000, "u8", {}), (32, 159808, 2738, "f16state", {}),
    (64, 2048, 1935, "f32", {"d_min": 77, "descending": True}), (1024, 65536, 1024, "f32", {}),
])
def test_sums_before_the_piece(nf, nt, nd, dtype, kw):
    p = FD.Plan(1200.0, 1600.0, nf, nt, nd, dtype, schedule="fused", host_only=True, **kw)
    es = 1 if dtype == "u8" else 4
    walks = p.fused_table(3).reshape(-1, 12).astype(np.int64)
    assert len(walks)
    moved = 0
    for dst, dst_row, x_lo, x_hi, width, col, a, e, dl0, bits, chan, flags in walks.tolist():
        grow = [(bits >> i) & 1 for i in range(e - a)]
        assert e - a < 32 and bits >> (e - a) == 0
        j, dl = a - dl0, dl0
        if not flags & MOVES:
            continue
        assert not flags & NO_UPPER
        # (column, first sample, terms) of each lane's sum, as the kernel keeps
        # them: columns -32 .. -1, and of the piece its first one
        kept = [(c, c - dl, j + 1) for c in range(-32, 0)]
        first = (0, -dl, j + 1)
        for g in grow:
            if g:
                dl += 1
                c, s, n = kept[-1]
                first = (0, s, n)
                kept = [None] + [(k[0] + 1, *k[1:]) if k else None for k in kept[:-1]]
                moved += 1
            else:
                j += 1
                first = (0, first[1], first[2] + 1)
                kept = [k and (k[0], k[1], k[2] + 1) for k in kept]
            assert first == (0, -dl, j + 1)
            assert x_hi - (32 + dl + j) * es >= UNDER
        assert x_hi - (32 + dl0 + a - dl0) * es >= UNDER
    assert moved > 0 or nf == 1024
