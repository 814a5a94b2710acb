"""The runs of the fused schedule (the ops of single and pair stages as the
kernel runs them) against the ops they are lowered from, on the CPU.

A run is expanded row by row with its step masks; every column it writes must
be one the stage's ops write, from the same shared-memory words, written once;
no read of the strip (the columns beside the rows included) may leave the
block's shared memory, and a strip stored whole must reach no column of
another row and stay between the staged rows and the descriptor slots.  The ops themselves are executed against the oracle in
test_fused_plan.py.
"""
import bisect

import numpy as np
import pytest

import paper_1411_5373_gb300 as FD
from fused_emulator import GENERAL, HI_ONE, KIND_MASK, LO_ONE, NO_HI, PADDED, PAIR, PIECE, SINGLE, STAGE_WORDS

RUN_STAGE = 64
WHOLE = 256


def _rows_of_run(run, pair):
    """(destination, first column, sources) of each row of a run."""
    dst, dst_row, col, width, p0, p1, p2, p3, g0, g1, g2, g3, n, inc, sub, flags = (int(v) for v in run)
    for r in range(n):
        yield r, col, (p0, p1, p2, p3)
        one, s = (inc >> r) & 1, (sub >> r) & 1
        if one:
            move = 0 if flags & NO_HI else 1
            col += move
            p0, p1 = p0 + move * ES, p1 + move * ES
            if s or not pair:
                p0, p1 = p0 + g0, p1 - ES
            else:
                p1 += g1
        elif s or not pair:
            p2, p3 = p2 + g2, p3 - ES
        else:
            p3 += g3


def _check(plan):
    global ES
    groups = plan.fused_table(0).reshape(-1, 16)
    tpls = plan.fused_table(1).reshape(-1, 8)
    ops = plan.fused_table(4).reshape(-1, 8).astype(np.int64)
    stages, run_stages = plan.fused_table(5), plan.fused_table(9)
    runs = plan.fused_table(8).reshape(-1, 16)
    over_read, desc = (int(v) for v in plan.fused_table(6)[4:6])
    assert len(stages) == len(run_stages)
    checked = 0
    for g in groups:
        smem, s_end, in_size = int(g[5]), int(g[8]), int(g[14])
        for tp in tpls[int(g[3]):int(g[3]) + int(g[4])]:
            sb, nst = int(tp[4]), int(tp[5])
            for si in range(nst):
                blk = stages[sb + si * STAGE_WORDS:sb + (si + 1) * STAGE_WORDS]
                rblk = run_stages[sb + si * STAGE_WORDS:sb + (si + 1) * STAGE_WORDS]
                kind = int(blk[0]) & KIND_MASK
                if kind not in (SINGLE, PAIR):
                    assert np.array_equal(blk, rblk)
                    continue
                assert int(rblk[0]) == int(blk[0]) | RUN_STAGE and np.all(np.diff(rblk[1:]) >= 0)
                pair, padded = kind == PAIR, bool(int(blk[0]) & PADDED)
                to_global = si == nst - 1
                ES = in_size if si == 0 else 4
                want = {}
                for d, p0, p1, p2, p3, width, flags, col in ops[int(blk[1]):int(blk[-1])].tolist():
                    src = [p0, p1 if pair and not flags & LO_ONE else None,
                           None if flags & NO_HI else (p2 if pair else p1),
                           p3 if pair and not flags & (NO_HI | HI_ONE) else None]
                    # bytes from the row's column 0
                    row = d if to_global else (d - (col + 4 * (col >> 4)) * 4 if padded else d - 4 * col)
                    at = want.setdefault(row, [0, [None if p is None else p - col * ES for p in src]])
                    assert at[1] == [None if p is None else p - col * ES for p in src]
                    at[0] = max(at[0], col + width)
                starts = sorted(want)
                got = {row: np.zeros(w, dtype=np.int32) for row, (w, _) in want.items()}
                for run in runs[int(rblk[1]):int(rblk[-1])]:
                    dst, dst_row, col0, width, n, flags = (int(run[i]) for i in (0, 1, 2, 3, 12, 15))
                    assert 1 <= n <= 32
                    assert int(blk[0]) & GENERAL or flags & ~WHOLE == 0
                    for r, col, p in _rows_of_run(run, pair):
                        if to_global:
                            row = dst + r
                        else:
                            row = dst + r * dst_row - (0 if padded else 4 * col0)
                        w, src = want[row]
                        assert w == width
                        for have, s in zip(p, src):
                            if s is None:
                                continue
                            assert have == s + col * ES, "a run reads other words than its op"
                            assert have >= 128 and have + PIECE * ES <= smem, "a strip leaves shared memory"
                            if si == 0:
                                lo = max(col, 0)
                                assert s + lo * ES >= 256 and s + min(col + PIECE, width) * ES <= s_end
                        if flags & WHOLE:
                            assert not to_global and not padded
                            b0, b1 = row + 4 * col, row + 4 * (col + PIECE)
                            assert b0 >= s_end and b1 <= smem - over_read - desc
                            i = bisect.bisect_left(starts, row)
                            assert i == 0 or starts[i - 1] + 4 * want[starts[i - 1]][0] <= b0
                            assert i + 1 == len(starts) or b1 <= starts[i + 1]
                        got[row][max(col, 0):min(col + PIECE, width)] += 1
                        checked += 1
                assert all((v == 1).all() for v in got.values()), "columns missing or written twice"
    return checked


@pytest.mark.parametrize("nf,nt,nd,dtype,kw", [
    (16, 256, 16, "f32", {}),
    (4, 64, 1, "f32", {}),
    (8, 4096, 4096, "f32", {}),  # delays far above the channels: runs cut at 32 rows
    (64, 1040, 300, "u8", {"tile": 512, "bounds": [0, 2, 4, 6]}),  # nodes a whole number of strips wide
    (128, 2064, 300, "f16state", {"tile": 192, "bounds": [0, 3, 4, 7]}),
    (257, 2048, 140, "u8", {"tile": 128}),
    (1000, 1024, 200, "f32", {"bounds": [0, 3, 6, 8, 10]}),
    (7, 256, 30, "u8", {"tile": 64, "bounds": [0, 1, 3]}),
    (64, 960, 64, "f32", {"tile": 64, "smem_budget": 48 * 1024, "search_widths": 6}),
    (100, 960, 90, "u8", {"tile": 256, "bounds": [0, 3, 7], "search_widths": 8}),
    (256, 4096, 2048, "f32", {"gamma": 1.5}),
    # budgets that only the compact layout fits
    (128, 2064, 399, "f32", {"tile": 128, "smem_budget": 12288, "bounds": [0, 3, 5, 7]}),
    (33, 448, 156, "u8", {"tile": 512, "smem_budget": 12288, "bounds": [0, 2, 4, 6], "staging": "boxes"}),
    (1024, 65536, 1024, "f32", {}),
    (1024, 65536, 1024, "u8", {"bounds": [0, 3, 6, 10]}),
])
def test_runs_are_the_ops(nf, nt, nd, dtype, kw):
    p = FD.Plan(1200.0, 1600.0, nf, nt, nd, dtype, schedule="fused", host_only=True, **kw)
    assert _check(p) > 0
