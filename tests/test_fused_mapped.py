"""A mapped plan's fused schedule (d_min pre-shift, descending channels) reads
the raw input through its first launch's copies: the emulated programme on
the raw rows must equal the oracle's mapping pass followed by its transform,
bit for bit, over channel orders, delays up to whole rows and beyond, data
types and row lengths."""
import numpy as np
import pytest

import filterbank_synth as fs
import oracle
import paper_1411_5373_gb300 as FD
from fused_emulator import check_bounds, emulate


@pytest.mark.parametrize("nf,nt,nd,dtype,d_min,desc,kw", [
    (16, 256, 16, "f32", 1, False, {}),
    (16, 256, 16, "f32", 0, True, {"staging": "blocks"}),
    (48, 452, 60, "f32", 37, True, {"tile": 64}),
    (33, 400, 40, "u8", 129, False, {"tile": 128}),
    (64, 448, 100, "u8", 1000, True, {"bounds": [0, 3, 6]}),  # delays past the row's end
    (64, 448, 64, "f16state", 15, True, {"tile": 128, "bounds": [0, 2, 6]}),
    (3, 192, 12, "f32", 5, True, {"bounds": [0, 1, 2]}),
])
def test_emulated_mapped_schedule_equals_oracle(nf, nt, nd, dtype, d_min, desc, kw):
    p = FD.Plan(1200.0, 1600.0, nf, nt, nd, dtype, schedule="fused", host_only=True, d_min=d_min, descending=desc, **kw)
    x = fs.random_u8(nf, nf, nt) if dtype == "u8" else fs.random_f32(nf, nf, nt)
    shifts = oracle.input_shifts(1200.0, 1600.0, nf, d_min)
    T = oracle.build_tables(1200.0, 1600.0, nf, nd)
    mode = {"u8": "i64", "f32": "f32", "f16state": "f16state"}[dtype]
    assert np.array_equal(emulate(p, x), oracle.fdmt(oracle.map_input(x, shifts, desc), T, mode))
    check_bounds(p)
