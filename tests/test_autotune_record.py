"""A tuned schedule's record makes the plan that was timed: the planner's own
pick has a tile per launch, and recording the first launch's as the tile of
all of them made another, slower plan."""
import json

import numpy as np
import pytest

import paper_1411_5373_gb300 as FD
from paper_1411_5373_gb300 import autotune


@pytest.mark.parametrize("tile", [0, 448])
@pytest.mark.parametrize("shape,dtype", [((1200.0, 1600.0, 1024, 65536, 1024), "f32"),
                                         ((1200.0, 1600.0, 1024, 65536, 1024), "u8"),
                                         ((1200.0, 1600.0, 100, 50004, 300), "f32"),
                                         ((1200.0, 1600.0, 64, 1024, 64), "f16state")])
@pytest.mark.parametrize("kib", [112, 72])
def test_record_makes_the_same_plan(shape, dtype, tile, kib):
    p = FD.Plan(*shape, dtype, schedule="fused", tile=tile, smem_budget=kib * 1024, host_only=True)
    bounds = p.schedule_info()[1]
    best = json.loads(json.dumps(autotune._trial(tile, kib, bounds, 1.0)))
    q = FD.Plan(*shape, dtype, host_only=True, **autotune._arguments(best))
    for kind in (0, 1, 2, 3, 8, 9):
        assert np.array_equal(p.fused_table(kind), q.fused_table(kind)), kind
