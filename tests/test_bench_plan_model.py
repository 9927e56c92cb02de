"""The benchmark's count of FP64 instructions per cell and step, from the plans
of the graphs a rank runs (no GPU needed)."""
import pytest

import bench
from paper_2107_00555_gb300 import _capi as C
from paper_2107_00555_gb300 import programs


def _plan(shape, steps, bc="periodic"):
    return programs.heat3d(shape, steps, bc, "f64", fuse=C.DCP_FUSE_ALL).plan()


def test_plans_of_a_sharded_rank_are_counted_with_their_own_forms():
    """A sharded rank passes one plan per chunk of steps: a 512^2 slab runs as
    columns, a small one as planes."""
    wl = bench.Stencil("heat3d")
    column, planes = _plan((260, 512, 512), 2), _plan((24, 24, 24), 2)
    assert column["groups"][0]["kernel_form"] == "column"
    assert planes["groups"][0]["kernel_form"] == "tile"
    per = {}
    for name, p in (("column", column), ("planes", planes)):
        wl.plan_model(p)
        per[name] = wl.fp64_inst_per_cell_step
    r = column["groups"][0]["rows_per_lane"]
    assert 4 + (r + 1) / r <= per["column"] < 6 <= per["planes"] <= 7
    wl.plan_model(column, column, planes)
    assert wl.fp64_inst_per_cell_step == pytest.approx((2 * per["column"] + per["planes"]) / 3)
