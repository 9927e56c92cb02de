"""Row reductions whose length is no multiple of a vector, and maps that follow
one reduction of a shared prologue before the next."""
import numpy as np
import pytest

import oracle
from paper_2107_00555_gb300 import Graph
from paper_2107_00555_gb300 import _capi as C


def _two_reductions(shape, dtype, axis):
    """sum(x*x) and max|x*x - x| along the axis: the second's maps come after
    the first's reduction."""
    g = Graph()
    x = g.input(dtype, shape)
    y = g.map("mul", [x, x])
    g.output(g.reduce(y, "sum", axis=axis))
    z = g.map("abs", [g.map("sub", [y, x])])
    g.output(g.reduce(z, "max", axis=axis))
    return g


def test_later_maps_join_the_axis_prologue():
    for axis in (0, 1):
        g = _two_reductions((30, 41), "f32", axis)
        assert g.fuse(C.DCP_FUSE_ALL) == 1
        (grp,) = g.plan()["groups"]
        assert (grp["kind"], grp["members"], grp["loads"], grp["reductions"]) == ("axis_reduce", 3, 1, 2)
    # a later map that is also stored, or reduced along another axis, keeps the maps apart
    for other in ("output", "axis"):
        g = Graph()
        x = g.input("f64", (30, 41))
        y = g.map("mul", [x, x])
        g.output(g.reduce(y, "sum", axis=1))
        z = g.map("sub", [y, x])
        g.output(z if other == "output" else g.reduce(z, "sum", axis=0))
        if other == "output":
            g.output(g.reduce(z, "sum", axis=1))
        g.fuse(C.DCP_FUSE_ALL)
        assert g.plan()["groups"][0]["kind"] == "map"


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("shape", [(1, 512), (7, 513), (9, 1026), (5, 4099), (3, 100003), (300, 515), (2, 3)])
def test_row_sums_of_any_length(shape, dtype):
    """Row starts at every alignment; the sum against the oracle's exactly
    rounded one within the backward-stable bound, the maximum exact."""
    from gpu_util import to_dev, to_host
    np_dt = np.float32 if dtype == "f32" else np.float64
    x = np.random.default_rng(sum(shape)).standard_normal(shape).astype(np_dt)
    g = _two_reductions(shape, dtype, 1)
    g.fuse(C.DCP_FUSE_ALL)
    s, m = (to_host(o).astype(np.float64) for o in g.run([to_dev(x)]))
    y = (x * x).astype(np.float64)  # one rounding in the element type, like the map
    _, fs, ab = oracle.reduce_axis("sum", y, 1)
    assert np.all(np.abs(s - fs) <= (1e-4 if dtype == "f32" else 1e-10) * ab)
    z = np.max(np.abs(y - x), axis=1)
    eps = np.finfo(np_dt).eps  # x*x and the difference round once each (or together)
    assert np.all(np.abs(m - z) <= 2 * eps * (np.max(y, axis=1) + np.max(np.abs(x), axis=1)))
