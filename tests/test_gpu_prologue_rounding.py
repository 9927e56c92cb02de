"""Rounding of the maps fused in front of a stencil: what is 0 operation by
operation is 0.  (The stencil is the identity, so the program's output is the
prologue's value.)"""
import numpy as np
import pytest

from paper_2107_00555_gb300 import _capi as C
from paper_2107_00555_gb300 import Graph, inputs

from gpu_util import to_dev, to_host

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [(3000,), (300, 310), (600, 640), (20, 30, 40)]


def _run(build, shape, dtype, bc):
    np_dt = np.float32 if dtype == "f32" else np.float64
    g = Graph()
    a, b = g.input(dtype, shape), g.input(dtype, shape)
    g.output(g.stencil(build(g, a, b), [(0,) * len(shape)], [1.0], bc, 1))
    assert g.fuse(C.DCP_FUSE_ALL) == 1
    x = [inputs.uniform(shape, -1.0, 1.0, 31 + k, np_dt) for k in range(2)]
    return x, to_host(g.run([to_dev(v) for v in x])[0])


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("bc", ["zero", "periodic"])
@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_a_product_less_itself_is_zero(shape, bc, dtype):
    def one(g, a, b):
        m = g.map("mul", [a, b])
        return g.map("sub", [m, m])

    def two(g, a, b):
        return g.map("sub", [g.map("mul", [a, b]), g.map("mul", [b, a])])

    for build in (one, two):
        _, got = _run(build, shape, dtype, bc)
        assert not got.any()


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_opposite_sums_of_a_product_cancel(shape, dtype):
    """(b - a b) + (a b - b), the first product negated by a map of its own: 0."""
    def build(g, a, b):
        m = g.map("mul", [a, b])
        return g.map("add", [g.map("add", [g.map("neg", [m]), b]), g.map("sub", [m, b])])

    _, got = _run(build, shape, dtype, "zero")
    assert not got.any()
