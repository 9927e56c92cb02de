"""Axis reductions of sums of several arrays, read element by element and in
vectors, along axes around the unrolled lengths."""
import numpy as np
import pytest

from paper_2107_00555_gb300 import _capi as C
from paper_2107_00555_gb300 import Graph

from gpu_util import to_dev, to_host

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("shape,axis", [((63, 41), 0), ((64, 41), 0), ((300, 7), 0), ((7, 63), 1), ((9, 65), 1),
                                        ((3, 50021), 1), ((3, 50020), 1), ((200, 1810), 1), ((200, 1808), 1)])
def test_sum_of_arrays_along_an_axis(shape, axis, dtype):
    """Integers small enough for every partial sum to be exact."""
    r = np.random.default_rng(shape[0])
    for arrays in (1, 2, 6, 16):
        g = Graph()
        name = "f32" if dtype == np.float32 else "f64"
        y = g.input(name, shape)
        for _ in range(arrays - 1):
            y = g.map("add", [y, g.input(name, shape)])
        g.output(g.reduce(y, "sum", axis=axis))
        g.output(g.reduce(y, "max", axis=axis))
        assert g.fuse(C.DCP_FUSE_ALL) == 1
        x = [r.integers(-8, 9, shape).astype(dtype) for _ in range(arrays)]
        s, m = (to_host(o) for o in g.run([to_dev(v) for v in x]))
        total = np.sum([v.astype(np.int64) for v in x], axis=0)
        assert np.array_equal(s, total.sum(axis)) and np.array_equal(m, total.max(axis))
