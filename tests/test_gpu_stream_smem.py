"""Warp-stream launches whose rings take exactly 48 KB, beside the shared memory
of a final reduction."""
import numpy as np
import pytest

from paper_2107_00555_gb300 import _capi as C
from paper_2107_00555_gb300 import inputs, programs
from paper_2107_00555_gb300.graph import Graph

from gpu_util import to_dev, to_host

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads", [352, 384, 416])
def test_rings_of_48_kb_with_a_reduction(threads):
    shape = (700, 640)
    u0 = inputs.uniform(shape, 0.0, 1.0, 3, np.float32)
    out = []
    for option in (False, True):
        g = Graph()
        u = g.stencil(g.input("f32", shape), programs.FIVE_POINT, programs.FIVE_WEIGHTS, "zero", 3)
        g.output(u)
        g.output(g.reduce(u, "max"))
        g.set_option(C.DCP_OPT_STENCIL_KERNEL, 1)
        if option:
            g.set_option(C.DCP_OPT_STREAM_THREADS, threads)
        g.fuse(C.DCP_FUSE_ALL)
        launch = g.plan()["launches"][-1]
        if option:
            assert launch["threads"] == threads and launch["smem"] == threads // 32 * 4096
        out.append([to_host(o).tobytes() for o in g.run([to_dev(u0)])])
    assert out[0] == out[1]
