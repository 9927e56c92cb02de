"""Stencils on rows of almost 2^31 elements, whose last strip reaches past what
an int holds.  All ones and power-of-two weights: every interior value stays 1,
and the ends equal those of a short array with the same boundary."""
import numpy as np
import pytest

from paper_2107_00555_gb300 import _capi as C
from paper_2107_00555_gb300 import Graph

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

OFFS, W = [(0,), (-1,), (1,), (2,)], [0.5, 0.25, 0.125, 0.125]


def _run(x, bc, steps):
    g = Graph()
    g.output(g.stencil(g.input("f32", tuple(x.shape)), OFFS, W, bc, steps))
    g.set_option(C.DCP_OPT_STENCIL_KERNEL, 1)
    g.fuse(C.DCP_FUSE_ALL)
    return g.run([x])[0]


@pytest.mark.parametrize("n", [(1 << 31) - 1, (1 << 31) - 64, (1 << 31) - 120])
@pytest.mark.parametrize("bc", ["zero", "periodic"])
def test_last_strip_of_the_longest_rows(bc, n):
    steps, m = 3, 64
    x = torch.ones(n, dtype=torch.float32, device="cuda")
    x[0], x[-1] = 4.0, 8.0  # the ends differ, so a wrapped read of the wrong cell shows
    short = torch.cat([x[:m], x[-m:]])
    got, want = _run(x, bc, steps), _run(short, bc, steps)
    assert torch.equal(got[:m // 2], want[:m // 2]) and torch.equal(got[-m // 2:], want[-m // 2:])
    assert int((got[m // 2:-m // 2] != 1).sum()) == 0
    del x, got
    torch.cuda.empty_cache()
