"""1-D streams against tiles, bit for bit, and the radius-2 star in every 2-D
form: lengths around a strip, its halos and a vector, each boundary, depth and
type, stored and reduced results, buffers off a vector boundary."""
import numpy as np
import pytest

from paper_2107_00555_gb300 import _capi as C
from paper_2107_00555_gb300 import Graph, inputs

from gpu_util import to_dev, to_host

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

STAR1 = {1: ([(0,), (-1,), (1,)], [0.5, 0.25, 0.25]),
         2: ([(0,), (-2,), (2,), (-1,), (1,)], [0.4, 0.1, 0.1, 0.2, 0.2])}
STAR2 = [(0, 0), (0, -1), (0, 1), (-1, 0), (1, 0), (0, -2), (0, 2), (-2, 0), (2, 0)]
W2 = [0.4, 0.1, 0.1, 0.1, 0.1, 0.05, 0.05, 0.05, 0.05]


def _run(x, offs, w, bc, steps, kernel, depth, off=False):
    g = Graph()
    u = g.stencil(g.input("f32" if x.dtype == np.float32 else "f64", x.shape), offs, w, bc, steps)
    g.output(u)
    g.output(g.reduce(u, "max"))
    g.set_option(C.DCP_OPT_STENCIL_KERNEL, kernel)
    g.set_option(C.DCP_OPT_TIME_TILE_DEPTH, depth)
    g.fuse(C.DCP_FUSE_ALL)
    assert g.plan()["groups"][0]["kernel_form"] == ("stream" if kernel else "tile")
    d = to_dev(x)
    outs = g.empty_outputs()
    if off:
        for k, t in enumerate((d, outs[0])):
            v = torch.empty(t.numel() + 1, dtype=t.dtype, device="cuda")[1:].view(t.shape)
            v.copy_(t)
            if k:
                outs[0] = v
            else:
                d = v
    return [to_host(o).tobytes() for o in g.run([d], outs)]


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("bc", ["zero", "periodic", "fixed_ring"])
def test_1d_streams_same_bits_as_tiles(bc, dtype):
    for n in (5, 60, 61, 62, 63, 64, 119, 120, 121, 124, 125, 128, 129, 1000, 4097, 70001):
        x = inputs.uniform((n,), -1.0, 1.0, n, dtype)
        for radius, (offs, w) in STAR1.items():
            ref = _run(x, offs, w, bc, 7, 0, 1)
            for depth in (1, 2, 3, 4):
                for off in (False, True):
                    assert _run(x, offs, w, bc, 7, 1, depth, off) == ref, (n, radius, depth, off)


@pytest.mark.parametrize("bc", ["zero", "periodic"])
@pytest.mark.parametrize("shape", [(37, 130), (300, 257)])
def test_radius_two_star_on_its_deferred_weight(shape, bc):
    x = inputs.uniform(shape, -1.0, 1.0, 5, np.float64)
    ref = _run(x, STAR2, W2, bc, 9, 0, 1)
    for kernel, depth in ((0, 3), (1, 1), (1, 2), (1, 4)):
        assert _run(x, STAR2, W2, bc, 9, kernel, depth) == ref
    u = x
    for _ in range(9):
        p = np.pad(u, 2, mode="wrap" if bc == "periodic" else "constant")
        u = sum(c * p[2 + dy:2 + dy + shape[0], 2 + dx:2 + dx + shape[1]] for c, (dy, dx) in zip(W2, STAR2))
    got = np.frombuffer(ref[0]).reshape(shape)
    # 9 convex steps of at most 10 roundings each on either side
    assert np.abs(got - u).max() <= 9 * 20 * np.finfo(np.float64).eps
