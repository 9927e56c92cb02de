"""The warp-streamed kernel forms against the shared-memory forms, bit for bit,
over the programs their dispatch accepts: 3-D columns (any boundary, partial
stars, extents around a warp's columns and rows, step epilogues, stored and
reduced results, buffers off a vector boundary) and periodic 2-D streams."""
import numpy as np
import pytest

import oracle
from oracle import programs as OP
from paper_2107_00555_gb300 import Graph, inputs, programs
from paper_2107_00555_gb300 import _capi as C

from gpu_util import assert_close, to_dev, to_host, tol_for

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NP = {"f32": np.float32, "f64": np.float64}
SEVEN, W7 = programs.SEVEN_POINT, programs.SEVEN_WEIGHTS


def _build(shape, dtype, bc, steps, offs, w, epi, post):
    g = Graph()
    u = g.input(dtype, shape)
    if epi is None:
        u = g.stencil(u, offs, w, bc, steps)
    else:
        for _ in range(steps):
            u = g.map(epi, [g.stencil(u, offs, w, bc, 1)])
    g.output(u)
    if post:
        g.output(g.map("add_s", [u], 0.25))
        g.output(g.reduce(u, "max"))
    return g


def _run(g, planes, dev):
    if planes:  # a tile option keeps the shared-memory planes
        g.set_option(C.DCP_OPT_CELLS_PER_THREAD, 2)
    g.fuse(C.DCP_FUSE_ALL)
    forms = {x["kernel_form"] for x in g.plan()["groups"] if x["kind"] == "stencil"}
    return forms, [to_host(o).tobytes() for o in g.run([dev])]


CASES = [
    # shape, steps, offsets, weights, epilogue, post
    ((40, 41, 43), 5, SEVEN, W7, None, False),
    ((97, 33, 64), 4, SEVEN, W7, None, True),
    ((70, 64, 121), 3, SEVEN, W7, None, False),
    ((65, 9, 260), 5, SEVEN, W7, None, True),
    ((3, 130, 128), 6, SEVEN, W7, None, False),
    ((50, 40, 119), 4, SEVEN, W7, "tanh", False),
    ((40, 60, 72), 3, [(0, 0, 0), (-1, 0, 0), (1, 0, 0)], [0.5, 0.25, 0.25], None, False),
    ((33, 48, 65), 4, [(0, 0, 1), (0, -1, 0), (0, 1, 0), (-1, 0, 0), (1, 0, 0)],
     [0.4, 0.15, 0.15, 0.15, 0.15], None, False),
    ((1, 50, 60), 3, SEVEN, W7, None, False),
    ((260, 5, 6), 3, SEVEN, W7, None, False),
]


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("bc", ["zero", "periodic", "fixed_ring"])
def test_columns_same_bits_as_planes(bc, dtype):
    seen = set()
    for k, (shape, steps, offs, w, epi, post) in enumerate(CASES):
        u0 = inputs.uniform(shape, -1.0, 1.0, 60 + k, NP[dtype])
        d = to_dev(u0)
        f, a = _run(_build(shape, dtype, bc, steps, offs, w, epi, post), False, d)
        _, b = _run(_build(shape, dtype, bc, steps, offs, w, epi, post), True, d)
        seen |= f
        assert a == b, (shape, offs, epi, post)
    if dtype == "f32":
        assert "column" in seen


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("bc", ["zero", "periodic"])
def test_columns_large_against_planes_and_oracle(bc, dtype):
    """A grid large enough for whole waves of columns in both types."""
    shape, steps = (130, 200, 256), 3
    u0 = inputs.uniform(shape, -1.0, 1.0, 71, NP[dtype])
    d = to_dev(u0)
    f, a = _run(_build(shape, dtype, bc, steps, SEVEN, W7, None, False), False, d)
    _, b = _run(_build(shape, dtype, bc, steps, SEVEN, W7, None, False), True, d)
    assert a == b and (dtype == "f64" or f == {"column"})
    ref = oracle.run(OP.heat3d(shape, steps, bc), [u0.astype(np.float64)])[-1]
    assert_close(np.frombuffer(a[0], NP[dtype]).reshape(shape), ref, tol_for(dtype), 1.0, "columns")


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("nd", [2, 3])
def test_buffers_off_a_vector_boundary(nd, dtype):
    """Inputs and outputs one element past a 16-byte boundary."""
    shape = (600, 640) if nd == 2 else (60, 64, 128)
    build = programs.jacobi2d if nd == 2 else programs.heat3d
    u0 = inputs.uniform(shape, -1.0, 1.0, 72, NP[dtype])
    n = u0.size
    g = build(shape, 5, "periodic", dtype, fuse=C.DCP_FUSE_ALL)
    ref = to_host(g.run([to_dev(u0)])[0])
    src = torch.empty(n + 1, dtype=torch.float32 if dtype == "f32" else torch.float64, device="cuda")
    dst = torch.empty_like(src)
    src[1:].view(shape).copy_(to_dev(u0))
    got = to_host(g.run([src[1:].view(shape)], [dst[1:].view(shape)])[0])
    assert got.tobytes() == ref.tobytes()


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("shape", [(5, 3), (1, 70), (70, 1), (37, 130), (300, 257), (64, 640)])
def test_periodic_stream_same_bits_as_tiles(shape, dtype):
    u0 = inputs.uniform(shape, 0.0, 1.0, 73, NP[dtype])
    d, T = to_dev(u0), 9
    res = []
    for kernel, depth, rows in ((0, 1, None), (1, 1, None), (1, 4, 7), (1, 9, None), (1, 3, 300)):
        g = programs.jacobi2d(shape, T, "periodic", dtype)
        g.set_option(C.DCP_OPT_STENCIL_KERNEL, kernel)
        g.set_option(C.DCP_OPT_TIME_TILE_DEPTH, depth)
        if rows is not None:
            g.set_option(C.DCP_OPT_STREAM_ROWS, rows)
        g.fuse(C.DCP_FUSE_ALL)
        assert g.plan()["groups"][0]["kernel_form"] == ("stream" if kernel else "tile")
        res.append(to_host(g.run([d])[0]).tobytes())
    assert all(r == res[0] for r in res)
    ref = oracle.run(OP.jacobi2d(shape, T, "periodic"), [u0.astype(np.float64)])[-1]
    assert_close(np.frombuffer(res[0], NP[dtype]).reshape(shape), ref, tol_for(dtype), 1.0, "periodic")
