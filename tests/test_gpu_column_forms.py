"""3-D columns in every form the planner can emit (rows per lane, lanes along
x, steps per launch), each forced through the autotuner's cache file, against
the shared-memory planes bit for bit: extents around a warp's rows and
columns, items shorter and longer than the grid, stored and reduced results,
buffers off a vector boundary."""
import json

import numpy as np
import pytest

import tune_util

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

STEPS = 3
SHAPES = [(13, 40, 70), (5, 33, 64), (20, 9, 121), (2, 17, 260), (9, 3, 5), (1, 1, 36)]
BCS = {"f32": ["zero", "periodic", "fixed_ring"], "f64": ["zero", "periodic"]}
FORMS = [("f64", cy, lx, 1) for cy in (8, 4, 2) for lx in (32, 16)] + \
        [("f32", cy, 32, depth) for cy in (4, 2) for depth in (1, 2)]


def _graph(dtype, shape, bc, post):
    from paper_2107_00555_gb300 import Graph, programs
    g = Graph()
    u = g.stencil(g.input(dtype, shape), programs.SEVEN_POINT, programs.SEVEN_WEIGHTS, bc, STEPS)
    g.output(u)
    if post:
        g.output(g.map("add_s", [u], 0.25))
        g.output(g.reduce(u, "max"))
    return g


def _off_boundary(t):
    """The same values one element past a 16-byte boundary."""
    buf = torch.empty(t.numel() + 1, dtype=t.dtype, device="cuda")
    v = buf[1:].view(t.shape)
    v.copy_(t)
    return v


def child(dtype):
    """Runs every grid twice as columns (the cache file's) and once as planes."""
    from gpu_util import to_dev, to_host
    from paper_2107_00555_gb300 import _capi as C
    from paper_2107_00555_gb300 import inputs
    bad, forms = [], set()
    for k, shape in enumerate(SHAPES):
        u0 = to_dev(inputs.uniform(shape, -1.0, 1.0, 40 + k, np.float32 if dtype == "f32" else np.float64))
        for bc in BCS[dtype]:
            post = k % 2 == 1
            ref = _graph(dtype, shape, bc, post)
            ref.set_option(C.DCP_OPT_CELLS_PER_THREAD, 2)  # keeps the planes
            ref.fuse(C.DCP_FUSE_ALL)
            assert ref.plan()["groups"][0]["kernel_form"] == "tile"
            want = [to_host(o).tobytes() for o in ref.run([u0])]
            g = _graph(dtype, shape, bc, post)
            g.fuse(C.DCP_FUSE_ALL | C.DCP_AUTOTUNE)
            aligned = [to_host(o).tobytes() for o in g.run([u0])]
            outs = [_off_boundary(o) if o.dim() else o for o in g.empty_outputs()]
            off = [to_host(o).tobytes() for o in g.run([_off_boundary(u0)], outs)]
            grp = g.plan()["groups"][0]
            forms.add((grp["kernel_form"], grp["rows_per_lane"], grp["lanes_x"], grp["depth"])
                      if grp["kernel_form"] == "column" else grp["kernel_form"])
            if aligned != want or off != want:
                bad.append([shape, bc, aligned != want, off != want])
    print(json.dumps({"forms": sorted(map(str, forms)), "bad": bad}))


@pytest.mark.parametrize("dtype,cy,lx,depth", FORMS)
def test_forced_columns_same_bits_as_planes(dtype, cy, lx, depth, tmp_path):
    from paper_2107_00555_gb300 import programs
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    entries = {}
    for k, shape in enumerate(SHAPES):
        for bc in BCS[dtype]:
            post = k % 2 == 1
            key = tune_util.key(sms, dtype, bc, shape, STEPS, programs.SEVEN_POINT, post=int(post),
                                reds=int(post), col=True)
            entries[key] = tune_util.column(cy, (4, 64)[k % 3 == 1], lx, depth)
    out = tune_util.run("import sys, test_gpu_column_forms as t; t.child(sys.argv[1])", entries, tmp_path, dtype)
    assert out["forms"] == [str(("column", cy, lx, depth))]
    assert out["bad"] == []
