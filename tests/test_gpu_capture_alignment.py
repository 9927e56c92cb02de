"""A caller's own CUDA-graph capture of a stencil whose buffers lie off a vector
boundary, after runs on aligned buffers only: the kernel variant for them is
loaded inside the capture."""
import numpy as np
import pytest

from paper_2107_00555_gb300 import _capi as C
from paper_2107_00555_gb300 import Graph, inputs, programs

from gpu_util import to_dev, to_host

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("reduced", [False, True])
@pytest.mark.parametrize("shape,dtype", [((600, 640), "f64"), ((700, 516), "f32"), ((80, 200, 256), "f32")])
def test_first_misaligned_run_inside_a_capture(shape, dtype, reduced):
    offs, w = ((programs.FIVE_POINT, programs.FIVE_WEIGHTS) if len(shape) == 2
               else (programs.SEVEN_POINT, programs.SEVEN_WEIGHTS))
    g = Graph()
    # (a weight of its own per parameter set: kernels no other test has loaded)
    u = g.stencil(g.input(dtype, shape), offs, [x * (0.875 if reduced else 0.9375) for x in w], "zero", 4)
    g.output(u)
    if reduced:
        g.output(g.reduce(u, "max"))
    g.fuse(C.DCP_FUSE_ALL)
    assert g.plan()["groups"][0]["kernel_form"] in ("stream", "column")
    u0 = to_dev(inputs.uniform(shape, -1.0, 1.0, 9, np.float32 if dtype == "f32" else np.float64))
    want = [to_host(o) for o in g.run([u0])]
    src = torch.empty(u0.numel() + 1, dtype=u0.dtype, device="cuda")[1:].view(shape)
    src.copy_(u0)
    outs = g.empty_outputs()
    outs[0] = torch.zeros(u0.numel() + 1, dtype=u0.dtype, device="cuda")[1:].view(shape)
    torch.cuda.synchronize()
    cg = torch.cuda.CUDAGraph()
    with torch.cuda.graph(cg):
        g.run([src], outs)
    cg.replay()
    torch.cuda.synchronize()
    for o, ref in zip(outs, want):
        assert to_host(o).tobytes() == ref.tobytes()
