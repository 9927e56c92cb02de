"""A prepared call takes a stream, or anything false for torch's current one."""
import numpy as np
import pytest

from paper_2107_00555_gb300 import _capi as C
from paper_2107_00555_gb300 import programs

from gpu_util import to_dev, to_host

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_prepared_call_streams():
    x = np.arange(300.0).reshape(15, 20)
    g = programs.jacobi2d(x.shape, 3, "zero", "f64", fuse=C.DCP_FUSE_ALL)
    d = to_dev(x)
    want = to_host(g.run([d])[0]).tobytes()
    call = g.prepare([d])
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    for stream in (None, 0, torch.cuda.current_stream(), side):
        call.outputs[0].zero_()
        side.wait_stream(torch.cuda.current_stream())
        out = call(stream)[0]
        torch.cuda.current_stream().wait_stream(side)
        assert to_host(out).tobytes() == want
