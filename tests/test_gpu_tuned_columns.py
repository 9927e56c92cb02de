"""A tuned configuration is applied only to stencil groups that can run it: 3-D
columns sum binary64 stars on a deferred weight, which depends on the weights
and on DCP_OPT_DEFERRED_WEIGHT, not on the neighbourhood alone."""
import pytest

import tune_util

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPE, STEPS = (30, 40, 66), 4

SCRIPT = """
import json, sys
import numpy as np
from paper_2107_00555_gb300 import Graph, inputs, programs
from paper_2107_00555_gb300 import _capi as C
from gpu_util import to_dev, to_host
from test_gpu_tuned_columns import SHAPE, STEPS

SEVEN = programs.SEVEN_POINT
even, uneven = programs.SEVEN_WEIGHTS, [0.37, 0.1, 0.11, 0.12, 0.13, 0.08, 0.09]
u0 = inputs.uniform(SHAPE, -1.0, 1.0, 5, np.float64)
out = []
for w, deferred in ((even, True), (uneven, True), (even, False)):
    g = Graph()
    g.output(g.stencil(g.input("f64", SHAPE), SEVEN, w, "periodic", STEPS))
    if not deferred:
        g.set_option(C.DCP_OPT_DEFERRED_WEIGHT, 0)
    g.fuse(C.DCP_FUSE_ALL | C.DCP_AUTOTUNE)
    d = to_dev(u0)
    got = [to_host(g.run([d])[0]) for _ in range(2)]
    ref = u0
    for _ in range(STEPS):
        ref = sum(c * np.roll(ref, [-o for o in off], (0, 1, 2)) for c, off in zip(w, SEVEN))
    err = max(float(np.abs(x - ref).max()) for x in got)
    out.append([g.plan()["groups"][0]["kernel_form"], err])
print(json.dumps(out))
"""


def test_columns_of_a_cache_file_only_where_they_apply(tmp_path):
    args = (torch.cuda.get_device_properties(0).multi_processor_count, "f64", "periodic", SHAPE, STEPS,
            [(0, 0, 0), (0, 0, -1), (0, 0, 1), (0, -1, 0), (0, 1, 0), (-1, 0, 0), (1, 0, 0)])
    entries = {tune_util.key(*args, col=c): tune_util.column(4, 8, 32) for c in (False, True)}
    (form, err), *others = tune_util.run(SCRIPT, entries, tmp_path)
    assert form == "column" and err <= 1e-13
    for form, err in others:
        assert form != "column" and err <= 1e-13


def test_entries_no_column_can_run_are_tuned_again(tmp_path):
    """No planes per item, too deep, rows or lanes no kernel has."""
    args = (torch.cuda.get_device_properties(0).multi_processor_count, "f64", "periodic", SHAPE, STEPS,
            [(0, 0, 0), (0, 0, -1), (0, 0, 1), (0, -1, 0), (0, 1, 0), (-1, 0, 0), (1, 0, 0)])
    for cfg in (tune_util.column(4, 0, 32), tune_util.column(4, 8, 32, depth=2), tune_util.column(3, 8, 32)):
        out = tune_util.run(SCRIPT, {tune_util.key(*args, col=True): cfg}, tmp_path)
        assert all(err <= 1e-13 for _, err in out)
