"""The plan description is JSON with one value per key."""
import json

import pytest

from paper_2107_00555_gb300 import _capi as C
from paper_2107_00555_gb300 import programs


def _unique(pairs):
    keys = [k for k, _ in pairs]
    assert len(set(keys)) == len(keys), keys
    return dict(pairs)


@pytest.mark.parametrize("build", [
    lambda: programs.heat3d((300, 320, 320), 3, "zero", "f32", fuse=C.DCP_FUSE_ALL),
    lambda: programs.heat3d((24, 24, 24), 3, "zero", "f64", fuse=C.DCP_FUSE_ALL),
    lambda: programs.jacobi2d((900, 800), 9, "zero", "f32", fuse=C.DCP_FUSE_ALL),
    lambda: programs.batch2d([40, 50], 4, "zero", "f32", fuse=C.DCP_FUSE_ALL | C.DCP_BATCH),
    lambda: programs.map_reduce((30, 41), "f32", fuse=C.DCP_FUSE_ALL, axis=1),
], ids=["columns", "planes", "stream", "batch", "axis"])
def test_keys_are_unique(build):
    g = build()
    plan = json.loads(C.dcp_plan_info(g._h), object_pairs_hook=_unique)
    assert plan["fused"] and plan["groups"] and plan["launches"]
