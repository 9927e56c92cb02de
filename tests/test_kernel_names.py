"""A kernel's name, and with it the key of its compiled module in memory and on
disk, changes with every skeleton its source includes, nested ones too."""
import json
import os
import shutil
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NAMES = """
import json, sys
sys.path.insert(0, sys.argv[1])
from paper_2107_00555_gb300 import Graph, build, _capi
build.build()
assert _capi.__file__.startswith(sys.argv[1])
out = {}
for op in ("tanh", "sqrt"):
    g = Graph()
    g.output(g.map(op, [g.input("f64", (100,))]))
    g.fuse(_capi.DCP_FUSE_ALL)
    out[op] = g.plan()["launches"][0]["kernel"]
print(json.dumps(out))
"""


def _names(root):
    r = subprocess.run([sys.executable, "-c", NAMES, str(root)], cwd=str(root), capture_output=True,
                       text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    return json.loads(r.stdout.splitlines()[-1])


def test_a_changed_table_changes_the_names_of_its_kernels(tmp_path):
    for d in ("paper_2107_00555_gb300", "include"):
        shutil.copytree(os.path.join(ROOT, d), tmp_path / d)
    before = _names(ROOT)
    table = tmp_path / "paper_2107_00555_gb300" / "csrc" / "kernels" / "k_tanh64_table.cuh"
    text = table.read_text()
    assert "0x1.084c29efe8664p-9" in text  # c0 of the first row
    table.write_text(text.replace("0x1.084c29efe8664p-9", "0x1.084c29efe8665p-9"))
    after = _names(tmp_path)
    assert after["tanh"] != before["tanh"]
    assert after["sqrt"] == before["sqrt"]
