"""Autotuner cache files written by hand: the key of a stencil group (the text
runtime.cpp hashes) and a run with chosen configurations in a process of its
own (a process reads the file once)."""
import json
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
DTYPE = {"f32": 1, "f64": 2}
BC = {"zero": 0, "periodic": 1, "fixed_ring": 2}


def key(sms, dtype, bc, shape, steps, offsets, epi=0, post=0, reds=0, col=False):
    """Key of one unbatched stencil group without a prologue."""
    pad = [tuple([0] * (3 - len(o))) + tuple(o) for o in offsets]
    text = "sm%d|k1|t%d|bc%d|s%s|n%d|o%s|p0,%d,%d%s%s" % (
        sms, DTYPE[dtype], BC[bc], "".join("%dx" % s for s in shape), steps,
        "".join("%d," % c for o in pad for c in o), post, reds, (",%d" % epi) * steps,
        "|col" if col else "")
    h = 1469598103934665603
    for c in text.encode():
        h = (h ^ c) * 1099511628211 % (1 << 64)
    return "%016x" % h


def column(rows_per_lane, planes, lanes, depth=1):
    """The configuration of 3-D columns."""
    return (depth, -3, rows_per_lane, planes, lanes)


def planes():
    """The configuration of the 3-D shared-memory planes."""
    return (1, 16, 8, 32, 1)


def run(script, entries, tmp_path, *args):
    """Runs a test module's script with a cache of {key: configuration}; its
    last line is JSON."""
    f = os.path.join(str(tmp_path), "tune.txt")
    with open(f, "w") as out:
        for k, cfg in entries.items():
            out.write("%s %s\n" % (k, " ".join(map(str, cfg))))
    env = dict(os.environ, DCP_TUNE_CACHE=f,
               PYTHONPATH=os.pathsep.join([ROOT, os.path.join(ROOT, "tests")]))
    r = subprocess.run([sys.executable, "-c", script] + [str(a) for a in args], env=env, cwd=ROOT,
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-3000:]
    return json.loads(r.stdout.splitlines()[-1])
