"""Performance cases: the work users of the package have it do, through its
public entry points (``dcp.program``, ``Graph.run`` / ``prepare`` /
``adjoint`` and ``autograd.apply``).

Each case is one program of a family the package is built for, at a size from
its tests, its benchmark or of the same kind:

* ``map``      y = exp(a*x + b) * sin(x) - 0.5*x*x over flat arrays, reduced to
               sum and max|y| and / or returned whole;
* ``axis``     the same maps with both reductions along one axis of a matrix;
* ``jacobi``   iterated 5-point averages in 2-D, as a stencil node or in the
               traced slice form (fixed ring);
* ``heat``     iterated 7-point steps in 3-D;
* ``batch``    many 2-D instances of uneven size in one program;
* ``adjoint``  value and gradient of sum(u_T^2), u_{t+1} = tanh(S u_t), in 2-D
               (through torch autograd) or 3-D (through ``Graph.adjoint``).
"""
import math

import numpy as np
import torch

import paper_2107_00555_gb300 as dcp
from paper_2107_00555_gb300 import _capi as C
from paper_2107_00555_gb300 import autograd, programs
from paper_2107_00555_gb300.graph import Graph

TORCH = {"f32": torch.float32, "f64": torch.float64}
SIZE = {"f32": 4, "f64": 8}


def listed():
    return [
        # a diagnostic evaluated inside a host loop: latency of one small call
        {"name": "map_small_f32", "kind": "map", "dtype": "f32", "n": 1500, "outputs": "reductions"},
        # the benchmark's fused map + reductions over a device-sized array
        {"name": "map_reduce_f32", "kind": "map", "dtype": "f32", "n": 1 << 26, "outputs": "reductions"},
        # scientific double precision, the mapped array kept; odd length
        {"name": "map_array_f64", "kind": "map", "dtype": "f64", "n": 10000019, "outputs": "both"},
        # per-row statistics of a matrix whose rows are not a multiple of 4 long
        {"name": "rows_f32_odd", "kind": "axis", "dtype": "f32", "ny": 6007, "nx": 4999, "axis": 1},
        # the small grid of the benchmark: ten steps that fit in L2
        {"name": "jacobi_small_f64", "kind": "jacobi", "dtype": "f64", "ny": 256, "nx": 256,
         "bc": "zero", "steps": 10},
        # the slice form of jacobi_2d in its usual single-precision run, long time loop
        {"name": "jacobi_ring_f32", "kind": "jacobi", "dtype": "f32", "ny": 4000, "nx": 4100,
         "bc": "ring", "steps": 50},
        # a periodic box in double precision with odd extents
        {"name": "jacobi_periodic_f64", "kind": "jacobi", "dtype": "f64", "ny": 2047, "nx": 2051,
         "bc": "periodic", "steps": 20},
        # the benchmark's default line: the large 3-D heat equation
        {"name": "heat_f64", "kind": "heat", "dtype": "f64", "nz": 512, "ny": 512, "nx": 512,
         "bc": "periodic", "steps": 50},
        # a ragged box in single precision with a zero border
        {"name": "heat_f32", "kind": "heat", "dtype": "f32", "nz": 300, "ny": 333, "nx": 381,
         "bc": "zero", "steps": 20},
        # the benchmark's batch: thousands of independent grids of uneven size
        {"name": "batch_f32", "kind": "batch", "dtype": "f32", "count": 4096, "lo": 32, "hi": 512,
         "sides_seed": 1004, "steps": 20},
        # gradient of a 3-D nonlinear chain in double precision (the benchmark's reverse pass)
        {"name": "adjoint3d_f64", "kind": "adjoint", "dtype": "f64", "nz": 256, "ny": 256, "nx": 256,
         "bc": "periodic", "steps": 20},
        # loss and gradient of a 2-D chain in a torch training step
        {"name": "adjoint2d_f32", "kind": "adjoint", "dtype": "f32", "nz": 0, "ny": 4096, "nx": 4096,
         "bc": "periodic", "steps": 20},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["map", "map", "axis", "jacobi", "jacobi", "heat", "heat", "batch", "adjoint"])
    dtype = rng.choice(["f32", "f64"])
    if kind == "map":
        return {"kind": kind, "dtype": dtype, "n": _log(rng, 1000, 1 << 26),
                "outputs": rng.choice(["reductions", "both"])}
    if kind == "axis":
        return {"kind": kind, "dtype": dtype, "ny": _log(rng, 64, 8192), "nx": _log(rng, 64, 8192),
                "axis": rng.choice([0, 1])}
    if kind == "jacobi":
        side = _log(rng, 48, 6000)
        return {"kind": kind, "dtype": dtype, "ny": side, "nx": max(32, int(side * rng.uniform(0.6, 1.3))),
                "bc": rng.choice(["zero", "periodic", "ring"]), "steps": rng.randint(5, 50)}
    if kind == "heat":
        n = [_log(rng, 40, 400) for _ in range(3)]
        return {"kind": kind, "dtype": dtype, "nz": n[0], "ny": n[1], "nx": n[2],
                "bc": rng.choice(["zero", "periodic"]), "steps": rng.randint(5, 30)}
    if kind == "batch":
        return {"kind": kind, "dtype": "f32", "count": _log(rng, 64, 2048), "lo": 32,
                "hi": rng.choice([128, 256, 512]), "sides_seed": rng.randint(1, 10**6),
                "steps": rng.randint(5, 30)}
    if rng.random() < 0.5:
        return {"kind": kind, "dtype": dtype, "nz": 0, "ny": _log(rng, 200, 3000),
                "nx": _log(rng, 200, 3000), "bc": rng.choice(["zero", "periodic"]),
                "steps": rng.randint(5, 20)}
    n = [_log(rng, 40, 200) for _ in range(3)]
    return {"kind": kind, "dtype": dtype, "nz": n[0], "ny": n[1], "nx": n[2],
            "bc": rng.choice(["zero", "periodic"]), "steps": rng.randint(5, 20)}


# -- inputs ------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _normal(case, shape, seed):
    """x, a, b ~ N(0, 1)."""
    g = _gen(seed)
    return [torch.randn(shape, generator=g, device="cuda", dtype=TORCH[case["dtype"]])
            for _ in range(3)]


def _field(case, seed):
    """Initial field: U[0, 1) in 2-D, U[-1, 1) in 3-D and for the nonlinear chains."""
    shape = _shape(case)
    u = torch.rand(shape, generator=_gen(seed), device="cuda", dtype=TORCH[case["dtype"]])
    return u if case["kind"] == "jacobi" else u * 2 - 1


def _shape(case):
    if case["kind"] == "map":
        return (case["n"],)
    if case.get("nz", 0):
        return (case["nz"], case["ny"], case["nx"])
    return (case["ny"], case["nx"])


def _sides(case):
    """Instance sides, log-uniform in [lo, hi]."""
    rng = np.random.default_rng(case["sides_seed"])
    s = np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]), size=case["count"]))
    return [int(v) for v in np.clip(np.rint(s), case["lo"], case["hi"])]


def _slab(sides):
    """Offsets of the instances in one buffer (each on a 128-byte boundary) and its length."""
    offs, at = [], 0
    for s in sides:
        offs.append(at)
        at += (s * s + 31) // 32 * 32
    return offs, at


def _instances(sides, seed):
    """All instances, U[0, 1), as one float32 buffer (its gaps are drawn too and never read)."""
    _, total = _slab(sides)
    return torch.rand(total, generator=_gen(seed), device="cuda", dtype=torch.float32)


def _views(buf, sides):
    offs, _ = _slab(sides)
    return [buf[o:o + s * s].view(s, s) for o, s in zip(offs, sides)]


# -- programs ----------------------------------------------------------------

def _map_program(case):
    spec = (case["dtype"], _shape(case))
    axis = case.get("axis")

    def f(x, a, b):
        y = dcp.exp(a * x + b) * dcp.sin(x) - 0.5 * x * x
        red = (y.sum(axis=axis), abs(y).max(axis=axis))
        return red + (y,) if case.get("outputs") == "both" else red

    return dcp.program(spec, spec, spec)(f)


def _jacobi_program(case):
    if case["bc"] == "ring":
        steps = case["steps"]

        def f(A):
            for _ in range(steps):
                A[1:-1, 1:-1] = 0.2 * (A[1:-1, 1:-1] + A[1:-1, :-2] + A[1:-1, 2:]
                                       + A[2:, 1:-1] + A[:-2, 1:-1])
            return A

        return dcp.program((case["dtype"], _shape(case)))(f).graph
    return programs.jacobi2d(_shape(case), case["steps"], case["bc"], case["dtype"],
                             fuse=C.DCP_FUSE_ALL)


def _adjoint_graph(case):
    if case["nz"]:
        return programs.tanh_chain(_shape(case), case["steps"], case["bc"], case["dtype"],
                                   fuse=C.DCP_FUSE_ALL)
    g = Graph()
    u = g.input(case["dtype"], _shape(case))
    for _ in range(case["steps"]):
        u = g.map("tanh", [g.stencil(u, programs.FIVE_POINT, programs.FIVE_WEIGHTS, case["bc"], 1)])
    g.output(g.reduce(g.map("square", [u]), "sum"))
    g.fuse(C.DCP_FUSE_ALL)
    return g


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("map", "axis"):
        return {"kind": kind, "program": _map_program(case),
                "args": _normal(case, _shape(case), seed)}
    if kind == "batch":
        sides = _sides(case)
        src = _instances(sides, seed)
        dst = torch.zeros_like(src)
        g = programs.batch2d(sides, case["steps"], "zero", case["dtype"],
                             fuse=C.DCP_FUSE_ALL | C.DCP_BATCH)
        # thousands of fixed buffers: marshalled once, as the benchmark does
        return {"kind": kind, "call": g.prepare(_views(src, sides), _views(dst, sides)), "out": dst,
                "keep": (g, src)}
    u = _field(case, seed)
    if kind == "jacobi":
        return {"kind": kind, "graph": _jacobi_program(case), "args": [u]}
    if kind == "heat":
        g = programs.heat3d(_shape(case), case["steps"], case["bc"], case["dtype"],
                            fuse=C.DCP_FUSE_ALL)
        return {"kind": kind, "graph": g, "args": [u]}
    g = _adjoint_graph(case)
    if case["nz"]:
        one = torch.ones((), dtype=u.dtype, device="cuda")
        return {"kind": "adjoint3d", "graph": g, "args": [u], "grads": [one],
                "into": [torch.empty_like(u)]}
    return {"kind": "adjoint2d", "graph": g, "u": u.requires_grad_(True)}


def run(state):
    kind = state["kind"]
    if kind in ("map", "axis"):
        return state["program"](*state["args"])
    if kind in ("jacobi", "heat"):
        return state["graph"].run(state["args"])
    if kind == "batch":
        state["call"]()
        return state["out"]
    if kind == "adjoint3d":
        return state["graph"].adjoint(state["args"], state["grads"], state["into"])
    loss = autograd.apply(state["graph"], state["u"])
    (grad,) = torch.autograd.grad(loss, state["u"])
    return {"loss": loss.detach(), "grad": grad}


# -- compulsory work ---------------------------------------------------------

def work(case):
    """Each input read once and each output written once; floating operations
    of the program as written (a 5-point sum 9, a 7-point sum 13; exp, sin and
    tanh counted as 10, 15 and 14, the operations of a binary64 evaluation)."""
    kind, sz = case["kind"], SIZE[case["dtype"]]
    if kind == "batch":
        cells = sum(s * s for s in _sides(case))
        return {"bytes": 2 * sz * cells, "flops": 9.0 * cells * case["steps"]}
    cells = math.prod(_shape(case))
    if kind == "map":
        whole = case["outputs"] == "both"
        return {"bytes": sz * cells * (4 if whole else 3) + 2 * sz, "flops": 33.0 * cells}
    if kind == "axis":
        kept = cells // (case["ny"] if case["axis"] == 0 else case["nx"])
        return {"bytes": sz * (3 * cells + 2 * kept), "flops": 33.0 * cells}
    if kind == "jacobi":
        return {"bytes": 2 * sz * cells, "flops": 9.0 * cells * case["steps"]}
    if kind == "heat":
        return {"bytes": 2 * sz * cells, "flops": 13.0 * cells * case["steps"]}
    p = 13 if case["nz"] else 9
    # the states and the gradient: u_0 read, the gradient written; per step the
    # forward sum and tanh, the transposed sum and the derivative
    return {"bytes": 2 * sz * cells, "flops": (2.0 * p + 14 + 3) * cells * case["steps"]}


# -- the same in 64 bits, plain torch ----------------------------------------

def _shift(u, axis, by, periodic):
    """v[p] = u[p + by] along axis; zero outside unless periodic."""
    v = torch.roll(u, -by, axis)
    if not periodic:
        v.narrow(axis, u.shape[axis] - 1 if by > 0 else 0, 1).zero_()
    return v


def _average(u, centre, side, periodic, axes):
    s = torch.zeros_like(u)
    for ax in axes:
        s += _shift(u, ax, -1, periodic)
        s += _shift(u, ax, 1, periodic)
    return centre * u + side * s


def _maps64(case, seed):
    x, a, b = (t.double() for t in _normal(case, _shape(case), seed))
    return torch.exp(a * x + b) * torch.sin(x) - 0.5 * x * x


def exact(case, seed):
    kind = case["kind"]
    if kind == "map":
        y = _maps64(case, seed)
        red = [y.sum(), y.abs().max()]
        return red + [y] if case["outputs"] == "both" else red
    if kind == "axis":
        y = _maps64(case, seed)
        return [y.sum(case["axis"]), y.abs().amax(case["axis"])]
    if kind == "batch":
        return _exact_batch(case, seed)
    u = _field(case, seed).double()
    periodic = case["bc"] == "periodic"
    three = bool(case.get("nz", 0))
    centre, side, axes = (0.4, 0.1, (2, 1, 0)) if three else (0.2, 0.2, (1, 0))
    if kind in ("jacobi", "heat"):
        for _ in range(case["steps"]):
            v = _average(u, centre, side, periodic, axes)
            if case["bc"] == "ring":
                u = u.clone()
                u[1:-1, 1:-1] = v[1:-1, 1:-1]
            else:
                u = v
        return [u]
    states = [u]
    for _ in range(case["steps"]):
        states.append(torch.tanh(_average(states[-1], centre, side, periodic, axes)))
    grad = 2 * states[-1]
    for t in range(case["steps"], 0, -1):
        # the average is its own transpose
        grad = _average(grad * (1 - states[t] ** 2), centre, side, periodic, axes)
    return [grad] if three else {"loss": states[-1].square().sum(), "grad": grad}


def _exact_batch(case, seed):
    sides = _sides(case)
    src = _instances(sides, seed).double()
    dst = torch.zeros_like(src)
    offs, _ = _slab(sides)
    order = sorted(range(len(sides)), key=lambda i: sides[i])
    for at in range(0, len(order), 64):  # instances of similar size side by side, zeros around
        part = order[at:at + 64]
        n = sides[part[-1]]
        u = torch.zeros(len(part), n, n, dtype=torch.float64, device="cuda")
        inside = torch.zeros_like(u)
        for k, i in enumerate(part):
            s = sides[i]
            u[k, :s, :s] = src[offs[i]:offs[i] + s * s].view(s, s)
            inside[k, :s, :s] = 1
        for _ in range(case["steps"]):
            u = _average(u, 0.2, 0.2, False, (2, 1)) * inside
        for k, i in enumerate(part):
            s = sides[i]
            dst[offs[i]:offs[i] + s * s] = u[k, :s, :s].reshape(-1)
    return dst
