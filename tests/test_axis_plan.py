"""Maps fused into the prologue of axis reductions: what the planner takes in,
and what it leaves room for."""
import pytest

from paper_2107_00555_gb300 import Graph
from paper_2107_00555_gb300 import _capi as C

SHAPE = (30, 41)


def _groups(g, flags=C.DCP_FUSE_ALL):
    g.fuse(flags)
    return [(p["kind"], p["members"], p["loads"], p["reductions"]) for p in g.plan()["groups"]]


def test_other_reductions_leave_room_for_those_of_the_prologue():
    """A reduction of the prologue's later maps always finds a place in its
    kernel (16 reductions), whatever was reduced in between."""
    g = Graph()
    x = g.input("f32", SHAPE)
    others = [g.input("f32", SHAPE) for _ in range(5)]
    y = g.map("square", [x])
    g.output(g.reduce(y, "sum", axis=1))
    for o in others:
        for op in ("sum", "min", "max"):
            g.output(g.reduce(o, op, axis=1))
    z = g.map("abs", [y])
    for op in ("sum", "min", "max"):
        g.output(g.reduce(z, op, axis=1))
    kinds = _groups(g)
    assert kinds[0] == ("axis_reduce", 2, 5, 16)  # y, z; 4 + 12 reductions of 1 + 4 arrays
    assert kinds[1:] == [("axis_reduce", 0, 1, 3)]


def test_other_reductions_leave_room_for_the_loads_of_the_prologue():
    """16 loads per kernel: the maps still to come read 13 arrays."""
    g = Graph()
    x = g.input("f32", SHAPE)
    operands = [g.input("f32", SHAPE) for _ in range(12)]
    others = [g.input("f32", SHAPE) for _ in range(5)]
    y = g.map("square", [x])
    g.output(g.reduce(y, "sum", axis=0))
    for o in others:
        g.output(g.reduce(o, "sum", axis=0))
    z = y
    for o in operands:
        z = g.map("add", [z, o])
    g.output(g.reduce(z, "sum", axis=0))
    assert _groups(g) == [("axis_reduce", 13, 16, 5), ("axis_reduce", 0, 2, 2)]


def test_maps_stay_apart_unless_maps_are_to_be_fused():
    """DCP_FUSE_SUBGRAPH alone takes a map into the reduction that reads it, and
    fuses no map with another."""
    g = Graph()
    x = g.input("f32", SHAPE)
    y = g.map("square", [x])
    g.output(g.reduce(y, "sum", axis=1))
    g.output(g.reduce(g.map("abs", [g.map("sub", [y, x])]), "max", axis=1))
    kinds = _groups(g, C.DCP_FUSE_SUBGRAPH)
    assert all(members <= 1 for _, members, _, _ in kinds)


@pytest.mark.parametrize("op,together", [("abs", True), ("sqrt", False), ("tanh", False), ("sin", False)])
def test_costly_binary64_maps_after_a_reduction_keep_their_own_kernel(op, together):
    """Counted over all the maps: those planned with the first reduction and
    those still to come."""
    g = Graph()
    y = g.map("square", [g.input("f64", SHAPE)])
    g.output(g.reduce(y, "sum", axis=0))
    g.output(g.reduce(g.map(op, [y]), "max", axis=0))
    kinds = [k for k, _, _, _ in _groups(g)]
    assert kinds == (["axis_reduce"] if together else ["map", "axis_reduce"])
