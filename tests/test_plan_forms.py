"""Which kernel form, depth and work split the planner gives stencil programs
whose best form is not the one their family usually takes (no GPU needed)."""
import pytest

from paper_2107_00555_gb300 import _capi as C
from paper_2107_00555_gb300 import Graph, programs

STAR2 = [(0, 0), (0, -1), (0, 1), (-1, 0), (1, 0), (0, -2), (0, 2), (-2, 0), (2, 0)]
W2 = [0.4, 0.1, 0.1, 0.1, 0.1, 0.05, 0.05, 0.05, 0.05]


def _stencil(shape, dtype, bc, steps, offs=programs.FIVE_POINT, w=programs.FIVE_WEIGHTS, arrays=1,
             reduced=False, flags=C.DCP_FUSE_ALL):
    g = Graph()
    u = g.input(dtype, shape)
    for _ in range(arrays - 1):
        u = g.map("add", [g.map("mul_s", [u], 0.5), g.input(dtype, shape)])
    u = g.stencil(u, offs, w, bc, steps)
    g.output(u)
    if reduced:
        g.output(g.reduce(u, "max"))
    g.fuse(flags)
    plan = g.plan()
    return plan["groups"][0], plan["launches"]


def test_periodic_binary64_sums_without_shared_pairs_run_in_tiles():
    grp, _ = _stencil((1000, 1001), "f64", "periodic", 7, STAR2, W2)
    assert grp["kernel_form"] == "tile" and grp["tile"][1:] == [32, 32]
    grp, _ = _stencil((1000, 1001), "f64", "periodic", 1)
    assert grp["kernel_form"] == "tile"
    # a long run of 5-point averages, which share their pairs, streams
    grp, _ = _stencil((2047, 2051), "f64", "periodic", 20)
    assert grp["kernel_form"] == "stream"


def test_narrow_periodic_binary64_grids_run_in_tiles():
    for shape in ((1000000, 4), (1000000, 1)):
        grp, _ = _stencil(shape, "f64", "periodic", 10)
        assert grp["kernel_form"] == "tile"


@pytest.mark.parametrize("shape", [(500, 513), (1000, 1001)])
def test_steps_on_many_arrays_run_in_tiles(shape):
    assert _stencil(shape, "f32", "periodic", 1, arrays=8)[0]["kernel_form"] == "tile"
    assert _stencil(shape, "f64", "zero", 1, arrays=8)[0]["kernel_form"] == "tile"
    # long runs stream: their first launch alone reads the arrays
    assert _stencil((1000, 1001), "f32", "periodic", 9, arrays=8)[0]["kernel_form"] == "stream"


def test_one_step_on_a_small_binary64_grid_takes_large_tiles():
    """4 x 16 cells keep a quarter of a CTA's threads busy."""
    grp, _ = _stencil((500, 513), "f64", "periodic", 1)
    assert grp["tile"][1] * grp["tile"][2] >= 512


def test_tile_heights_follow_the_number_of_sms():
    """512 rows in 16 strips: two tiles for each of 152 SMs."""
    grp, _ = _stencil((512, 512), "f64", "zero", 10)
    assert grp["kernel_form"] == "tile" and grp["tile"][1:] == [27, 32]


def test_small_periodic_binary64_batches_run_in_tiles():
    sides = [32 + k % 33 for k in range(64)]
    g = programs.batch2d(sides, 20, "periodic", "f64", fuse=C.DCP_FUSE_ALL | C.DCP_BATCH)
    assert g.plan()["groups"][0]["kernel_form"] == "tile"


def test_launches_that_reduce_share_tickets_between_binary32_warps():
    grp, launches = _stencil((1000, 1001), "f32", "zero", 14, reduced=True)
    assert grp["kernel_form"] == "stream" and grp["threads"] == 32
    assert [l["threads"] for l in launches] == [32] * (len(launches) - 1) + [128]
    _, launches = _stencil((3000, 3100), "f64", "zero", 1, reduced=True)
    assert launches[-1]["threads"] == 64


def test_deferred_weight_is_one_of_the_first_row():
    """Sides 0.1 and 0.05 are equally frequent; the row sums start at 0.05's
    point, which then needs no multiply."""
    _, launches = _stencil((1000, 1001), "f64", "zero", 3, STAR2, W2)
    scales = [s for l in launches for s in l["deferred_scales"]]
    assert scales[:2] == [1, 1] and scales[2] == pytest.approx(0.05 ** 3, rel=1e-15)


@pytest.mark.parametrize("axis", [0, 1, 2])
def test_columns_leave_extents_within_a_block_of_2p31_alone(axis):
    """A block of the last rows or columns would reach past what an int holds."""
    shape = [1, 1, 1]
    shape[axis] = (1 << 31) - 1
    grp, _ = _stencil(tuple(shape), "f32", "zero", 2, programs.SEVEN_POINT, programs.SEVEN_WEIGHTS)
    assert grp["kernel_form"] == "tile"
