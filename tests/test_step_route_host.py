"""Which kernel a default step runs, by box, storage, stencil and tau, in a captured
graph and launched by itself."""
import pytest

import launch_rules

TILE, ROW, SPLIT = range(3)


@pytest.mark.parametrize("box", [(8, 8, 8), (32, 32, 32), (100, 3, 3), (300, 5, 5), (64, 32, 16)])
@pytest.mark.parametrize("unit_tau", [True, False])
def test_small_fp32_steps_take_one_launch_unless_captured(box, unit_tau):
    assert launch_rules.step_route("f32", box, unit_tau=unit_tau, eager=True) == TILE
    assert launch_rules.step_route("f32", box, unit_tau=unit_tau) == SPLIT


@pytest.mark.parametrize("prec,box,stencil,route", [
    ("f32", (33, 33, 33), 4, SPLIT), ("f32", (3, 100, 100), 4, SPLIT), ("f64", (8, 8, 8), 4, SPLIT),
    ("f32", (100, 5, 5), 6, TILE), ("f32", (100, 5, 5), 8, TILE), ("f32", (8, 8, 8), 6, SPLIT),
    ("f32", (32, 32, 32), 8, SPLIT), ("f64", (100, 5, 5), 8, SPLIT),
])
def test_where_the_line_lies(prec, box, stencil, route):
    assert launch_rules.step_route(prec, box, stencil, eager=True) == route
    assert launch_rules.step_route(prec, box, stencil) == SPLIT


def test_a_graph_holds_128_kernels():
    """A graph is captured anew after every initialisation, so two kernels a step do not
    make it twice as long."""
    for box, route in (((64, 64, 64), SPLIT), ((128, 128, 128), ROW)):
        assert launch_rules.step_route("f32", box) == route
        assert launch_rules.steps_per_graph(route) * (2 if route == SPLIT else 1) == 128
