"""The row kernel's cuts (row_plan, row_batch_rows) stay inside what the kernel is
compiled for, over boxes of all shapes: a population's block with its widened copies
fits its slot, the interior its moments, the density warps their packed operands, the
collision turns the 32 bits of the wrap masks, a block's wrap in y its copies."""
import itertools
import random
import time

import pytest

import launch_rules


def boxes():
    rng = random.Random(7)
    sides = [3, 4, 5, 7, 8, 16, 31, 64, 100, 157, 256, 335]
    for b in itertools.product([3, 8, 33, 64, 157, 256, 440, 449, 512, 596, 597, 598, 768, 769], sides, sides):
        yield b
    for _ in range(600):
        yield tuple(int(round(2 ** rng.uniform(1.6, 9.6))) for _ in range(3))
    for b in [(3, 2000, 2000), (4, 1000, 1000), (16, 16, 4096), (64, 3, 5000), (201, 3, 2000), (768, 3, 400)]:
        yield b


def check_item(prec, box, by, zc, nd, nc):
    nx, ny, nz = box
    caps = launch_rules.row_caps(prec)
    ve = 8 if prec == "f16" else 4
    aligned = nx % ve == 0
    assert 1 <= by <= ny and 1 <= zc <= nz
    # a block with its shift (below 16 bytes), the step past the wrap (below two 16-byte
    # pieces) and the widened end
    assert (by + 2) * nx + (0 if aligned else 4 * ve) <= caps["slot"]
    assert by * nx <= caps["mcap"]
    assert (by + 2) * nx <= nd * caps["kd"] * 2
    turns = -(-by * nx // (2 * nc))
    assert turns * 2 <= 32
    assert nd + nc + 32 <= caps["threads"]
    # segments of a wrapping block: four for aligned rows, two for the others
    assert by + 2 <= (3 * ny if aligned else ny + 1)
    assert prec != "f16" or aligned


@pytest.mark.parametrize("prec", ["f32", "f16"])
def test_plans_fit(prec):
    planned = 0
    for box in boxes():
        p = launch_rules.row_plan(prec, box)
        if not p:
            continue
        planned += 1
        check_item(prec, box, p["by"], p["zc"], p["nd"], p["nc"])
        items = -(-box[1] // p["by"]) * -(-box[2] // p["zc"])
        assert p["items"] == items and p["grid"] == min(items, 152)
        assert p["aligned"] == (box[0] % (8 if prec == "f16" else 4) == 0)
    assert planned > 200


@pytest.mark.parametrize("prec", ["f32", "f16"])
def test_batch_items_fit(prec):
    caps = launch_rules.row_caps(prec)
    taken = 0
    for box in boxes():
        by = launch_rules.row_batch_rows(prec, 4, box)
        if by:
            taken += 1
            check_item(prec, box, by, box[2], caps["batch_nd"] * 32, caps["batch_nc"] * 32)
    assert taken > 200
    assert launch_rules.row_batch_rows(prec, 6, (64, 64, 64)) == 0
    assert launch_rules.row_batch_rows("f64", 4, (64, 64, 64)) == 0


def test_no_plan_for_fp64_and_small_boxes():
    assert launch_rules.row_plan("f64", (128, 128, 128)) is None
    assert launch_rules.row_plan("f32", (64, 64, 64)) is None
    assert launch_rules.row_plan("f32", (128, 128, 128))["ok"]


def test_a_long_box_is_planned_quickly():
    """Chunk counts that give the same planes are tried once: about 2 sqrt(nz) cuts per
    row count and not nz of them (14 million here)."""
    launch_rules.row_plan("f32", (64, 64, 100))
    t0 = time.perf_counter()
    launch_rules.row_plan("f32", (8, 8, 2000000))
    assert time.perf_counter() - t0 < 0.01


@pytest.mark.parametrize("prec,box,planned", [
    # blocks of few rows wrap around the box in y: three copies where one is usual
    ("f32", (64, 3, 5000), False), ("f32", (33, 3, 20000), False), ("f32", (32, 8, 8593), False),
    ("f32", (400, 6, 916), True), ("f32", (64, 24, 1432), True), ("f16", (64, 4, 8593), False),
    # items of one row, densities formed three times
    ("f32", (449, 80, 80), False), ("f32", (450, 64, 64), False), ("f32", (597, 64, 64), False),
    ("f32", (549, 100, 100), True), ("f32", (512, 100, 100), True), ("f32", (452, 30, 30), False),
    ("f16", (600, 64, 64), False), ("f16", (640, 20, 16), False), ("f16", (768, 100, 100), True),
    # ordinary boxes
    ("f32", (128, 128, 128), True), ("f32", (256, 256, 256), True), ("f32", (157, 157, 157), True),
    ("f32", (72, 72, 72), True), ("f32", (64, 64, 100), True), ("f32", (96, 96, 96), True), ("f32", (113, 113, 113), True), ("f32", (335, 335, 335), True),
    ("f32", (335, 41, 90), True), ("f32", (440, 48, 60), True), ("f16", (64, 64, 64), True),
    ("f16", (128, 128, 128), True), ("f16", (256, 256, 256), True), ("f16", (256, 40, 33), True),
])
def test_where_the_row_kernel_pays(prec, box, planned):
    """Measured on both sides of the line (GB300): the row kernel has a plan only where it is
    the faster one."""
    assert (launch_rules.row_plan(prec, box) is not None) == planned


@pytest.mark.parametrize("box", [(76, 72, 70), (440, 30, 28), (512, 40, 40)])
def test_without_the_psi_plane_rows_are_held_against_the_tile_kernels(box):
    """Boxes that the two passes take from the row kernel, where the workspace has no room
    for them: the moment kernel is slower than rows there."""
    assert launch_rules.row_plan("f32", box) is None
    assert launch_rules.row_plan("f32", box, passes=False)
